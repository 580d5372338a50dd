"""The bounded waits of the warm-start network: with one input row of a
streaming layer withheld (ADMM_OPT_TEST_CNN_STALL) every wait for it runs out,
the kernel ends, the device stays usable, and the next pass gives the bits of
an undisturbed one."""
import numpy as np
import pytest

import oracle.cnn as C
import synth as S

pytestmark = pytest.mark.gpu

SHAPE = (3, 48, 256)


@pytest.fixture(scope="module")
def ad():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.init()
    import paper_1210_2687_gb300 as mod
    return mod


@pytest.fixture
def stall(ad):
    """Arms the hook for the next pass; disarmed whatever the test does."""
    yield lambda: ad.admm_deconv_set_option(ad.ADMM_OPT_TEST_CNN_STALL, 1)
    ad.admm_deconv_set_option(ad.ADMM_OPT_TEST_CNN_STALL, 0)


def _net(ad, training=False):
    net = ad.Cnn(int(np.prod(SHAPE)), training=training)
    flat = np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in C.init_params(3)])
    net.set_params(flat.astype(np.float32))
    return net


def _inputs():
    import torch
    g = S.rng(8)
    y = torch.from_numpy(g.uniform(size=SHAPE).astype(np.float32)).cuda()
    m = torch.from_numpy((g.uniform(size=SHAPE) < 0.7).astype(np.uint8)).cuda()
    t = torch.from_numpy((0.5 * g.standard_normal((*SHAPE, 4))).astype(np.float32)).cuda()
    return y, m, t


def test_a_withheld_row_ends_and_the_device_stays_usable(ad, stall):
    import torch
    net = _net(ad)
    y, m, _ = _inputs()
    want, out = (torch.empty((*SHAPE, 4), device="cuda") for _ in range(2))
    net.forward(y, m, want)
    torch.cuda.synchronize()
    stall()
    try:
        net.forward(y, m, out)
        torch.cuda.synchronize()
        assert not torch.equal(out, want)
    finally:
        net.close()
    net = _net(ad)
    net.forward(y, m, out)
    assert torch.equal(out, want)
    net.close()
