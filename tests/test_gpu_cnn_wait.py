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


def test_the_next_call_reports_an_asynchronous_pass(ad, stall):
    import torch
    net = _net(ad)
    y, m, _ = _inputs()
    want, out = (torch.empty((*SHAPE, 4), device="cuda") for _ in range(2))
    net.forward(y, m, want)
    stall()
    net.forward(y, m, out)                       # does not wait for the device
    torch.cuda.synchronize()
    with pytest.raises(ad.AdmmError) as e:
        net.predict_start(y, m, (1.0, 1.0, 1.0, 0.0), out[..., 0].contiguous(), torch.empty(3 * out[..., 0].numel(), device="cuda"))
    assert e.value.code == ad.ADMM_ETIMEOUT
    net.forward(y, m, out)                       # reported once: the network is usable again
    assert torch.equal(out, want)
    net.close()


def test_gradients_and_training_report_and_leave_the_step_out(ad, stall):
    import torch
    y, m, t = _inputs()
    cw = (1.0, 0.5, 2.0, 2.0)
    g = [torch.empty(ad.Cnn.param_count(), device="cuda") for _ in range(2)]
    nets = [_net(ad, training=True) for _ in range(2)]
    nets[0].gradients(y, m, t, cw, g[0])
    stall()
    with pytest.raises(ad.AdmmError) as e:
        nets[1].gradients(y, m, t, cw, g[1])
    assert e.value.code == ad.ADMM_ETIMEOUT
    nets[1].gradients(y, m, t, cw, g[1])
    assert torch.equal(g[0], g[1])
    # steps that fail: one that is waited for, then one that is not with a good
    # one queued behind it (left out as well); Adam's count does not move
    nets[0].train_step(y, m, t, cw, 1e-3)
    nets[1].train_step(y, m, t, cw, 1e-3)
    before = nets[1].get_params()
    stall()
    with pytest.raises(ad.AdmmError):
        nets[1].train_step(y, m, t, cw, 1e-3)
    assert np.array_equal(nets[1].get_params(), before)
    stall()
    nets[1].train_step(y, m, t, cw, 1e-3, want_loss=False)
    nets[1].train_step(y, m, t, cw, 1e-3, want_loss=False)
    with pytest.raises(ad.AdmmError):
        nets[1].get_params()
    assert np.array_equal(nets[1].get_params(), before)
    for n in nets:
        n.train_step(y, m, t, cw, 1e-3)
    assert np.array_equal(nets[0].get_params(), nets[1].get_params())
    for n in nets:
        n.close()


def test_a_learned_start_that_fails_fails_the_call(ad, stall):
    import torch
    from paper_1210_2687_gb300 import warmstart as ws
    H, W = 128, 256
    g = S.rng(4)
    y = torch.from_numpy(g.uniform(size=(H, W)).astype(np.float32)).cuda()
    ad.admm_warmstart_load(ws.WEIGHTS_BIN)
    try:
        plans = [ad.Plan(H, W, S.psf_box(5), 1e-3, reg=reg, max_iters=4) for reg in ("tv", "tv", "haar")]
        xs = [[torch.empty_like(y) for _ in plans] for _ in range(2)]
        solve = lambda x: ad.solve_batch(plans, [y] * 3, None, x, use_warmstart=True)  # noqa: E731
        assert all(r.status == ad.ADMM_OK for r in solve(xs[0]))
        stall()
        res = solve(xs[1])
        assert [(r.status, r.iters, r.converged) for r in res] == [(ad.ADMM_ETIMEOUT, 0, 0)] * 3
        assert all(r.status == ad.ADMM_OK and r.iters == 4 for r in solve(xs[1]))
        assert all(torch.equal(a, b) for a, b in zip(*xs))
        for p in plans:
            p.close()
    finally:
        ad.admm_warmstart_load(None)
