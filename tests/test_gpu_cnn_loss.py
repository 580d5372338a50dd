"""The training loss as a sum in 64 bits: against numpy's over the network's own
output (whose bits the forward call returns), to one rounding per squared error
(a sum of N positive terms in any order is within N 2^-53 relative), and with
errors whose squares leave the FP32 range: large, tiny and infinite."""
import numpy as np
import pytest

import oracle.cnn as C
import synth as S

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("shape", [(1, 16, 16), (2, 48, 208), (3, 240, 256)])
@pytest.mark.parametrize("kind", ["ordinary", "large", "tiny", "one infinite"])
def test_loss_is_a_64_bit_sum(ad, shape, kind):
    import torch
    g = S.rng(31)
    y = torch.from_numpy(g.uniform(size=shape).astype(np.float32)).cuda()
    m = torch.from_numpy((g.uniform(size=shape) < 0.7).astype(np.uint8)).cuda()
    flat = np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in C.init_params(3)]).astype(np.float32)
    if kind == "tiny":
        flat[:] = 0.0                            # the network's output is 0, so the errors are the targets
    net = ad.Cnn(int(np.prod(shape)), training=True)
    net.set_params(flat)
    out = torch.empty((*shape, 4), device="cuda")
    net.forward(y, m, out)
    t = g.standard_normal((*shape, 4)).astype(np.float32)
    t *= {"ordinary": 1.0, "large": 1e21, "tiny": 1e-24, "one infinite": 1.0}[kind]
    if kind == "one infinite":
        t[0, 3, 5, 1] = np.inf
    cw = np.array([1.0, 0.5, 2.0, 0.25])
    loss = net.gradients(y, m, torch.from_numpy(t).cuda(), cw, torch.empty(ad.Cnn.param_count(), device="cuda"))
    net.close()
    e = (out.cpu().numpy() - t).astype(np.float64)   # (the error itself is an FP32 difference)
    want = float((cw * e ** 2).sum() / np.prod(shape))
    if kind == "one infinite":
        assert loss == want == np.inf
    else:
        assert abs(loss - want) <= e.size * 2.0 ** -53 * want and want > 0
