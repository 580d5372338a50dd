"""The network's layers streamed in strips of 128 columns, at the widths where
a strip is ragged or its rule changes over to 8 x 16 tiles (the strips may be
at most a quarter wider than the image), with fewer rows than CTAs, several
images per CTA and segments that end inside an image. Reference: the network
in 64-bit arithmetic with the values that are stored in BF16 rounded to BF16;
tolerance one BF16 unit in the last place (2^-8 relative, as a value that rounds the other way moves
by one), against a lost column, row or tap that moves it by far more."""
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


def _reference(ps, ybar, mask):
    import torch
    import torch.nn.functional as F
    bf = lambda v: v.to(torch.bfloat16).double()  # noqa: E731
    a = bf(torch.stack([torch.where(mask != 0, ybar, 0.0), mask.double()], 1))
    for l, (w, b) in enumerate(ps):
        z = F.conv2d(a, bf(torch.from_numpy(w.astype(np.float32)).double()), torch.from_numpy(b).float().double(), padding=1)
        a = bf(torch.relu(z)) if l < len(ps) - 1 else z
    return a.permute(0, 2, 3, 1)


@pytest.mark.parametrize("count,H,W", [(1, 16, 112), (1, 16, 128), (2, 32, 96), (3, 48, 208), (1, 176, 240),
                                       (5, 64, 272), (7, 80, 320), (2, 208, 512), (1, 32, 1040)])
def test_forward_at_strip_edges(ad, count, H, W):
    import torch
    ps = C.init_params(11)
    ps[-1][0] *= 10.0
    g = S.rng(3 * count + H + W)
    for _, b in ps:
        b[:] = 0.05 * g.standard_normal(b.shape)
    flat = np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in ps]).astype(np.float32)
    ybar = g.uniform(size=(count, H, W)).astype(np.float32)
    mask = (g.uniform(size=(count, H, W)) < 0.7).astype(np.uint8)
    y, m = torch.from_numpy(ybar).cuda(), torch.from_numpy(mask).cuda()
    net = ad.Cnn(count * H * W)
    net.set_params(flat)
    out = torch.full((count, H, W, 4), float("nan"), device="cuda")
    net.forward(y, m, out)
    x0, d0 = torch.empty(count, H, W, device="cuda"), torch.empty(count, 3 * H * W, device="cuda")
    sc = (0.5, 2.0, 0.25, 0.0)
    net.predict_start(y, m, sc, x0, d0)
    torch.cuda.synchronize()
    net.close()
    ref = _reference(ps, torch.from_numpy(ybar).double(), torch.from_numpy(mask))
    got = out.cpu().double()
    assert float((got - ref).norm() / ref.norm()) <= 2.0 ** -8
    # border rows and columns by themselves: a fault there is not hidden by the interior
    for sl in ((slice(None), 0), (slice(None), -1), (slice(None), slice(None), 0), (slice(None), slice(None), -1)):
        assert float((got[sl] - ref[sl]).norm() / ref[sl].norm()) <= 2.0 ** -7
    # the start is the output times its scales, in the solver's layout
    assert torch.equal(x0, sc[0] * out[..., 0])
    assert torch.equal(d0[:, :H * W].view(count, H, W), sc[1] * out[..., 1])
    assert torch.equal(d0[:, H * W:].view(count, H, W, 2), sc[2] * out[..., 2:])
