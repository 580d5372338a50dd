"""Weight and bias gradients on tcgen05 at the edges of their tiles (16 x 32
output pixels per tile, tiles walked by one CTA per SM): images narrower than
a tile, ragged in columns, several images, one tile per CTA and more tiles
than the CTAs and their three stages hold. Reference: the network in 64-bit
arithmetic with every value that the library stores in BF16 (weights,
activations, their gradients) rounded to BF16. Tolerance per parameter tensor:
one BF16 unit in the last place, 2^-8 relative (values that round the other
way after FP32 accumulation in another order); a lost tap, row, column or tile
is off by more than 1 / (number of pixels along an edge) > 2^-8 here."""
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


def _reference(params, ybar, mask, tgt, cw):
    import torch
    import torch.nn.functional as F
    bf = lambda v: v.to(torch.bfloat16).double()  # noqa: E731
    n, H, W = ybar.shape
    acts = [bf(torch.stack([torch.where(mask != 0, ybar, 0.0), mask.double()], 1))]
    ws = [bf(w) for w, _ in params]
    for l, (_, b) in enumerate(params):
        z = F.conv2d(acts[-1], ws[l], b, padding=1)
        acts.append(bf(torch.relu(z)) if l < len(params) - 1 else z)
    c = torch.tensor(cw, dtype=torch.float64).view(1, 4, 1, 1)
    e = acts[-1].float().double() - tgt.permute(0, 3, 1, 2)
    g = bf(2 * c * e / (n * H * W))
    out = []
    for l in range(len(params) - 1, -1, -1):
        p = F.pad(acts[l], (1, 1, 1, 1))
        gw = torch.stack([torch.einsum("nohw,nihw->oi", g, p[:, :, t // 3:t // 3 + H, t % 3:t % 3 + W])
                          for t in range(9)], -1)
        out.append((gw.reshape(-1), g.sum((0, 2, 3))))
        if l:
            g = bf(F.conv_transpose2d(g, ws[l], padding=1) * (acts[l] > 0))
    return out[::-1]


@pytest.mark.parametrize("count,H,W", [(1, 16, 16), (1, 16, 48), (3, 48, 80), (2, 32, 1024), (9, 160, 336)])
def test_gradients_at_tile_edges(ad, count, H, W):
    import torch
    ps = C.init_params(5)
    ps[-1][0] *= 10.0
    g = S.rng(7 * count + H + W)
    for _, b in ps:
        b[:] = 0.05 * g.standard_normal(b.shape)
    flat = np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in ps]).astype(np.float32)
    ybar = g.uniform(size=(count, H, W)).astype(np.float32)
    mask = (g.uniform(size=(count, H, W)) < 0.7).astype(np.uint8)
    tgt = (0.5 * g.standard_normal((count, H, W, 4))).astype(np.float32)
    cw = (1.0, 0.5, 2.0, 1.5)
    net = ad.Cnn(count * H * W, training=True)
    net.set_params(flat)
    dev = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    grads = [torch.full((net.param_count(),), float("nan"), device="cuda") for _ in range(2)]
    for v in grads:
        net.gradients(dev(ybar), dev(mask), dev(tgt), cw, v)
    net.close()
    assert torch.equal(grads[0], grads[1])           # the CTAs' shares are added in a fixed order
    got = grads[0].cpu().double()
    o = 0
    tp = [(torch.from_numpy(w.astype(np.float32)).double(), torch.from_numpy(b.astype(np.float32)).double()) for w, b in ps]
    ref = _reference(tp, torch.from_numpy(ybar).double(), torch.from_numpy(mask), torch.from_numpy(tgt).double(), cw)
    for l, parts in enumerate(ref):
        for k, r in enumerate(parts):
            v = got[o:o + r.numel()]
            o += r.numel()
            err = float((v - r).norm() / r.norm())
            assert err <= 2.0 ** -8, (l, "wb"[k], err)
    assert o == got.numel()
