"""The frame prior at every level count: the synthesis tile's halos (one to
four groups of columns) inside the image, across its edges, and on domains
that are no power of two. Compared with the FP64 oracle at the bound of the
frame iterates (2e-5: FP32 transforms and a few sums of 13 bands)."""
import numpy as np
import pytest

import oracle as O
import synth as S

pytestmark = pytest.mark.gpu

SIDES = [96, 160, 192, 320, 384, 640, 768, 1280, 1536]


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


@pytest.mark.parametrize("levels", [1, 2, 3, 4])
@pytest.mark.parametrize("H,W", [(64, 64), (96, 160), (160, 96), (64, 128)])
def test_every_level_count_matches_oracle(ad, H, W, levels):
    import torch
    g = S.rng(7 * levels + H + W)
    psf = S.psf_gaussian(7, 1.5)
    keep = (g.uniform(size=(H, W)) < 0.8).astype(np.uint8)
    ybar, mask, _ = S.observe(S.textured_image(H, W, g), psf, keep, 40.0, g)
    lam, mu1, mu2 = 1e-3, 3e-2, 1e-2
    st = O.State.zeros(H, W, "haar", levels)
    for _ in range(4):
        st = O.famd_step(st, ybar, mask, psf, lam, mu1, mu2, levels)
    plan = ad.Plan(H, W, psf, lam, mu1, mu2, "haar", levels=levels, max_iters=4)
    x = torch.full((H, W), float("nan"), device="cuda")
    ad.solve(plan, torch.from_numpy(ybar.astype(np.float32)).cuda(), torch.from_numpy(mask).cuda(), x)
    torch.cuda.synchronize()
    plan.close()
    assert np.linalg.norm(x.cpu().numpy() - st.x) <= 2e-5 * np.linalg.norm(st.x)
