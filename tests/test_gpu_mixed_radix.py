"""Every mixed-radix side as a row and as a column length (the leading radix-12
and radix-20 passes, the trailing radix 2 or none, a power of two beside it):
four TV iterations against the FP64 oracle, tolerance 2e-5 as for the other
short runs; rows and columns of 32 elements more or fewer change the pass plan."""
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


@pytest.mark.parametrize("side", SIDES)
@pytest.mark.parametrize("rows", [True, False])
def test_every_side_matches_oracle(ad, side, rows):
    import torch
    H, W = (64, side) if rows else (side, 96)
    g = S.rng(side)
    x = S.textured_image(H, W, g)
    psf = S.psf_motion(9.0, 40.0, 9)
    keep = (g.uniform(size=(H, W)) < 0.8).astype(np.uint8)
    ybar, mask, _ = S.observe(x, psf, keep, 40.0, g)
    lam, mu1, mu2 = 3e-4, 1e-2, 3e-3
    st = O.State.zeros(H, W, "tv")
    for _ in range(4):
        st = O.tvmd_step(st, ybar, mask, psf, lam, mu1, mu2)
    plan = ad.Plan(H, W, psf, lam, mu1, mu2, "tv", max_iters=4)
    xg = torch.full((H, W), float("nan"), device="cuda")
    ad.solve(plan, torch.from_numpy(ybar.astype(np.float32)).cuda(), torch.from_numpy(mask).cuda(), xg)
    plan.close()
    err = np.linalg.norm(xg.cpu().numpy() - st.x) / np.linalg.norm(st.x)
    assert err <= 2e-5, err
