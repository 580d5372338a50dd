"""Every compiled TV row configuration, and the choice that an untuned class
makes by the number of problems it solves, give the same bits: the strips and
the threads only divide the work."""
import numpy as np
import pytest

import oracle as O
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


def _problem(H, W, seed):
    g = S.rng(seed)
    psf = S.psf_gaussian(7, 1.5)
    keep = (g.uniform(size=(H, W)) < 0.7).astype(np.uint8)
    y, m, _ = S.observe(S.textured_image(H, W, g), psf, keep, 40.0, g)
    return psf, y, m


def _solve(ad, problems, general=True, **kw):
    import torch
    ad.admm_deconv_profile(general)      # per-phase timing keeps small images on the launches under test
    try:
        plans = [ad.Plan(*y.shape, psf, 3e-4, **kw) for psf, y, _ in problems]
        xs = [torch.full(y.shape, float("nan"), device="cuda") for _, y, _ in problems]
        ad.solve_batch(plans, [torch.from_numpy(y.astype(np.float32)).cuda() for _, y, _ in problems],
                       [torch.from_numpy(m).cuda() for _, _, m in problems], xs)
        torch.cuda.synchronize()
        for p in plans:
            p.close()
        return xs
    finally:
        ad.admm_deconv_profile(False)


@pytest.mark.parametrize("reg", ["tv", "tv_aniso"])
@pytest.mark.parametrize("W", [64, 128, 256, 512, 1024, 2048])
def test_every_row_configuration_gives_the_same_bits(ad, W, reg):
    import torch
    H = 64
    args = dict(reg=reg, max_iters=7, stop="rel_x", tol=0.0, check_every=3)
    p = [_problem(H, W, W)]
    want = _solve(ad, p, **args)[0]
    psf, y, m = p[0]
    if reg == "tv":
        mu1, mu2 = S.default_mu(3e-4)
        st = O.State.zeros(H, W, "tv")
        for _ in range(7):
            st = O.tvmd_step(st, y, m, psf, 3e-4, mu1, mu2)
        assert np.linalg.norm(want.cpu().numpy() - st.x) <= 2e-5 * np.linalg.norm(st.x)
    prev = ad.admm_deconv_get_tuning(H, W, "tv")
    rows, _ = ad.admm_deconv_variants(H, W, ad.ADMM_REG_TV)
    try:
        for v in range(rows):
            ad.admm_deconv_set_tuning({"H": H, "W": W, "reg": ad.ADMM_REG_TV, "haar_levels": 0, "row_variant": v,
                                       "col_variant": 0, "slot_ctas": 0, "lanes": 0})
            assert torch.equal(_solve(ad, p, **args)[0], want), v
    finally:
        ad.admm_deconv_set_tuning({**{k: prev[k] for k in ("H", "W", "reg", "haar_levels", "row_variant",
                                                           "col_variant", "slot_ctas", "lanes")}})


@pytest.mark.parametrize("H,W,count", [(256, 512, 9), (128, 1024, 9)])
def test_few_and_many_problems_give_the_same_bits(ad, H, W, count):
    import torch
    # (more than 1 Mpixel in flight: another strip than for one problem alone)
    problems = [_problem(H, W, 100 + i) for i in range(count)]
    args = dict(reg="tv", max_iters=9, stop="rel_x", tol=0.0, check_every=4)
    xs = _solve(ad, problems, general=False, **args)
    for i in (0, count - 1):
        assert torch.equal(_solve(ad, problems[i:i + 1], general=False, **args)[0], xs[i]), i
