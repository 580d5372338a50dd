"""Small TV images on teams of CTAs (clusters with distributed shared memory;
64 CTAs with a counter barrier at 256 x 256) against the general kernels, which
per-phase timing selects: the same iterates, duals and spectra bit for bit, over
every size, both differences' norms, all stop rules, warm starts, restored
states, several launches of one solve, more problems than are resident, padded
images and an observation that is not finite. Sums that only report (objective, relative changes) are added in
another order: 1e-6 relative, about a thousand FP64 roundings and one of FP32
per pixel's term."""
import numpy as np
import pytest

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
    x = S.textured_image(H, W, g)
    psf = S.psf_motion(7.0, 25.0, 7)
    keep = (g.uniform(size=(H, W)) < 0.75).astype(np.uint8)
    y, m, _ = S.observe(x, psf, keep, 40.0, g)
    return psf, y.astype(np.float32), m


def _run(ad, general, problems, plan_args, prepare=None):
    """x, full state and results of the problems solved in one call."""
    import torch
    ad.admm_deconv_profile(general)
    try:
        plans = [ad.Plan(*y.shape, psf, 3e-4, **plan_args) for psf, y, _ in problems]
        if prepare:
            for p in plans:
                prepare(p)
        ys = [torch.from_numpy(y).cuda() for _, y, _ in problems]
        ms = [torch.from_numpy(m).cuda() for _, _, m in problems]
        xs = [torch.full(y.shape, float("nan"), device="cuda") for y in ys]
        res = ad.solve_batch(plans, ys, ms, xs)
        states = []
        for p in plans:
            f = torch.empty(p.full_state_size(), device="cuda")
            p.get_full_state(f)
            states.append(f)
            p.close()
        return xs, states, res
    finally:
        ad.admm_deconv_profile(False)


def _same(a, b):
    import torch
    for i, (xa, xb) in enumerate(zip(a[0], b[0])):
        assert torch.equal(xa, xb), i
    for i, (sa, sb) in enumerate(zip(a[1], b[1])):
        assert torch.equal(sa, sb), i
    for ra, rb in zip(a[2], b[2]):
        assert (ra.iters, ra.converged, ra.status) == (rb.iters, rb.converged, rb.status)
        for f in ("objective", "rel_x", "primal_res"):
            u, v = getattr(ra, f), getattr(rb, f)
            assert u == v or abs(u - v) <= 1e-6 * abs(v), (f, u, v)


SIDES = (64, 128, 256)


@pytest.mark.parametrize("reg", ["tv", "tv_aniso"])
@pytest.mark.parametrize("H", SIDES)
@pytest.mark.parametrize("W", SIDES)
def test_same_bits_as_the_general_kernels(ad, H, W, reg):
    p = [_problem(H, W, H + 3 * W)]
    for args in (dict(max_iters=1), dict(max_iters=2), dict(max_iters=33),
                 dict(max_iters=60, stop="rel_x", tol=0.0, check_every=7),
                 dict(max_iters=400, stop="rel_x", tol=1e-3, check_every=3),
                 dict(max_iters=400, stop="rel_obj", tol=1e-3)):
        _same(_run(ad, False, p, dict(reg=reg, **args)), _run(ad, True, p, dict(reg=reg, **args)))


@pytest.mark.parametrize("H,W", [(64, 64), (128, 256), (256, 256)])
def test_starts_and_restarts(ad, H, W):
    import torch
    p = [_problem(H, W, 5)]
    g = torch.Generator().manual_seed(1)
    x0 = torch.rand(H, W, generator=g).cuda()
    d0 = (0.01 * torch.randn(3 * H * W, generator=g)).cuda()
    args = dict(max_iters=21, stop="rel_x", tol=0.0, check_every=4)
    warm = lambda pl: pl.warm_start(x0, d0)  # noqa: E731
    a = _run(ad, False, p, args, warm)
    _same(a, _run(ad, True, p, args, warm))
    resume = lambda pl: pl.set_state(a[1][0])  # noqa: E731
    _same(_run(ad, False, p, args, resume), _run(ad, True, p, args, resume))


@pytest.mark.parametrize("H,W", [(64, 128), (256, 256)])
def test_several_launches(ad, H, W):
    p = [_problem(H, W, 9)]
    args = dict(max_iters=1100, stop="rel_x", tol=0.0, check_every=10)
    _same(_run(ad, False, p, args), _run(ad, True, p, args))


@pytest.mark.parametrize("H,W,count", [(64, 64, 40), (128, 128, 14), (128, 256, 7), (256, 256, 2)])
def test_many_problems(ad, H, W, count):
    p = [_problem(H, W, 100 + i) for i in range(count)]
    args = dict(max_iters=300, stop="rel_x", tol=2e-3, check_every=5)
    a = _run(ad, False, p, args)
    _same(a, _run(ad, True, p, args))
    assert len({r.iters for r in a[2]}) > 1          # they retire at different iterations


def test_padded_and_not_finite(ad):
    p = [_problem(60, 101, 3)]
    args = dict(max_iters=25, pad=True, reg="tv")
    _same(_run(ad, False, p, args), _run(ad, True, p, args))
    psf, y, m = _problem(64, 64, 4)
    y = y.copy()
    y[tuple(np.argwhere(m)[0])] = np.inf
    a, b = (_run(ad, k, [(psf, y, m), _problem(64, 64, 6)], dict(max_iters=10)) for k in (False, True))
    assert [r.status for r in a[2]] == [r.status for r in b[2]] == [ad.ADMM_ENONFINITE, 0]
    assert (a[0][1] == b[0][1]).all()


@pytest.mark.parametrize("H,W", [(64, 64), (128, 256), (256, 256)])
def test_tuned_classes(ad, H, W):
    p = [_problem(H, W, 13)]
    args = dict(max_iters=25, stop="rel_x", tol=0.0, check_every=4)
    want = _run(ad, True, p, args)
    prev = ad.admm_deconv_get_tuning(H, W, "tv")
    keys = ("H", "W", "reg", "haar_levels", "row_variant", "col_variant", "slot_ctas", "lanes")
    try:
        for rv, cv in ((1, 0), (2, 1), (0, 3)):
            ad.admm_deconv_set_tuning({**{k: prev[k] for k in keys}, "row_variant": rv, "col_variant": cv})
            _same(_run(ad, False, p, args), want)
    finally:
        ad.admm_deconv_set_tuning({k: prev[k] for k in keys})
