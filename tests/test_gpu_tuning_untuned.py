"""The untuned class in the tuning table: its entry has every index 0, reading it
and setting it again changes nothing (its plans share a class, and so launches,
with plans made before), the autotuner may choose it, and row configuration 0 can
still be fixed by an entry that sets something else."""
import numpy as np
import pytest

import synth as S

pytestmark = pytest.mark.gpu

KEYS = ("H", "W", "reg", "haar_levels", "row_variant", "col_variant", "slot_ctas", "lanes")


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


@pytest.fixture(params=[(128, 512), (256, 1024), (512, 2048)])
def untuned(ad, request):
    """A class that no test has set before."""
    H, W = request.param
    zero = {"H": H, "W": W, "reg": ad.ADMM_REG_TV, "haar_levels": 0, "row_variant": 0, "col_variant": 0,
            "slot_ctas": 0, "lanes": 0}
    yield zero
    ad.admm_deconv_set_tuning(zero)


def _plan(ad, c):
    return ad.Plan(c["H"], c["W"], S.psf_box(5), 1e-3, max_iters=6)


def _solve(ad, plans):
    """x of every plan on one observation, and the kernels launched."""
    import torch
    H, W = plans[0].H, plans[0].W
    y = torch.from_numpy(S.rng(3).uniform(size=(H, W)).astype(np.float32)).cuda()
    xs = [torch.empty(H, W, device="cuda") for _ in plans]
    ad.admm_deconv_profile(False)
    ad.solve_batch(plans, [y] * len(plans), None, xs)
    return xs, ad.admm_deconv_profile(False).kernel_launches


def test_reading_and_setting_an_untuned_class_changes_nothing(ad, untuned):
    import torch
    got = ad.admm_deconv_get_tuning(untuned["H"], untuned["W"], "tv")
    assert all(got[k] == untuned[k] for k in KEYS)
    before = [_plan(ad, untuned) for _ in range(2)]
    ad.admm_deconv_set_tuning({k: got[k] for k in KEYS})
    after = _plan(ad, untuned)
    ad.admm_deconv_set_tuning({k: got[k] for k in KEYS} | {"lanes": 1})
    fixed = _plan(ad, untuned)
    want, launches = _solve(ad, before)
    xs, same = _solve(ad, [before[0], after])
    assert same == launches and all(torch.equal(a, b) for a, b in zip(xs, want))
    xs, other = _solve(ad, [before[0], fixed])   # two classes: other launches, the same bits
    assert other > launches and all(torch.equal(a, b) for a, b in zip(xs, want))
    for p in before + [after, fixed]:
        p.close()


def test_the_autotuners_winner_reads_back(ad):
    H, W = 256, 128
    zero = {"H": H, "W": W, "reg": ad.ADMM_REG_TV, "haar_levels": 0, "row_variant": 0, "col_variant": 0,
            "slot_ctas": 0, "lanes": 0}
    untouched = ad.admm_deconv_get_tuning(H, W, "tv")
    try:
        best, trials = ad.admm_deconv_autotune(H, W, "tv", problems=4, iters=8)
        got = ad.admm_deconv_get_tuning(H, W, "tv")
        assert all(got[k] == best[k] for k in (*KEYS, "rows_per_strip", "walk_depth", "row_threads", "us_per_iter"))
        # the trial with every index 0 is the untuned class: its rows are the default's, not entry 0's
        first = next(t for t in trials if all(t[k] == zero[k] for k in KEYS))
        ad.admm_deconv_set_tuning(zero)
        for got in (first, ad.admm_deconv_get_tuning(H, W, "tv")):
            assert all(got[k] == untouched[k] for k in (*KEYS, "rows_per_strip", "walk_depth", "row_threads"))
    finally:
        ad.admm_deconv_set_tuning(zero)
