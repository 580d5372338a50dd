"""Autotuner trials that come to the same launches: with few problems every slot
target puts all of them in flight, so the targets of one configuration share one
measurement, the default keeps the win, and the winner is the fastest."""
import pytest

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


@pytest.mark.parametrize("reg,H,W", [("tv", 64, 64), ("tv", 256, 512), ("haar", 128, 64)])
def test_one_measurement_per_layout(ad, reg, H, W):
    code = ad.ADMM_REG_TV if reg == "tv" else ad.ADMM_REG_HAAR
    try:
        best, trials = ad.admm_deconv_autotune(H, W, reg, problems=3, iters=8)
        nr, nc = ad.admm_deconv_variants(H, W, reg)
        assert len(trials) == nr * nc * 3 + 2
        assert best["us_per_iter"] == min(t["us_per_iter"] for t in trials) > 0
        assert best["slot_ctas"] == 0
        times = {}
        for t in trials[:-2]:
            if any(t[k] for k in ("row_variant", "col_variant", "slot_ctas", "lanes")):   # (all 0: rows by call)
                times.setdefault((t["row_variant"], t["col_variant"]), set()).add(t["us_per_iter"])
        assert all(len(v) == 1 for v in times.values())
    finally:
        ad.admm_deconv_set_tuning({"H": H, "W": W, "reg": code, "haar_levels": 4, "row_variant": 0, "col_variant": 0,
                                   "slot_ctas": 0, "lanes": 0})
