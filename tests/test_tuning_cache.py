"""The JSON tuning cache: an entry written under other defaults (no generation in
its key, as before, or another one) is not replayed but measured again; one that
this library has written is. The calls to the GPU are stood in for."""
import json

import pytest


@pytest.fixture(scope="module")
def ad():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1210_2687_gb300 as mod
    return mod


@pytest.mark.parametrize("problems", [0, 24])
def test_entries_of_other_defaults_are_measured_again(ad, monkeypatch, tmp_path, problems):
    calls = []
    old = {"H": 512, "W": 512, "reg": 0, "haar_levels": 0, "row_variant": 3, "col_variant": 0, "slot_ctas": 0,
           "lanes": 0, "us_per_iter": 4.5}
    best = dict(old, row_variant=1, us_per_iter=4.25)
    monkeypatch.setattr(ad, "admm_deconv_autotune", lambda *a, **k: calls.append("tune") or (best, [best]))
    monkeypatch.setattr(ad, "admm_deconv_set_tuning", lambda cfg: calls.append(cfg["row_variant"]))
    monkeypatch.setattr(ad, "admm_deconv_get_tuning", lambda *a, **k: dict(best))
    key = ad.tuning_cache_key(512, 512, "tv", device_name="GPU", problems=problems)
    before = "GPU|512x512|tv|0" + (f"|p{problems}" if problems else "")
    path = tmp_path / "tuning.json"
    path.write_text(json.dumps({before: old, before + "|g1": old}))
    run = lambda: ad.autotune_cached(512, 512, "tv", path=str(path), device_name="GPU", problems=problems)  # noqa: E731
    assert run()["source"] == "autotune" and calls == ["tune"]
    assert json.loads(path.read_text())[key] == best
    assert run()["source"] == "cache" and calls == ["tune", 1]
    assert len({ad.tuning_cache_key(*a, device_name="GPU", problems=p) for a in ((512, 512, "tv"), (512, 512, "haar"),
                (512, 256, "tv"), (512, 512, "haar", 3)) for p in (0, 24, 2)}) == 12
