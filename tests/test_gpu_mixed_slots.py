"""How many problems of a class iterate at once. Alone, as many as there are (up
to 9600 row-side CTAs); in a call of several classes about 3600 CTAs' worth (four
of the 1024 tiles of a 1024^2 frame image), and all where the rest would be no
more than half as many again."""
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


@pytest.mark.parametrize("count,mixed,at_once", [(7, False, 7), (6, True, 6), (7, True, 4), (9, True, 4)])
def test_problems_in_flight(ad, count, mixed, at_once):
    import torch
    frames = [ad.Plan(1024, 1024, S.psf_box(5), 1e-3, reg="haar", max_iters=6) for _ in range(count)]
    small = [ad.Plan(64, 64, S.psf_box(5), 1e-3, max_iters=6)] if mixed else []
    plans = frames + small
    g = S.rng(1)
    ys = [torch.from_numpy(g.uniform(size=(p.H, p.W)).astype(np.float32)).cuda() for p in plans]
    xs = [torch.empty_like(y) for y in ys]
    res = ad.solve_batch(plans, ys, None, xs)
    assert all(r.iters == 6 and r.status == ad.ADMM_OK for r in res)
    first_done = min(r.t_done_ms for r in res[:count])
    assert sum(r.t_start_ms < first_done for r in res[:count]) == at_once
    for p in plans:
        p.close()
