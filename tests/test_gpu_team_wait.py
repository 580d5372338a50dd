"""The bounded barrier of a 256 x 256 image's team (64 CTAs, a counter in L2):
with the stall hook one CTA gives up at the end of the first iteration. Where
nothing follows, its status alone tells; where an iteration follows, the other
CTAs' waits for it run out (about a second). Either way the problem retires with
ADMM_ETIMEOUT, and the next solve of the plan gives an undisturbed plan's bits."""
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


@pytest.mark.parametrize("args", [dict(max_iters=1), dict(max_iters=6), dict(max_iters=600, stop="rel_x", tol=0.0),
                                  dict(max_iters=6, stop="rel_obj", tol=0.0)])
def test_one_cta_gives_up(ad, args):
    import torch
    H = W = 256
    g = S.rng(21)
    psf = S.psf_box(9)
    y, m, _ = S.observe(S.textured_image(H, W, g), psf, None, 40.0, g)
    y, m = torch.from_numpy(y.astype(np.float32)).cuda(), torch.from_numpy(m).cuda()
    plans = [ad.Plan(H, W, psf, 3e-4, **args) for _ in range(2)]
    x = [torch.empty(H, W, device="cuda") for _ in range(2)]
    ad.admm_deconv_profile(False)                    # (read and reset the launch counter)
    ad.admm_deconv_set_option(ad.ADMM_OPT_TEST_STALL, 1)
    res = ad.solve(plans[0], y, m, x[0])
    assert res.status == ad.ADMM_ETIMEOUT and res.iters == 1 and res.converged == 0
    # one launch of the team: the general kernels, whose hook withholds a copy, take two per iteration
    launches = ad.admm_deconv_profile(False).kernel_launches
    for p, v in zip(plans, x):
        res = ad.solve(p, y, m, v)
        assert res.status == ad.ADMM_OK and res.iters == args["max_iters"]
    assert torch.equal(*x)
    again = ad.admm_deconv_profile(False).kernel_launches
    assert 2 * launches == again if args["max_iters"] <= 512 else 2 * launches + 2 == again
    for p in plans:
        p.close()
