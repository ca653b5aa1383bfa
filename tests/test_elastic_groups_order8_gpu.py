"""Shot groups of 8th-order elastic calls, whose kernels hold two CTAs on an SM: two
groups from 305 tiles on, with the results of the shots in smaller calls."""
import numpy as np
import pytest

from paper_2003_06027_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nshots,groups", [(50, 1), (51, 2), (52, 2), (77, 2)])  # 6 tiles a shot: 300 to 462
def test_groups_from_one_tile_per_resident_cta(fwi_lib, nshots, groups):
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_elastic(11, 70, 75, 60, nshots, 8, 10, nrec=5, f0=6.0)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    kw = fwi.problem_kwargs(d)
    model = [cu(d[k]) for k in ("vp", "vs", "rho")]
    rec = [cu(d[k]) for k in ("rec_iz", "rec_ix")]
    stf, x0, mt = (cu(d[k]) for k in ("stf", "x0", "mt"))
    obs = cu((np.random.default_rng(5).standard_normal((nshots, 2, 5, 60)) * 1e-2).astype(np.float32))

    def call(a, b):
        out = fwi.misfit_grad_elastic(*model, stf[a:b], x0[a:b], mt[a:b], *rec, obs[a:b].contiguous(), ckpt_every=25,
                                      want_seis=True, **kw)
        return out, fwi.last_timing().launches

    (J, g, gs, gx, seis), n = call(0, nshots)
    parts = [call(0, 25), call(25, nshots)]
    if nshots <= 75:  # both parts are one group
        # per group: 2 x 60 forward, 2 x 50 recomputed and 2 x 60 adjoint launches
        assert n - parts[0][1] == (groups - 1) * 340
    assert torch.equal(seis, torch.cat([p[0][4] for p in parts]))
    assert torch.equal(gs, torch.cat([p[0][2] for p in parts])) and torch.equal(gx, torch.cat([p[0][3] for p in parts]))
    assert torch.equal(seis, fwi.forward_elastic(*model, stf, x0, mt, *rec, **kw))
    # sums over shots in FP64, rounded to FP32 once here and once per part there
    a, b = (p[0][1].double() for p in parts)
    assert float((g.double() - (a + b)).norm()) <= 4 * 2.0**-24 * float(a.norm() + b.norm())


@pytest.mark.parametrize("nz,nx,nshots,groups", [(66, 914, 13, 1), (66, 914, 12, 2), (400, 700, 3, 1), (76, 108, 104, 2)])
def test_one_launch_of_two_waves_stays_one(fwi_lib, nz, nx, nshots, groups):
    # 585 tiles as 315 + 270, 540 as 270 + 270, 504 as 336 + 168, 624 as 312 + 312, of 304 places
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_elastic(5, nz, nx, 20, nshots, 8, 10, dx=5.0, dt=4e-4, nrec=3)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    kw, model = fwi.problem_kwargs(d), [cu(d[k]) for k in ("vp", "vs", "rho")]
    src, rec = [cu(d[k]) for k in ("stf", "x0", "mt")], [cu(d[k]) for k in ("rec_iz", "rec_ix")]
    seis = fwi.forward_elastic(*model, *src, *rec, **kw)
    n = fwi.last_timing().launches
    part = fwi.forward_elastic(*model, *[a[:1].contiguous() for a in src], *rec, **kw)  # one group
    assert n - fwi.last_timing().launches == (groups - 1) * 40  # 2 launches for each of 20 steps
    assert torch.equal(part, seis[:1])
