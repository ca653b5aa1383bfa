"""Elastic calls whose tiles exceed one per resident CTA run as two shot groups
on their own streams: the same results as the shots in smaller calls."""

import numpy as np
import pytest

from paper_2003_06027_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nshots", [77, 78])  # 6 tiles a shot: 462 and 468 tiles of 456; odd and even groups
def test_shot_groups_match_smaller_calls(fwi_lib, nshots):
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_elastic(11, 70, 75, 60, nshots, 4, 10, nrec=5, f0=6.0)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    kw = fwi.problem_kwargs(d)
    model = [cu(d[k]) for k in ("vp", "vs", "rho")]
    rec = [cu(d[k]) for k in ("rec_iz", "rec_ix")]
    stf, x0, mt = (cu(d[k]) for k in ("stf", "x0", "mt"))
    rng = np.random.default_rng(5)
    obs = cu((rng.standard_normal((nshots, 2, 5, 60)) * 1e-2).astype(np.float32))

    def call(a, b):
        return fwi.misfit_grad_elastic(*model, stf[a:b], x0[a:b], mt[a:b], *rec, obs[a:b].contiguous(), ckpt_every=25,
                                       want_seis=True, **kw)

    J, g, gs, gx, seis = call(0, nshots)
    assert torch.equal(seis, fwi.forward_elastic(*model, stf, x0, mt, *rec, **kw))
    h = nshots // 2
    parts = [call(0, h), call(h, nshots)]  # one group each
    assert torch.equal(seis, torch.cat([p[4] for p in parts]))
    assert torch.equal(gs, torch.cat([p[2] for p in parts])) and torch.equal(gx, torch.cat([p[3] for p in parts]))
    # sums over shots in FP64, rounded to FP32 once here and once per part there
    Js = float(parts[0][0][0] + parts[1][0][0])
    assert abs(float(J[0]) - Js) <= 1e-12 * Js
    gsum = parts[0][1].double() + parts[1][1].double()
    assert float((g.double() - gsum).norm()) <= 4 * 2.0**-24 * float(parts[0][1].double().norm() + parts[1][1].double().norm())
