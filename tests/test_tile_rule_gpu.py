"""The forward step's default tile height: launches whose 8-row tiles would take more
than one wave run 32-row ones, so the default is not slower than 32 rows asked for;
recording, keeping and recomputing steps of one gradient may differ in height."""
import numpy as np
import pytest

from paper_2003_06027_gb300 import synth

pytestmark = pytest.mark.gpu


def _problem(nz, nx, S, nt):
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_acoustic(S, nz, nx, nt, S, 4, 32, nrec=6)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    return fwi.problem_kwargs(d), [cu(d[k]) for k in ("c", "stf", "x0", "rec_iz", "rec_ix")]


# 720 tiles of 32 rows in two groups; 360 in one; 540 in groups of two shots and one
@pytest.mark.parametrize("nz,nx,S,groups", [(128, 256, 24, 0), (128, 256, 12, 1), (400, 700, 3, 0)])
def test_default_height_is_not_slower_than_32_rows(fwi_lib, nz, nx, S, groups):
    from paper_2003_06027_gb300 import fwi

    kw, args = _problem(nz, nx, S, 400)
    fwi.set_shot_groups(groups, 0)
    best = {}
    try:
        for _ in range(5):
            for rows in (0, 32):
                fwi.set_tile_shape(rows)
                fwi.forward(*args, **kw)
                best[rows] = min(best.get(rows, 1e9), fwi.last_timing().fwd_step_ms)
    finally:
        fwi.set_tile_shape(0)
        fwi.set_shot_groups(0, 0)
    # 8-row tiles took 1.45 to 1.6 times as long at these sizes
    assert best[0] <= 1.2 * best[32]


@pytest.mark.parametrize("nz,nx,S", [(400, 700, 3), (128, 256, 24), (70, 90, 5)])
def test_mixed_heights_give_the_same_bits(fwi_lib, nz, nx, S):
    import torch

    from paper_2003_06027_gb300 import fwi

    kw, args = _problem(nz, nx, S, 60)
    obs = torch.zeros((S, 6, 60), device="cuda")
    out = []
    for rows in (0, 32):
        fwi.set_tile_shape(rows)
        try:
            out.append(fwi.misfit_grad(*args, obs, ckpt_every=25, want_seis=True, **kw))
        finally:
            fwi.set_tile_shape(0)
    for a, b in zip(*out):
        assert a is None and b is None or torch.equal(a, b)


# 1200 and 1152 tiles: two launches a step would each take a second wave, three fit; 1380, 1408 and 1672: three
# launches, not all of one wave; 1500 and 2160 tiles: none of two, three or four fits
@pytest.mark.parametrize("nz,nx,S,order,npml", [
    (192, 320, 40, 8, 0), (192, 320, 40, 4, 0), (306, 310, 16, 4, 32), (128, 256, 46, 8, 32), (436, 436, 11, 4, 32),
    (536, 636, 8, 4, 32), (306, 310, 30, 4, 32), (32, 236, 100, 8, 32),
])
def test_default_groups_are_not_slower_than_four(fwi_lib, nz, nx, S, order, npml):
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_acoustic(S, nz, nx, 400, S, order, npml, nrec=6)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    kw, args, best, seis = fwi.problem_kwargs(d), [cu(d[k]) for k in ("c", "stf", "x0", "rec_iz", "rec_ix")], {}, {}
    try:
        for _ in range(5):
            for groups in (0, 4):
                fwi.set_shot_groups(groups, 0)
                seis[groups] = fwi.forward(*args, **kw)
                best[groups] = min(best.get(groups, 1e9), fwi.last_timing().fwd_step_ms)
    finally:
        fwi.set_shot_groups(0, 0)
    assert torch.equal(seis[0], seis[4])
    # two groups took 1.04 to 1.3 times as long as four at most of these sizes
    assert best[0] <= 1.05 * best[4]
