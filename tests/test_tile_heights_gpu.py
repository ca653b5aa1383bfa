"""The forward step's tile heights (8 rows by default on small grids, 32, 64)
give the same results bit for bit, for both acoustic operators."""

import numpy as np
import pytest

import oracle
from paper_2003_06027_gb300 import synth

pytestmark = pytest.mark.gpu


# padded heights around the tile edges: below one 8-row tile, one row past a multiple of 8, 32 and 64
@pytest.mark.parametrize("nz,nx,npml,order,op", [(5, 9, 0, 4, 0), (23, 66, 5, 8, 1), (47, 130, 9, 4, 1), (115, 59, 7, 8, 0)])
def test_tile_heights_agree(fwi_lib, nz, nx, npml, order, op):
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_acoustic(nz, nz, nx, 90, 2, order, npml, src_kind=0, nrec=6)
    d["rec_iz"][:2] = [nz - 1, 0]
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    kw = dict(fwi.problem_kwargs(d), op=op)
    args = [cu(d[k]) for k in ("c", "stf", "x0", "rec_iz", "rec_ix")]
    obs = torch.zeros((2, 6, 90), device="cuda")
    out = {}
    for rows in (0, 32, 64):
        fwi.set_tile_shape(rows)
        try:
            J, g, gs, _, seis = fwi.misfit_grad(*args, obs, ckpt_every=20, want_seis=True, **kw)
            out[rows] = (fwi.forward(*args, **kw), J, g, gs, seis)
        finally:
            fwi.set_tile_shape(0)
    for rows in (32, 64):
        for a, b in zip(out[0], out[rows]):
            assert torch.equal(a, b)
    assert torch.equal(out[0][0], out[0][4])
    geo = dict(nz=nz, nx=nx, npml=npml, order=order, nt=90, dz=d["dz"], dx=d["dx"], dt=d["dt"], src_kind=0,
               pml_R=d["pml_R"], pml_vmax=d["pml_vmax"], pml_f0=d["pml_f0"], rec_iz=d["rec_iz"], rec_ix=d["rec_ix"], op=op)
    do = oracle.acoustic_forward(geo, np.float64(d["c"]), np.float64(d["stf"]), np.float64(d["x0"]))
    # FP32 against FP64 over 90 steps: well inside the 1e-4 of the other parity tests
    assert np.linalg.norm(out[0][0].cpu().numpy() - do) <= 1e-4 * np.linalg.norm(do)
