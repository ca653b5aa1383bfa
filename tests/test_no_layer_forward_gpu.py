"""Recording steps without absorbing layers run a build of the 32-row step that holds
no layer operands: the same bits as 64- or 8-row tiles, both orders and operators, on
either side of the size up to which it is taken."""
import numpy as np
import pytest

from paper_2003_06027_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,op", [(4, 0), (8, 0), (4, 1), (8, 1)])
@pytest.mark.parametrize("nz,nx,S,nt", [(33, 70, 3, 80), (192, 320, 40, 40), (320, 640, 61, 12)])  # 12, 1200, 6100 tiles
def test_same_bits_as_other_heights(fwi_lib, nz, nx, S, nt, order, op):
    import torch

    from paper_2003_06027_gb300 import fwi

    d = synth.random_acoustic(nz, nz, nx, nt, S, order, 0, nrec=6)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    kw, args, seis = dict(fwi.problem_kwargs(d), op=op), [cu(d[k]) for k in ("c", "stf", "x0", "rec_iz", "rec_ix")], []
    for rows in (32, 0 if op else 64):  # 64 means 32 to the c^2 Laplacian; its 12 tiles run 8-row ones by default
        fwi.set_tile_shape(rows)
        try:
            seis.append(fwi.forward(*args, **kw))
        finally:
            fwi.set_tile_shape(0)
    assert torch.equal(seis[0], seis[1]) and bool(seis[0].abs().sum() > 0)
