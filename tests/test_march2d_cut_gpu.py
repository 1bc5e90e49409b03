"""The 2D kernel where its launch changes: rows of 129 to 256 nodes with the KL field at the Gauss points (its cosines lie in
a table that the block shares), three fields on wide, tall grids and just beside that line (three blocks to an SM), and batches
that one wave of units fills, against the oracle (the repository's 1e-5), with masked and raw residuals and imposed faces."""
import numpy as np
import pytest

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import check, make_problems, run_gpu

pytestmark = pytest.mark.gpu
KG, KN, ND = B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL

CASES = [(KG, False, 132, 9, 3, 1), (KG, True, 136, 3, 5, 2), (KG, False, 192, 70, 2, 5), (KG, False, 255, 21, 2, 3), (KG, True, 256, 64, 9, 1),
         (KG, False, 257, 12, 3, 2),
         (ND, True, 1024, 256, 1, 1), (ND, True, 1024, 255, 1, 1), (ND, True, 1020, 256, 2, 1), (ND, True, 1025, 256, 1, 1), (ND, True, 2048, 300, 1, 1),
         (ND, False, 64, 512, 74, 1), (KN, False, 128, 300, 37, 2), (KG, False, 513, 74, 33, 2)]


@pytest.mark.parametrize("mode,forcing,nx,ny,batch,m", CASES)
def test_cut(mode, forcing, nx, ny, batch, m):
    inp = inputs.random_inputs(2, nx, ny, 1, batch, m, seed=nx + ny, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == ND else None
    f = inputs.random_field(inp.u.shape, 9, scale=3.0) if forcing else None
    gJ = np.linspace(-1.5, 2.0, batch).astype(np.float32)
    for flags in (0, B.DN_NO_MASK, B.DN_IMPOSE_BC_ON_LOAD):
        po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
        Jo, _, _, ro = oracle.energy_grad(po, u, gJ=gJ.astype(np.float64))
        Jg, rg = run_gpu(pg, u, gJ=gJ)
        check(Jg, rg, Jo, ro, f"flags {flags}")
