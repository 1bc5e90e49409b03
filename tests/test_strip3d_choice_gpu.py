"""3D problems on both sides of every line between the scalar and the mirrored-pair kernel (rows of 8 to 256 nodes, with and
without nodal forcing, few and many modes), and the scalar kernel's eight nodes per lane (stored field with nodal forcing on
rows of more than 128 nodes), against the oracle (the repository's 1e-5), with masked and raw residuals."""
import numpy as np
import pytest

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import check, make_problems, run_gpu

pytestmark = pytest.mark.gpu
KG, KN, ND = B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL

CASES = [(ND, True, 136, 9, 5, 2, 1), (ND, True, 200, 12, 4, 1, 1), (ND, True, 256, 6, 7, 2, 1), (ND, False, 136, 7, 4, 1, 1), (ND, False, 128, 9, 5, 2, 1),
         (KG, False, 36, 9, 7, 2, 2), (KG, False, 124, 6, 5, 1, 8), (KG, False, 60, 40, 40, 23, 4), (KN, False, 100, 9, 6, 2, 3), (KN, True, 72, 9, 6, 2, 3),
         (KN, True, 128, 46, 46, 1, 2), (KG, True, 40, 9, 6, 3, 3), (KG, True, 112, 49, 48, 1, 5), (KG, False, 64, 22, 23, 1, 2), (KG, False, 64, 23, 23, 1, 2),
         (KN, False, 96, 18, 18, 1, 4)]


@pytest.mark.parametrize("mode,forcing,nx,ny,nz,batch,m", CASES)
def test_either_side(mode, forcing, nx, ny, nz, batch, m):
    inp = inputs.random_inputs(3, nx, ny, nz, batch, m, seed=nx + ny, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == ND else None
    f = inputs.random_field(inp.u.shape, 9, scale=3.0) if forcing else None
    gJ = np.linspace(-1.5, 2.0, batch).astype(np.float32)
    for flags in (0, B.DN_NO_MASK, B.DN_IMPOSE_BC_ON_LOAD):
        po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
        Jo, _, _, ro = oracle.energy_grad(po, u, gJ=gJ.astype(np.float64))
        Jg, rg = run_gpu(pg, u, gJ=gJ)
        check(Jg, rg, Jo, ro, f"flags {flags}")
