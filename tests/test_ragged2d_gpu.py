"""GPU parity of the 2D marching kernel on rows of any length and pointers of any alignment against the fp64 oracle: one
node short of a full unit, a full unit, one node left over (the Dirichlet column without a lane of its own), two left over,
strips that end anywhere, in every diffusivity mode, with every option, fused and energy only.

Tolerance: the repository's 1e-5 (J per sample, r against max |r|); fp32 sums of a node's 16 edge terms are good to 1e-6."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import check, dev, guarded, guards_intact, make_problems, run_gpu

pytestmark = pytest.mark.gpu

MODES = [B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL]
SIZES = [(2, 2, 1, 1), (3, 9, 2, 8), (31, 5, 3, 2), (33, 40, 2, 3), (34, 3, 5, 4), (63, 17, 2, 5), (65, 65, 3, 2), (66, 8, 1, 6),
         (127, 33, 2, 3), (129, 20, 2, 4), (130, 6, 2, 2), (253, 12, 1, 3), (257, 90, 2, 4), (513, 11, 2, 6), (1030, 7, 1, 7),
         (260, 9, 2, 3), (512, 40, 1, 4)]       # the last two: aligned rows in strips that the tiled kernel used to serve


def energy_only(pg, u):
    n = max(B.dn_workspace_bytes(pg), 256)
    whole, ws = guarded(n)
    J = torch.empty(pg.batch, device="cuda")
    B.dn_energy(pg, dev(u), J, ws)
    torch.cuda.synchronize()
    assert guards_intact(whole, n)
    return J.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("nx,ny,batch,m", SIZES)
def test_ragged_rows(nx, ny, batch, m, mode):
    inp = inputs.random_inputs(2, nx, ny, 1, batch, m, seed=nx + 5 * ny, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)                      # boundary values NOT satisfied
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    gJ = np.linspace(-1.5, 2.0, batch).astype(np.float32)
    for f in (None, inputs.random_field(inp.u.shape, 9, scale=3.0)):
        for flags in (0, B.DN_NO_MASK, B.DN_IMPOSE_BC_ON_LOAD, B.DN_IMPOSE_BC_ON_LOAD | B.DN_NO_MASK):
            po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
            Jo, _, _, ro = oracle.energy_grad(po, u, gJ=gJ.astype(np.float64))
            Jg, rg = run_gpu(pg, u, gJ=gJ)
            check(Jg, rg, Jo, ro, f"flags {flags} f {f is not None}")
            if not (flags & B.DN_NO_MASK):
                assert np.all(rg[..., 0] == 0.0) and np.all(rg[..., -1] == 0.0)
            J1 = energy_only(pg, u)
            Jo1 = oracle.energy_grad(po, u, want_r=False)[0]
            assert np.all(np.abs(J1 - Jo1) <= 1e-5 * np.abs(Jo1))


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(64, 30), (256, 19), (1024, 17)])
def test_unaligned_pointers_give_the_same_residual(nx, ny, off):
    """Fields that start at any float: the result is the one of the aligned call up to rounding."""
    inp = inputs.random_inputs(2, nx, ny, 1, 2, 3, seed=3, f_const=0.4)
    po, pg = make_problems(inp, B.DN_NU_KL_GAUSS)
    Jo, _, _, ro = oracle.energy_grad(po, inp.u)
    n = inp.u.size
    u = torch.zeros(n + 4, device="cuda")[off:off + n].view(pg.shape)
    u.copy_(dev(inp.u))
    r = torch.full((n + 4,), 7.0, device="cuda")
    J = torch.empty(2, device="cuda")
    B.dn_energy_grad(pg, u, None, J, r[off:off + n].view(pg.shape), B.new_workspace(pg))
    torch.cuda.synchronize()
    assert torch.all(r[:off] == 7.0) and torch.all(r[off + n:] == 7.0)
    check(J.cpu().numpy().astype(np.float64), r[off:off + n].view(pg.shape).cpu().numpy().astype(np.float64), Jo, ro, f"offset {off}")
