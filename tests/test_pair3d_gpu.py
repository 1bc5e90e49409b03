"""GPU parity of the mirrored-pair 3D kernel on rows of any length against the fp64 oracle: 2 to 17 nodes (lanes that reach
the far face), one node short of a full unit, a full unit, the middle node that has no lane (2^k + 1 nodes), odd and even
rows in between, with one and many tiles and chunks, in every diffusivity mode, with every option, fused and energy only.

Tolerance: the repository's 1e-5 (J per sample, r against max |r|); fp32 sums of a node's 8 contributions are good to 1e-6."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import check, dev, guarded, guards_intact, make_problems, run_gpu

pytestmark = pytest.mark.gpu

MODES = [B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL]
SIZES = [(2, 2, 2, 1, 1), (3, 3, 2, 2, 8), (4, 5, 3, 1, 2), (7, 4, 9, 3, 3), (9, 9, 9, 2, 2), (15, 6, 5, 1, 4), (16, 7, 4, 5, 5), (17, 17, 17, 2, 3),
         (18, 5, 6, 2, 6), (31, 9, 4, 1, 7), (33, 20, 12, 2, 2), (34, 3, 7, 1, 3), (63, 8, 5, 2, 2), (65, 21, 9, 1, 3), (66, 5, 5, 1, 8), (127, 6, 4, 1, 2),
         (129, 13, 7, 1, 4), (130, 4, 5, 1, 3), (200, 11, 3, 1, 2), (255, 4, 3, 1, 5), (257, 7, 4, 1, 3), (24, 11, 70, 1, 2)]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("nx,ny,nz,batch,m", SIZES)
def test_any_row_length(nx, ny, nz, batch, m, mode):
    inp = inputs.random_inputs(3, nx, ny, nz, batch, m, seed=nx + 5 * ny + nz, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)                      # boundary values NOT satisfied
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    gJ = np.linspace(-1.5, 2.0, batch).astype(np.float32)
    for f in (None, inputs.random_field(inp.u.shape, 9, scale=3.0)):
        for flags in (0, B.DN_NO_MASK, B.DN_IMPOSE_BC_ON_LOAD):
            po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
            Jo, _, _, ro = oracle.energy_grad(po, u, gJ=gJ.astype(np.float64))
            Jg, rg = run_gpu(pg, u, gJ=gJ)
            check(Jg, rg, Jo, ro, f"flags {flags} f {f is not None}")
            if not (flags & B.DN_NO_MASK):
                assert np.all(rg[..., 0] == 0.0) and np.all(rg[..., -1] == 0.0)
            n = max(B.dn_workspace_bytes(pg), 256)
            whole, ws = guarded(n)
            J = torch.empty(batch, device="cuda")
            B.dn_energy(pg, dev(u), J, ws)
            torch.cuda.synchronize()
            assert guards_intact(whole, n)
            Jo1 = oracle.energy_grad(po, u, want_r=False)[0]
            assert np.all(np.abs(J.cpu().numpy().astype(np.float64) - Jo1) <= 1e-5 * np.abs(Jo1))


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("n", [32, 64, 128])
def test_unaligned_pointers(n, off):
    inp = inputs.random_inputs(3, n, 9, 6, 2, 3, seed=3, f_const=0.4)
    po, pg = make_problems(inp, B.DN_NU_KL_GAUSS)
    Jo, _, _, ro = oracle.energy_grad(po, inp.u)
    k = inp.u.size
    u = torch.zeros(k + 4, device="cuda")[off:off + k].view(pg.shape)
    u.copy_(dev(inp.u))
    r = torch.full((k + 4,), 7.0, device="cuda")
    J = torch.empty(2, device="cuda")
    B.dn_energy_grad(pg, u, None, J, r[off:off + k].view(pg.shape), B.new_workspace(pg))
    torch.cuda.synchronize()
    assert torch.all(r[:off] == 7.0) and torch.all(r[off + k:] == 7.0)
    check(J.cpu().numpy().astype(np.float64), r[off:off + k].view(pg.shape).cpu().numpy().astype(np.float64), Jo, ro, f"offset {off}")
