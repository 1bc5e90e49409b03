"""The multigrid-preconditioned solver at the sizes where its levels can go wrong: one block and several, a grid that is its own
last level, axes of 2 and 3 nodes, even and odd extents, axes halved one after the other (stretched cells), one level shared
by all blocks and three, couplings of level 0 in shared memory and not; smooth and jumping coefficients.

Checked by the oracle's own residual of the returned field, which is |r| <= 1e-5 |r0| by the recurrence plus |K| |u| 2^-24 from
storing the field in fp32: 3e-5 |r0|, the bound of the other solver tests.  The iterations tell that the cycle preconditions:
the diagonal alone takes 60 and more on all but the smallest of these grids.  The scratch starts as NaN."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import dev, guarded, guards_intact

pytestmark = pytest.mark.gpu

GRIDS = [(2, 3, 2, 1, 2), (2, 3, 300, 1, 2), (2, 300, 2, 1, 3), (2, 24, 21, 1, 5), (2, 33, 33, 1, 3), (2, 41, 40, 1, 20), (2, 64, 63, 1, 2),
         (2, 104, 104, 1, 1), (2, 256, 32, 1, 9), (2, 32, 256, 1, 2), (2, 129, 130, 1, 30), (2, 257, 255, 1, 1), (2, 380, 380, 1, 1),
         (3, 3, 3, 3, 2), (3, 3, 2, 40, 2), (3, 8, 8, 8, 3), (3, 16, 16, 16, 5), (3, 17, 16, 18, 40), (3, 48, 16, 17, 2), (3, 16, 49, 33, 2),
         (3, 49, 49, 49, 1), (3, 31, 2, 31, 1),
         # the largest samples that are solved this way, and thin slabs, which need more than eight blocks
         (2, 512, 512, 1, 1), (2, 511, 511, 1, 2), (3, 63, 63, 63, 1), (3, 64, 64, 64, 1), (3, 100, 100, 8, 2), (3, 56, 192, 8, 1), (3, 96, 96, 24, 1)]


@pytest.mark.parametrize("mode", ["kl", "klnodal", "jump"])
@pytest.mark.parametrize("dim,nx,ny,nz,batch", GRIDS)
def test_solution_and_iterations(dim, nx, ny, nz, batch, mode):
    inp = inputs.random_inputs(dim, nx, ny, nz, batch, 3, seed=nx + ny + nz, sigma=1.0, f_const=1.5)
    bc = (0.75, -0.25)
    nu = None
    if mode == "jump":                                   # by up to 1e4 from one patch of 8 nodes per axis to the next
        rng = np.random.default_rng(nx)
        shape = inp.u.shape
        nu = 10.0 ** rng.integers(-2, 3, (batch,) + tuple((n + 7) // 8 for n in shape[1:]))
        for a in range(1, len(shape)):
            nu = nu.repeat(8, axis=a)
        nu = nu[tuple(slice(0, n) for n in shape)].astype(np.float32)
    gm, om = {"kl": (B.DN_NU_KL_GAUSS, oracle.NU_KL_GAUSS), "klnodal": (B.DN_NU_KL_NODAL, oracle.NU_KL_NODAL),
              "jump": (B.DN_NU_NODAL, oracle.NU_NODAL)}[mode]
    p = B.Problem(dim=dim, nx=nx, ny=ny, nz=nz, batch=batch, nu_mode=gm, nu=dev(nu), kl_modes=3, kl_w=dev(inp.kl_w), f_const=1.5,
                  bc_x0=bc[0], bc_x1=bc[1])
    u = dev(inp.u).clone()
    relres = torch.empty(batch, device="cuda"); its = torch.empty(batch, dtype=torch.int32, device="cuda")
    n = B.dn_cg_workspace_bytes(p)
    whole, ws = guarded(n)
    ws.fill_(0xFF)
    B.dn_cg_solve(p, u, 400, 1e-5, relres, its, ws)
    torch.cuda.synchronize()
    assert guards_intact(whole, n)
    assert torch.all(relres <= 1e-5) and torch.all(its > 0) and torch.all(its <= (100 if mode == "jump" else 14)), (relres, its)
    po = oracle.Problem(dim=dim, nx=nx, ny=ny, nz=nz, batch=batch, nu_mode=om, nu=nu, kl_modes=3, kl_w=inp.kl_w, f_const=1.5,
                        bc_x0=bc[0], bc_x1=bc[1])
    u0 = inp.u.copy(); u0[..., 0] = bc[0]; u0[..., -1] = bc[1]
    norm = lambda a: np.linalg.norm(oracle.energy_grad(po, a)[3].reshape(batch, -1), axis=1)
    assert np.all(norm(u.cpu().numpy()) <= 3e-5 * norm(u0)), norm(u.cpu().numpy()) / norm(u0)
    assert torch.all(u[..., 0] == bc[0]) and torch.all(u[..., -1] == bc[1])


@pytest.mark.parametrize("dim,nx,ny,nz,batch", [(2, 104, 90, 1, 3), (2, 33, 33, 1, 5), (3, 17, 16, 18, 4), (3, 100, 100, 8, 2)])
def test_captured_in_a_graph(dim, nx, ny, nz, batch):
    """Replays give bit for bit what the call gives, also on another field than the one captured."""
    inp = inputs.random_inputs(dim, nx, ny, nz, batch, 3, seed=7, sigma=1.0, f_const=1.5)
    p = B.Problem(dim=dim, nx=nx, ny=ny, nz=nz, batch=batch, nu_mode=B.DN_NU_KL_GAUSS, kl_modes=3, kl_w=dev(inp.kl_w), f_const=1.5)
    starts = [dev(inp.u), dev(inp.u).flip(0).contiguous()]
    eager = []
    ws = B.new_cg_workspace(p)
    for s in starts:
        u = s.clone()
        B.dn_cg_solve(p, u, 50, 1e-5, None, None, ws)
        eager.append(u)
    u = starts[0].clone()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        B.dn_cg_solve(p, u, 50, 1e-5, None, None, ws)
    for s, e in zip(starts, eager):
        u.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(u, e)
