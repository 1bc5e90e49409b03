"""dn_cg_solve on grids of two columns: every node lies on a Dirichlet face, so there is nothing to solve.  u takes the
boundary values, no iteration is made, the residual is 0, and not a byte outside u changes."""
import pytest
import torch

from paper_2007_12792_b200 import binding as B
from parity_util import guarded, guards_intact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,ny,nz,batch", [(2, 2, 1, 1), (2, 8, 1, 3), (2, 65, 1, 1), (2, 512, 1, 3), (2, 4000, 1, 2), (3, 2, 2, 1), (3, 40, 9, 3)])
@pytest.mark.parametrize("mode", [B.DN_NU_KL_GAUSS, B.DN_NU_NODAL])
def test_nothing_to_solve(dim, ny, nz, batch, mode):
    shape = (batch, nz, ny, 2) if dim == 3 else (batch, ny, 2)
    n = batch * nz * ny * 2
    g = torch.Generator(device="cuda"); g.manual_seed(ny)
    w = torch.rand((batch,) + (2,) * dim, generator=g, device="cuda")
    nu = torch.rand(shape, generator=g, device="cuda") + 0.5
    p = B.Problem(dim=dim, nx=2, ny=ny, nz=nz, batch=batch, nu_mode=mode, nu=nu, kl_modes=2, kl_w=w, f_const=1.0, bc_x0=0.75, bc_x1=-0.25)
    whole, bytes_ = guarded(4 * n)
    u = bytes_.view(torch.float32).view(shape)
    u.copy_(torch.randn(shape, generator=g, device="cuda"))
    wsn = B.dn_cg_workspace_bytes(p)
    ws_whole, ws = guarded(wsn)
    relres = torch.full((batch,), float("nan"), device="cuda"); its = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
    B.dn_cg_solve(p, u, 50, 1e-6, relres, its, ws)
    torch.cuda.synchronize()
    assert guards_intact(whole, 4 * n) and guards_intact(ws_whole, wsn)
    assert torch.all(u[..., 0] == 0.75) and torch.all(u[..., 1] == -0.25)
    assert torch.all(its == 0) and torch.all(relres == 0.0)
