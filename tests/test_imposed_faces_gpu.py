"""DN_IMPOSE_BC_ON_LOAD reads u as if its faces held the boundary values: what stands there in memory has no influence, not
even where a kernel's lanes reach beyond a row's end and drop what they compute.  Fields whose faces hold NaN or infinity give
bit for bit what a field with zeros there gives.  Rows of 2 to 18 nodes (every row that the lanes of a unit overhang), and
one node more and less than whole units."""
import pytest
import torch

from paper_2007_12792_b200 import binding as B

pytestmark = pytest.mark.gpu

NX = {2: [2, 3, 4, 5, 8, 12, 31, 32, 33, 34, 65, 129, 256, 257, 260, 1025], 3: list(range(2, 19)) + [20, 24, 33, 34, 36, 65, 66, 129, 136, 257, 260]}


@pytest.mark.parametrize("mode", [B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL])
@pytest.mark.parametrize("dim,nx", [(d, n) for d in NX for n in NX[d]])
def test_imposed_faces_are_not_read(dim, nx, mode):
    ny, nz, batch, m = 19, (5 if dim == 3 else 1), 2, 3
    shape = (batch, nz, ny, nx) if dim == 3 else (batch, ny, nx)
    g = torch.Generator(device="cuda"); g.manual_seed(nx)
    w = torch.rand((batch,) + (m,) * dim, generator=g, device="cuda") - 0.5
    u = torch.randn(shape, generator=g, device="cuda")
    nu = torch.rand(shape, generator=g, device="cuda") + 0.5
    fld = torch.randn(shape, generator=g, device="cuda")
    b0, b1 = torch.tensor([0.7, -0.4], device="cuda"), torch.tensor([-0.2, 1.5], device="cuda")
    for f in (None, fld):
        for flags in (B.DN_IMPOSE_BC_ON_LOAD, B.DN_IMPOSE_BC_ON_LOAD | B.DN_NO_MASK):
            p = B.Problem(dim=dim, nx=nx, ny=ny, nz=nz, batch=batch, nu_mode=mode, nu=nu, kl_modes=m, kl_w=w, f_const=0.3, f=f,
                          flags=flags, bc_x0_b=b0, bc_x1_b=b1)
            out = []
            for v in (0.0, float("nan"), float("inf")):
                u[..., 0] = v; u[..., -1] = v
                ws = B.new_workspace(p)
                J, J1, r = torch.empty(batch, device="cuda"), torch.empty(batch, device="cuda"), torch.zeros_like(u)
                B.dn_energy_grad(p, u, None, J, r, ws)
                B.dn_energy(p, u, J1, ws)
                out.append((J, J1, r))
            assert all(torch.isfinite(t).all() for t in out[0])
            for k in (1, 2):
                assert all(torch.equal(a, b) for a, b in zip(out[0], out[k])), f"f {f is not None} flags {flags}"
