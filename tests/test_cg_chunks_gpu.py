"""Batches that the solver takes in several chunks of samples: full chunks and a shorter last one, each sample with its own
diffusivity.  The library's residual of the returned field (its parity with the oracle is tested elsewhere) has fallen as far as
the solver says, and the samples around the chunks' ends are the ones that a solve of those alone returns, to what is left of
the residual (1e-5 of the first one: 2e-4 of the field, the bound of the other solver tests)."""
import pytest
import torch

from paper_2007_12792_b200 import binding as B

pytestmark = pytest.mark.gpu


def problem(nx, ny, nu, w, mode, sel=slice(None)):
    w = w[sel].contiguous()
    return B.Problem(dim=2, nx=nx, ny=ny, batch=w.shape[0], nu_mode=mode, nu=None if nu is None else nu[sel].contiguous(), kl_modes=2, kl_w=w, f_const=1.0)


@pytest.mark.parametrize("mode", [B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL])
def test_chunks(mode):
    nx, ny, batch = 140, 131, 601                        # 11 M nodes: couplings and probes of all take 1060 MB
    g = torch.Generator(device="cuda"); g.manual_seed(0)
    w = (2 * torch.rand((batch, 2, 2), generator=g, device="cuda") - 1) * 1.7
    u0 = torch.rand((batch, ny, nx), generator=g, device="cuda")
    nu = 0.5 + torch.rand((batch, ny, nx), generator=g, device="cuda") if mode == B.DN_NU_NODAL else None
    p = problem(nx, ny, nu, w, mode)
    assert B.dn_cg_workspace_bytes(p) < 600 << 20
    u = u0.clone()
    relres = torch.empty(batch, device="cuda"); its = torch.empty(batch, dtype=torch.int32, device="cuda")
    B.dn_cg_solve(p, u, 2000, 1e-5, relres, its, B.new_cg_workspace(p))
    assert torch.all(relres <= 1e-5) and torch.all(its < 2000) and torch.all(its > 0)
    r, r0 = torch.empty_like(u), torch.empty_like(u)
    start = u0.clone(); start[..., 0] = 1.0; start[..., -1] = 0.0
    B.dn_energy_grad(p, u, None, None, r, B.new_workspace(p))
    B.dn_energy_grad(p, start, None, None, r0, B.new_workspace(p))
    assert torch.all(r.flatten(1).norm(dim=1) <= 3e-5 * r0.flatten(1).norm(dim=1))
    for lo in (0, 148, 199, 298, 399, 449, 597):
        sel = slice(lo, lo + 4)
        q = problem(nx, ny, nu, w, mode, sel)
        v = u0[sel].clone()
        B.dn_cg_solve(q, v, 2000, 1e-5, None, None, B.new_cg_workspace(q))
        assert (v - u[sel]).abs().max() <= 2e-4 * v.abs().max()
