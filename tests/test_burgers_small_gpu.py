"""Small Burgers grids of any row length on both sides of the line between the one-thread-per-node kernel and the marching
one: each agrees with the oracle (the repository's 1e-5).  First sizes just below and above the line and narrow rows, then, all
above it, rows that leave 1 to 3 columns in the marching kernel's last lane, one column short of, at and beyond a strip's 120,
few rows; aligned and unaligned pointers."""
import numpy as np
import pytest
import torch

from oracle import burgers as ob
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs

pytestmark = pytest.mark.gpu
T32 = float(np.float32(0.2))


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("nx,nt,batch", [(3, 1000, 8), (5, 40, 60), (9, 9, 1), (17, 65, 64), (17, 129, 120), (129, 40, 4), (129, 301, 4), (129, 361, 5), (257, 129, 5),
                                         (257, 129, 6), (1025, 33, 5), (64, 64, 2),
                                         (119, 40, 60), (121, 40, 60), (122, 64, 40), (123, 12, 200), (361, 17, 40), (1001, 20, 12), (63, 40, 120), (33, 129, 100),
                                         (17, 129, 300), (13, 200, 400), (602, 3, 200)])
def test_both_kernels(nx, nt, batch, off):
    inp = inputs.burgers_inputs(nx, nt, batch)
    n = inp.u.size
    u = torch.zeros(n + 4, device="cuda")[off:off + n].view(inp.u.shape)
    u.copy_(torch.from_numpy(inp.u))
    Lo, Lp, Lb, go = ob.loss_grad(inp.u, inp.c.astype(np.float64), T=T32, lam=0.5)
    for flags in (0, B.DN_FORCE_GENERIC):
        p = B.Burgers(nx=nx, nt=nt, batch=batch, c=torch.from_numpy(inp.c).cuda(), T=T32, lam=0.5, flags=flags)
        whole = torch.full((n + 68,), 7.0, device="cuda")
        g = whole[32 + off:32 + off + n].view(inp.u.shape)
        L = torch.empty(batch, device="cuda"); parts = torch.empty(batch, 2, device="cuda")
        B.dn_burgers_loss_grad(p, u, None, L, parts, g, B.new_burgers_workspace(p))
        assert np.all(np.abs(L.cpu().numpy() - Lo) <= 1e-5 * np.abs(Lo))
        assert np.all(np.abs(parts.cpu().numpy() - np.stack([Lp, Lb], 1)) <= 1e-5 * np.abs(np.stack([Lp, Lb], 1)))
        assert np.abs(g.cpu().numpy() - go).max() <= 1e-5 * np.abs(go).max()
        assert torch.all(whole[:32 + off] == 7.0) and torch.all(whole[32 + off + n:] == 7.0)
