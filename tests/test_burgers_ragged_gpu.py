"""The Burgers marching kernel on rows of any length and pointers of any alignment against the fp64 oracle: 3 columns, one
column short of, at and beyond a strip's 120, rows that leave 1 to 3 columns in the last lane, few and many rows.
Tolerance: the repository's 1e-5 (L and its parts per sample, g against max |g|), see the error analysis of the aligned kernel,
whose arithmetic this is."""
import numpy as np
import pytest
import torch

from oracle import burgers as ob
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs

pytestmark = pytest.mark.gpu
T32 = float(np.float32(0.2))


def check(u_dev, g_dev, inp, gL=None):
    p = B.Burgers(nx=inp.nx, nt=inp.nt, batch=inp.batch, c=torch.from_numpy(inp.c).cuda(), T=T32, lam=0.5)
    L = torch.empty(inp.batch, device="cuda"); parts = torch.empty(inp.batch, 2, device="cuda")
    gLd = None if gL is None else torch.from_numpy(gL).cuda()
    B.dn_burgers_loss_grad(p, u_dev, gLd, L, parts, g_dev, B.new_burgers_workspace(p))
    Lo, Lp, Lb, go = ob.loss_grad(inp.u, inp.c.astype(np.float64), T=T32, lam=0.5)
    if gL is not None:
        go = go * gL.astype(np.float64)[:, None, None]
    assert np.all(np.abs(L.cpu().numpy() - Lo) <= 1e-5 * np.abs(Lo))
    assert np.all(np.abs(parts.cpu().numpy() - np.stack([Lp, Lb], 1)) <= 1e-5 * np.abs(np.stack([Lp, Lb], 1)))
    assert np.abs(g_dev.cpu().numpy() - go).max() <= 1e-5 * np.abs(go).max()
    L2 = torch.empty_like(L)
    B.dn_burgers_loss_grad(p, u_dev, gLd, L2, None, None, B.new_burgers_workspace(p))      # the loss alone
    assert torch.equal(L, L2)


@pytest.mark.parametrize("nx,nt,batch", [(3, 3, 2), (5, 40, 2), (7, 9, 1), (117, 20, 2), (119, 33, 1), (121, 12, 3), (122, 300, 1), (123, 8, 2),
                                         (257, 129, 4), (361, 17, 1), (1001, 20, 2)])
def test_rows_of_any_length(nx, nt, batch):
    inp = inputs.burgers_inputs(nx, nt, batch)
    whole = torch.full((inp.u.size + 64,), 7.0, device="cuda")
    g = whole[32:32 + inp.u.size].view(inp.u.shape)
    check(torch.from_numpy(inp.u).cuda(), g, inp, gL=np.linspace(-1.5, 2.0, batch).astype(np.float32))
    assert torch.all(whole[:32] == 7.0) and torch.all(whole[32 + inp.u.size:] == 7.0)


@pytest.mark.parametrize("off", [1, 2, 3])
def test_any_alignment(off):
    inp = inputs.burgers_inputs(256, 50, 2)
    n = inp.u.size
    u = torch.zeros(n + 4, device="cuda")[off:off + n].view(inp.u.shape)
    u.copy_(torch.from_numpy(inp.u))
    check(u, torch.empty(n + 4, device="cuda")[off:off + n].view(inp.u.shape), inp)
