"""Burgers losses of problems that do not fill the GPU, which march in chunks of a few rows: from one chunk to many, chunks that are
left over, with and without gradient, loss or parts; against the oracle (1e-5, as the other tests of this loss).  Rows that are no
multiple of four march in chunks of four to seven rows from about 160 000 nodes (the last six sizes); smaller ones run a thread per
node.  Two calls agree bit for bit."""
import numpy as np
import pytest
import torch

from oracle import burgers as ob
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nt,batch", [(4, 3, 1), (32, 32, 5), (33, 40, 3), (45, 45, 7), (46, 45, 2), (64, 64, 8), (120, 8, 1), (124, 70, 16), (257, 129, 16),
                                         (256, 170, 9), (256, 171, 3), (480, 130, 2), (129, 200, 4),
                                         (49, 224, 19), (53, 144, 26), (119, 256, 6), (239, 200, 4), (709, 41, 7), (1001, 60, 4)])
def test_small_problems(nx, nt, batch):
    inp = inputs.burgers_inputs(nx, nt, batch)
    T = float(np.float32(0.2))
    p = B.Burgers(nx=nx, nt=nt, batch=batch, c=torch.from_numpy(inp.c).cuda(), T=T, lam=0.7)
    u = torch.from_numpy(inp.u).cuda()
    gL = np.linspace(-1.0, 2.0, batch).astype(np.float32)
    gl = torch.from_numpy(gL).cuda()
    Lo, po, lb, go = ob.loss_grad(inp.u, inp.c.astype(np.float64), T=T, lam=0.7, gL=gL.astype(np.float64))
    out = []
    for rep in range(2):
        ws = B.new_burgers_workspace(p)
        ws.fill_(0xFF)
        L, parts, g = torch.empty(batch, device="cuda"), torch.empty(batch, 2, device="cuda"), torch.full_like(u, float("nan"))
        B.dn_burgers_loss_grad(p, u, gl, L, parts, g, ws)
        out.append((L, parts, g))
    assert all(torch.equal(a, b) for a, b in zip(*out))
    L, parts, g = (t.cpu().numpy().astype(np.float64) for t in out[0])
    assert np.all(np.abs(L - Lo) <= 1e-5 * np.abs(Lo))
    assert np.abs(g - go).max() <= 1e-5 * np.abs(go).max()
    assert np.all(np.abs(parts[:, 0] + 0.7 * parts[:, 1] - Lo) <= 2e-5 * np.abs(Lo))
    only = torch.empty(batch, device="cuda")
    B.dn_burgers_loss_grad(p, u, None, only, None, None, B.new_burgers_workspace(p))       # the loss alone
    assert torch.allclose(only, out[0][0], rtol=1e-6, atol=0)
    alone = torch.empty_like(u)
    B.dn_burgers_loss_grad(p, u, gl, None, None, alone, B.new_burgers_workspace(p))        # the gradient alone
    assert (alone - out[0][2]).abs().max() <= 1e-6 * alone.abs().max()                       # (another compilation of the same march)
