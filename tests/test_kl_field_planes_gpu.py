"""The nodal KL field of many small 3D grids, whose blocks take several whole planes: planes of 2 to 64 lines, plane counts that
the blocks divide or not, rows shorter and longer than a thread's four nodes, every alignment; one line more (65) and one
block fewer, where a block keeps to one plane.  Tolerance: that of the other tests of this field (1e-5, of which fp32 uses 4e-6)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import dev

pytestmark = pytest.mark.gpu

SIZES = [(2, 2, 20, 512, 1), (5, 3, 17, 300, 2), (8, 8, 8, 600, 4), (17, 33, 5, 500, 3), (4, 64, 9, 300, 8), (33, 32, 40, 60, 6), (3, 2, 2000, 3, 5),
         (4, 65, 9, 300, 2), (8, 7, 37, 64, 7), (8, 7, 36, 65, 1), (130, 5, 60, 50, 4)]


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("nx,ny,nz,batch,m", SIZES)
def test_planes(nx, ny, nz, batch, m, off):
    rng = np.random.default_rng(m + nx)
    w = np.stack([inputs.draw_weights(rng, 3, m) for _ in range(batch)])
    n = batch * nz * ny * nx
    buf = torch.full((n + 8,), -1.0, device="cuda")
    out = buf[off:off + n].view(batch, nz, ny, nx)
    B.dn_kl_field(3, nx, ny, nz, batch, m, dev(w), out)
    assert torch.all(buf[:off] == -1.0) and torch.all(buf[off + n:] == -1.0)
    got = out.cpu().numpy().astype(np.float64)
    pick = sorted({0, 1, batch // 2, batch - 1})
    ref = oracle.kl_field(3, nx, ny, nz, len(pick), m, w[pick])
    assert np.abs(got[pick] / ref.reshape(len(pick), nz, ny, nx) - 1).max() < 1e-5
    assert np.isfinite(got).all() and (got > 0).all()
