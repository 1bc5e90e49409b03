"""The nodal KL field at the edges of its blocks: one node more and less than a strip of 1024 nodes, rows shorter than a
thread's four nodes, one line more and less than a block's 64, planes of two lines, rows of any length and alignment.

Tolerance: the exponent is at most log2(nu) ~ 10 in size and carries m + 1 fp32 roundings of its terms and of the cosine
(2^-24 each, m <= 8), so nu is good to 10 ln 2 * 9 * 2^-24 = 4e-6 relative; the repository's 1e-5 is asked for."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import dev

pytestmark = pytest.mark.gpu

SIZES = [(2, 2, 2, 1, 1, 1), (2, 3, 129, 1, 2, 8), (2, 4, 65, 1, 3, 4), (2, 1020, 8, 1, 1, 3), (2, 1023, 9, 1, 2, 5), (2, 1024, 64, 1, 2, 6),
         (2, 1025, 7, 1, 2, 2), (2, 1028, 63, 1, 1, 7), (2, 2050, 3, 1, 1, 4), (2, 8, 2000, 1, 90, 2),
         (3, 2, 2, 2, 2, 8), (3, 5, 64, 3, 2, 8), (3, 12, 65, 2, 1, 5), (3, 129, 2, 9, 2, 4), (3, 257, 3, 3, 1, 1), (3, 32, 33, 34, 2, 6)]


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("dim,nx,ny,nz,batch,m", SIZES)
def test_kl_field_edges(dim, nx, ny, nz, batch, m, off):
    rng = np.random.default_rng(m + nx)
    w = np.stack([inputs.draw_weights(rng, dim, m) for _ in range(batch)])
    ref = oracle.kl_field(dim, nx, ny, nz, batch, m, w)
    n = ref.size
    buf = torch.full((n + 8,), -1.0, device="cuda")
    out = buf[off:off + n].view((batch, nz, ny, nx) if dim == 3 else (batch, ny, nx))
    B.dn_kl_field(dim, nx, ny, nz, batch, m, dev(w), out)
    got = out.cpu().numpy().astype(np.float64)
    assert torch.all(buf[:off] == -1.0) and torch.all(buf[off + n:] == -1.0)
    assert np.abs(got / ref.reshape(got.shape) - 1).max() < 1e-5
