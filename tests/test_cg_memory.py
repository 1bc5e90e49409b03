"""Scratch of dn_cg_solve (host arithmetic, no GPU): never less than the launches per iteration need, which every solve can
fall back on, and for solves in one launch bounded by that or by 512 MiB and a sample's share, however large the batch."""
import ctypes as C

import pytest

from paper_2007_12792_b200 import binding as B


@pytest.fixture(scope="module")
def L():
    from paper_2007_12792_b200 import build
    build.build()
    return B.lib()


def prob(dim, nx, ny, nz, batch, mode, m):
    p = B.DnProblem()
    p.grid = B.DnGrid(dim, nx, ny, nz)
    p.batch = batch; p.nu_mode = mode; p.kl_modes = m; p.kl_w = 0x100000
    p.nu = 0x100000 if mode == B.DN_NU_NODAL else None
    return p


@pytest.mark.parametrize("mode,m", [(B.DN_NU_KL_GAUSS, 8), (B.DN_NU_KL_NODAL, 3), (B.DN_NU_NODAL, 1)])
@pytest.mark.parametrize("dim,nx,ny,nz", [(2, 3, 3, 1), (2, 64, 64, 1), (2, 256, 256, 1), (2, 257, 257, 1), (2, 514, 60, 1), (2, 20, 4000, 1),
                                          (3, 3, 3, 3), (3, 16, 16, 16), (3, 48, 48, 48), (3, 49, 49, 49)])
def test_workspace_is_bounded(L, dim, nx, ny, nz, mode, m):
    nodes = nx * ny * nz
    for batch in (1, 2, 3, 16, 17, 100, 512, 4096, 7281, 7282):
        if batch * nodes > 1 << 31:
            continue
        p = prob(dim, nx, ny, nz, batch, mode, m)
        ws = L.dn_workspace_bytes(C.byref(p))
        least = 4 * 4 * batch * nodes + 2 * ws
        small = 64 * batch + 16 * batch * (nodes // 4096 + 1) + 4096          # scalars, partial sums, rounding
        got = L.dn_cg_workspace_bytes(C.byref(p))
        assert least <= got
        sample = 4 * 33 * nodes + L.dn_workspace_bytes(C.byref(prob(dim, nx, ny, nz, 9, mode, m)))
        assert got <= max(least + small, 512 << 20) + ws + sample, (batch, got, least)
