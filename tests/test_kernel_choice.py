"""Which kernel a call runs, decided on the host from the shape, the mode, the forcing and the pointers' alignment (no GPU)."""
import ctypes as C

import pytest

from paper_2007_12792_b200 import binding as B

KG, KN, ND = B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL


@pytest.fixture(scope="module")
def name():
    from paper_2007_12792_b200 import build
    build.build()
    L = B.lib()

    def f(dim, nx, ny, nz=1, mode=KG, forcing=False, batch=4, m=3, flags=0, u=0x100000, r=0x200000):
        p = B.DnProblem()
        p.grid = B.DnGrid(dim, nx, ny, nz)
        p.batch = batch; p.nu_mode = mode; p.kl_modes = m; p.kl_w = 0x100000; p.flags = flags
        p.nu = 0x300000 if mode == ND else None
        p.f = 0x400000 if forcing else None
        return L.dn_kernel_name(C.byref(p), u, r).decode()
    return f


def test_2d(name):
    for mode in (KG, KN, ND):
        for forcing in (False, True):
            for nx in (2, 5, 64, 129, 256, 260, 513, 2048, 2052):
                assert name(2, nx, 40, mode=mode, forcing=forcing) == "march2d"
                assert name(2, nx, 40, mode=mode, forcing=forcing, u=0x100004) == "march2d"
                assert name(2, nx, 40, mode=mode, forcing=forcing, flags=B.DN_FORCE_GENERIC) == "generic"
        assert name(2, 513, 40, mode=mode, r=None) == "march2d" and name(2, 2052, 40, mode=mode, r=None) == "march2d"
    assert name(2, 1024, 1024, batch=32, r=None) == "tiled2d"            # energy alone, rows that fill the tiled kernel
    assert name(2, 1024, 1024, batch=32, r=None, u=0x100004) == "march2d" and name(2, 1024, 1024, batch=32, r=None, forcing=True) == "march2d"
    assert name(4, 8, 8) == "invalid"


def test_3d(name):
    for mode in (KG, KN, ND):
        for forcing in (False, True):
            kw = dict(mode=mode, forcing=forcing)
            assert name(3, 32, 32, 32, **kw) == "strip3d" and name(3, 33, 33, 33, **kw) == "pair3d" and name(3, 257, 20, 20, **kw) == "pair3d"
            assert name(3, 32, 32, 32, u=0x100004, **kw) == "pair3d" and name(3, 6, 9, 9, **kw) == "pair3d"
            assert name(3, 256, 64, 64, r=None, **kw) == "strip3d" and name(3, 129, 64, 64, r=None, **kw) == "pair3d"
            assert name(3, 258, 20, 20, **kw) == "generic"
    # the residual on aligned rows of more than 32 nodes: both sides of every line of the rule
    assert name(3, 64, 64, 64, batch=32, m=2) == "pair3d" and name(3, 64, 22, 23, batch=1) == "strip3d" and name(3, 64, 23, 23, batch=1) == "pair3d"
    assert name(3, 96, 18, 18, batch=1, mode=KN) == "strip3d" and name(3, 96, 9, 9, batch=1) == "pair3d"
    assert name(3, 128, 128, 128, mode=ND) == "strip3d" and name(3, 136, 64, 64, mode=ND) == "pair3d"
    assert name(3, 136, 64, 64, mode=ND, forcing=True) == "strip3d" and name(3, 136, 64, 64, mode=KN, forcing=True) == "pair3d"
    assert name(3, 100, 100, 100, batch=16, m=3) == "strip3d" and name(3, 100, 100, 100, batch=16, m=4) == "pair3d"
    assert name(3, 100, 100, 100, batch=2, m=4) == "strip3d" and name(3, 100, 100, 100, batch=16, mode=KN, m=8) == "strip3d"
    assert name(3, 128, 64, 64, batch=4, m=3, forcing=True) == "strip3d" and name(3, 128, 64, 65, batch=4, m=3, forcing=True) == "pair3d"
    assert name(3, 128, 64, 32, batch=1, m=4, forcing=True) == "strip3d" and name(3, 128, 64, 33, batch=1, m=4, forcing=True) == "pair3d"
    assert name(3, 64, 64, 64, batch=64, mode=KN, forcing=True) == "strip3d" and name(3, 72, 64, 64, batch=64, mode=KN, forcing=True) == "pair3d"
    assert name(3, 260, 16, 16) == "tiled3d" and name(3, 512, 16, 16, mode=ND) == "tiled3d" and name(3, 260, 16, 16, mode=KN) == "generic"


def test_launches_of_small_3d_calls():
    """Tables of a 3D call in one launch or two, at both sides of every line of the rule (3: tables, kernel, seams and energies)."""
    def launches(nx, ny, nz, batch, m, mode=KG):
        p = B.DnProblem()
        p.grid = B.DnGrid(3, nx, ny, nz)
        p.batch = batch; p.nu_mode = mode; p.kl_modes = m; p.kl_w = 0x100000
        p.nu = 0x300000 if mode == ND else None
        return B.lib().dn_launches_per_call(C.byref(p))
    assert launches(33, 33, 33, 187, 2) == 3 and launches(33, 33, 33, 188, 2) == 4        # blocks (m^2 - 1) = 18 000: 6000 blocks
    assert launches(17, 17, 17, 140, 3) == 3 and launches(17, 17, 17, 928, 3) == 4
    assert launches(32, 32, 4, 2048, 3) == 4 and launches(16, 16, 16, 2272, 3) == 4 and launches(32, 32, 32, 64, 3) == 3
    assert launches(128, 145, 145, 3, 8) == 4 and launches(64, 224, 53, 4, 8) == 4 and launches(64, 64, 64, 1, 8) == 3
    assert launches(16, 16, 16, 4096, 1) == 3                                              # one mode: always
    assert launches(64, 64, 64, 8, 4, KN) == 3 and launches(64, 64, 64, 9, 4, KN) == 4
    assert launches(128, 128, 128, 7, 2, KN) == 3 and launches(128, 128, 128, 8, 2, KN) == 4
    assert launches(64, 64, 64, 1, 8, ND) == 2
    assert launches(256, 256, 256, 2, 2) == 5
