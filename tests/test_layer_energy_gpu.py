"""The energy alone on aligned 3D rows of more than 64 nodes (by layers, eight nodes per lane): 16 and 32 lanes, full and with lanes
beyond the grid, one and many tiles and chunks, every diffusivity mode, both kinds of forcing, imposed faces, cells that are
no cubes; against the oracle (the repository's 1e-5 per sample: fp32 sums per layer, double from there).  And 2D rows cut into units of
16 lanes, energy and residual."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import check, dev, guarded, guards_intact, make_problems, run_gpu

pytestmark = pytest.mark.gpu
MODES = [B.DN_NU_KL_GAUSS, B.DN_NU_KL_NODAL, B.DN_NU_NODAL]
SIZES = [(72, 2, 2, 3, 1), (72, 9, 30, 2, 8), (120, 21, 5, 1, 2), (128, 5, 13, 2, 3), (136, 3, 9, 1, 6), (200, 18, 4, 2, 4), (256, 11, 12, 1, 3)]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("nx,ny,nz,batch,m", SIZES)
def test_energy_alone(nx, ny, nz, batch, m, mode):
    inp = inputs.random_inputs(3, nx, ny, nz, batch, m, seed=nx + 5 * ny + nz, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)                      # boundary values NOT satisfied
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    for f in (None, inputs.random_field(inp.u.shape, 9, scale=3.0)):
        for flags in (0, B.DN_IMPOSE_BC_ON_LOAD):
            po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
            n = B.dn_workspace_bytes(pg)
            whole, ws = guarded(n)
            ws.fill_(0xFF)
            J = torch.empty(batch, device="cuda")
            B.dn_energy(pg, dev(u), J, ws)
            torch.cuda.synchronize()
            assert guards_intact(whole, n)
            Jo = oracle.energy_grad(po, u, want_r=False)[0]
            assert np.all(np.abs(J.cpu().numpy().astype(np.float64) - Jo) <= 1e-5 * np.abs(Jo)), (J, Jo)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("faces", [(1000.0, 1001.0), (1.0, 1.0 + 2.0 ** -10), (1.0, 0.0)])
@pytest.mark.parametrize("nx,ny,nz,batch,m", [(72, 9, 30, 2, 8), (128, 5, 13, 2, 3), (136, 3, 9, 1, 6), (256, 11, 12, 1, 3)])
def test_energy_of_fields_on_a_level(nx, ny, nz, batch, m, faces, mode):
    """Fields that vary little about a large mean, along all axes: the energy takes differences of the values given, so it loses
    nothing to the level.  Bound: differences of neighbours are exact here; an element's terms pass some 12 roundings and are
    positive, as are the sums per layer: 16 * 2^-24 = 1e-6, and as much for the KL exponents (up to 8, one rounding of each).
    Differences of values that are interpolated first are off by about 2 (2^-24 level / difference)^2 / 3 > 3e-6."""
    inp = inputs.random_inputs(3, nx, ny, nz, batch, m, seed=nx + ny, f_const=0.0)
    z, y, x = np.meshgrid(*(np.linspace(0.0, 1.0, n) for n in (nz, ny, nx)), indexing="ij")
    u = np.broadcast_to(faces[0] + (faces[1] - faces[0]) * (x + 0.25 * (y + z)), inp.u.shape).astype(np.float32)
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    for flags in (0, B.DN_IMPOSE_BC_ON_LOAD):
        po, pg = make_problems(inp, mode, nu=nu, flags=flags, f_const=0.0, bc=faces)
        J = torch.empty(batch, device="cuda")
        B.dn_energy(pg, dev(u), J, B.new_workspace(pg))
        Jo = oracle.energy_grad(po, u, want_r=False)[0]
        err = np.abs(J.cpu().numpy().astype(np.float64) / Jo - 1.0)
        assert np.all(err <= 2e-6), err


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("nx,ny,batch", [(150, 110, 64), (260, 65, 63), (513, 33, 64), (512, 70, 30)])
def test_2d_units_of_16_lanes(nx, ny, batch, mode):
    inp = inputs.random_inputs(2, nx, ny, 1, batch, 3, seed=nx, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    gJ = np.linspace(-1.5, 2.0, batch).astype(np.float32)
    for f in (None, inputs.random_field(inp.u.shape, 9, scale=3.0)):
        for flags in (0, B.DN_NO_MASK | B.DN_IMPOSE_BC_ON_LOAD):
            po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
            Jo, _, _, ro = oracle.energy_grad(po, u, gJ=gJ.astype(np.float64))
            Jg, rg = run_gpu(pg, u, gJ=gJ)
            check(Jg, rg, Jo, ro, f"flags {flags} f {f is not None}")


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("nx,ny,batch", [(148, 100, 200), (260, 65, 63), (284, 100, 100), (150, 110, 128), (513, 33, 128)])
def test_2d_units_of_16_lanes_of_both_calls(nx, ny, batch, mode):
    """The sizes from which the units have 16 lanes (2^20 nodes, 2^21 on ragged rows), the energy alone too: it runs other instantiations
    (with constant forcing on aligned rows the tiled kernel takes some of these calls).  The repository's 1e-5."""
    inp = inputs.random_inputs(2, nx, ny, 1, batch, 3, seed=nx, f_const=0.6)
    u = inputs.random_field(inp.u.shape, 8)
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    for f in (None, inputs.random_field(inp.u.shape, 9, scale=3.0)):
        for flags in (0, B.DN_IMPOSE_BC_ON_LOAD):
            po, pg = make_problems(inp, mode, nu=nu, f=f, flags=flags, bc=(0.8, -0.3))
            Jo, _, _, ro = oracle.energy_grad(po, u)
            Jg, rg = run_gpu(pg, u)
            check(Jg, rg, Jo, ro, f"flags {flags} f {f is not None}")
            n = B.dn_workspace_bytes(pg)
            whole, ws = guarded(n)
            ws.fill_(0xFF)
            J = torch.empty(batch, device="cuda")
            B.dn_energy(pg, dev(u), J, ws)
            torch.cuda.synchronize()
            assert guards_intact(whole, n)
            assert np.all(np.abs(J.cpu().numpy().astype(np.float64) - Jo) <= 1e-5 * np.abs(Jo)), (J, Jo)
