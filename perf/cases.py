"""Performance cases: the work a user of the library has it do, through its Python entry points.

A case is one call (or one training step) of
  grad      dn_energy_grad with an upstream gradient: energy and residual of a batch of fields, the body of a training loop
  train     the same loss as a PyTorch op: forward, batch mean, gradient back to the field
  sampled   a fresh diffusivity field per step (dn_kl_field), then dn_energy_grad with that stored field
  energy    dn_energy: the loss alone, as a line search or a validation pass asks for it
  cg        dn_cg_solve: the discrete solution the generator is compared with
  burgers   dn_burgers_loss_grad: loss, its two parts and the gradient of the Burgers finite-difference loss
on grids of 32 to 2048 nodes per axis in 2D and 16 to 256 in 3D.  Grids come with 2^k nodes per axis (what a
convolutional generator puts out), with 2^k + 1 (2^k elements per side) and with any other number (refinement studies).
"""
import math

import torch

from paper_2007_12792_b200 import autograd
from paper_2007_12792_b200 import binding as B

MODES = {"kl": B.DN_NU_KL_GAUSS, "klnodal": B.DN_NU_KL_NODAL, "stored": B.DN_NU_NODAL}
MOST_NODES = 1 << 26          # nodes of the largest listed cases (2048^2 x 16, 256^3 x 4)
MOST_RAGGED = 1 << 24         # ... and of the largest listed ones whose rows are not a multiple of 4 (513^2 x 64, 129^3 x 8)
MOST_CG = 1 << 20             # 256^2 x 16


def _case(op, nx, ny, nz, batch, name=None, **kw):
    c = {"op": op, "dim": 3 if nz > 1 else 2, "nx": nx, "ny": ny, "nz": nz, "batch": batch, "nu": "kl", "m": 4, "f": 0.0,
         "nodal_f": False, "impose": False, "field": "sines"}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest training grid: a call is a few microseconds of work, so launches and host time are what it costs
        _case("grad", 64, 64, 1, 8, "grad2d_64_b8", m=2, field="noise"),
        # the ordinary training step of a 2D generator, as a PyTorch op
        _case("train", 256, 256, 1, 64, "train2d_256_b64", m=4, f=1.0, field="noise"),
        # the largest 2D grid
        _case("grad", 2048, 2048, 1, 16, "grad2d_2048_b16", m=6),
        # a diffusivity field drawn and stored per step
        _case("sampled", 1024, 1024, 1, 32, "sampled2d_1024_b32", nu="stored", m=4),
        # 512 elements per side: odd rows; boundary data drawn per sample and imposed on load
        _case("grad", 513, 513, 1, 64, "grad2d_513_b64", nu="klnodal", m=4, impose=True),
        # the ordinary 3D training grid
        _case("grad", 64, 64, 64, 32, "grad3d_64_b32", m=2, field="noise"),
        # the largest 3D grid
        _case("grad", 256, 256, 256, 4, "grad3d_256_b4", m=3, f=1.0),
        # 128 elements per side in 3D with a measured (stored) coefficient: odd rows
        _case("grad", 129, 129, 129, 8, "grad3d_129_b8", nu="stored"),
        # a validation pass in 3D: the loss alone, with a forcing field
        _case("energy", 128, 128, 128, 8, "energy3d_128_b8", m=3, nodal_f=True),
        # reference solutions for a mini-batch: the conventional solver
        _case("cg", 256, 256, 1, 16, "cg2d_256_b16", m=4, f=1.0),
        # Burgers loss on the high-resolution outputs, and on a small space-time mesh with 2^k cells per side
        _case("burgers", 1024, 1024, 1, 64, "burgers_1024_b64", nu="none", m=0, field="wave"),
        _case("burgers", 257, 129, 1, 16, "burgers_257x129_b16", nu="none", m=0, field="wave"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, lo, hi):
    """Nodes along an axis: half of them a multiple of 8, a quarter one more than that, a quarter whatever comes."""
    n = _log_uniform(rng, lo, hi)
    kind = rng.random()
    if kind < 0.75:
        n = max(lo, n // 8 * 8) + (1 if kind < 0.25 else 0)
    return min(n, hi + 1)


def draw(rng):
    op = rng.choices(("grad", "train", "sampled", "energy", "cg", "burgers"), (40, 15, 10, 10, 10, 15))[0]
    dim = 2 if op == "burgers" else rng.choice((2, 3))
    if op == "cg":
        lo, hi, most = (32, 256, MOST_CG) if dim == 2 else (16, 48, MOST_CG)
    else:
        lo, hi, most = (32, 2048, MOST_NODES) if dim == 2 else (16, 256, MOST_NODES)
    nx = _extent(rng, lo, hi)
    ny, nz = nx, (nx if dim == 3 else 1)
    if rng.random() < 0.4:                        # not a square or a cube
        ny = _extent(rng, lo, hi)
        nz = _extent(rng, lo, hi) if dim == 3 else 1
    if nx % 4:
        most = min(most, MOST_RAGGED)
    while nx * ny * nz > most:
        ny, nz = max(lo, ny // 2), (max(lo, nz // 2) if dim == 3 else 1)
    batch = _log_uniform(rng, 1, max(1, min(64, most // (nx * ny * nz))))
    if op == "burgers":
        return _case(op, nx, ny, 1, batch, nu="none", m=0, field="wave")
    if op == "cg":
        return _case(op, nx, ny, nz, batch, nu=rng.choice(("kl", "stored")), m=rng.randint(1, 6), f=1.0)
    return _case(op, nx, ny, nz, batch, nu="stored" if op == "sampled" else rng.choice(("kl", "kl", "klnodal", "stored")),
                 m=rng.randint(1, 8), f=rng.choice((0.0, 1.0)), nodal_f=rng.random() < 0.2, impose=rng.random() < 0.3,
                 field=rng.choice(("noise", "sines")))


def _axis(n):
    return torch.linspace(0.0, 1.0, n, device="cuda", dtype=torch.float32)


def _fields(case, gen):
    """Stand-ins for generator outputs: the linear profile between the Dirichlet faces plus noise (early training) or
    plus a smooth random field of 16 sines (late training)."""
    nx, ny, nz, batch = case["nx"], case["ny"], case["nz"], case["batch"]
    shape = (batch, nz, ny, nx) if case["dim"] == 3 else (batch, ny, nx)
    if case["field"] == "noise":
        u = torch.randn(shape, generator=gen, device="cuda").mul_(0.1).add_(1.0 - _axis(nx))
    else:
        k = torch.randint(0, 5, (batch, 16, 3), generator=gen, device="cuda").float() * (2.0 * math.pi)
        k[:, :, 0] += (k.sum(-1) == 0) * (2.0 * math.pi)
        phi = torch.rand((batch, 16, 1), generator=gen, device="cuda") * (2.0 * math.pi)
        # sin(theta_rows + theta_x) summed over the sines as one product of small matrices per sample
        ty = k[:, :, 1:2] * _axis(ny) + phi                                      # [B][16][ny]
        if case["dim"] == 3:
            ty = (k[:, :, 2:3, None] * _axis(nz)[:, None] + ty[:, :, None, :]).flatten(2)
        tx = k[:, :, 0:1] * _axis(nx)
        rows = torch.cat([ty.sin(), ty.cos()], 1).transpose(1, 2)                # [B][rows][32]
        u = torch.bmm(rows, torch.cat([tx.cos(), tx.sin()], 1)).mul_(0.1 / 4.0).view(shape)
        u += 1.0 - _axis(nx)
    u[..., 0] = 1.0
    u[..., -1] = 0.0
    return u


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nx, ny, nz, batch, dim, op = (case[k] for k in ("nx", "ny", "nz", "batch", "dim", "op"))
    if op == "burgers":
        c = 3.0 + 3.0 * torch.rand(batch, generator=gen, device="cuda")
        wave = 2.0 * math.pi * c[:, None, None] * (_axis(nx) - 0.1 * _axis(ny)[:, None])
        u = wave.cos_().mul_(-0.5).add_(0.5).add_(torch.randn(wave.shape, generator=gen, device="cuda"), alpha=0.01)
        p = B.Burgers(nx=nx, nt=ny, batch=batch, c=c, T=0.2, lam=1.0)
        return {"op": op, "p": p, "u": u, "gL": torch.full((batch,), 1.0 / batch, device="cuda"),
                "L": torch.empty(batch, device="cuda"), "parts": torch.empty(batch, 2, device="cuda"),
                "g": torch.empty_like(u), "ws": B.new_burgers_workspace(p)}
    r3 = math.sqrt(3.0)
    w = (2.0 * torch.rand((batch,) + (case["m"],) * dim, generator=gen, device="cuda") - 1.0) * r3
    u = _fields(case, gen)
    nu = None
    if case["nu"] == "stored":
        nu = B.dn_kl_field(dim, nx, ny, nz, batch, case["m"], w, torch.empty_like(u))
    f = torch.randn(u.shape, generator=gen, device="cuda") if case["nodal_f"] else None
    bc = {}
    if case["impose"]:
        bc = {"flags": B.DN_IMPOSE_BC_ON_LOAD, "bc_x0_b": 0.5 + torch.rand(batch, generator=gen, device="cuda"),
              "bc_x1_b": 0.5 * torch.rand(batch, generator=gen, device="cuda")}
    p = B.Problem(dim=dim, nx=nx, ny=ny, nz=nz, batch=batch, nu_mode=MODES[case["nu"]], nu=nu, kl_modes=case["m"], kl_w=w,
                  f_const=case["f"], f=f, **bc)
    s = {"op": op, "p": p, "u": u, "w": w}
    if op == "cg":
        s["guess"] = u
        s["u"] = torch.empty_like(u)
        s["iters"] = 60 + 7 * max(nx, ny, nz) // 2
        s["ws"] = B.new_cg_workspace(p)
        return s
    s["ws"] = B.new_workspace(p)
    s["J"] = torch.empty(batch, device="cuda")
    if op == "train":
        u.requires_grad_(True)
    elif op != "energy":
        s["gJ"] = torch.full((batch,), 1.0 / batch, device="cuda")
        s["r"] = torch.empty_like(u)
    return s


def run(s):
    p, op = s["p"], s["op"]
    if op == "burgers":
        return B.dn_burgers_loss_grad(p, s["u"], s["gL"], s["L"], s["parts"], s["g"], s["ws"])
    if op == "train":
        J = autograd.energy(s["u"], p, s["ws"])
        (g,) = torch.autograd.grad(J.mean(), s["u"])
        return J.detach(), g
    if op == "energy":
        return B.dn_energy(p, s["u"], s["J"], s["ws"])
    if op == "cg":
        s["u"].copy_(s["guess"])
        B.dn_cg_solve(p, s["u"], s["iters"], 1e-5, None, None, s["ws"])
        return s["u"]
    if op == "sampled":
        B.dn_kl_field(p.dim, p.nx, p.ny, p.nz, p.batch, p.kl_modes, s["w"], p.nu)
        J, r = B.dn_energy_grad(p, s["u"], s["gJ"], s["J"], s["r"], s["ws"])
        return J, r, p.nu
    return B.dn_energy_grad(p, s["u"], s["gJ"], s["J"], s["r"], s["ws"])


def work(case):
    """Bytes: every field that goes in read once, every field that comes out written once (a solver iteration: solution,
    residual and direction in and out).  Flops: a count of the arithmetic per element or node of the closed form."""
    nodes = case["nx"] * case["ny"] * case["nz"] * case["batch"]
    d3, m, op = case["dim"] == 3, case["m"], case["op"]
    if op == "burgers":
        return {"bytes": 8.0 * nodes, "flops": 40.0 * nodes}
    points = 8 if d3 else 4
    exponents = {"kl": points * (2 * m + 1), "klnodal": 2 * m + 1, "stored": 0}[case["nu"]]
    flops = (180.0 if d3 else 40.0) + exponents
    if op == "energy":
        flops = (110.0 if d3 else 25.0) + exponents
    if op == "cg":
        iters = 60 + 7 * max(case["nx"], case["ny"], case["nz"]) // 2
        return {"bytes": 24.0 * nodes * iters, "flops": (flops + 13.0) * nodes * iters}
    fields = 1 + (case["nu"] == "stored") + case["nodal_f"] + (op != "energy")
    if op == "sampled":
        flops += 2 * m + 1
    if op == "train":
        flops += 1
    return {"bytes": 4.0 * fields * nodes, "flops": flops * nodes}


def tolerance(case):
    """Four times the largest distance from 64-bit results seen over listed and drawn cases (sums and exponentials in 32
    bits).  The solver stops at 1e-5 of its first residual: four times what is then left to the converged solution, since two
    implementations may stop an iteration apart."""
    if case["op"] == "cg":
        return {"rel": 5e-5, "max": 3e-4}
    return {"rel": 2e-6, "max": 4e-5}
