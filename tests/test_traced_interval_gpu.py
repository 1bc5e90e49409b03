"""dn_energy_grad_traced: r is complete where event_after is recorded, for every size (small 3D problems finish the energies in the launch
that adds the seams, which must then not stand behind the event); results bit for bit those of the plain call."""
import pytest
import torch

from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200 import inputs
from parity_util import dev, make_problems

pytestmark = pytest.mark.gpu


def kernels(call):
    """Names of the kernels that a call launches, in order."""
    from torch.profiler import ProfilerActivity, profile
    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    ev = [e for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA and "kernel" in e.name]
    return [e.name for e in sorted(ev, key=lambda e: e.time_range.start)]


@pytest.mark.parametrize("nx,ny,nz,batch,mode", [(64, 64, 64, 2, B.DN_NU_KL_GAUSS), (33, 40, 21, 3, B.DN_NU_KL_NODAL), (128, 20, 40, 1, B.DN_NU_NODAL),
                                                 (260, 260, 250, 1, B.DN_NU_KL_GAUSS), (256, 256, 257, 1, B.DN_NU_KL_GAUSS), (64, 64, 1, 2, B.DN_NU_KL_GAUSS)])
def test_seams_are_inside_the_interval(nx, ny, nz, batch, mode):
    inp = inputs.random_inputs(3 if nz > 1 else 2, nx, ny, nz, batch, 2, seed=nx, f_const=0.5)
    nu = inputs.random_positive_field(inp.u.shape, 5) if mode == B.DN_NU_NODAL else None
    _, p = make_problems(inp, mode, nu=nu)
    u, ws = dev(inp.u), B.new_workspace(p)
    J, J2 = torch.empty(batch, device="cuda"), torch.empty(batch, device="cuda")
    r, r2 = torch.empty_like(u), torch.empty_like(u)
    before, after = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    before.record(); after.record()                      # (creates them)
    names = kernels(lambda: B.dn_energy_grad_traced(p, u, None, J, r, ws, before, after))
    assert sum("finalize" in n for n in names) == 1 and "finalize" in names[-1], names      # behind the event: the energies alone
    assert not any("seam" in n for n in names[-1:])
    plain = kernels(lambda: B.dn_energy_grad(p, u, None, J2, r2, ws))
    assert len(plain) == B.dn_launches_per_call(p) or nx == 260, plain
    assert torch.equal(J, J2) and torch.equal(r, r2)
