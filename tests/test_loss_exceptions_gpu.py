"""Exceptions that pass through the native loss functions keep their type: what a saved-tensor hook raises, the early stop of
a non-reentrant checkpoint (an exception raised by such a hook), and running out of memory."""
import pytest
import torch
from torch.utils.checkpoint import checkpoint

from paper_2007_12792_b200 import binding as B
from paper_2007_12792_b200.autograd import burgers_loss, energy

pytestmark = pytest.mark.gpu


def losses(nx=32, ny=24, batch=2):
    g = torch.Generator(device="cuda"); g.manual_seed(0)
    p = B.Problem(dim=2, nx=nx, ny=ny, batch=batch, kl_modes=2, kl_w=torch.rand((batch, 2, 2), generator=g, device="cuda"), f_const=1.0)
    q = B.Burgers(nx=nx, nt=ny, batch=batch, c=torch.full((batch,), 3.5, device="cuda"))
    u = torch.randn(p.shape, generator=g, device="cuda")
    return u, [(energy, p, B.new_workspace(p)), (burgers_loss, q, B.new_burgers_workspace(q))]


class Stop(Exception):
    pass


def test_a_pack_hook_that_raises():
    u, fs = losses()
    def pack(_):
        raise Stop("pack")
    for loss, p, ws in fs:
        with torch.autograd.graph.saved_tensors_hooks(pack, lambda x: x), pytest.raises(Stop, match="pack"):
            loss(u.clone().requires_grad_(True), p, ws)


def test_an_unpack_hook_that_raises_and_one_that_moves():
    u, fs = losses()
    def unpack(_):
        raise Stop("unpack")
    for loss, p, ws in fs:
        with torch.autograd.graph.saved_tensors_hooks(lambda x: x, unpack):
            J = loss(u.clone().requires_grad_(True), p, ws)
        with pytest.raises(Stop, match="unpack"):
            J.sum().backward()
        x, y = u.clone().requires_grad_(True), u.clone().requires_grad_(True)
        with torch.autograd.graph.save_on_cpu():
            J = loss(x, p, ws)
        J.sum().backward()
        loss(y, p, ws).sum().backward()
        assert torch.equal(x.grad, y.grad)


@pytest.mark.parametrize("reentrant", [False, True])
def test_in_a_checkpoint(reentrant):
    u, fs = losses()
    for loss, p, ws in fs:
        x, y = u.clone().requires_grad_(True), u.clone().requires_grad_(True)
        checkpoint(lambda v: loss(torch.sin(v), p, ws), x, use_reentrant=reentrant).sum().backward()
        loss(torch.sin(y), p, ws).sum().backward()
        assert torch.equal(x.grad, y.grad)


def test_running_out_of_memory_is_reported_as_such():
    u, fs = losses(1024, 1024, 16)                       # 64 MiB: the residual needs as much again
    u.requires_grad_(True)
    torch.cuda.synchronize(); torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (16 << 20)) / total)
    held = []
    try:
        with pytest.raises(torch.OutOfMemoryError):      # until not even a hole in the allocator's blocks is left for it
            while True:
                held.append(torch.empty_like(u))
        for loss, p, ws in fs:
            with pytest.raises(torch.OutOfMemoryError):
                loss(u, p, ws)
    finally:
        del held
        torch.cuda.set_per_process_memory_fraction(1.0)
    for loss, p, ws in fs:                               # and the next call works
        assert torch.isfinite(loss(u, p, ws)).all()
