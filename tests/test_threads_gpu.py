"""Host threads that launch the same kernel for problems of different sizes at the same time, each on its own stream: every
call is accepted (the C entry points are called directly, so that the threads meet inside the library) and the last one
gives bit for bit what it gives alone."""
import ctypes as C
import threading

import pytest
import torch

from paper_2007_12792_b200 import binding as B

pytestmark = pytest.mark.gpu
CALLS = 2000


class Call:
    def __init__(self, entry, dim, nx, ny, nz, batch, m=2, mode=B.DN_NU_KL_GAUSS):
        g = torch.Generator(device="cuda"); g.manual_seed(nx + ny)
        shape = (batch, nz, ny, nx) if dim == 3 else (batch, ny, nx)
        self.p = B.Problem(dim=dim, nx=nx, ny=ny, nz=nz, batch=batch, nu_mode=mode, nu=0.5 + torch.rand(shape, generator=g, device="cuda"), kl_modes=m,
                           kl_w=torch.rand((batch,) + (m,) * dim, generator=g, device="cuda"), f_const=1.0)
        self.c = C.byref(self.p.c_struct())
        self.u = torch.rand(self.p.shape, generator=g, device="cuda")
        self.out = torch.zeros(batch if entry == "dn_energy" else self.p.shape, device="cuda")
        self.ws = B.new_cg_workspace(self.p) if entry == "dn_cg_solve" else B.new_workspace(self.p)
        self.f, self.entry = getattr(B.lib(), entry), entry
        torch.cuda.synchronize()

    def __call__(self, stream):
        u, out, ws, n = self.u.data_ptr(), self.out.data_ptr(), self.ws.data_ptr(), self.ws.numel()
        if self.entry == "dn_cg_solve":                   # no iterations: the launches only
            return self.f(self.c, out, 0, 0.0, None, None, ws, n, stream)
        if self.entry == "dn_energy":
            return self.f(self.c, u, out, ws, n, stream)
        return self.f(self.c, u, None, None, out, ws, n, stream)


# sizes that run the same kernel with different amounts of shared memory: slabs of 32 rows of 256 and of 250 nodes (2D solver),
# tiles of 8 and of 3 element rows (energy alone, residual)
ND = B.DN_NU_NODAL
PAIRS = [("dn_cg_solve", (2, 256, 249, 1, 1), (2, 250, 249, 1, 1)), ("dn_energy", (3, 256, 9, 9, 64, 1, ND), (3, 256, 4, 9, 150, 1, ND)),
         ("dn_energy_grad", (3, 256, 9, 9, 64, 1, ND), (3, 256, 4, 9, 150, 1, ND))]


@pytest.mark.parametrize("entry,a,b", PAIRS)
def test_two_sizes_in_several_threads(entry, a, b):
    calls = [Call(entry, *size) for size in (a, b) * 3]
    want = []
    for c in calls[:2]:
        assert c(torch.cuda.current_stream().cuda_stream) == B.DN_OK
        torch.cuda.synchronize()
        want.append(c.out.clone())
    streams, refused = [torch.cuda.Stream() for _ in calls], [0] * len(calls)
    torch.cuda.synchronize()

    def work(i):
        c, s, n = calls[i], streams[i].cuda_stream, 0
        for k in range(CALLS if entry != "dn_cg_solve" else CALLS // 4):
            n += c(s) != B.DN_OK
        refused[i] = n

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    [t.start() for t in ts]; [t.join() for t in ts]
    torch.cuda.synchronize()
    assert refused == [0] * len(calls)
    assert all(torch.equal(c.out, want[i % 2]) for i, c in enumerate(calls))
