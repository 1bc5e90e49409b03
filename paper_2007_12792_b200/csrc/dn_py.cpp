// Native marshalling of the Python entry points that a training loop calls per step: reads the fields of a Problem / Burgers
// object and the tensors' pointers, checks what the ctypes binding checks, calls the C entry point on the current stream.
// A call it does not recognise as plain (wrong type, device or layout of a tensor, a stream given) answers None, and the
// ctypes binding takes it, with its errors.  Also the two losses as autograd functions.
//
// Why: marshalling through ctypes cost more than the launches of a small problem (64^2 x 8: 17.5 us per call, of which 7.5 us
// are the three launches), and the autograd function in Python 20 us more per direction.
#include <torch/extension.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include "dn.h"

namespace {

struct Names {
    PyObject *dim, *nx, *ny, *nz, *batch, *nu_mode, *nu, *kl_modes, *kl_w, *f_const, *f, *bc_x0, *bc_x1, *flags, *bc_x0_b, *bc_x1_b, *nt, *T, *lam, *c;
} N;

struct NotPlain {};                                     // thrown where the ctypes binding has to look

struct Attr {                                           // an attribute of a Python object, owned
    PyObject* o;
    Attr(PyObject* from, PyObject* name) : o(PyObject_GetAttr(from, name)) { if (!o) { PyErr_Clear(); throw NotPlain{}; } }
    ~Attr() { Py_DECREF(o); }
    Attr(const Attr&) = delete;
    int32_t i32() const {
        const long v = PyLong_AsLong(o);
        if (v == -1 && PyErr_Occurred()) { PyErr_Clear(); throw NotPlain{}; }
        if (v < INT32_MIN || v > INT32_MAX) throw NotPlain{};
        return (int32_t)v;
    }
    float f32() const {
        const double v = PyFloat_AsDouble(o);
        if (v == -1.0 && PyErr_Occurred()) { PyErr_Clear(); throw NotPlain{}; }
        return (float)v;
    }
};

float* floats(PyObject* o) {                            // a contiguous float32 CUDA tensor, or None
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) throw NotPlain{};
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.scalar_type() != at::kFloat || !t.is_cuda() || !t.is_contiguous()) throw NotPlain{};
    return static_cast<float*>(t.data_ptr());
}
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) throw NotPlain{};
    return THPVariable_Unpack(o);
}
const float* floats_of(PyObject* from, PyObject* name) { return floats(Attr(from, name).o); }      // the object keeps it alive

dn_problem problem_of(PyObject* o) {
    dn_problem p{};
    p.grid.dim = Attr(o, N.dim).i32(); p.grid.nx = Attr(o, N.nx).i32(); p.grid.ny = Attr(o, N.ny).i32();
    p.grid.nz = p.grid.dim == 3 ? Attr(o, N.nz).i32() : 1;
    p.batch = Attr(o, N.batch).i32(); p.nu_mode = Attr(o, N.nu_mode).i32(); p.kl_modes = Attr(o, N.kl_modes).i32();
    p.nu = floats_of(o, N.nu); p.kl_w = floats_of(o, N.kl_w); p.f = floats_of(o, N.f);
    p.f_const = Attr(o, N.f_const).f32(); p.bc_x0 = Attr(o, N.bc_x0).f32(); p.bc_x1 = Attr(o, N.bc_x1).f32();
    p.flags = (uint32_t)Attr(o, N.flags).i32();
    p.bc_x0_b = floats_of(o, N.bc_x0_b); p.bc_x1_b = floats_of(o, N.bc_x1_b);
    return p;
}
dn_burgers burgers_of(PyObject* o) {
    dn_burgers p{};
    p.nx = Attr(o, N.nx).i32(); p.nt = Attr(o, N.nt).i32(); p.batch = Attr(o, N.batch).i32();
    p.T = Attr(o, N.T).f32(); p.lambda = Attr(o, N.lam).f32(); p.flags = (uint32_t)Attr(o, N.flags).i32();
    p.c = floats_of(o, N.c);
    return p;
}
void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// C++ exceptions become Python ones by torch's own translation: an allocation that fails is a torch.OutOfMemoryError, what a
// Python callback (a saved-tensor hook) raised keeps its type and traceback.
template <class F>
PyObject* call(F f) {                                   // the status as an int, or None
    HANDLE_TH_ERRORS
    try {
        return PyLong_FromLong((long)f());
    } catch (const NotPlain&) {
        Py_RETURN_NONE;
    }
    END_HANDLE_TH_ERRORS
}
#define DN_NO_GIL(x) [&]() { dn_status s_; Py_BEGIN_ALLOW_THREADS s_ = (x); Py_END_ALLOW_THREADS return s_; }()
#define DN_ARGS(n) do { if (nargs != (n)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; } } while (0)

PyObject* energy_grad(PyObject*, PyObject* const* a, Py_ssize_t nargs) {       // problem, u, gJ, J, r, workspace
    DN_ARGS(6);
    return call([&]() {
        const dn_problem p = problem_of(a[0]);
        const float *u = floats(a[1]), *gJ = floats(a[2]);
        float *J = floats(a[3]), *r = floats(a[4]);
        const at::Tensor& ws = tensor(a[5]);
        void *w = ws.data_ptr(), *s = current_stream();
        const size_t n = (size_t)ws.numel();
        return DN_NO_GIL(dn_energy_grad(&p, u, gJ, J, r, w, n, s));
    });
}
PyObject* energy(PyObject*, PyObject* const* a, Py_ssize_t nargs) {            // problem, u, J, workspace
    DN_ARGS(4);
    return call([&]() {
        const dn_problem p = problem_of(a[0]);
        const float* u = floats(a[1]);
        float* J = floats(a[2]);
        const at::Tensor& ws = tensor(a[3]);
        void *w = ws.data_ptr(), *s = current_stream();
        const size_t n = (size_t)ws.numel();
        return DN_NO_GIL(dn_energy(&p, u, J, w, n, s));
    });
}
PyObject* burgers_loss_grad(PyObject*, PyObject* const* a, Py_ssize_t nargs) { // problem, u, gL, L, parts, g, workspace
    DN_ARGS(7);
    return call([&]() {
        const dn_burgers p = burgers_of(a[0]);
        const float *u = floats(a[1]), *gL = floats(a[2]);
        float *L = floats(a[3]), *parts = floats(a[4]), *g = floats(a[5]);
        const at::Tensor& ws = tensor(a[6]);
        void *w = ws.data_ptr(), *s = current_stream();
        const size_t n = (size_t)ws.numel();
        return DN_NO_GIL(dn_burgers_loss_grad(&p, u, gL, L, parts, g, w, n, s, nullptr, nullptr));
    });
}

// ---- the losses as autograd functions: forward computes the loss and its gradient in one pass, backward scales it -----
struct LossFn : torch::autograd::Function<LossFn> {
    // status: out; p, q: the statement of the problem, one of them null (only read during forward)
    static at::Tensor forward(torch::autograd::AutogradContext* ctx, const at::Tensor& u_in, int64_t batch, int64_t p, int64_t q, int64_t ws, int64_t ws_bytes,
                              int64_t status) {
        const at::Tensor u = u_in.contiguous();
        at::Tensor loss = at::empty({batch}, u.options()), g = at::empty_like(u);
        void* s = current_stream();
        dn_status* st = reinterpret_cast<dn_status*>(status);
        const float* up = static_cast<const float*>(u.data_ptr());
        float *lp = static_cast<float*>(loss.data_ptr()), *gp = static_cast<float*>(g.data_ptr());
        void* w = reinterpret_cast<void*>(ws);
        if (p) *st = dn_energy_grad(reinterpret_cast<const dn_problem*>(p), up, nullptr, lp, gp, w, (size_t)ws_bytes, s);
        else *st = dn_burgers_loss_grad(reinterpret_cast<const dn_burgers*>(q), up, nullptr, lp, nullptr, gp, w, (size_t)ws_bytes, s, nullptr, nullptr);
        ctx->save_for_backward({g});
        return loss;
    }
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, torch::autograd::variable_list grads) {
        const at::Tensor g = ctx->get_saved_variables()[0];
        std::vector<int64_t> shape((size_t)g.dim(), 1);
        shape[0] = -1;
        at::Tensor none;
        return {grads[0].reshape(shape).to(g.scalar_type()) * g, none, none, none, none, none, none};
    }
};

template <class P>
PyObject* loss(PyObject* const* a, const P& p, int64_t batch, bool fem) {      // u, problem, workspace
    const at::Tensor& u = tensor(a[0]);
    if (u.scalar_type() != at::kFloat || !u.is_cuda() || u.dim() < 1) throw NotPlain{};
    const at::Tensor& ws = tensor(a[2]);
    dn_status st = DN_OK;
    const int64_t pp = reinterpret_cast<int64_t>(&p);
    at::Tensor out;
    {
        pybind11::gil_scoped_release no_gil;
        out = LossFn::apply(u, batch, fem ? pp : (int64_t)0, fem ? (int64_t)0 : pp, reinterpret_cast<int64_t>(ws.data_ptr()), ws.numel(),
                            reinterpret_cast<int64_t>(&st));
    }
    if (st != DN_OK) return PyLong_FromLong((long)st);
    return THPVariable_Wrap(out);
}
template <class F>
PyObject* call_loss(F f) {                              // the loss, a status as an int, or None
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const NotPlain&) {
        Py_RETURN_NONE;
    }
    END_HANDLE_TH_ERRORS
}
PyObject* energy_loss(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    DN_ARGS(3);
    return call_loss([&]() { const dn_problem p = problem_of(a[1]); return loss(a, p, p.batch, true); });
}
PyObject* burgers_loss(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    DN_ARGS(3);
    return call_loss([&]() { const dn_burgers p = burgers_of(a[1]); return loss(a, p, p.batch, false); });
}

PyMethodDef methods[] = {
    {"energy_grad", (PyCFunction)(void (*)(void))energy_grad, METH_FASTCALL, nullptr},
    {"energy", (PyCFunction)(void (*)(void))energy, METH_FASTCALL, nullptr},
    {"burgers_loss_grad", (PyCFunction)(void (*)(void))burgers_loss_grad, METH_FASTCALL, nullptr},
    {"energy_loss", (PyCFunction)(void (*)(void))energy_loss, METH_FASTCALL, nullptr},
    {"burgers_loss", (PyCFunction)(void (*)(void))burgers_loss, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
#define DN_NAME(x) N.x = PyUnicode_InternFromString(#x);
    DN_NAME(dim) DN_NAME(nx) DN_NAME(ny) DN_NAME(nz) DN_NAME(batch) DN_NAME(nu_mode) DN_NAME(nu) DN_NAME(kl_modes) DN_NAME(kl_w) DN_NAME(f_const)
    DN_NAME(f) DN_NAME(bc_x0) DN_NAME(bc_x1) DN_NAME(flags) DN_NAME(bc_x0_b) DN_NAME(bc_x1_b) DN_NAME(nt) DN_NAME(T) DN_NAME(lam) DN_NAME(c)
#undef DN_NAME
    return PyModule_Create(&module);
}
