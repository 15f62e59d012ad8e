// The per-call path from PyTorch tensors to libfmm (include/fmm.h), as a
// CPython extension module.
//
// What bounds a call on a small matrix is the host: checking five tensors,
// allocating the output, finding the stream and passing pointers took 12 us a
// call in Python beside 4 us for the launch, and a training step of five
// launches 230 us, most of it in Python on two threads that hand the
// interpreter lock to each other.  Here the same checks are a few loads, and
// the adjoint runs on the autograd thread without the interpreter: FusedMM
// 12 -> under 4 us of host time a call, the training step 229 -> 130 us, of which
// autograd's own hand-over between threads is about 75.
//
// Only the ordinary case is taken: plain tensors on the plan's device with the
// right dtype, shape and layout, outside of torch function and dispatch modes,
// function transforms, forward-mode differentiation and tracing.  Everything
// else returns NotImplemented, and the caller (fmm.py, autograd.py) takes its
// own path, which also raises the errors of wrong arguments.
#include <Python.h>

#include <memory>
#include <optional>

#include <ATen/Functions.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/jit/frontend/tracer.h>
#include <torch/version.h>

#include "fmm.h"

namespace {

using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::tensor_list;

constexpr int64_t kTypedMaxR = 512;   // widest bfloat16 rows of the typed adjoints

// A plan as the calls see it; handle is NULL once the plan is closed.
struct Plan {
    const fmm_plan *handle;
    int64_t m, n, r, nnz;
    at::ScalarType dtype;
    at::Device device;
};
using PlanPtr = std::shared_ptr<Plan>;

PyObject *g_check = nullptr;   // fmm._check(status, where): raises FmmError
const char *const kPlanName = "fmm plan";

// The plan of a capsule, or NULL (no capsule: a closed plan).
const PlanPtr *plan_of(PyObject *o)
{
    if (!PyCapsule_IsValid(o, kPlanName))
        return nullptr;
    return static_cast<const PlanPtr *>(PyCapsule_GetPointer(o, kPlanName));
}

// Whether no mode or transform wants to see the call.
bool plain_mode()
{
    return !at::impl::torch_function_mode_enabled() &&
           !c10::impl::TorchDispatchModeTLS::any_modes_set() &&
           !c10::impl::tls_is_dispatch_key_included(
               c10::DispatchKey::FuncTorchDynamicLayerFrontMode) &&
           !torch::jit::tracer::isTracing();
}

// A plain contiguous CUDA tensor of the given dtype on the given device.
bool plain(const Tensor &t, at::ScalarType dtype, at::Device device)
{
    return t.defined() && t.layout() == at::kStrided && t.has_storage() && t.is_cuda() &&
           t.device() == device && t.scalar_type() == dtype && t.is_contiguous();
}

const Tensor *tensor_of(PyObject *o)
{
    return THPVariable_CheckExact(o) ? &THPVariable_Unpack(o) : nullptr;
}

bool is_rows(const Tensor &t, int64_t rows, int64_t r)
{
    return t.dim() == 2 && t.size(0) == rows && t.size(1) == r;
}

bool is_list(const Tensor &t, int64_t n) { return t.dim() == 1 && t.size(0) == n; }

// The pointer the C interface expects: NULL for a tensor without elements.
template <typename P = void>
P *pointer(const Tensor &t)
{
    return t.defined() && t.numel() > 0 ? static_cast<P *>(t.data_ptr()) : nullptr;
}

Tensor empty(at::IntArrayRef shape, at::ScalarType dtype, at::Device device)
{
    return at::empty(shape, at::TensorOptions().dtype(dtype).device(device));
}

fmm_stream stream()
{
    return reinterpret_cast<fmm_stream>(c10::cuda::getCurrentCUDAStream().stream());
}

// Raises FmmError for a status in the calling thread (which holds the lock).
PyObject *raise_status(int status, const char *where)
{
    PyObject *r = PyObject_CallFunction(g_check, "is", status, where);
    Py_XDECREF(r);
    if (!PyErr_Occurred())
        PyErr_Format(PyExc_RuntimeError, "%s: status %d", where, status);
    return nullptr;
}

PyObject *not_implemented()
{
    Py_INCREF(Py_NotImplemented);
    return Py_NotImplemented;
}

struct Released {   // the interpreter lock, given up for a scope
    PyThreadState *s = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(s); }
};

// ------------------------------------------------------- calls on a plan
//
// args: plan, operands, out (None: allocated).  An operand kind per letter:
// v = float32, one per nonzero, or None; x = the same, not None; A, B = dense
// rows of S, of its columns; the output kind: V = one per nonzero, M, N = rows
// of S, of its columns (float32).
struct PlanCall {
    const char *name, *operands;
    char out;
    int (*fn4)(const fmm_plan *, const float *, const void *, const void *, float *, fmm_stream);
    int (*fn3)(const fmm_plan *, const float *, const void *, float *, fmm_stream);
};

const PlanCall kCalls[] = {
    {"fmm_sddmm", "vAB", 'V', fmm_sddmm, nullptr},
    {"fmm_spmm", "xB", 'M', nullptr, fmm_spmm},
    {"fmm_spmm_t", "xA", 'N', nullptr, fmm_spmm_t},
    {"fmm_fusedmm", "vAB", 'M', fmm_fusedmm, nullptr},
    {"fmm_fusedmm_t", "vAB", 'N', fmm_fusedmm_t, nullptr},
};

bool operand(char kind, const Tensor &t, const Plan &p)
{
    switch (kind) {
    case 'v': case 'x': case 'V': return plain(t, at::kFloat, p.device) && is_list(t, p.nnz);
    case 'A': return plain(t, p.dtype, p.device) && is_rows(t, p.m, p.r);
    case 'B': return plain(t, p.dtype, p.device) && is_rows(t, p.n, p.r);
    case 'M': return plain(t, at::kFloat, p.device) && is_rows(t, p.m, p.r);
    default: return plain(t, at::kFloat, p.device) && is_rows(t, p.n, p.r);
    }
}

bool operand(char kind, PyObject *o, const Plan &p, Tensor &t)
{
    if (o == Py_None)
        return kind == 'v';
    const Tensor *q = tensor_of(o);
    if (!q)
        return false;
    t = *q;
    return operand(kind, t, p);
}

PyObject *plan_call(const PlanCall &c, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const int k = c.fn4 ? 3 : 2;
    const PlanPtr *pp = n == k + 2 ? plan_of(args[0]) : nullptr;
    if (!pp || !plain_mode())
        return not_implemented();
    const Plan &p = **pp;
    Tensor t[3], out;
    for (int i = 0; i < k; ++i)
        if (!operand(c.operands[i], args[1 + i], p, t[i]))
            return not_implemented();
    PyObject *given = args[1 + k];
    if (given != Py_None && !operand(c.out, given, p, out))
        return not_implemented();
    int rc;
    {
        Released unlocked;
        if (!out.defined())
            out = c.out == 'V' ? empty({p.nnz}, at::kFloat, p.device)
                               : empty({c.out == 'M' ? p.m : p.n, p.r}, at::kFloat, p.device);
        rc = c.fn4 ? c.fn4(p.handle, pointer<float>(t[0]), pointer(t[1]), pointer(t[2]),
                           pointer<float>(out), stream())
                   : c.fn3(p.handle, pointer<float>(t[0]), pointer(t[1]), pointer<float>(out),
                           stream());
    }
    if (rc != FMM_OK)
        return raise_status(rc, c.name);
    if (given != Py_None) {
        Py_INCREF(given);
        return given;
    }
    return THPVariable_Wrap(out);
    END_HANDLE_TH_ERRORS
}

template <int I>
PyObject *call(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return plan_call(kCalls[I], args, n);
}

// ------------------------------------------------- conjugate gradients

// cg_update(lambda, x, res, p, q, rs)
PyObject *cg_update(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != 6 || !PyFloat_CheckExact(args[0]) || !plain_mode())
        return not_implemented();
    Tensor t[5];
    for (int i = 0; i < 5; ++i) {
        const Tensor *q = tensor_of(args[1 + i]);
        if (!q || !q->defined() || !plain(*q, at::kFloat, q->device()) ||
            (i > 0 && q->device() != t[0].device()))
            return not_implemented();
        t[i] = *q;
        if (i == 0 && t[0].dim() != 2)
            return not_implemented();
        if (!(i < 4 ? is_rows(t[i], t[0].size(0), t[0].size(1)) : is_list(t[i], t[0].size(0))))
            return not_implemented();
    }
    if (t[0].size(0) > INT32_MAX || t[0].size(1) > INT32_MAX)
        return not_implemented();
    const int rc = fmm_cg_update((int32_t)t[0].size(0), (int32_t)t[0].size(1),
                                 (float)PyFloat_AS_DOUBLE(args[0]), pointer<float>(t[0]),
                                 pointer<float>(t[1]), pointer<float>(t[2]), pointer<float>(t[3]),
                                 pointer<float>(t[4]), stream());
    if (rc != FMM_OK)
        return raise_status(rc, "fmm_cg_update");
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// -------------------------------------------------------------- autograd

struct Locked {   // the interpreter lock, taken for a scope
    PyGILState_STATE s = PyGILState_Ensure();
    ~Locked() { PyGILState_Release(s); }
};

// Keeps the Python plan (and with it the C plan) alive in a graph, and the
// Python adjoint for operands that this one does not take.
struct PlanRef : torch::CustomClassHolder {
    PlanPtr plan;
    PyObject *owner, *gradients;
    PlanRef(PlanPtr p, PyObject *o, PyObject *g) : plan(std::move(p)), owner(o), gradients(g)
    {
        Py_INCREF(owner);
        Py_INCREF(gradients);
    }
    ~PlanRef() override
    {
        if (!Py_IsInitialized())
            return;
        const Locked lock;
        Py_DECREF(owner);
        Py_DECREF(gradients);
    }
};

// The Python exception that is set, for a thread that gives up the lock.
[[noreturn]] void throw_python_error()
{
    python_error e;
    e.persist();
    throw e;
}

// FmmError on a thread without the lock.
[[noreturn]] void throw_status(int status, const char *where)
{
    const Locked lock;
    raise_status(status, where);
    throw_python_error();
}

// gradients(plan, transpose, vals, A, B, G, need) of autograd.py.
tensor_list python_gradients(const PlanRef &ref, bool transpose, const Tensor &vals, const Tensor &A,
                             const Tensor &B, const Tensor &G, bool need_A, bool need_B, bool need_s)
{
    const Locked lock;
    PyObject *r = PyObject_CallFunction(
        ref.gradients, "OONNNN(NNN)", ref.owner, transpose ? Py_True : Py_False,
        THPVariable_Wrap(vals), THPVariable_Wrap(A), THPVariable_Wrap(B), THPVariable_Wrap(G),
        PyBool_FromLong(need_A), PyBool_FromLong(need_B), PyBool_FromLong(need_s));
    if (!r)
        throw_python_error();
    Tensor d[3];
    for (int i = 0; i < 3; ++i) {
        PyObject *x = PySequence_GetItem(r, i);
        if (x && THPVariable_Check(x))
            d[i] = THPVariable_Unpack(x);
        Py_XDECREF(x);
    }
    Py_DECREF(r);
    if (PyErr_Occurred())
        throw_python_error();
    return {d[0], d[1], d[2], Tensor(), Tensor()};
}

struct FusedMM : torch::autograd::Function<FusedMM> {
    // vals comes last of the tensors: without it A and B keep their edges
    static Tensor forward(AutogradContext *ctx, const Tensor &A, const Tensor &B,
                          const std::optional<Tensor> &values,
                          const c10::intrusive_ptr<PlanRef> &ref, bool transpose)
    {
        const Tensor vals = values.value_or(Tensor());
        const Plan &p = *ref->plan;
        Tensor out = empty({transpose ? p.n : p.m, p.r}, at::kFloat, p.device);
        const int rc = (transpose ? fmm_fusedmm_t : fmm_fusedmm)(
            p.handle, pointer<float>(vals), pointer(A), pointer(B), pointer<float>(out), stream());
        if (rc != FMM_OK)
            throw_status(rc, transpose ? "fmm_fusedmm_t" : "fmm_fusedmm");
        ctx->saved_data["plan"] = c10::IValue::make_capsule(ref);
        ctx->saved_data["transpose"] = transpose;
        ctx->save_for_backward({vals, A, B});
        return out;
    }

    static tensor_list backward(AutogradContext *ctx, tensor_list grads)
    {
        const auto holder = ctx->saved_data["plan"].toCapsule();
        const PlanRef &ref = *static_cast<const PlanRef *>(holder.get());
        const Plan &p = *ref.plan;
        const bool transpose = ctx->saved_data["transpose"].toBool();
        const auto saved = ctx->get_saved_variables();
        const Tensor &vals = saved[0], &A = saved[1], &B = saved[2];
        Tensor G = grads[0].contiguous();
        if (G.scalar_type() != at::kFloat)
            G = G.to(at::kFloat);
        const bool need_s = vals.defined() && ctx->needs_input_grad(2);
        const bool need_A = ctx->needs_input_grad(0), need_B = ctx->needs_input_grad(1);
        Tensor ds, dA, dB;
        if (need_s || need_A || need_B) {
            // what a saved-tensor hook gave back may have any layout, shape,
            // dtype or device: the Python path raises its error
            if ((vals.defined() && !operand('v', vals, p)) || !operand('A', A, p) ||
                !operand('B', B, p) || !operand(transpose ? 'N' : 'M', G, p))
                return python_gradients(ref, transpose, vals, A, B, G, need_A, need_B, need_s);
            const bool typed = p.dtype != at::kFloat && p.r <= kTypedMaxR;
            const at::ScalarType dt = typed ? p.dtype : at::kFloat;
            if (need_s)
                ds = empty({p.nnz}, at::kFloat, p.device);
            if (need_A)
                dA = empty({p.m, p.r}, dt, p.device);
            if (need_B)
                dB = empty({p.n, p.r}, dt, p.device);
            const auto fn = transpose ? fmm_fusedmm_t_bwd_typed : fmm_fusedmm_bwd_typed;
            const char *name = transpose ? "fmm_fusedmm_t_bwd" : "fmm_fusedmm_bwd";
            const auto plain_fn = transpose ? fmm_fusedmm_t_bwd : fmm_fusedmm_bwd;
            const int rc =
                typed ? fn(p.handle, pointer<float>(vals), pointer(A), pointer(B), pointer<float>(G),
                           pointer(dA), pointer(dB), pointer<float>(ds), stream())
                      : plain_fn(p.handle, pointer<float>(vals), pointer(A), pointer(B),
                                 pointer<float>(G), pointer<float>(dA), pointer<float>(dB),
                                 pointer<float>(ds), stream());
            if (rc != FMM_OK)
                throw_status(rc, name);
            if (dA.defined() && dA.scalar_type() != A.scalar_type())
                dA = dA.to(A.scalar_type());
            if (dB.defined() && dB.scalar_type() != B.scalar_type())
                dB = dB.to(B.scalar_type());
        }
        return {dA, dB, ds, Tensor(), Tensor()};
    }
};

// autograd(plan capsule, plan object, vals, A, B, transpose, gradients)
PyObject *autograd(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const PlanPtr *pp = n == 7 ? plan_of(args[0]) : nullptr;
    if (!pp || !plain_mode())
        return not_implemented();
    const Plan &p = **pp;
    Tensor t[3];
    const char *kinds = "vAB";
    for (int i = 0; i < 3; ++i)
        if (!operand(kinds[i], args[2 + i], p, t[i]) ||
            (t[i].defined() && t[i]._fw_grad(/*level=*/0).defined()))
            return not_implemented();
    const int transpose = PyObject_IsTrue(args[5]);
    if (transpose < 0)
        return nullptr;
    auto ref = c10::make_intrusive<PlanRef>(*pp, args[1], args[6]);
    Tensor out;
    {
        Released unlocked;
        const std::optional<Tensor> vals =
            t[0].defined() ? std::optional<Tensor>(t[0]) : std::nullopt;
        out = FusedMM::apply(t[1], t[2], vals, ref, transpose != 0);
    }
    return THPVariable_Wrap(out);
    END_HANDLE_TH_ERRORS
}

// ---------------------------------------------------------------- module

void free_plan(PyObject *capsule)
{
    delete static_cast<PlanPtr *>(PyCapsule_GetPointer(capsule, kPlanName));
}

// plan(handle, m, n, r, nnz, bfloat16, device index) -> capsule
PyObject *make_plan(PyObject *, PyObject *args)
{
    unsigned long long handle;
    long long m, n, r, nnz;
    int bf16, device;
    if (!PyArg_ParseTuple(args, "KLLLLpi", &handle, &m, &n, &r, &nnz, &bf16, &device))
        return nullptr;
    auto *p = new PlanPtr(std::make_shared<Plan>(
        Plan{reinterpret_cast<const fmm_plan *>(handle), m, n, r, nnz, bf16 ? at::kBFloat16 : at::kFloat,
             at::Device(at::kCUDA, (c10::DeviceIndex)device)}));
    PyObject *o = PyCapsule_New(p, kPlanName, free_plan);
    if (!o)
        delete p;
    return o;
}

// close(capsule): graphs that still hold the plan get an error, not a freed handle
PyObject *close_plan(PyObject *, PyObject *o)
{
    if (const PlanPtr *p = plan_of(o))
        (*p)->handle = nullptr;
    Py_RETURN_NONE;
}

PyObject *set_check(PyObject *, PyObject *o)
{
    Py_INCREF(o);
    Py_XDECREF(g_check);
    g_check = o;
    Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef kMethods[] = {
    {"sddmm", FAST(call<0>)},
    {"spmm", FAST(call<1>)},
    {"spmm_t", FAST(call<2>)},
    {"fusedmm", FAST(call<3>)},
    {"fusedmm_t", FAST(call<4>)},
    {"cg_update", FAST(cg_update)},
    {"autograd", FAST(autograd)},
    {"plan", make_plan, METH_VARARGS, nullptr},
    {"close", close_plan, METH_O, nullptr},
    {"set_check", set_check, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "fmm_calls", nullptr, -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_fmm_calls(void)
{
    PyObject *m = PyModule_Create(&kModule);
    // the PyTorch it is built for: fmm.py uses it with no other
    if (m && PyModule_AddStringConstant(m, "torch_version", TORCH_VERSION) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
