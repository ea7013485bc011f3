// Python side of the transform calls: argument checks, output allocation, workspace and stream look-up, the C-ABI call
// and the autograd nodes, in native code.  No arithmetic: every step of the transforms runs in libcqt_b200.so.
//
// Why native: a call on a small batch is enqueued slower than the GPU runs it.  With ctypes marshalling, attribute
// look-ups and Python autograd functions the host needed 20 us per transform and 240 us per training step (two
// transforms and their adjoints) for 80 us of GPU work; see binding.py for the methods built on this.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/function.h>
#include <torch/csrc/autograd/functions/utils.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/Exceptions.h>

#include "../../include/cqt.h"

namespace {

enum Which { kAnalyse = 0, kSynthesiseAdjoint = 1, kSynthesise = 2, kAnalyseAdjoint = 3, kAnalyseStatic = 4 };
const char *const kNames[] = {"cqt_analyse", "cqt_synthesise_adjoint", "cqt_synthesise", "cqt_analyse_adjoint", "cqt_analyse_static_ws"};
bool to_coefficients(int which) { return which == kAnalyse || which == kSynthesiseAdjoint || which == kAnalyseStatic; }

PyObject *s_h, *s_ws, *s_workspace, *s_coeff_count, *s_N, *s_cuda_stream;   // interned attribute names
PyObject *g_error = nullptr;                                                 // CqtError

constexpr int64_t kAbsent = INT64_MIN;   // valid_len not given

// an exception is set
struct PyFailure {};

struct GilRelease {
    PyThreadState *state = PyEval_SaveThread();
    ~GilRelease() { PyEval_RestoreThread(state); }
};
struct GilAcquire {
    PyGILState_STATE state = PyGILState_Ensure();
    ~GilAcquire() { PyGILState_Release(state); }
};

void require(bool ok, const char *what) {
    if (ok) return;
    PyErr_SetString(PyExc_AssertionError, what);
    throw PyFailure();
}

long long int_attr(PyObject *o, PyObject *name) {
    PyObject *v = PyObject_GetAttr(o, name);
    if (!v) throw PyFailure();
    const long long r = PyLong_AsLongLong(v);
    Py_DECREF(v);
    if (r == -1 && PyErr_Occurred()) throw PyFailure();
    return r;
}

const at::Tensor &tensor_of(PyObject *o) {
    require(THPVariable_Check(o), "a torch tensor is needed");
    return THPVariable_Unpack(o);
}

void check_status(cqt_status s, const char *what) {
    if (s == CQT_OK) return;
    if (PyObject *e = PyObject_CallFunction(g_error, "is", (int)s, what)) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw PyFailure();
}

void *stream_of(PyObject *stream) {
    if (stream == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    return reinterpret_cast<void *>((intptr_t)int_attr(stream, s_cuda_stream));
}

// The library reads memory as it lies there, and a tensor may be a conjugate or a negative of it that is still to be
// computed.  Such an input is computed on the stream of the call: its memory is then given back in that stream's order too.
at::Tensor as_stored(const at::Tensor &t, void *stream) {
    if (!t.is_conj() && !t.is_neg()) return t;
    at::AutoDispatchBelowADInplaceOrView no_grad;
    const c10::cuda::CUDAStreamGuard guard(c10::cuda::getStreamFromExternal(reinterpret_cast<cudaStream_t>(stream), t.device().index()));
    return t.resolve_conj().resolve_neg();
}
void require_stored(const at::Tensor &t) { require(!t.is_conj() && !t.is_neg(), "the output is no conjugate or negative view"); }

// Plan._ws, grown by Plan.workspace when it is too small
at::Tensor workspace_of(PyObject *plan, const cqt_plan *p, int64_t batch) {
    PyObject *w = PyObject_GetAttr(plan, s_ws);
    if (!w) throw PyFailure();
    if (w == Py_None || (size_t)tensor_of(w).numel() < cqt_plan_workspace_bytes(p, batch)) {
        Py_DECREF(w);
        PyObject *n = PyLong_FromLongLong(batch);
        w = n ? PyObject_CallMethodOneArg(plan, s_workspace, n) : nullptr;
        Py_XDECREF(n);
        if (!w) throw PyFailure();
    }
    at::Tensor t = THPVariable_Check(w) ? THPVariable_Unpack(w) : at::Tensor();
    Py_DECREF(w);
    require(t.defined(), "the workspace is a tensor");
    return t;
}

// One transform.  out undefined: allocated.  Needs the GIL.
at::Tensor run(PyObject *plan, int which, const at::Tensor &in, int64_t valid_len, at::Tensor out, at::Tensor ws, PyObject *stream_arg) {
    const cqt_plan *p = reinterpret_cast<const cqt_plan *>((intptr_t)int_attr(plan, s_h));
    const bool forward = to_coefficients(which);
    const int64_t batch = in.dim() == 2 ? in.size(0) : 0;
    if (forward) {
        require(in.is_cuda() && in.scalar_type() == at::kFloat && in.dim() == 2 && in.stride(1) == 1,
                "x is a [batch, n] float32 CUDA tensor with unit column stride");
        if (valid_len == kAbsent) valid_len = in.size(1);
        if (!out.defined()) out = at::empty({batch, (int64_t)int_attr(plan, s_coeff_count)}, in.options().dtype(at::kComplexFloat));
    } else {
        require(in.is_cuda() && in.scalar_type() == at::kComplexFloat && in.dim() == 2 && in.is_contiguous() && in.size(1) == int_attr(plan, s_coeff_count),
                "c is a contiguous [batch, coeff_count] complex64 CUDA tensor");
        if (valid_len == kAbsent) valid_len = int_attr(plan, s_N);
        if (!out.defined()) out = at::empty({batch, valid_len}, in.options().dtype(at::kFloat));
    }
    require_stored(out);
    if (!ws.defined() && which != kAnalyseStatic && batch > 0) ws = workspace_of(plan, p, batch);
    void *stream = stream_of(stream_arg);
    const at::Tensor src = as_stored(in, stream);
    void *wp = ws.defined() ? ws.data_ptr() : nullptr;
    const size_t wn = ws.defined() ? (size_t)ws.numel() : 0;
    void *ip = src.data_ptr(), *op = out.data_ptr();
    cqt_status s;
    {
        GilRelease nogil;
        if (forward) {
            const float *x = (const float *)ip;
            cqt_c64 *c = (cqt_c64 *)op;
            const int64_t stride = src.stride(0);
            s = which == kAnalyse             ? cqt_analyse(p, x, stride, batch, valid_len, c, wp, wn, stream)
                : which == kSynthesiseAdjoint ? cqt_synthesise_adjoint(p, x, stride, batch, valid_len, c, wp, wn, stream)
                                              : cqt_analyse_static_ws(p, x, stride, batch, valid_len, c, stream);
        } else {
            const cqt_c64 *c = (const cqt_c64 *)ip;
            float *x = (float *)op;
            const int64_t stride = out.stride(0);
            s = which == kSynthesise ? cqt_synthesise(p, c, batch, valid_len, x, stride, wp, wn, stream)
                                     : cqt_analyse_adjoint(p, c, batch, valid_len, x, stride, wp, wn, stream);
        }
    }
    check_status(s, kNames[which]);
    return out;
}

int64_t optional_length(PyObject *o) {
    if (o == Py_None) return kAbsent;
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyFailure();
    return v;
}
at::Tensor optional_tensor(PyObject *o) { return o == Py_None ? at::Tensor() : tensor_of(o); }

template <class F>
PyObject *guarded(F f) {
    try {
        return f();
    } catch (const PyFailure &) {
        return nullptr;
    } catch (...) {
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}

// transform(plan, which, input, valid_len, out, ws, stream) -> output
PyObject *transform(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        require(n == 7, "seven arguments");
        return THPVariable_Wrap(run(a[0], (int)PyLong_AsLong(a[1]), tensor_of(a[2]), optional_length(a[3]), optional_tensor(a[4]),
                                    optional_tensor(a[5]), a[6]));
    });
}

// Backward of a transform: under <u, v> = Re(u^H v) the real adjoint applied to the cotangent, which is PyTorch's
// convention for complex tensors (the gradient of a real loss at c is dL/dRe c + i dL/dIm c).  Nothing of the forward
// pass is kept but the plan.
struct AdjointNode final : torch::autograd::Node {
    PyObject *plan;
    int which;            // the adjoint's own transform
    int64_t valid_len, width;   // width: columns of the forward input (signals)
    AdjointNode(PyObject *p, int w, int64_t vl, int64_t wd) : plan(p), which(w), valid_len(vl), width(wd) { Py_INCREF(plan); }
    ~AdjointNode() override {
        if (!Py_IsInitialized()) return;
        GilAcquire gil;
        Py_DECREF(plan);
    }
    torch::autograd::variable_list apply(torch::autograd::variable_list &&grads) override {
        if (!grads[0].defined()) return {at::Tensor()};
        at::AutoDispatchBelowADInplaceOrView no_grad;
        const at::Tensor g = grads[0].contiguous();
        at::Tensor out;
        // columns beyond valid_len were never read: zero gradient
        if (which == kAnalyseAdjoint && width != valid_len) out = at::zeros({g.size(0), width}, g.options().dtype(at::kFloat));
        GilAcquire gil;
        try {
            return {run(plan, which, g, valid_len, out, at::Tensor(), Py_None)};
        } catch (const PyFailure &) {
            python_error e;
            e.persist();
            throw e;
        }
    }
    std::string name() const override { return which == kAnalyseAdjoint ? "CqtAnalyseBackward" : "CqtSynthesiseBackward"; }
};

// differentiable(plan, which, input, valid_len) -> output; which: kAnalyse or kSynthesise
PyObject *differentiable(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        require(n == 4, "four arguments");
        const int which = (int)PyLong_AsLong(a[1]);
        const at::Tensor &x = tensor_of(a[2]);
        int64_t valid_len = optional_length(a[3]);
        require(which == kAnalyse || which == kSynthesise, "analyse or synthesise");
        require(x.dim() == 2, "a [batch, n] tensor");
        if (x._fw_grad(0).defined()) {   // its tangent would be lost without a word
            PyErr_SetString(PyExc_NotImplementedError, "the transforms have no forward-mode derivative: use the backward one, or transform the tangent");
            throw PyFailure();
        }
        if (valid_len == kAbsent) valid_len = which == kAnalyse ? x.size(1) : int_attr(a[0], s_N);
        at::Tensor out;
        {
            at::AutoDispatchBelowADInplaceOrView no_grad;
            out = run(a[0], which, x.contiguous(), valid_len, at::Tensor(), at::Tensor(), Py_None);
        }
        if (torch::autograd::compute_requires_grad(x)) {
            auto node = std::shared_ptr<AdjointNode>(
                new AdjointNode(a[0], which == kAnalyse ? kAnalyseAdjoint : kSynthesiseAdjoint, valid_len, x.size(1)), torch::autograd::deleteNode);
            node->set_next_edges(torch::autograd::collect_next_edges(x));
            torch::autograd::set_history(out, node);
        }
        return THPVariable_Wrap(std::move(out));
    });
}

// slicq_push(handle, x, stream) -> slices analysed so far; slicq_pull(handle, y, stream) -> frames written
PyObject *push(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        require(n == 3, "three arguments");
        cqt_slicq *s = reinterpret_cast<cqt_slicq *>((intptr_t)PyLong_AsLongLong(a[0]));
        void *stream = stream_of(a[2]);
        const at::Tensor x = as_stored(tensor_of(a[1]), stream);
        const int64_t frames = x.size(1);
        const float *p = frames ? (const float *)x.data_ptr() : nullptr;
        int64_t done = 0;
        cqt_status r;
        {
            GilRelease nogil;
            r = slicq_push(s, p, frames ? x.stride(0) : 0, frames, stream, &done);
        }
        check_status(r, "slicq_push");
        return PyLong_FromLongLong(done);
    });
}
PyObject *pull(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        require(n == 3, "three arguments");
        cqt_slicq *s = reinterpret_cast<cqt_slicq *>((intptr_t)PyLong_AsLongLong(a[0]));
        const at::Tensor &y = tensor_of(a[1]);
        require_stored(y);
        void *stream = stream_of(a[2]);
        int64_t wrote = 0;
        float *p = (float *)y.data_ptr();
        cqt_status r;
        {
            GilRelease nogil;
            r = slicq_pull(s, p, y.stride(0), y.size(1), stream, &wrote);
        }
        check_status(r, "slicq_pull");
        return PyLong_FromLongLong(wrote);
    });
}

PyObject *set_error(PyObject *, PyObject *cls) {
    Py_INCREF(cls);
    Py_XSETREF(g_error, cls);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"transform", (PyCFunction)(void (*)(void))transform, METH_FASTCALL, nullptr},
    {"differentiable", (PyCFunction)(void (*)(void))differentiable, METH_FASTCALL, nullptr},
    {"slicq_push", (PyCFunction)(void (*)(void))push, METH_FASTCALL, nullptr},
    {"slicq_pull", (PyCFunction)(void (*)(void))pull, METH_FASTCALL, nullptr},
    {"set_error", set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cqt_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cqt_torch() {
    s_h = PyUnicode_InternFromString("_h");
    s_ws = PyUnicode_InternFromString("_ws");
    s_workspace = PyUnicode_InternFromString("workspace");
    s_coeff_count = PyUnicode_InternFromString("coeff_count");
    s_N = PyUnicode_InternFromString("N");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
