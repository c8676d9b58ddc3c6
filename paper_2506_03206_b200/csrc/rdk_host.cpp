// CPython side of the binding's hot entry points: takes torch tensors apart (types, strides, device pointers, the
// current stream) and calls the C ABI of librdk_b200.so.  The calls of a decoding step are a few microseconds of GPU
// work each for a handful of rows; the same marshalling through ctypes costs more than that (45 us a step of three
// launches, against 16 us of GPU time for 1 x 5 rows of 128k tokens).  Argument errors raise what the ctypes
// binding raises; a non-zero status goes back to the caller, which turns it into RdkError.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/Functions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "rdk.h"

namespace {

PyObject* g_keys[10];           // names of the members of rdk_outputs, in the struct's order
const char* const kNames[10] = {"draft_token", "out_token", "accepted", "accept_prob", "alpha", "theta", "S",
                                "residual_mass", "accepted_len", "status_word"};

struct Raised {};               // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw Raised{};
}

const at::Tensor& tensor(PyObject* o, const char* what) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a torch tensor", what);
        throw Raised{};
    }
    return THPVariable_Unpack(o);
}
long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
const at::Tensor& rows2d(PyObject* o, const char* what) {
    const at::Tensor& t = tensor(o, what);
    if (t.dim() != 2 || t.stride(1) != 1) {
        PyErr_Format(PyExc_ValueError, "%s must be 2-D with contiguous rows", what);
        throw Raised{};
    }
    return t;
}
int dtype_code(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return RDK_F32;
    if (t.scalar_type() == at::kBFloat16) return RDK_BF16;
    PyErr_Format(PyExc_TypeError, "unsupported dtype torch.%s: the library takes float32 or bfloat16", at::toString(t.scalar_type()));
    throw Raised{};
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

rdk_outputs outputs(PyObject* dict) {
    if (!PyDict_Check(dict)) raise(PyExc_TypeError, "the outputs must be a dict of tensors");
    void* p[10];
    for (int k = 0; k < 10; ++k) {
        PyObject* o = PyDict_GetItemWithError(dict, g_keys[k]);
        if (!o && PyErr_Occurred()) throw Raised{};
        p[k] = (!o || o == Py_None) ? nullptr : tensor(o, kNames[k]).data_ptr();
    }
    rdk_outputs r;
    r.draft_token = static_cast<int32_t*>(p[0]); r.out_token = static_cast<int32_t*>(p[1]);
    r.accepted = static_cast<uint8_t*>(p[2]); r.accept_prob = static_cast<float*>(p[3]);
    r.alpha = static_cast<float*>(p[4]); r.theta = static_cast<float*>(p[5]); r.S = static_cast<float*>(p[6]);
    r.residual_mass = static_cast<float*>(p[7]); r.accepted_len = static_cast<int32_t*>(p[8]);
    r.status_word = static_cast<int32_t*>(p[9]);
    return r;
}

// index buffer, N, n, target or NULL, drafter or NULL, batch, positions, kind, flags
rdk_problem problem(PyObject* buffer, PyObject* N, PyObject* n, const at::Tensor* target, const at::Tensor* drafter,
                    PyObject* batch, PyObject* positions, PyObject* kind, long long flags) {
    rdk_problem p{};
    p.N = (int32_t)integer(N); p.n = (int32_t)integer(n);
    p.batch = (int32_t)integer(batch); p.positions = (int32_t)integer(positions);
    p.target_dtype = target ? dtype_code(*target) : RDK_F32;
    p.drafter_dtype = drafter ? dtype_code(*drafter) : RDK_F32;
    p.drafter_kind = (int32_t)integer(kind);
    p.flags = (int32_t)flags;
    p.target_row_stride = target ? target->stride(0) : 0;
    p.drafter_row_stride = drafter ? drafter->stride(0) : 0;
    p.kept_index = tensor(buffer, "index").data_ptr();
    return p;
}
long long per_row(const at::Tensor& uniforms, long long rows, bool check) {
    if (rows == 0) raise(PyExc_ZeroDivisionError, "no rows");
    if (check && (uniforms.scalar_type() != at::kFloat || !uniforms.is_contiguous() || uniforms.numel() % (rows * 4)))
        raise(PyExc_ValueError, "uniforms must be contiguous float32 [rows, trials, 4]");
    return uniforms.numel() / (rows * 4);
}
void arity(Py_ssize_t got, Py_ssize_t want) {
    if (got != want) raise(PyExc_TypeError, "wrong number of arguments");
}

// The library's calls run without the interpreter lock: a launch may have to wait for room in the stream's queue.  Only the
// C call itself belongs in here: whatever may throw (a pointer of a tensor without storage, a stride, the current stream) is
// worked out before, and the lock comes back on every way out.
class Unlocked {
public:
    Unlocked() : state_(PyEval_SaveThread()) {}
    ~Unlocked() { PyEval_RestoreThread(state_); }
    Unlocked(const Unlocked&) = delete;
    Unlocked& operator=(const Unlocked&) = delete;
private:
    PyThreadState* state_;
};
template <typename F> int unlocked(F f) {
    Unlocked lock;
    return f();
}
template <typename T> T* pointer(const at::Tensor& t) { return static_cast<T*>(t.data_ptr()); }

template <typename F> PyObject* guarded(F f) {
    try {
        return f();
    } catch (const Raised&) {
        return nullptr;
    } catch (const c10::IndexError& e) {
        PyErr_SetString(PyExc_IndexError, e.what_without_backtrace());
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// (buffer, N, n, mode, target, drafter, w, uniforms, batch, positions, kind, flags, out, ws) -> status
PyObject* sample(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arity(n, 14);
        const at::Tensor& target = rows2d(a[4], "target");
        const at::Tensor* drafter = a[5] == Py_None ? nullptr : &tensor(a[5], "drafter");
        const at::Tensor* w = a[6] == Py_None ? nullptr : &tensor(a[6], "w");
        const at::Tensor& u = tensor(a[7], "uniforms");
        const rdk_problem pb = problem(a[0], a[1], a[2], &target, drafter, a[8], a[9], a[10], integer(a[11]));
        const long long trials = per_row(u, (long long)pb.batch * pb.positions, true);
        const rdk_outputs o = outputs(a[12]);
        const at::Tensor& ws = tensor(a[13], "ws");
        const int mode = (int)integer(a[3]);
        const void *z = pointer<void>(target), *y = drafter ? pointer<void>(*drafter) : nullptr;
        const float *wp = w ? pointer<float>(*w) : nullptr, *up = pointer<float>(u);
        const int64_t w_stride = w ? w->stride(0) : 0;
        void *wsp = pointer<void>(ws), *s = stream();
        const size_t ws_bytes = (size_t)ws.numel();
        return PyLong_FromLong(unlocked([&] { return rdk_sample_and_verify(&pb, mode, z, y, wp, w_stride, up, (int32_t)trials, &o, wsp, ws_bytes, s); }));
    });
}

// a [N] prior is one row shared by all rows (stride 0); a [rows, N] prior has its row stride
long long prior_stride(const at::Tensor& prior, PyObject* o, const at::Tensor& target, long long N) {
    if (prior.scalar_type() != target.scalar_type()) raise(PyExc_ValueError, "the prior must have the target's dtype");
    if (prior.dim() == 1) {
        if (prior.numel() != N || !prior.is_contiguous()) raise(PyExc_ValueError, "a shared prior must be a contiguous [N] tensor");
        return 0;
    }
    return rows2d(o, "prior").stride(0);
}

// A workspace of a call's own from torch's allocator, which hands the memory out again in the order of the stream.  The call that
// takes it can do without: none (an undefined tensor) where the memory is not to be had, and while the stream is captured,
// where the allocator may have to be kept out of it.
at::Tensor own_workspace(size_t bytes, const at::Tensor& like, const c10::cuda::CUDAStream& current) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (!bytes || cudaStreamIsCapturing(current.stream(), &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) return at::Tensor();
    try {
        return at::empty({(int64_t)bytes}, like.options().dtype(at::kByte));
    } catch (const c10::OutOfMemoryError&) {
        return at::Tensor();
    }
}

// (buffer, N, n, target, prior, drafter, uniforms, batch, positions, kind, out[, ws or None]) -> status
PyObject* sample_prior(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 11) arity(n, 12);
        const at::Tensor& target = rows2d(a[3], "target");
        const at::Tensor& prior = tensor(a[4], "prior");
        const at::Tensor& drafter = rows2d(a[5], "drafter");
        const at::Tensor& u = tensor(a[6], "uniforms");
        const rdk_problem pb = problem(a[0], a[1], a[2], &target, &drafter, a[7], a[8], a[9], 0);
        const long long trials = per_row(u, (long long)pb.batch * pb.positions, false);
        const rdk_outputs o = outputs(a[10]);
        const long long stride = prior_stride(prior, a[4], target, pb.N);
        const void *z = pointer<void>(target), *pr = pointer<void>(prior), *y = pointer<void>(drafter);
        const float* up = pointer<float>(u);
        const c10::cuda::CUDAStream current = c10::cuda::getCurrentCUDAStream();
        void* s = current.stream();
        at::Tensor ws;
        if (n == 12 && a[11] != Py_None) ws = tensor(a[11], "ws");
        else ws = own_workspace(rdk_sample_prior_workspace_bytes(&pb, z, pr, stride, y, (int32_t)trials), target, current);
        void* wsp = ws.defined() && ws.numel() ? pointer<void>(ws) : nullptr;
        const size_t ws_bytes = wsp ? ws.nbytes() : 0;
        return PyLong_FromLong(unlocked([&] { return rdk_sample_and_verify_prior_ws(&pb, z, pr, stride, y, up, (int32_t)trials, &o, wsp, ws_bytes, s); }));
    });
}

// (buffer, N, n, target, prior or None, drafter, batch, positions, kind) -> (status, q~, theta, S)
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arity(n, 9);
        const at::Tensor& target = rows2d(a[3], "target");
        const at::Tensor& drafter = rows2d(a[5], "drafter");
        const rdk_problem pb = problem(a[0], a[1], a[2], &target, &drafter, a[6], a[7], a[8], 0);
        const int64_t rows = (int64_t)pb.batch * pb.positions;
        const auto opt = target.options().dtype(at::kFloat);
        const at::Tensor qt = at::empty({rows, pb.N}, opt), theta = at::empty({rows}, opt), S = at::empty({rows}, opt);
        const at::Tensor* prior = a[4] == Py_None ? nullptr : &tensor(a[4], "prior");
        const long long stride = prior ? prior_stride(*prior, a[4], target, pb.N) : 0;
        float *q = pointer<float>(qt), *th = pointer<float>(theta), *sum = pointer<float>(S);
        const void *z = pointer<void>(target), *pr = prior ? pointer<void>(*prior) : nullptr, *y = pointer<void>(drafter);
        void* s = stream();
        const int st = unlocked([&] {
            return prior ? rdk_redistribute_linear_prior(&pb, z, pr, stride, y, q, th, sum, s) : rdk_redistribute_linear(&pb, z, y, q, th, sum, s);
        });
        return Py_BuildValue("(iNNN)", st, THPVariable_Wrap(qt), THPVariable_Wrap(theta), THPVariable_Wrap(S));
    });
}

// (buffer, N, n, drafter, M data, M layout, M ld, batch, positions, kind, w, ws, status word or None) -> (status, S)
PyObject* exact(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arity(n, 13);
        const at::Tensor& drafter = rows2d(a[3], "drafter");
        const rdk_problem pb = problem(a[0], a[1], a[2], nullptr, &drafter, a[7], a[8], a[9], 0);
        rdk_affinity M{};
        M.data = tensor(a[4], "M").data_ptr(); M.layout = (int32_t)integer(a[5]); M.ld = integer(a[6]);
        const at::Tensor& w = tensor(a[10], "w_out");
        const at::Tensor& ws = tensor(a[11], "ws");
        void* status = a[12] == Py_None ? nullptr : tensor(a[12], "status_word").data_ptr();
        const at::Tensor S = at::empty({(int64_t)pb.batch * pb.positions}, drafter.options().dtype(at::kFloat));
        const void* y = pointer<void>(drafter);
        float *wp = pointer<float>(w), *sum = pointer<float>(S);
        void *wsp = pointer<void>(ws), *s = stream();
        const size_t ws_bytes = (size_t)ws.numel();
        const int st = unlocked([&] { return rdk_redistribute_exact(&pb, y, &M, wp, sum, wsp, ws_bytes, static_cast<int32_t*>(status), s); });
        return Py_BuildValue("(iN)", st, THPVariable_Wrap(S));
    });
}

// (N, batch, positions, bonus, uniforms, draft_token, accepted, out_token) -> (status, seq_tokens, seq_len)
PyObject* emit(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arity(n, 8);
        const at::Tensor& bonus = rows2d(a[3], "bonus_target");
        rdk_problem pb{};
        pb.N = (int32_t)integer(a[0]); pb.n = 1; pb.batch = (int32_t)integer(a[1]); pb.positions = (int32_t)integer(a[2]);
        pb.target_dtype = dtype_code(bonus);
        pb.flags = RDK_FLAG_PAD_SEQUENCES;
        const at::Tensor& u = tensor(a[4], "uniforms");
        const int64_t trials = per_row(u, (long long)pb.batch * pb.positions, false);
        const auto opt = bonus.options().dtype(at::kInt);
        const at::Tensor seq = at::empty({pb.batch, trials, (int64_t)pb.positions + 1}, opt), len = at::empty({pb.batch, trials}, opt);
        const at::Tensor &draft = tensor(a[5], "draft_token"), &acc = tensor(a[6], "accepted"), &out = tensor(a[7], "out_token");
        const void* z = pointer<void>(bonus);
        const int64_t z_stride = bonus.stride(0);
        const float* up = pointer<float>(u);
        const int32_t *d = pointer<int32_t>(draft), *o = pointer<int32_t>(out);
        const uint8_t* ap = pointer<uint8_t>(acc);
        int32_t *sp = pointer<int32_t>(seq), *lp = pointer<int32_t>(len);
        void* s = stream();
        const int st = unlocked([&] { return rdk_emit_sequences(&pb, z, z_stride, up, (int32_t)trials, d, ap, o, sp, lp, s); });
        return Py_BuildValue("(iNN)", st, THPVariable_Wrap(seq), THPVariable_Wrap(len));
    });
}

#define RDK_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {RDK_METHOD(sample), RDK_METHOD(sample_prior), RDK_METHOD(linear), RDK_METHOD(exact), RDK_METHOD(emit), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_rdk_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__rdk_host() {
    for (int k = 0; k < 10; ++k)
        if (!(g_keys[k] = PyUnicode_InternFromString(kNames[k]))) return nullptr;
    return PyModule_Create(&module);
}
