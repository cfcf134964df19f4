// The Python entry points' host path in native code: argument checks, output and workspace tensors, the call into
// libspecverify, the result object.  A verification of a small batch takes about as long on the GPU as its arguments
// took to marshal through ctypes (six checked tensors, five allocations, two structures), so a decoding loop over small
// batches was bound by the host: one sequence at V = 1000 took 36 us a call, of which the GPU was busy for 19.
//
// The module holds no state but the library's entry points, the result classes and interned names.  Workspaces are
// the caller's (a Workspace object of binding.py, grown by it).
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include "specverify.h"

namespace {

struct Library {
    decltype(&spec_workspace_bytes) workspace_bytes;
    decltype(&spec_analysis_workspace_bytes) analysis_workspace_bytes;
    decltype(&spec_verify_specinfer) specinfer, traversal;
    decltype(&spec_verify_otlp) otlp;
    decltype(&spec_tree_analysis) analysis;
    decltype(&spec_tree_probs) probs;
    decltype(&spec_sample_bonus) bonus;
} lib;
PyObject *verify_outputs_class, *analysis_outputs_class;
PyObject *n_buf, *n_get, *n_stream;
PyObject *n_out[10];
const char *const OUT_NAMES[10] = {"accepted_node", "accept_len", "out_tokens", "bonus_token", "status",
                                   "residual",      "node_thr",   "node_w_in",  "node_features", "margin"};

const char *error_name(int rc)
{
    static const char *const names[] = {"SPEC_OK", "SPEC_ERR_NULL", "SPEC_ERR_SHAPE", "SPEC_ERR_DTYPE", "SPEC_ERR_PARAM",
                                        "SPEC_ERR_WORKSPACE", "SPEC_ERR_UNSUPPORTED", "SPEC_ERR_CUDA"};
    return rc <= 0 && rc > -8 ? names[-rc] : "unknown error";
}

// an error that has been set as a Python exception
struct Raised {};
// a reference of this module's own
struct Owned {
    PyObject *o;
    explicit Owned(PyObject *p) : o(p) {}
    ~Owned() { Py_XDECREF(o); }
    Owned(const Owned &) = delete;
};
template <typename... A> [[noreturn]] void raise(const char *fmt, A... a)
{
    PyErr_Format(PyExc_RuntimeError, fmt, a...);
    throw Raised{};
}
void check(int rc, const char *what) { if (rc) raise("%s failed: %s", what, error_name(rc)); }

// Calls f, which touches no Python object, with the interpreter's lock released: a launch may wait (a full queue, the first use of
// a kernel), and other threads run meanwhile, as with ctypes.
template <typename F> int unlocked(F f)
{
    struct Released {
        PyThreadState *state = PyEval_SaveThread();
        ~Released() { PyEval_RestoreThread(state); }
    } released;
    return f();
}

const at::Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) { PyErr_Format(PyExc_TypeError, "%s must be a tensor", name); throw Raised{}; }
    return THPVariable_Unpack(o);
}
const at::Tensor &cuda_tensor(PyObject *o, const char *name)
{
    const at::Tensor &t = tensor(o, name);
    if (!t.is_cuda()) raise("%s must live on a CUDA device (there is no CPU path)", name);
    return t;
}
void *pointer_or_null(PyObject *o, const char *name) { return o == Py_None ? nullptr : tensor(o, name).data_ptr(); }
double number(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised{};
    return v;
}
long long integer(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
int truncated(PyObject *o)        // int(x), as the callers write it
{
    if (PyLong_Check(o)) return (int)integer(o);
    PyObject *i = PyNumber_Long(o);
    if (!i) throw Raised{};
    const long long v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return (int)v;
}
void *stream_of(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *s = PyObject_GetAttr(o, n_stream);
    if (!s) throw Raised{};
    void *p = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    if (!p && PyErr_Occurred()) throw Raised{};
    return p;
}
at::Tensor empty(at::IntArrayRef sizes, at::ScalarType t, const at::Device &d)
{
    return at::Tensor(at::detail::empty_cuda(sizes, t, d, std::nullopt));
}

// the caller's Workspace: its buffer, grown by the object itself when too small (held until the call has been enqueued: another
// thread may grow the object meanwhile)
struct Scratch { void *ptr; int64_t bytes; at::Tensor buf; };
Scratch scratch_of(PyObject *workspace, int64_t bytes)
{
    for (int attempt = 0;; ++attempt) {
        PyObject *buf = PyObject_GetAttr(workspace, n_buf);
        if (!buf) throw Raised{};
        if (buf != Py_None) {
            const Owned held(buf);
            const at::Tensor t = tensor(buf, "buf");
            const int64_t have = t.numel();
            char *base = (char *)t.data_ptr();
            if (have >= bytes + 256) {
                const int64_t off = (256 - ((intptr_t)base & 255)) & 255;
                return {base + off, have - off, t};
            }
        } else {
            Py_DECREF(buf);
        }
        if (attempt) raise("the workspace did not grow");
        PyObject *n = PyLong_FromLongLong(bytes), *r = n ? PyObject_CallMethodOneArg(workspace, n_get, n) : nullptr;
        Py_XDECREF(n);
        if (!r) throw Raised{};
        Py_DECREF(r);
    }
}

void check_vector(const at::Tensor &t, const char *name, at::ScalarType dt, const char *type)
{
    if (t.scalar_type() != dt || !t.is_contiguous()) raise("%s must be a contiguous %s tensor", name, type);
}

// arguments 0 .. 9 of every call on a batch of trees: target, draft, parent, token, u_accept, u_bonus, temperature, top_k,
// top_p, temperature_per_seq
SpecIn spec_in(PyObject *const *a)
{
    const at::Tensor &zp = cuda_tensor(a[0], "target_logits"), &zq = cuda_tensor(a[1], "draft_logits");
    const at::Tensor &parent = cuda_tensor(a[2], "parent"), &token = cuda_tensor(a[3], "token");
    const at::Tensor &ua = cuda_tensor(a[4], "u_accept"), &ub = cuda_tensor(a[5], "u_bonus");
    const auto dt = zp.scalar_type();
    if ((dt != at::kFloat && dt != at::kBFloat16) || zq.scalar_type() != dt) raise("logits must both be float32 or both bfloat16");
    if (zp.dim() != 3 || zp.stride(2) != 1 || zq.dim() != 3 || zq.strides() != zp.strides())
        raise("logits must be [B,N,V] with a contiguous vocabulary axis and equal strides");
    const int64_t B = zp.size(0), N = zp.size(1), V = zp.size(2);
    check_vector(parent, "parent", at::kInt, "torch.int32");
    check_vector(token, "token", at::kInt, "torch.int32");
    check_vector(ua, "u_accept", at::kFloat, "torch.float32");
    check_vector(ub, "u_bonus", at::kFloat, "torch.float32");
    const auto is_bn = [&](const at::Tensor &t) { return t.dim() == 2 && t.size(0) == B && t.size(1) == N; };
    if (!is_bn(token) || !is_bn(ua) || !is_bn(ub)) raise("token, u_accept and u_bonus must be [B,N]");
    if (!(parent.dim() == 1 && parent.size(0) == N) && !is_bn(parent)) raise("parent must be [N] or [B,N]");
    SpecIn in = {};
    in.B = (int32_t)B; in.N = (int32_t)N; in.V = (int32_t)V;
    in.logits_dtype = dt == at::kFloat ? SPEC_F32 : SPEC_BF16;
    in.target_logits = zp.data_ptr(); in.draft_logits = zq.data_ptr();
    in.seq_stride = zp.stride(0); in.node_stride = zp.stride(1);
    in.parent = (const int32_t *)parent.data_ptr(); in.topo_seq_stride = parent.dim() == 1 ? 0 : N;
    in.token = (const int32_t *)token.data_ptr();
    in.temperature = (float)number(a[6]); in.top_k = truncated(a[7]); in.top_p = (float)number(a[8]);
    in.temperature_per_seq = (const float *)pointer_or_null(a[9], "temperature_per_seq");
    in.u_accept = (const float *)ua.data_ptr(); in.u_bonus = (const float *)ub.data_ptr();
    return in;
}

template <typename F> PyObject *guarded(F f)
{
    try {
        return f();
    } catch (const Raised &) {
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
bool arity(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
    return false;
}

// an object of one of the result classes from n tensors (undefined ones: None)
PyObject *result(PyObject *cls, const at::Tensor *t, int n)
{
    PyObject *args[10];
    int made = 0;
    for (; made < n; ++made) {
        args[made] = t[made].defined() ? THPVariable_Wrap(t[made]) : Py_NewRef(Py_None);
        if (!args[made]) break;
    }
    PyObject *r = made == n ? PyObject_Vectorcall(cls, args, n, nullptr) : nullptr;
    while (made > 0) Py_DECREF(args[--made]);
    if (!r) throw Raised{};
    return r;
}

// verify(code, <10 batch arguments>, outputs, workspace, stream, flags): code 0 SpecInfer, 1 Traversal, 2 + s the walk with
// OTLP solver s; flags: optional outputs to allocate, bit i for output 5 + i
PyObject *py_verify(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 15)) return nullptr;
    return guarded([&]() -> PyObject * {
        const int code = (int)integer(a[0]), flags = (int)integer(a[14]);
        const SpecIn in = spec_in(a + 1);
        int64_t bytes = 0;
        check(lib.workspace_bytes(&in, &bytes), "spec_workspace_bytes");
        const Scratch ws = scratch_of(a[12], bytes);
        PyObject *given = a[11];
        at::Tensor t[10];
        void *p[10] = {};
        if (given == Py_None) {
            const at::Device dev = THPVariable_Unpack(a[1]).device();
            const int64_t B = in.B, N = in.N;
            for (int i = 0; i < 5; ++i) t[i] = i == 2 ? empty({B, N}, at::kInt, dev) : empty({B}, at::kInt, dev);
            if (flags & 1) t[5] = empty({B, (int64_t)in.V}, at::kFloat, dev);
            if (flags & 2) t[6] = empty({B, N}, at::kFloat, dev);
            if (flags & 4) t[7] = empty({B, N}, at::kFloat, dev);
            if (flags & 8) t[8] = empty({B, N, 4}, at::kFloat, dev);
            if (flags & 16) t[9] = empty({B, N + 1}, at::kFloat, dev);
            for (int i = 0; i < 10; ++i) if (t[i].defined()) p[i] = t[i].data_ptr();
        } else {
            for (int i = 0; i < 10; ++i) {
                const Owned o(PyObject_GetAttr(given, n_out[i]));
                if (!o.o) throw Raised{};
                if (o.o == Py_None) continue;
                t[i] = tensor(o.o, OUT_NAMES[i]);          // (held until the call has been enqueued: the attribute may be computed)
                p[i] = t[i].data_ptr();
            }
        }
        const SpecOut out = {(int32_t *)p[0], (int32_t *)p[1], (int32_t *)p[2], (int32_t *)p[3], (int32_t *)p[4],
                             (float *)p[5], (float *)p[6], (float *)p[7], (float *)p[8], (float *)p[9]};
        void *st = stream_of(a[13]);
        const int rc = unlocked([&] {
            return code == 0   ? lib.specinfer(&in, &out, ws.ptr, ws.bytes, st)
                   : code == 1 ? lib.traversal(&in, &out, ws.ptr, ws.bytes, st)
                               : lib.otlp(&in, &out, code - 2, ws.ptr, ws.bytes, st);
        });
        check(rc, code == 0 ? "spec_verify_specinfer" : code == 1 ? "spec_verify_traversal" : "spec_verify_otlp");
        return given == Py_None ? result(verify_outputs_class, t, 10) : Py_NewRef(given);
    });
}

// tree_analysis(<10 batch arguments>, workspace, stream)
PyObject *py_analysis(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 12)) return nullptr;
    return guarded([&]() -> PyObject * {
        const SpecIn in = spec_in(a);
        const at::Device dev = THPVariable_Unpack(a[0]).device();
        const int64_t B = in.B, N = in.N;
        at::Tensor t[5] = {empty({B, N, 4}, at::kFloat, dev), empty({B, N, 3}, at::kFloat, dev), empty({5, B, N}, at::kFloat, dev),
                           empty({5, B, N}, at::kFloat, dev), empty({5, B}, at::kFloat, dev)};
        int64_t bytes = 0;
        check(lib.analysis_workspace_bytes(&in, &bytes), "spec_analysis_workspace_bytes");
        const Scratch ws = scratch_of(a[10], bytes);
        const SpecAnalysisOut out = {(float *)t[0].data_ptr(), (float *)t[1].data_ptr(), (float *)t[2].data_ptr(),
                                     (float *)t[3].data_ptr(), (float *)t[4].data_ptr()};
        void *st = stream_of(a[11]);
        check(unlocked([&] { return lib.analysis(&in, &out, ws.ptr, ws.bytes, st); }), "spec_tree_analysis");
        return result(analysis_outputs_class, t, 5);
    });
}

// tree_probs(logits, which, temperature, top_k, top_p, temperature_per_seq, want_probs, want_stats, workspace, stream)
PyObject *py_probs(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 10)) return nullptr;
    return guarded([&]() -> PyObject * {
        const at::Tensor &z = cuda_tensor(a[0], "logits");
        const auto dt = z.scalar_type();
        if (z.dim() != 3 || z.stride(2) != 1 || (dt != at::kFloat && dt != at::kBFloat16))
            raise("logits must be [B,N,V] float32 / bfloat16 with a contiguous vocabulary axis");
        const int64_t B = z.size(0), N = z.size(1), V = z.size(2);
        SpecIn in = {};
        in.B = (int32_t)B; in.N = (int32_t)N; in.V = (int32_t)V;
        in.logits_dtype = dt == at::kFloat ? SPEC_F32 : SPEC_BF16;
        in.target_logits = in.draft_logits = z.data_ptr();
        in.seq_stride = z.stride(0); in.node_stride = z.stride(1);
        in.temperature = (float)number(a[2]); in.top_k = truncated(a[3]); in.top_p = (float)number(a[4]);
        in.temperature_per_seq = (const float *)pointer_or_null(a[5], "temperature_per_seq");
        at::Tensor probs, stats;
        if (PyObject_IsTrue(a[6])) probs = empty({B, N, V}, at::kFloat, z.device());
        if (PyObject_IsTrue(a[7])) stats = empty({B, N, 6}, at::kFloat, z.device());
        int64_t bytes = 0;
        check(lib.workspace_bytes(&in, &bytes), "spec_workspace_bytes");
        const Scratch ws = scratch_of(a[8], bytes);        // holds the rows' records when truncating
        const int which = truncated(a[1]);
        float *pr = probs.defined() ? (float *)probs.data_ptr() : nullptr, *st = stats.defined() ? (float *)stats.data_ptr() : nullptr;
        void *stream = stream_of(a[9]);
        check(unlocked([&] { return lib.probs(&in, which, pr, st, ws.ptr, ws.bytes, stream); }), "spec_tree_probs");
        PyObject *p = probs.defined() ? THPVariable_Wrap(probs) : Py_NewRef(Py_None);
        PyObject *s = stats.defined() ? THPVariable_Wrap(stats) : Py_NewRef(Py_None);
        PyObject *r = p && s ? PyTuple_Pack(2, p, s) : nullptr;
        Py_XDECREF(p);
        Py_XDECREF(s);
        return r;
    });
}

// sample_bonus(weights, u, want_margin, stream)
PyObject *py_bonus(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 4)) return nullptr;
    return guarded([&]() -> PyObject * {
        const at::Tensor &w = cuda_tensor(a[0], "weights"), &u = cuda_tensor(a[1], "u");
        if (w.scalar_type() != at::kFloat || !w.is_contiguous() || w.dim() != 2) raise("weights must be a contiguous [R,V] float32 tensor");
        if (u.scalar_type() != at::kFloat || !u.is_contiguous() || u.numel() != w.size(0))
            raise("u must be a contiguous float32 tensor with one entry per row");
        const bool want = PyObject_IsTrue(a[2]);
        at::Tensor token = empty({w.size(0)}, at::kInt, w.device()), margin;
        if (want) margin = empty({w.size(0)}, at::kFloat, w.device());
        const float *wp = (const float *)w.data_ptr(), *up = (const float *)u.data_ptr();
        const int32_t R = (int32_t)w.size(0), V = (int32_t)w.size(1);
        int32_t *tp = (int32_t *)token.data_ptr();
        float *mp = want ? (float *)margin.data_ptr() : nullptr;
        void *st = stream_of(a[3]);
        check(unlocked([&] { return lib.bonus(wp, R, V, up, tp, mp, nullptr, 0, st); }), "spec_sample_bonus");
        PyObject *t = THPVariable_Wrap(token);
        if (!want || !t) return t;
        PyObject *m = THPVariable_Wrap(margin), *r = m ? PyTuple_Pack(2, t, m) : nullptr;
        Py_DECREF(t);
        Py_XDECREF(m);
        return r;
    });
}

// launch(code, SpecIn address, SpecOut address, workspace address, workspace bytes, stream): one of the two verifiers on
// structures that the caller has filled and keeps
PyObject *py_launch(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 6)) return nullptr;
    return guarded([&]() -> PyObject * {
        const auto at_ = [&](int i) { return (void *)(intptr_t)integer(a[i]); };
        const bool traversal = integer(a[0]) != 0;
        const SpecIn *in = (const SpecIn *)at_(1);
        const SpecOut *out = (const SpecOut *)at_(2);
        void *ws = at_(3), *st = stream_of(a[5]);
        const int64_t bytes = integer(a[4]);
        check(unlocked([&] { return (traversal ? lib.traversal : lib.specinfer)(in, out, ws, bytes, st); }),
              traversal ? "spec_verify_traversal" : "spec_verify_specinfer");
        Py_RETURN_NONE;
    });
}

// init(path of libspecverify.so, VerifyOutputs, AnalysisOutputs)
PyObject *py_init(PyObject *, PyObject *args)
{
    const char *path;
    PyObject *v, *an;
    if (!PyArg_ParseTuple(args, "sOO", &path, &v, &an)) return nullptr;
    void *h = dlopen(path, RTLD_NOW | RTLD_LOCAL);
    if (!h) return PyErr_Format(PyExc_RuntimeError, "%s", dlerror());
    bool ok = true;
    const auto find = [&](auto &f, const char *name) {
        f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(dlsym(h, name));
        ok = ok && f;
    };
    find(lib.workspace_bytes, "spec_workspace_bytes");
    find(lib.analysis_workspace_bytes, "spec_analysis_workspace_bytes");
    find(lib.specinfer, "spec_verify_specinfer");
    find(lib.traversal, "spec_verify_traversal");
    find(lib.otlp, "spec_verify_otlp");
    find(lib.analysis, "spec_tree_analysis");
    find(lib.probs, "spec_tree_probs");
    find(lib.bonus, "spec_sample_bonus");
    if (!ok) return PyErr_Format(PyExc_RuntimeError, "%s lacks an entry point", path);
    verify_outputs_class = Py_NewRef(v);
    analysis_outputs_class = Py_NewRef(an);
    n_buf = PyUnicode_InternFromString("buf");
    n_get = PyUnicode_InternFromString("get");
    n_stream = PyUnicode_InternFromString("cuda_stream");
    for (int i = 0; i < 10; ++i) n_out[i] = PyUnicode_InternFromString(OUT_NAMES[i]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"init", py_init, METH_VARARGS, nullptr},
    {"verify", (PyCFunction)(void *)py_verify, METH_FASTCALL, nullptr},
    {"tree_analysis", (PyCFunction)(void *)py_analysis, METH_FASTCALL, nullptr},
    {"tree_probs", (PyCFunction)(void *)py_probs, METH_FASTCALL, nullptr},
    {"sample_bonus", (PyCFunction)(void *)py_bonus, METH_FASTCALL, nullptr},
    {"launch", (PyCFunction)(void *)py_launch, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_torch_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_calls(void) { return PyModule_Create(&module_def); }
