// Python front end of the C ABI: reads tensors (shape, strides, data pointer) and calls libdssd.so.
//
// A round of a small batch takes about 10 us on the GPU, and marshalling one call in Python through
// ctypes took about 8 us of host time, so the calls of a serving loop were bound by it.  Here a call costs
// well under 1 us besides the launches.  Nothing is computed and nothing allocated: every function
// takes the caller's tensors and hands pointers on.  binding.py holds the entry points with their
// arguments, defaults and allocations.
#include <Python.h>

#include <dlfcn.h>

#include <vector>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "dssd.h"

namespace {

// ---- the library's entry points, resolved from the handle that binding.py loaded ----
#define DSSD_CALLS(X)                                                                                         \
    X(dssd_edge_verify) X(dssd_edge_verify_p16) X(dssd_device_resample) X(dssd_device_resample_p16)           \
    X(dssd_device_resample_static) X(dssd_device_resample_rejected) X(dssd_edge_verify_topk)                  \
    X(dssd_device_resample_topk) X(dssd_dsd_verify) X(dssd_edge_verify_bonus) X(dssd_round_host)              \
    X(dssd_round_host_topk) X(dssd_edge_partial) X(dssd_edge_combine) X(dssd_edge_emit_shard)                 \
    X(dssd_resample_shard_mass) X(dssd_resample_shard_draw)
struct Calls {
#define X(name) decltype(&::name) name;
    DSSD_CALLS(X)
#undef X
} lib;

struct Raised {};  // a Python exception has been set

[[noreturn]] void raise(PyObject *type, const char *text)
{
    PyErr_SetString(type, text);
    throw Raised();
}

void require(bool ok, const char *text)
{
    if (!ok) raise(PyExc_AssertionError, text);
}

const at::Tensor &tensor(PyObject *o)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a tensor");
    return THPVariable_Unpack(o);
}

// None and empty tensors are NULL
void *ptr(PyObject *o)
{
    if (o == nullptr || o == Py_None) return nullptr;
    const at::Tensor &t = tensor(o);
    return t.numel() ? t.data_ptr() : nullptr;
}
template <class T>
T *ptr_as(PyObject *o)
{
    return static_cast<T *>(ptr(o));
}

// References that a mapping other than a dict gave out, kept until the call that asked for them returns.
thread_local std::vector<PyObject *> kept;
PyObject *keep(PyObject *v)
{
    if (v == nullptr) throw Raised();
    kept.push_back(v);
    return v;
}

// out["name"]; a missing key is an error
PyObject *item(PyObject *out, const char *name)
{
    if (!PyDict_CheckExact(out)) return keep(PyMapping_GetItemString(out, name));
    PyObject *v = PyDict_GetItemString(out, name);
    if (v == nullptr) {
        PyErr_SetString(PyExc_KeyError, name);
        throw Raised();
    }
    return v;
}
template <class T>
T *need(PyObject *out, const char *name)
{
    return static_cast<T *>(tensor(item(out, name)).data_ptr());
}
// out.get("name"): NULL where there is none
template <class T>
T *maybe(PyObject *out, const char *name)
{
    return ptr_as<T>(PyDict_CheckExact(out) ? PyDict_GetItemString(out, name) : keep(PyObject_CallMethod(out, "get", "s", name)));
}

double number(PyObject *o)
{
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) throw Raised();
    return x;
}
long integer(PyObject *o)
{
    const long x = PyLong_AsLong(o);
    if (x == -1 && PyErr_Occurred()) throw Raised();
    return x;
}
int size_arg(PyObject *o) { return (int)integer(o); }

// None: torch's current stream; else a torch stream, or a cudaStream_t as an integer or an object that converts to one
void *stream(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_Check(o)) return PyLong_AsVoidPtr(o);
    PyObject *h = PyObject_HasAttrString(o, "cuda_stream") ? PyObject_GetAttrString(o, "cuda_stream") : PyNumber_Long(o);
    if (h == nullptr) throw Raised();
    void *s = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (PyErr_Occurred()) throw Raised();
    return s;
}

dssd_dtype dtype_code(const at::Tensor &t)
{
    if (t.scalar_type() == at::kBFloat16) return DSSD_BF16;
    if (t.scalar_type() == at::kFloat) return DSSD_F32;
    raise(PyExc_TypeError, "target_logits must be float32 or bfloat16");
}

// a [B, gamma+1, V] tensor with unit stride along V and equally spaced rows
struct Rows {
    const void *data;
    dssd_dtype dtype;
    int64_t stride;
    int B, gamma, V;
};
int64_t row_stride(const at::Tensor &t, const char *what)
{
    const int64_t B = t.size(0), n = t.size(1), V = t.size(2);
    const int64_t s = n > 1 ? t.stride(1) : (V > t.stride(0) ? V : t.stride(0));
    if (B > 1 && t.stride(0) != n * s) raise(PyExc_ValueError, what);
    return s;
}
Rows rows(PyObject *o, bool cuda = true)
{
    const at::Tensor &t = tensor(o);
    require(t.is_cuda() == cuda && t.dim() == 3, "target_logits must be a [B, gamma+1, V] tensor on the right device");
    require(t.stride(2) == 1 || t.size(2) == 1, "target_logits must have unit stride along V");
    Rows r;
    r.B = (int)t.size(0);
    r.gamma = (int)t.size(1) - 1;
    r.V = (int)t.size(2);
    if (cuda) r.stride = row_stride(t, "rows of target_logits must be equally spaced");
    else require(t.is_contiguous(), "target_logits must be contiguous");
    r.dtype = dtype_code(t);
    r.data = t.data_ptr();
    return r;
}

const float *draft_rows(PyObject *o, int64_t B, int64_t gamma, int64_t V)
{
    if (gamma <= 0) return nullptr;
    const at::Tensor &q = tensor(o);
    require(q.is_contiguous() && q.scalar_type() == at::kFloat && q.numel() == B * gamma * V,
            "draft_q must be a contiguous float32 [B, gamma, V] tensor");
    return q.numel() ? static_cast<const float *>(q.data_ptr()) : nullptr;
}

struct Space {
    void *data;
    size_t bytes;
};
Space space(PyObject *o)
{
    const at::Tensor &t = tensor(o);
    return {t.data_ptr(), (size_t)t.numel()};
}

// elements between rows of a [B, V] float32 tensor with unit stride along V
int64_t rows_2d(const at::Tensor &t)
{
    require(t.is_cuda() && t.dim() == 2 && t.scalar_type() == at::kFloat && (t.stride(1) == 1 || t.size(1) == 1),
            "rows must be a float32 [B, V] CUDA tensor with unit stride along V");
    return t.size(0) > 1 ? (t.size(1) > t.stride(0) ? t.size(1) : t.stride(0)) : t.size(1);
}

struct QShard {
    const float *data;
    int64_t stride;
};
QShard q_shard(PyObject *o, int64_t B, int64_t gamma, int64_t Vs)
{
    if (gamma == 0 || o == Py_None) return {nullptr, Vs};
    const at::Tensor &q = tensor(o);
    require(q.is_cuda() && q.scalar_type() == at::kFloat && q.dim() == 3 && q.size(0) == B && q.size(1) == gamma &&
                q.size(2) == Vs && (q.stride(2) == 1 || Vs == 1),
            "draft_q_shard must be a float32 [B, gamma, V_shard] CUDA tensor with unit stride along V");
    return {q.numel() ? static_cast<const float *>(q.data_ptr()) : nullptr, row_stride(q, "rows of draft_q_shard must be equally spaced")};
}

// The library's call without the interpreter lock, once every argument has been read: a round on host buffers waits for
// the GPU and copies from pageable memory, and any launch waits while the stream's queue is full.  Other threads run
// meanwhile, a host callback on the stream among them.
template <class... P, class... A>
dssd_status call(dssd_status (*fn)(P...), A... args)
{
    PyThreadState *const state = PyEval_SaveThread();
    const dssd_status st = fn(args...);
    PyEval_RestoreThread(state);
    return st;
}

// ---- one function per entry point: (arguments ...) -> status -----------------------------------

// target_logits, draft_tokens, draft_q_tok, uniforms, temperature, out, workspace, stream, half
dssd_status edge_verify(PyObject *const *a)
{
    const Rows r = rows(a[0]);
    const bool half = PyObject_IsTrue(a[8]) == 1;
    const at::Tensor &p = tensor(item(a[5], "p_row"));
    require(p.scalar_type() == (half ? at::kHalf : at::kFloat), "out[\"p_row\"] must have the payload's type");
    const Space ws = space(a[6]);
    const int32_t *tok = ptr_as<const int32_t>(a[1]);
    const float *q = ptr_as<const float>(a[2]), *u = ptr_as<const float>(a[3]);
    const float T = (float)number(a[4]);
    int32_t *n = need<int32_t>(a[5], "accept_len");
    float *pt = maybe<float>(a[5], "p_tok"), *lse = maybe<float>(a[5], "lse");
    uint32_t *fl = maybe<uint32_t>(a[5], "flags");
    void *s = stream(a[7]);
    if (half)
        return call(lib.dssd_edge_verify_p16, r.data, r.dtype, r.stride, tok, q, u, T, r.B, r.gamma, r.V, n,
                                        static_cast<uint16_t *>(p.data_ptr()), pt, lse, fl, ws.data, ws.bytes, s);
    return call(lib.dssd_edge_verify, r.data, r.dtype, r.stride, tok, q, u, T, r.B, r.gamma, r.V, n,
                                static_cast<float *>(p.data_ptr()), pt, lse, fl, ws.data, ws.bytes, s);
}

const at::Tensor &payload(PyObject *o, bool half_too)
{
    const at::Tensor &p = tensor(o);
    require(p.is_cuda() && p.dim() == 2 && p.is_contiguous() &&
                (p.scalar_type() == at::kFloat || (half_too && p.scalar_type() == at::kHalf)),
            "p_row must be a contiguous [B, V] CUDA tensor of the payload's type");
    return p;
}

// p_row, draft_q, accept_len, uniforms_rs, gamma, out, workspace, stream
dssd_status device_resample(PyObject *const *a)
{
    const at::Tensor &p = payload(a[0], true);
    const int B = (int)p.size(0), V = (int)p.size(1), gamma = size_arg(a[4]);
    const float *q = draft_rows(a[1], B, gamma, V);
    const Space ws = space(a[6]);
    const int32_t *n = static_cast<const int32_t *>(tensor(a[2]).data_ptr());
    const float *u = static_cast<const float *>(tensor(a[3]).data_ptr());
    int32_t *tok = need<int32_t>(a[5], "token");
    uint32_t *fl = maybe<uint32_t>(a[5], "flags");
    void *s = stream(a[7]);
    if (p.scalar_type() == at::kHalf)
        return call(lib.dssd_device_resample_p16, static_cast<const uint16_t *>(p.data_ptr()), q, n, u, B, gamma, V, tok, fl, ws.data,
                                            ws.bytes, s);
    return call(lib.dssd_device_resample, static_cast<const float *>(p.data_ptr()), q, n, u, B, gamma, V, tok, fl, ws.data, ws.bytes, s);
}

// the same for the rejected sequences only
dssd_status device_resample_rejected(PyObject *const *a)
{
    const at::Tensor &p = payload(a[0], false);
    const int B = (int)p.size(0), V = (int)p.size(1), gamma = size_arg(a[4]);
    const float *q = draft_rows(a[1], B, gamma, V);
    const Space ws = space(a[6]);
    return call(lib.dssd_device_resample_rejected, static_cast<const float *>(p.data_ptr()), q,
                                             static_cast<const int32_t *>(tensor(a[2]).data_ptr()),
                                             static_cast<const float *>(tensor(a[3]).data_ptr()), B, gamma, V,
                                             need<int32_t>(a[5], "token"), maybe<uint32_t>(a[5], "flags"), ws.data, ws.bytes,
                                             stream(a[7]));
}

// p_row, draft_q, accept_len, uniforms_rs, gamma, out, stream
dssd_status device_resample_static(PyObject *const *a)
{
    const at::Tensor &p = payload(a[0], false);
    const int B = (int)p.size(0), V = (int)p.size(1), gamma = size_arg(a[4]);
    return call(lib.dssd_device_resample_static, static_cast<const float *>(p.data_ptr()), gamma > 0 ? ptr_as<const float>(a[1]) : nullptr,
                                           static_cast<const int32_t *>(tensor(a[2]).data_ptr()),
                                           static_cast<const float *>(tensor(a[3]).data_ptr()), B, gamma, V,
                                           need<int32_t>(a[5], "token"), maybe<uint32_t>(a[5], "flags"), stream(a[6]));
}

// target_logits, draft_tokens, draft_q_tok, uniforms, temperature, k, out, workspace, stream
dssd_status edge_verify_topk(PyObject *const *a)
{
    const Rows r = rows(a[0]);
    const Space ws = space(a[7]);
    return call(lib.dssd_edge_verify_topk, r.data, r.dtype, r.stride, ptr_as<const int32_t>(a[1]), ptr_as<const float>(a[2]),
                                     ptr_as<const float>(a[3]), (float)number(a[4]), r.B, r.gamma, r.V, size_arg(a[5]),
                                     need<int32_t>(a[6], "accept_len"), need<int32_t>(a[6], "p_idx"), need<float>(a[6], "p_val"),
                                     maybe<float>(a[6], "p_tok"), maybe<uint32_t>(a[6], "flags"), ws.data, ws.bytes, stream(a[8]));
}

// p_idx, p_val, q_idx, q_val, accept_len, uniforms_rs, gamma, out, stream
dssd_status device_resample_topk(PyObject *const *a)
{
    const at::Tensor &pi = tensor(a[0]), &pv = tensor(a[1]);
    require(pi.is_cuda() && pi.dim() == 2 && pi.is_contiguous() && pi.scalar_type() == at::kInt && pv.is_contiguous() &&
                pv.scalar_type() == at::kFloat && pv.sizes() == pi.sizes(),
            "p_idx (int32) and p_val (float32) must be contiguous [B, k] CUDA tensors");
    const int B = (int)pi.size(0), k = (int)pi.size(1), gamma = size_arg(a[6]);
    const int32_t *qi = nullptr;
    const float *qv = nullptr;
    if (gamma > 0) {
        const at::Tensor &ti = tensor(a[2]), &tv = tensor(a[3]);
        const int64_t want = (int64_t)B * gamma * k;
        require(ti.is_contiguous() && ti.scalar_type() == at::kInt && ti.numel() == want && tv.is_contiguous() &&
                    tv.scalar_type() == at::kFloat && tv.numel() == want,
                "q_idx (int32) and q_val (float32) must be contiguous [B, gamma, k] tensors");
        qi = ptr_as<const int32_t>(a[2]);
        qv = ptr_as<const float>(a[3]);
    }
    return call(lib.dssd_device_resample_topk, static_cast<const int32_t *>(pi.data_ptr()), static_cast<const float *>(pv.data_ptr()), qi, qv,
                                         static_cast<const int32_t *>(tensor(a[4]).data_ptr()),
                                         static_cast<const float *>(tensor(a[5]).data_ptr()), B, gamma, k,
                                         need<int32_t>(a[7], "token"), maybe<uint32_t>(a[7], "flags"), stream(a[8]));
}

// target_logits, draft_q, draft_tokens, uniforms, uniforms_rs, temperature, out, workspace, stream
dssd_status dsd_verify(PyObject *const *a)
{
    const Rows r = rows(a[0]);
    const float *q = draft_rows(a[1], r.B, r.gamma, r.V);
    const Space ws = space(a[7]);
    return call(lib.dssd_dsd_verify, r.data, r.dtype, r.stride, q, ptr_as<const int32_t>(a[2]), ptr_as<const float>(a[3]),
                               static_cast<const float *>(tensor(a[4]).data_ptr()), (float)number(a[5]), r.B, r.gamma, r.V,
                               need<int32_t>(a[6], "accept_len"), need<int32_t>(a[6], "token"),
                               maybe<uint32_t>(a[6], "edge_flags"), maybe<uint32_t>(a[6], "rs_flags"), ws.data, ws.bytes,
                               stream(a[8]));
}

// target_logits, draft_tokens, draft_q_tok, uniforms, uniforms_bonus, temperature, out, workspace, stream
dssd_status edge_verify_bonus(PyObject *const *a)
{
    const Rows r = rows(a[0]);
    const Space ws = space(a[7]);
    return call(lib.dssd_edge_verify_bonus, r.data, r.dtype, r.stride, ptr_as<const int32_t>(a[1]), ptr_as<const float>(a[2]),
                                      ptr_as<const float>(a[3]), static_cast<const float *>(tensor(a[4]).data_ptr()),
                                      (float)number(a[5]), r.B, r.gamma, r.V, need<int32_t>(a[6], "accept_len"),
                                      need<float>(a[6], "p_row"), need<int32_t>(a[6], "token"), maybe<float>(a[6], "p_tok"),
                                      maybe<float>(a[6], "lse"), maybe<uint32_t>(a[6], "flags"),
                                      maybe<uint32_t>(a[6], "token_flags"), ws.data, ws.bytes, stream(a[8]));
}

// host dict, temperature, arena, out, stream
dssd_status round_host(PyObject *const *a)
{
    const Rows r = rows(item(a[0], "target_logits"), false);
    const Space ar = space(a[2]);
    return call(lib.dssd_round_host, r.data, r.dtype, maybe<const int32_t>(a[0], "draft_tokens"), maybe<const float>(a[0], "draft_q_tok"),
                               maybe<const float>(a[0], "uniforms"), maybe<const float>(a[0], "draft_q"),
                               need<const float>(a[0], "uniforms_rs"), (float)number(a[1]), r.B, r.gamma, r.V,
                               need<int32_t>(a[3], "accept_len"), need<int32_t>(a[3], "token"),
                               maybe<uint32_t>(a[3], "edge_flags"), maybe<uint32_t>(a[3], "rs_flags"), maybe<float>(a[3], "p_row"),
                               ar.data, ar.bytes, stream(a[4]));
}

// host dict, temperature, k, arena, out, stream
dssd_status round_host_topk(PyObject *const *a)
{
    const Rows r = rows(item(a[0], "target_logits"), false);
    const Space ar = space(a[3]);
    return call(lib.dssd_round_host_topk, r.data, r.dtype, maybe<const int32_t>(a[0], "draft_tokens"),
                                    maybe<const float>(a[0], "draft_q_tok"), maybe<const float>(a[0], "uniforms"),
                                    maybe<const int32_t>(a[0], "q_idx"), maybe<const float>(a[0], "q_val"),
                                    need<const float>(a[0], "uniforms_rs"), (float)number(a[1]), r.B, r.gamma, r.V, size_arg(a[2]),
                                    need<int32_t>(a[4], "accept_len"), need<int32_t>(a[4], "token"),
                                    maybe<uint32_t>(a[4], "edge_flags"), maybe<uint32_t>(a[4], "rs_flags"),
                                    maybe<int32_t>(a[4], "p_idx"), maybe<float>(a[4], "p_val"), ar.data, ar.bytes, stream(a[5]));
}

// logits_shard, draft_tokens, v_begin, temperature, out, workspace, stream
dssd_status edge_partial(PyObject *const *a)
{
    const Rows r = rows(a[0]);
    const Space ws = space(a[5]);
    return call(lib.dssd_edge_partial, r.data, r.dtype, r.stride, ptr_as<const int32_t>(a[1]), size_arg(a[2]), (float)number(a[3]), r.B,
                                 r.gamma, r.V, need<float>(a[4], "part_ref"), need<double>(a[4], "part_sum"),
                                 ptr_as<float>(item(a[4], "tok_logit")), ws.data, ws.bytes, stream(a[6]));
}

// part_ref, part_sum, tok_logit, draft_tokens, draft_q_tok, uniforms, temperature, V, out, stream
dssd_status edge_combine(PyObject *const *a)
{
    const at::Tensor &pr = tensor(a[0]), &ps = tensor(a[1]), &tl = tensor(a[2]);
    require(pr.is_cuda() && pr.dim() == 3 && pr.is_contiguous() && pr.scalar_type() == at::kFloat,
            "part_ref must be a contiguous float32 [G, B, gamma+1] CUDA tensor");
    require(ps.sizes() == pr.sizes() && ps.is_contiguous() && ps.scalar_type() == at::kDouble,
            "part_sum must be a contiguous float64 tensor of part_ref's shape");
    const int G = (int)pr.size(0), B = (int)pr.size(1), gamma = (int)pr.size(2) - 1;
    require(tl.is_contiguous() && tl.scalar_type() == at::kFloat && tl.numel() == (int64_t)G * B * gamma,
            "tok_logit must be a contiguous float32 [G, B, gamma] tensor");
    return call(lib.dssd_edge_combine, static_cast<const float *>(pr.data_ptr()), static_cast<const double *>(ps.data_ptr()),
                                 ptr_as<const float>(a[2]), G, ptr_as<const int32_t>(a[3]), ptr_as<const float>(a[4]),
                                 ptr_as<const float>(a[5]), (float)number(a[6]), B, gamma, size_arg(a[7]),
                                 need<int32_t>(a[8], "accept_len"), need<float>(a[8], "row_scale"), maybe<float>(a[8], "p_tok"),
                                 maybe<float>(a[8], "lse"), maybe<uint32_t>(a[8], "flags"), stream(a[9]));
}

// logits_shard, accept_len, row_scale, temperature, out tensor, stream
dssd_status edge_emit_shard(PyObject *const *a)
{
    const Rows r = rows(a[0]);
    const at::Tensor &o = tensor(a[4]);
    require(o.dim() == 2 && o.size(0) == r.B && o.size(1) == r.V, "out must be a [B, V_shard] tensor");
    return call(lib.dssd_edge_emit_shard, r.data, r.dtype, r.stride, static_cast<const int32_t *>(tensor(a[1]).data_ptr()),
                                    static_cast<const float *>(tensor(a[2]).data_ptr()), (float)number(a[3]), r.B, r.gamma, r.V,
                                    static_cast<float *>(o.data_ptr()), rows_2d(o), stream(a[5]));
}

// p_row_shard, draft_q_shard, accept_len, gamma, out tensor, workspace, stream
dssd_status resample_shard_mass(PyObject *const *a)
{
    const at::Tensor &p = tensor(a[0]);
    const int64_t ps = rows_2d(p);
    const int B = (int)p.size(0), Vs = (int)p.size(1), gamma = size_arg(a[3]);
    const QShard q = q_shard(a[1], B, gamma, Vs);
    const Space ws = space(a[5]);
    return call(lib.dssd_resample_shard_mass, static_cast<const float *>(p.data_ptr()), ps, q.data, q.stride,
                                        static_cast<const int32_t *>(tensor(a[2]).data_ptr()), B, gamma, Vs,
                                        static_cast<double *>(tensor(a[4]).data_ptr()), ws.data, ws.bytes, stream(a[6]));
}

// masses, g, v_begin, p_row_shard, draft_q_shard, accept_len, uniforms_rs, gamma, workspace, out, stream
dssd_status resample_shard_draw(PyObject *const *a)
{
    const at::Tensor &m = tensor(a[0]), &p = tensor(a[3]);
    require(m.is_cuda() && m.dim() == 3 && m.is_contiguous() && m.scalar_type() == at::kDouble,
            "masses must be a contiguous float64 [G, B, 2] CUDA tensor");
    const int64_t ps = rows_2d(p);
    const int B = (int)p.size(0), Vs = (int)p.size(1), gamma = size_arg(a[7]);
    const QShard q = q_shard(a[4], B, gamma, Vs);
    const Space ws = space(a[8]);
    return call(lib.dssd_resample_shard_draw, static_cast<const double *>(m.data_ptr()), (int)m.size(0), size_arg(a[1]), size_arg(a[2]),
                                        static_cast<const float *>(p.data_ptr()), ps, q.data, q.stride,
                                        static_cast<const int32_t *>(tensor(a[5]).data_ptr()),
                                        static_cast<const float *>(tensor(a[6]).data_ptr()), B, gamma, Vs,
                                        need<int32_t>(a[9], "token"), maybe<uint32_t>(a[9], "flags"), ws.data, ws.bytes,
                                        stream(a[10]));
}

// ---- glue -----------------------------------------------------------------------------------

template <dssd_status (*fn)(PyObject *const *), Py_ssize_t kArgs>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != kArgs) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", kArgs, n);
        return nullptr;
    }
    const size_t before = kept.size();
    PyObject *result = nullptr;
    try {
        result = PyLong_FromLong(fn(args));
    } catch (const Raised &) {
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    while (kept.size() > before) {  // (after an error too: the references' owners may run Python code of their own)
        PyObject *type, *value, *trace;
        PyErr_Fetch(&type, &value, &trace);
        PyObject *v = kept.back();
        kept.pop_back();
        Py_DECREF(v);
        PyErr_Restore(type, value, trace);
    }
    return result;
}

// the handle that dlopen gave for libdssd.so
PyObject *bind(PyObject *, PyObject *arg)
{
    void *handle = PyLong_AsVoidPtr(arg);
    if (PyErr_Occurred()) return nullptr;
    Calls c;
#define X(name)                                                          \
    c.name = reinterpret_cast<decltype(c.name)>(dlsym(handle, #name));   \
    if (!c.name) {                                                       \
        PyErr_SetString(PyExc_ImportError, "libdssd.so lacks " #name);   \
        return nullptr;                                                  \
    }
    DSSD_CALLS(X)
#undef X
    lib = c;
    Py_RETURN_NONE;
}

#define ENTRY(name, n) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<name, n>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    ENTRY(edge_verify, 9),
    ENTRY(device_resample, 8),
    ENTRY(device_resample_rejected, 8),
    ENTRY(device_resample_static, 7),
    ENTRY(edge_verify_topk, 9),
    ENTRY(device_resample_topk, 9),
    ENTRY(dsd_verify, 9),
    ENTRY(edge_verify_bonus, 9),
    ENTRY(round_host, 5),
    ENTRY(round_host_topk, 6),
    ENTRY(edge_partial, 7),
    ENTRY(edge_combine, 10),
    ENTRY(edge_emit_shard, 6),
    ENTRY(resample_shard_mass, 7),
    ENTRY(resample_shard_draw, 11),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
