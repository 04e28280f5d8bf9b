// Python-side argument marshalling of the calls that a serving loop makes step after step: tensors in, the C ABI of
// include/l4l.h out, nothing kept. A small call (one decode step of one user, a short prompt) is bound by its host side:
// reading some thirty tensor attributes from Python and building ctypes structures took two thirds of it. Host time per
// call through ctypes and here: a prompt of 128 tokens 21.1 and 5.2 us, one user's rope-fused step 26.8 and 5.8 us (3 us
// of either are the launch). Each function returns the library's status; the Python wrappers, which hold the signatures
// and the documentation, turn it into an exception.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <c10/cuda/CUDAStream.h>

#include "../../include/l4l.h"

namespace {

using at::Tensor;

[[noreturn]] void type_error(const std::string &what) { TORCH_CHECK_TYPE(false, what); throw 0; }
[[noreturn]] void value_error(const std::string &what) { TORCH_CHECK_VALUE(false, what); throw 0; }

const Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) type_error(std::string(name) + " must be a tensor");
    return THPVariable_Unpack(o);
}
bool is_none(PyObject *o) { return o == nullptr || o == Py_None; }

int as_int(PyObject *o)                                          // int(o), narrowed as a ctypes call narrows it
{
    THPObjectPtr n(PyNumber_Long(o));
    if (!n) throw python_error();
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(n.get());
    if (PyErr_Occurred()) throw python_error();
    return (int)v;
}
float as_float(PyObject *o)
{
    THPObjectPtr f(PyNumber_Float(o));
    if (!f) throw python_error();
    return (float)PyFloat_AS_DOUBLE(f.get());
}

const Tensor &bf16(PyObject *o, const char *name)
{
    const Tensor &t = tensor(o, name);
    if (!(t.is_cuda() && t.scalar_type() == at::kBFloat16 && t.stride(-1) == 1))
        type_error(std::string(name) + " must be a CUDA bfloat16 tensor with a contiguous last dimension");
    return t;
}

l4l_tensor4 tensor4(PyObject *o, const char *name)               // [B, T, H, D] view
{
    const Tensor &t = bf16(o, name);
    if (t.dim() != 4) value_error(std::string(name) + " must have 4 dimensions [B, T, H, D]");
    return l4l_tensor4{t.data_ptr(), t.stride(0), t.stride(1), t.stride(2)};
}

// caches [B, Hkv, slot, D], or page pools [page, Hkv, slot, D]: the same fields
struct Cache {
    const Tensor *k = nullptr, *v = nullptr;
    l4l_kv_cache contiguous() const
    {
        if (!k) return l4l_kv_cache{nullptr, nullptr, 0, 0, 0, 0};
        return l4l_kv_cache{k->data_ptr(), v->data_ptr(), k->stride(0), k->stride(1), k->stride(2), (int32_t)k->size(2)};
    }
    l4l_paged_kv paged() const
    {
        return l4l_paged_kv{k->data_ptr(), v->data_ptr(), k->stride(0), k->stride(1), k->stride(2), (int32_t)k->size(2),
                            (int32_t)k->size(0)};
    }
};
Cache cache_of(PyObject *ko, PyObject *vo, bool paged, bool fp8)
{
    Cache c;
    if (fp8) {
        for (int i = 0; i < 2; ++i) {
            const char *name = i ? "cache_v8" : "cache_k8";
            const Tensor &t = tensor(i ? vo : ko, name);
            if (!(t.is_cuda() && (t.scalar_type() == at::kByte || t.scalar_type() == at::kFloat8_e4m3fn) && t.dim() == 4 && t.stride(-1) == 1))
                type_error(std::string(name) + " must be a CUDA uint8 / float8_e4m3fn tensor [B, Hkv, max_len, D] with D contiguous");
            (i ? c.v : c.k) = &t;
        }
        if (c.k->sizes() != c.v->sizes() || c.k->strides() != c.v->strides())
            value_error("cache_k8 and cache_v8 must have equal shapes and strides");
        return c;
    }
    if (is_none(ko) && is_none(vo) && !paged) return c;
    c.k = &bf16(ko, paged ? "pool_k" : "cache_k");
    c.v = &bf16(vo, paged ? "pool_v" : "cache_v");
    if (c.k->dim() != 4 || c.k->sizes() != c.v->sizes() || c.k->strides() != c.v->strides())
        value_error(paged ? "pool_k and pool_v must be [pages, Hkv, page_size, D] views with equal shapes and strides"
                          : "cache_k and cache_v must be [B, Hkv, max_len, D] views with equal shapes and strides");
    return c;
}

const int32_t *i32(PyObject *o, const char *name)
{
    if (is_none(o)) return nullptr;
    const Tensor &t = tensor(o, name);
    if (!(t.is_cuda() && t.scalar_type() == at::kInt && t.is_contiguous()))
        type_error(std::string(name) + " must be a contiguous CUDA int32 tensor");
    return static_cast<const int32_t *>(t.data_ptr());
}

float *f32(PyObject *o, const char *name, at::IntArrayRef shape)
{
    if (is_none(o)) return nullptr;
    const Tensor &t = tensor(o, name);
    if (!(t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous()))
        type_error(std::string(name) + " must be a contiguous CUDA float32 tensor");
    if (t.sizes() != shape) {
        std::string s = "(";
        for (size_t i = 0; i < shape.size(); ++i) s += (i ? ", " : "") + std::to_string(shape[i]);
        value_error(std::string(name) + " must have shape " + s + (shape.size() == 1 ? ",)" : ")"));
    }
    return static_cast<float *>(t.data_ptr());
}

float *lse_of(PyObject *o, at::IntArrayRef shape, const char *what)
{
    if (is_none(o)) return nullptr;
    const Tensor &t = tensor(o, "lse");
    if (!(t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous() && t.sizes() == shape))
        type_error(std::string("lse must be a contiguous CUDA float32 tensor ") + what);
    return static_cast<float *>(t.data_ptr());
}

struct Table { const int32_t *ids; int stride; };
Table table_of(PyObject *o, int64_t B)
{
    const Tensor &t = tensor(o, "block_table");
    if (!(t.is_cuda() && t.scalar_type() == at::kInt && t.dim() == 2 && t.size(0) == B && t.is_contiguous()))
        type_error("block_table must be a contiguous CUDA int32 tensor [B, pages per sequence]");
    return {static_cast<const int32_t *>(t.data_ptr()), (int)t.size(1)};
}

struct Workspace { void *ptr; size_t bytes; };
Workspace workspace_of(PyObject *o)
{
    const Tensor &t = tensor(o, "workspace");
    return {t.data_ptr(), (size_t)t.numel() * t.element_size()};
}

// The library is called without the interpreter lock, as a ctypes call is: a launch may wait for room in the stream's queue.
struct Unlocked {
    PyThreadState *state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};

l4l_stream stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

struct Dims { int B, S, Hq, D; };
Dims dims4(PyObject *o, const char *name)
{
    const Tensor &t = tensor(o, name);
    if (t.dim() != 4) value_error(std::string(name) + " must have 4 dimensions [B, T, H, D]");
    return {(int)t.size(0), (int)t.size(1), (int)t.size(2), (int)t.size(3)};
}
int size_at(PyObject *o, const char *name, int dim) { return (int)tensor(o, name).size(dim); }

#define L4L_ARGS(count)                                                                \
    HANDLE_TH_ERRORS                                                                   \
    if (n != (count)) {                                                                \
        PyErr_Format(PyExc_TypeError, "%zd arguments instead of %d", n, (int)(count)); \
        return nullptr;                                                                \
    }
// the call itself, on the current stream s and without the interpreter lock
#define L4L_CALL(expr)                           \
    {                                            \
        const l4l_stream s = stream();           \
        l4l_status st;                           \
        {                                        \
            Unlocked unlocked;                   \
            st = (expr);                         \
        }                                        \
        return PyLong_FromLong((long)st);        \
    }
#define L4L_END END_HANDLE_TH_ERRORS

// q, k, v, o, seq_lens, scale, workspace, cache_k, cache_v, lse
PyObject *prefill(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    L4L_ARGS(10)
    const Dims d = dims4(a[0], "q");
    const int Hkv = size_at(a[1], "k", 2);
    float *lse = lse_of(a[9], {d.B, d.Hq, d.S}, "[B, Hq, S]");
    const l4l_tensor4 q = tensor4(a[0], "q"), k = tensor4(a[1], "k"), v = tensor4(a[2], "v"), o = tensor4(a[3], "o");
    const l4l_kv_cache cache = cache_of(a[7], a[8], false, false).contiguous();
    const int32_t *lens = i32(a[4], "seq_lens");
    const Workspace w = workspace_of(a[6]);
    const float scale = as_float(a[5]);
    L4L_CALL(l4l_attn_prefill(q, k, v, o, cache, lens, d.S, d.B, d.Hq, Hkv, d.D, scale, lse, w.ptr, w.bytes, s))
    L4L_END
}

// q, o, cache_k, cache_v, past_lens, q_lens, scale, workspace, lse
PyObject *prefill_chunk(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    L4L_ARGS(9)
    const Dims d = dims4(a[0], "q");
    const int Hkv = size_at(a[2], "cache_k", 1);
    float *lse = lse_of(a[8], {d.B, d.Hq, d.S}, "[B, Hq, S]");
    const l4l_tensor4 q = tensor4(a[0], "q"), o = tensor4(a[1], "o");
    const l4l_kv_cache cache = cache_of(a[2], a[3], false, false).contiguous();
    const int32_t *past = i32(a[4], "past_lens"), *lens = i32(a[5], "q_lens");
    const Workspace w = workspace_of(a[7]);
    const float scale = as_float(a[6]);
    L4L_CALL(l4l_attn_prefill_chunk(q, o, cache, past, lens, d.S, d.B, d.Hq, Hkv, d.D, scale, lse, w.ptr, w.bytes, s))
    L4L_END
}

// q, k_new, v_new, o, cache_k, cache_v, past_lens, q_lens, scale, workspace, lse, block_table
PyObject *prefill_chunk_append(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    L4L_ARGS(12)
    const Dims d = dims4(a[0], "q");
    const int Hkv = size_at(a[1], "k_new", 2);
    float *lse = lse_of(a[10], {d.B, d.Hq, d.S}, "[B, Hq, S]");
    const int32_t *past = i32(a[6], "past_lens"), *lens = i32(a[7], "q_lens");
    const float scale = as_float(a[8]);
    const Workspace w = workspace_of(a[9]);
    const bool paged = !is_none(a[11]);
    const Table t = paged ? table_of(a[11], d.B) : Table{nullptr, 0};
    const l4l_tensor4 q = tensor4(a[0], "q"), k = tensor4(a[1], "k_new"), v = tensor4(a[2], "v_new"), o = tensor4(a[3], "o");
    const Cache c = cache_of(a[4], a[5], paged, false);
    if (paged) {
        const l4l_paged_kv pool = c.paged();
        L4L_CALL(l4l_attn_prefill_chunk_paged_append(q, k, v, o, pool, t.ids, t.stride, past, lens, d.S, d.B, d.Hq, Hkv, d.D, scale, lse,
                                                     w.ptr, w.bytes, s))
    }
    const l4l_kv_cache cache = c.contiguous();
    L4L_CALL(l4l_attn_prefill_chunk_append(q, k, v, o, cache, past, lens, d.S, d.B, d.Hq, Hkv, d.D, scale, lse, w.ptr, w.bytes, s))
    L4L_END
}

// q, k_new, v_new, cache_k, cache_v, pos, n_new, cos, sin, q_weight, k_weight, eps
PyObject *rope_kv_append(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    L4L_ARGS(12)
    const Dims d = dims4(a[0], "q");
    const int Hkv = size_at(a[1], "k_new", 2), n_pos = size_at(a[7], "cos", 0);
    const l4l_tensor4 q = tensor4(a[0], "q"), k = tensor4(a[1], "k_new"), v = tensor4(a[2], "v_new");
    const l4l_kv_cache cache = cache_of(a[3], a[4], false, false).contiguous();
    const int32_t *pos = i32(a[5], "pos"), *n_new = i32(a[6], "n_new");
    const float *cs = f32(a[7], "cos", {n_pos, d.D / 2}), *sn = f32(a[8], "sin", {n_pos, d.D / 2});
    const float *qw = f32(a[9], "q_weight", {d.D}), *kw = f32(a[10], "k_weight", {d.D});
    const float eps = as_float(a[11]);
    L4L_CALL(l4l_rope_kv_append(q, k, v, cache, pos, n_new, d.S, d.B, d.Hq, Hkv, d.D, cs, sn, n_pos, qw, kw, eps, s))
    L4L_END
}

// What a decode call is, said by the entry point: an argument that is missing never makes it another operation.
// (binding.py has the same values.)
enum Form {
    kNewShapes = 1, kLseShape = 2,                               // shapes that are looked at: those of k_new and v_new, that of lse
    kAppend = 4, kRope = 8, kFp8 = 16, kPaged = 32,              // the operation
    kMaybePaged = 64,                                            // paged where a block table is given
};

// Every decode step: q, o, k, v, k_scale, v_scale (fp8 caches), block_table (paged), k_new, v_new (fused append), kv_lens,
// max_kv_len, scale, cos, sin, q_weight, k_weight, eps (rope), workspace, lse, form. What the form has no use for is None.
PyObject *decode(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    L4L_ARGS(20)
    const int form = as_int(a[19]);
    const bool fp8 = form & kFp8, append = form & kAppend, rope = form & kRope;
    const bool paged = (form & kPaged) || ((form & kMaybePaged) && !is_none(a[6]));
    // (a missing sin or scale is a null pointer, which the library refuses)
    if (append) tensor(a[7], "k_new"), tensor(a[8], "v_new");
    if (paged) tensor(a[6], "block_table");
    if (rope) tensor(a[12], "cos");
    const Tensor &q = bf16(a[0], "q"), &o = bf16(a[1], "o");
    if (!(q.is_contiguous() && o.is_contiguous() && q.dim() == 3 && q.sizes() == o.sizes())) value_error("q and o must be dense [B, Hq, D]");
    const int B = (int)q.size(0), Hq = (int)q.size(1), D = (int)q.size(2);
    const Cache c = cache_of(a[2], a[3], paged, fp8);
    if (!c.k) type_error("cache_k must be a tensor");
    const int Hkv = (int)c.k->size(1);
    l4l_tensor4 kn{}, vn{};
    if (append) {
        const int64_t want[4] = {B, 1, Hkv, D};
        if ((form & kNewShapes) && (tensor(a[7], "k_new").sizes() != at::IntArrayRef(want, 4) ||
                                    tensor(a[8], "v_new").sizes() != at::IntArrayRef(want, 4)))
            value_error("k_new and v_new must be [B, 1, Hkv, D]");
        kn = tensor4(a[7], "k_new");
        vn = tensor4(a[8], "v_new");
    }
    float *lse = (form & kLseShape) ? lse_of(a[18], {B, Hq}, "[B, Hq]")
                              : is_none(a[18]) ? nullptr : static_cast<float *>(tensor(a[18], "lse").data_ptr());
    const Table t = paged ? table_of(a[6], B) : Table{nullptr, 0};
    const int32_t *lens = i32(a[9], "kv_lens");
    const int max_len = as_int(a[10]);
    const float scale = as_float(a[11]);
    const float *ks = nullptr, *vs = nullptr, *cs = nullptr, *sn = nullptr, *qw = nullptr, *kw = nullptr;
    int n_pos = 0;
    float eps = 0.f;
    if (rope) {
        n_pos = size_at(a[12], "cos", 0);
        cs = f32(a[12], "cos", {n_pos, D / 2});
        sn = f32(a[13], "sin", {n_pos, D / 2});
        qw = f32(a[14], "q_weight", {D});
        kw = f32(a[15], "k_weight", {D});
        eps = as_float(a[16]);
    }
    const Workspace w = workspace_of(a[17]);
    if (fp8) {
        ks = f32(a[4], "k_scale", {Hkv});
        vs = f32(a[5], "v_scale", {Hkv});
    }
    void *qp = q.data_ptr(), *op = o.data_ptr();
    const l4l_kv_cache cache = c.contiguous();
    const l4l_paged_kv pool = paged ? c.paged() : l4l_paged_kv{};
    const l4l_stream s = stream();
    l4l_status st;
    {
    Unlocked unlocked;
    if (fp8 && rope)
        st = paged ? l4l_attn_decode_paged_rope_append_fp8(qp, op, pool, ks, vs, t.ids, t.stride, kn, vn, lens, max_len, B, Hq, Hkv, D, scale,
                                                           cs, sn, n_pos, qw, kw, eps, lse, w.ptr, w.bytes, s)
                   : l4l_attn_decode_rope_append_fp8(qp, op, cache, ks, vs, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, cs, sn,
                                                     n_pos, qw, kw, eps, lse, w.ptr, w.bytes, s);
    else if (fp8 && append)
        st = paged ? l4l_attn_decode_paged_append_fp8(qp, op, pool, ks, vs, t.ids, t.stride, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, lse,
                                                      w.ptr, w.bytes, s)
                   : l4l_attn_decode_append_fp8(qp, op, cache, ks, vs, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr,
                                                w.bytes, s);
    else if (fp8)
        st = paged ? l4l_attn_decode_paged_fp8(qp, op, pool, ks, vs, t.ids, t.stride, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr,
                                               w.bytes, s)
                   : l4l_attn_decode_fp8(qp, op, cache, ks, vs, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr, w.bytes, s);
    else if (rope)
        st = paged ? l4l_attn_decode_paged_rope_append(qp, op, pool, t.ids, t.stride, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, cs, sn,
                                                       n_pos, qw, kw, eps, lse, w.ptr, w.bytes, s)
                   : l4l_attn_decode_rope_append(qp, op, cache, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, cs, sn, n_pos, qw, kw,
                                                 eps, lse, w.ptr, w.bytes, s);
    else if (append)
        st = paged ? l4l_attn_decode_paged_append(qp, op, pool, t.ids, t.stride, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr,
                                                  w.bytes, s)
                   : l4l_attn_decode_append(qp, op, cache, kn, vn, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr, w.bytes, s);
    else
        st = paged ? l4l_attn_decode_paged(qp, op, pool, t.ids, t.stride, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr, w.bytes, s)
                   : l4l_attn_decode(qp, op, cache, lens, max_len, B, Hq, Hkv, D, scale, lse, w.ptr, w.bytes, s);
    }
    return PyLong_FromLong((long)st);
    L4L_END
}

// x, gate_x, gate_a, a_param, state, y, workspace, position, seq_lens
PyObject *rglru_scan(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    L4L_ARGS(9)
    const Tensor &x = tensor(a[0], "x");
    const char *names[4] = {"x", "gate_x", "gate_a", "y"};
    const int arg[4] = {0, 1, 2, 5};
    void *ptr[4];
    for (int i = 0; i < 4; ++i) {
        const Tensor &t = bf16(a[arg[i]], names[i]);
        if (!(t.dim() == 3 && t.is_contiguous() && t.sizes() == x.sizes()))
            value_error(std::string(names[i]) + " must be a dense [B, T, W] tensor of the same shape as x");
        ptr[i] = t.data_ptr();
    }
    const int B = (int)x.size(0), T = (int)x.size(1), W = (int)x.size(2);
    const int32_t *position = nullptr;
    if (!is_none(a[7])) {
        const Tensor &t = tensor(a[7], "position");
        const int64_t want[2] = {B, T};
        if (!(t.is_cuda() && t.scalar_type() == at::kInt && t.is_contiguous() && t.sizes() == at::IntArrayRef(want, 2)))
            type_error("position must be a contiguous CUDA int32 tensor [B, T]");
        position = static_cast<const int32_t *>(t.data_ptr());
    }
    const float *ap = f32(a[3], "a_param", {W});
    const int32_t *lens = i32(a[8], "seq_lens");
    float *state = f32(a[4], "state", {B, W});
    const Workspace w = workspace_of(a[6]);
    L4L_CALL(l4l_rglru_scan(ptr[0], ptr[1], ptr[2], ap, position, lens, state, ptr[3], B, T, W, w.ptr, w.bytes, s))
    L4L_END
}

#define L4L_METHOD(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    L4L_METHOD(prefill),        L4L_METHOD(prefill_chunk), L4L_METHOD(prefill_chunk_append),
    L4L_METHOD(rope_kv_append), L4L_METHOD(decode),        L4L_METHOD(rglru_scan),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_l4l_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__l4l_marshal()
{
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "BUILT_FOR", L4L_BUILT_FOR) < 0) Py_CLEAR(m);
    return m;
}
