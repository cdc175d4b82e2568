// The serving calls of binding.py -- prefill, the decode steps, the 8-bit append, the paged layer calls -- as a CPython
// extension over torch tensors: the same checks, messages and results as the ctypes form of the other calls.
//
// Why: what such a call does in Python (two dozen attribute reads, shape tuples, conversions, the allocation of its
// result) took 6 - 16 us, as long as the launches themselves, and the small calls are bound by it: a whole-layer decode step
// 32 us on the host against 31 on the device, a quantised prompt load 15 against 11.  Here it takes 1 - 3 us.
// The C library stays the one that binding.py has loaded: its entry points come in as addresses (bind).
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>

#include <array>
#include <initializer_list>
#include <string>
#include <string_view>

#include "gta.h"

namespace {

using at::Tensor;

#define GTA_ENTRIES(X)                                                                                               \
    X(gta_prefill_workspace_bytes) X(gta_prefill) X(gta_decode_workspace_bytes) X(gta_decode_append)                  \
    X(gta_layer_prefill_workspace_bytes) X(gta_layer_prefill_paged) X(gta_layer_decode_paged_workspace_bytes)         \
    X(gta_layer_decode_paged) X(gta_cache_append_fp8) X(gta_decode_fp8_workspace_bytes) X(gta_decode_fp8)

#define GTA_POINTER(name) decltype(&::name) name = nullptr;
struct Library { GTA_ENTRIES(GTA_POINTER) } lib;

struct Refused {};       // a Python exception is set
[[noreturn]] void refuse(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw Refused();
}
void need(bool ok, const char* what) {
    if (!ok) refuse(PyExc_ValueError, what);
}

const Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) refuse(PyExc_TypeError, "expected a torch.Tensor");
    return THPVariable_Unpack(o);
}
void* ptr(const Tensor& t) { return t.data_ptr(); }
void* ptr_or_null(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
long integer(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Refused();
    return v;
}
int32_t int32(PyObject* o) {
    const long v = integer(o);
    if (v != (int32_t)v) refuse(PyExc_ValueError, "integer out of range");
    return (int32_t)v;
}
float real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Refused();
    return (float)v;
}
void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw Refused();
    void* s = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (s == nullptr && PyErr_Occurred()) throw Refused();
    return s;
}

using Sizes = std::initializer_list<int64_t>;
bool is(const Tensor& t, Sizes want) { return t.sizes() == at::IntArrayRef(want); }
// sizes of a tensor that must have `n` dimensions
template <size_t n>
std::array<int64_t, n> dims(const Tensor& t) {
    need(t.dim() == (int64_t)n, "operator tensor with the wrong number of dimensions");
    std::array<int64_t, n> d;
    for (size_t i = 0; i < n; ++i) d[i] = t.size((int64_t)i);
    return d;
}

// one CUDA device, one dtype, contiguous
void check_tensors(std::initializer_list<const Tensor*> ts) {
    const Tensor& first = **ts.begin();
    for (const Tensor* t : ts) {
        need(t->scalar_type() == first.scalar_type() && t->device() == first.device(),
             "all operator tensors must share one device and one dtype");
        need(t->is_contiguous(), "operator tensors must be contiguous");
        need(t->is_cuda(), "operator tensors must live on a CUDA device");
    }
}
// The lengths of B sequences, which the kernels read and advance as they are; None goes on to the library, which refuses it.
void* lens_ptr(PyObject* o, const Tensor& like, int64_t B) {
    if (o == Py_None) return nullptr;
    const Tensor& t = tensor(o);
    need(t.scalar_type() == at::kInt && t.device() == like.device() && t.is_contiguous(),
         "seq_lens must be a contiguous int32 tensor on the operator's device");
    need(is(t, {B}), "seq_lens must hold one length per sequence");
    return t.data_ptr();
}
int32_t dtype_code(const Tensor& t) {
    if (t.scalar_type() == at::kFloat) return GTA_F32;
    if (t.scalar_type() == at::kBFloat16) return GTA_BF16;
    refuse(PyExc_TypeError, "unsupported dtype: the library takes float32 or bfloat16");
}
gta_shape_t shape_of(int64_t B, int64_t N, int64_t H, int64_t n_h, int64_t n_q, int64_t n_k, int64_t n_c, int64_t d_h,
                     int64_t d_l, int32_t dtype, int32_t causal, float scale) {
    return gta_shape_t{(int32_t)B, (int32_t)N, (int32_t)H, (int32_t)n_h, (int32_t)n_q, (int32_t)n_k,
                       (int32_t)n_c, (int32_t)d_h, (int32_t)d_l, causal, dtype, scale};
}

// result and workspace of a call: the caller's, or new ones
struct Buffers {
    Tensor out, ws;
    void *out_p, *ws_p;
    size_t ws_bytes;
    PyObject* given;
    Buffers(PyObject* o, PyObject* w, Sizes sizes, const Tensor& like, size_t bytes) : given(o) {
        out = o == Py_None ? at::empty(sizes, like.options()) : tensor(o);
        ws = w == Py_None ? at::empty({(int64_t)(bytes < 256 ? 256 : bytes)}, like.options().dtype(at::kByte)) : tensor(w);
        out_p = out.data_ptr();
        ws_p = ws.data_ptr();
        ws_bytes = ws.nbytes();
    }
};
size_t workspace_bytes(PyObject* given, size_t (*f)(const gta_shape_t*), const gta_shape_t& s) {
    return given == Py_None ? f(&s) : 0;
}

// The call itself, without the interpreter lock.  0: the result; anything else: the status, as an int.
template <class F>
PyObject* finish(Buffers& b, F call) {
    gta_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    if (st != GTA_OK) return PyLong_FromLong((long)st);
    if (b.given != Py_None) {
        Py_INCREF(b.given);
        return b.given;
    }
    return THPVariable_Wrap(b.out);
}

struct Paged { int32_t n_pages, page_size, max_pages; };
Paged check_pools(const Tensor& k, const Tensor& c, const Tensor& table) {
    need(table.scalar_type() == at::kInt && table.device() == k.device() && table.is_contiguous() && table.dim() == 2,
         "block_table must be a contiguous int32 [B, max_pages] tensor on the pools' device");
    const auto kd = dims<4>(k), cd = dims<4>(c);
    need(cd[0] == kd[0] && cd[2] == kd[2], "inconsistent pool tensor shapes");
    return Paged{(int32_t)kd[0], (int32_t)kd[2], (int32_t)table.size(1)};
}
struct Fp8Caches { int64_t B, n_k, n_c, cap, d_h, d_l; };
Fp8Caches check_fp8(const Tensor& k, const Tensor& c, const Tensor& ks, const Tensor& cs) {
    static const char* what = "8-bit caches: codes uint8 [B, groups, S_cap, width], scales float32 [B, groups, S_cap]";
    need(k.dim() == 4 && c.dim() == 4, what);
    const Fp8Caches f{k.size(0), k.size(1), c.size(1), k.size(2), k.size(3), c.size(3)};
    need(k.scalar_type() == at::kByte && c.scalar_type() == at::kByte && ks.scalar_type() == at::kFloat &&
         cs.scalar_type() == at::kFloat && is(c, {f.B, f.n_c, f.cap, f.d_l}) && is(ks, {f.B, f.n_k, f.cap}) &&
         is(cs, {f.B, f.n_c, f.cap}), what);
    for (const Tensor* t : {&k, &c, &ks, &cs})
        need(t->is_contiguous() && t->is_cuda() && t->device() == k.device(), "cache tensors must be contiguous CUDA tensors of one device");
    return f;
}

// q, k, c, x, w_p, w_g, causal, softmax_scale, out, workspace, status_word, stream
PyObject* prefill(PyObject* const* a) {
    const Tensor &q = tensor(a[0]), &k = tensor(a[1]), &c = tensor(a[2]), &x = tensor(a[3]), &wp = tensor(a[4]), &wg = tensor(a[5]);
    check_tensors({&q, &k, &c, &x, &wp, &wg});
    const auto [B, n_q, N, d_h] = dims<4>(q);
    const int64_t n_k = dims<4>(k)[1], n_c = dims<4>(c)[1], d_l = c.size(3), n_h = dims<3>(wp)[0], H = dims<3>(x)[2];
    need(is(k, {B, n_k, N, d_h}) && is(c, {B, n_c, N, d_l}) && is(x, {B, N, H}) && is(wp, {n_h, d_l, d_h}) &&
         is(wg, {H, n_h * d_h}), "inconsistent operator tensor shapes");
    const gta_shape_t s = shape_of(B, N, H, n_h, n_q, n_k, n_c, d_h, d_l, dtype_code(q), (int32_t)integer(a[6]), real(a[7]));
    Buffers b(a[8], a[9], {B, N, n_h, d_h}, q, workspace_bytes(a[9], lib.gta_prefill_workspace_bytes, s));
    void* status = ptr_or_null(a[10]);
    void* stream = stream_of(a[11]);
    return finish(b, [&] { return lib.gta_prefill(&s, ptr(q), ptr(k), ptr(c), ptr(x), ptr(wp), ptr(wg), b.out_p, b.ws_p,
                                                  b.ws_bytes, (int32_t*)status, stream); });
}

// q, k_cache, c_cache, k_new, c_new, seq_lens, x_t, w_p, w_g, softmax_scale, out, workspace, status_word, stream
PyObject* decode_append(PyObject* const* a) {
    const Tensor &q = tensor(a[0]), &k = tensor(a[1]), &c = tensor(a[2]), &kn = tensor(a[3]), &cn = tensor(a[4]),
                 &x = tensor(a[6]), &wp = tensor(a[7]), &wg = tensor(a[8]);
    check_tensors({&q, &k, &c, &kn, &cn, &x, &wp, &wg});
    const int64_t n_q = dims<3>(q)[1], n_h = dims<3>(wp)[0], H = dims<2>(x)[1];
    const auto [B, n_k, cap, d_h] = dims<4>(k);
    const int64_t n_c = dims<4>(c)[1], d_l = c.size(3);
    need(is(q, {B, n_q, d_h}) && is(c, {B, n_c, cap, d_l}) && is(x, {B, H}) && is(wp, {n_h, d_l, d_h}) &&
         is(wg, {H, n_h * d_h}), "inconsistent operator tensor shapes");
    need(kn.numel() == B * n_k * d_h && cn.numel() == B * n_c * d_l, "k_new / c_new hold one row per sequence and group");
    void* lens = lens_ptr(a[5], q, B);
    const gta_shape_t s = shape_of(B, 0, H, n_h, n_q, n_k, n_c, d_h, d_l, dtype_code(q), 1, real(a[9]));
    Buffers b(a[10], a[11], {B, n_h, d_h}, q,
              a[11] == Py_None ? lib.gta_decode_workspace_bytes(&s, (int32_t)cap) : 0);
    void* status = ptr_or_null(a[12]);
    void* stream = stream_of(a[13]);
    return finish(b, [&] { return lib.gta_decode_append(&s, ptr(q), ptr(k), ptr(c), ptr(kn), ptr(cn), (int32_t*)lens,
                                                        (int32_t)cap, ptr(x), ptr(wp), ptr(wg), b.out_p, b.ws_p, b.ws_bytes,
                                                        (int32_t*)status, stream); });
}

// k_codes, c_codes, k_scales, c_scales, k_new, c_new, seq_lens, status_word, stream
PyObject* cache_append_fp8(PyObject* const* a) {
    const Tensor &k = tensor(a[0]), &c = tensor(a[1]), &ks = tensor(a[2]), &cs = tensor(a[3]), &kn = tensor(a[4]),
                 &cn = tensor(a[5]);
    const Fp8Caches f = check_fp8(k, c, ks, cs);
    check_tensors({&kn, &cn});
    need(kn.device() == k.device(), "the new rows and the caches must share one device");
    void* lens = lens_ptr(a[6], k, f.B);
    need(kn.dim() == 4, "inconsistent new-row shapes");
    const int64_t n_new = kn.size(2);
    need(is(kn, {f.B, f.n_k, n_new, f.d_h}) && is(cn, {f.B, f.n_c, n_new, f.d_l}), "inconsistent new-row shapes");
    const int64_t n_q = f.n_k * f.n_c;     // any map count that both group counts divide: the append does not look at it
    const gta_shape_t s = shape_of(f.B, 0, 8, n_q, n_q, f.n_k, f.n_c, f.d_h, f.d_l, dtype_code(kn), 1, 0.f);
    void* status = ptr_or_null(a[7]);
    void* stream = stream_of(a[8]);
    gta_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = lib.gta_cache_append_fp8(&s, ptr(k), ptr(c), (float*)ptr(ks), (float*)ptr(cs), (int32_t)f.cap, ptr(kn), ptr(cn),
                                  (int32_t)n_new, (int32_t*)lens, (int32_t*)status, stream);
    Py_END_ALLOW_THREADS
    if (st != GTA_OK) return PyLong_FromLong((long)st);
    Py_INCREF(a[6]);
    return a[6];
}

// q, k_codes, c_codes, k_scales, c_scales, seq_lens, x_t, w_p, w_g, softmax_scale, out, workspace, status_word, stream
PyObject* decode_fp8(PyObject* const* a) {
    const Tensor &q = tensor(a[0]), &k = tensor(a[1]), &c = tensor(a[2]), &ks = tensor(a[3]), &cs = tensor(a[4]),
                 &x = tensor(a[6]), &wp = tensor(a[7]), &wg = tensor(a[8]);
    const Fp8Caches f = check_fp8(k, c, ks, cs);
    check_tensors({&q, &x, &wp, &wg});
    need(q.device() == k.device(), "the operator tensors and the caches must share one device");
    void* lens = lens_ptr(a[5], q, f.B);
    need(q.dim() >= 2 && wp.dim() >= 1 && x.dim() >= 2, "inconsistent operator tensor shapes");
    const int64_t n_q = q.size(1), n_h = wp.size(0), H = x.size(1);
    need(is(q, {f.B, n_q, f.d_h}) && is(wp, {n_h, f.d_l, f.d_h}) && is(wg, {H, n_h * f.d_h}) && is(x, {f.B, H}),
         "inconsistent operator tensor shapes");
    const gta_shape_t s = shape_of(f.B, 0, H, n_h, n_q, f.n_k, f.n_c, f.d_h, f.d_l, dtype_code(q), 1, real(a[9]));
    Buffers b(a[10], a[11], {f.B, n_h, f.d_h}, q,
              a[11] == Py_None ? lib.gta_decode_fp8_workspace_bytes(&s, (int32_t)f.cap) : 0);
    void* status = ptr_or_null(a[12]);
    void* stream = stream_of(a[13]);
    return finish(b, [&] { return lib.gta_decode_fp8(&s, ptr(q), ptr(k), ptr(c), (const float*)ptr(ks), (const float*)ptr(cs),
                                                     (const int32_t*)lens, (int32_t)f.cap, ptr(x), ptr(wp), ptr(wg),
                                                     b.out_p, b.ws_p, b.ws_bytes, (int32_t*)status, stream); });
}

// the tensors of a whole-layer call over pools; B rows of x
struct Layer {
    const Tensor &x, &w_qkc, &wp, &wg, &wo, &k, &c, &table;
    Paged p;
    int64_t B, H, n_h, d_l, d_h, n_k, n_c;
    Layer(PyObject* const* a, int64_t n_q)
        : x(tensor(a[0])), w_qkc(tensor(a[1])), wp(tensor(a[2])), wg(tensor(a[3])), wo(tensor(a[4])), k(tensor(a[5])),
          c(tensor(a[6])), table(tensor(a[7])) {
        check_tensors({&x, &w_qkc, &wp, &wg, &wo, &k, &c});
        p = check_pools(k, c, table);
        need(x.dim() >= 2, "inconsistent layer tensor shapes");
        B = x.size(0);
        H = x.size(x.dim() - 1);
        const auto w = dims<3>(wp);
        n_h = w[0]; d_l = w[1]; d_h = w[2];
        n_k = k.size(1); n_c = c.size(1);
        need(k.size(3) == d_h && c.size(3) == d_l && table.size(0) == B && is(w_qkc, {H, (n_q + n_k) * d_h + n_c * d_l}) &&
             is(wg, {H, n_h * d_h}) && is(wo, {n_h * d_h, H}), "inconsistent layer tensor shapes");
    }
};

// x, w_qkc, w_p, w_g, w_o, k_pool, c_pool, block_table, pos0, rope_base, n_q, softmax_scale, out, workspace, status_word, stream
PyObject* layer_prefill_paged(PyObject* const* a) {
    const int32_t n_q = int32(a[10]);
    const Layer w(a, n_q);
    need(w.x.dim() == 3, "inconsistent layer tensor shapes");
    const int64_t N = w.x.size(1);
    const gta_shape_t s = shape_of(w.B, N, w.H, w.n_h, n_q, w.n_k, w.n_c, w.d_h, w.d_l, dtype_code(w.x), 1, real(a[11]));
    const int32_t pos0 = int32(a[8]);
    const float base = real(a[9]);
    Buffers b(a[12], a[13], {w.B, N, w.H}, w.x, workspace_bytes(a[13], lib.gta_layer_prefill_workspace_bytes, s));
    void* status = ptr_or_null(a[14]);
    void* stream = stream_of(a[15]);
    return finish(b, [&] {
        return lib.gta_layer_prefill_paged(&s, pos0, base, ptr(w.x), ptr(w.w_qkc), ptr(w.wp), ptr(w.wg), ptr(w.wo), ptr(w.k),
                                           ptr(w.c), (const int32_t*)ptr(w.table), w.p.page_size, w.p.n_pages, w.p.max_pages,
                                           b.out_p, b.ws_p, b.ws_bytes, (int32_t*)status, stream); });
}

// x_t, w_qkc, w_p, w_g, w_o, k_pool, c_pool, block_table, seq_lens, rope_base, n_q, softmax_scale, out, workspace, status_word, stream
PyObject* layer_decode_paged(PyObject* const* a) {
    const int32_t n_q = int32(a[10]);
    const Tensor& lens = tensor(a[8]);
    const Layer w(a, n_q);
    need(lens.scalar_type() == at::kInt && lens.device() == w.k.device() && lens.is_contiguous(),
         "seq_lens must be a contiguous int32 tensor on the pools' device");
    need(w.x.dim() == 2 && is(lens, {w.B}), "inconsistent pool tensor shapes");
    const gta_shape_t s = shape_of(w.B, 0, w.H, w.n_h, n_q, w.n_k, w.n_c, w.d_h, w.d_l, dtype_code(w.x), 1, real(a[11]));
    const float base = real(a[9]);
    Buffers b(a[12], a[13], {w.B, w.H}, w.x,
              a[13] == Py_None ? lib.gta_layer_decode_paged_workspace_bytes(&s, w.p.page_size, w.p.max_pages) : 0);
    void* status = ptr_or_null(a[14]);
    void* stream = stream_of(a[15]);
    return finish(b, [&] {
        return lib.gta_layer_decode_paged(&s, (const int32_t*)ptr(w.table), w.p.page_size, w.p.n_pages, w.p.max_pages, base,
                                          ptr(w.x), ptr(w.w_qkc), ptr(w.wp), ptr(w.wg), ptr(w.wo), ptr(w.k), ptr(w.c),
                                          (int32_t*)ptr(lens), b.out_p, b.ws_p, b.ws_bytes, (int32_t*)status, stream); });
}

template <PyObject* (*F)(PyObject* const*), int kArgs>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    try {
        if (n != kArgs) refuse(PyExc_TypeError, "wrong number of arguments");
        return F(args);
    } catch (const Refused&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// bind(name, address): an entry point of the C library
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    const char* name = n == 2 ? PyUnicode_AsUTF8(args[0]) : nullptr;
    void* at = name ? PyLong_AsVoidPtr(args[1]) : nullptr;
    if (!at) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "bind(name, address)");
        return nullptr;
    }
    const std::string_view key(name);
#define GTA_BIND(entry_name) if (key == #entry_name) lib.entry_name = reinterpret_cast<decltype(lib.entry_name)>(at);
    GTA_ENTRIES(GTA_BIND)
    Py_RETURN_NONE;
}

#define GTA_METHOD(name, n) {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
    GTA_METHOD(prefill, 12), GTA_METHOD(decode_append, 14), GTA_METHOD(cache_append_fp8, 9), GTA_METHOD(decode_fp8, 14),
    GTA_METHOD(layer_prefill_paged, 16), GTA_METHOD(layer_decode_paged, 16), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_gta_binding", nullptr, -1, methods};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__gta_binding() { return PyModule_Create(&module); }
