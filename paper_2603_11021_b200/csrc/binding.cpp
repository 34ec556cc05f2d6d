// Python binding of the entry points that launch work (the module paper_2603_11021_b200._native): argument checks, the output
// tensor and the call into the C ABI of include/llvq.h in one native function each.  A small product runs for about as long as
// the host needs to launch it, so what the host does per call is part of its time: through ctypes, with the checks in Python,
// a call cost 12.8 us of host time, of which the launch itself is a quarter.
//
// Every function takes the context as the address in Context._ptr, tensors as they are, sizes as integers and the stream as a
// CUDA stream address or None (PyTorch's current stream), and returns the output tensor, or a nonzero LLVQ status as an int
// for the caller to raise.  Violated expectations raise AssertionError, tensors of the wrong kind TypeError.
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>

#include "llvq.h"

namespace {

struct Args {
    PyObject* const* a;
    bool ok = true;

    bool expect(bool cond)
    {
        if (!cond && ok) { PyErr_SetNone(PyExc_AssertionError); ok = false; }
        return ok;
    }
    const at::Tensor* tensor(int i, const char* name)
    {
        if (!ok) return nullptr;
        if (!THPVariable_Check(a[i])) { wrong(name); return nullptr; }
        return &THPVariable_Unpack(a[i]);
    }
    const at::Tensor* tensor_or_none(int i, const char* name) { return a[i] == Py_None ? nullptr : tensor(i, name); }
    void wrong(const char* name)
    {
        if (ok) PyErr_Format(PyExc_TypeError, "%s must be a contiguous CUDA tensor", name);
        ok = false;
    }
    void* device(const at::Tensor* t, const char* name)
    {
        if (!ok || !t) return nullptr;
        if (!t->is_cuda() || !t->is_contiguous()) { wrong(name); return nullptr; }
        return t->data_ptr();
    }
    int64_t integer(int i)
    {
        if (!ok) return 0;
        const long long v = PyLong_AsLongLong(a[i]);
        if (v == -1 && PyErr_Occurred()) ok = false;
        return v;
    }
    const llvq_ctx* context(int i)
    {
        if (!ok) return nullptr;
        void* p = PyLong_AsVoidPtr(a[i]);
        if (!p && PyErr_Occurred()) ok = false;
        return static_cast<const llvq_ctx*>(p);
    }
    void* stream(int i)
    {
        if (!ok) return nullptr;
        if (a[i] == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        void* p = PyLong_AsVoidPtr(a[i]);
        if (!p && PyErr_Occurred()) ok = false;
        return p;
    }
    at::ScalarType dtype(int i)
    {
        if (!ok) return at::kFloat;
        if (!THPDtype_Check(a[i])) { PyErr_SetString(PyExc_TypeError, "y_dtype must be a torch.dtype"); ok = false; return at::kFloat; }
        return reinterpret_cast<THPDtype*>(a[i])->scalar_type;
    }
};

uint64_t bytes_of(const at::Tensor& t) { return (uint64_t)t.numel() * (uint64_t)t.element_size(); }

at::Tensor new_tensor(at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like)
{
    return at::empty(shape, at::TensorOptions().dtype(type).device(like.device()));
}

// the output tensor, or the status
PyObject* result(int status, at::Tensor&& y)
{
    if (status != LLVQ_OK) return PyLong_FromLong(status);
    return THPVariable_Wrap(std::move(y));
}

template <typename F>
int call(F f)
{
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = f();
    Py_END_ALLOW_THREADS
    return s;
}

int y_code(at::ScalarType t) { return t == at::kFloat ? LLVQ_F32 : LLVQ_BF16; }
// Whether w has room for rows x cols with leading dimension ld (the product may exceed 64 bits).
bool holds(const at::Tensor& w, int64_t rows, int64_t cols, int64_t ld) { return rows == 0 || (__int128)w.numel() >= ((__int128)rows - 1) * ld + cols; }
uint64_t blocks_of(int64_t rows, int64_t cols) { return (uint64_t)rows * (uint64_t)((cols + 23) / 24); }

// C++ exceptions become the Python ones that PyTorch's own functions raise for them (torch.OutOfMemoryError and so on).
#define LLVQ_FUNC(name, count)                                                                                    \
    PyObject* name##_body(Args& A);                                                                               \
    PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t n)                                                 \
    {                                                                                                             \
        HANDLE_TH_ERRORS                                                                                          \
        if (n != count) { PyErr_Format(PyExc_TypeError, #name " takes %d arguments", count); return nullptr; }    \
        Args A{args};                                                                                             \
        PyObject* r = name##_body(A);                                                                             \
        return A.ok ? r : nullptr;                                                                                \
        END_HANDLE_TH_ERRORS                                                                                      \
    }                                                                                                             \
    PyObject* name##_body(Args& A)

// (ctx, weights, gain, n_out, k_in, x, y or None, y_dtype, stream, sorted)
LLVQ_FUNC(gemv, 10)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *w = A.tensor(1, "d_idx"), *g = A.tensor(2, "d_gain"), *x = A.tensor(5, "d_x"), *y0 = A.tensor_or_none(6, "d_y");
    const int64_t n_out = A.integer(3), k_in = A.integer(4);
    const at::ScalarType yt = y0 ? y0->scalar_type() : A.dtype(7);
    const bool sorted = A.a[9] == Py_True;
    if (!A.ok) return nullptr;
    at::Tensor y = y0 ? *y0 : new_tensor({n_out}, yt, *w);
    A.expect(x->scalar_type() == at::kBFloat16 && x->numel() >= k_in && g->scalar_type() == at::kHalf);
    A.expect((y.scalar_type() == at::kFloat || y.scalar_type() == at::kBFloat16) && y.numel() >= n_out);
    const uint64_t nblocks = blocks_of(n_out, k_in);
    A.expect((uint64_t)g->numel() >= nblocks && bytes_of(*w) >= (sorted ? llvq_sorted_bytes(ctx, n_out, k_in) : llvq_index_bytes(ctx, nblocks)));
    const void* pw = A.device(w, sorted ? "d_sorted" : "d_idx");
    const uint16_t *pg = static_cast<const uint16_t*>(A.device(g, "d_gain")), *px = static_cast<const uint16_t*>(A.device(x, "d_x"));
    void* py = A.device(&y, "d_y");
    void* st = A.stream(8);
    if (!A.ok) return nullptr;
    const int s = call([&] {
        return sorted ? llvq_gemv_sorted(ctx, pw, pg, n_out, k_in, px, py, y_code(y.scalar_type()), st)
                      : llvq_gemv(ctx, pw, pg, n_out, k_in, px, py, y_code(y.scalar_type()), st);
    });
    return result(s, std::move(y));
}

// codebook and row scales of the shape-gain form
struct SgPtrs { const float *cb, *rs; };
SgPtrs sg_args(Args& A, const at::Tensor* cb, const at::Tensor* rs, int64_t gain_bits, int64_t rows)
{
    A.expect(cb->scalar_type() == at::kFloat && gain_bits >= 0 && gain_bits < 32 && cb->numel() >= (1ll << gain_bits));
    A.expect(!rs || (rs->scalar_type() == at::kFloat && rs->numel() >= rows));
    return {static_cast<const float*>(A.device(cb, "d_codebook")), static_cast<const float*>(A.device(rs, "d_row_scale"))};
}

// (ctx, fields, gain_bits, codebook, row_scale or None, n_out, k_in, x, y or None, y_dtype, stream, sorted)
LLVQ_FUNC(gemv_sg, 12)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *w = A.tensor(1, "d_fields"), *cb = A.tensor(3, "d_codebook"), *rs = A.tensor_or_none(4, "d_row_scale"),
                     *x = A.tensor(7, "d_x"), *y0 = A.tensor_or_none(8, "d_y");
    const int64_t bits = A.integer(2), n_out = A.integer(5), k_in = A.integer(6);
    const at::ScalarType yt = y0 ? y0->scalar_type() : A.dtype(9);
    const bool sorted = A.a[11] == Py_True;
    if (!A.ok) return nullptr;
    at::Tensor y = y0 ? *y0 : new_tensor({n_out}, yt, *w);
    A.expect(x->scalar_type() == at::kBFloat16 && x->numel() >= k_in);
    A.expect((y.scalar_type() == at::kFloat || y.scalar_type() == at::kBFloat16) && y.numel() >= n_out);
    if (!A.ok) return nullptr;
    const SgPtrs p = sg_args(A, cb, rs, bits, n_out);
    A.expect(bytes_of(*w) >= (sorted ? llvq_sorted_bytes(ctx, n_out, k_in) : llvq_field_bytes(ctx, blocks_of(n_out, k_in), (int)bits)));
    const void* pw = A.device(w, sorted ? "d_sorted" : "d_fields");
    const uint16_t* px = static_cast<const uint16_t*>(A.device(x, "d_x"));
    void* py = A.device(&y, "d_y");
    void* st = A.stream(10);
    if (!A.ok) return nullptr;
    const int s = call([&] {
        return sorted ? llvq_gemv_sorted_sg(ctx, pw, (int)bits, p.cb, p.rs, n_out, k_in, px, py, y_code(y.scalar_type()), st)
                      : llvq_gemv_sg(ctx, pw, (int)bits, p.cb, p.rs, n_out, k_in, px, py, y_code(y.scalar_type()), st);
    });
    return result(s, std::move(y));
}

// (ctx, weights, gain, n_out, k_in, X, Y or None, stream, form): form 0 stored stream, 1 sorted layout, 2 the call that allocates nothing
LLVQ_FUNC(gemm, 9)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *w = A.tensor(1, "d_idx"), *g = A.tensor(2, "d_gain"), *x = A.tensor(5, "d_x"), *y0 = A.tensor_or_none(6, "d_y");
    const int64_t n_out = A.integer(3), k_in = A.integer(4);
    const int64_t form = A.integer(8);
    if (!A.ok) return nullptr;
    if (!A.expect(x->scalar_type() == at::kBFloat16 && x->dim() == 2 && x->size(1) == k_in && g->scalar_type() == at::kHalf)) return nullptr;
    const int64_t batch = x->size(0);
    if (!A.expect(form != 2 || y0)) return nullptr;             // that call allocates nothing: Y has to be passed in
    at::Tensor y = y0 ? *y0 : new_tensor({batch, n_out}, at::kBFloat16, *w);
    A.expect(y.scalar_type() == at::kBFloat16 && y.numel() >= batch * n_out);
    const uint64_t nblocks = blocks_of(n_out, k_in);
    A.expect(form == 2 || ((uint64_t)g->numel() >= nblocks &&
                           bytes_of(*w) >= (form == 1 ? llvq_sorted_gemm_bytes(ctx, n_out, k_in) : llvq_index_bytes(ctx, nblocks))));
    const void* pw = A.device(w, form == 1 ? "d_sorted" : "d_idx");
    const uint16_t *pg = static_cast<const uint16_t*>(A.device(g, "d_gain")), *px = static_cast<const uint16_t*>(A.device(x, "d_x"));
    uint16_t* py = static_cast<uint16_t*>(A.device(&y, "d_y"));
    void* st = A.stream(7);
    if (!A.ok) return nullptr;
    const int s = call([&] {
        return form == 1   ? llvq_gemm_small_batch_sorted(ctx, pw, pg, n_out, k_in, px, (int)batch, py, st)
               : form == 2 ? llvq_gemm_small_batch_noalloc(ctx, pw, pg, n_out, k_in, px, (int)batch, py, st)
                           : llvq_gemm_small_batch(ctx, pw, pg, n_out, k_in, px, (int)batch, py, st);
    });
    return result(s, std::move(y));
}

// (ctx, fields, gain_bits, codebook, row_scale or None, n_out, k_in, X, Y or None, stream, sorted)
LLVQ_FUNC(gemm_sg, 11)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *w = A.tensor(1, "d_fields"), *cb = A.tensor(3, "d_codebook"), *rs = A.tensor_or_none(4, "d_row_scale"),
                     *x = A.tensor(7, "d_x"), *y0 = A.tensor_or_none(8, "d_y");
    const int64_t bits = A.integer(2), n_out = A.integer(5), k_in = A.integer(6);
    const bool sorted = A.a[10] == Py_True;
    if (!A.ok) return nullptr;
    if (!A.expect(x->scalar_type() == at::kBFloat16 && x->dim() == 2 && x->size(1) == k_in)) return nullptr;
    const int64_t batch = x->size(0);
    at::Tensor y = y0 ? *y0 : new_tensor({batch, n_out}, at::kBFloat16, *w);
    if (!A.expect(y.scalar_type() == at::kBFloat16 && y.numel() >= batch * n_out)) return nullptr;
    const SgPtrs p = sg_args(A, cb, rs, bits, n_out);
    A.expect(bytes_of(*w) >= (sorted ? llvq_sorted_gemm_bytes(ctx, n_out, k_in) : llvq_field_bytes(ctx, blocks_of(n_out, k_in), (int)bits)));
    const void* pw = A.device(w, sorted ? "d_sorted" : "d_fields");
    const uint16_t* px = static_cast<const uint16_t*>(A.device(x, "d_x"));
    uint16_t* py = static_cast<uint16_t*>(A.device(&y, "d_y"));
    void* st = A.stream(9);
    if (!A.ok) return nullptr;
    const int s = call([&] {
        return sorted ? llvq_gemm_small_batch_sorted_sg(ctx, pw, (int)bits, p.cb, p.rs, n_out, k_in, px, (int)batch, py, st)
                      : llvq_gemm_small_batch_sg(ctx, pw, (int)bits, p.cb, p.rs, n_out, k_in, px, (int)batch, py, st);
    });
    return result(s, std::move(y));
}

// (ctx, mats, y_dtype, stream, sorted): mats a sequence of (weights, gain, n_out, k_in, x, y); returns the status
LLVQ_FUNC(gemv_multi, 5)
{
    const llvq_ctx* ctx = A.context(0);
    const at::ScalarType yt = A.dtype(2);
    const bool sorted = A.a[4] == Py_True;
    if (!A.expect(yt == at::kFloat || yt == at::kBFloat16)) return nullptr;
    PyObject* mats = PySequence_Fast(A.a[1], "mats must be a sequence");
    if (!mats) { A.ok = false; return nullptr; }
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(mats);
    std::vector<llvq_gemv_desc> d((size_t)n);
    for (Py_ssize_t i = 0; i < n && A.ok; ++i) {
        PyObject* m = PySequence_Fast(PySequence_Fast_GET_ITEM(mats, i), "a matrix is (weights, gain, n_out, k_in, x, y)");
        if (!m) { A.ok = false; break; }
        if (PySequence_Fast_GET_SIZE(m) != 6) {
            PyErr_SetString(PyExc_ValueError, "a matrix is (weights, gain, n_out, k_in, x, y)");
            A.ok = false;
        } else {
            Args M{PySequence_Fast_ITEMS(m)};
            const at::Tensor *w = M.tensor(0, "d_weights"), *g = M.tensor(1, "d_gain"), *x = M.tensor(4, "d_x"), *y = M.tensor(5, "d_y");
            llvq_gemv_desc& q = d[(size_t)i];
            q.n_out = M.integer(2);
            q.k_in = M.integer(3);
            if (M.ok) {
                M.expect(x->scalar_type() == at::kBFloat16 && x->numel() >= q.k_in && g->scalar_type() == at::kHalf);
                M.expect(y->scalar_type() == yt && y->numel() >= q.n_out && g->numel() >= (int64_t)blocks_of(q.n_out, q.k_in));
            }
            q.d_weights = M.device(w, "d_weights");
            q.d_gain_f16 = static_cast<const uint16_t*>(M.device(g, "d_gain"));
            q.d_x_bf16 = static_cast<const uint16_t*>(M.device(x, "d_x"));
            q.d_y = M.device(y, "d_y");
            A.ok = M.ok;
        }
        Py_DECREF(m);
    }
    int s = LLVQ_OK;
    void* st = A.stream(3);
    if (A.ok)
        s = call([&] {
            return sorted ? llvq_gemv_sorted_multi(ctx, d.data(), (int)n, y_code(yt), st) : llvq_gemv_multi(ctx, d.data(), (int)n, y_code(yt), st);
        });
    Py_DECREF(mats);
    return A.ok ? PyLong_FromLong(s) : nullptr;
}

// (ctx, idx, gain, rows, cols, layout, W or None, ld, stream)
LLVQ_FUNC(dequant, 9)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *idx = A.tensor(1, "d_idx"), *g = A.tensor(2, "d_gain"), *w0 = A.tensor_or_none(6, "d_w");
    const int64_t rows = A.integer(3), cols = A.integer(4), layout = A.integer(5), ld = A.integer(7);
    if (!A.ok) return nullptr;
    at::Tensor w = w0 ? *w0 : new_tensor({rows, ld}, at::kBFloat16, *idx);
    A.expect(w.scalar_type() == at::kBFloat16 && g->scalar_type() == at::kHalf);
    const uint64_t nblocks = layout == LLVQ_LAYOUT_FLAT ? ((uint64_t)rows * (uint64_t)cols + 23) / 24 : blocks_of(rows, cols);
    A.expect((uint64_t)g->numel() >= nblocks && bytes_of(*idx) >= llvq_index_bytes(ctx, nblocks));
    A.expect(holds(w, rows, cols, ld));
    const void* pi = A.device(idx, "d_idx");
    const uint16_t* pg = static_cast<const uint16_t*>(A.device(g, "d_gain"));
    uint16_t* pw = static_cast<uint16_t*>(A.device(&w, "d_w"));
    void* st = A.stream(8);
    if (!A.ok) return nullptr;
    const int s = call([&] { return llvq_dequant_matrix(ctx, pi, pg, rows, cols, (int)layout, pw, ld, st); });
    return result(s, std::move(w));
}

// (ctx, fields, gain_bits, codebook, row_scale or None, rows, cols, W or None, ld, stream)
LLVQ_FUNC(dequant_sg, 10)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *f = A.tensor(1, "d_fields"), *cb = A.tensor(3, "d_codebook"), *rs = A.tensor_or_none(4, "d_row_scale"), *w0 = A.tensor_or_none(7, "d_w");
    const int64_t bits = A.integer(2), rows = A.integer(5), cols = A.integer(6), ld = A.integer(8);
    if (!A.ok) return nullptr;
    at::Tensor w = w0 ? *w0 : new_tensor({rows, ld}, at::kBFloat16, *f);
    A.expect(w.scalar_type() == at::kBFloat16);
    if (!A.expect(holds(w, rows, cols, ld))) return nullptr;
    const SgPtrs p = sg_args(A, cb, rs, bits, rows);
    A.expect(bytes_of(*f) >= llvq_field_bytes(ctx, blocks_of(rows, cols), (int)bits));
    const void* pf = A.device(f, "d_fields");
    uint16_t* pw = static_cast<uint16_t*>(A.device(&w, "d_w"));
    void* st = A.stream(9);
    if (!A.ok) return nullptr;
    const int s = call([&] { return llvq_dequant_matrix_sg(ctx, pf, (int)bits, p.cb, p.rs, rows, cols, pw, ld, st); });
    return result(s, std::move(w));
}

// (ctx, idx, nblocks, points or None, stream)
LLVQ_FUNC(decode, 5)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *idx = A.tensor(1, "d_idx"), *p0 = A.tensor_or_none(3, "d_points");
    const int64_t n = A.integer(2);
    if (!A.ok) return nullptr;
    at::Tensor p = p0 ? *p0 : new_tensor({n, 24}, at::kChar, *idx);
    A.expect(p.scalar_type() == at::kChar && p.numel() >= n * 24);
    A.expect(bytes_of(*idx) >= llvq_index_bytes(ctx, (uint64_t)n));
    const void* pi = A.device(idx, "d_idx");
    int8_t* pp = static_cast<int8_t*>(A.device(&p, "d_points"));
    void* st = A.stream(4);
    if (!A.ok) return nullptr;
    const int s = call([&] { return llvq_decode_blocks(ctx, pi, (uint64_t)n, pp, st); });
    return result(s, std::move(p));
}

// (ctx, v, metric, points or None, index or None, stream) -> (points, index)
LLVQ_FUNC(encode, 6)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *v = A.tensor(1, "d_v"), *p0 = A.tensor_or_none(3, "d_points"), *i0 = A.tensor_or_none(4, "d_index");
    const int64_t metric = A.integer(2);
    if (!A.ok) return nullptr;
    if (!A.expect(v->scalar_type() == at::kFloat && v->dim() == 2 && v->size(1) == 24)) return nullptr;
    const int64_t n = v->size(0);
    at::Tensor p = p0 ? *p0 : new_tensor({n, 24}, at::kChar, *v), ix = i0 ? *i0 : new_tensor({n}, at::kLong, *v);
    A.expect(p.scalar_type() == at::kChar && p.numel() >= n * 24 && ix.scalar_type() == at::kLong && ix.numel() >= n);
    const float* pv = static_cast<const float*>(A.device(v, "d_v"));
    int8_t* pp = static_cast<int8_t*>(A.device(&p, "d_points"));
    uint64_t* pi = static_cast<uint64_t*>(A.device(&ix, "d_index"));
    void* st = A.stream(5);
    if (!A.ok) return nullptr;
    const int s = call([&] { return llvq_encode_blocks(ctx, pv, (uint64_t)n, (int)metric, pp, pi, st); });
    if (s != LLVQ_OK) return PyLong_FromLong(s);
    PyObject *a = THPVariable_Wrap(std::move(p)), *b = THPVariable_Wrap(std::move(ix));
    PyObject* r = a && b ? PyTuple_Pack(2, a, b) : nullptr;
    Py_XDECREF(a);
    Py_XDECREF(b);
    if (!r) A.ok = false;
    return r;
}

// (ctx, points, index or None, stream)
LLVQ_FUNC(rank, 4)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *p = A.tensor(1, "d_points"), *i0 = A.tensor_or_none(2, "d_index");
    if (!A.ok) return nullptr;
    if (!A.expect(p->scalar_type() == at::kChar && p->dim() == 2 && p->size(1) == 24)) return nullptr;
    const int64_t n = p->size(0);
    at::Tensor ix = i0 ? *i0 : new_tensor({n}, at::kLong, *p);
    A.expect(ix.scalar_type() == at::kLong && ix.numel() >= n);
    const int8_t* pp = static_cast<const int8_t*>(A.device(p, "d_points"));
    uint64_t* pi = static_cast<uint64_t*>(A.device(&ix, "d_index"));
    void* st = A.stream(3);
    if (!A.ok) return nullptr;
    const int s = call([&] { return llvq_rank_blocks(ctx, pp, (uint64_t)n, pi, st); });
    return result(s, std::move(ix));
}

// (ctx, index, gain_index or None, gain_bits, fields or None, stream)
LLVQ_FUNC(pack, 6)
{
    const llvq_ctx* ctx = A.context(0);
    const at::Tensor *ix = A.tensor(1, "d_index"), *k = A.tensor_or_none(2, "d_gain_index"), *f0 = A.tensor_or_none(4, "d_fields");
    const int64_t bits = A.integer(3);
    if (!A.ok) return nullptr;
    if (!A.expect(ix->scalar_type() == at::kLong)) return nullptr;
    const int64_t n = ix->numel();
    const uint64_t nbytes = llvq_field_bytes(ctx, (uint64_t)n, (int)bits);
    at::Tensor f = f0 ? *f0 : new_tensor({(int64_t)nbytes}, at::kByte, *ix);
    A.expect(bytes_of(f) >= nbytes);
    A.expect(bits == 0 || (k && k->scalar_type() == at::kByte && k->numel() >= n));
    const uint64_t* pi = static_cast<const uint64_t*>(A.device(ix, "d_index"));
    const uint8_t* pk = bits == 0 ? nullptr : static_cast<const uint8_t*>(A.device(k, "d_gain_index"));
    void* pf = A.device(&f, "d_fields");
    void* st = A.stream(5);
    if (!A.ok) return nullptr;
    const int s = call([&] { return llvq_pack_fields(ctx, pi, pk, (int)bits, (uint64_t)n, pf, st); });
    return result(s, std::move(f));
}

#define LLVQ_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {LLVQ_METHOD(gemv), LLVQ_METHOD(gemv_sg), LLVQ_METHOD(gemm), LLVQ_METHOD(gemm_sg), LLVQ_METHOD(gemv_multi),
                         LLVQ_METHOD(dequant), LLVQ_METHOD(dequant_sg), LLVQ_METHOD(decode), LLVQ_METHOD(encode), LLVQ_METHOD(rank),
                         LLVQ_METHOD(pack), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Entry points of libllvq.so on PyTorch tensors.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (LLVQ_BUILT_FOR: the PyTorch and Python whose headers this was compiled with, looked for in the file before it is loaded)
PyMODINIT_FUNC PyInit__native()
{
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", LLVQ_BUILT_FOR) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
