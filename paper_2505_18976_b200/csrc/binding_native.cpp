// The per-call host path of the Python binding, as a CPython extension.
//
// A call of the compression library costs its caller about as much host time as a small batch costs the GPU: with
// ctypes, argument checks and marshalling in Python took 12-16 us per call on the GPU machine's host cores (20 us for a
// call whose kernel runs 10 us), so small calls ran at the pace of the interpreter.  Here the ordinary case -- CUDA
// tensors of the documented dtypes and layouts -- is checked and marshalled on the tensors' C++ objects (about 1 us
// plus the launch itself).  Whatever is out of the ordinary (host tensors, raw pointers, a wrong dtype or layout)
// is not judged here: the function returns None and the Python code in binding.py takes the call, with its checks
// and its exceptions.  The library's entry points are handed over by address (bind), so that exactly one copy of
// the library is loaded, the one that binding.py chose.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <c10/util/Exception.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/grass.h"

namespace {

// entry points of libgrass_b200.so
struct Api {
    decltype(&::grass_compress_ws) compress = nullptr;
    decltype(&::grass_compress_workspace_bytes) compress_bytes = nullptr;
    decltype(&::factgrass_compress_workspace_bytes) layer_bytes = nullptr;
    decltype(&::factgrass_compress_varlen) factgrass_varlen = nullptr;
    decltype(&::factgrass_compress_grouped_out) grouped_out = nullptr;
    decltype(&::factgrass_compress_grouped_varlen) grouped_varlen = nullptr;
    decltype(&::grass_score) score = nullptr;
    decltype(&::grass_score_bf16) score_bf16 = nullptr;
    PyObject* error = nullptr;     // binding.GrassError
} api;

const at::Tensor* as_tensor(PyObject* o)
{
    return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr;
}

// a tensor of this process's GPUs whose elements the kernels may address
bool is_cuda(const at::Tensor& t) { return t.is_cuda() && t.layout() == at::kStrided && !t.is_neg(); }

bool elem_dtype(const at::Tensor& t, int* dt)
{
    const auto s = t.scalar_type();
    if (s == at::kFloat) { *dt = GRASS_F32; return true; }
    if (s == at::kBFloat16) { *dt = GRASS_BF16; return true; }
    return false;
}

// None or a contiguous 1-D list of 4-byte integers
bool mask_list(PyObject* o, bool none_ok, const uint32_t** p, int64_t* n)
{
    *p = nullptr;
    *n = 0;
    if (o == Py_None) return none_ok;
    const at::Tensor* t = as_tensor(o);
    if (!t || !is_cuda(*t) || t->dim() != 1 || !t->is_contiguous()) return false;
    if (t->scalar_type() != at::kInt && t->scalar_type() != at::kUInt32) return false;
    *p = static_cast<const uint32_t*>(t->const_data_ptr());
    *n = t->numel();
    return true;
}

bool status_word(PyObject* o, uint32_t** p)
{
    *p = nullptr;
    if (o == Py_None) return true;
    const at::Tensor* t = as_tensor(o);
    if (!t || !is_cuda(*t)) return false;
    *p = static_cast<uint32_t*>(t->data_ptr());
    return true;
}

bool as_int(PyObject* o, int64_t* v)
{
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    *v = PyLong_AsLongLongAndOverflow(o, &overflow);
    return overflow == 0;
}

// k, s of a projection; the seed is taken modulo 2^64
bool sjlt_spec(PyObject* k, PyObject* s, PyObject* seed, grass_sjlt_spec* sp)
{
    int64_t kv, sv;
    if (!as_int(k, &kv) || !as_int(s, &sv) || !PyLong_CheckExact(seed)) return false;
    if (kv < 0 || kv > 0xFFFFFFFFLL || sv < 0 || sv > 0xFFFFFFFFLL) return false;
    sp->k = (uint32_t)kv;
    sp->s = (uint32_t)sv;
    sp->seed = PyLong_AsUnsignedLongLongMask(seed);
    return true;
}

void* current_stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor empty2(int64_t rows, int64_t cols, at::ScalarType dtype, at::Device dev)
{
    const int64_t size[2] = {rows, cols};
    return at::detail::empty_cuda(at::IntArrayRef(size, 2), dtype, dev, std::nullopt);
}

// the result object of a call that was made: `owned` (a new tensor) or the caller's `out`; NULL with GrassError set
PyObject* finish(grass_status rc, const char* where, PyObject* out, at::Tensor& made)
{
    if (rc != GRASS_OK) {
        PyObject* e = PyObject_CallFunction(api.error, "is", (int)rc, where);
        if (e) {
            PyErr_SetObject(api.error, e);
            Py_DECREF(e);
        }
        return nullptr;
    }
    if (out != Py_None) return Py_NewRef(out);
    return THPVariable_Wrap(std::move(made));
}

// the rows of `out` (NULL: not ordinary, the Python path decides); makes one of rows x cols where it is None
const at::Tensor* out_rows(PyObject* out, int64_t rows, int64_t cols, at::ScalarType dtype, at::Device dev,
                           at::Tensor* made)
{
    if (out == Py_None) {
        *made = empty2(rows, cols, dtype, dev);
        return made;
    }
    const at::Tensor* t = as_tensor(out);
    if (!t || !is_cuda(*t) || t->dim() != 2 || t->stride(1) != 1) return nullptr;
    return t;
}

// Scratch that the library can do without: none where the pool has no more to give.  It comes from torch's stream-ordered pool
// of the device whose current stream the call is enqueued on, so it may be handed out again as soon as this tensor is gone, to
// work that is enqueued behind the kernels that use it.
void* optional_scratch(size_t* bytes, at::Tensor* keep)
{
    if (*bytes == 0) return nullptr;
    try {
        *keep = empty2(1, (int64_t)*bytes, at::kByte, at::Device(at::kCUDA, c10::cuda::current_device()));
        return keep->data_ptr();
    } catch (const c10::OutOfMemoryError&) {
        *bytes = 0;
        return nullptr;
    }
}

#define ORDINARY(cond) do { if (!(cond)) Py_RETURN_NONE; } while (0)
#define GUARD_BEGIN try {
// as torch reports them: an allocation that fails is torch.OutOfMemoryError
#define GUARD_END                                                           \
    } catch (const std::exception&) {                                       \
        torch::translate_exception_to_python(std::current_exception());     \
        return nullptr;                                                     \
    }

// grass_compress(g, idx, k, s, seed, out, p, dev_status, out_dtype)
PyObject* py_grass_compress(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 9);
    const at::Tensor* g = as_tensor(a[0]);
    int dt, odt;
    const uint32_t* idx;
    int64_t kprime;
    grass_sjlt_spec sp;
    uint32_t* dev_status;
    ORDINARY(g && is_cuda(*g) && g->dim() == 2 && g->stride(1) == 1 && elem_dtype(*g, &dt));
    ORDINARY(mask_list(a[1], true, &idx, &kprime) && sjlt_spec(a[2], a[3], a[4], &sp) && status_word(a[7], &dev_status));
    ORDINARY(THPDtype_Check(a[8]));
    const int64_t rows = g->size(0), ld = rows > 1 ? g->stride(0) : g->size(1);
    int64_t p = g->size(1);
    ORDINARY(a[6] == Py_None || as_int(a[6], &p));
    if (a[1] == Py_None) kprime = p;
    at::Tensor made;
    const at::Tensor* o = out_rows(a[5], rows, sp.k, reinterpret_cast<THPDtype*>(a[8])->scalar_type, g->device(), &made);
    ORDINARY(o && elem_dtype(*o, &odt));
    const int64_t ld_out = rows > 1 ? o->stride(0) : std::max<int64_t>(o->size(1), sp.k);
    void* const st = current_stream();
    const void* gp = g->const_data_ptr();
    void* op = o->data_ptr();
    at::Tensor scratch;
    size_t wbytes = idx ? 0 : api.compress_bytes((grass_dtype)dt, rows, p, idx, &sp);
    void* const wp = optional_scratch(&wbytes, &scratch);
    grass_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = api.compress(gp, (grass_dtype)dt, rows, p, ld, idx, kprime, &sp, op, (grass_dtype)odt, ld_out, wp, wbytes, dev_status, st);
    Py_END_ALLOW_THREADS
    return finish(rc, "grass_compress", a[5], made);
    GUARD_END
}

// factgrass_compress(A, G, mask_in, mask_out, k, s, seed, out, dev_status)
PyObject* py_factgrass_compress(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 9);
    const at::Tensor *A = as_tensor(a[0]), *G = as_tensor(a[1]);
    int dt;
    const uint32_t *mi, *mo;
    int64_t kin, kout;
    grass_sjlt_spec sp;
    uint32_t* dev_status;
    ORDINARY(A && G && is_cuda(*A) && is_cuda(*G) && A->dim() == 3 && G->dim() == 3 && A->is_contiguous() && G->is_contiguous());
    ORDINARY(A->scalar_type() == G->scalar_type() && elem_dtype(*A, &dt) && A->size(0) == G->size(0) && A->size(1) == G->size(1));
    ORDINARY(mask_list(a[2], false, &mi, &kin) && mask_list(a[3], false, &mo, &kout));
    ORDINARY(sjlt_spec(a[4], a[5], a[6], &sp) && status_word(a[8], &dev_status));
    const int64_t B = A->size(0), T = A->size(1), d_in = A->size(2), d_out = G->size(2);
    ORDINARY(B <= INT32_MAX && T <= INT32_MAX && d_in <= INT32_MAX && d_out <= INT32_MAX && kin <= INT32_MAX && kout <= INT32_MAX);
    at::Tensor made;
    const at::Tensor* o = out_rows(a[7], B, sp.k, at::kFloat, A->device(), &made);
    ORDINARY(o && o->scalar_type() == at::kFloat);
    const int64_t ld_out = B > 1 ? o->stride(0) : std::max<int64_t>(o->size(1), sp.k);
    void* const st = current_stream();
    const void *ap = A->const_data_ptr(), *gp = G->const_data_ptr();
    float* op = static_cast<float*>(o->data_ptr());
    at::Tensor scratch;
    size_t wbytes = api.layer_bytes((grass_dtype)dt, (int32_t)B, (int32_t)T, (int32_t)kin, (int32_t)kout, &sp);
    void* const wp = optional_scratch(&wbytes, &scratch);
    const factgrass_layer layer = {ap, gp, mi, mo, (int32_t)d_in, (int32_t)d_out, (int32_t)kin, (int32_t)kout, sp, 0};
    grass_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = api.grouped_out(&layer, 1, (grass_dtype)dt, (int32_t)B, (int32_t)T, op, GRASS_F32, ld_out, wp, wbytes, dev_status, st);
    Py_END_ALLOW_THREADS
    return finish(rc, "factgrass_compress", a[7], made);
    GUARD_END
}

// None, or a contiguous list of B entries of the given type
bool token_list(PyObject* o, at::ScalarType dtype, int64_t B, const void** p)
{
    *p = nullptr;
    if (o == Py_None) return true;
    const at::Tensor* t = as_tensor(o);
    if (!t || !is_cuda(*t) || t->scalar_type() != dtype || t->numel() != B || !t->is_contiguous()) return false;
    *p = t->const_data_ptr();
    return true;
}

// factgrass_compress_varlen(A, G, mask_in, mask_out, k, s, seed, B, T_max, tok_begin, tok_count, out, dev_status)
PyObject* py_factgrass_compress_varlen(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 13);
    const at::Tensor *A = as_tensor(a[0]), *G = as_tensor(a[1]);
    int dt;
    const uint32_t *mi, *mo;
    int64_t kin, kout, B, T;
    grass_sjlt_spec sp;
    uint32_t* dev_status;
    const void *tb, *tcnt;
    ORDINARY(A && G && is_cuda(*A) && is_cuda(*G) && A->dim() >= 1 && G->dim() >= 1 && A->is_contiguous() && G->is_contiguous());
    ORDINARY(A->scalar_type() == G->scalar_type() && elem_dtype(*A, &dt));
    ORDINARY(mask_list(a[2], false, &mi, &kin) && mask_list(a[3], false, &mo, &kout));
    ORDINARY(sjlt_spec(a[4], a[5], a[6], &sp) && as_int(a[7], &B) && as_int(a[8], &T) && status_word(a[12], &dev_status));
    ORDINARY(B >= 0 && B <= INT32_MAX && T >= 0 && T <= INT32_MAX);
    ORDINARY(token_list(a[9], at::kLong, B, &tb) && token_list(a[10], at::kInt, B, &tcnt));
    const int64_t d_in = A->size(-1), d_out = G->size(-1);
    ORDINARY(d_in <= INT32_MAX && d_out <= INT32_MAX && kin <= INT32_MAX && kout <= INT32_MAX);
    ORDINARY(tb || (A->numel() >= B * T * d_in && G->numel() >= B * T * d_out));
    at::Tensor made;
    const at::Tensor* o = out_rows(a[11], B, sp.k, at::kFloat, A->device(), &made);
    ORDINARY(o && o->scalar_type() == at::kFloat);
    const int64_t ld_out = B > 1 ? o->stride(0) : std::max<int64_t>(o->size(1), sp.k);
    void* const st = current_stream();
    const void *ap = A->const_data_ptr(), *gp = G->const_data_ptr();
    float* op = static_cast<float*>(o->data_ptr());
    grass_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = api.factgrass_varlen(ap, gp, (grass_dtype)dt, (int32_t)B, (int32_t)T, (const int64_t*)tb, (const int32_t*)tcnt,
                              (int32_t)d_in, (int32_t)d_out, mi, (int32_t)kin, mo, (int32_t)kout, &sp, op, ld_out,
                              dev_status, st);
    Py_END_ALLOW_THREADS
    return finish(rc, "factgrass_compress_varlen", a[11], made);
    GUARD_END
}

// Interned keys of the layer dicts.
enum { K_A, K_G, K_MASK_IN, K_MASK_OUT, K_K, K_S, K_SEED, K_OFF, K_COUNT };
PyObject* keys[K_COUNT];

// fill_layers(layers, address of a factgrass_layer array) -> (dtype, B, T), or None
PyObject* py_fill_layers(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 2 && PyList_CheckExact(a[0]) && PyLong_CheckExact(a[1]));
    auto* table = static_cast<factgrass_layer*>(PyLong_AsVoidPtr(a[1]));
    const Py_ssize_t L = PyList_GET_SIZE(a[0]);
    ORDINARY(table && L > 0);
    const at::Tensor* A0 = nullptr;
    int dt = 0;
    for (Py_ssize_t i = 0; i < L; ++i) {
        PyObject* d = PyList_GET_ITEM(a[0], i);
        ORDINARY(PyDict_CheckExact(d));
        PyObject* v[K_COUNT];
        for (int q = 0; q < K_COUNT; ++q) {
            v[q] = PyDict_GetItemWithError(d, keys[q]);     // borrowed
            if (!v[q]) {
                PyErr_Clear();
                Py_RETURN_NONE;
            }
        }
        const at::Tensor *A = as_tensor(v[K_A]), *G = as_tensor(v[K_G]);
        ORDINARY(A && G && is_cuda(*A) && is_cuda(*G) && A->is_contiguous() && G->is_contiguous());
        if (i == 0) {
            A0 = A;
            ORDINARY(A->dim() >= 2 && elem_dtype(*A, &dt));
        }
        // every layer shares the token layout and dtype of the first; the kernels index with these
        const int64_t nd = A0->dim();
        ORDINARY(A->dim() == nd && G->dim() == nd && A->scalar_type() == A0->scalar_type() && G->scalar_type() == A0->scalar_type());
        for (int64_t q = 0; q + 1 < nd; ++q) ORDINARY(A->size(q) == A0->size(q) && G->size(q) == A0->size(q));
        const uint32_t *mi, *mo;
        int64_t kin, kout, off;
        ORDINARY(mask_list(v[K_MASK_IN], false, &mi, &kin) && mask_list(v[K_MASK_OUT], false, &mo, &kout));
        ORDINARY(as_int(v[K_OFF], &off) && off >= 0);
        factgrass_layer& l = table[i];
        ORDINARY(sjlt_spec(v[K_K], v[K_S], v[K_SEED], &l.spec));
        const int64_t d_in = A->size(-1), d_out = G->size(-1);
        ORDINARY(d_in <= INT32_MAX && d_out <= INT32_MAX && kin <= INT32_MAX && kout <= INT32_MAX);
        l.A = A->const_data_ptr();
        l.G = G->const_data_ptr();
        l.mask_in = mi;
        l.mask_out = mo;
        l.d_in = (int32_t)d_in;
        l.d_out = (int32_t)d_out;
        l.kin = (int32_t)kin;
        l.kout = (int32_t)kout;
        l.out_offset = off;
    }
    return Py_BuildValue("iLL", dt, (long long)A0->size(0), (long long)A0->size(1));
    GUARD_END
}

// the arguments every grouped call shares
bool grouped_args(PyObject* table, PyObject* L, PyObject* dt, PyObject* B, PyObject* T, int64_t (&v)[4], const factgrass_layer** t)
{
    if (!PyLong_CheckExact(table) || !as_int(L, &v[0]) || !as_int(dt, &v[1]) || !as_int(B, &v[2]) || !as_int(T, &v[3])) return false;
    for (int64_t x : v)
        if (x < INT32_MIN || x > INT32_MAX) return false;
    *t = static_cast<const factgrass_layer*>(PyLong_AsVoidPtr(table));
    return true;
}

// factgrass_compress_grouped(table, L, dtype, B, T, out, workspace, dev_status)
PyObject* py_grouped(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 8);
    int64_t v[4];
    const factgrass_layer* t;
    const at::Tensor *o = as_tensor(a[5]), *w = as_tensor(a[6]);
    uint32_t* dev_status;
    int odt;
    ORDINARY(grouped_args(a[0], a[1], a[2], a[3], a[4], v, &t) && status_word(a[7], &dev_status));
    ORDINARY(o && w && is_cuda(*o) && is_cuda(*w) && o->dim() == 2 && o->stride(1) == 1 && elem_dtype(*o, &odt));
    const int64_t ld_out = o->size(0) > 1 ? o->stride(0) : o->size(1);
    void *op = o->data_ptr(), *wp = w->data_ptr(), *st = current_stream();
    const size_t wbytes = (size_t)w->numel() * w->element_size();
    grass_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = api.grouped_out(t, (int32_t)v[0], (grass_dtype)v[1], (int32_t)v[2], (int32_t)v[3], op, (grass_dtype)odt, ld_out,
                         wp, wbytes, dev_status, st);
    Py_END_ALLOW_THREADS
    at::Tensor none;
    return finish(rc, "factgrass_compress_grouped", a[5], none);
    GUARD_END
}

// factgrass_compress_grouped_varlen(table, L, dtype, B, T_max, out, workspace, tok_begin, tok_count, dev_status)
PyObject* py_grouped_varlen(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 10);
    int64_t v[4];
    const factgrass_layer* t;
    const at::Tensor *o = as_tensor(a[5]), *w = as_tensor(a[6]);
    uint32_t* dev_status;
    const void *tb, *tcnt;
    ORDINARY(grouped_args(a[0], a[1], a[2], a[3], a[4], v, &t) && status_word(a[9], &dev_status));
    ORDINARY(o && w && is_cuda(*o) && is_cuda(*w) && o->dim() == 2 && o->stride(1) == 1 && o->scalar_type() == at::kFloat &&
             o->size(0) == v[2]);
    ORDINARY(token_list(a[7], at::kLong, v[2], &tb) && token_list(a[8], at::kInt, v[2], &tcnt));
    const int64_t ld_out = o->size(0) > 1 ? o->stride(0) : o->size(1);
    float* op = static_cast<float*>(o->data_ptr());
    void *wp = w->data_ptr(), *st = current_stream();
    const size_t wbytes = (size_t)w->numel() * w->element_size();
    grass_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = api.grouped_varlen(t, (int32_t)v[0], (grass_dtype)v[1], (int32_t)v[2], (int32_t)v[3], (const int64_t*)tb,
                            (const int32_t*)tcnt, op, ld_out, wp, wbytes, dev_status, st);
    Py_END_ALLOW_THREADS
    at::Tensor none;
    return finish(rc, "factgrass_compress_grouped_varlen", a[5], none);
    GUARD_END
}

// grass_score(train, test, out) and grass_score_bf16(train, test, out)
template <bool BF16>
PyObject* py_score(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GUARD_BEGIN
    ORDINARY(n == 3);
    constexpr auto want = BF16 ? at::kBFloat16 : at::kFloat;
    const at::Tensor *tr = as_tensor(a[0]), *te = as_tensor(a[1]);
    ORDINARY(tr && te && is_cuda(*tr) && is_cuda(*te) && tr->dim() == 2 && te->dim() == 2);
    ORDINARY(tr->scalar_type() == want && te->scalar_type() == want && tr->stride(1) == 1 && te->stride(1) == 1);
    const int64_t N = tr->size(0), D = tr->size(1), M = te->size(0);
    ORDINARY(te->size(1) == D);
    at::Tensor made;
    const at::Tensor* o = out_rows(a[2], N, M, at::kFloat, tr->device(), &made);
    ORDINARY(o && o->scalar_type() == at::kFloat);
    const int64_t ldt = N > 1 ? tr->stride(0) : D, lde = M > 1 ? te->stride(0) : D, lds = N > 1 ? o->stride(0) : M;
    void* st = current_stream();
    const void *tp = tr->const_data_ptr(), *ep = te->const_data_ptr();
    float* op = static_cast<float*>(o->data_ptr());
    grass_status rc;
    Py_BEGIN_ALLOW_THREADS
    if (BF16) rc = api.score_bf16(tp, N, ldt, ep, M, lde, D, op, lds, st);
    else rc = api.score((const float*)tp, N, ldt, (const float*)ep, M, lde, D, op, lds, st);
    Py_END_ALLOW_THREADS
    return finish(rc, BF16 ? "grass_score_bf16" : "grass_score", a[2], made);
    GUARD_END
}

// bind(GrassError, addresses...): the library's entry points, in the order of struct Api
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    void* p[8];
    if (n != 9) {
        PyErr_SetString(PyExc_TypeError, "bind(GrassError, 8 addresses)");
        return nullptr;
    }
    for (int i = 0; i < 8; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i + 1]);
        if (PyErr_Occurred()) return nullptr;
    }
    api.compress = (decltype(api.compress))p[0];
    api.compress_bytes = (decltype(api.compress_bytes))p[7];
    api.layer_bytes = (decltype(api.layer_bytes))p[1];
    api.factgrass_varlen = (decltype(api.factgrass_varlen))p[2];
    api.grouped_out = (decltype(api.grouped_out))p[3];
    api.grouped_varlen = (decltype(api.grouped_varlen))p[4];
    api.score = (decltype(api.score))p[5];
    api.score_bf16 = (decltype(api.score_bf16))p[6];
    Py_XSETREF(api.error, Py_NewRef(a[0]));
    Py_RETURN_NONE;
}

template <typename F>
PyCFunction fast(F f) { return (PyCFunction)(void (*)(void))f; }

PyMethodDef methods[] = {
    {"bind", fast(py_bind), METH_FASTCALL, nullptr},
    {"grass_compress", fast(py_grass_compress), METH_FASTCALL, nullptr},
    {"factgrass_compress", fast(py_factgrass_compress), METH_FASTCALL, nullptr},
    {"factgrass_compress_varlen", fast(py_factgrass_compress_varlen), METH_FASTCALL, nullptr},
    {"fill_layers", fast(py_fill_layers), METH_FASTCALL, nullptr},
    {"factgrass_compress_grouped", fast(py_grouped), METH_FASTCALL, nullptr},
    {"factgrass_compress_grouped_varlen", fast(py_grouped_varlen), METH_FASTCALL, nullptr},
    {"grass_score", fast(py_score<false>), METH_FASTCALL, nullptr},
    {"grass_score_bf16", fast(py_score<true>), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    static const char* const names[K_COUNT] = {"A", "G", "mask_in", "mask_out", "k", "s", "seed", "out_offset"};
    for (int i = 0; i < K_COUNT; ++i)
        if (!(keys[i] = PyUnicode_InternFromString(names[i]))) return nullptr;
    return PyModule_Create(&module);
}
