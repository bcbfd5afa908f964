// Native half of binding.py: takes the tensors of a call apart, allocates its outputs and calls the C entry point.
//
// A pass over a short history is four calls of five or six launches; marshalling them in Python (some twenty tensor and stream
// queries and a ctypes conversion per call) took 65 to 75 us of host time per pass, longer than the kernels.  Positional
// arguments in the order of binding.py's signatures; checks and errors are the same, and so is the absence of any fallback.
#include <Python.h>

#include <dlfcn.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <string>
#include <vector>

#include "../../include/janus.h"

// read by build.py: the library is built again when torch or the interpreter is another
extern "C" __attribute__((used, visibility("default"))) const char janus_native_mark[] = JANUS_NATIVE_MARK;

namespace {

// ---- state set once by init(): the C entry points and the Python objects the calls need
struct Api {
    decltype(&janus_indexer_scores) indexer_scores;
    decltype(&janus_topk) topk;
    decltype(&janus_indexer_topk_workspace_size) indexer_topk_workspace_size;
    decltype(&janus_indexer_topk) indexer_topk;
    decltype(&janus_page_demand) page_demand;
    decltype(&janus_page_union) page_union;
    decltype(&janus_sparse_attn_prefill) sparse_attn_prefill;
    decltype(&janus_topk_entries) topk_entries;
    decltype(&janus_entry_pool_scores) entry_pool_scores;
    decltype(&janus_entry_expand) entry_expand;
    decltype(&janus_indexer_scores_batch) indexer_scores_batch;
    decltype(&janus_topk_batch) topk_batch;
    decltype(&janus_page_demand_batch) page_demand_batch;
    decltype(&janus_sparse_attn_decode) sparse_attn_decode;
    decltype(&janus_last_cuda_error) last_cuda_error;
} api;
PyObject* janus_error = nullptr;        // exception class
PyObject* status_tensor_fn = nullptr;   // binding.dev_status_tensor
auto& status_words = *new std::vector<at::Tensor>;   // by device, as binding.dev_status_tensor made them; never destroyed (outlives CUDA's own teardown)
PyObject *key_bitmap, *key_pages, *key_runs, *key_counts, *key_miss_pages, *key_miss_runs;

struct PyError {};                      // a Python exception is set
[[noreturn]] void fail(PyObject* type, const std::string& what) {
    PyErr_SetString(type, what.c_str());
    throw PyError{};
}

// ---- arguments
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a tensor");
    return THPVariable_Unpack(o);
}
void* ptr(const at::Tensor& t) {
    if (!t.is_cuda()) fail(janus_error, "expected a CUDA tensor (the library takes device pointers)");
    return t.data_ptr();
}
void* ptr_or_null(PyObject* o) { return o == Py_None ? nullptr : ptr(tensor(o)); }
int64_t integer(PyObject* o) {
    if (PyLong_CheckExact(o)) {
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) throw PyError{};
        return v;
    }
    PyObject* n = PyNumber_Long(o);
    if (n == nullptr) throw PyError{};
    const long long v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw PyError{};
    return v;
}
// A size of something this call allocates: whole numbers only, as for any tensor's shape.
int64_t size(PyObject* o) {
    PyObject* n = PyNumber_Index(o);
    if (n == nullptr) throw PyError{};
    const long long v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw PyError{};
    return v;
}
double number(PyObject* o) {
    PyObject* f = PyNumber_Float(o);
    if (f == nullptr) throw PyError{};
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return v;
}
bool truth(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw PyError{};
    return v != 0;
}
void want_dims(const at::Tensor& t, int64_t n, const char* name) {
    if (t.dim() != n) fail(PyExc_ValueError, std::string(name) + " must have " + std::to_string(n) + " dimensions, not " + std::to_string(t.dim()));
}
const at::Tensor& item(PyObject* dict, PyObject* key, at::Tensor& hold) {
    PyObject* o = PyObject_GetItem(dict, key);
    if (o == nullptr) throw PyError{};
    if (!THPVariable_Check(o)) {
        Py_DECREF(o);
        fail(PyExc_TypeError, "expected a tensor");
    }
    hold = THPVariable_Unpack(o);
    Py_DECREF(o);
    return hold;
}

// ---- what every call passes along
int32_t* status_word() {
    const int dev = c10::cuda::current_device();
    if (static_cast<size_t>(dev) >= status_words.size()) status_words.resize(dev + 1);
    if (!status_words[dev].defined()) {
        PyObject* t = PyObject_CallNoArgs(status_tensor_fn);
        if (t == nullptr) throw PyError{};
        status_words[dev] = THPVariable_Unpack(t);
        Py_DECREF(t);
    }
    return static_cast<int32_t*>(status_words[dev].data_ptr());
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor make(at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) { return at::empty(shape, like.options().dtype(type)); }
PyObject* wrap(at::Tensor t) { return THPVariable_Wrap(std::move(t)); }
PyObject* none() { return Py_NewRef(Py_None); }

PyObject* triple(PyObject* a, const at::Tensor& b, const at::Tensor& c) {      // b, c undefined -> None; steals a
    PyObject* t = PyTuple_New(3);
    PyTuple_SET_ITEM(t, 0, a);
    PyTuple_SET_ITEM(t, 1, b.defined() ? wrap(b) : none());
    PyTuple_SET_ITEM(t, 2, c.defined() ? wrap(c) : none());
    return t;
}

void check(int rc, const char* what) {
    if (rc == JANUS_OK) return;
    static const char* names[] = {"", "JANUS_ERR_INVALID_ARG", "JANUS_ERR_UNSUPPORTED", "JANUS_ERR_WORKSPACE_TOO_SMALL", "JANUS_ERR_CUDA"};
    std::string text = std::string(what) + " failed: " + (rc >= 1 && rc <= 4 ? names[rc] : std::to_string(rc));
    if (rc == JANUS_ERR_CUDA) text += " (cudaError " + std::to_string(api.last_cuda_error()) + ")";
    fail(janus_error, text);
}

// Calls a C entry point without the GIL (a full launch queue blocks).
template <class F, class... A>
void call(const char* what, F f, A... a) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f(a...);
    Py_END_ALLOW_THREADS
    check(rc, what);
}

int idx_dtype_code(const at::Tensor& t) {
    if (t.scalar_type() == at::kBFloat16) return JANUS_DTYPE_BF16;
    if (t.scalar_type() == at::kByte || t.scalar_type() == at::kFloat8_e4m3fn) return JANUS_DTYPE_FP8_E4M3;
    fail(janus_error, std::string("indexer operands must be bfloat16 or E4M3 bytes, got ") + c10::toString(t.scalar_type()));
}
struct IdxDtypes {
    int code;
    int64_t k_stride;
};
IdxDtypes idx_dtypes(const at::Tensor& q, const at::Tensor& k, bool fp4) {
    const int code = idx_dtype_code(q);
    if (fp4) {
        if (code != JANUS_DTYPE_FP8_E4M3 || k.scalar_type() != at::kByte) fail(janus_error, "FP4 keys are uint8 (two per byte) and go with E4M3 queries");
        return {JANUS_DTYPE_FP8_Q_FP4_K, k.stride(0) * 2};
    }
    if (idx_dtype_code(k) != code) fail(janus_error, "q_idx and k_idx must share a dtype");
    return {code, k.stride(0)};
}
int64_t q_scale_stride(PyObject* q_scale, int64_t H) { return q_scale != Py_None && tensor(q_scale).dim() == 2 ? H : 0; }
int i32(int64_t v) { return static_cast<int>(v); }
template <class T>
T* as(void* p) { return static_cast<T*>(p); }

// ---- the calls: (arguments in the order of binding.py) -> new reference
using Args = PyObject* const*;

PyObject* indexer_scores(Args a) {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]);
    want_dims(q, 3, "q_idx");
    const int64_t M = q.size(0), H = q.size(1), D = q.size(2), n_keys = k.size(0);
    const IdxDtypes dt = idx_dtypes(q, k, truth(a[10]));
    at::Tensor scores = a[9] == Py_None ? make({M, (n_keys + 31) / 32 * 32}, at::kFloat, q) : tensor(a[9]);
    call("janus_indexer_scores", api.indexer_scores, ptr(q), q.stride(0), ptr(k), dt.k_stride, as<const float>(ptr_or_null(a[2])),
         as<const float>(ptr_or_null(a[3])), q_scale_stride(a[3], H), as<const float>(ptr_or_null(a[4])), as<const float>(ptr_or_null(a[5])),
         as<const float>(ptr_or_null(a[6])), i32(M), i32(H), i32(D), n_keys, integer(a[7]), i32(truth(a[8])), dt.code, as<float>(ptr(scores)),
         scores.stride(0), nullptr, size_t(0), status_word(), stream());
    return a[9] == Py_None ? wrap(scores) : Py_NewRef(a[9]);
}

PyObject* topk(Args a) {
    const at::Tensor& scores = tensor(a[0]);
    const int64_t M = scores.size(0), k = a[7] == Py_None ? size(a[2]) : integer(a[2]);
    at::Tensor idx = a[7] == Py_None ? make({M, k}, at::kInt, scores) : tensor(a[7]), count, kth;
    if (truth(a[5])) count = make({M}, at::kInt, scores);
    if (truth(a[6])) kth = make({M}, at::kFloat, scores);
    call("janus_topk", api.topk, as<const float>(ptr(scores)), scores.stride(0), i32(M), integer(a[1]), integer(a[3]), i32(truth(a[4])), i32(k),
         as<int32_t>(ptr(idx)), as<int32_t>(count.defined() ? ptr(count) : nullptr), as<float>(kth.defined() ? ptr(kth) : nullptr), nullptr, size_t(0),
         status_word(), stream());
    return triple(a[7] == Py_None ? wrap(idx) : Py_NewRef(a[7]), count, kth);
}

PyObject* indexer_topk(Args a) {
    const at::Tensor &q = tensor(a[0]), &k_idx = tensor(a[1]);
    want_dims(q, 3, "q_idx");
    const int64_t M = q.size(0), H = q.size(1), D = q.size(2), n_keys = k_idx.size(0), k = a[13] == Py_None ? size(a[3]) : integer(a[3]), q_pos0 = integer(a[8]);
    const IdxDtypes dt = idx_dtypes(q, k_idx, truth(a[14]));
    const int causal = i32(truth(a[9]));
    const size_t need = api.indexer_topk_workspace_size(i32(M), i32(H), i32(D), n_keys, q_pos0, causal, dt.code, i32(k));
    at::Tensor ws;
    if (a[12] != Py_None) ws = tensor(a[12]);
    if (!ws.defined() || ws.numel() < static_cast<int64_t>(need)) ws = make({static_cast<int64_t>(need > 16 ? need : 16)}, at::kByte, q);
    at::Tensor idx, count, kth;
    if (a[13] == Py_None) {
        idx = make({M, k}, at::kInt, q);
    } else {
        idx = tensor(a[13]);
        if (idx.dim() != 2 || idx.size(0) != M || idx.size(1) != k || number(a[3]) != static_cast<double>(k) || idx.scalar_type() != at::kInt || !idx.is_contiguous())
            fail(janus_error, "idx must be a contiguous [M, k] int32 tensor");
    }
    if (truth(a[10])) count = make({M}, at::kInt, q);
    if (truth(a[11])) kth = make({M}, at::kFloat, q);
    call("janus_indexer_topk", api.indexer_topk, ptr(q), q.stride(0), ptr(k_idx), dt.k_stride, as<const float>(ptr_or_null(a[2])),
         as<const float>(ptr_or_null(a[4])), q_scale_stride(a[4], H), as<const float>(ptr_or_null(a[5])), as<const float>(ptr_or_null(a[6])),
         as<const float>(ptr_or_null(a[7])), i32(M), i32(H), i32(D), n_keys, q_pos0, causal, dt.code, i32(k), as<int32_t>(ptr(idx)),
         as<int32_t>(count.defined() ? ptr(count) : nullptr), as<float>(kth.defined() ? ptr(kth) : nullptr), ptr(ws), static_cast<size_t>(ws.numel()),
         status_word(), stream());
    return triple(a[13] == Py_None ? wrap(idx) : Py_NewRef(a[13]), count, kth);
}

// Output buffers of a page-demand call: the dict of page_demand_buffers().
struct PageOut {
    at::Tensor bitmap, pages, runs, counts, miss_pages, miss_runs;
    int32_t *n_pages, *n_runs, *miss_p = nullptr, *n_miss = nullptr, *miss_r = nullptr, *n_miss_runs = nullptr;
    int64_t capacity;
    PageOut(PyObject* out, PyObject* cap, bool want_miss) {
        item(out, key_bitmap, bitmap);
        item(out, key_pages, pages);
        item(out, key_runs, runs);
        item(out, key_counts, counts);
        n_pages = as<int32_t>(counts.data_ptr());
        n_runs = n_pages + 1;
        const int has = want_miss ? PySequence_Contains(out, key_miss_pages) : 0;
        if (has < 0) throw PyError{};
        if (has) {
            miss_p = as<int32_t>(ptr(item(out, key_miss_pages, miss_pages)));
            n_miss = n_pages + 2;
            miss_r = as<int32_t>(ptr(item(out, key_miss_runs, miss_runs)));
            n_miss_runs = n_pages + 3;
        }
        capacity = cap == Py_None ? pages.numel() : integer(cap);
    }
};

PyObject* page_demand(Args a) {       // idx, demand_limit, page_size, page_table, n_phys_pages, predicted, capacity, want_miss, out
    const at::Tensor &idx = tensor(a[0]), &table = tensor(a[3]);
    want_dims(idx, 2, "idx");
    PageOut o(a[8], a[6], truth(a[7]));
    call("janus_page_demand", api.page_demand, as<const int32_t>(ptr(idx)), idx.size(0), i32(idx.size(1)), integer(a[1]), i32(integer(a[2])),
         as<const int32_t>(ptr(table)), table.numel(), integer(a[4]), as<const uint32_t>(ptr_or_null(a[5])), as<uint32_t>(ptr(o.bitmap)),
         as<int32_t>(ptr(o.pages)), o.n_pages, as<int32_t>(ptr(o.runs)), o.n_runs, o.miss_p, o.n_miss, o.miss_r, o.n_miss_runs, o.capacity, nullptr,
         size_t(0), status_word(), stream());
    return Py_NewRef(a[8]);
}

PyObject* page_demand_batch(Args a) { // idx, demand_limits, page_size, page_tables, table_offsets, n_phys_pages, predicted, capacity, want_miss, out
    const at::Tensor& idx = tensor(a[0]);
    want_dims(idx, 2, "idx");
    PageOut o(a[9], a[7], truth(a[8]));
    call("janus_page_demand_batch", api.page_demand_batch, as<const int32_t>(ptr(idx)), idx.size(0), i32(idx.size(1)),
         as<const int64_t>(ptr_or_null(a[1])), i32(integer(a[2])), as<const int32_t>(ptr_or_null(a[3])), as<const int64_t>(ptr_or_null(a[4])),
         integer(a[5]), as<const uint32_t>(ptr_or_null(a[6])), as<uint32_t>(ptr(o.bitmap)), as<int32_t>(ptr(o.pages)), o.n_pages,
         as<int32_t>(ptr(o.runs)), o.n_runs, o.miss_p, o.n_miss, o.miss_r, o.n_miss_runs, o.capacity, status_word(), stream());
    return Py_NewRef(a[9]);
}

PyObject* page_union(Args a) {        // dst, src, n_phys_pages
    call("janus_page_union", api.page_union, as<uint32_t>(ptr_or_null(a[0])), as<const uint32_t>(ptr_or_null(a[1])), integer(a[2]), stream());
    return Py_NewRef(a[0]);
}

// q, k_pool, v_pool, idx, page tables, table offsets (None: prefill), page_size, softmax_scale, d_v, want_lse, out
PyObject* sparse_attn(Args a) {
    const at::Tensor &q = tensor(a[0]), &kp = tensor(a[1]), &vp = tensor(a[2]), &idx = tensor(a[3]), &table = tensor(a[4]);
    want_dims(q, 3, "q");
    const bool batch = a[5] != Py_None;
    const int64_t M = q.size(0), H = q.size(1), d_qk = q.size(2), n_kv = kp.size(2), d_v = a[10] == Py_None ? size(a[8]) : integer(a[8]);
    at::Tensor out = a[10] == Py_None ? make({M, H, d_v}, at::kBFloat16, q) : tensor(a[10]), lse;
    if (truth(a[9])) lse = make({M, H}, at::kFloat, q);
    if (!batch && vp.data_ptr() != kp.data_ptr() && vp.strides() != kp.strides()) fail(janus_error, "k_pool and v_pool must share strides");
    float* lse_p = lse.defined() ? as<float>(ptr(lse)) : nullptr;
    if (batch)
        call("janus_sparse_attn_decode", api.sparse_attn_decode, ptr(q), i32(M), i32(H), i32(d_qk), ptr(kp), ptr(vp), kp.stride(0), kp.stride(1),
             kp.stride(2), i32(n_kv), i32(d_v), as<const int32_t>(ptr(idx)), i32(idx.size(1)), i32(integer(a[6])), as<const int32_t>(ptr(table)),
             as<const int64_t>(ptr_or_null(a[5])), static_cast<float>(number(a[7])), ptr(out), lse_p, status_word(), stream());
    else
        call("janus_sparse_attn_prefill", api.sparse_attn_prefill, ptr(q), i32(M), i32(H), i32(d_qk), ptr(kp), ptr(vp), kp.stride(0), kp.stride(1),
             kp.stride(2), i32(n_kv), i32(d_v), as<const int32_t>(ptr(idx)), i32(idx.size(1)), i32(integer(a[6])), as<const int32_t>(ptr(table)),
             table.numel(), static_cast<float>(number(a[7])), ptr(out), lse_p, nullptr, size_t(0), status_word(), stream());
    PyObject* t = PyTuple_New(2);
    PyTuple_SET_ITEM(t, 0, a[10] == Py_None ? wrap(out) : Py_NewRef(a[10]));
    PyTuple_SET_ITEM(t, 1, lse.defined() ? wrap(lse) : none());
    return t;
}

PyObject* topk_entries(Args a) {      // scores, n_entries, k, q_pos0, entry_size, want_count, want_kth
    const at::Tensor& scores = tensor(a[0]);
    const int64_t M = scores.size(0), k = size(a[2]);
    at::Tensor idx = make({M, k}, at::kInt, scores), count, kth;
    if (truth(a[5])) count = make({M}, at::kInt, scores);
    if (truth(a[6])) kth = make({M}, at::kFloat, scores);
    call("janus_topk_entries", api.topk_entries, as<const float>(ptr(scores)), scores.stride(0), i32(M), integer(a[1]), integer(a[3]),
         i32(integer(a[4])), i32(k), as<int32_t>(ptr(idx)), as<int32_t>(count.defined() ? ptr(count) : nullptr),
         as<float>(kth.defined() ? ptr(kth) : nullptr), status_word(), stream());
    return triple(wrap(idx), count, kth);
}

PyObject* entry_pool_scores(Args a) { // scores, n_keys, entry_size, q_pos0, causal
    const at::Tensor& scores = tensor(a[0]);
    const int64_t M = scores.size(0), n_keys = integer(a[1]), entry = size(a[2]);
    if (entry == 0) fail(PyExc_ZeroDivisionError, "entry_size is zero");
    const int64_t n_entries = (n_keys + entry - 1) / entry, ld = n_entries > 4 ? (n_entries + 3) / 4 * 4 : 4;
    at::Tensor out = make({M, ld}, at::kFloat, scores);
    call("janus_entry_pool_scores", api.entry_pool_scores, as<const float>(ptr(scores)), scores.stride(0), i32(M), n_keys, integer(a[3]),
         i32(truth(a[4])), i32(entry), as<float>(ptr(out)), ld, stream());
    return wrap(out);
}

PyObject* entry_expand(Args a) {      // idx_entries, q_pos0, entry_size
    const at::Tensor& e = tensor(a[0]);
    want_dims(e, 2, "idx_entries");
    const int64_t M = e.size(0), k_e = e.size(1), entry = size(a[2]);
    at::Tensor out = make({M, k_e * entry}, at::kInt, e);
    call("janus_entry_expand", api.entry_expand, as<const int32_t>(ptr(e)), i32(M), i32(k_e), i32(entry), integer(a[1]), as<int32_t>(ptr(out)), stream());
    return wrap(out);
}

PyObject* indexer_scores_batch(Args a) {      // q, k, w, key_offsets, max_keys, q_scale, k_scale, row_bias, col_bias, scores, keys_fp4
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]);
    want_dims(q, 3, "q_idx");
    const int64_t n = q.size(0), H = q.size(1), D = q.size(2), total = k.size(0);
    const bool fp4 = truth(a[10]);
    const int code = fp4 ? JANUS_DTYPE_FP8_Q_FP4_K : idx_dtype_code(q);
    at::Tensor scores = a[9] == Py_None ? make({total}, at::kFloat, q) : tensor(a[9]);
    call("janus_indexer_scores_batch", api.indexer_scores_batch, ptr(q), ptr(k), k.stride(0) * (fp4 ? 2 : 1), as<const float>(ptr_or_null(a[2])),
         as<const float>(ptr_or_null(a[5])), q_scale_stride(a[5], H), as<const float>(ptr_or_null(a[6])), as<const float>(ptr_or_null(a[7])),
         as<const float>(ptr_or_null(a[8])), i32(n), i32(H), i32(D), as<const int64_t>(ptr_or_null(a[3])), total, integer(a[4]), code,
         as<float>(ptr(scores)), status_word(), stream());
    return a[9] == Py_None ? wrap(scores) : Py_NewRef(a[9]);
}

PyObject* topk_batch(Args a) {        // scores, row_offsets, k, row_lengths, want_count, want_kth
    const at::Tensor &scores = tensor(a[0]), &off = tensor(a[1]);
    const int64_t n = off.numel() - 1, k = size(a[2]);
    at::Tensor idx = make({n, k}, at::kInt, scores), count, kth;
    if (truth(a[4])) count = make({n}, at::kInt, scores);
    if (truth(a[5])) kth = make({n}, at::kFloat, scores);
    call("janus_topk_batch", api.topk_batch, as<const float>(ptr(scores)), as<const int64_t>(ptr(off)), as<const int64_t>(ptr_or_null(a[3])), i32(n),
         i32(k), as<int32_t>(ptr(idx)), as<int32_t>(count.defined() ? ptr(count) : nullptr), as<float>(kth.defined() ? ptr(kth) : nullptr),
         status_word(), stream());
    return triple(wrap(idx), count, kth);
}

// ---- module
template <PyObject* (*F)(Args), int N>
PyObject* entry(PyObject*, Args args, Py_ssize_t n) {
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const PyError&) {
    } catch (...) {      // torch's own exceptions by their own names: out of memory, a dimension that is not there
        torch::translate_exception_to_python(std::current_exception());
    }
    return nullptr;
}

PyObject* init(PyObject*, Args args, Py_ssize_t n) {      // path of libjanus.so, exception class, dev_status_tensor
    if (n != 3) {
        PyErr_SetString(PyExc_TypeError, "init(path, error, dev_status_tensor)");
        return nullptr;
    }
    const char* path = PyUnicode_AsUTF8(args[0]);
    if (path == nullptr) return nullptr;
    void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
    if (lib == nullptr) {
        PyErr_SetString(args[1], dlerror());
        return nullptr;
    }
    bool ok = true;
    auto find = [&](auto& f, const char* name) {
        f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(dlsym(lib, name));
        ok = ok && f != nullptr;
    };
    find(api.indexer_scores, "janus_indexer_scores");
    find(api.topk, "janus_topk");
    find(api.indexer_topk_workspace_size, "janus_indexer_topk_workspace_size");
    find(api.indexer_topk, "janus_indexer_topk");
    find(api.page_demand, "janus_page_demand");
    find(api.page_union, "janus_page_union");
    find(api.sparse_attn_prefill, "janus_sparse_attn_prefill");
    find(api.topk_entries, "janus_topk_entries");
    find(api.entry_pool_scores, "janus_entry_pool_scores");
    find(api.entry_expand, "janus_entry_expand");
    find(api.indexer_scores_batch, "janus_indexer_scores_batch");
    find(api.topk_batch, "janus_topk_batch");
    find(api.page_demand_batch, "janus_page_demand_batch");
    find(api.sparse_attn_decode, "janus_sparse_attn_decode");
    find(api.last_cuda_error, "janus_last_cuda_error");
    if (!ok) {
        PyErr_SetString(args[1], "libjanus.so lacks an entry point");
        return nullptr;
    }
    janus_error = Py_NewRef(args[1]);
    status_tensor_fn = Py_NewRef(args[2]);
    return Py_NewRef(Py_None);
}

#define JANUS_METHOD(name, n) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<&name, n>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"init", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&init)), METH_FASTCALL, nullptr},
    JANUS_METHOD(indexer_scores, 11),
    JANUS_METHOD(topk, 8),
    JANUS_METHOD(indexer_topk, 15),
    JANUS_METHOD(page_demand, 9),
    JANUS_METHOD(page_demand_batch, 10),
    JANUS_METHOD(page_union, 3),
    JANUS_METHOD(sparse_attn, 11),
    JANUS_METHOD(topk_entries, 7),
    JANUS_METHOD(entry_pool_scores, 5),
    JANUS_METHOD(entry_expand, 3),
    JANUS_METHOD(indexer_scores_batch, 11),
    JANUS_METHOD(topk_batch, 6),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
    key_bitmap = PyUnicode_InternFromString("bitmap");
    key_pages = PyUnicode_InternFromString("pages");
    key_runs = PyUnicode_InternFromString("runs");
    key_counts = PyUnicode_InternFromString("counts");
    key_miss_pages = PyUnicode_InternFromString("miss_pages");
    key_miss_runs = PyUnicode_InternFromString("miss_runs");
    return PyModule_Create(&module);
}
