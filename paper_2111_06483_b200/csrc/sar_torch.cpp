// Python-facing fast path of api.py: allocates the outputs with torch's allocator and calls libsar's C entry points, in
// native code.  Nothing is computed here; every function is what its counterpart in api.py documents.
//
// Why it exists: a pass over a small graph is a handful of launches of about 5 us each.  Marshalled by ctypes, with
// every output allocated through Python, one layer forward and backward of the tiny workload took 53 us of host time for
// 14 us of kernels.  A call here costs an argument check, an allocation per output (about 0.5 us each) and the launches.
//
// The entry points are looked up in the library that binding.py has loaded, so there is one libsar per process.
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/cuda/CUDAContext.h>
#include <ATen/cuda/EmptyTensor.h>
#include <dlfcn.h>

#include <vector>

#include "sar.h"

namespace {

#define SAR_TABLE(X)                                                                                                   \
    X(sar_status_string) X(sar_gat_workspace_bytes) X(sar_gat_fwd) X(sar_gat_fwd_fused) X(sar_gat_bwd_prepare)         \
    X(sar_gat_bwd) X(sar_gat_bwd_fused) X(sar_spmm_agg) X(sar_spmm_workspace_bytes) X(sar_spmm_agg_scaled)             \
    X(sar_propagate) X(sar_propagate_workspace_bytes_at) X(sar_relu) X(sar_gat_project) X(sar_gat_project_bwd) X(sar_gat_project_workspace_bytes)              \
    X(sar_linear_workspace_bytes) X(sar_linear) X(sar_linear_accumulate) X(sar_linear_project)                         \
    X(sar_linear_bwd_input) X(sar_linear_bwd_input_relu) X(sar_linear_bwd_weight) X(sar_bn_workspace_bytes)            \
    X(sar_bn_stats) X(sar_bn_rstd) X(sar_bn_apply) X(sar_bn_bwd_stats) X(sar_bn_bwd_apply)                             \
    X(sar_graph_workspace_bytes) X(sar_graph_from_coo) X(sar_csr_split_indptr) X(sar_csr_split_indices)                \
    X(sar_csc_slice_indptr) X(sar_plan_many_workspace_bytes) X(sar_plan_count_many) X(sar_plan_fill_many) X(sar_gather_i64)

struct Lib {
#define X(f) decltype(&::f) f;
    SAR_TABLE(X)
#undef X
};
Lib L;
PyObject *g_error = nullptr, *g_oom = nullptr;   // binding.SarError, torch.OutOfMemoryError

// A failed call or check: the Python error is set, the C++ exception unwinds to the entry point.
struct Failed {};

[[noreturn]] void fail(PyObject *type, const char *text) {
    PyErr_SetString(type, text);
    throw Failed{};
}

void check(const char *fn, sar_status s) {
    if (s == SAR_OK) return;
    PyObject *e = g_error ? PyObject_CallFunction(g_error, "sis", fn, (int)s, L.sar_status_string(s)) : nullptr;
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Failed{};
}
#define SAR(fn, ...) check(#fn, L.fn(__VA_ARGS__))

// ---- arguments -----------------------------------------------------------------------------------------------------------
struct Args {
    PyObject *const *a;
    Py_ssize_t n, i = 0;
    PyObject *next() {
        if (i >= n) fail(PyExc_TypeError, "too few arguments");
        return a[i++];
    }
    const at::Tensor &tensor() {
        PyObject *o = next();
        if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a tensor");
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_AssertionError, "libsar takes contiguous CUDA tensors");
        return t;
    }
    at::Tensor optional() {   // a tensor or None
        if (i < n && a[i] == Py_None) {
            ++i;
            return at::Tensor();
        }
        return tensor();
    }
    long long integer() {
        const long long v = PyLong_AsLongLong(next());
        if (v == -1 && PyErr_Occurred()) throw Failed{};
        return v;
    }
    double real() {
        const double v = PyFloat_AsDouble(next());
        if (v == -1.0 && PyErr_Occurred()) throw Failed{};
        return v;
    }
    bool flag() {
        const int v = PyObject_IsTrue(next());
        if (v < 0) throw Failed{};
        return v != 0;
    }
    const sar_part *part() { return reinterpret_cast<const sar_part *>(integer()); }
    std::vector<int64_t> integers() {
        PyObject *s = PySequence_Fast(next(), "expected a sequence of integers");
        if (!s) throw Failed{};
        std::vector<int64_t> v((size_t)PySequence_Fast_GET_SIZE(s));
        for (size_t k = 0; k < v.size(); ++k) v[k] = PyLong_AsLongLong(PySequence_Fast_GET_ITEM(s, (Py_ssize_t)k));
        Py_DECREF(s);
        if (PyErr_Occurred()) throw Failed{};
        return v;
    }
};

sar_dtype code(const at::Tensor &t) {
    if (t.scalar_type() == at::kFloat) return SAR_F32;
    if (t.scalar_type() == at::kBFloat16) return SAR_BF16;
    fail(PyExc_TypeError, "unsupported storage dtype");
}
void require(bool ok, const char *text) {
    if (!ok) fail(PyExc_AssertionError, text);
}
// The library sees a pointer, so what it will read behind it is checked here: the type and at least n elements.
const float *f32(const at::Tensor &t, int64_t n) {
    if (!t.defined()) return nullptr;
    require(t.scalar_type() == at::kFloat, "expected a float32 tensor");
    require(t.numel() >= n, "a float32 tensor is smaller than its use");
    return static_cast<const float *>(t.const_data_ptr());
}
void require_like(const at::Tensor &t, const at::Tensor &like, int64_t n) {
    require(t.scalar_type() == like.scalar_type(), "tensors of one storage type expected");
    require(t.numel() >= n, "a tensor is smaller than its use");
}
void require_matrix(const at::Tensor &t, const at::Tensor &like, int64_t rows, int64_t cols) {
    require(t.dim() == 2 && t.size(0) == rows && t.size(1) == cols, "a weight matrix of another shape");
    require(t.scalar_type() == like.scalar_type(), "tensors of one storage type expected");
}
void require_rows(const at::Tensor &t, int64_t n) { require(t.dim() > 0 && t.size(0) >= n, "a node array has fewer rows than the graph"); }
// ... of every piece of a graph: its destinations and its slice of the sources
void require_pieces(const std::vector<int64_t> &parts, const std::vector<int64_t> &bounds, int64_t n_src, int64_t n_dst) {
    require(!parts.empty() && bounds.size() == parts.size() + 1, "one more bound than partitions expected");
    for (size_t q = 0; q < parts.size(); ++q) {
        const sar_part *g = reinterpret_cast<const sar_part *>(parts[q]);
        require(g->n_dst <= n_dst && bounds[q] >= 0 && bounds[q] + g->n_src <= n_src, "a node array has fewer rows than the graph");
    }
}
float *f32m(const at::Tensor &t) { return t.defined() ? static_cast<float *>(t.mutable_data_ptr()) : nullptr; }
const void *ptr(const at::Tensor &t) { return t.const_data_ptr(); }
void *ptrm(const at::Tensor &t) { return t.mutable_data_ptr(); }
// rows from s on
const char *rows(const at::Tensor &t, int64_t s) {
    const int64_t n = t.size(0);
    return static_cast<const char *>(t.const_data_ptr()) + (n ? (size_t)s * (t.nbytes() / n) : 0);
}
char *rowsm(const at::Tensor &t, int64_t s) { return const_cast<char *>(rows(t, s)); }

at::Tensor empty(at::IntArrayRef size, at::ScalarType type, const at::Tensor &like) {
    return at::detail::empty_cuda(size, type, like.device(), c10::nullopt);
}
at::Tensor bytes(size_t n, const at::Tensor &like) { return empty({(int64_t)(n < 256 ? 256 : n)}, at::kByte, like); }
void *stream() { return at::cuda::getCurrentCUDAStream().stream(); }

PyObject *wrap(const at::Tensor &t) {
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}
template <typename... Ts>
PyObject *tuple(const Ts &...ts) {
    PyObject *r = PyTuple_New(sizeof...(Ts));
    Py_ssize_t k = 0;
    ((PyTuple_SET_ITEM(r, k++, wrap(ts))), ...);
    return r;
}

// ---- graph preparation -----------------------------------------------------------------------------------------------------
// The sizes that the host needs (edges of the partitions, long rows and segments of the plans) come over in ONE copy, so
// that the stream is drained once: with a copy per plan and partition a small graph in 4 parts took 1.2 ms, nearly all of
// it waiting.
PyObject *from_coo(Args &a) {   // n, src, dst, bounds, threshold, t_threshold, parts -> ((4 arrays), plans, parts)
    const int64_t n = a.integer();
    const at::Tensor &src = a.tensor(), &dst = a.tensor();
    const auto bounds = a.integers();
    const int32_t threshold = (int32_t)a.integer(), t_threshold = (int32_t)a.integer();
    const int64_t k = a.flag() ? (int64_t)bounds.size() - 1 : 0, nnz = src.numel();
    const at::Tensor indptr = empty({n + 1}, at::kLong, src), t_indptr = empty({n + 1}, at::kLong, src);
    const at::Tensor indices = empty({nnz}, at::kInt, src), t_indices = empty({nnz}, at::kInt, src);
    auto i64 = [](const at::Tensor &t) { return static_cast<int64_t *>(t.mutable_data_ptr()); };
    auto i32 = [](const at::Tensor &t) { return static_cast<int32_t *>(t.mutable_data_ptr()); };
    const at::Tensor ws = bytes(L.sar_graph_workspace_bytes(nnz, n), src);
    SAR(sar_graph_from_coo, n, nnz, i32(src), i32(dst), i64(indptr), i32(indices), i64(t_indptr), i32(t_indices), ptrm(ws), ws.nbytes(), stream());

    at::Tensor indptr_all, indices_all;
    std::vector<at::Tensor> t_ip;
    if (k > 0) {
        indptr_all = empty({k, n + 1}, at::kLong, src);
        indices_all = empty({nnz > 0 ? nnz : 1}, at::kInt, src);
        SAR(sar_csr_split_indptr, n, i64(indptr), i32(indices), (int32_t)k, bounds.data(), i64(indptr_all), ptrm(ws), ws.nbytes(), stream());
        for (int64_t q = 0; q < k; ++q) {
            t_ip.push_back(empty({bounds[q + 1] - bounds[q] + 1}, at::kLong, src));
            SAR(sar_csc_slice_indptr, bounds[q], bounds[q + 1], i64(t_indptr), i64(t_ip.back()), stream());
        }
    }
    std::vector<sar_plan_job> jobs;
    if (threshold) jobs.push_back({n, i64(indptr), threshold, nullptr, nullptr});
    if (t_threshold) jobs.push_back({n, i64(t_indptr), t_threshold, nullptr, nullptr});
    for (int64_t q = 0; threshold && q < k; ++q) {
        jobs.push_back({n, i64(indptr_all) + q * (n + 1), threshold, nullptr, nullptr});
        jobs.push_back({bounds[q + 1] - bounds[q], i64(t_ip[q]), threshold, nullptr, nullptr});
    }
    const int32_t nj = (int32_t)jobs.size();
    const at::Tensor sizes = empty({2 * nj + k + 1}, at::kLong, src), plan_ws = bytes(L.sar_plan_many_workspace_bytes(nj, jobs.data()), src);
    SAR(sar_plan_count_many, nj, jobs.data(), i64(sizes), ptrm(plan_ws), plan_ws.nbytes(), stream());
    std::vector<int64_t> host((size_t)(2 * nj + k + 1), 0);
    if (k > 0) {   // a partition's edges are a run of the whole CSC: its first source's first edge to the next one's
        std::vector<const int64_t *> from((size_t)k + 1);
        for (int64_t q = 0; q <= k; ++q) from[q] = i64(t_indptr) + bounds[q];
        SAR(sar_gather_i64, (int32_t)k + 1, from.data(), i64(sizes) + 2 * nj, stream());
    }
    if (nj > 0 || k > 0) {
        cudaError_t e;
        Py_BEGIN_ALLOW_THREADS
        e = cudaMemcpyAsync(host.data(), i64(sizes), host.size() * 8, cudaMemcpyDeviceToHost, at::cuda::getCurrentCUDAStream());
        if (e == cudaSuccess) e = cudaStreamSynchronize(at::cuda::getCurrentCUDAStream());
        Py_END_ALLOW_THREADS
        check("sar_plan_count_many", e == cudaSuccess ? SAR_OK : SAR_ERR_CUDA);
    }
    const int64_t *first = host.data() + 2 * nj;
    if (k > 0)
        SAR(sar_csr_split_indices, n, i64(indptr), i32(indices), (int32_t)k, bounds.data(), i64(indptr_all), first, i32(indices_all), stream());
    PyObject *plans = PyTuple_New(nj);
    for (int32_t j = 0; j < nj; ++j) {
        const at::Tensor row = empty({host[2 * j]}, at::kInt, src), seg = empty({host[2 * j] + 1}, at::kLong, src);
        jobs[j].long_row = host[2 * j] > 0 ? i32(row) : i32(ws);
        jobs[j].long_seg = i64(seg);
        PyTuple_SET_ITEM(plans, j, Py_BuildValue("(LLNN)", (long long)host[2 * j], (long long)host[2 * j + 1], wrap(row), wrap(seg)));
    }
    SAR(sar_plan_fill_many, nj, jobs.data(), ptrm(plan_ws), plan_ws.nbytes(), stream());
    PyObject *parts = PyTuple_New(k);
    for (int64_t q = 0; q < k; ++q) {
        const int64_t cnt = first[q + 1] - first[q];
        PyTuple_SET_ITEM(parts, q, Py_BuildValue("(NNNNL)", wrap(indptr_all.select(0, q)), wrap(indices_all.narrow(0, first[q], cnt)), wrap(t_ip[q]),
                                                 wrap(t_indices.narrow(0, first[q], cnt)), (long long)cnt));
    }
    return Py_BuildValue("(NNN)", tuple(indptr, indices, t_indptr, t_indices), plans, parts);
}

// ---- aggregation -----------------------------------------------------------------------------------------------------------
struct Dims {
    int64_t n;
    int32_t H, F;
    sar_dtype t;
    explicit Dims(const at::Tensor &x) {
        if (x.dim() != 3) fail(PyExc_ValueError, "expected [n, heads, features]");
        n = x.size(0);
        H = (int32_t)x.size(1);
        F = (int32_t)x.size(2);
        t = code(x);
    }
};

bool forward_needs_workspace(const sar_part *g, const Dims &d) {
    const size_t es = d.t == SAR_BF16 ? 2 : 4;
    return (g->split && g->split->n_long > 0) || ((size_t)d.F * es) % 16 != 0;
}

struct Forward {
    at::Tensor out, m, d;
};
Forward forward_fused(const sar_part *g, const std::vector<int64_t> &bounds, const at::Tensor &feat, const at::Tensor &el,
                      const at::Tensor &er, double slope, at::Tensor ws, bool relu) {
    const Dims d(feat);
    require_rows(feat, g->n_src);
    const float *pl = f32(el, g->n_dst * d.H), *pr = f32(er, g->n_src * d.H);
    Forward r;
    r.m = empty({g->n_dst, d.H}, at::kFloat, feat);
    r.d = empty({g->n_dst, d.H}, at::kFloat, feat);
    r.out = empty({g->n_dst, d.H, d.F}, feat.scalar_type(), feat);
    if (!ws.defined() && forward_needs_workspace(g, d)) ws = bytes(L.sar_gat_workspace_bytes(g, d.H, d.F, d.t), feat);
    void *w = ws.defined() ? ptrm(ws) : nullptr;
    const size_t wb = ws.defined() ? ws.nbytes() : 0;
    if (relu)   // the un-split graph as one partition holding all sources
        SAR(sar_gat_fwd, g, ptr(feat), pl, pr, d.H, d.F, d.t, (float)slope, SAR_FIRST | SAR_LAST | SAR_RELU_OUT, nullptr,
            f32m(r.m), f32m(r.d), ptrm(r.out), w, wb, stream());
    else
        SAR(sar_gat_fwd_fused, g, (int32_t)bounds.size() - 1, bounds.data(), ptr(feat), pl, pr, d.H, d.F, d.t, (float)slope,
            f32m(r.m), f32m(r.d), ptrm(r.out), w, wb, stream());
    return r;
}

struct Backward {
    at::Tensor dfeat, del, der;
};
Backward backward_outputs(const at::Tensor &feat, const Dims &d, int64_t n_dst) {
    Backward r;
    r.dfeat = empty(feat.sizes(), feat.scalar_type(), feat);
    r.del = empty({n_dst, d.H}, at::kFloat, feat);
    r.der = empty({d.n, d.H}, at::kFloat, feat);
    return r;
}
Backward backward_fused(const sar_part *g, const std::vector<int64_t> &bounds, const at::Tensor &feat, const at::Tensor &el,
                        const at::Tensor &er, const at::Tensor &m, const at::Tensor &dd, const at::Tensor &gout, double slope, at::Tensor ws) {
    const Dims d(feat);
    const int64_t nh = g->n_dst * d.H;
    require_rows(feat, g->n_src);
    require_like(gout, feat, nh * d.F);
    const float *pl = f32(el, nh), *pr = f32(er, g->n_src * d.H), *pm = f32(m, nh), *pd = f32(dd, nh);
    Backward r = backward_outputs(feat, d, g->n_dst);
    if (!ws.defined()) ws = bytes(L.sar_gat_workspace_bytes(g, d.H, d.F, d.t), feat);
    SAR(sar_gat_bwd_fused, g, (int32_t)bounds.size() - 1, bounds.data(), ptr(feat), pl, pr, pm, pd, ptr(gout), d.H, d.F,
        d.t, (float)slope, ptrm(r.dfeat), f32m(r.del), f32m(r.der), ptrm(ws), ws.nbytes(), stream());
    return r;
}

size_t parts_workspace(const std::vector<int64_t> &parts, const Dims &d) {
    size_t nb = 0;
    for (int64_t p : parts) {
        const size_t b = L.sar_gat_workspace_bytes(reinterpret_cast<const sar_part *>(p), d.H, d.F, d.t);
        nb = b > nb ? b : nb;
    }
    return nb;
}
unsigned step_flags(size_t q, size_t k) { return (q == 0 ? SAR_FIRST : 0u) | (q + 1 == k ? SAR_LAST : 0u); }

PyObject *gat_forward(Args &a) {   // part, bounds, feat, el, er, slope, workspace, relu
    const sar_part *g = a.part();
    const auto bounds = a.integers();
    const at::Tensor &feat = a.tensor(), &el = a.tensor(), &er = a.tensor();
    const double slope = a.real();
    const at::Tensor ws = a.optional();
    const Forward r = forward_fused(g, bounds, feat, el, er, slope, ws, a.flag());
    return tuple(r.out, r.m, r.d);
}

PyObject *gat_backward(Args &a) {   // part, bounds, feat, el, er, m, d, gout, slope, workspace
    const sar_part *g = a.part();
    const auto bounds = a.integers();
    const at::Tensor &feat = a.tensor(), &el = a.tensor(), &er = a.tensor(), &m = a.tensor(), &d = a.tensor(), &gout = a.tensor();
    const double slope = a.real();
    const Backward r = backward_fused(g, bounds, feat, el, er, m, d, gout, slope, a.optional());
    return tuple(r.dfeat, r.del, r.der);
}

PyObject *gat_forward_parts(Args &a) {   // parts, bounds, n_dst, feat, el, er, slope, keep, relu
    const auto parts = a.integers(), bounds = a.integers();
    const int64_t n_dst = a.integer();
    const at::Tensor &feat = a.tensor(), &el = a.tensor(), &er = a.tensor();
    const double slope = a.real();
    const bool keep = a.flag(), relu = a.flag();
    const Dims d(feat);
    const size_t k = parts.size();
    require_pieces(parts, bounds, d.n, n_dst);
    const float *pl = f32(el, n_dst * d.H);
    f32(er, bounds[k] * d.H);
    const at::Tensor m = empty({n_dst, d.H}, at::kFloat, feat), dd = empty({n_dst, d.H}, at::kFloat, feat);
    const at::Tensor out = empty({n_dst, d.H, d.F}, feat.scalar_type(), feat);
    at::Tensor acc;
    if (k > 1 || keep) acc = empty({n_dst, d.H, d.F}, at::kFloat, feat);
    const at::Tensor ws = bytes(parts_workspace(parts, d), feat);
    for (size_t q = 0; q < k; ++q) {
        unsigned flags = step_flags(q, k);
        if (q + 1 == k) flags |= (keep ? SAR_KEEP_NUMERATOR : 0u) | (relu ? SAR_RELU_OUT : 0u);
        SAR(sar_gat_fwd, reinterpret_cast<const sar_part *>(parts[q]), rows(feat, bounds[q]), pl,
            reinterpret_cast<const float *>(rows(er, bounds[q])), d.H, d.F, d.t, (float)slope, flags, f32m(acc), f32m(m), f32m(dd), ptrm(out),
            ptrm(ws), ws.nbytes(), stream());
    }
    return tuple(out, m, dd, acc);
}

PyObject *gat_backward_parts(Args &a) {   // parts, bounds, n_dst, feat, el, er, m, d, gout, slope, out_or_acc, is_numerator
    const auto parts = a.integers(), bounds = a.integers();
    const int64_t n_dst = a.integer();
    const at::Tensor &feat = a.tensor(), &el = a.tensor(), &er = a.tensor(), &m = a.tensor(), &dd = a.tensor(), &gout = a.tensor();
    const double slope = a.real();
    const at::Tensor &oa = a.tensor();
    const bool numerator = a.flag();
    const Dims d(feat);
    const size_t k = parts.size();
    const int64_t nh = n_dst * d.H;
    require_pieces(parts, bounds, d.n, n_dst);
    require_like(gout, feat, nh * d.F);
    if (numerator) f32(oa, nh * d.F);
    else require_like(oa, feat, nh * d.F);
    const float *pl = f32(el, nh), *pm = f32(m, nh), *pd = f32(dd, nh);
    f32(er, bounds[k] * d.H);
    const Backward r = backward_outputs(feat, d, n_dst);
    const at::Tensor ws = bytes(parts_workspace(parts, d), feat);
    SAR(sar_gat_bwd_prepare, n_dst, d.H, d.F, d.t, ptr(oa), numerator ? 1 : 0, ptr(gout), pl, pm, pd, nullptr, ptrm(ws), ws.nbytes(), stream());
    for (size_t q = 0; q < k; ++q) {
        const int64_t s = bounds[q];
        SAR(sar_gat_bwd, reinterpret_cast<const sar_part *>(parts[q]), rows(feat, s), pl, reinterpret_cast<const float *>(rows(er, s)),
            pm, pd, ptr(gout), d.H, d.F, d.t, (float)slope, step_flags(q, k) | (q > 0 ? SAR_SAME_WORKSPACE : 0u), rowsm(r.dfeat, s), f32m(r.del),
            reinterpret_cast<float *>(rowsm(r.der, s)), ptrm(ws), ws.nbytes(), stream());
    }
    return tuple(r.dfeat, r.del, r.der);
}

// ---- sums ----------------------------------------------------------------------------------------------------------------
size_t sum_workspace(const sar_part *g, const at::Tensor &x) {
    const int32_t F = (int32_t)x.size(1);
    const bool ragged = ((size_t)F * x.element_size()) % 16 != 0;
    return ((g->split && g->split->n_long > 0) || ragged) ? L.sar_spmm_workspace_bytes(g, F, code(x)) : 0;
}
// scratch that serves one sum after another (they follow each other on the stream)
struct Scratch {
    at::Tensor t;
    void *get(size_t n, const at::Tensor &like) {
        if (n && (!t.defined() || t.nbytes() < n)) t = bytes(n, like);
        return t.defined() ? ptrm(t) : nullptr;
    }
    size_t size() const { return t.defined() ? t.nbytes() : 0; }
};
void sum_scaled(const sar_part *g, const void *x, const at::Tensor &like, unsigned flags, const float *src, const float *dst, void *out, Scratch &ws) {
    void *w = ws.get(sum_workspace(g, like), like);
    SAR(sar_spmm_agg_scaled, g, x, (int32_t)like.size(1), code(like), flags, src, dst, out, w, ws.size(), stream());
}

PyObject *spmm(Args &a) {   // part, feat, flags, deg_total
    const sar_part *g = a.part();
    const at::Tensor &x = a.tensor();
    const unsigned flags = (unsigned)a.integer();
    const at::Tensor deg = a.optional();
    require_rows(x, g->n_src);
    require(!deg.defined() || (deg.scalar_type() == at::kLong && deg.numel() >= g->n_dst), "expected an int64 degree per node");
    const at::Tensor out = empty({g->n_dst, x.size(1)}, x.scalar_type(), x);
    Scratch ws;
    void *w = ws.get(sum_workspace(g, x), x);
    SAR(sar_spmm_agg, g, ptr(x), (int32_t)x.size(1), code(x), flags, deg.defined() ? static_cast<const int64_t *>(ptr(deg)) : nullptr, ptrm(out),
        w, ws.size(), stream());
    return wrap(out);
}

PyObject *spmm_scaled(Args &a) {   // part, feat, flags, src_scale, dst_scale, out
    const sar_part *g = a.part();
    const at::Tensor &x = a.tensor();
    const unsigned flags = (unsigned)a.integer();
    const at::Tensor src = a.optional(), dst = a.optional();
    at::Tensor out = a.optional();
    require_rows(x, g->n_src);
    if (out.defined()) require_like(out, x, g->n_dst * x.size(1));
    else out = empty({g->n_dst, x.size(1)}, x.scalar_type(), x);
    Scratch ws;
    sum_scaled(g, ptr(x), x, flags, f32(src, g->n_src), f32(dst, g->n_dst), ptrm(out), ws);
    return wrap(out);
}

PyObject *propagate(Args &a) {   // parts, bounds, x0, alpha, iters, src_scale, dst_scale
    const auto parts = a.integers(), bounds = a.integers();
    const at::Tensor &x0 = a.tensor();
    const double alpha = a.real();
    const int64_t iters = a.integer();
    const at::Tensor src = a.optional(), dst = a.optional();
    if (iters <= 0) return wrap(x0.clone());
    std::vector<const sar_part *> ps;
    for (int64_t p : parts) ps.push_back(reinterpret_cast<const sar_part *>(p));
    require_pieces(parts, bounds, x0.size(0), x0.size(0));
    const float *ss = f32(src, ps[0]->n_dst), *ds = f32(dst, ps[0]->n_dst);
    const int32_t k = (int32_t)ps.size(), F = (int32_t)x0.size(1);
    const at::Tensor out = empty(x0.sizes(), x0.scalar_type(), x0);
    const at::Tensor ws = bytes(L.sar_propagate_workspace_bytes_at(k, ps.data(), ptr(x0), F, code(x0), ptr(out)), x0);
    SAR(sar_propagate, k, ps.data(), bounds.data(), ptr(x0), F, code(x0), (float)alpha, iters, ss, ds, ptrm(out), ptrm(ws), ws.nbytes(), stream());
    return wrap(out);
}

// sum over the pieces of one graph of inv * A x
void aggregate(const std::vector<int64_t> &parts, const std::vector<int64_t> &bounds, const at::Tensor &h, const at::Tensor &inv, const at::Tensor &agg, Scratch &ws) {
    for (size_t q = 0; q < parts.size(); ++q)
        sum_scaled(reinterpret_cast<const sar_part *>(parts[q]), rows(h, bounds[q]), h, step_flags(q, parts.size()), nullptr, f32(inv, reinterpret_cast<const sar_part *>(parts[q])->n_dst), ptrm(agg), ws);
}
// dh of every piece's sources (+)= what their out-edges hand back of dagg
void scatter(const std::vector<int64_t> &parts, const std::vector<int64_t> &bounds, const at::Tensor &dagg, const at::Tensor &inv, const at::Tensor &dh, unsigned first, Scratch &ws) {
    for (size_t q = 0; q < parts.size(); ++q) {
        const sar_part *g = reinterpret_cast<const sar_part *>(parts[q]);
        const sar_part t{g->n_src, g->n_dst, g->nnz, g->t_indptr, g->t_indices, g->indptr, g->indices, g->t_split, g->split};
        sum_scaled(&t, ptr(dagg), dagg, first | SAR_LAST, f32(inv, g->n_dst), nullptr, rowsm(dh, bounds[q]), ws);
    }
}

// ---- layers --------------------------------------------------------------------------------------------------------------
PyObject *layer_forward(Args &a) {   // part, bounds, h, W, a_l, a_r, slope, relu_input
    const sar_part *g = a.part();
    const auto bounds = a.integers();
    const at::Tensor &h = a.tensor(), &W = a.tensor(), &al = a.tensor(), &ar = a.tensor();
    const double slope = a.real();
    const bool relu = a.flag();
    const int64_t n = h.size(0);
    const int32_t d_in = (int32_t)h.size(1), H = (int32_t)al.size(0), F = (int32_t)al.size(1);
    const sar_dtype t = code(h);
    require_matrix(W, h, d_in, (int64_t)H * F);
    require_rows(h, g->n_src);
    const float *pal = f32(al, (int64_t)H * F), *par = f32(ar, (int64_t)H * F);
    if (relu) SAR(sar_relu, h.numel(), t, ptrm(h), stream());
    const at::Tensor z = empty({n, H, F}, h.scalar_type(), h), el = empty({n, H}, at::kFloat, h), er = empty({n, H}, at::kFloat, h);
    {
        const at::Tensor ws = bytes(L.sar_linear_workspace_bytes(n, d_in, H * F), h);
        if (F % 8 == 0 && 128 % F == 0) {   // the scores leave the projection's epilogue
            SAR(sar_linear_project, n, d_in, H, F, t, ptr(h), ptr(W), pal, par, ptrm(z), f32m(el), f32m(er), nullptr, ptrm(ws), ws.nbytes(), stream());
        } else {
            SAR(sar_linear, n, d_in, H * F, t, ptr(h), ptr(W), ptrm(z), ptrm(ws), ws.nbytes(), stream());
            SAR(sar_gat_project, n, H, F, t, ptrm(z), pal, par, f32m(el), f32m(er), 0u, stream());
        }
    }
    const Forward r = forward_fused(g, bounds, z, el, er, slope, at::Tensor(), false);
    return tuple(r.out, z, el, er, r.m, r.d);
}

PyObject *layer_backward(Args &a) {   // part, bounds, h, W, a_l, a_r, z, el, er, m, d, gout, slope, relu_input
    const sar_part *g = a.part();
    const auto bounds = a.integers();
    const at::Tensor &h = a.tensor(), &W = a.tensor(), &al = a.tensor(), &ar = a.tensor();
    const at::Tensor &z = a.tensor(), &el = a.tensor(), &er = a.tensor(), &m = a.tensor(), &d = a.tensor(), &gout = a.tensor();
    const double slope = a.real();
    const bool relu = a.flag();
    const int64_t n = h.size(0);
    const int32_t d_in = (int32_t)h.size(1), H = (int32_t)al.size(0), F = (int32_t)al.size(1);
    const sar_dtype t = code(h);
    require_matrix(W, h, d_in, (int64_t)H * F);
    require(z.dim() == 3 && z.size(0) == n && z.size(1) == H && z.size(2) == F, "expected the z of the forward call");
    require_like(z, h, 0);
    const float *pal = f32(al, (int64_t)H * F), *par = f32(ar, (int64_t)H * F);
    const Backward b = backward_fused(g, bounds, z, el, er, m, d, gout, slope, at::Tensor());
    const at::Tensor dal = empty({H, F}, at::kFloat, h), dar = empty({H, F}, at::kFloat, h);
    {
        const at::Tensor ws = bytes(L.sar_gat_project_workspace_bytes(H, F), h);
        SAR(sar_gat_project_bwd, n, H, F, t, ptr(z), pal, par, f32(b.del, n * H), f32(b.der, n * H), ptrm(b.dfeat), f32m(dal), f32m(dar), 0u, ptrm(ws), ws.nbytes(), stream());
    }
    const at::Tensor ws = bytes(L.sar_linear_workspace_bytes(n, d_in, H * F), h);
    const at::Tensor dW = empty({d_in, (int64_t)H * F}, at::kFloat, h), dh = empty(h.sizes(), h.scalar_type(), h);
    SAR(sar_linear_bwd_weight, n, d_in, H * F, t, ptr(h), ptr(b.dfeat), f32m(dW), ptrm(ws), ws.nbytes(), stream());
    if (relu)   // the mask of the input's ReLU is applied in the GEMM's epilogue
        SAR(sar_linear_bwd_input_relu, n, d_in, H * F, t, ptr(b.dfeat), ptr(W), ptr(h), ptrm(dh), ptrm(ws), ws.nbytes(), stream());
    else
        SAR(sar_linear_bwd_input, n, d_in, H * F, t, ptr(b.dfeat), ptr(W), ptrm(dh), ptrm(ws), ws.nbytes(), stream());
    return tuple(dh, dW, dal, dar);
}

PyObject *sage_forward(Args &a) {   // parts, bounds, h, W, W_res, inv
    const auto parts = a.integers(), bounds = a.integers();
    const at::Tensor &h = a.tensor(), &W = a.tensor(), &Wr = a.tensor(), &inv = a.tensor();
    const int64_t n = h.size(0);
    const int32_t d_in = (int32_t)h.size(1), d_out = (int32_t)W.size(1);
    const sar_dtype t = code(h);
    require_pieces(parts, bounds, n, n);
    require_matrix(W, h, d_in, d_out);
    require_matrix(Wr, h, d_in, d_out);
    const at::Tensor agg = empty(h.sizes(), h.scalar_type(), h), pre = empty({n, d_out}, h.scalar_type(), h);
    Scratch sws;
    aggregate(parts, bounds, h, inv, agg, sws);
    const at::Tensor ws = bytes(L.sar_linear_workspace_bytes(n, d_in, d_out), h);
    SAR(sar_linear, n, d_in, d_out, t, ptr(h), ptr(Wr), ptrm(pre), ptrm(ws), ws.nbytes(), stream());
    SAR(sar_linear_accumulate, n, d_in, d_out, t, ptr(agg), ptr(W), ptrm(pre), ptrm(ws), ws.nbytes(), stream());
    return tuple(pre, agg);
}

PyObject *sage_backward(Args &a) {   // parts, bounds, h, W, W_res, agg, inv, gpre
    const auto parts = a.integers(), bounds = a.integers();
    const at::Tensor &h = a.tensor(), &W = a.tensor(), &Wr = a.tensor(), &agg = a.tensor(), &inv = a.tensor(), &g = a.tensor();
    const int64_t n = h.size(0);
    const int32_t d_in = (int32_t)h.size(1), d_out = (int32_t)W.size(1);
    const sar_dtype t = code(h);
    require_pieces(parts, bounds, n, n);
    require_matrix(W, h, d_in, d_out);
    require_matrix(Wr, h, d_in, d_out);
    require_like(agg, h, n * d_in);
    require_like(g, h, n * d_out);
    const at::Tensor ws = bytes(L.sar_linear_workspace_bytes(n, d_in, d_out), h);
    const at::Tensor dW = empty({d_in, d_out}, at::kFloat, h), dWr = empty({d_in, d_out}, at::kFloat, h);
    SAR(sar_linear_bwd_weight, n, d_in, d_out, t, ptr(agg), ptr(g), f32m(dW), ptrm(ws), ws.nbytes(), stream());
    SAR(sar_linear_bwd_weight, n, d_in, d_out, t, ptr(h), ptr(g), f32m(dWr), ptrm(ws), ws.nbytes(), stream());
    const at::Tensor dh = empty(h.sizes(), h.scalar_type(), h), dagg = empty(h.sizes(), h.scalar_type(), h);
    SAR(sar_linear_bwd_input, n, d_in, d_out, t, ptr(g), ptr(Wr), ptrm(dh), ptrm(ws), ws.nbytes(), stream());   // the residual path
    SAR(sar_linear_bwd_input, n, d_in, d_out, t, ptr(g), ptr(W), ptrm(dagg), ptrm(ws), ws.nbytes(), stream());
    Scratch sws;
    scatter(parts, bounds, dagg, inv, dh, 0u, sws);   // plus what every out-edge hands back
    return tuple(dh, dW, dWr);
}

// ---- batch normalisation (one worker) ------------------------------------------------------------------------------------
PyObject *bn_forward(Args &a) {   // x, eps, gamma, beta
    const at::Tensor &x = a.tensor();
    const double eps = a.real();
    const at::Tensor gamma = a.optional(), beta = a.optional();
    const int64_t n = x.size(0);
    const int32_t C = (int32_t)x.size(1);
    const sar_dtype t = code(x);
    const float *pg = f32(gamma, C), *pb = f32(beta, C);
    const at::Tensor ws = bytes(L.sar_bn_workspace_bytes(C), x);
    const at::Tensor mean = empty({C}, at::kFloat, x), m2 = empty({C}, at::kFloat, x), rstd = empty({C}, at::kFloat, x);
    const at::Tensor y = empty(x.sizes(), x.scalar_type(), x);
    SAR(sar_bn_stats, n, C, t, ptr(x), f32m(mean), f32m(m2), ptrm(ws), ws.nbytes(), stream());
    SAR(sar_bn_rstd, C, f32(m2, C), n > 1 ? n : 1, (float)eps, f32m(rstd), stream());
    SAR(sar_bn_apply, n, C, t, ptr(x), f32(mean, C), f32(rstd, C), pg, pb, ptrm(y), stream());
    return tuple(y, mean, rstd);
}

PyObject *bn_backward(Args &a) {   // x, gy, mean, rstd, gamma, count
    const at::Tensor &x = a.tensor(), &gy = a.tensor(), &mean = a.tensor(), &rstd = a.tensor();
    const at::Tensor gamma = a.optional();
    const int64_t count = a.integer(), n = x.size(0);
    const int32_t C = (int32_t)x.size(1);
    const sar_dtype t = code(x);
    require_like(gy, x, n * C);
    const float *pm = f32(mean, C), *pr = f32(rstd, C), *pg = f32(gamma, C);
    const at::Tensor ws = bytes(L.sar_bn_workspace_bytes(C), x);
    const at::Tensor s0 = empty({C}, at::kFloat, x), s1 = empty({C}, at::kFloat, x), gx = empty(x.sizes(), x.scalar_type(), x);
    SAR(sar_bn_bwd_stats, n, C, t, ptr(x), pm, pr, ptr(gy), f32m(s0), f32m(s1), ptrm(ws), ws.nbytes(), stream());
    SAR(sar_bn_bwd_apply, n, C, t, ptr(x), pm, pr, pg, ptr(gy), f32(s0, C), f32(s1, C), (float)(1.0 / (double)(count > 1 ? count : 1)), ptrm(gx), stream());
    return tuple(gx, s1, s0);
}

// ---- module --------------------------------------------------------------------------------------------------------------
PyObject *init(Args &a) {   // handle of the loaded library, binding.SarError, torch.OutOfMemoryError
    void *handle = reinterpret_cast<void *>(a.integer());
    g_error = a.next();
    g_oom = a.next();
    Py_INCREF(g_error);
    Py_INCREF(g_oom);
#define X(f)                                                     \
    L.f = reinterpret_cast<decltype(&::f)>(dlsym(handle, #f));   \
    if (!L.f) fail(PyExc_RuntimeError, "libsar lacks " #f);
    SAR_TABLE(X)
#undef X
    Py_RETURN_NONE;
}

// Entry point of a function: argument errors and library errors are Python errors already, torch's become RuntimeError.
template <PyObject *(*F)(Args &)>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
    try {
        Args a{args, n};
        return F(a);
    } catch (const Failed &) {
        return nullptr;
    } catch (const c10::OutOfMemoryError &e) {
        PyErr_SetString(g_oom, e.what());
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
#define M(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<f>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {M(init), M(from_coo), M(gat_forward), M(gat_backward), M(gat_forward_parts), M(gat_backward_parts), M(spmm), M(spmm_scaled),
                           M(propagate), M(layer_forward), M(layer_backward), M(sage_forward), M(sage_backward), M(bn_forward), M(bn_backward),
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_sar_torch", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject *PyInit__sar_torch() { return PyModule_Create(&g_module); }
