// Marshalling between torch tensors and librsd's C ABI (include/rsd.h), as a CPython extension: api.py's functions hand
// their arguments on to the functions below, which read sizes, strides and device pointers off the tensors and call the
// entry point of the same name on the current CUDA stream.  Nothing is computed here.  A call through ctypes spent 20 to 40 us
// on attribute look-ups and conversions, more than a small draft or walk takes on the GPU; this takes two to three.
#include <Python.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include <c10/cuda/CUDAStream.h>

#include <vector>

#include "../../include/rsd.h"

namespace {

PyObject* g_error = nullptr;   // api.RsdError

decltype(&rsd_last_error) p_last_error;
decltype(&rsd_filter_rows) p_filter_rows;
decltype(&rsd_gumbel_topk_draft) p_gumbel;
decltype(&rsd_sbs_step) p_sbs_step;
decltype(&rsd_sbs_step_static) p_sbs_step_static;
decltype(&rsd_sbs_draft_tree) p_sbs_draft_tree;
decltype(&rsd_verify_tree) p_verify_tree;
decltype(&rsd_verify_tree_rule) p_verify_tree_rule;
decltype(&rsd_resample_residual) p_resample;

struct Failed {};   // a Python error is set

[[noreturn]] void fail(const char* message) {
    PyErr_SetString(g_error, message);
    throw Failed();
}
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "a tensor is expected, got %s", Py_TYPE(o)->tp_name);
        throw Failed();
    }
    return THPVariable_Unpack(o);
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
long long low_bits(PyObject* n) {   // takes the reference
    if (!n) throw Failed();
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(n);
    Py_DECREF(n);
    if (PyErr_Occurred()) throw Failed();
    return (long long)v;
}
long long integer(PyObject* o) { return low_bits(PyNumber_Index(o)); }       // an integer; a float or a text is refused
long long as_integer(PyObject* o) { return low_bits(PyNumber_Long(o)); }     // int(o)
double real(PyObject* o) {   // float(o)
    if (PyFloat_CheckExact(o)) return PyFloat_AS_DOUBLE(o);
    PyObject* n = PyNumber_Float(o);
    if (!n) throw Failed();
    const double v = PyFloat_AsDouble(n);
    Py_DECREF(n);
    return v;
}
bool truth(PyObject* o) {
    const int t = PyObject_IsTrue(o);
    if (t < 0) throw Failed();
    return t != 0;
}
std::vector<int32_t> integers(PyObject* o) {
    PyObject* s = PySequence_Fast(o, "a sequence of integers is expected");
    if (!s) throw Failed();
    std::vector<int32_t> v((size_t)PySequence_Fast_GET_SIZE(s));
    try {
        for (size_t i = 0; i < v.size(); ++i) v[i] = (int32_t)as_integer(PySequence_Fast_GET_ITEM(s, i));
    } catch (Failed&) {
        Py_DECREF(s);
        throw;
    }
    Py_DECREF(s);
    return v;
}
rsd_rows rows_of(const at::Tensor& t, bool is_logprob, double temperature) {
    if (!t.is_cuda()) fail("rows must live on a CUDA device");
    rsd_rows r;
    if (t.scalar_type() == at::kFloat) r.dtype = RSD_F32;
    else if (t.scalar_type() == at::kBFloat16) r.dtype = RSD_BF16;
    else fail("rows must be float32 or bfloat16");
    const int64_t n = t.dim();
    if (n < 1 || t.stride(n - 1) != 1) fail("rows must be dense along the vocabulary");
    if (n != 2 && n != 3) fail("rows must be [B, R, V] or [B, V]");
    r.data = t.data_ptr();
    r.is_logprob = is_logprob;
    r.seq_stride = t.stride(0);
    r.row_stride = n == 3 ? t.stride(1) : t.size(1);
    r.temperature = (float)temperature;
    return r;
}
void want_dims(const at::Tensor& t, int n) {
    if (t.dim() == n) return;
    PyErr_Format(PyExc_ValueError, "a tensor of %d dimensions is expected, got %d", n, (int)t.dim());
    throw Failed();
}
rsd_stream_t stream() { return (rsd_stream_t)c10::cuda::getCurrentCUDAStream().stream(); }

template <typename F>
PyObject* call(F f) {   // f: the library call, without the interpreter's lock
    int code;
    Py_BEGIN_ALLOW_THREADS
    code = f();
    Py_END_ALLOW_THREADS
    if (code != 0) {
        PyErr_Format(g_error, "librsd error %d: %s", code, p_last_error());
        return nullptr;
    }
    Py_RETURN_NONE;
}
template <PyObject* (*F)(PyObject* const*), int N>
PyObject* entry(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!g_error) {
        PyErr_SetString(PyExc_RuntimeError, "the library is not bound");
        return nullptr;
    }
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "%d arguments are expected, got %zd", N, n);
        return nullptr;
    }
    try {
        return F(a);
    } catch (Failed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// rows, temperature, top_k, top_p, out rows, kept, status
PyObject* filter_rows(PyObject* const* a) {
    const at::Tensor &t = tensor(a[0]), &out = tensor(a[4]);
    want_dims(t, 3);
    if (!out.is_contiguous() || out.scalar_type() != t.scalar_type()) fail("out rows must be contiguous and of the rows' dtype");
    const rsd_rows r = rows_of(t, false, real(a[1]));
    const int top_k = (int)as_integer(a[2]);
    const float top_p = (float)real(a[3]);
    void *rows = out.data_ptr(), *kept = ptr(a[5]), *status = ptr(a[6]);
    const rsd_stream_t s = stream();
    const int B = (int)t.size(0), R = (int)t.size(1), V = (int)t.size(2);
    return call([&] { return p_filter_rows(&r, B, R, V, top_k, top_p, rows, (int32_t*)kept, (int32_t*)status, s); });
}

// draft, is_logprob, temperature, k_per_row, rng_node, max_k, seed, step, seq_base, token, perturbed, logprob, child_base, node_token,
// status
PyObject* gumbel_topk_draft(PyObject* const* a) {
    const at::Tensor& t = tensor(a[0]);
    want_dims(t, 3);
    const rsd_rows r = rows_of(t, truth(a[1]), real(a[2]));
    const int B = (int)t.size(0), R = (int)t.size(1), V = (int)t.size(2);
    const std::vector<int32_t> k = integers(a[3]), node = integers(a[4]);
    std::vector<int32_t> base;
    if (a[12] != Py_None) base = integers(a[12]);
    if ((int)k.size() < R || (int)node.size() < R || (a[12] != Py_None && (int)base.size() < R)) fail("k_per_row, rng_node and child_base must have an entry per row");
    const int max_k = (int)integer(a[5]);
    const uint64_t seed = (uint64_t)integer(a[6]);
    const uint32_t step = (uint32_t)integer(a[7]), seq = (uint32_t)integer(a[8]);
    int32_t* node_token = nullptr;
    int node_stride = 0;
    if (a[13] != Py_None) {
        const at::Tensor& nt = tensor(a[13]);
        if (nt.scalar_type() != at::kInt || !nt.is_contiguous()) fail("node_token must be contiguous int32");
        node_token = (int32_t*)nt.data_ptr();
        node_stride = (int)nt.size(1);
    }
    void *token = ptr(a[9]), *pert = ptr(a[10]), *lp = ptr(a[11]), *status = ptr(a[14]);
    const rsd_stream_t s = stream();
    return call([&] {
        return p_gumbel(&r, B, R, V, k.data(), node.data(), max_k, seed, step, seq, (int32_t*)token, (float*)pert, (float*)lp,
                        a[12] == Py_None ? nullptr : base.data(), node_token, node_stride, (int32_t*)status, s);
    });
}

void same_stride(const at::Tensor& x, const at::Tensor& y, const char* message) {
    if (x.dim() != 2 || y.dim() != 2 || x.stride(0) != y.stride(0) || x.stride(1) != 1 || y.stride(1) != 1) fail(message);
}

// draft_level, is_logprob, temperature, W, first_parent_node, sum_in, gumbel_in, seed, step, seq_base, token, parent, parent_base, sum,
// gumbel, count, status, workspace (None: the library's built-in scratch)
PyObject* sbs_step(PyObject* const* a) {
    const at::Tensor &t = tensor(a[0]), &token = tensor(a[10]), &parent = tensor(a[11]);
    want_dims(t, 3);
    const rsd_rows r = rows_of(t, truth(a[1]), real(a[2]));
    const int B = (int)t.size(0), n_par = (int)t.size(1), V = (int)t.size(2), W = (int)integer(a[3]);
    const int32_t first = (int32_t)integer(a[4]), base = (int32_t)integer(a[12]);
    const float *sum_in = (const float*)ptr(a[5]), *gum_in = (const float*)ptr(a[6]);
    const uint64_t seed = (uint64_t)integer(a[7]);
    const uint32_t step = (uint32_t)integer(a[8]), seq = (uint32_t)integer(a[9]);
    same_stride(token, parent, "out token/parent must share a row stride and be dense along the picks");
    int32_t *tok = (int32_t*)token.data_ptr(), *par = (int32_t*)parent.data_ptr(), *count = (int32_t*)ptr(a[15]), *status = (int32_t*)ptr(a[16]);
    float *sum = (float*)ptr(a[13]), *gum = (float*)ptr(a[14]);
    const int64_t stride = token.stride(0);
    const rsd_stream_t s = stream();
    if (a[17] == Py_None)
        return call([&] {
            return p_sbs_step_static(&r, B, n_par, V, W, first, sum_in, gum_in, seed, step, seq, tok, par, stride, base, sum, gum, count, status, s);
        });
    const at::Tensor& ws = tensor(a[17]);
    void* wp = ws.data_ptr();
    const size_t wn = (size_t)ws.numel();
    return call([&] {
        return p_sbs_step(&r, B, n_par, V, W, first, sum_in, gum_in, seed, step, seq, tok, par, stride, base, sum, gum, count, status, wp, wn, s);
    });
}

// draft, is_logprob, temperature, W, L, seed, step, seq_base, node_token, node_parent, sum, gumbel, count, status, workspace
PyObject* sbs_draft_tree(PyObject* const* a) {
    const at::Tensor &t = tensor(a[0]), &token = tensor(a[8]), &parent = tensor(a[9]), &ws = tensor(a[14]);
    want_dims(t, 3);
    const int B = (int)t.size(0), V = (int)t.size(2), W = (int)integer(a[3]), L = (int)integer(a[4]);
    const int64_t P = 1 + (int64_t)(L - 1) * W;
    if (t.size(1) != P) {
        PyErr_Format(g_error, "draft must hold 1 + (L - 1) W = %lld rows per sequence, got %lld", (long long)P, (long long)t.size(1));
        throw Failed();
    }
    same_stride(token, parent, "node_token / node_parent must share a row stride and be dense along the nodes");
    const rsd_rows r = rows_of(t, truth(a[1]), real(a[2]));
    const uint64_t seed = (uint64_t)integer(a[5]);
    const uint32_t step = (uint32_t)integer(a[6]), seq = (uint32_t)integer(a[7]);
    int32_t *tok = (int32_t*)token.data_ptr(), *par = (int32_t*)parent.data_ptr(), *count = (int32_t*)ptr(a[12]), *status = (int32_t*)ptr(a[13]);
    float *sum = (float*)ptr(a[10]), *gum = (float*)ptr(a[11]);
    const int64_t stride = token.stride(0);
    void* wp = ws.data_ptr();
    const size_t wn = (size_t)ws.numel();
    const rsd_stream_t s = stream();
    return call([&] { return p_sbs_draft_tree(&r, B, V, W, L, seed, step, seq, tok, par, stride, sum, gum, count, status, wp, wn, s); });
}

// draft, draft temperature, target, target temperature, parent, token, num_levels, seed, step, seq_base, rule, gamma, final_sampler,
// always through rsd_verify_tree_rule, accepted_len, accepted_node, accepted_token, last_token, stop_reason, theta, status
PyObject* verify_tree(PyObject* const* a) {
    const at::Tensor &target = tensor(a[2]), &parent = tensor(a[4]), &token = tensor(a[5]);
    want_dims(target, 3);
    want_dims(token, 2);
    if (parent.scalar_type() != at::kInt || token.scalar_type() != at::kInt) fail("parent and token must be int32");
    if (!parent.is_contiguous() || !token.is_contiguous()) fail("parent and token must be contiguous");
    const rsd_rows d = rows_of(tensor(a[0]), false, real(a[1])), t = rows_of(target, false, real(a[3]));
    rsd_tree tree;
    tree.num_levels = (int32_t)integer(a[6]);
    tree.num_nodes = (int32_t)token.size(1);
    tree.parent = (const int32_t*)parent.data_ptr();
    tree.token = (const int32_t*)token.data_ptr();
    tree.topology_is_shared = parent.dim() == 1;
    const int B = (int)target.size(0), V = (int)target.size(2);
    const uint64_t seed = (uint64_t)integer(a[7]);
    const uint32_t step = (uint32_t)integer(a[8]), seq = (uint32_t)integer(a[9]);
    const int rule = (int)as_integer(a[10]), sampler = (int)as_integer(a[12]);
    const float gamma = (float)real(a[11]);
    int32_t *len = (int32_t*)ptr(a[14]), *node = (int32_t*)ptr(a[15]), *tok = (int32_t*)ptr(a[16]), *last = (int32_t*)ptr(a[17]), *reason = (int32_t*)ptr(a[18]),
            *status = (int32_t*)ptr(a[20]);
    float* theta = (float*)ptr(a[19]);
    const rsd_stream_t s = stream();
    if (rule == RSD_RULE_RRS && sampler == RSD_FINAL_INVERSE_CDF && !truth(a[13]))
        return call([&] { return p_verify_tree(&d, &t, &tree, B, V, seed, step, seq, len, node, tok, last, reason, theta, status, s); });
    return call([&] { return p_verify_tree_rule(&d, &t, &tree, B, V, rule, gamma, sampler, seed, step, seq, len, node, tok, last, reason, theta, status, s); });
}

// draft_row, draft temperature, target_row, target temperature, rejected, rng_node, seed, step, seq_base, token, residual, status
PyObject* resample_residual(PyObject* const* a) {
    const at::Tensor& target = tensor(a[2]);
    want_dims(target, 2);
    const rsd_rows t = rows_of(target, false, real(a[3])), d = a[0] == Py_None ? t : rows_of(tensor(a[0]), false, real(a[1]));
    const int32_t* rejected = nullptr;
    int max_k = 0;
    if (a[4] != Py_None) {
        const at::Tensor& rj = tensor(a[4]);
        want_dims(rj, 2);
        if (rj.scalar_type() != at::kInt || !rj.is_contiguous()) fail("rejected must be contiguous int32");
        rejected = (const int32_t*)rj.data_ptr();
        max_k = (int)rj.size(1);
    }
    const int B = (int)target.size(0), V = (int)target.size(1);
    const uint64_t seed = (uint64_t)integer(a[6]);
    const uint32_t step = (uint32_t)integer(a[7]), seq = (uint32_t)integer(a[8]);
    const int32_t* node = (const int32_t*)ptr(a[5]);
    int32_t *token = (int32_t*)ptr(a[9]), *status = (int32_t*)ptr(a[11]);
    float* residual = (float*)ptr(a[10]);
    const rsd_stream_t s = stream();
    return call([&] { return p_resample(&d, &t, B, V, rejected, max_k, node, seed, step, seq, token, residual, status, s); });
}

// bind(path of librsd, exception class)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    const char* path = n == 2 ? PyUnicode_AsUTF8(a[0]) : nullptr;
    if (!path) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "bind(path, exception class)");
        return nullptr;
    }
    static PyObject* bound = nullptr;         // one library per process: the entry points below are not per caller
    if (bound && PyUnicode_Compare(bound, a[0]) != 0) {
        PyErr_Format(PyExc_RuntimeError, "already bound to %U", bound);
        return nullptr;
    }
    void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
    if (!lib) {
        PyErr_SetString(PyExc_OSError, dlerror());
        return nullptr;
    }
    bool all = true;
    auto find = [&](auto& f, const char* name) {
        f = (std::remove_reference_t<decltype(f)>)dlsym(lib, name);
        all = all && f;
    };
    find(p_last_error, "rsd_last_error");
    find(p_filter_rows, "rsd_filter_rows");
    find(p_gumbel, "rsd_gumbel_topk_draft");
    find(p_sbs_step, "rsd_sbs_step");
    find(p_sbs_step_static, "rsd_sbs_step_static");
    find(p_sbs_draft_tree, "rsd_sbs_draft_tree");
    find(p_verify_tree, "rsd_verify_tree");
    find(p_verify_tree_rule, "rsd_verify_tree_rule");
    find(p_resample, "rsd_resample_residual");
    if (!all) {
        PyErr_Format(PyExc_OSError, "%s lacks an entry point", path);
        return nullptr;
    }
    if (!bound) {
        Py_INCREF(a[0]);
        bound = a[0];
    }
    Py_INCREF(a[1]);
    Py_XDECREF(g_error);
    g_error = a[1];
    Py_RETURN_NONE;
}

#define RSD_ENTRY(f, n) {#f, (PyCFunction)(void (*)(void))entry<f, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
    RSD_ENTRY(filter_rows, 7),
    RSD_ENTRY(gumbel_topk_draft, 15),
    RSD_ENTRY(sbs_step, 18),
    RSD_ENTRY(sbs_draft_tree, 15),
    RSD_ENTRY(verify_tree, 21),
    RSD_ENTRY(resample_residual, 12),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_rsdbind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__rsdbind() { return PyModule_Create(&module); }
