// CPython front of the C ABI for the calls a decode loop makes every step: unpacks the arguments (tensors by their
// data_ptr(), sequence lists, the current stream) and calls the entry point of the same name with the interpreter
// lock released.  Nothing is computed here.
//
// Tensors and the current stream are read through torch's C++ interface; through Python calls they took 0.6 us of a call's
// 3.2 (2.6 now, of which the launch is 1.9 and the unpacking 0.2).
//
// Why not ctypes for these: with ctypes a decode-step call spent 8.3 us on the host (torch.cuda.current_stream()
// 3.2, argument conversion about 1.2, the entry point itself 3.7), and a program that launches its steps directly is
// bound by that, not by kernels of 2 to 6 us.  The rarely used entry points stay with ctypes.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <vector>

#include "../../include/tokenbutler.h"

// Read from the file by build.py and binding.py: another torch or Python needs another build.
extern "C" __attribute__((used, visibility("default"))) const char tb_calls_abi[] = TB_CALLS_ABI;

namespace {

PyObject* g_data_ptr;        // "data_ptr"
PyObject* g_cuda_stream;     // "cuda_stream"
PyObject* g_shape;           // "shape"

// Each reader returns false with a Python exception set, or throws what torch throws (a tensor without storage, no
// device): guarded() makes that a Python exception.

bool read_pointer(PyObject* o, void** out) {      // a tensor, or None
    *out = nullptr;
    if (o == Py_None) return true;
    if (THPVariable_Check(o)) {
        *out = THPVariable_Unpack(o).data_ptr();
        return true;
    }
    PyObject* v = PyObject_CallMethodNoArgs(o, g_data_ptr);   // whatever else says where it is
    if (!v) return false;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return *out || !PyErr_Occurred();
}

bool read_address(PyObject* o, void** out) {      // an integer address, or None
    *out = nullptr;
    if (o == Py_None) return true;
    *out = PyLong_AsVoidPtr(o);
    return *out || !PyErr_Occurred();
}

bool read_int(PyObject* o, int32_t* out) {
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    if (v == (unsigned long)-1 && PyErr_Occurred()) return false;
    *out = (int32_t)v;
    return true;
}

// A list of integers, or None.  Short lists (a call takes at most 64 sequences) live on the stack.
struct IntList {
    int32_t small[64];
    std::vector<int32_t> large;
    const int32_t* data = nullptr;
    Py_ssize_t n = 0;
    bool read(PyObject* o) {
        if (o == Py_None) return true;
        PyObject* seq = PySequence_Fast(o, "a sequence of integers is expected");
        if (!seq) return false;
        n = PySequence_Fast_GET_SIZE(seq);
        int32_t* dst = small;
        if (n > 64) large.resize(n), dst = large.data();
        data = dst;
        for (Py_ssize_t i = 0; i < n; ++i) {
            PyObject* item = PySequence_Fast_GET_ITEM(seq, i);
            bool ok;
            if (PyLong_CheckExact(item)) {
                ok = read_int(item, dst + i);
            } else {                              // whatever int() takes
                PyObject* v = PyNumber_Long(item);
                ok = v && read_int(v, dst + i);
                Py_XDECREF(v);
            }
            if (!ok) { Py_DECREF(seq); return false; }
        }
        Py_DECREF(seq);
        return true;
    }
};

// A ctypes structure, through the buffer protocol.
template <typename T>
bool read_struct(PyObject* o, T* out) {
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    const bool ok = b.len == (Py_ssize_t)sizeof(T);
    if (ok) *out = *static_cast<const T*>(b.buf);
    PyBuffer_Release(&b);
    if (!ok) PyErr_SetString(PyExc_TypeError, "not the structure this call takes");
    return ok;
}

// A torch stream, or None for the current stream of the current device.
bool read_stream(PyObject* o, void** out) {
    if (o == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* v = PyObject_GetAttr(o, g_cuda_stream);
    if (!v) return false;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return *out || !PyErr_Occurred();
}

bool want(Py_ssize_t got, Py_ssize_t n) {
    if (got == n) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", n, got);
    return false;
}

template <typename F>
PyObject* call(F&& f) {
    tb_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

// (ctx, layer_begin, layer_count, seq_ids, n_new, k, v, stream)
PyObject* append_kv(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void *ctx, *k, *v, *stream;
    int32_t lb, lc;
    IntList ids, n_new;
    if (!want(n, 8) || !read_address(a[0], &ctx) || !read_int(a[1], &lb) || !read_int(a[2], &lc) || !ids.read(a[3]) ||
        !n_new.read(a[4]) || !read_pointer(a[5], &k) || !read_pointer(a[6], &v) || !read_stream(a[7], &stream))
        return nullptr;
    return call([&] { return tb_append_kv((tb_ctx*)ctx, lb, lc, ids.data, n_new.data, (int32_t)n_new.n, k, v, stream); });
}

// (ctx, layer_begin, layer_count, seq_ids, pos_begin, pos_end, n_seq, stream)
PyObject* project_keys(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void *ctx, *stream;
    int32_t lb, lc, n_seq;
    IntList ids, pb, pe;
    if (!want(n, 8) || !read_address(a[0], &ctx) || !read_int(a[1], &lb) || !read_int(a[2], &lc) || !ids.read(a[3]) ||
        !pb.read(a[4]) || !pe.read(a[5]) || !read_int(a[6], &n_seq) || !read_stream(a[7], &stream))
        return nullptr;
    return call([&] { return tb_project_keys((tb_ctx*)ctx, lb, lc, ids.data, pb.data, pe.data, n_seq, stream); });
}

// (ctx, layer_begin, layer_count, seq_ids, n_seq, q_imp, params, idx_out, cnt_out, stream)
PyObject* select_topk(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void *ctx, *q_imp, *idx, *cnt, *stream;
    int32_t lb, lc, n_seq;
    IntList ids;
    tb_select_params p;
    if (!want(n, 10) || !read_address(a[0], &ctx) || !read_int(a[1], &lb) || !read_int(a[2], &lc) || !ids.read(a[3]) ||
        !read_int(a[4], &n_seq) || !read_pointer(a[5], &q_imp) || !read_struct(a[6], &p) || !read_pointer(a[7], &idx) ||
        !read_pointer(a[8], &cnt) || !read_stream(a[9], &stream))
        return nullptr;
    return call([&] {
        return tb_select_topk((tb_ctx*)ctx, lb, lc, ids.data, n_seq, (const float*)q_imp, &p, (int32_t*)idx, (int32_t*)cnt, stream);
    });
}

// (ctx, layer_begin, layer_count, seq_ids, n_seq, q, params, idx, cnt, sm_scale, out, lse, stream)
PyObject* sparse_decode_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void *ctx, *q, *idx, *cnt, *out, *lse, *stream;
    int32_t lb, lc, n_seq;
    IntList ids;
    tb_select_params p;
    if (!want(n, 13) || !read_address(a[0], &ctx) || !read_int(a[1], &lb) || !read_int(a[2], &lc) || !ids.read(a[3]) ||
        !read_int(a[4], &n_seq) || !read_pointer(a[5], &q) || !read_struct(a[6], &p) || !read_pointer(a[7], &idx) ||
        !read_pointer(a[8], &cnt))
        return nullptr;
    const double scale = PyFloat_AsDouble(a[9]);
    if (scale == -1.0 && PyErr_Occurred()) return nullptr;
    if (!read_pointer(a[10], &out) || !read_pointer(a[11], &lse) || !read_stream(a[12], &stream)) return nullptr;
    return call([&] {
        return tb_sparse_decode_attention((tb_ctx*)ctx, lb, lc, ids.data, n_seq, q, &p, (const int32_t*)idx, (const int32_t*)cnt,
                                          (float)scale, (float*)out, (float*)lse, stream);
    });
}

// A tensor (or whatever else has a shape and says where it is) and its leading sizes; `cols` may be null.
bool read_matrix(PyObject* o, void** out, int32_t* rows, int32_t* cols) {
    int32_t* sizes[2] = {rows, cols};
    if (THPVariable_Check(o) && THPVariable_Unpack(o).dim() >= (cols ? 2 : 1)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        *out = t.data_ptr();
        for (int i = 0; i < (cols ? 2 : 1); ++i) *sizes[i] = (int32_t)t.size(i);
        return true;
    }
    PyObject* shape = PyObject_GetAttr(o, g_shape);
    if (!shape) return false;
    bool ok = true;
    for (int i = 0; i < (cols ? 2 : 1) && ok; ++i) {
        PyObject* n = PySequence_GetItem(shape, i);    // (an IndexError where there are fewer)
        ok = n && read_int(n, sizes[i]);
        Py_XDECREF(n);
    }
    Py_DECREF(shape);
    return ok && o != Py_None && read_pointer(o, out);
}

// (dtype, n_q_heads, n_slots, imp_dim, activation, ln_eps, ln_weight, ln_bias, w1, w2, hidden, scratch, q_imp, stream)
PyObject* predict_importance_queries(PyObject*, PyObject* const* a, Py_ssize_t n) {
    tb_predictor p;
    void *lw, *lb, *w1, *w2, *hidden, *scratch, *q_imp, *stream;
    int32_t n_tok;
    if (!want(n, 14) || !read_int(a[0], &p.dtype) || !read_int(a[1], &p.n_q_heads) || !read_int(a[2], &p.n_slots) ||
        !read_int(a[3], &p.imp_dim) || !read_int(a[4], &p.activation))
        return nullptr;
    const double eps = PyFloat_AsDouble(a[5]);
    if (eps == -1.0 && PyErr_Occurred()) return nullptr;
    if (!read_pointer(a[6], &lw) || !read_pointer(a[7], &lb) || !read_matrix(a[8], &w1, &p.hidden_dim, nullptr) || !read_pointer(a[9], &w2) ||
        !read_matrix(a[10], &hidden, &n_tok, &p.model_dim) || !read_pointer(a[11], &scratch) || !read_pointer(a[12], &q_imp) ||
        !read_stream(a[13], &stream))
        return nullptr;
    p.ln_eps = (float)eps;
    p.ln_weight = lw, p.ln_bias = lb, p.w1 = w1, p.w2 = w2;
    return call([&] { return tb_predict_importance_queries(&p, hidden, n_tok, (float*)scratch, (float*)q_imp, stream); });
}

template <PyObject* (*f)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    return f(self, a, n);
    END_HANDLE_TH_ERRORS
}

#define TB_METHOD(name) {#name, (PyCFunction)(void (*)(void))guarded<name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {TB_METHOD(append_kv), TB_METHOD(project_keys), TB_METHOD(select_topk), TB_METHOD(sparse_decode_attention),
                         TB_METHOD(predict_importance_queries), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tokenbutler", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tokenbutler(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    g_shape = PyUnicode_InternFromString("shape");
    if (!g_data_ptr || !g_cuda_stream || !g_shape) return nullptr;
    return PyModule_Create(&module);
}
