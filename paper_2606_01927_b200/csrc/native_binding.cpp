// Argument marshalling of the Python binding, in native code.
//
// A sampling call is a kernel of 5 to 20 us on small and ordinary batches; turning two dozen Python
// arguments into pointers with ctypes, allocating the outputs and looking up the stream through
// torch's Python layer took 19 us of host time per call, which was the rate such batches ran at.
// The same steps against torch's C++ interface take about a quarter of that.  Nothing of the sampling
// path is here: this file checks tensors, allocates what the caller did not pass, and calls the C ABI.

#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <stdexcept>
#include <string>

#include "albireo_sample.h"

namespace {

struct BadArgument : std::runtime_error { using std::runtime_error::runtime_error; };
struct PythonError {};      // a Python exception is already set

const at::Tensor *tensor_or_null(PyObject *o, const char *name) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) throw BadArgument(std::string(name) + " must be a torch tensor");
    return &THPVariable_Unpack(o);
}

// an optional contiguous array of one type, on the CUDA device or (host entry) in host memory
template <class T>
T *array(PyObject *o, const char *name, at::ScalarType dtype, bool cuda) {
    const at::Tensor *t = tensor_or_null(o, name);
    if (!t) return nullptr;
    if (t->scalar_type() != dtype || !t->is_contiguous() || (cuda ? !t->is_cuda() : !t->is_cpu()))
        throw BadArgument(std::string("expected contiguous ") + c10::toString(dtype) + " tensor on " + (cuda ? "cuda" : "cpu") +
                          " for " + name + ", got " + c10::toString(t->scalar_type()) + " on " + t->device().str());
    return (T *)t->data_ptr();
}

int64_t as_int(PyObject *o, const char *name) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) {
        if (!PyErr_ExceptionMatches(PyExc_TypeError)) throw PythonError{};
        PyErr_Clear();
        PyObject *i = PyNumber_Index(o);
        if (!i) { PyErr_Clear(); throw BadArgument(std::string(name) + " must be an integer"); }
        const long long w = PyLong_AsLongLong(i);
        Py_DECREF(i);
        if (w == -1 && PyErr_Occurred()) throw PythonError{};
        return w;
    }
    return v;
}
uint64_t as_u64(PyObject *o, const char *name) {
    PyObject *i = PyNumber_Index(o);
    if (!i) { PyErr_Clear(); throw BadArgument(std::string(name) + " must be an integer"); }
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(i);      // modulo 2^64, as a C conversion does
    Py_DECREF(i);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) throw PythonError{};
    return v;
}
bool as_bool(PyObject *o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw PythonError{};
    return v != 0;
}

// what the outputs of one call are allocated on
struct Where {
    bool host;
    c10::Device device;
    at::Tensor make(at::IntArrayRef shape, at::ScalarType dtype) const {
        return at::empty(shape, host ? at::TensorOptions(dtype).pinned_memory(true) : at::TensorOptions(dtype).device(device));
    }
};

// a caller's output tensor, or a new one
at::Tensor output(PyObject *o, const char *name, const Where &w, at::IntArrayRef shape, at::ScalarType dtype) {
    const at::Tensor *t = tensor_or_null(o, name);
    return t ? *t : w.make(shape, dtype);
}
at::Tensor list_output(PyObject *o, const char *name, const Where &w, int64_t B, int64_t n, at::ScalarType dtype) {
    const at::Tensor *t = tensor_or_null(o, name);
    if (!t) return w.make({B, n}, dtype);
    if (t->scalar_type() != dtype || t->numel() < B * n || !t->is_contiguous())
        throw BadArgument(std::string(name) + " must be a contiguous " + (dtype == at::kInt ? "int32" : "float32") + " tensor of B * num_top entries");
    return *t;
}

PyObject *wrap(const at::Tensor &t) {
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}

enum Entry { DEVICE = 0, HOST = 1, FIXED = 2 };
// positions of the positional arguments of sample()
enum Arg {
    A_ENTRY, A_HANDLE, A_DEVICE, A_LOGITS, A_T, A_K, A_TOPP, A_MINP, A_REP, A_PRES, A_FREQ, A_HID, A_HOFF, A_SEEDS, A_STEP,
    A_OUT_TOK, A_OUT_LP, A_STREAM, A_ROW_BASE, A_NUM_TOP, A_COUNTS, A_DBG_CAP, A_STATUS, A_FLAGS, A_B, A_V, A_EXP1,
    A_BF_IDS, A_BF_INDEX, A_RING, A_RING_HEAD, A_OUT_START, A_SEGS, A_SEG_ROW, A_OUT_TOP_IDS, A_OUT_TOP_LP, A_HTOT, A_COUNT
};

int dtype_code(const at::Tensor &t) {
    switch (t.scalar_type()) {
        case at::kFloat: return ALBIREO_F32;
        case at::kBFloat16: return ALBIREO_BF16;
        case at::kHalf: return ALBIREO_F16;
        default: throw BadArgument("logits must be float32, bfloat16 or float16");
    }
}

PyObject *sample_checked(PyObject *const *a) {
    const int entry = (int)as_int(a[A_ENTRY], "entry");
    albireo_sampler_t *h = (albireo_sampler_t *)(uintptr_t)as_u64(a[A_HANDLE], "handle");
    const at::Tensor *lp_ = tensor_or_null(a[A_LOGITS], "logits");
    if (!lp_) throw BadArgument("logits must be a torch tensor");
    const at::Tensor &logits = *lp_;
    const bool host = entry == HOST, cuda = !host;
    const int dt = dtype_code(logits);
    if (cuda ? !logits.is_cuda() : !logits.is_cpu()) throw BadArgument(std::string("logits must be on ") + (cuda ? "a CUDA device" : "the host"));
    const c10::Device dev(c10::kCUDA, host ? (c10::DeviceIndex)as_int(a[A_DEVICE], "device") : logits.device().index());

    albireo_sample_ext_t ext = {};
    ext.struct_size = sizeof ext;
    ext.flags = (uint32_t)as_int(a[A_FLAGS], "flags");
    ext.row_base = (uint32_t)as_int(a[A_ROW_BASE], "row_base");

    // the shape of the batch: [B, V], or rows in pieces [t, B, V / t]
    int64_t B, V, row_stride;
    if (entry == DEVICE && logits.dim() == 3) {
        if (logits.stride(2) != 1) throw BadArgument("logits in pieces must be [t, B, V/t] with unit stride along the last axis");
        const int64_t nseg = logits.size(0);
        B = a[A_B] == Py_None ? logits.size(1) : as_int(a[A_B], "B");
        V = a[A_V] == Py_None ? nseg * logits.size(2) : as_int(a[A_V], "V");
        ext.num_segments = (int32_t)nseg;
        ext.segment_stride_elems = logits.stride(0);
        ext.row_stride_elems = row_stride = logits.stride(1);
    } else {
        if (logits.dim() != 2 || (entry == DEVICE && logits.stride(1) != 1)) throw BadArgument("logits must be [B, V] with unit stride along V");
        B = a[A_B] == Py_None ? logits.size(0) : as_int(a[A_B], "B");
        V = a[A_V] == Py_None ? logits.size(1) : as_int(a[A_V], "V");
        row_stride = B > 1 ? logits.stride(0) : V;
        if (entry == DEVICE) ext.row_stride_elems = row_stride == V ? 0 : row_stride;
    }

    const Where where{host, dev};
    at::Tensor tokens = output(a[A_OUT_TOK], "out_tokens", where, {B}, at::kInt);
    at::Tensor logprobs = output(a[A_OUT_LP], "out_logprobs", where, {B}, at::kFloat);
    at::Tensor top_ids, top_lps, num_kept, num_topk, dbg, status;
    const int64_t num_top = as_int(a[A_NUM_TOP], "num_top"), dbg_cap = as_int(a[A_DBG_CAP], "dbg_cap");
    ext.num_top = (int32_t)num_top;
    if (num_top > 0) {
        top_ids = list_output(a[A_OUT_TOP_IDS], "out_top_ids", where, B, num_top, at::kInt);
        top_lps = list_output(a[A_OUT_TOP_LP], "out_top_logprobs", where, B, num_top, at::kFloat);
        ext.out_top_ids = (int32_t *)top_ids.data_ptr();
        ext.out_top_logprobs = (float *)top_lps.data_ptr();
    }
    if (as_bool(a[A_COUNTS])) {
        num_kept = where.make({B}, at::kInt);
        num_topk = where.make({B}, at::kInt);
        ext.out_num_kept = (int32_t *)num_kept.data_ptr();
        ext.out_num_topk = (int32_t *)num_topk.data_ptr();
    }
    if (dbg_cap > 0) {
        dbg = where.make({B, dbg_cap}, at::kInt);
        ext.dbg_cap = (int32_t)dbg_cap;
        ext.dbg_topk_ids = (int32_t *)dbg.data_ptr();
    }
    if (as_bool(a[A_STATUS])) {
        status = where.make({B}, at::kInt);
        ext.out_row_status = (uint32_t *)status.data_ptr();
    }

    ext.history_output_start = array<const int32_t>(a[A_OUT_START], "output_start", at::kInt, true);
    const void *seg_ptrs[ALBIREO_MAX_SEGMENTS];
    if (a[A_SEGS] != Py_None) {
        // one [rows, V/t] buffer per piece (e.g. the peers' vocabulary shards in symmetric memory), read in place
        PyObject *seq = PySequence_Fast(a[A_SEGS], "segment_tensors must be a sequence of tensors");
        if (!seq) throw PythonError{};
        struct Release { PyObject *o; ~Release() { Py_DECREF(o); } } release{seq};
        const Py_ssize_t t = PySequence_Fast_GET_SIZE(seq);
        const at::Tensor *first = nullptr;
        for (Py_ssize_t j = 0; j < t; ++j) {
            const at::Tensor *x = tensor_or_null(PySequence_Fast_GET_ITEM(seq, j), "segment_tensors");
            if (x && !first) first = x;
            if (!x || x->dim() != 2 || x->stride(1) != 1 || x->scalar_type() != first->scalar_type() || x->size(1) != first->size(1) ||
                x->stride(0) != first->stride(0))
                throw BadArgument("segment_tensors must be same-shaped [rows, V/t] tensors with unit stride along V/t");
            if (j < ALBIREO_MAX_SEGMENTS) seg_ptrs[j] = x->data_ptr();
        }
        if (!first) throw BadArgument("segment_tensors must not be empty");
        ext.num_segments = (int32_t)t;
        ext.segment_ptrs = seg_ptrs;
        ext.segment_row_offset = as_int(a[A_SEG_ROW], "segment_row_offset");
        ext.row_stride_elems = first->stride(0);
    }
    if (const at::Tensor *e = tensor_or_null(a[A_EXP1], "exp1")) {
        if (e->scalar_type() != at::kFloat || e->dim() != 2 || e->stride(1) != 1 || e->device() != logits.device())
            throw BadArgument("exp1 must be a float32 [B, V] tensor on the logits' device");
        ext.exp1 = (const float *)e->data_ptr();
        ext.exp1_stride_elems = (B <= 1 || e->stride(0) == V) ? 0 : e->stride(0);
    }
    if (const at::Tensor *ids = tensor_or_null(a[A_BF_IDS], "backfill_ids")) {
        ext.backfill_ids = array<int32_t>(a[A_BF_IDS], "backfill_ids", at::kInt, true);
        ext.backfill_index = array<const int32_t>(a[A_BF_INDEX], "backfill_index", at::kInt, true);
        ext.backfill_len = ids->numel();
    }
    if (const at::Tensor *ring = tensor_or_null(a[A_RING], "feedback_ring")) {
        if (ring->scalar_type() != at::kLong || !ring->is_contiguous())
            throw BadArgument("feedback_ring must be a contiguous int64 tensor (device, or pinned host memory)");
        ext.feedback_ring = (uint64_t *)ring->data_ptr();
        ext.feedback_cap = ring->numel();
        ext.feedback_head = as_int(a[A_RING_HEAD], "feedback_head");
    }

    const float *T = array<const float>(a[A_T], "temperature", at::kFloat, cuda);
    const int32_t *k = array<const int32_t>(a[A_K], "top_k", at::kInt, cuda);
    const float *topp = array<const float>(a[A_TOPP], "top_p", at::kFloat, cuda), *minp = array<const float>(a[A_MINP], "min_p", at::kFloat, cuda);
    const float *rep = array<const float>(a[A_REP], "repetition_penalty", at::kFloat, cuda);
    const float *pres = array<const float>(a[A_PRES], "presence_penalty", at::kFloat, cuda);
    const float *freq = array<const float>(a[A_FREQ], "frequency_penalty", at::kFloat, cuda);
    const int32_t *hid = array<const int32_t>(a[A_HID], "history_ids", at::kInt, cuda);
    const int32_t *hoff = array<const int32_t>(a[A_HOFF], "history_offsets", at::kInt, cuda);
    const uint64_t *seeds = array<const uint64_t>(a[A_SEEDS], "seeds", at::kLong, cuda);
    const uint64_t step = as_u64(a[A_STEP], "step");
    int64_t htot = 0;
    if (a[A_HTOT] != Py_None) htot = as_int(a[A_HTOT], "history_total");
    else if (const at::Tensor *t = tensor_or_null(a[A_HID], "history_ids")) htot = t->numel();

    void *stream;
    if (a[A_STREAM] == Py_None) stream = c10::cuda::getCurrentCUDAStream(dev.index()).stream();
    else {
        PyObject *s = PyObject_GetAttrString(a[A_STREAM], "cuda_stream");
        if (!s) throw PythonError{};
        const uint64_t v = as_u64(s, "stream");
        Py_DECREF(s);
        stream = (void *)(uintptr_t)v;
    }

    int rc;
    {
        c10::cuda::CUDAGuard guard(dev);
        const void *x = logits.data_ptr();
        int32_t *tok = (int32_t *)tokens.data_ptr();
        float *lp = (float *)logprobs.data_ptr();
        const int32_t b32 = (int32_t)B, v32 = (int32_t)V;
        // other Python threads run meanwhile: the host entry waits for the device, and a launch waits for it where
        // the queue is full
        PyThreadState *ts = PyEval_SaveThread();
        rc = entry == DEVICE ? albireo_sample(h, x, b32, v32, dt, T, k, topp, minp, rep, pres, freq, hid, hoff, seeds, step, tok, lp, stream, &ext)
             : entry == HOST ? albireo_sample_host(h, x, b32, v32, dt, T, k, topp, minp, rep, pres, freq, hid, hoff, htot, seeds, step, tok, lp, stream, &ext)
                             : albireo_sample_fixed_scratch(x, b32, v32, dt, T, k, topp, minp, rep, pres, freq, hid, hoff, htot, seeds, step, tok, lp, stream, &ext);
        PyEval_RestoreThread(ts);
    }
    if (rc != ALBIREO_OK) return PyLong_FromLong(rc);
    // a tensor the caller passed is returned as the object it passed
    auto given = [&](int i, const at::Tensor &t) -> PyObject * { if (a[i] != Py_None) { Py_INCREF(a[i]); return a[i]; } return wrap(t); };
    PyObject *out = PyTuple_New(8);
    if (!out) throw PythonError{};
    PyTuple_SET_ITEM(out, 0, given(A_OUT_TOK, tokens));
    PyTuple_SET_ITEM(out, 1, given(A_OUT_LP, logprobs));
    PyTuple_SET_ITEM(out, 2, num_top > 0 ? given(A_OUT_TOP_IDS, top_ids) : wrap(top_ids));
    PyTuple_SET_ITEM(out, 3, num_top > 0 ? given(A_OUT_TOP_LP, top_lps) : wrap(top_lps));
    PyTuple_SET_ITEM(out, 4, wrap(num_kept));
    PyTuple_SET_ITEM(out, 5, wrap(num_topk));
    PyTuple_SET_ITEM(out, 6, wrap(dbg));
    PyTuple_SET_ITEM(out, 7, wrap(status));
    return out;
}

// (torch's own errors reach Python as torch's types: out of memory as torch.OutOfMemoryError)
PyObject *sample(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != A_COUNT) { PyErr_Format(PyExc_TypeError, "sample takes %d positional arguments, got %zd", (int)A_COUNT, n); return nullptr; }
    try {
        return sample_checked(args);
    } catch (const BadArgument &e) {
        PyErr_SetString(PyExc_ValueError, e.what());
    } catch (const PythonError &) {
    }
    return nullptr;
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"sample", (PyCFunction)(void (*)(void))sample, METH_FASTCALL,
     "One sampling call with its arguments in the order of the binding; a tuple of output tensors, or the C ABI's error code."},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of the sampler's Python binding.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
