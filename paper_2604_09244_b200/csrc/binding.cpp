// Native side of the Python binding (module `_native`): turns the arguments of the C-ABI calls -- tensors, sample
// descriptors, output records -- into plain pointers and calls libmvla_prune.so.  No arithmetic of the method here.
//
// A step of the smallest sizes is 12 us of GPU work, so what a call costs on the host is part of its time: the same
// marshalling through ctypes (two structures, some fourteen tensors checked one by one, the current stream) took 8.7 us
// of interpreter work per call, here about 1 us.
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>

#include <cstring>

#include "mvla_prune.h"

namespace {

constexpr int kMaxBatch = 64;       // samples per call (the library refuses more)

// Attribute names of StepOutputs, in the order of mvla_outputs, and of the sample descriptors.
enum { OUT_HIDDEN, OUT_K, OUT_V, KEPT, OFFSETS, BUDGETS, ATTN, AHAT, Z, DIAG, PATCH_X, PATCH_XHAT, PATCH_INFO, PATCH_DIAG, N_OUT };
const char* const kOutNames[N_OUT] = {"out_hidden", "out_k", "out_v", "kept_idx", "out_offsets", "budgets", "attn",
                                      "ahat", "z", "diag", "patch_x", "patch_xhat", "patch_info", "patch_diag"};
const char* const kSampleInts[8] = {"seq_off", "off_txt", "n_txt", "off_2d", "n_2d", "off_3d", "n_3d", "state_slot"};
const char* const kSampleFloats[3] = {"keep_2d", "keep_3d", "keep_total"};
PyObject* g_out_names[N_OUT];
PyObject* g_int_names[8];
PyObject* g_float_names[3];
PyObject* g_cuda_stream;            // "cuda_stream"

// Device pointer of a tensor, null for None.  False: a Python exception is set.
bool tensor_ptr(PyObject* o, void** p, const at::Tensor** tensor = nullptr)
{
    *p = nullptr;
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor or None");
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
        PyErr_SetString(PyExc_AssertionError, "device-resident contiguous tensors only");
        return false;
    }
    *p = t.data_ptr();
    if (tensor) *tensor = &t;
    return true;
}

// Rows of the packed tensor q (its first dimension).
bool rows_of(PyObject* q, int64_t* rows)
{
    if (!THPVariable_Check(q) || THPVariable_Unpack(q).dim() < 1) {
        PyErr_SetString(PyExc_TypeError, "q must be a tensor of [rows, heads, head_dim]");
        return false;
    }
    *rows = THPVariable_Unpack(q).size(0);
    return true;
}

bool int_of(PyObject* o, int64_t* v)
{
    *v = PyLong_AsLongLong(o);
    if (*v == -1 && PyErr_Occurred()) {                       // not an int (a NumPy integer, say): what int() makes of it
        PyErr_Clear();
        PyObject* i = PyNumber_Long(o);
        if (!i) return false;
        *v = PyLong_AsLongLong(i);
        Py_DECREF(i);
        if (*v == -1 && PyErr_Occurred()) return false;
    }
    return true;
}

// One descriptor from an object with the descriptor's field names.
bool sample_from(PyObject* o, mvla_sample* s)
{
    int32_t* const ints[8] = {&s->seq_off, &s->off_txt, &s->n_txt, &s->off_2d, &s->n_2d, &s->off_3d, &s->n_3d, &s->state_slot};
    double* const floats[3] = {&s->keep_2d, &s->keep_3d, &s->keep_total};
    for (int i = 0; i < 8; ++i) {
        PyObject* a = PyObject_GetAttr(o, g_int_names[i]);
        if (!a) {
            if (i < 7 || !PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
            PyErr_Clear();                                    // state_slot may be missing: slot 0
            s->state_slot = 0;
            continue;
        }
        int64_t v = 0;
        const bool ok = int_of(a, &v);
        Py_DECREF(a);
        if (!ok) return false;
        *ints[i] = static_cast<int32_t>(v);
    }
    for (int i = 0; i < 3; ++i) {
        PyObject* a = PyObject_GetAttr(o, g_float_names[i]);
        if (!a) return false;
        *floats[i] = PyFloat_AsDouble(a);
        Py_DECREF(a);
        if (*floats[i] == -1.0 && PyErr_Occurred()) return false;
    }
    return true;
}

// The call's descriptors: the caller's ctypes array as it lies in memory, or a list / tuple of objects converted here.
struct Samples {
    mvla_sample own[kMaxBatch];
    const mvla_sample* ptr = nullptr;
    int n = 0;
    Py_buffer view;
    bool viewed = false;
    ~Samples() { if (viewed) PyBuffer_Release(&view); }
    bool take(PyObject* o)
    {
        if (PyList_Check(o) || PyTuple_Check(o)) {
            const Py_ssize_t len = PySequence_Fast_GET_SIZE(o);
            n = static_cast<int>(len);
            ptr = own;
            // more than the library takes: only the count matters, it answers MVLA_ERR_CAPACITY
            for (Py_ssize_t i = 0; i < len && i < kMaxBatch; ++i)
                if (!sample_from(PySequence_Fast_GET_ITEM(o, i), own + i)) return false;
            return true;
        }
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) == 0) {
            viewed = true;
            if (view.len % static_cast<Py_ssize_t>(sizeof(mvla_sample)) != 0) {
                PyErr_SetString(PyExc_TypeError, "samples: not an array of sample descriptors");
                return false;
            }
            ptr = static_cast<const mvla_sample*>(view.buf);
            n = static_cast<int>(view.len / static_cast<Py_ssize_t>(sizeof(mvla_sample)));
            return true;
        }
        PyErr_Clear();
        PyObject* seq = PySequence_List(o);                   // any other sequence of objects
        if (!seq) return false;
        const bool ok = take(seq);
        Py_DECREF(seq);
        return ok;
    }
    int64_t visual() const
    {
        int64_t v = 0;
        for (int i = 0; i < n && i < kMaxBatch; ++i) v += ptr[i].n_2d + ptr[i].n_3d;
        return v;
    }
};

bool stream_of(PyObject* o, void** st)
{
    if (o == Py_None) {
        *st = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = PyObject_GetAttr(o, g_cuda_stream);
    if (!h) return false;
    *st = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

bool arg_count(Py_ssize_t got, Py_ssize_t want)
{
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return false;
}

// Pointers of a StepOutputs record; the tensors stay alive through the record.
bool outputs_of(PyObject* out, mvla_outputs* o, unsigned wanted)
{
    std::memset(o, 0, sizeof *o);
    void** const dst[N_OUT] = {&o->out_hidden, &o->out_k, &o->out_v, reinterpret_cast<void**>(&o->kept_idx),
                               reinterpret_cast<void**>(&o->out_offsets), reinterpret_cast<void**>(&o->budgets),
                               reinterpret_cast<void**>(&o->attn), reinterpret_cast<void**>(&o->ahat),
                               reinterpret_cast<void**>(&o->z), reinterpret_cast<void**>(&o->diag),
                               reinterpret_cast<void**>(&o->patch_x), reinterpret_cast<void**>(&o->patch_xhat),
                               reinterpret_cast<void**>(&o->patch_info), reinterpret_cast<void**>(&o->patch_diag)};
    for (int i = 0; i < N_OUT; ++i) {
        if (!((wanted >> i) & 1u)) continue;
        PyObject* a = PyObject_GetAttr(out, g_out_names[i]);
        if (!a) return false;
        const bool ok = tensor_ptr(a, dst[i]);
        Py_DECREF(a);
        if (!ok) return false;
    }
    return true;
}

// The library call itself runs without the interpreter lock: a launch may block when the device's queue is full.
template <class F>
int32_t unlocked(F call)
{
    PyThreadState* save = PyEval_SaveThread();
    const int32_t rc = call();
    PyEval_RestoreThread(save);
    return rc;
}
mvla_ctx* ctx_of(PyObject* h) { return static_cast<mvla_ctx*>(PyLong_AsVoidPtr(h)); }

#define MVLA_TRY try {
#define MVLA_CATCH                                                                    \
    } catch (const std::exception& e) {                                               \
        PyErr_SetString(PyExc_RuntimeError, e.what());                                \
        return nullptr;                                                               \
    }

// prune_step(ctx, point, samples, mode, flags, q, k, v, hidden, rand_u, changed_rows, out, stream) -> rows kept, or < 0
PyObject* py_prune_step(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 13)) return nullptr;
    int64_t point, mode, flags;
    if (!int_of(a[1], &point) || !int_of(a[3], &mode) || !int_of(a[4], &flags)) return nullptr;
    Samples s;
    if (!s.take(a[2])) return nullptr;
    mvla_tensors in;
    std::memset(&in, 0, sizeof in);
    void *q, *k, *v, *hidden, *u, *st;
    if (!tensor_ptr(a[5], &q) || !tensor_ptr(a[6], &k) || !tensor_ptr(a[7], &v) || !tensor_ptr(a[8], &hidden) ||
        !tensor_ptr(a[9], &u) || !rows_of(a[5], &in.rows))
        return nullptr;
    in.q = q; in.k = k; in.v = v; in.hidden = hidden; in.rand_u = static_cast<const float*>(u);
    Py_buffer mask;
    const bool masked = a[10] != Py_None;
    if (masked) {                                             // a host byte per row, read during the call
        if (PyObject_GetBuffer(a[10], &mask, PyBUF_SIMPLE) != 0) return nullptr;
        if (mask.len != in.rows) {
            PyBuffer_Release(&mask);
            PyErr_SetString(PyExc_AssertionError, "one byte per row of the packed tensors");
            return nullptr;
        }
        in.changed_rows = static_cast<const uint8_t*>(mask.buf);
    }
    mvla_outputs out;
    int32_t rc = 0, total = 0;
    const bool ok = outputs_of(a[11], &out, ~0u) && stream_of(a[12], &st);
    mvla_ctx* ctx = ctx_of(a[0]);
    if (ok)
        rc = unlocked([&] {
            return mvla_prune_step(ctx, static_cast<int32_t>(point), s.n, s.ptr, static_cast<int32_t>(mode),
                                   static_cast<uint32_t>(flags), &in, &out, &total, st);
        });
    if (masked) PyBuffer_Release(&mask);
    if (!ok) return nullptr;
    return PyLong_FromLong(rc != MVLA_OK ? rc : total);
    MVLA_CATCH
}

// salience(ctx, samples, q, k, hidden, attn_out, l1_out, stream) -> (status, attn_out, l1_out); a missing attn_out, and a
// missing l1_out beside `hidden`, is allocated on q's device
PyObject* py_salience(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 8)) return nullptr;
    Samples s;
    if (!s.take(a[1])) return nullptr;
    int64_t rows;
    void *q, *k, *hidden, *attn, *l1, *st;
    const at::Tensor* qt = nullptr;
    if (!tensor_ptr(a[2], &q, &qt) || !tensor_ptr(a[3], &k) || !tensor_ptr(a[4], &hidden) || !rows_of(a[2], &rows) ||
        !stream_of(a[7], &st))
        return nullptr;
    PyObject *attn_o = a[5], *l1_o = a[6];
    Py_INCREF(attn_o);
    Py_INCREF(l1_o);
    auto fresh = [&](PyObject** o) {
        Py_DECREF(*o);
        *o = THPVariable_Wrap(at::empty({s.visual()}, qt->options().dtype(at::kFloat)));
    };
    if (attn_o == Py_None) fresh(&attn_o);
    if (l1_o == Py_None && hidden) fresh(&l1_o);
    PyObject* ret = nullptr;
    if (attn_o && l1_o && tensor_ptr(attn_o, &attn) && tensor_ptr(l1_o, &l1)) {
        mvla_ctx* ctx = ctx_of(a[0]);
        const int32_t rc = unlocked([&] {
            return mvla_salience(ctx, s.n, s.ptr, q, k, hidden, rows, static_cast<float*>(attn), static_cast<float*>(l1), st);
        });
        ret = Py_BuildValue("(iOO)", rc, attn_o, l1_o);
    }
    Py_XDECREF(attn_o);
    Py_XDECREF(l1_o);
    return ret;
    MVLA_CATCH
}

// select(ctx, point, samples, mode, flags, attn, l1, out, stream) -> status
PyObject* py_select(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 9)) return nullptr;
    int64_t point, mode, flags;
    if (!int_of(a[1], &point) || !int_of(a[3], &mode) || !int_of(a[4], &flags)) return nullptr;
    Samples s;
    void *attn, *l1, *st;
    mvla_outputs o;
    constexpr unsigned kWanted = 1u << KEPT | 1u << OFFSETS | 1u << BUDGETS | 1u << AHAT | 1u << Z | 1u << DIAG;
    if (!s.take(a[2]) || !tensor_ptr(a[5], &attn) || !tensor_ptr(a[6], &l1) || !outputs_of(a[7], &o, kWanted) ||
        !stream_of(a[8], &st))
        return nullptr;
    mvla_ctx* ctx = ctx_of(a[0]);
    return PyLong_FromLong(unlocked([&] {
        return mvla_select(ctx, static_cast<int32_t>(point), s.n, s.ptr, static_cast<int32_t>(mode),
                           static_cast<uint32_t>(flags), static_cast<const float*>(attn), static_cast<const float*>(l1),
                           o.kept_idx, o.out_offsets, o.budgets, o.ahat, o.z, o.diag, st);
    }));
    MVLA_CATCH
}

// compact(ctx, samples, kept_idx, out_offsets, total, hidden, k, v, out_hidden, out_k, out_v, stream) -> status
PyObject* py_compact(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 12)) return nullptr;
    Samples s;
    int64_t total;
    void *kept, *offs, *src[3], *dst[3], *st;
    if (!s.take(a[1]) || !tensor_ptr(a[2], &kept) || !tensor_ptr(a[3], &offs) || !int_of(a[4], &total)) return nullptr;
    for (int i = 0; i < 3; ++i)
        if (!tensor_ptr(a[5 + i], &src[i]) || !tensor_ptr(a[8 + i], &dst[i])) return nullptr;
    if (!stream_of(a[11], &st)) return nullptr;
    mvla_ctx* ctx = ctx_of(a[0]);
    return PyLong_FromLong(unlocked([&] {
        return mvla_compact(ctx, s.n, s.ptr, static_cast<const int32_t*>(kept), static_cast<const int32_t*>(offs),
                            static_cast<int32_t>(total), src[0], src[1], src[2], dst[0], dst[1], dst[2], st);
    }));
    MVLA_CATCH
}

// patch_indicators(ctx, samples, q, k, hidden, attn_out, x_out, stream) -> status
PyObject* py_patch_indicators(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 8)) return nullptr;
    Samples s;
    int64_t rows;
    void *q, *k, *hidden, *attn, *x, *st;
    if (!s.take(a[1]) || !tensor_ptr(a[2], &q) || !tensor_ptr(a[3], &k) || !tensor_ptr(a[4], &hidden) ||
        !tensor_ptr(a[5], &attn) || !tensor_ptr(a[6], &x) || !rows_of(a[2], &rows) || !stream_of(a[7], &st))
        return nullptr;
    mvla_ctx* ctx = ctx_of(a[0]);
    return PyLong_FromLong(unlocked([&] {
        return mvla_patch_indicators(ctx, s.n, s.ptr, q, k, hidden, rows, static_cast<float*>(attn), static_cast<float*>(x), st);
    }));
    MVLA_CATCH
}

// patch_select(ctx, point, samples, flags, attn, x, rand_u, out, stream) -> status
PyObject* py_patch_select(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 9)) return nullptr;
    int64_t point, flags;
    if (!int_of(a[1], &point) || !int_of(a[3], &flags)) return nullptr;
    Samples s;
    void *attn, *x, *u, *st;
    mvla_outputs o;
    constexpr unsigned kWanted = 1u << KEPT | 1u << OFFSETS | 1u << BUDGETS | 1u << PATCH_XHAT | 1u << PATCH_INFO | 1u << PATCH_DIAG;
    if (!s.take(a[2]) || !tensor_ptr(a[4], &attn) || !tensor_ptr(a[5], &x) || !tensor_ptr(a[6], &u) ||
        !outputs_of(a[7], &o, kWanted) || !stream_of(a[8], &st))
        return nullptr;
    mvla_ctx* ctx = ctx_of(a[0]);
    return PyLong_FromLong(unlocked([&] {
        return mvla_patch_select(ctx, static_cast<int32_t>(point), s.n, s.ptr, static_cast<uint32_t>(flags),
                                 static_cast<const float*>(attn), static_cast<const float*>(x), static_cast<const float*>(u),
                                 o.kept_idx, o.out_offsets, o.budgets, o.patch_xhat, o.patch_info, o.patch_diag, st);
    }));
    MVLA_CATCH
}

// fill_samples(array, sequence): descriptors from objects with the descriptor's field names, into a ctypes array
PyObject* py_fill_samples(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    MVLA_TRY
    if (!arg_count(n, 2)) return nullptr;
    PyObject* seq = PySequence_Fast(a[1], "samples: expected a sequence");
    if (!seq) return nullptr;
    Py_buffer view;
    bool ok = PyObject_GetBuffer(a[0], &view, PyBUF_WRITABLE) == 0;
    if (ok) {
        const Py_ssize_t len = PySequence_Fast_GET_SIZE(seq);
        if (view.len < len * static_cast<Py_ssize_t>(sizeof(mvla_sample))) {
            PyErr_SetString(PyExc_ValueError, "array too small");
            ok = false;
        }
        for (Py_ssize_t i = 0; ok && i < len; ++i)
            ok = sample_from(PySequence_Fast_GET_ITEM(seq, i), static_cast<mvla_sample*>(view.buf) + i);
        PyBuffer_Release(&view);
    }
    Py_DECREF(seq);
    if (!ok) return nullptr;
    Py_RETURN_NONE;
    MVLA_CATCH
}

#define MVLA_FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {MVLA_FAST("prune_step", py_prune_step), MVLA_FAST("salience", py_salience),
                          MVLA_FAST("select", py_select), MVLA_FAST("compact", py_compact),
                          MVLA_FAST("patch_indicators", py_patch_indicators), MVLA_FAST("patch_select", py_patch_select),
                          MVLA_FAST("fill_samples", py_fill_samples), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of libmvla_prune.so", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native()
{
    for (int i = 0; i < N_OUT; ++i) if (!(g_out_names[i] = PyUnicode_InternFromString(kOutNames[i]))) return nullptr;
    for (int i = 0; i < 8; ++i) if (!(g_int_names[i] = PyUnicode_InternFromString(kSampleInts[i]))) return nullptr;
    for (int i = 0; i < 3; ++i) if (!(g_float_names[i] = PyUnicode_InternFromString(kSampleFloats[i]))) return nullptr;
    if (!(g_cuda_stream = PyUnicode_InternFromString("cuda_stream"))) return nullptr;
    return PyModule_Create(&kModule);
}
