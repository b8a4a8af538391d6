// Native argument marshalling for binding.py (module paper_2607_24953_b200._host).
//
// The kernels of a small layer run a few microseconds each, less than a ctypes call spends on turning tensors into
// pointers: 20 us for a quantizer call and 18 us for a product, of which the launch itself is about 3.  These functions
// take the Python arguments as they are, allocate the outputs, and call the C entry points through the addresses that
// binding.py hands over once (so that a library chosen by FP4Q_LIB stays the one that is used): 8 and 7 us.  No state is
// kept from one call to the next.  Whatever a call allocates or clears is allocated and cleared in the order of the stream that
// its kernels run in (OnStream).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <algorithm>
#include <optional>
#include <vector>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>

#include "fp4q.h"

namespace {

struct Entry {
    decltype(&fp4q_quantize2d) quantize2d;
    decltype(&fp4q_quantize2d_multi) quantize2d_multi;
    decltype(&fp4q_quantize2d_multi_f32) quantize2d_multi_f32;
    decltype(&fp4q_mxfp8_quantize1d) mxfp8_quantize1d, mxfp8_quantize1d_t;
    decltype(&fp4q_quantize1d) quantize1d;
    decltype(&fp4q_quantize1d_t) quantize1d_t;
    decltype(&fp4q_gemm_fwd) gemm_fwd, gemm_dgrad;
    decltype(&fp4q_gemm_wgrad) gemm_wgrad;
    decltype(&fp4q_gemm_fwd_b16) gemm_fwd_b16, gemm_dgrad_b16;
    decltype(&fp4q_gemm_wgrad_b16) gemm_wgrad_b16;
    decltype(&fp4q_gemm_fwd_quantized) gemm_fwd_quantized, gemm_dgrad_quantized;
    decltype(&fp4q_gemm_fwd_act1d) gemm_fwd_act1d;
    decltype(&fp4q_gemm_wgrad_act1d) gemm_wgrad_act1d;
    decltype(&fp4q_mxfp8_qk) mxfp8_qk;
    decltype(&fp4q_mxfp8_gemm) mxfp8_gemm;
    decltype(&fp4q_workspace_bytes) workspace_bytes;
} lib;

PyObject *g_qtensor = nullptr, *g_fail = nullptr;   // binding.QTensor; binding._check
PyObject *s_rows, *s_cols, *s_q_rm, *s_q_t, *s_scale, *s_granularity;

// A Python exception is set: unwinds to the entry point, which returns NULL.
struct PyError {};

struct Ref {   // owned reference
    PyObject *p;
    explicit Ref(PyObject *o) : p(o) { if (!p) throw PyError(); }
    ~Ref() { Py_DECREF(p); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

// The interpreter lock is given up around allocations and library calls, as torch.empty and ctypes do (the layer's passes run
// without it altogether).
struct Unlock {
    PyThreadState *state = PyGILState_Check() ? PyEval_SaveThread() : nullptr;
    ~Unlock() { if (state) PyEval_RestoreThread(state); }
};
template <typename F, typename... A>
fp4q_status unlocked(F fn, A... args)
{
    Unlock u;
    return fn(args...);
}

[[noreturn]] void value_error(const char *text) { PyErr_SetString(PyExc_ValueError, text); throw PyError(); }

int64_t as_i64(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyError();
    return v;
}
uint64_t as_bits(PyObject *o)   // seeds and modes: anything with __index__ (NumPy's and torch's whole numbers), modulo 2^64, as ctypes does
{
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) throw PyError();
    return v;
}
int as_int(PyObject *o) { return (int)(uint32_t)as_bits(o); }
uint32_t id_at(PyObject *ids, Py_ssize_t j)   // int(ids[j]), of a list, an array or a tensor
{
    Ref index(PyLong_FromSsize_t(j)), item(PyObject_GetItem(ids, index.p)), number(PyNumber_Long(item.p));
    return (uint32_t)as_bits(number.p);
}
bool as_bool(PyObject *o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw PyError();
    return v != 0;
}
const at::Tensor &as_tensor(PyObject *o)
{
    if (!THPVariable_Check(o)) { PyErr_Format(PyExc_TypeError, "expected a tensor, got %s", Py_TYPE(o)->tp_name); throw PyError(); }
    return THPVariable_Unpack(o);
}
// The stream a call runs in: the current stream of the current device (None) or another one, given by its handle.  In the
// second case that stream is made current while the call lasts: outputs, their zero fill and the default workspace belong to its
// order and, freed, to its pool.  What the call returns is also recorded for the caller's stream, where it is likely to be
// read and dropped.
struct OnStream {
    void *handle;
    std::optional<c10::cuda::CUDAStream> caller;
    std::optional<c10::cuda::CUDAStreamGuard> guard;
    OnStream() : handle(c10::cuda::getCurrentCUDAStream().stream()) {}
    OnStream(PyObject *o, const at::Tensor *like)
    {
        if (o == Py_None) {
            handle = c10::cuda::getCurrentCUDAStream().stream();
            return;
        }
        handle = PyLong_AsVoidPtr(o);
        if (PyErr_Occurred()) throw PyError();
        if (!like || !like->is_cuda()) return;
        const auto device = like->device().index();
        const auto raw = handle == (void *)cudaStreamLegacy ? nullptr : static_cast<cudaStream_t>(handle);
        const auto now = c10::cuda::getCurrentCUDAStream(device);
        if (raw == now.stream()) return;
        caller.emplace(now);
        guard.emplace(c10::cuda::getStreamFromExternal(raw, device));
    }
    const at::Tensor &returned(const at::Tensor &t) const
    {
        if (caller && t.defined()) t.record_stream(caller->unwrap());
        return t;
    }
};
uint8_t *bytes_of(const at::Tensor &t) { return static_cast<uint8_t *>(t.data_ptr()); }

// Error status: binding._check raises.
void check(fp4q_status st, const char *where)
{
    if (st == FP4Q_OK) return;
    Ref r(PyObject_CallFunction(g_fail, "is", (int)st, where));
}

int64_t pad16(int64_t n) { return (n + 15) / 16 * 16; }
int64_t ceil_to(int64_t a, int64_t b) { return (a + b - 1) / b; }

at::Tensor empty2(int64_t r, int64_t c, at::ScalarType dt, const at::Tensor &like)
{
    Unlock u;
    return at::empty({r, c}, at::TensorOptions().dtype(dt).device(like.device()));
}

// x: BF16 [rows, cols], unit stride along the columns.
const at::Tensor &as_matrix(PyObject *o, const char *name, const char *what)
{
    const at::Tensor &x = as_tensor(o);
    if (!x.is_cuda()) { PyErr_Format(PyExc_ValueError, "%s must live on a CUDA device (there is no CPU path)", name); throw PyError(); }
    if (x.scalar_type() != at::kBFloat16 || x.dim() != 2 || (x.numel() && x.stride(1) != 1)) value_error(what);
    return x;
}
// The caller's workspace, or one that lasts for this call: its memory is reused in the order of the call's stream.
at::Tensor workspace(PyObject *o, const at::Tensor &like)
{
    if (o != Py_None) return as_tensor(o);
    Unlock u;
    return at::zeros({(int64_t)lib.workspace_bytes()}, at::TensorOptions().dtype(at::kByte).device(like.device()));
}
const char kXText[] = "x must be a 2-D BF16 tensor with contiguous rows";
int64_t pitch(const at::Tensor &x) { return x.size(0) ? x.stride(0) : x.size(1); }

// Leading dimensions the C interface asks for, as in binding.alloc_qtensor.
struct QBuffers { at::Tensor q_rm, q_t, scale; };
QBuffers alloc_q(const OnStream &on, int64_t rows, int64_t cols, const at::Tensor &like, bool want_t, int64_t g)
{
    QBuffers b;
    b.q_rm = empty2(rows, std::max<int64_t>(pad16(ceil_to(cols, 32) * 16), 16), at::kByte, like);
    if (want_t) b.q_t = empty2(cols, std::max<int64_t>(pad16(ceil_to(rows, 32) * 16), 16), at::kByte, like);
    b.scale = empty2(ceil_to(rows, g), std::max<int64_t>(ceil_to(cols, g), 1), at::kByte, like);
    for (const at::Tensor *t : {&b.q_rm, &b.q_t, &b.scale}) on.returned(*t);
    return b;
}
fp4q_tensor c_tensor(int64_t rows, int64_t cols, const at::Tensor &q_rm, const at::Tensor &q_t, const at::Tensor &scale)
{
    fp4q_tensor t;
    t.rows = rows; t.cols = cols;
    t.q_rm = bytes_of(q_rm); t.ld_rm = q_rm.stride(0);
    t.q_t = q_t.defined() ? bytes_of(q_t) : nullptr; t.ld_t = q_t.defined() ? q_t.stride(0) : 0;
    t.scale = bytes_of(scale); t.ld_s = scale.stride(0);
    return t;
}
PyObject *new_qtensor(int64_t rows, int64_t cols, const QBuffers &b, int64_t g)
{
    Ref r(PyLong_FromLongLong(rows)), c(PyLong_FromLongLong(cols)), rm(THPVariable_Wrap(b.q_rm));
    Ref t(b.q_t.defined() ? THPVariable_Wrap(b.q_t) : Py_NewRef(Py_None)), s(THPVariable_Wrap(b.scale)), gr(PyLong_FromLongLong(g));
    PyObject *args[6] = {r.p, c.p, rm.p, t.p, s.p, gr.p};
    PyObject *q = PyObject_Vectorcall(g_qtensor, args, 6, nullptr);
    if (!q) throw PyError();
    return q;
}
// The C view of a QTensor; granularity: the scale granularity the callee expects (0 = any).
fp4q_tensor from_qtensor(PyObject *q, long granularity)
{
    if (granularity) {
        Ref g(PyObject_GetAttr(q, s_granularity));
        const long have = PyLong_AsLong(g.p);
        if (have == -1 && PyErr_Occurred()) throw PyError();
        if (have != granularity) {
            PyErr_Format(PyExc_ValueError, "this call takes tensors quantized in %ld x %ld blocks (scale matrix of that granularity); got %ld",
                         granularity, granularity, have);
            throw PyError();
        }
    }
    Ref r(PyObject_GetAttr(q, s_rows)), c(PyObject_GetAttr(q, s_cols)), rm(PyObject_GetAttr(q, s_q_rm)), t(PyObject_GetAttr(q, s_q_t)),
        s(PyObject_GetAttr(q, s_scale));
    return c_tensor(as_i64(r.p), as_i64(c.p), as_tensor(rm.p), t.p == Py_None ? at::Tensor() : as_tensor(t.p), as_tensor(s.p));
}
at::Tensor qtensor_payload(PyObject *q)
{
    Ref rm(PyObject_GetAttr(q, s_q_rm));
    return as_tensor(rm.p);
}

// An output matrix: rows padded to whole 16 bytes, the padding cut off the returned view.
at::Tensor out_buffer(const OnStream &on, int64_t rows, int64_t cols, int dt, const at::Tensor &like)
{
    const int64_t per16 = dt == FP4Q_OUT_BF16 ? 8 : 4, ld = std::max(ceil_to(cols, per16) * per16, per16);
    at::Tensor t = empty2(rows, ld, dt == FP4Q_OUT_BF16 ? at::kBFloat16 : at::kFloat, like);
    on.returned(t);
    return ld == cols ? t : t.slice(1, 0, cols);
}
// The type as the library takes it: an output that was allocated here is padded, a caller's is written up to its last column.  (Callers of this
// module name types 0 and 1 only; the library refuses anything else.)
fp4q_out out_type(int dt, bool ours) { return (fp4q_out)(dt & FP4Q_OUT_PADDED ? 0xFF : ours ? dt | FP4Q_OUT_PADDED : dt); }
int64_t out_pitch(const at::Tensor &out, int64_t cols) { return out.numel() ? out.stride(0) : cols; }

struct Groups {
    fp4q_groups g;
    const fp4q_groups *ptr = nullptr;
    Groups(PyObject *row_offsets, int alignment)
    {
        if (row_offsets == Py_None) return;
        const at::Tensor &t = as_tensor(row_offsets);
        if (!t.is_cuda()) value_error("row_offsets must live on a CUDA device (there is no CPU path)");
        if (t.scalar_type() != at::kLong || !t.is_contiguous()) value_error("row_offsets must be a contiguous int64 device tensor");
        g.n_groups = (int32_t)(t.numel() - 1);
        g.row_alignment = alignment;
        g.row_offsets = static_cast<const int64_t *>(t.data_ptr());
        ptr = &g;
    }
};

typedef PyObject *const *Args;

void want(Py_ssize_t got, Py_ssize_t n)
{
    if (got != n) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", n, got); throw PyError(); }
}

// x, out | None, mode, seed, tensor_id, flags, want_t, stream
PyObject *quantize2d(Args a, Py_ssize_t n)
{
    want(n, 8);
    const at::Tensor &x = as_matrix(a[0], "x", kXText);
    const int64_t rows = x.size(0), cols = x.size(1);
    const uint32_t flags = (uint32_t)as_bits(a[5]);
    const int64_t g = (flags & FP4Q_BLOCK_16) ? 16 : 32;
    const OnStream on(a[7], &x);
    fp4q_tensor t;
    QBuffers b;
    if (a[1] == Py_None) {
        b = alloc_q(on, rows, cols, x, as_bool(a[6]), g);
        t = c_tensor(rows, cols, b.q_rm, b.q_t, b.scale);
    } else {
        t = from_qtensor(a[1], 0);
    }
    check(unlocked(lib.quantize2d, x.data_ptr(), rows, cols, pitch(x), &t, (fp4q_round)as_int(a[2]), as_bits(a[3]), (uint32_t)as_bits(a[4]), flags,
                         on.handle), "fp4q_quantize2d");
    return a[1] == Py_None ? new_qtensor(rows, cols, b, g) : Py_NewRef(a[1]);
}

// xs, outs | None, mode, seed, tensor_ids | None, flags, want_t, stream
PyObject *quantize2d_multi(Args a, Py_ssize_t n)
{
    want(n, 8);
    // Copies of the lists: the loop below lets other threads and the caller's own attributes run, which may change them.
    if (PyObject_Size(a[0]) < 0) throw PyError();
    Ref xs(PySequence_Tuple(a[0]));
    const Py_ssize_t k = PyTuple_GET_SIZE(xs.p);
    const bool own = a[1] == Py_None;
    Ref outs(own ? PyList_New(0) : PySequence_Tuple(a[1]));
    const uint32_t flags = (uint32_t)as_bits(a[5]);
    const bool want_t = as_bool(a[6]);
    if (!own && PyTuple_GET_SIZE(outs.p) < k) {
        PyErr_SetString(PyExc_IndexError, "list index out of range");
        throw PyError();
    }
    const OnStream on(a[7], k > 0 ? &as_tensor(PyTuple_GET_ITEM(xs.p, 0)) : nullptr);
    std::vector<fp4q_tensor> ts((size_t)k);
    std::vector<fp4q_quantize_job> jobs((size_t)(k > 0 ? k : 1));
    for (Py_ssize_t j = 0; j < k; j++) {
        char name[32];
        snprintf(name, sizeof name, "xs[%zd]", j);
        const at::Tensor &x = as_matrix(PyTuple_GET_ITEM(xs.p, j), name, "every input must be a 2-D BF16 tensor with contiguous rows");
        if (own) {
            const QBuffers b = alloc_q(on, x.size(0), x.size(1), x, want_t, 32);
            Ref q(new_qtensor(x.size(0), x.size(1), b, 32));
            if (PyList_Append(outs.p, q.p) < 0) throw PyError();
            ts[j] = c_tensor(x.size(0), x.size(1), b.q_rm, b.q_t, b.scale);
        } else {
            ts[j] = from_qtensor(PyTuple_GET_ITEM(outs.p, j), 32);
        }
        jobs[j].x_bf16 = x.data_ptr();
        jobs[j].rows = x.size(0); jobs[j].cols = x.size(1); jobs[j].ld_x = pitch(x);
        jobs[j].out = &ts[j];
        jobs[j].tensor_id = a[4] == Py_None ? (uint32_t)j : id_at(a[4], j);
        jobs[j].flags = flags;
    }
    for (Py_ssize_t j = k; !own && j < PyTuple_GET_SIZE(outs.p); j++) from_qtensor(PyTuple_GET_ITEM(outs.p, j), 32);   // refused as a whole
    check(unlocked(lib.quantize2d_multi, jobs.data(), (int32_t)k, (fp4q_round)as_int(a[2]), as_bits(a[3]), on.handle), "fp4q_quantize2d_multi");
    return own ? Py_NewRef(outs.p) : Py_NewRef(a[1]);
}

PyObject *pair(const OnStream &on, const at::Tensor &q, const at::Tensor &s)
{
    Ref x(THPVariable_Wrap(on.returned(q))), y(THPVariable_Wrap(on.returned(s)));
    return PyTuple_Pack(2, x.p, y.p);
}

// x, stream; transposed: the encoding of x^T
template <bool T>
PyObject *mxfp8_quantize1d(Args a, Py_ssize_t n)
{
    want(n, 2);
    const at::Tensor &x = as_matrix(a[0], "x", kXText);
    const int64_t rows = x.size(0), cols = x.size(1), along = T ? rows : cols, across = T ? cols : rows;
    const OnStream on(a[1], &x);
    const at::Tensor q = empty2(across, std::max<int64_t>(ceil_to(along, 32) * 32, 32), at::kByte, x);
    const at::Tensor s = empty2(across, std::max<int64_t>(ceil_to(along, 32), 1), at::kByte, x);
    check(unlocked(T ? lib.mxfp8_quantize1d_t : lib.mxfp8_quantize1d, x.data_ptr(), rows, cols, pitch(x), bytes_of(q), q.stride(0), bytes_of(s),
                                                              s.stride(0), on.handle),
          T ? "fp4q_mxfp8_quantize1d_t" : "fp4q_mxfp8_quantize1d");
    return pair(on, q, s);
}

// x, mode, seed, tensor_id, stream
PyObject *quantize1d(Args a, Py_ssize_t n)
{
    want(n, 5);
    const at::Tensor &x = as_matrix(a[0], "x", kXText);
    const int64_t rows = x.size(0), cols = x.size(1);
    const OnStream on(a[4], &x);
    const at::Tensor q = empty2(rows, std::max<int64_t>(pad16(ceil_to(cols, 32) * 16), 16), at::kByte, x);
    const at::Tensor s = empty2(rows, std::max<int64_t>(ceil_to(cols, 32), 1), at::kByte, x);
    check(unlocked(lib.quantize1d, x.data_ptr(), rows, cols, pitch(x), bytes_of(q), q.stride(0), bytes_of(s), s.stride(0), (fp4q_round)as_int(a[1]),
                         as_bits(a[2]), (uint32_t)as_bits(a[3]), on.handle), "fp4q_quantize1d");
    return pair(on, q, s);
}

// x, stream
PyObject *quantize1d_t(Args a, Py_ssize_t n)
{
    want(n, 2);
    const at::Tensor &x = as_matrix(a[0], "x", kXText);
    const int64_t rows = x.size(0), cols = x.size(1);
    const OnStream on(a[1], &x);
    const at::Tensor q = empty2(cols, std::max<int64_t>(pad16(ceil_to(rows, 32) * 16), 16), at::kByte, x);
    const at::Tensor s = empty2(cols, std::max<int64_t>(ceil_to(rows, 32), 1), at::kByte, x);
    check(unlocked(lib.quantize1d_t, x.data_ptr(), rows, cols, pitch(x), bytes_of(q), q.stride(0), bytes_of(s), s.stride(0), on.handle),
          "fp4q_quantize1d_t");
    return pair(on, q, s);
}

// which (0 fwd, 1 dgrad, 2 wgrad), a, b, out_rows, out_cols, out | None, dt, accumulate, row_offsets | None, row_alignment, ws | None, stream
PyObject *gemm(Args a, Py_ssize_t n)
{
    want(n, 12);
    static const char *const names[3] = {"fp4q_gemm_fwd", "fp4q_gemm_dgrad", "fp4q_gemm_wgrad"};
    const int which = as_int(a[0]), dt = as_int(a[6]), accumulate = as_int(a[7]);
    const int64_t rows = as_i64(a[3]), cols = as_i64(a[4]);
    const at::Tensor like = qtensor_payload(a[1]);
    const OnStream on(a[11], &like);
    const at::Tensor out = a[5] == Py_None ? out_buffer(on, rows, cols, dt, like) : as_tensor(a[5]);
    if (a[5] == Py_None && accumulate) out.zero_();
    const fp4q_tensor ta = from_qtensor(a[1], 32), tb = from_qtensor(a[2], 32);
    const Groups g(a[8], as_int(a[9]));
    const at::Tensor ws = workspace(a[10], like);
    const int64_t ld = out_pitch(out, cols);
    const fp4q_status s =
        which == 2 ? unlocked(lib.gemm_wgrad, &ta, &tb, out.data_ptr(), ld, out_type(dt, a[5] == Py_None), accumulate, g.ptr, ws.data_ptr(), (size_t)ws.numel(), on.handle)
                   : unlocked(which == 1 ? lib.gemm_dgrad : lib.gemm_fwd, &ta, &tb, out.data_ptr(), ld, out_type(dt, a[5] == Py_None), g.ptr, ws.data_ptr(),
                                                                  (size_t)ws.numel(), on.handle);
    check(s, names[which]);
    return a[5] == Py_None ? THPVariable_Wrap(out) : Py_NewRef(a[5]);
}

// which, a, b, out_rows, out_cols, out | None, dt, accumulate, ws | None, stream
PyObject *gemm_b16(Args a, Py_ssize_t n)
{
    want(n, 10);
    static const char *const names[3] = {"fp4q_gemm_fwd_b16", "fp4q_gemm_dgrad_b16", "fp4q_gemm_wgrad_b16"};
    const int which = as_int(a[0]), dt = as_int(a[6]), accumulate = as_int(a[7]);
    const int64_t rows = as_i64(a[3]), cols = as_i64(a[4]);
    const at::Tensor like = qtensor_payload(a[1]);
    const OnStream on(a[9], &like);
    const at::Tensor out = a[5] == Py_None ? out_buffer(on, rows, cols, dt, like) : as_tensor(a[5]);
    if (a[5] == Py_None && accumulate) out.zero_();
    const fp4q_tensor ta = from_qtensor(a[1], 16), tb = from_qtensor(a[2], 16);
    const at::Tensor ws = workspace(a[8], like);
    const int64_t ld = out_pitch(out, cols);
    const fp4q_status s =
        which == 2 ? unlocked(lib.gemm_wgrad_b16, &ta, &tb, out.data_ptr(), ld, out_type(dt, a[5] == Py_None), accumulate, ws.data_ptr(), (size_t)ws.numel(), on.handle)
                   : unlocked(which == 1 ? lib.gemm_dgrad_b16 : lib.gemm_fwd_b16, &ta, &tb, out.data_ptr(), ld, out_type(dt, a[5] == Py_None), ws.data_ptr(),
                                                                          (size_t)ws.numel(), on.handle);
    check(s, names[which]);
    return a[5] == Py_None ? THPVariable_Wrap(out) : Py_NewRef(a[5]);
}

// which (0 fwd, 1 dgrad), a, b, out_rows, out_cols, out | None, mode, seed, tensor_id, want_t, row_offsets | None, ws | None, stream
PyObject *gemm_quantized(Args a, Py_ssize_t n)
{
    want(n, 13);
    const int which = as_int(a[0]);
    const Groups g(a[10], 256);
    const int64_t rows = as_i64(a[3]), cols = as_i64(a[4]);
    const at::Tensor like = qtensor_payload(a[1]);
    const OnStream on(a[12], &like);
    QBuffers b;
    fp4q_tensor tc;
    if (a[5] == Py_None) {
        b = alloc_q(on, rows, cols, like, as_bool(a[9]), 32);
        tc = c_tensor(rows, cols, b.q_rm, b.q_t, b.scale);
    }
    const fp4q_tensor ta = from_qtensor(a[1], 32), tb = from_qtensor(a[2], 32);
    if (a[5] != Py_None) tc = from_qtensor(a[5], 32);
    const at::Tensor ws = workspace(a[11], like);
    check(unlocked(which ? lib.gemm_dgrad_quantized : lib.gemm_fwd_quantized, &ta, &tb, &tc, (fp4q_round)as_int(a[6]), as_bits(a[7]),
                                                                      (uint32_t)as_bits(a[8]), g.ptr, ws.data_ptr(), (size_t)ws.numel(),
                                                                      on.handle),
          which ? "fp4q_gemm_dgrad_quantized" : "fp4q_gemm_fwd_quantized");
    return a[5] == Py_None ? new_qtensor(rows, cols, b, 32) : Py_NewRef(a[5]);
}

// xq, xs, T, W, out | None, dt, ws | None, stream
PyObject *gemm_fwd_act1d(Args a, Py_ssize_t n)
{
    want(n, 8);
    const at::Tensor &xq = as_tensor(a[0]), &xs = as_tensor(a[1]);
    const int64_t T = as_i64(a[2]);
    const int dt = as_int(a[5]);
    Ref wr(PyObject_GetAttr(a[3], s_rows));
    const OnStream on(a[7], &xq);
    const at::Tensor out = a[4] == Py_None ? out_buffer(on, T, as_i64(wr.p), dt, xq) : as_tensor(a[4]);
    const fp4q_tensor w = from_qtensor(a[3], 32);
    const at::Tensor ws = workspace(a[6], xq);
    check(unlocked(lib.gemm_fwd_act1d, bytes_of(xq), xq.stride(0), bytes_of(xs), xs.stride(0), T, &w, out.data_ptr(), out.stride(0), out_type(dt, a[4] == Py_None),
                             ws.data_ptr(), (size_t)ws.numel(), on.handle), "fp4q_gemm_fwd_act1d");
    return a[4] == Py_None ? THPVariable_Wrap(out) : Py_NewRef(a[4]);
}

// dY, xtq, xts, K, out | None, dt, accumulate, ws | None, stream
PyObject *gemm_wgrad_act1d(Args a, Py_ssize_t n)
{
    want(n, 9);
    const at::Tensor &xq = as_tensor(a[1]), &xs = as_tensor(a[2]);
    const int64_t K = as_i64(a[3]);
    const int dt = as_int(a[5]), accumulate = as_bool(a[6]) ? 1 : 0;
    Ref dc(PyObject_GetAttr(a[0], s_cols));
    const OnStream on(a[8], &xq);
    const at::Tensor out = a[4] == Py_None ? out_buffer(on, as_i64(dc.p), K, dt, xq) : as_tensor(a[4]);
    if (a[4] == Py_None && accumulate) out.zero_();
    const fp4q_tensor d = from_qtensor(a[0], 32);
    const at::Tensor ws = workspace(a[7], xq);
    check(unlocked(lib.gemm_wgrad_act1d, &d, bytes_of(xq), xq.stride(0), bytes_of(xs), xs.stride(0), K, out.data_ptr(), out.stride(0), out_type(dt, a[4] == Py_None),
                               accumulate, ws.data_ptr(), (size_t)ws.numel(), on.handle), "fp4q_gemm_wgrad_act1d");
    return a[4] == Py_None ? THPVariable_Wrap(out) : Py_NewRef(a[4]);
}

// aq, as, bq, bs, M, N, K, dt, ws | None, stream
PyObject *mxfp8_gemm(Args a, Py_ssize_t n)
{
    want(n, 10);
    const at::Tensor &aq = as_tensor(a[0]), &as = as_tensor(a[1]), &bq = as_tensor(a[2]), &bs = as_tensor(a[3]);
    const int64_t M = as_i64(a[4]), N = as_i64(a[5]), K = as_i64(a[6]);
    const int dt = as_int(a[7]);
    const OnStream on(a[9], &aq);
    const at::Tensor out = out_buffer(on, M, N, dt, aq);
    const at::Tensor ws = workspace(a[8], aq);
    const int64_t per16 = dt == FP4Q_OUT_BF16 ? 8 : 4, ld = std::max(ceil_to(N, per16) * per16, per16);
    check(unlocked(lib.mxfp8_gemm, bytes_of(aq), aq.stride(0), bytes_of(as), as.stride(0), M, bytes_of(bq), bq.stride(0), bytes_of(bs), bs.stride(0), N,
                         K, out.data_ptr(), ld, out_type(dt, true), ws.data_ptr(), (size_t)ws.numel(), on.handle), "fp4q_mxfp8_gemm");
    return THPVariable_Wrap(out);
}

// xq, xs, wq_q | None, wq_s | None, wk_q | None, wk_s | None, T, K, N, dt, ws | None, stream
PyObject *mxfp8_qk(Args a, Py_ssize_t n)
{
    want(n, 12);
    const at::Tensor &xq = as_tensor(a[0]), &xs = as_tensor(a[1]);
    at::Tensor w[4];
    uint8_t *p[4];
    for (int i = 0; i < 4; i++) {
        if (a[2 + i] != Py_None) w[i] = as_tensor(a[2 + i]);
        p[i] = w[i].defined() ? bytes_of(w[i]) : nullptr;
    }
    const int64_t T = as_i64(a[6]), K = as_i64(a[7]), N = as_i64(a[8]);
    const int dt = as_int(a[9]);
    const int64_t per16 = dt == FP4Q_OUT_BF16 ? 8 : 4, ld = std::max(ceil_to(N, per16) * per16, per16);
    const OnStream on(a[11], &xq);
    at::Tensor out[2];
    for (int i = 0; i < 2; i++) if (w[2 * i].defined()) out[i] = out_buffer(on, T, N, dt, xq);
    const at::Tensor &wref = w[0].defined() ? w[0] : w[2], &sref = w[0].defined() ? w[1] : w[3];
    if (!wref.defined() || !sref.defined()) { PyErr_SetString(PyExc_AttributeError, "'NoneType' object has no attribute 'stride'"); throw PyError(); }
    const at::Tensor ws = workspace(a[10], xq);
    check(unlocked(lib.mxfp8_qk, bytes_of(xq), xq.stride(0), bytes_of(xs), xs.stride(0), T, K, p[0], p[1], p[2], p[3], wref.stride(0), sref.stride(0), N,
                       out[0].defined() ? out[0].data_ptr() : nullptr, out[1].defined() ? out[1].data_ptr() : nullptr, ld, out_type(dt, true),
                       ws.data_ptr(), (size_t)ws.numel(), on.handle), "fp4q_mxfp8_qk");
    Ref q(out[0].defined() ? THPVariable_Wrap(out[0]) : Py_NewRef(Py_None)), k(out[1].defined() ? THPVariable_Wrap(out[1]) : Py_NewRef(Py_None));
    return PyTuple_Pack(2, q.p, k.p);
}

// ---- the straight-through layer of autograd.py as one native autograd node
//
// The layer's kernels run 20 to 90 us forward and backward at the sizes where layers are small; through a Python autograd
// function and the calls above the interpreter took as long, forward in the caller's thread and backward, with the lock, in the
// engine's (128 x 256 x 256, forward and backward, 122-139 -> 87 us, of which the engine's own change of threads is 36).
void check_unlocked(fp4q_status st, const char *where)
{
    if (st == FP4Q_OK) return;
    const PyGILState_STATE gil = PyGILState_Ensure();
    python_error e;
    try {
        check(st, where);
    } catch (const PyError &) {
        e.persist();
    }
    PyGILState_Release(gil);
    throw e;
}
struct LinearCall {
    at::Tensor ws;
    uint64_t seed;
    uint32_t tensor_id;
};
// Places in one allocation, for the arrays of quantized tensors (pitches as in alloc_q): one by one, twelve allocations a step
// would be a tenth of its host time.
struct Block {
    int64_t bytes = 0;
    int64_t add(int64_t n)
    {
        const int64_t at = bytes;
        bytes += ceil_to(n, 256) * 256;
        return at;
    }
};
struct Placed {   // a quantized [rows, cols]: where its arrays lie in their blocks
    fp4q_tensor t = {};
    int64_t rm = 0, tr = 0, sc = 0, n_rm, n_t, n_s;
    Placed(int64_t rows, int64_t cols)
    {
        t.rows = rows; t.cols = cols;
        t.ld_rm = std::max<int64_t>(pad16(ceil_to(cols, 32) * 16), 16);
        t.ld_t = std::max<int64_t>(pad16(ceil_to(rows, 32) * 16), 16);
        t.ld_s = std::max<int64_t>(ceil_to(cols, 32), 1);
        n_rm = rows * t.ld_rm; n_t = cols * t.ld_t; n_s = ceil_to(rows, 32) * t.ld_s;
    }
    void place_rm(Block &b) { rm = b.add(n_rm); }
    void place_t(Block &b) { tr = b.add(n_t); sc = b.add(n_s); }
    void bind_rm(uint8_t *base) { t.q_rm = n_rm ? base + rm : nullptr; }
    void bind_t(uint8_t *base) { t.q_t = n_t ? base + tr : nullptr; t.scale = n_s ? base + sc : nullptr; }
};
at::Tensor block(const Block &b, const at::Tensor &like) { return at::empty({b.bytes}, at::TensorOptions().dtype(at::kByte).device(like.device())); }
at::Tensor as_bf16(const at::Tensor &t)
{
    const at::Tensor c = t.scalar_type() == at::kBFloat16 ? t : t.to(at::kBFloat16);
    return c.is_contiguous() ? c : c.contiguous();
}
// What the quantizer reads of an operand: an FP32 one as it is, where its rows start on 16 bytes (a BF16 copy of a 2048 x 2048 weight
// took 6 us, and 7 of host time); else BF16.  A single row is contiguous whatever its pitch, and the quantizer checks the pitch.  The
// copy is also what resolves a tensor whose memory does not hold its values: the negative bit, and zeros without memory.
at::Tensor as_source(const at::Tensor &t)
{
    const bool as_it_is = t.scalar_type() == at::kFloat && t.is_contiguous() && t.size(1) % 4 == 0 && pitch(t) % 4 == 0 &&
                          reinterpret_cast<uintptr_t>(t.data_ptr()) % 16 == 0 && !t.is_neg() && !t._is_zerotensor();
    return as_it_is ? t : as_bf16(t);
}
at::Tensor as_type(const at::Tensor &t, int64_t dtype) { return t.scalar_type() == (at::ScalarType)dtype ? t : t.to((at::ScalarType)dtype); }

struct LinearNode : torch::autograd::Function<LinearNode> {
    static at::Tensor forward(torch::autograd::AutogradContext *ctx, const at::Tensor &x, const at::Tensor &weight, const LinearCall &call)
    {
        const OnStream on;
        const at::Tensor xb = as_source(x), wb = as_source(weight);
        const int64_t T = xb.size(0), K = xb.size(1), N = wb.size(0);
        Placed qx(T, K), qw(N, wb.size(1));
        Block keep, drop;   // backward reads the transposed codes and the scales
        qx.place_t(keep); qw.place_t(keep); qx.place_rm(drop); qw.place_rm(drop);
        const at::Tensor kept = block(keep, xb), dropped = block(drop, xb);
        for (Placed *q : {&qx, &qw}) { q->bind_t(bytes_of(kept)); q->bind_rm(bytes_of(dropped)); }
        fp4q_quantize_job jobs[2] = {};
        jobs[0].x_bf16 = xb.data_ptr(); jobs[0].rows = T; jobs[0].cols = K; jobs[0].ld_x = pitch(xb); jobs[0].out = &qx.t;
        jobs[1].x_bf16 = wb.data_ptr(); jobs[1].rows = N; jobs[1].cols = wb.size(1); jobs[1].ld_x = pitch(wb); jobs[1].out = &qw.t;
        const uint8_t is_f32[2] = {xb.scalar_type() == at::kFloat, wb.scalar_type() == at::kFloat};
        check_unlocked(lib.quantize2d_multi_f32(jobs, is_f32, 2, FP4Q_ROUND_NEAREST, 0, on.handle), "fp4q_quantize2d");
        const at::Tensor y = out_buffer(on, T, N, FP4Q_OUT_BF16, xb);
        check_unlocked(lib.gemm_fwd(&qx.t, &qw.t, y.data_ptr(), out_pitch(y, N), out_type(FP4Q_OUT_BF16, true), nullptr, call.ws.data_ptr(), (size_t)call.ws.numel(), on.handle),
                       "fp4q_gemm_fwd");
        ctx->saved_data["kept"] = kept;
        ctx->saved_data["ws"] = call.ws;
        ctx->saved_data["numbers"] = std::vector<int64_t>{K, (int64_t)call.seed, (int64_t)call.tensor_id, (int64_t)x.scalar_type(), (int64_t)weight.scalar_type()};
        return y.is_contiguous() ? y : y.contiguous();
    }
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext *ctx, torch::autograd::variable_list grads)
    {
        TORCH_CHECK(!ctx->saved_data.empty(),
                    "fp4_linear: the quantized operands are freed when backward has run; run the layer again instead of going through its graph a second time");
        const OnStream on;
        const at::Tensor kept = ctx->saved_data["kept"].toTensor(), ws = ctx->saved_data["ws"].toTensor(), dy = as_bf16(grads[0]);
        const auto numbers = ctx->saved_data["numbers"].toIntVector();
        const int64_t T = dy.size(0), N = dy.size(1), K = numbers[0];
        Placed qx(T, K), qw(N, K), q(T, N);
        Block keep, own;
        qx.place_t(keep); qw.place_t(keep); q.place_rm(own); q.place_t(own);
        const at::Tensor codes = block(own, dy);
        qx.bind_t(bytes_of(kept)); qw.bind_t(bytes_of(kept));
        q.bind_rm(bytes_of(codes)); q.bind_t(bytes_of(codes));
        check_unlocked(lib.quantize2d(dy.data_ptr(), T, N, pitch(dy), &q.t, FP4Q_ROUND_STOCHASTIC, (uint64_t)numbers[1], (uint32_t)numbers[2], 0, on.handle),
                       "fp4q_quantize2d");
        at::Tensor dx, dw;
        if (ctx->needs_input_grad(0)) {
            dx = out_buffer(on, T, K, FP4Q_OUT_BF16, dy);
            check_unlocked(lib.gemm_dgrad(&q.t, &qw.t, dx.data_ptr(), out_pitch(dx, K), out_type(FP4Q_OUT_BF16, true), nullptr, ws.data_ptr(), (size_t)ws.numel(), on.handle),
                           "fp4q_gemm_dgrad");
            dx = as_type(dx, numbers[3]);
        }
        if (ctx->needs_input_grad(1)) {
            dw = out_buffer(on, N, K, FP4Q_OUT_F32, dy);
            check_unlocked(lib.gemm_wgrad(&q.t, &qx.t, dw.data_ptr(), out_pitch(dw, K), out_type(FP4Q_OUT_F32, true), 0, nullptr, ws.data_ptr(), (size_t)ws.numel(), on.handle),
                           "fp4q_gemm_wgrad");
            dw = as_type(dw, numbers[4]);
        }
        ctx->saved_data.clear();
        return {dx, dw, at::Tensor()};
    }
};

// x [T, K], weight [N, K], seed, tensor_id, ws
PyObject *linear(Args a, Py_ssize_t n)
{
    want(n, 5);
    const at::Tensor x = as_tensor(a[0]), weight = as_tensor(a[1]);
    const LinearCall call{as_tensor(a[4]), as_bits(a[2]), (uint32_t)as_bits(a[3])};
    at::Tensor y;
    {
        Unlock u;
        y = LinearNode::apply(x, weight, call);
    }
    return THPVariable_Wrap(y);
}

template <typename F>
void set_entry(PyObject *addresses, const char *name, F &slot)
{
    PyObject *v = PyDict_GetItemString(addresses, name);
    if (!v) { PyErr_Format(PyExc_KeyError, "%s", name); throw PyError(); }
    slot = reinterpret_cast<F>(PyLong_AsVoidPtr(v));
    if (PyErr_Occurred()) throw PyError();
}

// {name: address of the C entry point}, QTensor, _check
PyObject *init(Args a, Py_ssize_t n)
{
    want(n, 3);
    set_entry(a[0], "fp4q_quantize2d", lib.quantize2d);
    set_entry(a[0], "fp4q_quantize2d_multi", lib.quantize2d_multi);
    set_entry(a[0], "fp4q_quantize2d_multi_f32", lib.quantize2d_multi_f32);
    set_entry(a[0], "fp4q_mxfp8_quantize1d", lib.mxfp8_quantize1d);
    set_entry(a[0], "fp4q_mxfp8_quantize1d_t", lib.mxfp8_quantize1d_t);
    set_entry(a[0], "fp4q_quantize1d", lib.quantize1d);
    set_entry(a[0], "fp4q_quantize1d_t", lib.quantize1d_t);
    set_entry(a[0], "fp4q_gemm_fwd", lib.gemm_fwd);
    set_entry(a[0], "fp4q_gemm_dgrad", lib.gemm_dgrad);
    set_entry(a[0], "fp4q_gemm_wgrad", lib.gemm_wgrad);
    set_entry(a[0], "fp4q_gemm_fwd_b16", lib.gemm_fwd_b16);
    set_entry(a[0], "fp4q_gemm_dgrad_b16", lib.gemm_dgrad_b16);
    set_entry(a[0], "fp4q_gemm_wgrad_b16", lib.gemm_wgrad_b16);
    set_entry(a[0], "fp4q_gemm_fwd_quantized", lib.gemm_fwd_quantized);
    set_entry(a[0], "fp4q_gemm_dgrad_quantized", lib.gemm_dgrad_quantized);
    set_entry(a[0], "fp4q_gemm_fwd_act1d", lib.gemm_fwd_act1d);
    set_entry(a[0], "fp4q_gemm_wgrad_act1d", lib.gemm_wgrad_act1d);
    set_entry(a[0], "fp4q_mxfp8_qk", lib.mxfp8_qk);
    set_entry(a[0], "fp4q_mxfp8_gemm", lib.mxfp8_gemm);
    set_entry(a[0], "fp4q_workspace_bytes", lib.workspace_bytes);
    Py_XSETREF(g_qtensor, Py_NewRef(a[1]));
    Py_XSETREF(g_fail, Py_NewRef(a[2]));
    return Py_NewRef(Py_None);
}

// What a call throws becomes a Python exception: its own, or torch's (out of memory, a failed CUDA call).
template <PyObject *(*F)(Args, Py_ssize_t)>
PyObject *entry(PyObject *, Args a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    try {
        return F(a, n);
    } catch (const PyError &) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

#define METHOD(name, fn) {name, (PyCFunction)(void (*)(void))entry<fn>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD("init", init),
                         METHOD("quantize2d", quantize2d),
                         METHOD("quantize2d_multi", quantize2d_multi),
                         METHOD("mxfp8_quantize1d", mxfp8_quantize1d<false>),
                         METHOD("mxfp8_quantize1d_t", mxfp8_quantize1d<true>),
                         METHOD("quantize1d", quantize1d),
                         METHOD("quantize1d_t", quantize1d_t),
                         METHOD("gemm", gemm),
                         METHOD("gemm_b16", gemm_b16),
                         METHOD("gemm_quantized", gemm_quantized),
                         METHOD("gemm_fwd_act1d", gemm_fwd_act1d),
                         METHOD("gemm_wgrad_act1d", gemm_wgrad_act1d),
                         METHOD("mxfp8_gemm", mxfp8_gemm),
                         METHOD("mxfp8_qk", mxfp8_qk),
                         METHOD("linear", linear),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", "argument marshalling of binding.py", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host(void)
{
    s_rows = PyUnicode_InternFromString("rows");
    s_cols = PyUnicode_InternFromString("cols");
    s_q_rm = PyUnicode_InternFromString("q_rm");
    s_q_t = PyUnicode_InternFromString("q_t");
    s_scale = PyUnicode_InternFromString("scale");
    s_granularity = PyUnicode_InternFromString("scale_granularity");
    return PyModule_Create(&module);
}
