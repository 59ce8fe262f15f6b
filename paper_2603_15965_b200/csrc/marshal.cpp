// Argument marshalling of the hot entry points, as a CPython extension over the C ABI in include/molora.h.
//
// What a small call costs is mostly this: reading the shapes, strides, types and pointers of up to 33 tensors, three output
// allocations and the current stream.  Done attribute by attribute from Python it took 35 - 60 us per step, several times
// what the kernels take (one decode layer of seven projections: 58 us per call against 11 us of GPU time); here it is a few
// microseconds.  Every call does all of it again: nothing is kept between calls.
//
// Checks, messages and results are those documented in binding.py, which keeps the public signatures and calls the
// functions below with positional arguments.  A refused call raises MoloraError through `raise_status`.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <string>
#include <vector>

#include "molora.h"

namespace {

PyObject* g_raise_status = nullptr;      // binding._check(function name, status)
PyObject *s_x, *s_y, *s_A, *s_B, *s_scale, *s_row_scale, *s_cuda_stream, *s_data_ptr;

struct PyRaised {};                      // a Python exception is set
[[noreturn]] void raise(PyObject* type, const std::string& text)
{
    PyErr_SetString(type, text.c_str());
    throw PyRaised{};
}
struct Ref {                             // owned reference
    PyObject* p;
    explicit Ref(PyObject* q) : p(q)
    {
        if (p == nullptr) throw PyRaised{};
    }
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
};

// Other Python threads run while a call allocates and enqueues: either may block (an allocation that goes to the driver, a launch
// into a full queue).
struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(state); }
};

void check(const char* fn, molora_status_t status)
{
    if (status == MOLORA_OK) return;
    Ref r(PyObject_CallFunction(g_raise_status, "si", fn, (int)status));
    raise(PyExc_RuntimeError, std::string(fn) + " was refused");      // (not reached: the callable raises)
}

const at::Tensor& tensor(PyObject* o, const char* name)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string(name) + ": expected a tensor");
    return THPVariable_Unpack(o);
}
// device pointer of a tensor, or of anything else that has data_ptr(); None is a null pointer, which the library judges
void* ptr(PyObject* o)
{
    if (o == Py_None) return nullptr;
    if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
    Ref v(PyObject_CallMethodNoArgs(o, s_data_ptr));
    void* p = PyLong_AsVoidPtr(v.p);
    if (p == nullptr && PyErr_Occurred()) throw PyRaised{};
    return p;
}
PyObject* wrap(const at::Tensor& t)
{
    PyObject* o = THPVariable_Wrap(t);
    if (o == nullptr) throw PyRaised{};
    return o;
}
int64_t integer(PyObject* o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyRaised{};
    return v;
}
// the stream of a call: the one given, or the current one
struct Stream {
    void* p;
    bool given;
    explicit Stream(PyObject* o) : p(nullptr), given(o != Py_None)
    {
        if (!given) {
            p = c10::cuda::getCurrentCUDAStream().stream();
            return;
        }
        Ref v(PyObject_HasAttr(o, s_cuda_stream) ? PyObject_GetAttr(o, s_cuda_stream) : PyNumber_Long(o));
        p = PyLong_AsVoidPtr(v.p);
        if (p == nullptr && PyErr_Occurred()) throw PyRaised{};
    }
};
const at::Tensor& i32_dev(PyObject* o, const char* name)
{
    const at::Tensor& t = tensor(o, name);
    if (!t.is_cuda() || t.scalar_type() != at::kInt || !t.is_contiguous())
        raise(PyExc_ValueError, std::string(name) + ": expected a contiguous int32 CUDA tensor");
    return t;
}
// What a call allocates belongs to the stream that it runs on: memory that the current stream's allocator hands out may still be in
// use there, and is handed out again there as soon as the call has returned.
template <class F>
at::Tensor allocate(const Stream& stream, F f)
{
    if (!stream.given) return f();
    c10::cuda::OptionalCUDAStreamGuard on;
    // (odd values are not addresses but the runtime's names of its default streams)
    if (stream.p != c10::cuda::getCurrentCUDAStream().stream() && ((uintptr_t)stream.p & 1u) == 0)
        on.reset_stream(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(stream.p), c10::cuda::current_device()));
    return f();
}
// an output: the caller's tensor, or n words allocated on first use
struct Out {
    at::Tensor t;
    at::Device dev;
    int64_t n;
    Out(PyObject* o, const char* name, int64_t n_, const at::Device& dev_) : dev(dev_), n(n_)
    {
        if (o != Py_None) t = i32_dev(o, name);
    }
    int32_t* get(const Stream& stream)
    {
        if (!t.defined()) t = allocate(stream, [&] { return at::empty({n}, at::TensorOptions().dtype(at::kInt).device(dev)); });
        return static_cast<int32_t*>(t.data_ptr());
    }
};
molora_dtype_t dtype_code(const at::Tensor& t)
{
    if (t.scalar_type() == at::kFloat) return MOLORA_F32;
    if (t.scalar_type() == at::kBFloat16) return MOLORA_BF16;
    raise(PyExc_TypeError, std::string("unsupported element type ") + c10::toString(t.scalar_type()) + ": fp32 or bf16 only");
}
struct Matrix {
    int64_t rows, cols, pitch;
};
Matrix matrix(const at::Tensor& t, const char* name)
{
    if (!t.is_cuda() || t.dim() != 2 || (t.size(1) > 1 && t.stride(1) != 1))
        raise(PyExc_ValueError, std::string(name) + ": expected a 2-D row-major CUDA tensor");
    const int64_t rows = t.size(0), cols = t.size(1);
    return {rows, cols, rows > 1 ? t.stride(0) : std::max<int64_t>(t.stride(0), cols)};
}
// the caller's workspace, or one of `need` bytes allocated by make()
struct Workspace {
    at::Tensor t;
    void* p = nullptr;
    size_t n = 0, need = 0;
    Workspace(PyObject* o, size_t need_)
    {
        if (o != Py_None) t = tensor(o, "ws");
        else need = need_;
    }
    void make(const at::Device& dev, bool zero, const Stream& stream)
    {
        const auto opt = at::TensorOptions().dtype(at::kByte).device(dev);
        if (need > 0) t = allocate(stream, [&] { return zero ? at::zeros({(int64_t)need}, opt) : at::empty({(int64_t)need}, opt); });
        if (!t.defined()) return;
        p = t.data_ptr();
        n = (size_t)t.numel() * t.element_size();
    }
};
// ---- descriptors of a batched apply: from ProjDesc objects, or the array that pack_proj_descs returned
struct Projs {
    std::vector<molora_proj_desc_t> own;
    Py_buffer view{};
    const molora_proj_desc_t* d = nullptr;
    int32_t P = 0;
    int64_t N = 0, C = 0;
    molora_dtype_t dt = MOLORA_F32;

    Projs(PyObject* projs, PyObject* packed)
    {
        if (packed != Py_None) {
            Ref arr(PySequence_GetItem(packed, 0)), n(PySequence_GetItem(packed, 1)), c(PySequence_GetItem(packed, 2)),
                t(PySequence_GetItem(packed, 3));
            N = integer(n.p), C = integer(c.p), dt = (molora_dtype_t)integer(t.p);
            if (PyObject_GetBuffer(arr.p, &view, PyBUF_SIMPLE) != 0) throw PyRaised{};
            d = static_cast<const molora_proj_desc_t*>(view.buf);
            P = (int32_t)(view.len / (Py_ssize_t)sizeof(molora_proj_desc_t));
            return;
        }
        Ref seq(PySequence_Fast(projs, "projs: expected a sequence of ProjDesc"));
        P = (int32_t)PySequence_Fast_GET_SIZE(seq.p);
        own.resize((size_t)P);
        for (int32_t i = 0; i < P; ++i) fill(PySequence_Fast_GET_ITEM(seq.p, i), own[(size_t)i], i == 0);
        d = own.data();
    }
    ~Projs()
    {
        if (view.obj != nullptr) PyBuffer_Release(&view);
    }
    Projs(const Projs&) = delete;
    Projs& operator=(const Projs&) = delete;

    size_t apply_bytes() const
    {
        size_t need = 0;
        for (int32_t i = 0; i < P; ++i) need += molora_apply_workspace_bytes(N, (int32_t)C, d[i].d_in, d[i].d_out, d[i].rank);
        return need;
    }

private:
    void fill(PyObject* o, molora_proj_desc_t& out, bool first)
    {
        Ref ox(PyObject_GetAttr(o, s_x)), oy(PyObject_GetAttr(o, s_y)), oA(PyObject_GetAttr(o, s_A)), oB(PyObject_GetAttr(o, s_B)),
            osc(PyObject_GetAttr(o, s_scale));
        const at::Tensor &x = tensor(ox.p, "x"), &y = tensor(oy.p, "y"), &A = tensor(oA.p, "A"), &B = tensor(oB.p, "B");
        const Matrix mx = matrix(x, "x"), my = matrix(y, "y");
        const auto st = x.scalar_type();
        if (my.rows != mx.rows || y.scalar_type() != st || A.scalar_type() != st || B.scalar_type() != st)
            raise(PyExc_ValueError, "x, y, A, B must share the token count and the element type");
        if (A.dim() < 3) raise(PyExc_IndexError, "A: expected 3 dimensions");
        const int64_t c = A.size(0), rank = A.size(2);
        if (!A.is_contiguous() || !B.is_contiguous() || A.size(1) != mx.cols || B.dim() != 3 || B.size(0) != c || B.size(1) != rank ||
            B.size(2) != my.cols)
            raise(PyExc_ValueError, "A / B shapes do not match x / y");
        const molora_dtype_t code = dtype_code(x);
        if (first) {
            N = mx.rows;
            C = c;
            dt = code;
        } else if (N != mx.rows || C != c || dt != code) {
            raise(PyExc_ValueError, "all projections of a batched apply share N, C and the element type");
        }
        out.row_scale = nullptr;
        PyObject* rs = PyObject_GetAttr(o, s_row_scale);
        if (rs == nullptr) {
            if (!PyErr_ExceptionMatches(PyExc_AttributeError)) throw PyRaised{};
            PyErr_Clear();
        } else {
            Ref hold(rs);
            if (rs != Py_None) {
                const at::Tensor& t = tensor(rs, "row_scale");
                if (t.scalar_type() != at::kFloat || t.numel() != mx.rows || !t.is_contiguous())
                    raise(PyExc_ValueError, "row_scale must be a dense fp32 tensor with one factor per token");
                out.row_scale = static_cast<const float*>(t.data_ptr());
            }
        }
        const double scale = PyFloat_AsDouble(osc.p);
        if (scale == -1.0 && PyErr_Occurred()) throw PyRaised{};
        out.x = x.data_ptr();
        out.ldx = mx.pitch;
        out.y = y.data_ptr();
        out.ldy = my.pitch;
        out.A = A.data_ptr();
        out.B = B.data_ptr();
        out.d_in = (int32_t)mx.cols;
        out.d_out = (int32_t)my.cols;
        out.rank = (int32_t)rank;
        out.scale = (float)scale;
    }
};

int32_t* i32(const at::Tensor& t) { return static_cast<int32_t*>(t.data_ptr()); }
float* f32(PyObject* o) { return static_cast<float*>(ptr(o)); }
// one call of the library: f() allocates what it needs, enqueues and returns the status
template <class F>
void call(const char* fn, F f)
{
    molora_status_t status;
    {
        const NoGil others;
        status = f();
    }
    check(fn, status);
}
uint32_t* status_word(PyObject* o) { return static_cast<uint32_t*>(ptr(o)); }

// ---- (ids, breaks, r_out, dev_status, stream.p)
PyObject* route_vocab(PyObject* const* a)
{
    const at::Tensor &ids = i32_dev(a[0], "ids"), &breaks = i32_dev(a[1], "breaks");
    const int64_t N = ids.numel();
    Out r(a[2], "r_out", N, ids.device());
    uint32_t* status = status_word(a[3]);
    const Stream stream(a[4]);
    call("molora_route_vocab", [&] { return molora_route_vocab(i32(ids), N, i32(breaks), (int32_t)breaks.numel() - 1, r.get(stream), status, stream.p); });
    return wrap(r.t);
}

// ---- (ids, adapter, breaks, n_adapters, r_out, dev_status, stream.p)
PyObject* route_composite(PyObject* const* a)
{
    const at::Tensor &ids = i32_dev(a[0], "ids"), &adapter = i32_dev(a[1], "adapter"), &breaks = i32_dev(a[2], "breaks");
    const int64_t N = ids.numel();
    if (adapter.numel() != N) raise(PyExc_ValueError, "adapter must hold one index per token");
    Ref n(PyNumber_Long(a[3]));
    const int32_t n_adapters = (int32_t)integer(n.p);
    Out r(a[4], "r_out", N, ids.device());
    uint32_t* status = status_word(a[5]);
    const Stream stream(a[6]);
    call("molora_route_composite", [&] {
        return molora_route_composite(i32(ids), i32(adapter), N, i32(breaks), (int32_t)breaks.numel() - 1, n_adapters, r.get(stream), status, stream.p);
    });
    return wrap(r.t);
}

// ---- (x, G, bias, r_out, logits_out, ws, dev_status, stream, prepared)
PyObject* route_gate(PyObject* const* a)
{
    const at::Tensor &x = tensor(a[0], "x"), &G = tensor(a[1], "G");
    const Matrix m = matrix(x, "x");
    if (G.scalar_type() != at::kFloat || !G.is_cuda() || !G.is_contiguous() || G.dim() != 2 || G.size(0) != m.cols)
        raise(PyExc_ValueError, "G: expected a contiguous fp32 CUDA tensor of shape [d, C]");
    const int32_t C = (int32_t)G.size(1), d = (int32_t)m.cols;
    if (a[2] != Py_None) {
        const at::Tensor& b = tensor(a[2], "bias");
        if (b.scalar_type() != at::kFloat || b.numel() != C || !b.is_contiguous())
            raise(PyExc_ValueError, "bias: expected contiguous fp32 [C]");
    }
    if (a[4] != Py_None) {
        const at::Tensor& z = tensor(a[4], "logits_out");
        if (z.scalar_type() != at::kFloat || z.dim() != 2 || z.size(0) != m.rows || z.size(1) != C || !z.is_contiguous())
            raise(PyExc_ValueError, "logits_out: expected contiguous fp32 [N, C]");
    }
    const molora_dtype_t dt = dtype_code(x);
    Out r(a[3], "r_out", m.rows, x.device());
    const float *g = f32(a[1]), *bias = f32(a[2]);
    float* logits = f32(a[4]);
    uint32_t* status = status_word(a[6]);
    const Stream stream(a[7]);
    if (a[8] != Py_None) {
        const at::Tensor& prepared = tensor(a[8], "prepared");
        call("molora_route_gate_prepared", [&] {
            return molora_route_gate_prepared(x.data_ptr(), dt, m.rows, d, m.pitch, g, bias, C, r.get(stream), logits, prepared.data_ptr(),
                                              (size_t)prepared.numel(), status, stream.p);
        });
        return wrap(r.t);
    }
    Workspace ws(a[5], molora_route_gate_workspace_bytes(dt, d, C));
    call("molora_route_gate", [&] {
        ws.make(x.device(), false, stream);        // (the weight images are written before they are read: the scratch need not be cleared)
        return molora_route_gate(x.data_ptr(), dt, m.rows, d, m.pitch, g, bias, C, r.get(stream), logits, ws.p, ws.n, status, stream.p);
    });
    return wrap(r.t);
}

// ---- (x, W1, b1, W2, b2, r_out, logits_out, ws, dev_status, stream, prepared)
PyObject* route_mlp(PyObject* const* a)
{
    const at::Tensor &x = tensor(a[0], "x"), &W1 = tensor(a[1], "W1"), &W2 = tensor(a[3], "W2");
    const Matrix m = matrix(x, "x");
    if (W1.scalar_type() != at::kFloat || W2.scalar_type() != at::kFloat || !W1.is_contiguous() || !W2.is_contiguous())
        raise(PyExc_ValueError, "W1 [d, H] and W2 [H, C] must be dense fp32 tensors");
    if (W2.dim() != 2) raise(PyExc_ValueError, "W2 must be [H, C]");
    const int32_t H = (int32_t)W2.size(0), C = (int32_t)W2.size(1), d = (int32_t)m.cols;
    if (W1.dim() != 2 || W1.size(0) != d || W1.size(1) != H) raise(PyExc_ValueError, "W1 must be [d, H]");
    const molora_dtype_t dt = dtype_code(x);
    Out r(a[5], "r_out", m.rows, x.device());
    const float *w1 = f32(a[1]), *b1 = f32(a[2]), *w2 = f32(a[3]), *b2 = f32(a[4]);
    float* logits = f32(a[6]);
    uint32_t* status = status_word(a[8]);
    const Stream stream(a[9]);
    if (a[10] != Py_None) {
        const at::Tensor& prepared = tensor(a[10], "prepared");
        call("molora_route_mlp_prepared", [&] {
            return molora_route_mlp_prepared(x.data_ptr(), dt, m.rows, d, m.pitch, w1, b1, H, w2, b2, C, r.get(stream), logits, prepared.data_ptr(),
                                             (size_t)prepared.numel(), status, stream.p);
        });
        return wrap(r.t);
    }
    Workspace ws(a[7], molora_route_mlp_workspace_bytes(dt, d, H, C));
    call("molora_route_mlp", [&] {
        ws.make(x.device(), false, stream);
        return molora_route_mlp(x.data_ptr(), dt, m.rows, d, m.pitch, w1, b1, H, w2, b2, C, r.get(stream), logits, ws.p, ws.n, status, stream.p);
    });
    return wrap(r.t);
}

PyObject* tuple_of(std::initializer_list<at::Tensor> ts)
{
    PyObject* t = PyTuple_New((Py_ssize_t)ts.size());
    if (t == nullptr) throw PyRaised{};
    Py_ssize_t i = 0;
    for (const at::Tensor& x : ts) {
        PyObject* o = THPVariable_Wrap(x);
        if (o == nullptr) {
            Py_DECREF(t);
            throw PyRaised{};
        }
        PyTuple_SET_ITEM(t, i++, o);
    }
    return t;
}

// ---- (r, C, counts, offsets, perm, ws, dev_status, stream.p)
PyObject* group(PyObject* const* a)
{
    const at::Tensor& r = i32_dev(a[0], "r");
    const int64_t N = r.numel(), C = integer(a[1]);
    const at::Device dev = r.device();
    Out counts(a[2], "counts", C, dev), offsets(a[3], "offsets", C + 1, dev), perm(a[4], "perm", std::max<int64_t>(N, 1), dev);
    Workspace ws(a[5], molora_group_workspace_bytes(N, (int32_t)C));
    uint32_t* status = status_word(a[6]);
    const Stream stream(a[7]);
    call("molora_group", [&] {
        int32_t *c = counts.get(stream), *o = offsets.get(stream), *p = perm.get(stream);
        ws.make(dev, true, stream);
        return molora_group(i32(r), N, (int32_t)C, c, o, p, ws.p, ws.n, status, stream.p);
    });
    return tuple_of({counts.t, offsets.t, perm.t});
}

// ---- (projs, offsets, perm, ws, dev_status, stream, packed)
PyObject* apply_batched(PyObject* const* a)
{
    const Projs pr(a[0], a[6]);
    const auto *offsets = static_cast<const int32_t*>(ptr(a[1])), *perm = static_cast<const int32_t*>(ptr(a[2]));
    Workspace ws(a[3], a[3] == Py_None ? pr.apply_bytes() : 0);
    const at::Device dev = ws.need > 0 ? tensor(a[1], "offsets").device() : at::Device(at::kCUDA);
    uint32_t* status = status_word(a[4]);
    const Stream stream(a[5]);
    call("molora_apply_batched", [&] {
        ws.make(dev, true, stream);
        return molora_apply_batched(pr.d, pr.P, pr.dt, pr.N, (int32_t)pr.C, offsets, perm, ws.p, ws.n, status, stream.p);
    });
    Py_RETURN_NONE;
}

// ---- (r, projs, C, counts, offsets, perm, ws, dev_status, stream, packed)
PyObject* group_apply_batched(PyObject* const* a)
{
    const at::Tensor& r = i32_dev(a[0], "r");
    const Projs pr(a[1], a[9]);
    const int64_t C = a[2] == Py_None ? pr.C : integer(a[2]);
    if (r.numel() != pr.N || C != pr.C) raise(PyExc_ValueError, "r must hold one routing decision per token of the projections");
    const at::Device dev = r.device();
    Out counts(a[3], "counts", C, dev), offsets(a[4], "offsets", C + 1, dev), perm(a[5], "perm", std::max<int64_t>(pr.N, 1), dev);
    Workspace ws(a[6], a[6] == Py_None ? pr.apply_bytes() : 0);
    uint32_t* status = status_word(a[7]);
    const Stream stream(a[8]);
    call("molora_group_apply_batched", [&] {
        int32_t *c = counts.get(stream), *o = offsets.get(stream), *p = perm.get(stream);
        ws.make(dev, true, stream);
        return molora_group_apply_batched(i32(r), pr.N, (int32_t)C, c, o, p, pr.d, pr.P, pr.dt, ws.p, ws.n, status, stream.p);
    });
    return tuple_of({counts.t, offsets.t, perm.t});
}

// ---- (logits, k, stream)
PyObject* topk_softmax(PyObject* const* a)
{
    const at::Tensor& z = tensor(a[0], "logits");
    if (z.scalar_type() != at::kFloat || z.dim() != 2 || !z.is_contiguous()) raise(PyExc_ValueError, "logits must be a dense fp32 [N, C] tensor");
    Ref kk(PyNumber_Long(a[1]));
    const int64_t k = integer(kk.p), N = z.size(0);
    const Stream stream(a[2]);
    at::Tensor idx, w;
    call("molora_topk_softmax", [&] {
        idx = allocate(stream, [&] { return at::empty({k, N}, at::TensorOptions().dtype(at::kInt).device(z.device())); });
        w = allocate(stream, [&] { return at::empty({k, N}, at::TensorOptions().dtype(at::kFloat).device(z.device())); });
        return molora_topk_softmax(static_cast<const float*>(z.data_ptr()), N, (int32_t)z.size(1), (int32_t)k, i32(idx),
                                   static_cast<float*>(w.data_ptr()), stream.p);
    });
    return tuple_of({idx, w});
}

// ---- (projs, idx, w, C, ws, dev_status, stream.p)
PyObject* apply_topk(PyObject* const* a)
{
    const Projs pr(a[0], Py_None);
    const at::Tensor &idx0 = tensor(a[1], "idx"), &w0 = tensor(a[2], "w");
    const int64_t C = integer(a[3]);
    if (pr.C != C || idx0.scalar_type() != at::kInt || w0.scalar_type() != at::kFloat || idx0.dim() != 2 || idx0.sizes() != w0.sizes() ||
        idx0.size(1) != pr.N)
        raise(PyExc_ValueError, "idx int32 [k, N] and w fp32 [k, N] must match the projections");
    const bool zero = pr.apply_bytes() > 0;
    Workspace ws(a[4], a[4] == Py_None ? molora_apply_topk_workspace_bytes(pr.d, pr.P, pr.N, (int32_t)C) + 256 : 0);
    uint32_t* status = status_word(a[5]);
    const Stream stream(a[6]);
    at::Tensor idx, w;
    call("molora_apply_topk", [&] {
        idx = allocate(stream, [&] { return idx0.contiguous(); });
        w = allocate(stream, [&] { return w0.contiguous(); });
        ws.make(idx.device(), zero, stream);        // (only the apply part has to start cleared, and only where a kernel keeps control words in it)
        const size_t off = std::min((size_t)(-(intptr_t)ws.p) % 256, ws.n);      // (a shorter workspace is refused as too small)
        return molora_apply_topk(pr.d, pr.P, pr.dt, pr.N, (int32_t)C, (int32_t)idx.size(0), i32(idx), static_cast<const float*>(w.data_ptr()),
                                 static_cast<char*>(ws.p) + off, ws.n - off, status, stream.p);
    });
    Py_RETURN_NONE;
}

// ---- (raise_status)
PyObject* bind(PyObject* const* a)
{
    Py_INCREF(a[0]);
    Py_XDECREF(g_raise_status);
    g_raise_status = a[0];
    Py_RETURN_NONE;
}

// fixed number of positional arguments; C++ exceptions end here
template <PyObject* (*F)(PyObject* const*), int ARGS>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    if (n != ARGS) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", ARGS, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const PyRaised&) {
    } catch (...) {
        torch::translate_exception_to_python(std::current_exception());      // (out of memory is torch.OutOfMemoryError, as from torch itself)
    }
    return nullptr;
}

#define ENTRY(name, n) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<name, n>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(route_vocab, 5), ENTRY(route_composite, 7), ENTRY(route_gate, 9), ENTRY(route_mlp, 11), ENTRY(group, 8),
                         ENTRY(apply_batched, 7), ENTRY(group_apply_batched, 10), ENTRY(topk_softmax, 3), ENTRY(apply_topk, 7), ENTRY(bind, 1),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal()
{
    s_x = PyUnicode_InternFromString("x");
    s_y = PyUnicode_InternFromString("y");
    s_A = PyUnicode_InternFromString("A");
    s_B = PyUnicode_InternFromString("B");
    s_scale = PyUnicode_InternFromString("scale");
    s_row_scale = PyUnicode_InternFromString("row_scale");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return PyModule_Create(&module);
}
