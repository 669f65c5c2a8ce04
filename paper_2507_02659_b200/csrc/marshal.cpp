// Argument marshalling of the binding's calls as a Python extension: tensors become raw device
// pointers, the current stream becomes the `stream` argument, and the C ABI is called.
//
// Why it is native: a verification step passes 31 tensors, and looking at each from Python (type,
// device, layout, pointer) costs 0.5 us, 15 to 20 us a call for 12 us of work on the device.
//
// Every function takes the arguments of its wrapper in binding.py and returns the status of the
// call, or None where an argument is not what the call takes as it stands (another type, device or
// layout, a number out of range): nothing has been called then, and the wrapper goes on to its
// own checks, which raise. No tensor or address is kept from one call to the next.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>

#include "omnidraft.h"

namespace {

// The arguments of one call, read in order.
struct Args {
    PyObject *const *a;
    Py_ssize_t n, at = 0;
    c10::Device dev;
    bool ok = true;

    Args(PyObject *const *args, Py_ssize_t nargs, Py_ssize_t want) : a(args), n(nargs), dev(c10::DeviceType::CPU)
    {
        ok = nargs == want;
    }
    PyObject *next() { return ok && at < n ? a[at++] : (ok = false, nullptr); }

    long long integer()
    {
        PyObject *o = next();
        if (!o || !PyLong_CheckExact(o)) { ok = false; return 0; }
        int over = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &over);
        if (over) ok = false;
        return v;
    }
    int32_t i32()
    {
        const long long v = integer();
        if (v < INT32_MIN || v > INT32_MAX) ok = false;
        return (int32_t)v;
    }
    // a step number: any Python integer modulo 2^64
    uint64_t u64()
    {
        PyObject *o = next();
        if (!o || !PyLong_CheckExact(o)) { ok = false; return 0; }
        return (uint64_t)PyLong_AsUnsignedLongLongMask(o);
    }
    float f32()
    {
        PyObject *o = next();
        if (!o || !PyFloat_CheckExact(o)) { ok = false; return 0.f; }
        return (float)PyFloat_AS_DOUBLE(o);
    }
    // the context: its handle (an integer) and the index of its device
    od_ctx *ctx()
    {
        PyObject *o = next();
        if (!o || !PyLong_CheckExact(o)) { ok = false; return nullptr; }
        void *p = PyLong_AsVoidPtr(o);
        if (!p) { PyErr_Clear(); ok = false; }
        dev = c10::Device(c10::DeviceType::CUDA, (c10::DeviceIndex)integer());
        return (od_ctx *)p;
    }
    const at::Tensor *tensor(bool may_be_none = false)
    {
        PyObject *o = next();
        if (!o || (may_be_none && o == Py_None)) return nullptr;
        if (!THPVariable_Check(o)) { ok = false; return nullptr; }
        const at::Tensor &t = THPVariable_Unpack(o);
        if (t.device() != dev) { ok = false; return nullptr; }
        return &t;
    }
    template <typename T>
    T *ptr(c10::ScalarType type, bool may_be_none = false)
    {
        const at::Tensor *t = tensor(may_be_none);
        if (!t) return nullptr;
        if (t->scalar_type() != type || !t->is_contiguous()) { ok = false; return nullptr; }
        return (T *)t->data_ptr();
    }
    float *pf(bool may_be_none = false) { return ptr<float>(c10::kFloat, may_be_none); }
    int32_t *pi(bool may_be_none = false) { return ptr<int32_t>(c10::kInt, may_be_none); }
    uint32_t *pu() { return ptr<uint32_t>(c10::kInt); }
    uint8_t *pb() { return ptr<uint8_t>(c10::kByte); }
    double *pd() { return ptr<double>(c10::kDouble); }
    uint64_t *pl() { return ptr<uint64_t>(c10::kLong); }

    // drafter's distributions [B, K, v_q]
    float *q_rows(int64_t B, int64_t K, int64_t v_q)
    {
        const at::Tensor *t = tensor();
        if (!t || t->scalar_type() != c10::kFloat || !t->is_contiguous() || t->dim() != 3 || t->size(0) != B ||
            t->size(1) != K || t->size(2) != v_q) {
            ok = false;
            return nullptr;
        }
        return (float *)t->data_ptr();
    }
    void *stream() const { return (void *)c10::cuda::getCurrentCUDAStream(dev.index()).stream(); }
};

// logits [B, K + 1, row] with dense rows
struct Logits {
    const void *p = nullptr;
    int32_t dtype = 0;
    int64_t row_stride = 0, seq_stride = 0;
    Logits(Args &x, int64_t B, int64_t K, int64_t row)
    {
        const at::Tensor *t = x.tensor();
        if (!t || t->dim() != 3 || t->size(0) != B || t->size(1) != K + 1 || t->size(2) != row || t->stride(2) != 1 ||
            (t->scalar_type() != c10::kFloat && t->scalar_type() != c10::kBFloat16)) {
            x.ok = false;
            return;
        }
        p = t->data_ptr();
        dtype = t->scalar_type() == c10::kFloat ? OD_F32 : OD_BF16;
        row_stride = t->stride(1); seq_stride = t->stride(0);
    }
};

// calls fn with the tuple's elements (a braced tuple evaluates its elements in order) and the current stream
template <typename F, typename T>
PyObject *call(const Args &x, F fn, const T &args)
{
    if (!x.ok || x.at != x.n) Py_RETURN_NONE;
    void *stream = x.stream();
    int32_t status;
    Py_BEGIN_ALLOW_THREADS
    status = std::apply([&](auto... v) { return fn(v..., stream); }, args);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

PyObject *map_proposals(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 14);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32();
    std::tuple args{c, B, K, x.pi(), x.pi(), x.pf(), x.pi(), x.pf(), x.pi(), x.pi(), x.pi(), x.pb(), x.pu()};
    return call(x, od_map_proposals, args);
}

PyObject *verify(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 20);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), v_p = x.i32();
    const Logits l(x, B, K, v_p);
    std::tuple args{c, B, K, l.p, l.dtype, l.row_stride, l.seq_stride, x.pi(), x.pf(), x.pi(), x.pi(), x.pf(), x.pl(),
                    x.u64(), x.pf(), x.pf(), x.pf(), x.pf(), x.pi(), x.pi(), x.pu()};
    return call(x, od_verify, args);
}

PyObject *sample_residual(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 24);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), v_q = x.i32(), v_p = x.i32();
    const Logits l(x, B, K, v_p);
    std::tuple args{c, B, K, l.p, l.dtype, l.row_stride, l.seq_stride, x.pf(), x.pf(), x.q_rows(B, K, v_q), x.pi(), x.pi(),
                    x.pf(), x.pi(), x.pi(), x.pi(), x.pb(), x.pi(), x.pf(), x.pl(), x.u64(), x.pi(), x.pf(), x.pu()};
    return call(x, od_sample_residual, args);
}

PyObject *step(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 31);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), v_q = x.i32(), v_p = x.i32();
    int32_t *ids = x.pi(), *len = x.pi();
    float *q_sel = x.pf(), *q = x.q_rows(B, K, v_q);
    const Logits l(x, B, K, v_p);
    std::tuple args{c, B, K, ids, len, q_sel, q, l.p, l.dtype, l.row_stride, l.seq_stride, x.pf(), x.pl(), x.u64(),
                    x.pi(), x.pf(), x.pi(), x.pi(), x.pi(), x.pb(), x.pu(),
                    x.pf(), x.pf(), x.pf(), x.pf(), x.pi(), x.pi(), x.pu(), x.pi(), x.pf(), x.pu()};
    return call(x, od_step, args);
}

PyObject *exit_rule(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 10);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32();
    std::tuple args{c, B, K, x.pf(), x.pi(true), x.f32(), x.pi(), x.pf(), x.pu()};
    return call(x, od_exit_rule, args);
}

PyObject *distill_loss(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 20);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), v_p = x.i32();
    float *q = x.pf();
    int32_t *ids = x.pi(), *tgt = x.pi(), *s0 = x.pi(), *sl = x.pi(), *m = x.pi();
    const Logits l(x, B, K, v_p);
    std::tuple args{c, B, K, q, ids, tgt, s0, sl, m, l.p, l.dtype, l.row_stride, l.seq_stride, x.pf(), x.pf(), x.pf(),
                    x.pf(), x.f32(), x.i32(), x.pf(), x.pf(true)};
    return call(x, od_distill_loss, args);
}

PyObject *verify_shard_stats(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 11);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), lo = x.i32(), len = x.i32();
    const Logits l(x, B, K, len);
    std::tuple args{c, B, K, lo, len, l.p, l.dtype, l.row_stride, l.seq_stride, x.pi(), x.pi(), x.pf(), x.pf()};
    return call(x, od_verify_shard_stats, args);
}

PyObject *verify_shard_finish(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 20);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), shards = x.i32();
    std::tuple args{c, B, K, shards, x.pf(), x.pi(), x.pf(), x.pi(), x.pi(), x.pf(), x.pl(), x.u64(),
                    x.pf(), x.pf(), x.pf(), x.pf(), x.pi(), x.pi(), x.pu()};
    return call(x, od_verify_shard_finish, args);
}

PyObject *sample_shard_mass(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 21);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), v_q = x.i32(), lo = x.i32(), len = x.i32();
    const Logits l(x, B, K, len);
    std::tuple args{c, B, K, lo, len, l.p, l.dtype, l.row_stride, l.seq_stride, x.pf(), x.pf(), x.q_rows(B, K, v_q), x.pi(),
                    x.pi(), x.pf(), x.pi(), x.pi(), x.pi(), x.pb(), x.pi(), x.pf(), x.pd()};
    return call(x, od_sample_shard_mass, args);
}

PyObject *sample_shard_pick(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 27);
    od_ctx *c = x.ctx();
    const int32_t B = x.i32(), K = x.i32(), shards = x.i32(), index = x.i32(), lo = x.i32(), len = x.i32();
    double *mass = x.pd();
    const Logits l(x, B, K, len);
    std::tuple args{c, B, K, shards, index, lo, len, mass, l.p, l.dtype, l.row_stride, l.seq_stride, x.pf(), x.pf(), x.pf(),
                    x.pi(), x.pi(), x.pf(), x.pi(), x.pi(), x.pi(), x.pb(), x.pi(), x.pf(), x.pl(), x.u64(), x.pi(), x.pf(),
                    x.pu()};
    return call(x, od_sample_shard_pick, args);
}

PyObject *cache_insert(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 6);
    od_ctx *c = x.ctx();
    const int32_t N = x.i32();
    std::tuple args{c, N, x.pi(), x.pi(), x.pi()};
    return call(x, od_cache_insert, args);
}

PyObject *cache_trim(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args x(a, n, 2);
    std::tuple args{x.ctx()};
    return call(x, od_cache_trim, args);
}

// a tensor without memory of its own (one that is being traced or mapped over) throws when asked
// for its address: not an argument to take as it stands
template <PyObject *(*F)(PyObject *, PyObject *const *, Py_ssize_t)>
PyObject *guarded(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    try {
        return F(self, a, n);
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

#define METHOD(f) {#f, (PyCFunction)(void (*)(void))guarded<f>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(map_proposals), METHOD(verify), METHOD(sample_residual), METHOD(step), METHOD(exit_rule),
                         METHOD(distill_loss), METHOD(verify_shard_stats), METHOD(verify_shard_finish),
                         METHOD(sample_shard_mass), METHOD(sample_shard_pick), METHOD(cache_insert), METHOD(cache_trim),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void)
{
    PyObject *m = PyModule_Create(&module);
    // it reads tensors by the layout of the torch that it was compiled against: the binding compares
    if (m && PyModule_AddStringConstant(m, "built_for", OD_BUILT_FOR) != 0) Py_CLEAR(m);
    return m;
}
