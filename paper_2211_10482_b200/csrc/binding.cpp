// Python side of the C ABI: argument checks, output and workspace allocation, the current stream and the call, without a
// Python frame or a ctypes conversion in between.  The kernels of a small call run a few microseconds, so what the
// host does per call is what such a call costs: st_packed_axpby 8.4 us through ctypes, of which the launch itself is 2.2.
// The module holds no kernel and no reference to a particular library: bind() receives the addresses of the entry points.
#include <Python.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <cstdint>
#include <cstring>
#include <exception>
#include <initializer_list>
#include <map>
#include <string>
#include <tuple>
#include <utility>
#include "structtensor.h"

namespace {

struct Api {
    decltype(&st_packed_elems) packed_elems;
    decltype(&st_dense_elems) dense_elems;
    decltype(&st_workspace_bytes) workspace_bytes;
    decltype(&st_pack) pack;
    decltype(&st_unpack) unpack;
    decltype(&st_thp) thp;
    decltype(&st_packed_axpby) packed_axpby;
    decltype(&st_packed_mul) packed_mul;
    decltype(&st_sym_moment2) sym_moment2;
    decltype(&st_sym_moment3) sym_moment3;
    decltype(&st_sym_moment4) sym_moment4;
    decltype(&st_mttkrp_tri) mttkrp_tri;
    decltype(&st_mttkrp_slice) mttkrp_slice;
    decltype(&st_ttm_blockdiag) ttm_blockdiag;
    decltype(&st_ttm_packed) ttm_packed;
} api;

PyObject *error_class, *allocator;             // StError; callable or null
PyObject *dtype_f32, *dtype_u8;                // torch.float32, torch.uint8
PyObject *s_kind, *s_d, *s_inner, *s_kl, *s_ku, *s_nblocks, *s_bs, *s_dtype, *s_device, *s_view;
PyObject *last_ws;                             // dict: device index -> workspace of the most recent compute call

struct Failed {};                              // a Python error is set

[[noreturn]] void fail(PyObject *type, const char *text)
{
    PyErr_SetString(type, text);
    throw Failed();
}

void check(st_status rc, const char *where)
{
    if (rc == ST_OK) return;
    PyObject *e = PyObject_CallFunction(error_class, "is", (int)rc, where);
    if (e) {
        PyErr_SetObject(error_class, e);
        Py_DECREF(e);
    }
    throw Failed();
}

const at::Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
        throw Failed();
    }
    return THPVariable_Unpack(o);
}

void *device_ptr(const at::Tensor &t, const char *name)
{
    if (!t.is_cuda()) {
        PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor", name);
        throw Failed();
    }
    if (!t.is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
        throw Failed();
    }
    return t.data_ptr();
}

const float *f32_ptr(const at::Tensor &t, const char *name) { return (const float *)device_ptr(t, name); }

// The kernels run on one device and take every pointer as its memory.
void want_device_of(const at::Tensor &x, const at::Tensor &t, const char *name)
{
    if (t.device() != x.device()) {
        PyErr_Format(PyExc_ValueError, "%s must be on the device of the first operand", name);
        throw Failed();
    }
}

// The address that `bytes` bytes of results go to.
void *result_ptr(const at::Tensor &x, PyObject *out, size_t bytes)
{
    const at::Tensor &t = tensor(out, "out");
    void *p = device_ptr(t, "out");
    want_device_of(x, t, "out");
    if (t.nbytes() < bytes) {
        PyErr_Format(PyExc_ValueError, "out has %zu bytes, the result %zu", (size_t)t.nbytes(), bytes);
        throw Failed();
    }
    return p;
}

int64_t integer(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return v;
}
// What int() makes of it.
int64_t whole(PyObject *o)
{
    PyObject *v = PyNumber_Long(o);
    if (!v) throw Failed();
    const long long x = PyLong_AsLongLong(v);
    Py_DECREF(v);
    if (x == -1 && PyErr_Occurred()) throw Failed();
    return x;
}
unsigned flag_bits(PyObject *o)
{
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw Failed();
    return (unsigned)v;
}
float real(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Failed();
    return (float)v;
}

// The product, or -1, which no element count equals, where it leaves 64 bits.
int64_t times(std::initializer_list<int64_t> factors)
{
    int64_t n = 1;
    for (const int64_t f : factors)
        if (f < 0 || __builtin_mul_overflow(n, f, &n)) return -1;
    return n;
}

int64_t field(PyObject *layout, PyObject *name)
{
    PyObject *v = PyObject_GetAttr(layout, name);
    if (!v) throw Failed();
    const long long x = PyLong_AsLongLong(v);
    Py_DECREF(v);
    if (x == -1 && PyErr_Occurred()) throw Failed();
    return x;
}
st_layout layout_of(PyObject *o)
{
    st_layout l;
    l.kind = (int32_t)field(o, s_kind);
    l.reserved = 0;
    l.d = field(o, s_d);
    l.inner = field(o, s_inner);
    l.kl = field(o, s_kl);
    l.ku = field(o, s_ku);
    l.nblocks = field(o, s_nblocks);
    l.bs = field(o, s_bs);
    return l;
}

// Element type of st_pack / st_unpack: bit copies, so any type of the same size travels.
st_dtype copy_dtype(const at::Tensor &t)
{
    switch (t.scalar_type()) {
    case at::kFloat: case at::kInt: case at::kUInt32: return ST_F32;
    case at::kBFloat16: case at::kHalf: case at::kShort: case at::kUInt16: return ST_BF16;
    case at::kDouble: case at::kLong: return ST_F64;
    default: fail(PyExc_TypeError, "unsupported dtype");
    }
}

// A new tensor as a Python object, from torch or from the allocator of set_allocator().
PyObject *allocate(PyObject *like, const at::Tensor &t, at::IntArrayRef shape, at::ScalarType type, PyObject *py_type)
{
    if (!allocator) return THPVariable_Wrap(at::empty(shape, t.options().dtype(type).requires_grad(false)));
    int64_t n = 1;
    for (const int64_t s : shape) n *= s;
    PyObject *device = PyObject_GetAttr(like, s_device);
    PyObject *r = device ? PyObject_CallFunction(allocator, "LOO", (long long)n, py_type, device) : nullptr;
    Py_XDECREF(device);
    if (r && shape.size() != 1) {
        PyObject *dims = PyTuple_New((Py_ssize_t)shape.size());
        for (size_t i = 0; i < shape.size(); ++i) PyTuple_SET_ITEM(dims, (Py_ssize_t)i, PyLong_FromLongLong(shape[i]));
        PyObject *v = PyObject_CallMethodOneArg(r, s_view, dims);
        Py_DECREF(dims);
        Py_DECREF(r);
        r = v;
    }
    return r;
}

// Owned Python reference.
struct Ref {
    PyObject *o;
    explicit Ref(PyObject *p) : o(p) { if (!p) throw Failed(); }
    Ref(const Ref &) = delete;
    Ref(Ref &&r) noexcept : o(r.o) { r.o = nullptr; }
    ~Ref() { Py_XDECREF(o); }
    PyObject *release() { PyObject *p = o; o = nullptr; return p; }
};

// The caller's tensor or a new one of `shape`.
PyObject *output(PyObject *given, PyObject *like, const at::Tensor &t, at::IntArrayRef shape)
{
    if (given != Py_None) {
        (void)tensor(given, "out");
        Py_INCREF(given);
        return given;
    }
    return allocate(like, t, shape, at::kFloat, dtype_f32);
}

struct Workspace {
    Ref ref;                                   // held until the call has been enqueued (another thread may replace last_ws)
    void *ptr;
    size_t bytes;
};

// Workspace bytes by request; the current device decides too (its SM count).  Bounded: forgotten when it grows past
// what a program with many shapes uses.  Accessed with the GIL held.
size_t workspace_size(int op, int64_t a, int64_t b, int64_t c, int64_t e, unsigned flags)
{
    typedef std::tuple<int, int, int64_t, int64_t, int64_t, int64_t, unsigned> Key;
    static std::map<Key, size_t> known;
    const Key key(c10::cuda::current_device(), op, a, b, c, e, flags);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    if (known.size() >= 1024) known.clear();
    const size_t n = api.workspace_bytes((st_op)op, a, b, c, e, flags);
    return known[key] = n < 256 ? 256 : n;
}

// The caller's workspace or a new one of the request's size; remembered as its device's last.
Workspace workspace(PyObject *given, PyObject *like, const at::Tensor &t, int op, int64_t a, int64_t b, int64_t c, int64_t e,
                    unsigned flags)
{
    PyObject *o = given;
    if (given == Py_None) {
        const int64_t n = (int64_t)workspace_size(op, a, b, c, e, flags);
        o = allocate(like, t, {n}, at::kByte, dtype_u8);
    } else {
        Py_INCREF(given);
    }
    Ref hold(o);
    const at::Tensor &ws = tensor(o, "ws");
    void *ptr = device_ptr(ws, "ws");
    want_device_of(t, ws, "ws");
    Ref index(PyLong_FromLong(ws.get_device()));
    if (PyDict_SetItem(last_ws, index.o, o) != 0) throw Failed();
    const size_t bytes = ws.nbytes();
    return Workspace{std::move(hold), ptr, bytes};
}

void *stream() { return (void *)c10::cuda::getCurrentCUDAStream().stream(); }

// The C call with the interpreter lock released, as a launch may have to wait for room in the queue.
template <typename F>
void call(const char *where, F f)
{
    void *s = stream();
    st_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f(s);
    Py_END_ALLOW_THREADS
    check(rc, where);
}

void want_f32(const at::Tensor &t, const char *what)
{
    if (t.scalar_type() != at::kFloat) {
        PyErr_Format(PyExc_TypeError, "%s must be float32", what);
        throw Failed();
    }
}
void want_2d(const at::Tensor &t, const char *what)
{
    if (t.dim() != 2) {
        PyErr_Format(PyExc_ValueError, "%s must have two dimensions", what);
        throw Failed();
    }
}

PyObject *py_pack(PyObject *const *v)                    // dense, layout, out
{
    const at::Tensor &dense = tensor(v[0], "dense");
    const st_layout l = layout_of(v[1]);
    const int64_t n = api.packed_elems(&l);
    if (n < 0) check(ST_ERR_SHAPE, "st_packed_elems");
    if (dense.numel() != api.dense_elems(&l)) {
        PyErr_Format(PyExc_ValueError, "dense has %lld elements, layout needs %lld", (long long)dense.numel(), (long long)api.dense_elems(&l));
        throw Failed();
    }
    const st_dtype type = copy_dtype(dense);
    void *src = device_ptr(dense, "dense");
    Ref out(Py_None == v[2] ? [&] { Ref ty(PyObject_GetAttr(v[0], s_dtype)); return allocate(v[0], dense, {n}, dense.scalar_type(), ty.o); }()
                            : (Py_INCREF(v[2]), v[2]));
    void *dst = result_ptr(dense, out.o, (size_t)n * dense.element_size());
    call("st_pack", [&](void *s) { return api.pack(&l, type, src, dst, s); });
    return out.release();
}

PyObject *py_unpack(PyObject *const *v)                  // packed, layout, fill, out
{
    const at::Tensor &packed = tensor(v[0], "packed");
    const st_layout l = layout_of(v[1]);
    const int64_t n = api.dense_elems(&l);
    if (n < 0) check(ST_ERR_SHAPE, "st_dense_elems");
    if (packed.numel() != api.packed_elems(&l)) {
        PyErr_Format(PyExc_ValueError, "packed has %lld elements, layout needs %lld", (long long)packed.numel(), (long long)api.packed_elems(&l));
        throw Failed();
    }
    const st_dtype type = copy_dtype(packed);
    const st_fill fill = (st_fill)whole(v[2]);
    void *src = device_ptr(packed, "packed");
    Ref out(Py_None == v[3] ? [&] { Ref ty(PyObject_GetAttr(v[0], s_dtype)); return allocate(v[0], packed, {n}, packed.scalar_type(), ty.o); }()
                            : (Py_INCREF(v[3]), v[3]));
    void *dst = result_ptr(packed, out.o, (size_t)n * packed.element_size());
    call("st_unpack", [&](void *s) { return api.unpack(&l, type, src, dst, fill, s); });
    return out.release();
}

PyObject *py_thp(PyObject *const *v)                     // Bp, C, layout, out
{
    const at::Tensor &B = tensor(v[0], "Bp"), &C = tensor(v[1], "C");
    want_f32(B, "inputs");
    want_f32(C, "inputs");
    const st_layout l = layout_of(v[2]);
    if (B.numel() != api.packed_elems(&l) || C.numel() != api.dense_elems(&l)) fail(PyExc_ValueError, "shape mismatch");
    const float *b = f32_ptr(B, "Bp"), *c = f32_ptr(C, "C");
    want_device_of(B, C, "C");
    Ref out(output(v[3], v[0], B, B.sizes()));
    float *o = (float *)result_ptr(B, out.o, sizeof(float) * (size_t)B.numel());
    call("st_thp", [&](void *s) { return api.thp(&l, b, c, o, s); });
    return out.release();
}

void want_pair(const at::Tensor &a, const at::Tensor &b)
{
    if (a.scalar_type() != at::kFloat || b.scalar_type() != at::kFloat || a.numel() != b.numel())
        fail(PyExc_ValueError, "two float32 arrays of the same size are needed");
}

PyObject *py_axpby(PyObject *const *v)                   // alpha, a, beta, b, out
{
    const float alpha = real(v[0]), beta = real(v[2]);
    const at::Tensor &a = tensor(v[1], "a"), &b = tensor(v[3], "b");
    want_pair(a, b);
    const float *pa = f32_ptr(a, "a"), *pb = f32_ptr(b, "b");
    want_device_of(a, b, "b");
    Ref out(output(v[4], v[1], a, a.sizes()));
    float *o = (float *)result_ptr(a, out.o, sizeof(float) * (size_t)a.numel());
    const int64_t n = a.numel();
    call("st_packed_axpby", [&](void *s) { return api.packed_axpby(n, alpha, pa, beta, pb, o, s); });
    return out.release();
}

PyObject *py_mul(PyObject *const *v)                     // a, b, out
{
    const at::Tensor &a = tensor(v[0], "a"), &b = tensor(v[1], "b");
    want_pair(a, b);
    const float *pa = f32_ptr(a, "a"), *pb = f32_ptr(b, "b");
    want_device_of(a, b, "b");
    Ref out(output(v[2], v[0], a, a.sizes()));
    float *o = (float *)result_ptr(a, out.o, sizeof(float) * (size_t)a.numel());
    const int64_t n = a.numel();
    call("st_packed_mul", [&](void *s) { return api.packed_mul(n, pa, pb, o, s); });
    return out.release();
}

PyObject *py_moment2(PyObject *const *v)                 // X, out, ws, flags
{
    const at::Tensor &X = tensor(v[0], "X");
    want_2d(X, "X");
    const bool bf16 = X.scalar_type() == at::kBFloat16;
    if (!bf16 && X.scalar_type() != at::kFloat) fail(PyExc_TypeError, "X must be float32 or bfloat16");
    const st_dtype type = bf16 ? ST_BF16 : ST_F32;
    const int64_t N = X.size(0), d = X.size(1), ldx = X.stride(0);
    const unsigned flags = flag_bits(v[3]);
    const void *x = device_ptr(X, "X");
    Ref out(output(v[1], v[0], X, {d * (d + 1) / 2}));
    const Workspace w = workspace(v[2], v[0], X, ST_OP_SYM_MOMENT2, N, d, type, 0, flags);
    float *o = (float *)result_ptr(X, out.o, sizeof(float) * (size_t)(d * (d + 1) / 2));
    call("st_sym_moment2", [&](void *s) { return api.sym_moment2(x, type, N, d, ldx, o, w.ptr, w.bytes, flags, s); });
    return out.release();
}

PyObject *moment34(PyObject *const *v, int order)        // X, out, ws, flags
{
    const at::Tensor &X = tensor(v[0], "X");
    want_2d(X, "X");
    want_f32(X, "X");
    const int64_t N = X.size(0), d = X.size(1), ldx = X.stride(0);
    const unsigned flags = flag_bits(v[3]);
    const int64_t tet = d * (d + 1) * (d + 2) / 6;
    const float *x = f32_ptr(X, "X");
    Ref out(output(v[1], v[0], X, {order == 3 ? tet : tet * (d + 3) / 4}));
    const Workspace w = workspace(v[2], v[0], X, order == 3 ? ST_OP_SYM_MOMENT3 : ST_OP_SYM_MOMENT4, N, d, 0, 0, flags);
    float *o = (float *)result_ptr(X, out.o, sizeof(float) * (size_t)(order == 3 ? tet : tet * (d + 3) / 4));
    const auto f = order == 3 ? api.sym_moment3 : api.sym_moment4;
    call(order == 3 ? "st_sym_moment3" : "st_sym_moment4", [&](void *s) { return f(x, N, d, ldx, o, w.ptr, w.bytes, flags, s); });
    return out.release();
}
PyObject *py_moment3(PyObject *const *v) { return moment34(v, 3); }
PyObject *py_moment4(PyObject *const *v) { return moment34(v, 4); }

PyObject *py_mttkrp_tri(PyObject *const *v)              // Bp, C, D, out, ws, flags
{
    const at::Tensor &B = tensor(v[0], "Bp"), &C = tensor(v[1], "C"), &D = tensor(v[2], "D");
    want_2d(C, "C");
    want_2d(D, "D");
    for (const at::Tensor *t : {&B, &C, &D}) want_f32(*t, "inputs");
    const int64_t I = C.size(0), R = C.size(1), K = D.size(0);
    const unsigned flags = flag_bits(v[5]);
    const int64_t want = (flags & ST_FLAG_DENSE_CONTROL) ? times({I, I, K}) : times({I % 2 ? I : I / 2, I % 2 ? (I + 1) / 2 : I + 1, K});
    if (B.numel() != want || D.size(1) != R) fail(PyExc_ValueError, "shape mismatch");
    const float *b = f32_ptr(B, "Bp"), *c = f32_ptr(C, "C"), *d = f32_ptr(D, "D");
    want_device_of(B, C, "C");
    want_device_of(B, D, "D");
    Ref out(output(v[3], v[0], B, {I, R}));
    const Workspace w = workspace(v[4], v[0], B, ST_OP_MTTKRP_TRI, I, K, R, 0, flags);
    float *o = (float *)result_ptr(B, out.o, sizeof(float) * (size_t)(I * R));
    call("st_mttkrp_tri", [&](void *s) { return api.mttkrp_tri(b, I, K, c, d, R, o, w.ptr, w.bytes, flags, s); });
    return out.release();
}

PyObject *py_mttkrp_slice(PyObject *const *v)            // Bp, C, D, I, fixed_i, fixed_j, out, ws, flags
{
    const at::Tensor &B = tensor(v[0], "Bp"), &C = tensor(v[1], "C"), &D = tensor(v[2], "D");
    want_2d(C, "C");
    want_2d(D, "D");
    for (const at::Tensor *t : {&B, &C, &D}) want_f32(*t, "inputs");
    const int64_t J = C.size(0), R = C.size(1), K = D.size(0), I = integer(v[3]), fi = integer(v[4]), fj = integer(v[5]);
    const unsigned flags = flag_bits(v[8]);
    const int64_t rows = fi >= 0 ? (fj >= 0 ? 1 : J) : I;
    if (B.numel() != times({rows, K}) || D.size(1) != R) fail(PyExc_ValueError, "shape mismatch");
    const float *b = f32_ptr(B, "Bp"), *c = f32_ptr(C, "C"), *d = f32_ptr(D, "D");
    want_device_of(B, C, "C");
    want_device_of(B, D, "D");
    Ref out(output(v[6], v[0], B, {I, R}));
    const Workspace w = workspace(v[7], v[0], B, ST_OP_MTTKRP_SLICE, I, J, K, R, flags);
    float *o = (float *)result_ptr(B, out.o, sizeof(float) * (size_t)(I * R));
    call("st_mttkrp_slice", [&](void *s) { return api.mttkrp_slice(b, I, J, K, fi, fj, c, d, R, o, w.ptr, w.bytes, flags, s); });
    return out.release();
}

PyObject *py_ttm_blockdiag(PyObject *const *v)           // Bp, U, nblocks, bs, out, ws, flags
{
    const at::Tensor &B = tensor(v[0], "Bp"), &U = tensor(v[1], "U");
    want_2d(U, "U");
    want_f32(B, "inputs");
    want_f32(U, "inputs");
    const int64_t K = U.size(0), R = U.size(1), nb = integer(v[2]), bs = integer(v[3]), d = times({nb, bs});
    const unsigned flags = flag_bits(v[6]);
    const int64_t rows = (flags & ST_FLAG_DENSE_CONTROL) ? times({d, d}) : times({d, bs});
    if (B.numel() != times({rows, K})) fail(PyExc_ValueError, "shape mismatch");
    const float *b = f32_ptr(B, "Bp"), *u = f32_ptr(U, "U");
    want_device_of(B, U, "U");
    Ref out(output(v[4], v[0], B, {rows, R}));
    const Workspace w = workspace(v[5], v[0], B, ST_OP_TTM_BLOCKDIAG, nb, bs, K, R, flags);
    float *o = (float *)result_ptr(B, out.o, sizeof(float) * (size_t)(rows * R));
    call("st_ttm_blockdiag", [&](void *s) { return api.ttm_blockdiag(b, nb, bs, K, u, R, o, w.ptr, w.bytes, flags, s); });
    return out.release();
}

PyObject *py_ttm_packed(PyObject *const *v)              // Bp, U, layout, out, ws, flags
{
    const at::Tensor &B = tensor(v[0], "Bp"), &U = tensor(v[1], "U");
    want_2d(U, "U");
    want_f32(B, "inputs");
    want_f32(U, "inputs");
    const int64_t K = U.size(0), R = U.size(1);
    const st_layout l = layout_of(v[2]);
    if (l.inner != K || B.numel() != api.packed_elems(&l)) fail(PyExc_ValueError, "shape mismatch");
    const int64_t rows = B.numel() / K;
    const unsigned flags = flag_bits(v[5]);
    const float *b = f32_ptr(B, "Bp"), *u = f32_ptr(U, "U");
    want_device_of(B, U, "U");
    Ref out(output(v[3], v[0], B, {rows, R}));
    const Workspace w = workspace(v[4], v[0], B, ST_OP_TTM_BLOCKDIAG, rows, 1, K, R, flags);
    float *o = (float *)result_ptr(B, out.o, sizeof(float) * (size_t)(rows * R));
    call("st_ttm_packed", [&](void *s) { return api.ttm_packed(&l, b, u, R, o, w.ptr, w.bytes, flags, s); });
    return out.release();
}

// Argument count, and C++ errors as Python ones.
template <PyObject *(*F)(PyObject *const *), int N>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
        return nullptr;
    }
    if (!api.pack) {
        PyErr_SetString(PyExc_RuntimeError, "bind() has not been called");
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Failed &) {
    } catch (...) {
        torch::translate_exception_to_python(std::current_exception());
    }
    return nullptr;
}

// bind(addresses: dict name -> int, StError, torch.float32, torch.uint8, last_ws: dict)
PyObject *py_bind(PyObject *, PyObject *args)
{
    PyObject *table, *err, *f32, *u8, *last;
    if (!PyArg_ParseTuple(args, "O!OOOO!", &PyDict_Type, &table, &err, &f32, &u8, &PyDict_Type, &last)) return nullptr;
    Api a;
    const struct { const char *name; void *slot; } want[] = {
        {"st_packed_elems", &a.packed_elems}, {"st_dense_elems", &a.dense_elems}, {"st_workspace_bytes", &a.workspace_bytes},
        {"st_pack", &a.pack}, {"st_unpack", &a.unpack}, {"st_thp", &a.thp}, {"st_packed_axpby", &a.packed_axpby},
        {"st_packed_mul", &a.packed_mul}, {"st_sym_moment2", &a.sym_moment2}, {"st_sym_moment3", &a.sym_moment3},
        {"st_sym_moment4", &a.sym_moment4}, {"st_mttkrp_tri", &a.mttkrp_tri}, {"st_mttkrp_slice", &a.mttkrp_slice},
        {"st_ttm_blockdiag", &a.ttm_blockdiag}, {"st_ttm_packed", &a.ttm_packed}};
    for (const auto &w : want) {
        PyObject *v = PyDict_GetItemString(table, w.name);
        void *p = v ? PyLong_AsVoidPtr(v) : nullptr;
        if (!p) {
            if (!PyErr_Occurred()) PyErr_Format(PyExc_KeyError, "%s", w.name);
            return nullptr;
        }
        std::memcpy(w.slot, &p, sizeof(p));
    }
    for (PyObject *o : {err, f32, u8, last}) Py_INCREF(o);
    error_class = err;
    dtype_f32 = f32;
    dtype_u8 = u8;
    last_ws = last;
    api = a;
    Py_RETURN_NONE;
}

PyObject *py_set_allocator(PyObject *, PyObject *fn)
{
    PyObject *old = allocator;
    allocator = fn == Py_None ? nullptr : (Py_INCREF(fn), fn);
    Py_XDECREF(old);
    Py_RETURN_NONE;
}

#define ENTRY(name, n) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(&entry<py_##name, n>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", py_bind, METH_VARARGS, nullptr},
    {"set_allocator", py_set_allocator, METH_O, nullptr},
    ENTRY(pack, 3), ENTRY(unpack, 4), ENTRY(thp, 4), ENTRY(axpby, 5), ENTRY(mul, 3), ENTRY(moment2, 4), ENTRY(moment3, 4),
    ENTRY(moment4, 4), ENTRY(mttkrp_tri, 6), ENTRY(mttkrp_slice, 9), ENTRY(ttm_blockdiag, 7), ENTRY(ttm_packed, 6),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void)
{
    s_kind = PyUnicode_InternFromString("kind");
    s_d = PyUnicode_InternFromString("d");
    s_inner = PyUnicode_InternFromString("inner");
    s_kl = PyUnicode_InternFromString("kl");
    s_ku = PyUnicode_InternFromString("ku");
    s_nblocks = PyUnicode_InternFromString("nblocks");
    s_bs = PyUnicode_InternFromString("bs");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_device = PyUnicode_InternFromString("device");
    s_view = PyUnicode_InternFromString("view");
    return PyModule_Create(&module);
}
