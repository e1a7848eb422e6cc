// CPython module over the C ABI (include/dig_gla.h) for torch CUDA tensors: checks, allocation of results and
// workspace, the current stream and the call, without a line of Python in between.  Through ctypes a call of one
// launch took 14 to 19 us of host time (3.4 us of it to ask for the current stream, 2.6 us per allocation, 0.6 us
// per checked tensor), more than the small problems take on the GPU; here it takes 4 to 5 us, the launch
// included.  dig.py holds the documented functions, which hand their arguments over by position.
// The interpreter lock is released around every library call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>
#include <string>
#include <vector>

#include "dig_gla.h"

namespace {

using at::Tensor;
using at::ScalarType;

PyObject *g_error = nullptr;        // dig.DigError(status, where)

struct Raised {};                    // a Python exception is set

[[noreturn]] void raise(PyObject *type, const std::string &msg)
{
    PyErr_SetString(type, msg.c_str());
    throw Raised{};
}
void check(int status, const char *where)
{
    if (status == DIG_OK) return;
    PyObject *e = PyObject_CallFunction(g_error, "is", status, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Raised{};
}

// ---- arguments -------------------------------------------------------------------------------------
bool none(PyObject *o) { return o == Py_None; }
const Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string(name) + ": need a torch tensor, got " + Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}
int integer(PyObject *o)
{
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    if (v < INT_MIN || v > INT_MAX) raise(PyExc_OverflowError, "integer argument out of range");
    return (int)v;
}
// A set of scan orders, one bit each, of which the library takes the lowest four and refuses the others up to 32.
unsigned order_mask(PyObject *o)
{
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw Raised{};
    return (unsigned)v;
}
bool truth(PyObject *o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw Raised{};
    return v != 0;
}
float real(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised{};
    return (float)v;
}

std::string text(at::IntArrayRef s)
{
    std::string t = "(";
    for (size_t i = 0; i < s.size(); ++i) t += (i ? ", " : "") + std::to_string(s[i]);
    return t + (s.size() == 1 ? ",)" : ")");
}
// Device pointer of a checked tensor.
void *dev(const Tensor &t, ScalarType st, const char *name)
{
    if (!t.is_cuda() || !t.is_contiguous() || t.scalar_type() != st)
        raise(PyExc_ValueError, std::string(name) + ": need a contiguous CUDA tensor of " + c10::toString(st) + ", got " +
                                    c10::toString(t.scalar_type()) + " on " + t.device().str());
    return t.data_ptr();
}
// ... of the given shape, on the device of `like`.
void *dev(const Tensor &t, ScalarType st, at::IntArrayRef shape, const char *name, const Tensor &like)
{
    void *p = dev(t, st, name);
    if (t.sizes() != shape) raise(PyExc_ValueError, std::string(name) + ": shape " + text(t.sizes()) + " != " + text(shape));
    if (t.device() != like.device()) raise(PyExc_ValueError, std::string(name) + ": on " + t.device().str() + ", the other tensors on " + like.device().str());
    return p;
}
void *dev(PyObject *o, ScalarType st, at::IntArrayRef shape, const char *name, const Tensor &like) { return dev(tensor(o, name), st, shape, name, like); }
void *dev_opt(PyObject *o, ScalarType st, at::IntArrayRef shape, const char *name, const Tensor &like)
{
    return none(o) ? nullptr : dev(o, st, shape, name, like);
}

Tensor empty(at::IntArrayRef shape, ScalarType st, const Tensor &like)
{
    return at::detail::empty_cuda(shape, st, like.device(), std::nullopt);
}
// The caller's tensor where there is one, else a new one.
Tensor given(PyObject *o, at::IntArrayRef shape, ScalarType st, const Tensor &like, const char *name)
{
    if (none(o)) return empty(shape, st, like);
    return tensor(o, name);
}
PyObject *wrap(Tensor t) { return THPVariable_Wrap(std::move(t)); }
PyObject *wrap_opt(const Tensor &t) { return t.defined() ? wrap(t) : Py_NewRef(Py_None); }
PyObject *pack(std::initializer_list<Tensor> ts)
{
    PyObject *r = PyTuple_New((Py_ssize_t)ts.size());
    Py_ssize_t i = 0;
    for (const Tensor &t : ts) PyTuple_SET_ITEM(r, i++, wrap_opt(t));
    return r;
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

constexpr ScalarType kF32 = ScalarType::Float, kBf16 = ScalarType::BFloat16, kByte = ScalarType::Byte;
int dtype_of(const Tensor &t, bool f32_out)
{
    if (t.scalar_type() == kF32) return DIG_F32;
    if (t.scalar_type() == kBf16) return f32_out ? DIG_BF16_F32OUT : DIG_BF16;
    raise(PyExc_TypeError, std::string("unsupported storage type ") + c10::toString(t.scalar_type()));
}
ScalarType storage(int dtype) { return dtype == DIG_F32 ? kF32 : kBf16; }
ScalarType out_storage(int dtype) { return dtype == DIG_BF16 ? kBf16 : kF32; }

struct Ws {
    Tensor t;
    void *p = nullptr;
    size_t n = 0;
};
Ws workspace(PyObject *o, size_t need, const Tensor &like)
{
    Ws w;
    if (none(o)) {
        w.t = empty({(int64_t)(need > 16 ? need : 16)}, kByte, like);
    } else {                             // any type and shape: it is scratch
        w.t = tensor(o, "workspace");
        if (!w.t.is_cuda() || !w.t.is_non_overlapping_and_dense() || w.t.device() != like.device())
            raise(PyExc_ValueError, "workspace: need a dense tensor on " + like.device().str() + ", got one on " + w.t.device().str());
    }
    w.p = w.t.data_ptr();
    w.n = (size_t)w.t.numel() * w.t.element_size();
    return w;
}

// Shapes and types shared by the GLA entry points; q, k, v and the gate checked.
struct Gla {
    const Tensor &q_t;
    int B, L, H, dk, dv, gh, gw, chunk, dtype;
    std::vector<int64_t> ks, vs;
    ScalarType st, ost;
    void *q, *k, *v;
    float *gate;
    Gla(PyObject *const *a, PyObject *gh_, PyObject *gw_, PyObject *chunk_, bool f32_out) : q_t(tensor(a[0], "q"))
    {
        const Tensor &v_t = tensor(a[2], "v");
        if (q_t.dim() != 4) raise(PyExc_ValueError, "q: need 4 dimensions [B, L, H, d_k], got shape " + text(q_t.sizes()));
        if (v_t.dim() < 1) raise(PyExc_ValueError, "v: need 4 dimensions [B, L, H, d_v], got shape " + text(v_t.sizes()));
        ks = q_t.sizes().vec();
        vs = ks;
        vs[3] = v_t.size(-1);
        B = (int)ks[0]; L = (int)ks[1]; H = (int)ks[2]; dk = (int)ks[3]; dv = (int)vs[3];
        gh = integer(gh_); gw = integer(gw_); chunk = integer(chunk_);
        dtype = dtype_of(q_t, f32_out);
        st = storage(dtype);
        ost = out_storage(dtype);
        q = dev(q_t, st, "q");
        k = dev(a[1], st, ks, "k", q_t);
        v = dev(v_t, st, vs, "v", q_t);
        gate = (float *)dev(a[3], kF32, ks, "gate", q_t);
    }
    std::vector<int64_t> state() const { return {B, H, dk, dv}; }
};

#define CALL(expr, where)            \
    do {                             \
        int st_;                     \
        Py_BEGIN_ALLOW_THREADS       \
        st_ = (int)(expr);           \
        Py_END_ALLOW_THREADS         \
        check(st_, where);           \
    } while (0)

// ---- entry points (arguments by position, in the order dig.py passes them) ----------------------------
PyObject *gate_logsigmoid(PyObject *const *a)
{
    const Tensor &g = tensor(a[0], "g");
    if (g.dim() != 4) raise(PyExc_ValueError, "g: need 4 dimensions [B, L, H, d_k], got shape " + text(g.sizes()));
    const int B = (int)g.size(0), L = (int)g.size(1), H = (int)g.size(2), dk = (int)g.size(3), dtype = dtype_of(g, false);
    PyObject *seq = PySequence_Fast(a[1], "tau_per_head: need a sequence of numbers");
    if (!seq) throw Raised{};
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    std::vector<float> tau(H, 0.f);
    bool bad = n > H;
    if (bad) PyErr_SetString(PyExc_IndexError, "tau_per_head: more values than heads");
    for (Py_ssize_t i = 0; i < n && !bad; ++i) {
        const double v = PyFloat_AsDouble(PySequence_Fast_GET_ITEM(seq, i));
        bad = v == -1.0 && PyErr_Occurred();
        tau[i] = (float)v;
    }
    Py_DECREF(seq);
    if (bad) throw Raised{};
    void *gp = dev(g, storage(dtype), "g");
    Tensor gate = given(a[2], g.sizes(), kF32, g, "gate");
    float *op = (float *)dev(gate, kF32, g.sizes(), "gate", g);
    void *s = stream();
    CALL(dig_gate_logsigmoid(gp, tau.data(), op, B, L, H, dk, dtype, s), "dig_gate_logsigmoid");
    return wrap(gate);
}

// q k v gate grid_h grid_w chunk direction f32_out out workspace
PyObject *gla_fwd(PyObject *const *a)
{
    const Gla g(a, a[4], a[5], a[6], truth(a[8]));
    const int dir = integer(a[7]);
    Tensor out = given(a[9], g.vs, g.ost, g.q_t, "out");
    void *op = dev(out, g.ost, g.vs, "out", g.q_t);
    const Ws w = workspace(a[10], none(a[10]) ? dig_gla_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 0) : 0, g.q_t);
    void *s = stream();
    CALL(dig_gla_fwd(g.q, g.k, g.v, g.gate, op, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir, g.dtype, w.p, w.n, s), "dig_gla_fwd");
    return wrap(out);
}

// The four gradients: the caller's or new ones.
struct Grads {
    Tensor dq, dk, dv, dg;
    void *pq, *pk, *pv;
    float *pg;
    Grads(PyObject *o, const Gla &g)
    {
        if (none(o)) {
            dq = empty(g.ks, g.ost, g.q_t);
            dk = empty(g.ks, g.ost, g.q_t);
            dv = empty(g.vs, g.ost, g.q_t);
            dg = empty(g.ks, kF32, g.q_t);
        } else {
            PyObject *seq = PySequence_Fast(o, "grads: need (dq, dk, dv, dgate)");
            if (!seq) throw Raised{};
            const bool four = PySequence_Fast_GET_SIZE(seq) == 4;
            PyObject **it = PySequence_Fast_ITEMS(seq);
            bool tensors = four;
            for (int i = 0; i < 4 && tensors; ++i) tensors = THPVariable_Check(it[i]);
            if (tensors) {
                dq = THPVariable_Unpack(it[0]);
                dk = THPVariable_Unpack(it[1]);
                dv = THPVariable_Unpack(it[2]);
                dg = THPVariable_Unpack(it[3]);
            }
            Py_DECREF(seq);
            if (!tensors) raise(PyExc_ValueError, "grads: need four tensors (dq, dk, dv, dgate)");
        }
        pq = dev(dq, g.ost, g.ks, "dq", g.q_t);
        pk = dev(dk, g.ost, g.ks, "dk", g.q_t);
        pv = dev(dv, g.ost, g.vs, "dv", g.q_t);
        pg = (float *)dev(dg, kF32, g.ks, "dgate", g.q_t);
    }
};

// q k v gate d_out grid_h grid_w chunk direction f32_out grads workspace
PyObject *gla_bwd(PyObject *const *a)
{
    const Gla g(a, a[5], a[6], a[7], truth(a[9]));
    const int dir = integer(a[8]);
    void *dop = dev(a[4], g.st, g.vs, "d_out", g.q_t);
    const Grads r(a[10], g);
    const Ws w = workspace(a[11], none(a[11]) ? dig_gla_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 1) : 0, g.q_t);
    void *s = stream();
    CALL(dig_gla_bwd(g.q, g.k, g.v, g.gate, dop, r.pq, r.pk, r.pv, r.pg, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir, g.dtype, w.p, w.n, s),
         "dig_gla_bwd");
    return pack({r.dq, r.dk, r.dv, r.dg});
}

// q k v gate s_in grid_h grid_w chunk direction f32_out want_s_out workspace
PyObject *gla_fwd_state(PyObject *const *a)
{
    const Gla g(a, a[5], a[6], a[7], truth(a[9]));
    const int dir = integer(a[8]);
    const float *si = (const float *)dev_opt(a[4], kF32, g.state(), "s_in", g.q_t);
    Tensor out = empty(g.vs, g.ost, g.q_t), so;
    if (truth(a[10])) so = empty(g.state(), kF32, g.q_t);
    const Ws w = workspace(a[11], none(a[11]) ? dig_gla_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 0) : 0, g.q_t);
    void *op = out.data_ptr();
    float *sop = so.defined() ? (float *)so.data_ptr() : nullptr;
    void *s = stream();
    CALL(dig_gla_fwd_state(g.q, g.k, g.v, g.gate, si, op, sop, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir, g.dtype, w.p, w.n, s),
         "dig_gla_fwd_state");
    return pack({out, so});
}

// q k v gate d_out s_in ds_out grid_h grid_w chunk direction f32_out workspace
PyObject *gla_bwd_state(PyObject *const *a)
{
    const Gla g(a, a[7], a[8], a[9], truth(a[11]));
    const int dir = integer(a[10]);
    void *dop = dev(a[4], g.st, g.vs, "d_out", g.q_t);
    const float *si = (const float *)dev_opt(a[5], kF32, g.state(), "s_in", g.q_t), *dso = (const float *)dev_opt(a[6], kF32, g.state(), "ds_out", g.q_t);
    const Grads r(Py_None, g);
    Tensor dsi = empty(g.state(), kF32, g.q_t);
    float *dsip = (float *)dsi.data_ptr();
    const Ws w = workspace(a[12], none(a[12]) ? dig_gla_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 1) : 0, g.q_t);
    void *s = stream();
    CALL(dig_gla_bwd_state(g.q, g.k, g.v, g.gate, dop, si, dso, r.pq, r.pk, r.pv, r.pg, dsip, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir,
                           g.dtype, w.p, w.n, s), "dig_gla_bwd_state");
    return pack({r.dq, r.dk, r.dv, r.dg, dsi});
}

// q k v gate grid_h grid_w mask chunk f32_out out workspace
PyObject *gla_fwd_multi(PyObject *const *a)
{
    const Gla g(a, a[4], a[5], a[7], truth(a[8]));
    const unsigned mask = order_mask(a[6]);
    Tensor out = given(a[9], g.vs, g.ost, g.q_t, "out");
    void *op = dev(out, g.ost, g.vs, "out", g.q_t);
    const Ws w = workspace(a[10], none(a[10]) ? dig_gla_multi_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 0) : 0, g.q_t);
    void *s = stream();
    CALL(dig_gla_fwd_multi(g.q, g.k, g.v, g.gate, op, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, mask, g.dtype, w.p, w.n, s), "dig_gla_fwd_multi");
    return wrap(out);
}

// q k v gate d_out grid_h grid_w mask chunk f32_out grads workspace
PyObject *gla_bwd_multi(PyObject *const *a)
{
    const Gla g(a, a[5], a[6], a[8], truth(a[9]));
    const unsigned mask = order_mask(a[7]);
    void *dop = dev(a[4], g.st, g.vs, "d_out", g.q_t);
    const Grads r(a[10], g);
    const Ws w = workspace(a[11], none(a[11]) ? dig_gla_multi_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 1) : 0, g.q_t);
    void *s = stream();
    CALL(dig_gla_bwd_multi(g.q, g.k, g.v, g.gate, dop, r.pq, r.pk, r.pv, r.pg, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, mask, g.dtype, w.p, w.n, s),
         "dig_gla_bwd_multi");
    return pack({r.dq, r.dk, r.dv, r.dg});
}

size_t beta_need(const Gla &g, int backward)
{
    const size_t need = dig_gla_beta_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, backward);
    if (need == 0) check(DIG_ERR_UNSUPPORTED, "dig_gla_beta_workspace_bytes");
    return need;
}
// q k v gate bgate grid_h grid_w chunk direction f32_out workspace
PyObject *gla_fwd_beta(PyObject *const *a)
{
    const Gla g(a, a[5], a[6], a[7], truth(a[9]));
    const int dir = integer(a[8]);
    const float *bg = (const float *)dev(a[4], kF32, g.vs, "bgate", g.q_t);
    const Ws w = workspace(a[10], beta_need(g, 0), g.q_t);
    Tensor out = empty(g.vs, g.ost, g.q_t);
    void *op = out.data_ptr(), *s = stream();
    CALL(dig_gla_fwd_beta(g.q, g.k, g.v, g.gate, bg, op, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir, g.dtype, w.p, w.n, s), "dig_gla_fwd_beta");
    return wrap(out);
}
// q k v gate bgate d_out grid_h grid_w chunk direction f32_out workspace
PyObject *gla_bwd_beta(PyObject *const *a)
{
    const Gla g(a, a[6], a[7], a[8], truth(a[10]));
    const int dir = integer(a[9]);
    const float *bg = (const float *)dev(a[4], kF32, g.vs, "bgate", g.q_t);
    void *dop = dev(a[5], g.st, g.vs, "d_out", g.q_t);
    const Ws w = workspace(a[11], beta_need(g, 1), g.q_t);
    const Grads r(Py_None, g);
    Tensor db = empty(g.vs, kF32, g.q_t);
    float *dbp = (float *)db.data_ptr();
    void *s = stream();
    CALL(dig_gla_bwd_beta(g.q, g.k, g.v, g.gate, bg, dop, r.pq, r.pk, r.pv, r.pg, dbp, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir, g.dtype, w.p,
                          w.n, s), "dig_gla_bwd_beta");
    return pack({r.dq, r.dk, r.dv, r.dg, db});
}

// q k v gate r grid_h grid_w chunk direction ln_w ln_b eps f32_out want_out workspace
PyObject *gla_fwd_outgate(PyObject *const *a)
{
    const Gla g(a, a[5], a[6], a[7], truth(a[12]));
    const int dir = integer(a[8]);
    const void *rp = dev(a[4], g.st, g.vs, "r", g.q_t);
    const float *lw = (const float *)dev_opt(a[9], kF32, {g.dv}, "ln_w", g.q_t), *lb = (const float *)dev_opt(a[10], kF32, {g.dv}, "ln_b", g.q_t);
    const float eps = real(a[11]);
    Tensor out, z = empty(g.vs, g.ost, g.q_t);
    if (truth(a[13])) out = empty(g.vs, g.ost, g.q_t);
    const Ws w = workspace(a[14], none(a[14]) ? dig_gla_workspace_bytes(g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, g.dtype, 0) : 0, g.q_t);
    void *op = out.defined() ? out.data_ptr() : nullptr, *zp = z.data_ptr(), *s = stream();
    CALL(dig_gla_fwd_outgate(g.q, g.k, g.v, g.gate, rp, lw, lb, eps, op, zp, g.B, g.H, g.gh, g.gw, g.dk, g.dv, g.chunk, dir, g.dtype, w.p, w.n, s),
         "dig_gla_fwd_outgate");
    return pack({out, z});
}

// The rows of a tensor [..., d].
void rows_of(const Tensor &o, int &d, long long &rows)
{
    if (o.dim() < 1 || o.size(-1) < 1) raise(PyExc_ValueError, "o: need rows of at least one value, got shape " + text(o.sizes()));
    d = (int)o.size(-1);
    rows = o.numel() / d;
}
// o r ln_w ln_b eps f32_out
PyObject *outgate_fwd(PyObject *const *a)
{
    const Tensor &o = tensor(a[0], "o");
    int d;
    long long rows;
    rows_of(o, d, rows);
    const int dtype = dtype_of(o, truth(a[5]));
    const ScalarType st = storage(dtype);
    const void *op = dev(o, st, "o"), *rp = dev(a[1], st, o.sizes(), "r", o);
    const float *lw = (const float *)dev_opt(a[2], kF32, {d}, "ln_w", o), *lb = (const float *)dev_opt(a[3], kF32, {d}, "ln_b", o);
    const float eps = real(a[4]);
    Tensor z = empty(o.sizes(), out_storage(dtype), o);
    void *zp = z.data_ptr(), *s = stream();
    CALL(dig_gla_outgate_fwd(op, rp, lw, lb, zp, rows, d, eps, dtype, s), "dig_gla_outgate_fwd");
    return wrap(z);
}
// o r dz ln_w ln_b eps affine_grads f32_out workspace
PyObject *outgate_bwd(PyObject *const *a)
{
    const Tensor &o = tensor(a[0], "o");
    int d;
    long long rows;
    rows_of(o, d, rows);
    const int dtype = dtype_of(o, truth(a[7]));
    const ScalarType st = storage(dtype);
    const void *op = dev(o, st, "o"), *rp = dev(a[1], st, o.sizes(), "r", o), *zp = dev(a[2], st, o.sizes(), "dz", o);
    const float *lw = (const float *)dev_opt(a[3], kF32, {d}, "ln_w", o), *lb = (const float *)dev_opt(a[4], kF32, {d}, "ln_b", o);
    const float eps = real(a[5]);
    Tensor d_o = empty(o.sizes(), out_storage(dtype), o), d_r = empty(o.sizes(), out_storage(dtype), o), dw, db;
    Ws w;
    if (truth(a[6])) {
        dw = empty({d}, kF32, o);
        db = empty({d}, kF32, o);
        if (!none(a[8])) dev(tensor(a[8], "workspace"), kByte, "workspace");
        w = workspace(a[8], none(a[8]) ? dig_gla_outgate_bwd_workspace_bytes(rows, d) : 0, o);
    }
    void *dop = d_o.data_ptr(), *drp = d_r.data_ptr(), *s = stream();
    float *dwp = dw.defined() ? (float *)dw.data_ptr() : nullptr, *dbp = db.defined() ? (float *)db.data_ptr() : nullptr;
    CALL(dig_gla_outgate_bwd(op, rp, lw, lb, zp, dop, drp, dwp, dbp, rows, d, eps, dtype, w.p, w.n, s), "dig_gla_outgate_bwd");
    return pack({d_o, d_r, dw, db});
}

// x w bias grid_h grid_w direction f32_out y
PyObject *dwconv(PyObject *const *a)
{
    const Tensor &x = tensor(a[0], "x");
    if (x.dim() != 3) raise(PyExc_ValueError, "x: need 3 dimensions [B, L, D], got shape " + text(x.sizes()));
    const int64_t D = x.size(2);
    const int gh = integer(a[3]), gw = integer(a[4]), dir = integer(a[5]);
    if (x.size(1) != (int64_t)gh * gw) raise(PyExc_ValueError, "x: L != grid_h*grid_w");
    const int dtype = dtype_of(x, truth(a[6]));
    const ScalarType st = storage(dtype), ost = out_storage(dtype);
    const void *xp = dev(x, st, "x"), *wp = dev(a[1], st, {3, 3, D}, "w", x), *bp = dev_opt(a[2], st, {D}, "bias", x);
    Tensor y = given(a[7], x.sizes(), ost, x, "y");
    void *yp = dev(y, ost, x.sizes(), "y", x), *s = stream();
    const int B = (int)x.size(0);
    CALL(dig_srem_dwconv(xp, wp, bp, yp, B, gh, gw, (int)D, dir, dtype, s), "dig_srem_dwconv");
    return wrap(y);
}
// x w dy grid_h grid_w direction with_bias f32_out workspace
PyObject *dwconv_bwd(PyObject *const *a)
{
    const Tensor &x = tensor(a[0], "x");
    if (x.dim() != 3) raise(PyExc_ValueError, "x: need 3 dimensions [B, L, D], got shape " + text(x.sizes()));
    const int64_t D = x.size(2);
    const int gh = integer(a[3]), gw = integer(a[4]), dir = integer(a[5]), B = (int)x.size(0);
    if (x.size(1) != (int64_t)gh * gw) raise(PyExc_ValueError, "x.shape[1] must equal grid_h * grid_w");
    const int dtype = dtype_of(x, truth(a[7]));
    const ScalarType st = storage(dtype);
    const size_t need = dig_srem_dwconv_bwd_workspace_bytes(B, gh, gw, (int)D);
    if (need == 0) raise(PyExc_ValueError, "dig_srem_dwconv_bwd: unsupported sizes");
    const void *xp = dev(x, st, "x"), *wp = dev(a[1], st, {3, 3, D}, "w", x), *gp = dev(a[2], st, x.sizes(), "dy", x);
    if (!none(a[8])) dev(tensor(a[8], "workspace"), kByte, "workspace");
    const Ws w = workspace(a[8], need, x);
    Tensor dx = empty(x.sizes(), out_storage(dtype), x), dw = empty({3, 3, D}, kF32, x), db;
    if (truth(a[6])) db = empty({D}, kF32, x);
    void *dxp = dx.data_ptr(), *s = stream();
    float *dwp = (float *)dw.data_ptr(), *dbp = db.defined() ? (float *)db.data_ptr() : nullptr;
    CALL(dig_srem_dwconv_bwd(xp, wp, gp, dxp, dwp, dbp, B, gh, gw, (int)D, dir, dtype, w.p, w.n, s), "dig_srem_dwconv_bwd");
    return pack({dx, dw, db});
}

template <PyObject *(*F)(PyObject *const *), int N>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "need %d arguments, got %zd", N, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Raised &) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

PyObject *set_error(PyObject *, PyObject *cls)
{
    Py_XSETREF(g_error, Py_NewRef(cls));
    Py_RETURN_NONE;
}

#define FAST(name, n) {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    {"set_error", set_error, METH_O, nullptr},
    FAST(gate_logsigmoid, 3), FAST(gla_fwd, 11), FAST(gla_bwd, 12), FAST(gla_fwd_state, 12), FAST(gla_bwd_state, 13),
    FAST(gla_fwd_multi, 11), FAST(gla_bwd_multi, 12), FAST(gla_fwd_beta, 11), FAST(gla_bwd_beta, 12), FAST(gla_fwd_outgate, 15),
    FAST(outgate_fwd, 6), FAST(outgate_bwd, 9), FAST(dwconv, 8), FAST(dwconv_bwd, 9),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&kModule); }
