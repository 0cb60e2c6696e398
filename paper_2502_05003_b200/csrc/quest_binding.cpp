// CPython binding of the calls a training or serving loop makes once per layer: it allocates the outputs that the
// caller did not provide and calls the C ABI (quest.h) with the current stream, without the Python-level argument
// marshalling (a layer with every output to allocate: 38 us of host time through ctypes, more than the GPU needs).
//
// Every function takes the positional arguments of the Python function of the same name (__init__.py) and returns
//   * its result, when the call was made and accepted;
//   * an int, the quest_status of a call that the library refused;
//   * None, when the arguments are not the plain case (an argument of another type, a tensor that is not in CUDA
//     memory, a tensor subclass, an unsupported dtype, strides that the C ABI does not take, a buffer that is too small,
//     a shape the library has no workspace for): nothing has been
//     done, and the Python function goes on to raise what it raises for such arguments or to handle them.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "quest.h"

namespace {

struct NotPlain {};                     // thrown to hand the call back to Python

// A new reference that is dropped when the scope is left without release().
struct Ref {
    PyObject *p;
    explicit Ref(PyObject *q) : p(q) { if (!q) throw python_error(); }
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
    PyObject *release() { PyObject *q = p; p = nullptr; return q; }
};

const at::Tensor &plain_tensor(PyObject *o, bool cuda = true) {
    if (!o || !THPVariable_CheckExact(o)) throw NotPlain();
    const at::Tensor &t = THPVariable_Unpack(o);
    if (t.layout() != at::kStrided || (cuda && !t.is_cuda())) throw NotPlain();
    return t;
}
const at::Tensor &matrix(PyObject *o) {
    const at::Tensor &t = plain_tensor(o);
    if (t.dim() != 2) throw NotPlain();
    return t;
}
const at::Tensor &dense(PyObject *o) {   // a matrix without gaps: the layer calls take no leading dimension
    const at::Tensor &t = matrix(o);
    if (!t.is_contiguous()) throw NotPlain();
    return t;
}
const at::Tensor &dense_like(PyObject *o, const at::Tensor &x) {         // w beside x
    const at::Tensor &t = dense(o);
    if (t.scalar_type() != x.scalar_type() || t.size(1) != x.size(1)) throw NotPlain();
    return t;
}
void *room(PyObject *o, int64_t bytes) {  // a buffer of at least that size, or None
    if (!o || o == Py_None) return nullptr;
    const at::Tensor &t = plain_tensor(o);
    if (!t.is_contiguous() || (int64_t)t.nbytes() < bytes) throw NotPlain();
    return t.data_ptr();
}
void *ptr(PyObject *o) {                // a tensor, or None
    if (!o || o == Py_None) return nullptr;
    return plain_tensor(o, false).data_ptr();
}
int code_of(at::ScalarType t) {
    if (t == at::kFloat) return QUEST_F32;
    if (t == at::kBFloat16) return QUEST_BF16;
    throw NotPlain();
}
at::ScalarType dtype_arg(PyObject *o) {
    if (!THPDtype_Check(o)) throw NotPlain();
    const at::ScalarType t = reinterpret_cast<THPDtype *>(o)->scalar_type;
    code_of(t);
    return t;
}
int64_t int_arg(PyObject *o) {
    if (!PyLong_CheckExact(o)) throw NotPlain();
    int overflow = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
    if (overflow || v < INT32_MIN || v > INT32_MAX) throw NotPlain();
    return v;
}
float float_arg(PyObject *o) {
    if (PyFloat_CheckExact(o)) return (float)PyFloat_AS_DOUBLE(o);
    return (float)int_arg(o);
}
bool bool_arg(PyObject *o) {
    if (o == Py_True) return true;
    if (o == Py_False) return false;
    throw NotPlain();
}
int bits_arg(PyObject *o) {
    const int64_t b = int_arg(o);
    if (b < 1 || b > 8) throw NotPlain();
    return (int)b;
}
int64_t container(int bits) { return bits == 1 ? 1 : bits == 2 ? 2 : bits <= 4 ? 4 : 8; }

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor fresh(at::IntArrayRef shape, at::ScalarType t, const at::Device &dev) {
    return at::empty(shape, at::TensorOptions().dtype(t).device(dev));
}

// Interned dictionary keys, made when the module is loaded.
#define QUEST_KEYS(X) \
    X(xq) X(sx) X(mx) X(wq) X(sw) X(mw) X(y) X(xh) X(dx) X(dw) X(h) X(workspace) X(operand_in_workspace) \
    X(wgq) X(swg) X(mwg) X(wuq) X(swu) X(mwu) X(hq) X(sh) X(mh) X(wdq) X(swd) X(mwd)
#define QUEST_KEY_DECLARE(name) PyObject *k_##name = nullptr;
QUEST_KEYS(QUEST_KEY_DECLARE)
PyObject *item(PyObject *dict, PyObject *key) {            // borrowed; NULL where missing
    PyObject *v = PyDict_GetItemWithError(dict, key);
    if (!v && PyErr_Occurred()) throw python_error();
    return v;
}

// A dict of named tensors under construction.
struct Named {
    PyObject *d;
    at::Device dev;
    PyObject *get(PyObject *key) const {                   // borrowed; NULL where missing or None
        PyObject *v = item(d, key);
        return v == Py_None ? nullptr : v;
    }
    void set(PyObject *key, PyObject *v) { if (PyDict_SetItem(d, key, v) < 0) throw python_error(); }
    // the tensor under that name, with room for that shape (`any`: as it is), or a new one; its memory
    void *need(PyObject *key, at::IntArrayRef shape, at::ScalarType t, bool any = false) {
        if (PyObject *given = get(key)) {
            if (any) return ptr(given);
            int64_t n = (int64_t)c10::elementSize(t);
            for (const int64_t s : shape) n *= s;
            return room(given, n);
        }
        at::Tensor made = fresh(shape, t, dev);
        void *const p = made.data_ptr();
        Ref v(THPVariable_Wrap(std::move(made)));
        set(key, v.p);
        return p;
    }
    void *at(PyObject *key) const { return ptr(get(key)); }
};

PyObject *copy_of_dict(PyObject *o) {
    if (o == Py_None) return PyDict_New();
    if (!PyDict_CheckExact(o)) throw NotPlain();
    return PyDict_Copy(o);
}

template <typename F>
int unlocked(F &&f) {
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = f();
    Py_END_ALLOW_THREADS
    return s;
}

template <PyObject *(*F)(PyObject *const *)>
PyObject *guarded(PyObject *const *args) {
    HANDLE_TH_ERRORS
    try {
        return F(args);
    } catch (const NotPlain &) {
        Py_RETURN_NONE;
    }
    END_HANDLE_TH_ERRORS
}
template <PyObject *(*F)(PyObject *const *), int N>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != N) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    return guarded<F>(args);
}

// x, bits, had_block, trust_factor, codes, scales, mask, want_mask
PyObject *quantize(PyObject *const *a) {
    const at::Tensor &x = matrix(a[0]);
    const int bits = bits_arg(a[1]);
    const int64_t g = int_arg(a[2]), rows = x.size(0), cols = x.size(1);
    const float trust = float_arg(a[3]);
    const int dt = code_of(x.scalar_type());
    if (x.stride(1) != 1) throw NotPlain();
    auto given = [](PyObject *o) { if (o != Py_None) plain_tensor(o); return o != Py_None; };
    const bool gc = given(a[4]), gs = given(a[5]), gm = given(a[6]), want = bool_arg(a[7]) || gm;
    auto own = [](PyObject *o) { Py_INCREF(o); return o; };
    Ref codes(gc ? own(a[4]) : THPVariable_Wrap(fresh({rows, cols * container(bits) / 8}, at::kByte, x.device())));
    Ref scales(gs ? own(a[5]) : THPVariable_Wrap(fresh({rows}, at::kFloat, x.device())));
    Ref mask(gm ? own(a[6]) : want ? THPVariable_Wrap(fresh({rows, cols / 8}, at::kByte, x.device())) : own(Py_None));
    const void *xp = x.data_ptr();
    void *cp = ptr(codes.p), *sp = ptr(scales.p), *mp = ptr(mask.p), *st = stream();
    const int64_t ld = x.stride(0);
    const int s = unlocked([&] {
        return quest_quantize(xp, dt, rows, cols, ld, bits, (int)g, trust, (uint8_t *)cp, (float *)sp, (uint8_t *)mp, st);
    });
    if (s) return PyLong_FromLong(s);
    return PyTuple_Pack(3, codes.p, scales.p, mask.p);
}

// xq, sx, bits_x, wq, sw, bits_w, K, out_dtype, y, want_acc, acc, workspace, want_y
PyObject *lowbit_gemm(PyObject *const *a) {
    const at::Tensor &xq = matrix(a[0]), &sx = plain_tensor(a[1]), &wq = matrix(a[3]), &sw = plain_tensor(a[4]);
    const int bx = bits_arg(a[2]), bw = bits_arg(a[5]);
    const int64_t K = int_arg(a[6]), M = xq.size(0), N = wq.size(0);
    const at::ScalarType ot = dtype_arg(a[7]);
    const bool gy = a[8] != Py_None, ga = a[10] != Py_None;
    const bool want_y = bool_arg(a[12]) || gy, want_acc = bool_arg(a[9]) || ga;
    const at::Tensor y = gy ? matrix(a[8]) : want_y ? fresh({M, N}, ot, xq.device()) : at::Tensor();
    const at::Tensor acc = ga ? plain_tensor(a[10]) : want_acc ? fresh({M, N}, at::kInt, xq.device()) : at::Tensor();
    at::Tensor ws;
    if (a[11] != Py_None) {
        ws = plain_tensor(a[11]);
    } else {
        const size_t n = quest_workspace_bytes(M, N, K, bx, bw);
        if (!n) throw NotPlain();
        ws = fresh({(int64_t)n}, at::kByte, xq.device());
    }
    const int ydt = y.defined() ? code_of(y.scalar_type()) : 0;
    const int64_t ldy = y.defined() ? y.stride(0) : N;
    void *yp = y.defined() ? y.data_ptr() : nullptr, *ap = acc.defined() ? acc.data_ptr() : nullptr, *st = stream();
    const int s = unlocked([&] {
        return quest_lowbit_gemm((const uint8_t *)xq.data_ptr(), (const float *)sx.data_ptr(), bx, (const uint8_t *)wq.data_ptr(),
                                 (const float *)sw.data_ptr(), bw, M, N, K, yp, ydt, ldy, (int32_t *)ap, ws.data_ptr(),
                                 (size_t)ws.numel(), st);
    });
    if (s) return PyLong_FromLong(s);
    auto out = [](bool given, PyObject *o, const at::Tensor &t) {
        if (given || !t.defined()) { PyObject *r = given ? o : Py_None; Py_INCREF(r); return r; }
        return THPVariable_Wrap(t);
    };
    Ref ry(out(gy, a[8], y)), ra(out(ga, a[10], acc));
    return PyTuple_Pack(2, ry.p, ra.p);
}

// x, w, bits, had_block, trust_factor, out_dtype, y, saved, w_cached, workspace, want_masks
PyObject *linear_fwd(PyObject *const *a) {
    const at::Tensor &x = dense(a[0]);
    const int bits = bits_arg(a[2]);
    const int64_t g = int_arg(a[3]), M = x.size(0), K = x.size(1), cb = container(bits);
    const float trust = float_arg(a[4]);
    const int xdt = code_of(x.scalar_type());
    const void *wp = a[1] == Py_None ? nullptr : plain_tensor(a[1]).data_ptr();
    const at::ScalarType ot = a[5] == Py_None ? x.scalar_type() : dtype_arg(a[5]);
    const bool masks = bool_arg(a[10]);
    Ref dict(copy_of_dict(a[7]));
    Named out{dict.p, x.device()};
    int cached = 0;
    int64_t N;
    if (a[8] != Py_None) {
        if (!PyDict_CheckExact(a[8])) throw NotPlain();
        PyObject *wq = item(a[8], k_wq), *sw = item(a[8], k_sw);
        N = matrix(wq).size(0);
        plain_tensor(sw);
        out.set(k_wq, wq);
        out.set(k_sw, sw);
        PyObject *held = item(a[8], k_operand_in_workspace);
        const int h = held ? PyObject_IsTrue(held) : 0;
        if (h < 0) throw python_error();
        cached = h ? 2 : 1;
    } else {
        N = dense_like(a[1], x).size(0);
    }
    uint8_t *xq = (uint8_t *)out.need(k_xq, {M, K * cb / 8}, at::kByte);
    float *sx = (float *)out.need(k_sx, {M}, at::kFloat);
    uint8_t *wq = (uint8_t *)out.need(k_wq, {N, K * cb / 8}, at::kByte);
    float *sw = (float *)out.need(k_sw, {N}, at::kFloat);
    // masks: those that are wanted, and any that the caller gives
    uint8_t *mx = nullptr, *mw = nullptr;
    if (masks || out.get(k_mx)) mx = (uint8_t *)out.need(k_mx, {M, K / 8}, at::kByte);
    if (!cached && (masks || out.get(k_mw))) mw = (uint8_t *)out.need(k_mw, {N, K / 8}, at::kByte);
    for (PyObject *key : {k_mx, k_mw})
        if (!item(dict.p, key)) out.set(key, Py_None);
    at::Tensor y, ws;
    if (a[6] != Py_None) {
        y = plain_tensor(a[6]);
        code_of(y.scalar_type());
        room(a[6], M * N * y.element_size());
    } else {
        y = fresh({M, N}, ot, x.device());
    }
    if (a[9] != Py_None) {
        ws = plain_tensor(a[9]);
    } else {
        const size_t n = quest_workspace_bytes(M, N, K, bits, bits);
        if (!n) throw NotPlain();
        ws = fresh({(int64_t)n}, at::kByte, x.device());
    }
    const int ydt = code_of(y.scalar_type());
    void *st = stream();
    const int s = unlocked([&] {
        return quest_linear_fwd(x.data_ptr(), wp, xdt, M, N, K, bits, (int)g, trust, y.data_ptr(), ydt, xq, sx, mx, wq, sw, mw,
                                cached, ws.data_ptr(), (size_t)ws.numel(), st);
    });
    if (s) return PyLong_FromLong(s);
    if (a[6] != Py_None) {
        out.set(k_y, a[6]);
    } else {
        Ref v(THPVariable_Wrap(y));
        out.set(k_y, v.p);
    }
    return dict.release();
}

// dy, fwd, bits, had_block, K, out_dtype, dx, dw, want_dx, want_dw, workspace
PyObject *linear_bwd(PyObject *const *a) {
    const at::Tensor &dy = matrix(a[0]);
    if (dy.scalar_type() != at::kBFloat16 || !dy.is_contiguous() || !PyDict_CheckExact(a[1])) throw NotPlain();
    const int bits = bits_arg(a[2]);
    const int64_t g = int_arg(a[3]), K = int_arg(a[4]), M = dy.size(0), N = dy.size(1);
    const at::ScalarType ot = dtype_arg(a[5]);
    const bool gx = a[6] != Py_None, gw = a[7] != Py_None;
    const bool want_x = bool_arg(a[8]) || gx, want_w = bool_arg(a[9]) || gw;
    if (!want_x && !want_w) throw NotPlain();
    const void *in[6];
    PyObject *const keys[6] = {k_xq, k_sx, k_mx, k_wq, k_sw, k_mw};
    for (int i = 0; i < 6; ++i) {
        PyObject *v = item(a[1], keys[i]);
        if (!v) throw NotPlain();
        in[i] = v == Py_None ? nullptr : plain_tensor(v).data_ptr();
    }
    at::Tensor dx, dw, ws;
    if (gx) dx = plain_tensor(a[6]);
    if (gw) dw = plain_tensor(a[7]);
    size_t n = 0;
    if (a[10] != Py_None) ws = plain_tensor(a[10]);
    else if (!(n = quest_bwd_workspace_bytes(M, N, K))) throw NotPlain();
    if (want_x && !gx) dx = fresh({M, K}, ot, dy.device());
    if (want_w && !gw) dw = fresh({N, K}, ot, dy.device());
    if (n) ws = fresh({(int64_t)n}, at::kByte, dy.device());
    const int odt = code_of((dx.defined() ? dx : dw).scalar_type());
    void *dxp = dx.defined() ? dx.data_ptr() : nullptr, *dwp = dw.defined() ? dw.data_ptr() : nullptr, *st = stream();
    const int s = unlocked([&] {
        return quest_linear_bwd(dy.data_ptr(), M, N, K, bits, (int)g, (const uint8_t *)in[0], (const float *)in[1],
                                (const uint8_t *)in[2], (const uint8_t *)in[3], (const float *)in[4], (const uint8_t *)in[5], dxp,
                                dwp, odt, ws.data_ptr(), (size_t)ws.numel(), st);
    });
    if (s) return PyLong_FromLong(s);
    Ref d(PyDict_New());
    Named out{d.p, dy.device()};
    auto put = [&](PyObject *key, bool given, PyObject *o, const at::Tensor &t) {
        if (given || !t.defined()) { out.set(key, given ? o : Py_None); return; }
        Ref v(THPVariable_Wrap(t));
        out.set(key, v.p);
    };
    put(k_dx, gx, a[6], dx);
    put(k_dw, gw, a[7], dw);
    return d.release();
}

// x, w, had_block, trust_factor, out_dtype, w_cached, workspace
PyObject *linear_fwd_fp4(PyObject *const *a) {
    const at::Tensor &x = dense(a[0]);
    const int64_t g = int_arg(a[2]), M = x.size(0), K = x.size(1);
    const float trust = float_arg(a[3]);
    const int xdt = code_of(x.scalar_type());
    const void *wp = a[1] == Py_None ? nullptr : plain_tensor(a[1]).data_ptr();
    const at::ScalarType ot = a[4] == Py_None ? x.scalar_type() : dtype_arg(a[4]);
    Ref dict(PyDict_New());
    Named out{dict.p, x.device()};
    int64_t N;
    const bool cached = a[5] != Py_None;
    if (cached) {
        if (!PyDict_CheckExact(a[5])) throw NotPlain();
        PyObject *wq = item(a[5], k_wq), *sw = item(a[5], k_sw);
        N = matrix(wq).size(0);
        plain_tensor(sw);
        out.set(k_wq, wq);
        out.set(k_sw, sw);
        out.set(k_mw, Py_None);
    } else {
        N = dense_like(a[1], x).size(0);
    }
    uint8_t *wq = (uint8_t *)out.need(k_wq, {N, K / 2}, at::kByte);
    float *sw = (float *)out.need(k_sw, {N}, at::kFloat);
    uint8_t *mw = cached ? nullptr : (uint8_t *)out.need(k_mw, {N, K / 8}, at::kByte);
    void *wsp = nullptr;
    size_t wsn = 0;
    if (a[6] != Py_None) {
        const at::Tensor &t = plain_tensor(a[6]);
        wsp = t.data_ptr();
        wsn = (size_t)t.numel();
    }
    uint8_t *xq = (uint8_t *)out.need(k_xq, {M, K / 2}, at::kByte);
    float *sx = (float *)out.need(k_sx, {M}, at::kFloat);
    uint8_t *mx = (uint8_t *)out.need(k_mx, {M, K / 8}, at::kByte);
    Ref yv(THPVariable_Wrap(fresh({M, N}, ot, x.device())));
    void *yp = ptr(yv.p), *st = stream();
    const int s = unlocked([&] {
        return quest_linear_fwd_fp4(x.data_ptr(), wp, xdt, M, N, K, (int)g, trust, yp, code_of(ot), xq, sx, mx, wq, sw, mw,
                                    cached ? 1 : 0, wsp, wsn, st);
    });
    if (s) return PyLong_FromLong(s);
    out.set(k_y, yv.p);
    return dict.release();
}

// x, w, bits_w, had_block, trust_factor, out_dtype, out, workspace
PyObject *linear_fwd_weight_only(PyObject *const *a) {
    const at::Tensor &x = matrix(a[0]), &w = matrix(a[1]);
    if (x.stride(1) != 1 || w.stride(1) != 1 || x.size(1) != w.size(1)) throw NotPlain();
    const int bits = bits_arg(a[2]);
    const int64_t g = int_arg(a[3]), M = x.size(0), K = x.size(1), N = w.size(0);
    const float trust = float_arg(a[4]);
    const int xdt = code_of(x.scalar_type()), wdt = code_of(w.scalar_type());
    const at::ScalarType ot = dtype_arg(a[5]);
    Ref dict(copy_of_dict(a[6]));
    Named out{dict.p, x.device()};
    for (PyObject *key : {k_y, k_xh, k_wq, k_sw, k_mw})
        if (PyObject *v = out.get(key)) plain_tensor(v);
    size_t n = 0;
    at::Tensor ws;
    if (a[7] != Py_None) ws = plain_tensor(a[7]);
    else if (!(n = quest_weight_only_workspace_bytes(M, N, K))) throw NotPlain();
    out.need(k_y, {M, N}, ot, true);
    out.need(k_xh, {M, K}, at::kBFloat16, true);
    out.need(k_wq, {N, K * container(bits) / 8}, at::kByte, true);
    out.need(k_sw, {N}, at::kFloat, true);
    out.need(k_mw, {N, K / 8}, at::kByte, true);
    if (n) ws = fresh({(int64_t)n}, at::kByte, x.device());
    const at::Tensor &y = matrix(out.get(k_y));
    const int ydt = code_of(y.scalar_type());
    void *xh = out.at(k_xh), *wq = out.at(k_wq), *sw = out.at(k_sw), *mw = out.at(k_mw), *st = stream();
    const int64_t ldx = x.stride(0), ldw = w.stride(0), ldy = y.stride(0);
    const int s = unlocked([&] {
        return quest_linear_fwd_weight_only(x.data_ptr(), xdt, ldx, w.data_ptr(), wdt, ldw, M, N, K, bits, (int)g, trust,
                                            y.data_ptr(), ydt, ldy, xh, (uint8_t *)wq, (float *)sw, (uint8_t *)mw, ws.data_ptr(),
                                            (size_t)ws.numel(), st);
    });
    if (s) return PyLong_FromLong(s);
    return dict.release();
}

// x, w_gate, w_up, w_down, bits, had_block, trust_factor, buffers
PyObject *mlp_fwd(PyObject *const *a) {
    const at::Tensor &x = matrix(a[0]), &wg = matrix(a[1]), &wu = matrix(a[2]), &wd = matrix(a[3]);
    const int64_t T = x.size(0), H = x.size(1), I = wg.size(0);
    for (const at::Tensor *t : {&x, &wg, &wu, &wd})
        if (!t->is_contiguous() || t->scalar_type() != x.scalar_type()) throw NotPlain();
    if (wg.size(1) != H || wu.size(0) != I || wu.size(1) != H || wd.size(0) != H || wd.size(1) != I) throw NotPlain();
    const int bits = bits_arg(a[4]);
    const int64_t g = int_arg(a[5]);
    const float trust = float_arg(a[6]);
    const int dt = code_of(x.scalar_type());
    if (!PyDict_CheckExact(a[7])) throw NotPlain();
    Named b{a[7], x.device()};
    quest_mlp_saved sv;
    sv.xq = (uint8_t *)b.at(k_xq); sv.sx = (float *)b.at(k_sx); sv.mx = (uint8_t *)b.at(k_mx);
    sv.wgq = (uint8_t *)b.at(k_wgq); sv.swg = (float *)b.at(k_swg); sv.mwg = (uint8_t *)b.at(k_mwg);
    sv.wuq = (uint8_t *)b.at(k_wuq); sv.swu = (float *)b.at(k_swu); sv.mwu = (uint8_t *)b.at(k_mwu);
    sv.hq = (uint8_t *)b.at(k_hq); sv.sh = (float *)b.at(k_sh); sv.mh = (uint8_t *)b.at(k_mh);
    sv.wdq = (uint8_t *)b.at(k_wdq); sv.swd = (float *)b.at(k_swd); sv.mwd = (uint8_t *)b.at(k_mwd);
    const at::Tensor &h = plain_tensor(b.get(k_h), false), &y = plain_tensor(b.get(k_y), false), &ws = plain_tensor(b.get(k_workspace), false);
    const int ydt = code_of(y.scalar_type());
    void *st = stream();
    const int s = unlocked([&] {
        return quest_mlp_fwd(x.data_ptr(), wg.data_ptr(), wu.data_ptr(), wd.data_ptr(), dt, T, H, I, bits, (int)g, trust,
                             h.data_ptr(), y.data_ptr(), ydt, &sv, ws.data_ptr(), (size_t)ws.numel(), st);
    });
    if (s) return PyLong_FromLong(s);
    Py_INCREF(a[7]);
    return a[7];
}

// QUEST_BINDING: the module's name (build.py: it carries the version of torch)
#define QUEST_STRING_(X) #X
#define QUEST_STRING(X) QUEST_STRING_(X)
#define QUEST_INIT_(X) PyInit_##X
#define QUEST_INIT(X) QUEST_INIT_(X)
#define QUEST_METHOD(NAME, N) {#NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<NAME, N>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    QUEST_METHOD(quantize, 8), QUEST_METHOD(lowbit_gemm, 13), QUEST_METHOD(linear_fwd, 11), QUEST_METHOD(linear_bwd, 11),
    QUEST_METHOD(linear_fwd_fp4, 7), QUEST_METHOD(linear_fwd_weight_only, 8), QUEST_METHOD(mlp_fwd, 8),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, QUEST_STRING(QUEST_BINDING), nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC QUEST_INIT(QUEST_BINDING)(void) {
#define QUEST_KEY_INTERN(name) if (!(k_##name = PyUnicode_InternFromString(#name))) return nullptr;
    QUEST_KEYS(QUEST_KEY_INTERN)
    return PyModule_Create(&module_def);
}
