// CPython binding of libssd (include/ssd.h) for torch tensors: the argument checks, output and scratch allocation and
// pointer extraction of libssd.py's wrappers, in native code.  A decode step is a few microseconds of kernel: marshalled
// through ctypes its host side took 15 us per call and set the pace of a generation loop.
//
// Every function takes positional arguments (None where the Python wrapper has None), launches on the given stream or,
// for None, on the current one, and returns its tensors; a negative SSD_* code of the library comes back as an int, for
// the wrapper to raise.
#include <ATen/ATen.h>
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "ssd.h"

namespace {

// Raised as the Python exception it names; anything torch throws is translated by HANDLE_TH_ERRORS.
struct PyError {
    PyObject *type;
    const char *msg;
};

const at::Tensor &tensor(PyObject *o) {
    if (!THPVariable_Check(o)) throw PyError{PyExc_TypeError, "a torch tensor is required"};
    return THPVariable_Unpack(o);
}
void *ptr(PyObject *o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
float *fptr(PyObject *o) { return (float *)ptr(o); }
long long num(PyObject *o) {
    if (PyFloat_Check(o)) return (long long)PyFloat_AS_DOUBLE(o);
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
}
void *stream_of(PyObject *o) {
    if (o == Py_None) return (void *)c10::cuda::getCurrentCUDAStream().stream();
    PyObject *v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw python_error();
    void *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!p && PyErr_Occurred()) throw python_error();
    return p;
}
int dtype_code(const at::Tensor &t, const char *msg) {
    if (t.scalar_type() == at::kBFloat16) return SSD_DTYPE_BF16;
    if (t.scalar_type() == at::kFloat) return SSD_DTYPE_F32;
    throw PyError{PyExc_TypeError, msg};
}
void require(bool ok, PyObject *type, const char *msg) {
    if (!ok) throw PyError{type, msg};
}
at::Tensor f32_like(const at::Tensor &ref, at::IntArrayRef sizes) { return at::empty(sizes, ref.options().dtype(at::kFloat)); }
at::Tensor bytes(const at::Tensor &ref, size_t n) { return at::empty({(int64_t)n}, ref.options().dtype(at::kByte)); }
size_t nbytes(const at::Tensor &ws) { return (size_t)ws.numel() * ws.element_size(); }
// the caller's tensor as it is, or a new one
template <typename F> PyObject *given_or(PyObject *o, F make) {
    if (o == Py_None) return THPVariable_Wrap(make());
    tensor(o);
    Py_INCREF(o);
    return o;
}

template <typename F> PyObject *guarded(Py_ssize_t n, Py_ssize_t want, F body) {
    HANDLE_TH_ERRORS
    try {
        require(n == want, PyExc_TypeError, "wrong number of arguments");
        return body();
    } catch (const PyError &e) {
        PyErr_SetString(e.type, e.msg);
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// The library call itself, without the interpreter lock (its arguments are read from the Python objects before).
template <typename... P, typename... A> int unlocked(int (*call)(P...), A... args) {
    PyThreadState *ts = PyEval_SaveThread();
    const int rc = call(args...);
    PyEval_RestoreThread(ts);
    return rc;
}

// Owned references of a function's results, released if it throws or returns an error code.
struct Results {
    PyObject *r[8];
    int n = 0;
    PyObject *add(PyObject *o) {
        if (!o) throw python_error();
        return r[n++] = o;
    }
    ~Results() {
        for (int i = 0; i < n; ++i) Py_DECREF(r[i]);
    }
    PyObject *tuple() {
        PyObject *t = PyTuple_New(n);
        if (!t) throw python_error();
        for (int i = 0; i < n; ++i) PyTuple_SET_ITEM(t, i, r[i]);
        n = 0;
        return t;
    }
};

// ---- decode_step(x, dt, A, Bm, Cm, D, h, y, stream): y
PyObject *decode_step(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 9, [&]() -> PyObject * {
        at::Tensor x = tensor(a[0]), dt = tensor(a[1]), Bm = tensor(a[3]), Cm = tensor(a[4]);
        const at::Tensor &h = tensor(a[6]);
        require(x.is_cuda() && h.is_cuda(), PyExc_ValueError, "device tensors required");
        static const char *const kToken = "ssd_decode_step takes one token: x [B,1,H,P], dt [B,1,H], Bm/Cm [B,1,G,N]";
        require(x.dim() == 4 && Bm.dim() == 4, PyExc_ValueError, kToken);
        const int64_t B = x.size(0), H = x.size(2), P = x.size(3), G = Bm.size(2), N = Bm.size(3);
        require(x.size(1) == 1 && dt.dim() == 3 && dt.size(0) == B && dt.size(1) == 1 && dt.size(2) == H && Cm.sizes() == Bm.sizes() &&
                    Bm.size(0) == B && Bm.size(1) == 1,
                PyExc_ValueError, kToken);
        require(h.dim() == 4 && h.size(0) == B && h.size(1) == H && h.size(2) == P && h.size(3) == N && h.scalar_type() == at::kFloat &&
                    h.is_contiguous(),
                PyExc_ValueError, "h must be a contiguous float32 [B,H,P,N] tensor");
        static const char *const kDtype = "x, Bm, Cm must share dtype float32 or bfloat16";
        const int code = dtype_code(x, kDtype);
        require(Bm.scalar_type() == x.scalar_type() && Cm.scalar_type() == x.scalar_type(), PyExc_TypeError, kDtype);
        // one-token slices of longer tensors are made dense here (a few KB); the C call also takes batch strides
        if (!x.is_contiguous()) x = x.contiguous();
        if (!dt.is_contiguous()) dt = dt.contiguous();
        if (!Bm.is_contiguous()) Bm = Bm.contiguous();
        if (!Cm.is_contiguous()) Cm = Cm.contiguous();
        Results out;
        PyObject *y = out.add(given_or(a[7], [&] { return at::empty({B, 1, H, P}, x.options()); }));
        const at::Tensor &yt = tensor(y);
        require(yt.is_contiguous() && yt.sizes() == x.sizes() && yt.scalar_type() == x.scalar_type(), PyExc_ValueError,
                "y must be a dense tensor like x");
        ssd_shape_t s = {(int32_t)B, 1, (int32_t)H, (int32_t)P, (int32_t)N, (int32_t)G, 0, 0, code, 0, 0, 0, 0};
        const int rc = unlocked(ssd_decode_step, &s, x.data_ptr(), (const float *)dt.data_ptr(), fptr(a[2]), Bm.data_ptr(), Cm.data_ptr(), fptr(a[5]),
                                       (float *)h.data_ptr(), yt.data_ptr(), stream_of(a[8]));
        if (rc) return PyLong_FromLong(rc);
        Py_INCREF(y);
        return y;
    });
}

// ---- the layer calls share the checks of x, dt, A, Bm, Cm, D and the shape
ssd_shape_t layer_shape(PyObject *const *a, PyObject *chunk, PyObject *seg, PyObject *flags) {
    static const char *const kMsg[6] = {"x must be a contiguous CUDA tensor", "dt must be a contiguous CUDA tensor",
                                        "A must be a contiguous CUDA tensor", "Bm must be a contiguous CUDA tensor",
                                        "Cm must be a contiguous CUDA tensor", "D must be a contiguous CUDA tensor"};
    for (int i = 0; i < 6; ++i) {
        const at::Tensor &t = tensor(a[i]);
        require(t.is_cuda() && t.is_contiguous(), PyExc_ValueError, kMsg[i]);
    }
    const at::Tensor &x = tensor(a[0]), &Bm = tensor(a[3]);
    require(tensor(a[1]).scalar_type() == at::kFloat && tensor(a[2]).scalar_type() == at::kFloat && tensor(a[5]).scalar_type() == at::kFloat,
            PyExc_TypeError, "dt, A, D must be float32");
    require(Bm.scalar_type() == x.scalar_type() && tensor(a[4]).scalar_type() == x.scalar_type(), PyExc_TypeError,
            "Bm, Cm must have the dtype of x");
    require(x.dim() == 4 && Bm.dim() == 4, PyExc_ValueError, "x must be [B,L,H,P] and Bm [B,L,G,N]");
    return ssd_shape_t{(int32_t)x.size(0), (int32_t)x.size(1), (int32_t)x.size(2), (int32_t)x.size(3), (int32_t)Bm.size(3),
                       (int32_t)Bm.size(2), (int32_t)num(chunk), (int32_t)num(seg), dtype_code(x, "x must be float32 or bfloat16"),
                       (int32_t)num(flags), 0, 0, 0};
}

// ---- fwd(x, dt, A, Bm, Cm, D, h0, chunk, seg, flags, y, h_final, boundary, ws, stream): y, h_final[, boundary]
//      boundary == False: ssd_fwd; None or a tensor: ssd_fwd_segmented
PyObject *fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 15, [&]() -> PyObject * {
        const ssd_shape_t s = layer_shape(a, a[7], a[8], a[9]);
        const bool seg = a[12] != Py_False;
        const at::Tensor &x = tensor(a[0]);
        Results out;
        PyObject *y = out.add(given_or(a[10], [&] { return at::empty_like(x); }));
        PyObject *hf = out.add(given_or(a[11], [&] { return f32_like(x, {s.B, s.H, s.P, s.N}); }));
        PyObject *bd = nullptr;
        if (seg) {
            const size_t nb = a[12] == Py_None ? ssd_boundary_bytes(&s) : 1;
            if (!nb) return PyLong_FromLong(SSD_EINVAL);
            bd = out.add(given_or(a[12], [&] { return f32_like(x, {s.B, (int64_t)(nb / (4ull * s.B * s.H * s.P * s.N)), s.H, s.P, s.N}); }));
        }
        const size_t need = a[13] == Py_None ? ssd_workspace_bytes(&s, seg ? SSD_OP_FWD_SEG : SSD_OP_FWD) : 1;
        if (!need) return PyLong_FromLong(SSD_EINVAL);
        const at::Tensor ws = a[13] == Py_None ? bytes(x, need) : tensor(a[13]);
        void *st = stream_of(a[14]);
        const int rc = seg ? unlocked(ssd_fwd_segmented, &s, x.data_ptr(), fptr(a[1]), fptr(a[2]), ptr(a[3]), ptr(a[4]), fptr(a[5]), fptr(a[6]), ptr(y), fptr(hf),
                                               fptr(bd), ws.data_ptr(), nbytes(ws), st)
                           : unlocked(ssd_fwd, &s, x.data_ptr(), fptr(a[1]), fptr(a[2]), ptr(a[3]), ptr(a[4]), fptr(a[5]), fptr(a[6]), ptr(y), fptr(hf),
                                     ws.data_ptr(), nbytes(ws), st);
        if (rc) return PyLong_FromLong(rc);
        return out.tuple();
    });
}

// ---- bwd(x, dt, A, Bm, Cm, D, boundary, dy, dh_final, chunk, seg, flags, dx, ddt, dA, dB, dC, dD, dh0, ws, stream): 0
PyObject *bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 21, [&]() -> PyObject * {
        const ssd_shape_t s = layer_shape(a, a[9], a[10], a[11]);
        const at::Tensor &x = tensor(a[0]);
        const size_t need = a[19] == Py_None ? ssd_workspace_bytes(&s, SSD_OP_BWD_SEG) : 1;
        if (!need) return PyLong_FromLong(SSD_EINVAL);
        const at::Tensor ws = a[19] == Py_None ? bytes(x, need) : tensor(a[19]);
        return PyLong_FromLong(unlocked(ssd_bwd_segmented, &s, x.data_ptr(), fptr(a[1]), fptr(a[2]), ptr(a[3]), ptr(a[4]), fptr(a[5]), fptr(a[6]), ptr(a[7]),
                                                 fptr(a[8]), ptr(a[12]), fptr(a[13]), fptr(a[14]), ptr(a[15]), ptr(a[16]), fptr(a[17]), fptr(a[18]),
                                                 ws.data_ptr(), nbytes(ws), stream_of(a[20])));
    });
}

struct ConvArgs {
    int B, L, C, code;
    long long bs;
};
ConvArgs conv_args(const at::Tensor &u) {
    const int code = dtype_code(u, "u must be float32 or bfloat16");
    require(u.is_cuda() && u.dim() == 3 && u.stride(2) == 1 && u.stride(1) == u.size(2), PyExc_ValueError,
            "u must be a CUDA tensor [B, L, C] with contiguous rows");
    return ConvArgs{(int)u.size(0), (int)u.size(1), (int)u.size(2), code, u.size(0) > 1 ? (long long)u.stride(0) : 0ll};
}

// ---- conv_fwd(u, w, bias, state_in, out, state_out, stream): out, state_out
PyObject *conv_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&]() -> PyObject * {
        const at::Tensor &u = tensor(a[0]);
        const ConvArgs c = conv_args(u);
        Results out;
        PyObject *o = out.add(given_or(a[4], [&] { return at::empty_like(u); }));
        PyObject *so = out.add(given_or(a[5], [&] { return at::empty({c.B, 3, c.C}, u.options()); }));
        const int rc = unlocked(ssd_conv_fwd, c.B, c.L, c.C, c.code, u.data_ptr(), c.bs, fptr(a[1]), fptr(a[2]), ptr(a[3]), ptr(o), ptr(so), stream_of(a[6]));
        if (rc) return PyLong_FromLong(rc);
        return out.tuple();
    });
}

// ---- conv_bwd(u, w, bias, state_in, dout, dtail, du, dstate, dw, dbias, accumulate, ws, stream): du, dstate, dw, dbias
PyObject *conv_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 13, [&]() -> PyObject * {
        const at::Tensor &u = tensor(a[0]);
        const ConvArgs c = conv_args(u);
        const auto f32 = u.options().dtype(at::kFloat);
        Results out;
        PyObject *du = out.add(given_or(a[6], [&] { return at::empty_like(u); }));
        PyObject *ds = out.add(given_or(a[7], [&] { return at::empty({c.B, 3, c.C}, f32); }));
        PyObject *dw = out.add(given_or(a[8], [&] { return at::zeros({c.C, 4}, f32); }));
        PyObject *db = out.add(given_or(a[9], [&] { return at::zeros({c.C}, f32); }));
        const at::Tensor ws = a[11] == Py_None ? bytes(u, ssd_conv_workspace_bytes(c.B, c.L, c.C)) : tensor(a[11]);
        const int rc = unlocked(ssd_conv_bwd, c.B, c.L, c.C, c.code, u.data_ptr(), c.bs, fptr(a[1]), fptr(a[2]), ptr(a[3]), ptr(a[4]), fptr(a[5]), ptr(du),
                                    fptr(ds), fptr(dw), fptr(db), PyObject_IsTrue(a[10]), ws.data_ptr(), nbytes(ws), stream_of(a[12]));
        if (rc) return PyLong_FromLong(rc);
        return out.tuple();
    });
}

struct NormArgs {
    long long rows;
    int D, group, code;
};
NormArgs norm_args(const at::Tensor &y, PyObject *group) {
    const int code = dtype_code(y, "y must be float32 or bfloat16");
    require(y.is_cuda() && y.dim() > 0 && y.is_contiguous(), PyExc_ValueError, "y must be a contiguous CUDA tensor [..., D]");
    const long long D = y.size(-1);
    return NormArgs{D ? (long long)y.numel() / D : 0, (int)D, group == Py_None ? (int)D : (int)num(group), code};
}
float real(PyObject *o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw python_error();
    return (float)v;
}

// ---- gated_norm_fwd(y, z, gamma, group, eps, out, stream): out
PyObject *gated_norm_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&]() -> PyObject * {
        const at::Tensor &y = tensor(a[0]);
        const NormArgs c = norm_args(y, a[3]);
        Results out;
        PyObject *o = out.add(given_or(a[5], [&] { return at::empty_like(y); }));
        const int rc = unlocked(ssd_gated_norm_fwd, c.rows, c.D, c.group, c.code, y.data_ptr(), ptr(a[1]), fptr(a[2]), real(a[4]), ptr(o), stream_of(a[6]));
        if (rc) return PyLong_FromLong(rc);
        Py_INCREF(o);
        return o;
    });
}

// ---- gated_norm_bwd(y, z, gamma, dout, group, eps, dy, dz, dgamma, accumulate, ws, stream): dy, dz, dgamma
PyObject *gated_norm_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 12, [&]() -> PyObject * {
        const at::Tensor &y = tensor(a[0]);
        const NormArgs c = norm_args(y, a[4]);
        Results out;
        PyObject *dy = out.add(given_or(a[6], [&] { return at::empty_like(y); }));
        PyObject *dz = out.add(given_or(a[7], [&] { return at::empty_like(y); }));
        PyObject *dg = out.add(given_or(a[8], [&] { return at::zeros({c.D}, y.options().dtype(at::kFloat)); }));
        const at::Tensor ws = a[10] == Py_None ? bytes(y, ssd_gated_norm_workspace_bytes(c.rows, c.D)) : tensor(a[10]);
        const int rc = unlocked(ssd_gated_norm_bwd, c.rows, c.D, c.group, c.code, y.data_ptr(), ptr(a[1]), fptr(a[2]), real(a[5]), ptr(a[3]), ptr(dy), ptr(dz),
                                          fptr(dg), PyObject_IsTrue(a[9]), ws.data_ptr(), nbytes(ws), stream_of(a[11]));
        if (rc) return PyLong_FromLong(rc);
        return out.tuple();
    });
}

ssd_shape_t glue_shape(const at::Tensor &t) {
    const int code = dtype_code(t, "tensor must be float32 or bfloat16");
    require(t.is_cuda() && t.dim() == 4 && t.is_contiguous(), PyExc_ValueError, "tensor must be a contiguous CUDA tensor");
    return ssd_shape_t{(int32_t)t.size(0), (int32_t)t.size(1), (int32_t)t.size(2), (int32_t)t.size(3), 1, 1, 64, 0, code, 0, 0, 0, 0};
}

// ---- glue_fwd(x, y, W, x_next, stream), glue_bwd(g_next, W, dz, stream): 0
PyObject *glue_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 5, [&]() -> PyObject * {
        const ssd_shape_t s = glue_shape(tensor(a[0]));
        return PyLong_FromLong(unlocked(ssd_glue_fwd, &s, ptr(a[0]), ptr(a[1]), fptr(a[2]), ptr(a[3]), stream_of(a[4])));
    });
}
PyObject *glue_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 4, [&]() -> PyObject * {
        const ssd_shape_t s = glue_shape(tensor(a[0]));
        return PyLong_FromLong(unlocked(ssd_glue_bwd, &s, ptr(a[0]), fptr(a[1]), ptr(a[2]), stream_of(a[3])));
    });
}

#define SSD_METHOD(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SSD_METHOD(decode_step), SSD_METHOD(fwd), SSD_METHOD(bwd), SSD_METHOD(conv_fwd), SSD_METHOD(conv_bwd),
                         SSD_METHOD(gated_norm_fwd), SSD_METHOD(gated_norm_bwd), SSD_METHOD(glue_fwd), SSD_METHOD(glue_bwd),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module_def); }
