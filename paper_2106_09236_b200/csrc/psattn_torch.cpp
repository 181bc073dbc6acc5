// Native side of the Python binding: one object per plan whose methods take torch tensors, allocate the outputs that the
// caller left out, and call the C entry points on the current stream.  It marshals arguments and computes nothing.
//
// Why it exists: the small calls are bound by the host.  Marshalled in Python (ctypes objects for eight pointers, two
// torch.empty, the stream object) one psattn_forward kept a core busy for 15-19 us, longer than the kernel of a short
// utterance runs; here the same call is a few microseconds, most of it the launch.
//
// The addresses of the C entry points come from the caller (bind), so whichever build of the library the binding has
// loaded is the one that runs, and this module links against nothing of it.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/zeros.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

#ifdef PSATTN_BUILT_FOR
// read back from the file by build.py: a module compiled against another torch or Python is built again, not loaded
extern "C" __attribute__((used)) const char psattn_built_for[] = PSATTN_BUILT_FOR;
#endif

namespace {

typedef int (*fn_forward)(void *, const void *, const void *, const void *, const void *, const void *, void *, void *,
                          void *, void *, size_t, void *);
typedef int (*fn_reuse)(void *, const void *, const void *, const void *, const void *, const void *, void *, void *,
                        size_t, void *);
typedef int (*fn_measure)(void *, const void *, const void *, const void *, const void *, void *, void *, size_t, void *);
typedef int (*fn_exact)(void *, const void *, const void *, const void *, void *, void *, size_t, void *);
typedef int (*fn_qkv)(void *, const void *, const void *, int32_t, const void *, void *, void *, void *, void *, void *,
                      size_t, void *);
typedef int (*fn_out)(void *, const void *, const void *, const void *, const void *, int32_t, void *, void *, size_t,
                      void *);
typedef int (*fn_select)(void *, const void *, const void *, void *, void *, size_t, void *);      // also mean_v
typedef int (*fn_rows)(void *, const void *, const void *, const void *, const void *, const void *, int32_t, void *,
                       void *, size_t, void *);
typedef int (*fn_dense)(void *, const void *, const void *, const void *, const void *, void *, void *, size_t, void *);

enum Entry { kForward, kReuse, kMeasure, kExact, kQkv, kQkvZeroed, kOut, kOutZeroed, kSelect, kMeanV, kRows, kDense, kEntries };
void *g_entry[kEntries];
PyObject *g_check;                       // binding._check(rc, handle): raises

struct Caller {
    PyObject_HEAD
    void *plan, *ws;
    size_t ws_bytes;
    int64_t B, H, T, D, u_max;
    int bf16;
};

// The address behind an argument: None is a null pointer, a tensor its data, anything else is asked for data_ptr().
bool address(PyObject *o, void **out) {
    if (o == Py_None) { *out = nullptr; return true; }
    if (THPVariable_Check(o)) { *out = THPVariable_Unpack(o).data_ptr(); return true; }
    PyObject *r = PyObject_CallMethod(o, "data_ptr", nullptr);
    if (!r) return false;
    *out = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return !PyErr_Occurred();
}

bool device_of(PyObject *o, c10::Device *out) {
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a torch tensor"); return false; }
    *out = THPVariable_Unpack(o).device();
    return true;
}

// A new tensor for an output that the caller left out (new reference), or the caller's own.
PyObject *output(PyObject *given, c10::IntArrayRef shape, c10::ScalarType type, c10::Device dev, bool zero = false) {
    if (given != Py_None) { Py_INCREF(given); return given; }
    const auto opt = at::TensorOptions().dtype(type).device(dev);
    return THPVariable_Wrap(zero ? at::zeros(shape, opt) : at::empty(shape, opt));
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

bool failed(Caller *c, int rc) {
    if (rc == 0) return false;
    PyObject *h = c->plan ? PyLong_FromVoidPtr(c->plan) : Py_NewRef(Py_None);
    PyObject *r = PyObject_CallFunction(g_check, "iO", rc, h);
    Py_XDECREF(h);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "psattn call failed");
    return true;
}

bool count_is(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

// Owned references that are dropped on every way out of a method.
struct Ref {
    PyObject *p;
    explicit Ref(PyObject *x = nullptr) : p(x) {}
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref &) = delete;
    PyObject *give() { PyObject *x = p; p = nullptr; return x; }
};

#define PSATTN_CALL(type, entry, ...)                                                      \
    Py_BEGIN_ALLOW_THREADS                                                                 \
    rc = ((type)g_entry[entry])(__VA_ARGS__);                                              \
    Py_END_ALLOW_THREADS

c10::ScalarType element(const Caller *c) { return c->bf16 ? c10::kBFloat16 : c10::kFloat; }

#define PSATTN_METHOD(name, nargs) \
    PyObject *name(PyObject *self, PyObject *const *a, Py_ssize_t n) { \
        Caller *c = reinterpret_cast<Caller *>(self);                  \
        if (!count_is(n, nargs)) return nullptr;                       \
        HANDLE_TH_ERRORS                                               \
        int rc;                                                        \
        c10::Device dev(c10::kCPU);
#define PSATTN_METHOD_END \
        END_HANDLE_TH_ERRORS \
    }
// The first `count` arguments as addresses p[0..count).
#define PSATTN_POINTERS(count)                             \
        void *p[count];                                    \
        for (int k = 0; k < (count); ++k)                  \
            if (!address(a[k], &p[k])) return nullptr;

// forward(Q, K, V, lengths, sample_idx, O, sel_idx, M_out) -> (O, sel_idx)
PSATTN_METHOD(caller_forward, 8)
    PSATTN_POINTERS(5)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref O(output(a[5], {c->B, c->H, c->T, c->D}, element(c), dev));
    Ref S(output(a[6], {c->B, c->H, c->u_max}, c10::kInt, dev));
    void *o, *s, *m;
    if (!O.p || !S.p || !address(O.p, &o) || !address(S.p, &s) || !address(a[7], &m)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_forward, kForward, c->plan, p[0], p[1], p[2], p[3], p[4], o, s, m, c->ws, c->ws_bytes, st)
    if (failed(c, rc)) return nullptr;
    return PyTuple_Pack(2, O.p, S.p);
PSATTN_METHOD_END

// forward_with_selection(Q, K, V, lengths, sel_idx_in, O) -> O
PSATTN_METHOD(caller_reuse, 6)
    PSATTN_POINTERS(5)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref O(output(a[5], {c->B, c->H, c->T, c->D}, element(c), dev));
    void *o;
    if (!O.p || !address(O.p, &o)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_reuse, kReuse, c->plan, p[0], p[1], p[2], p[3], p[4], o, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : O.give();
PSATTN_METHOD_END

// measure(Q, K, lengths, sample_idx, M_out) -> M_out
PSATTN_METHOD(caller_measure, 5)
    PSATTN_POINTERS(4)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref M(output(a[4], {c->B, c->H, c->T}, c10::kFloat, dev));
    void *m;
    if (!M.p || !address(M.p, &m)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_measure, kMeasure, c->plan, p[0], p[1], p[2], p[3], m, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : M.give();
PSATTN_METHOD_END

// exact_measure(Q, K, lengths, M_out) -> M_out
PSATTN_METHOD(caller_exact, 4)
    PSATTN_POINTERS(3)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref M(output(a[3], {c->B, c->H, c->T}, c10::kFloat, dev));
    void *m;
    if (!M.p || !address(M.p, &m)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_exact, kExact, c->plan, p[0], p[1], p[2], m, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : M.give();
PSATTN_METHOD_END

// project_qkv(X, Wt, d_x, lengths, Q, K, V, vbar) -> (Q, K, V).  A caller that leaves out all three outputs gets
// tensors whose padded rows are zero; the call writes these zeros itself, so that no pass over the outputs precedes it.
PSATTN_METHOD(caller_qkv, 8)
    void *x, *w, *len, *vb, *q, *k, *v;
    if (!address(a[0], &x) || !address(a[1], &w) || !address(a[3], &len) || !address(a[7], &vb)) return nullptr;
    const long dx = PyLong_AsLong(a[2]);
    if (dx == -1 && PyErr_Occurred()) return nullptr;
    if (!device_of(a[0], &dev)) return nullptr;
    const bool fresh = a[4] == Py_None && a[5] == Py_None && a[6] == Py_None;
    const int64_t shape[4] = {c->B, c->H, c->T, c->D};
    Ref Q(output(a[4], shape, element(c), dev, !fresh)), K(output(a[5], shape, element(c), dev, !fresh)),
        V(output(a[6], shape, element(c), dev, !fresh));
    if (!Q.p || !K.p || !V.p || !address(Q.p, &q) || !address(K.p, &k) || !address(V.p, &v)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_qkv, fresh ? kQkvZeroed : kQkv, c->plan, x, w, (int32_t)dx, len, q, k, v, vb, c->ws, c->ws_bytes, st)
    if (failed(c, rc)) return nullptr;
    return PyTuple_Pack(3, Q.p, K.p, V.p);
PSATTN_METHOD_END

// project_out(O, sel_idx, lengths, Wot, d_y, Y) -> Y; a Y left out has zeros in its padded rows, as above
PSATTN_METHOD(caller_out, 6)
    PSATTN_POINTERS(4)
    const long dy = PyLong_AsLong(a[4]);
    if (dy == -1 && PyErr_Occurred()) return nullptr;
    if (!device_of(a[0], &dev)) return nullptr;
    const bool fresh = a[5] == Py_None;
    Ref Y(output(a[5], {c->B, c->T, (int64_t)dy}, element(c), dev));
    void *y;
    if (!Y.p || !address(Y.p, &y)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_out, fresh ? kOutZeroed : kOut, c->plan, p[0], p[1], p[2], p[3], (int32_t)dy, y, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : Y.give();
PSATTN_METHOD_END

// select(M, lengths, sel_idx) -> sel_idx
PSATTN_METHOD(caller_select, 3)
    PSATTN_POINTERS(2)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref S(output(a[2], {c->B, c->H, c->u_max}, c10::kInt, dev));
    void *s;
    if (!S.p || !address(S.p, &s)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_select, kSelect, c->plan, p[0], p[1], s, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : S.give();
PSATTN_METHOD_END

// mean_v(V, lengths, vbar) -> vbar
PSATTN_METHOD(caller_mean_v, 3)
    PSATTN_POINTERS(2)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref S(output(a[2], {c->B, c->H, c->D}, c10::kFloat, dev));
    void *s;
    if (!S.p || !address(S.p, &s)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_select, kMeanV, c->plan, p[0], p[1], s, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : S.give();
PSATTN_METHOD_END

// attend_rows(Q, K, V, lengths, row_idx, n_rows, out) -> out
PSATTN_METHOD(caller_rows, 7)
    PSATTN_POINTERS(5)
    const long rows = PyLong_AsLong(a[5]);
    if (rows == -1 && PyErr_Occurred()) return nullptr;
    if (!device_of(a[0], &dev)) return nullptr;
    Ref O(output(a[6], {c->B, c->H, (int64_t)rows, c->D}, c10::kFloat, dev));
    void *o;
    if (!O.p || !address(O.p, &o)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_rows, kRows, c->plan, p[0], p[1], p[2], p[3], p[4], (int32_t)rows, o, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : O.give();
PSATTN_METHOD_END

// dense_forward(Q, K, V, lengths, O) -> O
PSATTN_METHOD(caller_dense, 5)
    PSATTN_POINTERS(4)
    if (!device_of(a[0], &dev)) return nullptr;
    Ref O(output(a[4], {c->B, c->H, c->T, c->D}, element(c), dev));
    void *o;
    if (!O.p || !address(O.p, &o)) return nullptr;
    void *st = stream();
    PSATTN_CALL(fn_dense, kDense, c->plan, p[0], p[1], p[2], p[3], o, c->ws, c->ws_bytes, st)
    return failed(c, rc) ? nullptr : O.give();
PSATTN_METHOD_END

// close(): the plan is gone; later calls get the library's null-pointer status
PyObject *caller_close(PyObject *self, PyObject *) {
    reinterpret_cast<Caller *>(self)->plan = nullptr;
    Py_RETURN_NONE;
}

// set_workspace(address, bytes)
PyObject *caller_set_workspace(PyObject *self, PyObject *args) {
    unsigned long long ws, bytes;
    if (!PyArg_ParseTuple(args, "KK", &ws, &bytes)) return nullptr;
    reinterpret_cast<Caller *>(self)->ws = (void *)(uintptr_t)ws;
    reinterpret_cast<Caller *>(self)->ws_bytes = (size_t)bytes;
    Py_RETURN_NONE;
}

#define PSATTN_FAST(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, nullptr}
PyMethodDef caller_methods[] = {
    PSATTN_FAST("forward", caller_forward), PSATTN_FAST("forward_with_selection", caller_reuse),
    PSATTN_FAST("measure", caller_measure), PSATTN_FAST("exact_measure", caller_exact),
    PSATTN_FAST("project_qkv", caller_qkv), PSATTN_FAST("project_out", caller_out),
    PSATTN_FAST("select", caller_select), PSATTN_FAST("mean_v", caller_mean_v),
    PSATTN_FAST("attend_rows", caller_rows), PSATTN_FAST("dense_forward", caller_dense),
    {"set_workspace", caller_set_workspace, METH_VARARGS, nullptr}, {"close", caller_close, METH_NOARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};

// Caller(plan, workspace, workspace_bytes, B, H, T_max, d_head, u_max, bf16): addresses and sizes as integers
int caller_init(PyObject *self, PyObject *args, PyObject *) {
    Caller *c = reinterpret_cast<Caller *>(self);
    unsigned long long plan, ws, bytes;
    long long B, H, T, D, u;
    int bf16;
    if (!PyArg_ParseTuple(args, "KKKLLLLLi", &plan, &ws, &bytes, &B, &H, &T, &D, &u, &bf16)) return -1;
    c->plan = (void *)(uintptr_t)plan; c->ws = (void *)(uintptr_t)ws; c->ws_bytes = (size_t)bytes;
    c->B = B; c->H = H; c->T = T; c->D = D; c->u_max = u; c->bf16 = bf16;
    return 0;
}

PyTypeObject caller_type = {PyVarObject_HEAD_INIT(nullptr, 0)};

// bind(check, addresses): `addresses` holds kEntries integers in the order of Entry
PyObject *bind(PyObject *, PyObject *args) {
    PyObject *check, *list;
    if (!PyArg_ParseTuple(args, "OO!", &check, &PyTuple_Type, &list)) return nullptr;
    if (!count_is(PyTuple_GET_SIZE(list), kEntries)) return nullptr;
    for (int k = 0; k < kEntries; ++k) {
        g_entry[k] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(list, k));
        if (PyErr_Occurred()) return nullptr;
    }
    Py_XSETREF(g_check, Py_NewRef(check));
    Py_RETURN_NONE;
}

PyMethodDef module_methods[] = {{"bind", bind, METH_VARARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "psattn_torch", nullptr, -1, module_methods};

}  // namespace

PyMODINIT_FUNC PyInit_psattn_torch(void) {
    caller_type.tp_name = "psattn_torch.Caller";
    caller_type.tp_basicsize = sizeof(Caller);
    caller_type.tp_flags = Py_TPFLAGS_DEFAULT;
    caller_type.tp_new = PyType_GenericNew;
    caller_type.tp_init = caller_init;
    caller_type.tp_methods = caller_methods;
    if (PyType_Ready(&caller_type) < 0) return nullptr;
    PyObject *m = PyModule_Create(&module_def);
    if (!m || PyModule_AddObjectRef(m, "Caller", reinterpret_cast<PyObject *>(&caller_type)) < 0) return nullptr;
    return m;
}
