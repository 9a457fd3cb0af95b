// osd_binding.cpp -- the Python calls in native code.  Each function takes what the
// Python function of the same name takes, positionally, and either makes the C call
// and returns its result (or the status of a call that failed), or returns None,
// having done nothing, where an argument is not of the plain kind it handles: the
// Python code then checks the arguments itself and raises what is wrong with them.
//
// A call on small inputs is bound by the host: through ctypes, with every tensor
// property fetched as a Python object, one took 14 to 24 us of a Grace core (distill 13.9,
// verify 13.5 and with fresh results 23.6, tree 20.7), where the kernels behind it take
// 8 to 25.  Here distill and verify take 2.5 us, tree 2.7, verify with fresh results 7.2.
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

#include "osd.h"

namespace {

PyObject* g_verify_result = nullptr;    // VerifyResult, DistillAcceptedResult, TreeResult
PyObject* g_accepted_result = nullptr;
PyObject* g_tree_result = nullptr;
PyObject* g_cuda_stream = nullptr;      // "cuda_stream"

// The arguments of one call: every tensor a plain CUDA tensor (no subclass, no
// transform's wrapper, no mode that wants to see the call) on the current device.
struct Call {
    bool ok = true;
    int dev = -1;

    Call() { ok = !at::impl::torch_function_mode_enabled() && !c10::impl::TorchDispatchModeTLS::any_modes_set(); }

    const at::Tensor* tensor(PyObject* o) {
        if (!ok || !THPVariable_CheckExact(o)) return fail();
        const at::Tensor& t = THPVariable_Unpack(o);
        constexpr c10::DispatchKeySet wrappers(
            {c10::DispatchKey::Python, c10::DispatchKey::Functionalize, c10::DispatchKey::FuncTorchBatched,
             c10::DispatchKey::FuncTorchGradWrapper});
        if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage() || t.key_set().has_any(wrappers))
            return fail();
        const int d = t.device().index();
        if (dev < 0) {
            dev = d;
            if (c10::cuda::current_device() != d) return fail();
        }
        if (d != dev) return fail();
        for (int64_t n : t.sizes())
            if (n > INT_MAX) return fail();
        return &t;
    }
    const at::Tensor* optional(PyObject* o) { return o == Py_None ? nullptr : tensor(o); }
    const at::Tensor* fail() {
        ok = false;
        return nullptr;
    }
    bool need(bool cond) { return ok = ok && cond; }

    double number(PyObject* o) {
        if (!ok) return 0.0;
        if (PyFloat_CheckExact(o)) return PyFloat_AS_DOUBLE(o);
        if (!PyLong_CheckExact(o)) {
            ok = false;
            return 0.0;
        }
        const double v = PyLong_AsDouble(o);
        if (v == -1.0 && PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return v;
    }
    void* stream(PyObject* o) {
        if (!ok) return nullptr;
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(dev)).stream();
        PyObject* v = PyObject_GetAttr(o, g_cuda_stream);
        void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
        Py_XDECREF(v);
        if (PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return p;
    }
    int kind(PyObject* o) {
        if (!ok) return -1;
        if (PyLong_CheckExact(o)) {
            const long v = PyLong_AsLong(o);
            if ((v == -1 && PyErr_Occurred()) || v < INT_MIN || v > INT_MAX) {
                PyErr_Clear();
                ok = false;
            }
            return static_cast<int>(v);
        }
        static const char* const names[] = {"fkl", "rkl", "jsd", "tvd", "ce"};
        if (PyUnicode_CheckExact(o))
            for (int i = 0; i < 5; ++i)
                if (PyUnicode_CompareWithASCIIString(o, names[i]) == 0) return i;
        ok = false;
        return -1;
    }
    // an output the caller may have brought, by its place in a result tuple
    const at::Tensor* member(PyObject* out, Py_ssize_t i) { return ok ? optional(PyTuple_GET_ITEM(out, i)) : nullptr; }
};

int dtype_code(const at::Tensor& t) {
    return t.scalar_type() == at::kFloat ? OSD_F32 : (t.scalar_type() == at::kBFloat16 ? OSD_BF16 : -1);
}
bool shaped(const at::Tensor& t, at::IntArrayRef sizes) { return t.sizes() == sizes && t.is_contiguous(); }
void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
at::Tensor fresh(at::IntArrayRef sizes, at::ScalarType type, int dev) {
    return at::empty(sizes, at::TensorOptions().dtype(type).device(at::kCUDA, static_cast<c10::DeviceIndex>(dev)));
}
// A result tuple of class `cls` holding `n` tensors (undefined ones as None).
PyObject* result(PyObject* cls, const at::Tensor* ts, int n) {
    PyObject* items = PyTuple_New(n);
    if (!items) return nullptr;
    for (int i = 0; i < n; ++i) {
        PyObject* o = ts[i].defined() ? THPVariable_Wrap(ts[i]) : Py_NewRef(Py_None);
        if (!o) {
            Py_DECREF(items);
            return nullptr;
        }
        PyTuple_SET_ITEM(items, i, o);
    }
    if (!cls) return items;
    PyObject* args = PyTuple_Pack(1, items);
    Py_DECREF(items);
    if (!args) return nullptr;
    PyObject* r = PyTuple_Type.tp_new(reinterpret_cast<PyTypeObject*>(cls), args, nullptr);
    Py_DECREF(args);
    return r;
}
template <typename F>
osd_status released(F&& f) {
    osd_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return st;
}
// C++ exceptions (an allocation that fails) become the Python error of the slow path.
template <typename F>
PyObject* guarded(F&& f) {
    try {
        return f();
    } catch (const std::exception&) {
        Py_RETURN_NONE;
    }
}

// draft, target, tokens, uniforms, temperature, diagnostics, workspace, out, stream
PyObject* verify(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 9) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        Call c;
        const at::Tensor* target = c.tensor(a[1]);
        if (!c.ok || target->dim() != 3 || target->size(1) < 1) Py_RETURN_NONE;
        const int64_t B = target->size(0), k = target->size(1) - 1, V = target->size(2);
        const at::Tensor *draft = c.optional(a[0]), *tokens = c.tensor(a[2]), *uniforms = c.optional(a[3]);
        const int dt = dtype_code(*target);
        if (!c.need(dt >= 0 && target->is_contiguous())) Py_RETURN_NONE;
        if (draft) c.need(draft->scalar_type() == target->scalar_type() && shaped(*draft, {B, k, V}));
        c.need(tokens->scalar_type() == at::kInt && shaped(*tokens, {B, k}));
        if (uniforms) c.need(uniforms->scalar_type() == at::kFloat && shaped(*uniforms, {B, k + 1}));
        const double temperature = c.number(a[4]);
        const bool diagnostics = a[5] == Py_True;
        c.need(diagnostics || a[5] == Py_False);
        void* stream = c.stream(a[8]);
        size_t need = 0;
        if (!c.ok || osd_verify_workspace_size(int(B), int(k), int(V), &need) != OSD_OK) Py_RETURN_NONE;
        const at::Tensor* given = c.optional(a[6]);
        const at::Tensor* o[5] = {};
        at::Tensor made[5];
        const bool own = a[7] == Py_None;
        if (!own) {
            if (!c.need(Py_TYPE(a[7]) == reinterpret_cast<PyTypeObject*>(g_verify_result))) Py_RETURN_NONE;
            for (int i = 0; i < 5; ++i) o[i] = c.member(a[7], i);
        }
        if (!c.ok) Py_RETURN_NONE;
        at::Tensor ws;
        if (!given) {
            ws = fresh({int64_t(need)}, at::kByte, c.dev);
            given = &ws;
        }
        if (own) {
            made[0] = fresh({B}, at::kInt, c.dev);
            made[1] = fresh({B, k + 1}, at::kInt, c.dev);
            made[2] = fresh({B, k}, at::kByte, c.dev);
            if (diagnostics) {
                made[3] = fresh({B, k}, at::kFloat, c.dev);
                made[4] = fresh({B}, at::kFloat, c.dev);
            }
            for (int i = 0; i < 5; ++i) o[i] = made[i].defined() ? &made[i] : nullptr;
        }
        const void *zp = ptr(draft), *tp = ptr(target);
        const auto *yp = static_cast<const int32_t*>(ptr(tokens));
        const auto* up = static_cast<const float*>(ptr(uniforms));
        void* p[5];
        for (int i = 0; i < 5; ++i) p[i] = ptr(o[i]);
        void* wp = ptr(given);
        const size_t wbytes = size_t(given->numel()) * given->element_size();
        const osd_status st = released([&]() {
            return osd_verify(zp, tp, osd_dtype(dt), int(B), int(k), int(V), yp, up, float(temperature),
                              static_cast<int32_t*>(p[0]), static_cast<int32_t*>(p[1]), static_cast<uint8_t*>(p[2]),
                              static_cast<float*>(p[3]), static_cast<float*>(p[4]), wp, wbytes, stream);
        });
        if (st != OSD_OK) return PyLong_FromLong(st);
        return own ? result(g_verify_result, made, 5) : Py_NewRef(a[7]);
    });
}

// A [N, V] or [G, P, V] view with contiguous rows.
struct Rows {
    int64_t G, P, V, sg, sp;
    bool of(const at::Tensor& t) {
        if (t.dim() == 2) {
            G = t.size(0), P = 1, V = t.size(1), sg = t.stride(0), sp = 0;
        } else if (t.dim() == 3) {
            G = t.size(0), P = t.size(1), V = t.size(2), sg = t.stride(0), sp = t.stride(1);
        } else {
            return false;
        }
        return t.stride(-1) == 1;
    }
};

// draft, target, mask, kind, beta, temperature, loss, dlogits, status, stream
PyObject* distill(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 10) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        Call c;
        const at::Tensor *draft = c.tensor(a[0]), *target = c.tensor(a[1]);
        Rows d, t;
        if (!c.ok || !d.of(*draft) || !t.of(*target) || draft->sizes() != target->sizes()) Py_RETURN_NONE;
        const int dt = dtype_code(*draft);
        c.need(dt >= 0 && draft->scalar_type() == target->scalar_type());
        const at::Tensor *mask = c.optional(a[2]), *loss = c.optional(a[6]), *dlogits = c.optional(a[7]),
                         *status = c.optional(a[8]);
        const int kind = c.kind(a[3]);
        const double beta = c.number(a[4]), temperature = c.number(a[5]);
        void* stream = c.stream(a[9]);
        if (!c.ok) Py_RETURN_NONE;
        const at::IntArrayRef full = draft->sizes(), lead = full.slice(0, full.size() - 1);
        if (mask) c.need(mask->scalar_type() == at::kByte && shaped(*mask, lead));
        if (loss) c.need(loss->scalar_type() == at::kFloat && shaped(*loss, lead));
        if (dlogits) c.need(dlogits->scalar_type() == at::kFloat && shaped(*dlogits, full));
        if (!c.ok) Py_RETURN_NONE;
        at::Tensor made[2];
        if (!loss) loss = &(made[0] = fresh(lead, at::kFloat, c.dev));
        if (!dlogits) dlogits = &(made[1] = fresh(full, at::kFloat, c.dev));
        const void *zp = ptr(draft), *tp = ptr(target);
        const auto* mp = static_cast<const uint8_t*>(ptr(mask));
        auto *lp = static_cast<float*>(ptr(loss)), *gp = static_cast<float*>(ptr(dlogits));
        auto* sp = static_cast<int32_t*>(ptr(status));
        const osd_status st = released([&]() {
            return osd_distill(zp, tp, osd_dtype(dt), int(d.G), int(d.P), int(d.V), d.sg, d.sp, t.sg, t.sp, mp,
                               osd_loss(kind), float(beta), float(temperature), lp, gp, sp, stream);
        });
        if (st != OSD_OK) return PyLong_FromLong(st);
        PyObject* l = made[0].defined() ? THPVariable_Wrap(made[0]) : Py_NewRef(a[6]);
        PyObject* g = made[1].defined() ? THPVariable_Wrap(made[1]) : Py_NewRef(a[7]);
        PyObject* r = (l && g) ? PyTuple_Pack(2, l, g) : nullptr;
        Py_XDECREF(l);
        Py_XDECREF(g);
        return r;
    });
}

// draft, target, accepted, kind, beta, temperature, out, status, stream
PyObject* distill_accepted(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 9) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        Call c;
        const at::Tensor *draft = c.tensor(a[0]), *target = c.tensor(a[1]), *acc = c.tensor(a[2]);
        if (!c.ok || draft->dim() != 3) Py_RETURN_NONE;
        const int64_t B = draft->size(0), k = draft->size(1), V = draft->size(2);
        const int dt = dtype_code(*draft);
        c.need(dt >= 0 && draft->is_contiguous() && target->scalar_type() == draft->scalar_type() &&
               shaped(*target, {B, k + 1, V}) && acc->scalar_type() == at::kInt && shaped(*acc, {B}));
        const int kind = c.kind(a[3]);
        const double beta = c.number(a[4]), temperature = c.number(a[5]);
        const at::Tensor* status = c.optional(a[7]);
        void* stream = c.stream(a[8]);
        const at::Tensor* o[4] = {};
        at::Tensor made[4];
        const bool own = a[6] == Py_None;
        if (!own) {
            if (!c.need(Py_TYPE(a[6]) == reinterpret_cast<PyTypeObject*>(g_accepted_result))) Py_RETURN_NONE;
            for (int i = 0; i < 4; ++i) o[i] = c.member(a[6], i);
        }
        if (!c.ok) Py_RETURN_NONE;
        if (own) {
            made[0] = fresh({B}, at::kFloat, c.dev);
            made[1] = fresh({B, V}, at::kFloat, c.dev);
            made[2] = fresh({B}, at::kInt, c.dev);
            made[3] = fresh({1}, at::kInt, c.dev);
            for (int i = 0; i < 4; ++i) o[i] = &made[i];
        }
        const void *zp = ptr(draft), *tp = ptr(target);
        const auto* ap = static_cast<const int32_t*>(ptr(acc));
        void* p[4];
        for (int i = 0; i < 4; ++i) p[i] = ptr(o[i]);
        auto* sp = static_cast<int32_t*>(ptr(status));
        const osd_status st = released([&]() {
            return osd_distill_accepted(zp, tp, osd_dtype(dt), int(B), int(k), int(V), ap, osd_loss(kind), float(beta),
                                        float(temperature), static_cast<float*>(p[0]), static_cast<float*>(p[1]),
                                        static_cast<int32_t*>(p[2]), static_cast<int32_t*>(p[3]), sp, stream);
        });
        if (st != OSD_OK) return PyLong_FromLong(st);
        return own ? result(g_accepted_result, made, 4) : Py_NewRef(a[6]);
    });
}

// draft, target, uniforms, beta, temperature, tokens, cdf_gap, status, stream
PyObject* mixed_sample(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 9) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        Call c;
        const at::Tensor *draft = c.tensor(a[0]), *target = c.tensor(a[1]), *u = c.tensor(a[2]);
        auto rows = [](const at::Tensor& t) { return t.dim() == 2 && (t.size(1) <= 1 || t.stride(1) == 1); };
        if (!c.ok || !rows(*draft) || !rows(*target) || draft->sizes() != target->sizes()) Py_RETURN_NONE;
        const int64_t N = draft->size(0), V = draft->size(1);
        const int dt = dtype_code(*draft);
        c.need(dt >= 0 && target->scalar_type() == draft->scalar_type() && u->scalar_type() == at::kFloat && shaped(*u, {N}));
        const double beta = c.number(a[3]), temperature = c.number(a[4]);
        const at::Tensor *tokens = c.optional(a[5]), *gap = c.optional(a[6]), *status = c.optional(a[7]);
        void* stream = c.stream(a[8]);
        if (!c.ok) Py_RETURN_NONE;
        at::Tensor made;
        if (!tokens) tokens = &(made = fresh({N}, at::kInt, c.dev));
        const void *zp = ptr(draft), *tp = ptr(target);
        const int64_t ds = draft->stride(0), ts = target->stride(0);
        const auto* up = static_cast<const float*>(ptr(u));
        auto* yp = static_cast<int32_t*>(ptr(tokens));
        auto* gp = static_cast<float*>(ptr(gap));
        auto* sp = static_cast<int32_t*>(ptr(status));
        const osd_status st = released([&]() {
            return osd_mixed_sample(zp, tp, osd_dtype(dt), int(N), int(V), ds, ts, up, float(beta), float(temperature), yp,
                                    gp, sp, stream);
        });
        if (st != OSD_OK) return PyLong_FromLong(st);
        PyObject* y = made.defined() ? THPVariable_Wrap(made) : Py_NewRef(a[5]);
        PyObject* r = y ? PyTuple_Pack(2, y, a[6]) : nullptr;
        Py_XDECREF(y);
        return r;
    });
}

// draft, target, parent, tokens, uniforms, temperature, diagnostics, workspace, out, stream
PyObject* verify_tree(PyObject*, PyObject* const* a, Py_ssize_t n_args) {
    if (n_args != 10) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        Call c;
        const at::Tensor* target = c.tensor(a[1]);
        if (!c.ok || target->dim() != 3) Py_RETURN_NONE;
        const int64_t B = target->size(0), n = target->size(1), V = target->size(2);
        const at::Tensor *draft = c.optional(a[0]), *tokens = c.tensor(a[3]), *uniforms = c.optional(a[4]);
        const int dt = dtype_code(*target);
        if (!c.need(dt >= 0 && target->is_contiguous() && n <= OSD_TREE_MAX_NODES)) Py_RETURN_NONE;
        if (draft) c.need(draft->scalar_type() == target->scalar_type() && shaped(*draft, {B, n, V}));
        c.need(tokens->scalar_type() == at::kInt && shaped(*tokens, {B, n}));
        if (uniforms) c.need(uniforms->scalar_type() == at::kFloat && shaped(*uniforms, {B, n}));
        int32_t parent[OSD_TREE_MAX_NODES];
        if (!c.need(PyList_CheckExact(a[2]) && PyList_GET_SIZE(a[2]) == n)) Py_RETURN_NONE;
        for (int64_t i = 0; i < n; ++i) {
            PyObject* o = PyList_GET_ITEM(a[2], i);
            if (!PyLong_CheckExact(o)) Py_RETURN_NONE;
            const long v = PyLong_AsLong(o);
            if ((v == -1 && PyErr_Occurred()) || v < INT_MIN || v > INT_MAX) {
                PyErr_Clear();
                Py_RETURN_NONE;
            }
            parent[i] = static_cast<int32_t>(v);
        }
        const double temperature = c.number(a[5]);
        const bool diagnostics = a[6] == Py_True;
        c.need(diagnostics || a[6] == Py_False);
        void* stream = c.stream(a[9]);
        size_t need = 0;
        if (!c.ok || osd_verify_tree_workspace_size(int(B), int(n), int(V), &need) != OSD_OK) Py_RETURN_NONE;
        const at::Tensor* given = c.optional(a[7]);
        const at::Tensor* o[6] = {};
        at::Tensor made[6];
        const bool own = a[8] == Py_None;
        if (!own) {
            if (!c.need(Py_TYPE(a[8]) == reinterpret_cast<PyTypeObject*>(g_tree_result))) Py_RETURN_NONE;
            for (int i = 0; i < 6; ++i) o[i] = c.member(a[8], i);
        }
        if (!c.ok) Py_RETURN_NONE;
        at::Tensor ws;
        if (!given) {
            ws = fresh({int64_t(need < 16 ? 16 : need)}, at::kByte, c.dev);
            given = &ws;
        }
        if (own) {
            made[0] = fresh({B}, at::kInt, c.dev);
            made[1] = fresh({B, n}, at::kInt, c.dev);
            made[2] = fresh({B, n}, at::kInt, c.dev);
            made[3] = fresh({B}, at::kInt, c.dev);
            if (diagnostics) {
                made[4] = fresh({B, n}, at::kFloat, c.dev);
                made[5] = fresh({B}, at::kFloat, c.dev);
            }
            for (int i = 0; i < 6; ++i) o[i] = made[i].defined() ? &made[i] : nullptr;
        }
        const void *zp = ptr(draft), *tp = ptr(target);
        const auto* yp = static_cast<const int32_t*>(ptr(tokens));
        const auto* up = static_cast<const float*>(ptr(uniforms));
        void* p[6];
        for (int i = 0; i < 6; ++i) p[i] = ptr(o[i]);
        void* wp = ptr(given);
        const size_t wbytes = size_t(given->numel()) * given->element_size();
        const osd_status st = released([&]() {
            return osd_verify_tree(zp, tp, osd_dtype(dt), int(B), int(n), int(V), parent, yp, up, float(temperature),
                                   static_cast<int32_t*>(p[0]), static_cast<int32_t*>(p[1]), static_cast<int32_t*>(p[2]),
                                   static_cast<int32_t*>(p[3]), static_cast<float*>(p[4]), static_cast<float*>(p[5]), wp,
                                   wbytes, stream);
        });
        if (st != OSD_OK) return PyLong_FromLong(st);
        return own ? result(g_tree_result, made, 6) : Py_NewRef(a[8]);
    });
}

// VerifyResult, DistillAcceptedResult, TreeResult: the tuple classes the results come in
PyObject* setup(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 3 || !PyType_Check(a[0]) || !PyType_Check(a[1]) || !PyType_Check(a[2])) {
        PyErr_SetString(PyExc_TypeError, "setup takes the three result classes");
        return nullptr;
    }
    g_verify_result = Py_NewRef(a[0]);
    g_accepted_result = Py_NewRef(a[1]);
    g_tree_result = Py_NewRef(a[2]);
    Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {{"setup", FAST(setup)},
                         {"verify", FAST(verify)},
                         {"distill", FAST(distill)},
                         {"distill_accepted", FAST(distill_accepted)},
                         {"mixed_sample", FAST(mixed_sample)},
                         {"verify_tree", FAST(verify_tree)},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return g_cuda_stream ? PyModule_Create(&module) : nullptr;
}
