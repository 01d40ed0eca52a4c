// The Python binding's calls of every iteration in native code: the direct loss call, prepared calls re-issued, the ring's push
// and sample.  The tensors of a call are checked and their addresses handed to the library's function.  In Python the checks
// alone -- type, device, shape and layout of fourteen tensors, an attribute access each -- take four times as long as the
// launch itself, and a prepared call of 25 arguments as long as the launch.
//
// A call is served here only if every argument is exactly as it should be: plain dense tensors (no subclass, no wrapper of a
// transform, no lazily negated view), coefficients that are Python floats and ints in range.  Anything else gets None, and
// the caller goes the way that names the argument at fault.  Nothing is kept from one call for the next but what a prepared
// call was prepared with.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/TensorBase.h>
#include <c10/core/DispatchKeySet.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <limits>
#include <new>

#include "impact.h"

namespace {

using LossCall = int32_t (*)(const impact_loss_call*, void*);
LossCall g_loss_call = nullptr;

// A plain dense tensor of the device's memory (or the host's), contiguous?  Its tensor, or nullptr.
const at::Tensor* plain(PyObject* o, bool on_host) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    const c10::TensorImpl* const impl = t.unsafeGetTensorImpl();
    struct Keys {
        c10::DispatchKeySet bare, with_autograd;
        Keys(c10::DispatchKey key, c10::BackendComponent where)
            : bare(c10::DispatchKeySet(key) | c10::getAutocastRelatedKeySetFromBackend(where)),
              with_autograd(bare | c10::getAutogradRelatedKeySetFromBackend(where)) {}
    };
    static const Keys of_device(c10::DispatchKey::CUDA, c10::BackendComponent::CUDABit);
    static const Keys of_host(c10::DispatchKey::CPU, c10::BackendComponent::CPUBit);
    const c10::DispatchKeySet bare = on_host ? of_host.bare : of_device.bare;
    const c10::DispatchKeySet with_autograd = on_host ? of_host.with_autograd : of_device.with_autograd;
    const c10::DispatchKeySet keys = impl->key_set();
    if ((keys != with_autograd && keys != bare) || !impl->has_storage() || impl->layout() != c10::kStrided ||
        impl->is_python_dispatch() || !impl->is_contiguous())
        return nullptr;
    return &t;
}

const at::Tensor* plain_cuda(PyObject* o) { return plain(o, false); }

struct Shape {
    int64_t d[3];
    int n;
};
bool address(PyObject* o, c10::ScalarType type, const Shape& shape, void** out) {
    const at::Tensor* const t = plain_cuda(o);
    if (!t || t->scalar_type() != type || t->dim() != shape.n) return false;
    const auto sizes = t->sizes();
    for (int i = 0; i < shape.n; ++i)
        if (sizes[i] != shape.d[i]) return false;
    *out = t->data_ptr();
    return true;
}

// (a value that a float does not hold is left to the caller)
bool number(PyObject* coef, PyObject* name, float* out) {
    PyObject* const v = PyObject_GetAttr(coef, name);
    if (!v) return false;
    bool ok = PyFloat_CheckExact(v) || PyLong_CheckExact(v);
    if (ok) {
        const double x = PyFloat_AsDouble(v);
        ok = !(x == -1.0 && PyErr_Occurred()) && !(std::isfinite(x) && std::fabs(x) > (double)std::numeric_limits<float>::max());
        *out = (float)x;
    }
    Py_DECREF(v);
    return ok;
}
bool integer(PyObject* coef, PyObject* name, int64_t* out) {
    PyObject* const v = PyObject_GetAttr(coef, name);
    if (!v) return false;
    bool ok = PyLong_CheckExact(v);
    if (ok) {
        int overflow = 0;
        *out = PyLong_AsLongLongAndOverflow(v, &overflow);
        ok = overflow == 0;
    }
    Py_DECREF(v);
    return ok;
}

enum { kRhoBar, kCBar, kClipEps, kVfCoef, kEntCoef, kKlCoef, kLam, kRhoTw, kIsSource, kRatioMode, kObjective, kGlobalSteps, kNames };
PyObject* g_names[kNames];

// A stream's handle, None for the current one.  (Numbers only: what else stands for a stream is the caller's to turn into one.)
bool stream_of(PyObject* o, void** stream) {
    if (o == Py_None) {
        *stream = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    if (!PyLong_CheckExact(o)) return false;
    *stream = PyLong_AsVoidPtr(o);
    return *stream || !PyErr_Occurred();
}

bool fill(PyObject* const* a, impact_loss_call* c, void** stream) {
    const at::Tensor* const learner = plain_cuda(a[0]);
    const at::Tensor* const dlogits = plain_cuda(a[10]);
    if (!learner || !dlogits || learner->dim() != 3) return false;
    const auto sizes = learner->sizes();
    if (sizes[2] > std::numeric_limits<int32_t>::max()) return false;
    const Shape bta = {{sizes[0], sizes[1], sizes[2]}, 3}, bt = {{sizes[0], sizes[1], 0}, 2}, b = {{sizes[0], 0, 0}, 1}, terms = {{8, 0, 0}, 1};
    const c10::ScalarType lt = learner->scalar_type(), gt = dlogits->scalar_type(), f32 = at::kFloat;
    if ((lt != f32 && lt != at::kBFloat16) || (gt != f32 && gt != at::kBFloat16)) return false;
    void* p[15] = {};
    if (!address(a[0], lt, bta, &p[0]) || !address(a[1], lt, bta, &p[1]) || !address(a[2], f32, bt, &p[2]) ||
        !address(a[3], at::kInt, bt, &p[3]) || !address(a[4], f32, bt, &p[4]) || !address(a[5], f32, bt, &p[5]) ||
        !address(a[6], f32, bt, &p[6]) || !address(a[7], f32, b, &p[7]) || !address(a[9], f32, terms, &p[8]) ||
        !address(a[10], gt, bta, &p[9]) || !address(a[11], f32, bt, &p[10]) ||
        (a[12] != Py_None && !address(a[12], f32, bt, &p[11])) || (a[13] != Py_None && !address(a[13], f32, bt, &p[12])) ||
        (a[15] != Py_None && !address(a[15], lt, bta, &p[14])))
        return false;
    const at::Tensor* const workspace = plain_cuda(a[14]);
    if (!workspace || workspace->scalar_type() != at::kByte) return false;
    c->learner_logits = p[0];
    c->target_logits = p[1];
    c->worker_logp = static_cast<const float*>(p[2]);
    c->actions = static_cast<const int32_t*>(p[3]);
    c->rewards = static_cast<const float*>(p[4]);
    c->discounts = static_cast<const float*>(p[5]);
    c->values = static_cast<const float*>(p[6]);
    c->bootstrap_values = static_cast<const float*>(p[7]);
    c->logits_dtype = lt == f32 ? IMPACT_DTYPE_F32 : IMPACT_DTYPE_BF16;
    c->A = (int32_t)sizes[2];
    c->B = sizes[0];
    c->T = sizes[1];
    c->loss_terms = static_cast<float*>(p[8]);
    c->dlogits = p[9];
    c->dvalues = static_cast<float*>(p[10]);
    c->vtarget = static_cast<float*>(p[11]);
    c->advantage = static_cast<float*>(p[12]);
    c->workspace = workspace->data_ptr();
    c->workspace_bytes = (size_t)workspace->numel();
    c->target_logits_copy = p[14];
    PyObject* const coef = a[8];
    int64_t is_source, ratio_mode, objective, global_steps;
    if (!number(coef, g_names[kRhoBar], &c->rho_bar) || !number(coef, g_names[kCBar], &c->c_bar) ||
        !number(coef, g_names[kClipEps], &c->clip_eps) || !number(coef, g_names[kVfCoef], &c->coef.vf_coef) ||
        !number(coef, g_names[kEntCoef], &c->coef.ent_coef) || !number(coef, g_names[kKlCoef], &c->coef.kl_coef) ||
        !number(coef, g_names[kLam], &c->coef.lambda_) || !number(coef, g_names[kRhoTw], &c->coef.rho_tw) ||
        !integer(coef, g_names[kIsSource], &is_source) || !integer(coef, g_names[kRatioMode], &ratio_mode) ||
        !integer(coef, g_names[kObjective], &objective) || !integer(coef, g_names[kGlobalSteps], &global_steps))
        return false;
    if (is_source != (int32_t)is_source || ratio_mode != (int32_t)ratio_mode || objective != (int32_t)objective) return false;
    c->coef.is_source = (int32_t)is_source;
    c->coef.ratio_mode = (int32_t)ratio_mode;
    c->coef.objective = (int32_t)objective;
    c->coef.global_steps = global_steps;
    c->coef.dlogits_dtype = gt == f32 ? IMPACT_DTYPE_F32 : IMPACT_DTYPE_BF16;
    return stream_of(a[16], stream);
}

// loss(learner_logits, target_logits, worker_logp, actions, rewards, discounts, values, bootstrap_values, coef, loss_terms,
// dlogits, dvalues, vtarget, advantage, workspace, target_logits_copy, stream) -> status, or None: not served here
PyObject* loss(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 17 || !g_loss_call) {
        PyErr_SetString(PyExc_TypeError, "loss takes 17 arguments, after bind");
        return nullptr;
    }
    impact_loss_call call = {};
    void* stream = nullptr;
    bool served = false;
    try {
        served = fill(a, &call, &stream);
    } catch (...) {  // (what torch throws about an argument is found again, and named, the other way)
        served = false;
    }
    if (!served) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    int32_t status;
    Py_BEGIN_ALLOW_THREADS
    status = g_loss_call(&call, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// bind(address of impact_loss_fwd_bwd_call)
PyObject* bind(PyObject*, PyObject* address) {
    void* const p = PyLong_AsVoidPtr(address);
    if (!p) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no address");
        return nullptr;
    }
    g_loss_call = reinterpret_cast<LossCall>(p);
    Py_RETURN_NONE;
}

// ---- prepared calls: the function's address and its arguments, kept in a capsule that the binding's object holds beside
// whatever the addresses point into
struct Prepared {
    int32_t (*issue)(const Prepared&, void* stream);
    void* fn;
    void* p[18];
    float f[3];
    int64_t n[4];
    size_t bytes;
};
constexpr const char* kPrepared = "impact prepared call";

int32_t issue_loss(const Prepared& c, void* stream) {
    return reinterpret_cast<LossCall>(c.fn)(static_cast<const impact_loss_call*>(c.p[0]), stream);
}
int32_t issue_gaussian(const Prepared& c, void* stream) {
    auto in = [&](int i) { return static_cast<const float*>(c.p[i]); };
    auto out = [&](int i) { return static_cast<float*>(c.p[i]); };
    return reinterpret_cast<decltype(&impact_loss_fwd_bwd_gaussian)>(c.fn)(
        in(0), in(1), in(2), in(3), in(4), in(5), in(6), in(7), in(8), in(9), c.f[0], c.f[1], c.f[2],
        static_cast<const impact_coefficients*>(c.p[10]), c.n[0], c.n[1], (int32_t)c.n[2], out(11), out(12), out(13), out(14), out(15),
        out(16), c.p[17], c.bytes, stream);
}
int32_t issue_step(const Prepared& c, void* stream) {
    return reinterpret_cast<decltype(&impact_buffer_device_step)>(c.fn)(
        static_cast<impact_buffer*>(c.p[0]), static_cast<const impact_ring_field_map*>(c.p[1]), c.p[2], static_cast<const float*>(c.p[3]),
        static_cast<const float*>(c.p[4]), static_cast<const void* const*>(c.p[5]), (int32_t)c.n[0],
        static_cast<impact_loss_inputs*>(c.p[6]), stream);
}

// prepare(kind, address of the function, addresses, floats, integers) -> capsule.  kind: 0 loss call, 1 Gaussian loss, 2 step.
PyObject* prepare(PyObject*, PyObject* const* a, Py_ssize_t n) {
    static const struct {
        int32_t (*issue)(const Prepared&, void*);
        Py_ssize_t addresses, floats, integers;
    } kinds[] = {{issue_loss, 1, 0, 0}, {issue_gaussian, 18, 3, 4}, {issue_step, 7, 0, 1}};
    const long kind = n == 5 ? PyLong_AsLong(a[0]) : -1;
    if (kind < 0 || kind > 2 || !PyTuple_CheckExact(a[2]) || !PyTuple_CheckExact(a[3]) || !PyTuple_CheckExact(a[4]) ||
        PyTuple_GET_SIZE(a[2]) != kinds[kind].addresses || PyTuple_GET_SIZE(a[3]) != kinds[kind].floats ||
        PyTuple_GET_SIZE(a[4]) != kinds[kind].integers) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "prepare: not a call's arguments");
        return nullptr;
    }
    Prepared* const c = new (std::nothrow) Prepared();
    if (!c) return PyErr_NoMemory();
    c->issue = kinds[kind].issue;
    c->fn = PyLong_AsVoidPtr(a[1]);
    for (Py_ssize_t i = 0; i < kinds[kind].addresses; ++i) {
        PyObject* const v = PyTuple_GET_ITEM(a[2], i);
        c->p[i] = v == Py_None ? nullptr : PyLong_AsVoidPtr(v);
    }
    for (Py_ssize_t i = 0; i < kinds[kind].floats; ++i) c->f[i] = (float)PyFloat_AsDouble(PyTuple_GET_ITEM(a[3], i));
    for (Py_ssize_t i = 0; i < kinds[kind].integers; ++i) c->n[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(a[4], i));
    c->bytes = (size_t)c->n[3];
    PyObject* const capsule = PyErr_Occurred() || !c->fn ? nullptr : PyCapsule_New(c, kPrepared, [](PyObject* o) {
        delete static_cast<Prepared*>(PyCapsule_GetPointer(o, kPrepared));
    });
    if (!capsule) {
        delete c;
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no address");
    }
    return capsule;
}

// issue(capsule, stream) -> status, or None: not a stream's handle
PyObject* issue(PyObject*, PyObject* const* a, Py_ssize_t n) {
    const Prepared* const c = n == 2 ? static_cast<Prepared*>(PyCapsule_GetPointer(a[0], kPrepared)) : nullptr;
    if (!c) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "issue takes a prepared call and a stream");
        return nullptr;
    }
    void* stream = nullptr;
    bool served = false;
    try {
        served = stream_of(a[1], &stream);
    } catch (...) {
        served = false;
    }
    if (!served) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    int32_t status;
    Py_BEGIN_ALLOW_THREADS
    status = c->issue(*c, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// ---- the ring's calls
decltype(&impact_buffer_push) g_push = nullptr;
decltype(&impact_buffer_sample) g_sample = nullptr;

// push(buffer, fields, bytes of each field, stream) -> (status, slot), or None: not served here
PyObject* push(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 4 || !g_push) {
        PyErr_SetString(PyExc_TypeError, "push takes 4 arguments, after bind");
        return nullptr;
    }
    constexpr Py_ssize_t kMost = 16;
    const void* src[kMost] = {};
    void *buffer = nullptr, *stream = nullptr;
    int32_t where = IMPACT_SRC_DEVICE;
    bool served = false;
    try {
        served = [&] {
            if (!PyLong_CheckExact(a[0]) || !(buffer = PyLong_AsVoidPtr(a[0])) || !PyList_CheckExact(a[2])) return false;
            const bool list = PyList_CheckExact(a[1]);
            if (!list && !PyTuple_CheckExact(a[1])) return false;
            const Py_ssize_t fields = PyList_GET_SIZE(a[2]);
            if (fields > kMost || (list ? PyList_GET_SIZE(a[1]) : PyTuple_GET_SIZE(a[1])) != fields) return false;
            bool known = false;
            for (Py_ssize_t f = 0; f < fields; ++f) {
                PyObject* const o = list ? PyList_GET_ITEM(a[1], f) : PyTuple_GET_ITEM(a[1], f);
                if (o == Py_None) continue;
                const at::Tensor* t = plain(o, known && where == IMPACT_SRC_HOST);
                if (!t && !known && (t = plain(o, true))) where = IMPACT_SRC_HOST;
                if (!t) return false;
                known = true;
                if ((long long)t->nbytes() != PyLong_AsLongLong(PyList_GET_ITEM(a[2], f))) return false;
                src[f] = t->data_ptr();
            }
            return stream_of(a[3], &stream);
        }();
    } catch (...) {
        served = false;
    }
    if (!served || PyErr_Occurred()) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    int32_t status, slot = -1;
    Py_BEGIN_ALLOW_THREADS
    status = g_push(static_cast<impact_buffer*>(buffer), src, where, &slot, stream);
    Py_END_ALLOW_THREADS
    return Py_BuildValue("(ii)", (int)status, (int)slot);
}

// sample(buffer, stream) -> (status, slot, k), or None: not served here
PyObject* sample(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 2 || !g_sample) {
        PyErr_SetString(PyExc_TypeError, "sample takes 2 arguments, after bind");
        return nullptr;
    }
    void *buffer = nullptr, *stream = nullptr;
    bool served = false;
    try {
        served = PyLong_CheckExact(a[0]) && (buffer = PyLong_AsVoidPtr(a[0])) && stream_of(a[1], &stream);
    } catch (...) {
        served = false;
    }
    if (!served) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    int32_t status, slot = -1, k = -1;
    Py_BEGIN_ALLOW_THREADS
    status = g_sample(static_cast<impact_buffer*>(buffer), &slot, &k, nullptr, stream);
    Py_END_ALLOW_THREADS
    return Py_BuildValue("(iii)", (int)status, (int)slot, (int)k);
}

// bind_ring(addresses of impact_buffer_push and impact_buffer_sample)
PyObject* bind_ring(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void *push_at = nullptr, *sample_at = nullptr;
    if (n != 2 || !(push_at = PyLong_AsVoidPtr(a[0])) || !(sample_at = PyLong_AsVoidPtr(a[1]))) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no address");
        return nullptr;
    }
    g_push = reinterpret_cast<decltype(g_push)>(push_at);
    g_sample = reinterpret_cast<decltype(g_sample)>(sample_at);
    Py_RETURN_NONE;
}

#define IMPACT_FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    IMPACT_FAST(prepare),
    IMPACT_FAST(issue),
    IMPACT_FAST(push),
    IMPACT_FAST(sample),
    IMPACT_FAST(bind_ring),
    {"loss", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&loss)), METH_FASTCALL, nullptr},
    {"bind", &bind, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (the module's name says which Python and torch it was built for: IMPACT_MARSHAL, see build.py)
#define IMPACT_INIT_OF(name) PyInit_##name
#define IMPACT_INIT(name) IMPACT_INIT_OF(name)
PyMODINIT_FUNC IMPACT_INIT(IMPACT_MARSHAL)() {
    static const char* const names[kNames] = {"rho_bar", "c_bar", "clip_eps", "vf_coef", "ent_coef", "kl_coef", "lam", "rho_tw",
                                              "is_source", "ratio_mode", "objective", "global_steps"};
    for (int i = 0; i < kNames; ++i)
        if (!(g_names[i] = PyUnicode_InternFromString(names[i]))) return nullptr;
    return PyModule_Create(&g_module);
}
