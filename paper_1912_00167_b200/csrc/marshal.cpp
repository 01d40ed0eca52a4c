// The Python binding's direct loss call in native code: the tensors of one call checked and their addresses handed to
// impact_loss_fwd_bwd_call.  In Python the checks alone -- type, device, shape and layout of fourteen tensors, an
// attribute access each -- take four times as long as the launch itself.
//
// A call is served here only if every argument is exactly as it should be: plain dense CUDA tensors (no subclass, no
// wrapper of a transform, no lazily negated view), coefficients that are Python floats and ints in range.  Anything else
// gets None, and the caller goes the way that names the argument at fault.  Nothing is kept from one call for the next.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/TensorBase.h>
#include <c10/core/DispatchKeySet.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <limits>

#include "impact.h"

namespace {

using LossCall = int32_t (*)(const impact_loss_call*, void*);
LossCall g_loss_call = nullptr;

// A plain dense CUDA tensor of the type and shape, contiguous?  Its tensor, or nullptr.
const at::Tensor* plain_cuda(PyObject* o) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    const c10::TensorImpl* const impl = t.unsafeGetTensorImpl();
    static const c10::DispatchKeySet bare = c10::DispatchKeySet(c10::DispatchKey::CUDA) |
                                            c10::getAutocastRelatedKeySetFromBackend(c10::BackendComponent::CUDABit);
    static const c10::DispatchKeySet with_autograd = bare | c10::getAutogradRelatedKeySetFromBackend(c10::BackendComponent::CUDABit);
    const c10::DispatchKeySet keys = impl->key_set();
    if ((keys != with_autograd && keys != bare) || !impl->has_storage() || impl->layout() != c10::kStrided ||
        impl->is_python_dispatch() || !impl->is_contiguous())
        return nullptr;
    return &t;
}

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
    if (a[16] == Py_None) {
        *stream = c10::cuda::getCurrentCUDAStream().stream();
    } else {
        if (!PyLong_CheckExact(a[16])) return false;
        *stream = PyLong_AsVoidPtr(a[16]);
        if (!*stream && PyErr_Occurred()) return false;
    }
    return true;
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

PyMethodDef g_methods[] = {
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
