// Python entry of the hot calls: what binding.py would do for every Actor step -- check the tensors,
// allocate the results, find the current stream, call the C ABI -- in native code.  At the small
// batches of a single Actor the step is bound by exactly this host work: the CartPole step at batch
// 160 took 15.0 us through ctypes and torch's Python functions, of which the GPU needed five.
//
// Every function returns the results, the status code (an int) of a call that failed, or None when
// the arguments are not what the fast path takes (binding.py then checks them one by one, raises for what a
// kernel could not read, and goes through ctypes with the rest).
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "accerl.h"

namespace {

// a CUDA tensor of the given type whose elements are contiguous, or null
const at::Tensor *cuda_tensor(PyObject *o, at::ScalarType type)
{
    if (!THPVariable_Check(o)) return nullptr;
    const at::Tensor &t = THPVariable_Unpack(o);
    return t.is_cuda() && t.scalar_type() == type && t.is_contiguous() ? &t : nullptr;
}

// did a conversion fail?  (binding.py's own then takes what it always took, or raises)
bool not_for_us()
{
    if (!PyErr_Occurred()) return false;
    PyErr_Clear();
    return true;
}

// the stream argument: an integer, or None for torch's current stream of `device`
bool stream_of(PyObject *o, c10::DeviceIndex device, void **stream)
{
    if (o == Py_None) {
        *stream = (void *)c10::cuda::getCurrentCUDAStream(device).stream();
        return true;
    }
    *stream = PyLong_AsVoidPtr(o);
    return *stream || !not_for_us();
}

at::Tensor empty(at::IntArrayRef size, at::ScalarType type, const at::Tensor &like)
{
    return at::detail::empty_cuda(size, type, like.device(), std::nullopt);
}

template <typename F>
accerl_status without_gil(F &&call)
{
    accerl_status st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    return st;
}

PyObject *wrapped(at::Tensor t) { return THPVariable_Wrap(std::move(t)); }

struct Names {
    PyObject *logits, *actions, *logp, *entropy, *value, *use_smaller;
} names;

void put(PyObject *dict, PyObject *key, at::Tensor t)
{
    PyObject *v = wrapped(std::move(t));
    PyDict_SetItem(dict, key, v);
    Py_XDECREF(v);
}

// what an observation batch and its uniforms have to be for the fast path
bool act_inputs(PyObject *u8, PyObject *obs_o, PyObject *u_o, const at::Tensor **obs, const at::Tensor **u, int64_t *b)
{
    *obs = cuda_tensor(obs_o, u8 == Py_True ? at::kByte : at::kFloat);
    *u = cuda_tensor(u_o, at::kFloat);
    if (!*obs || !*u || (*obs)->dim() < 1) return false;
    *b = (*obs)->size(0);
    return (*u)->numel() == *b && *b > 0 && *b <= INT32_MAX;
}

// act(handle, n_actions, frames, obs, uniforms, out, stream) -> (logits, actions, logp), or `out`
PyObject *py_act(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 7) return Py_BuildValue("");
    void *handle = PyLong_AsVoidPtr(a[0]);
    const int64_t A = PyLong_AsLongLong(a[1]);
    const at::Tensor *obs, *u;
    int64_t b;
    void *stream;
    if (not_for_us()) Py_RETURN_NONE;
    if (!act_inputs(a[2], a[3], a[4], &obs, &u, &b) || !stream_of(a[6], obs->device().index(), &stream)) Py_RETURN_NONE;
    void *dst[3];
    at::Tensor t[3];
    if (a[5] == Py_None) {
        t[0] = empty({b, A}, at::kFloat, *obs);
        t[1] = empty({b}, at::kInt, *obs);
        t[2] = empty({b}, at::kFloat, *obs);
        for (int i = 0; i < 3; ++i) dst[i] = t[i].data_ptr();
    } else {
        if (!PyTuple_Check(a[5]) || PyTuple_GET_SIZE(a[5]) != 3) Py_RETURN_NONE;
        for (int i = 0; i < 3; ++i) {
            PyObject *o = PyTuple_GET_ITEM(a[5], i);
            if (!THPVariable_Check(o)) Py_RETURN_NONE;
            dst[i] = THPVariable_Unpack(o).data_ptr();
        }
    }
    const void *obs_p = obs->data_ptr();
    const float *u_p = (const float *)u->data_ptr();
    const accerl_status st = without_gil([&] {
        return accerl_policy_act((accerl_policy *)handle, obs_p, u_p, (int32_t)b, (float *)dst[0], (int32_t *)dst[1],
                                 (float *)dst[2], stream);
    });
    if (st != ACCERL_OK) return PyLong_FromLong(st);
    if (a[5] != Py_None) {
        Py_INCREF(a[5]);
        return a[5];
    }
    PyObject *r = PyTuple_New(3);
    if (!r) return nullptr;
    for (int i = 0; i < 3; ++i) PyTuple_SET_ITEM(r, i, wrapped(std::move(t[i])));
    return r;
}

// act_ex(handle, n_actions, frames, value_head, obs, uniforms, stream) -> dict
PyObject *py_act_ex(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 7) return Py_BuildValue("");
    void *handle = PyLong_AsVoidPtr(a[0]);
    const int64_t A = PyLong_AsLongLong(a[1]);
    const at::Tensor *obs, *u;
    int64_t b;
    void *stream;
    if (not_for_us()) Py_RETURN_NONE;
    if (!act_inputs(a[2], a[4], a[5], &obs, &u, &b) || !stream_of(a[6], obs->device().index(), &stream)) Py_RETURN_NONE;
    at::Tensor logits = empty({b, A}, at::kFloat, *obs), actions = empty({b}, at::kInt, *obs),
               logp = empty({b}, at::kFloat, *obs), entropy = empty({b}, at::kFloat, *obs), value;
    if (a[3] == Py_True) value = empty({b}, at::kFloat, *obs);
    const void *obs_p = obs->data_ptr();
    const float *u_p = (const float *)u->data_ptr();
    float *value_p = value.defined() ? (float *)value.data_ptr() : nullptr;
    const accerl_status st = without_gil([&] {
        return accerl_policy_act_ex((accerl_policy *)handle, obs_p, u_p, (int32_t)b, (float *)logits.data_ptr(),
                                    (int32_t *)actions.data_ptr(), (float *)logp.data_ptr(), value_p,
                                    (float *)entropy.data_ptr(), stream);
    });
    if (st != ACCERL_OK) return PyLong_FromLong(st);
    PyObject *d = PyDict_New();
    if (!d) return nullptr;
    put(d, names.logits, std::move(logits));
    put(d, names.actions, std::move(actions));
    put(d, names.logp, std::move(logp));
    put(d, names.entropy, std::move(entropy));
    if (value.defined()) put(d, names.value, std::move(value));
    return d;
}

// act_mixed(smaller, original, n_actions, frames, value, obs, uniforms, select, alpha, stream) -> dict
PyObject *py_act_mixed(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 10) return Py_BuildValue("");
    void *smaller = PyLong_AsVoidPtr(a[0]), *original = PyLong_AsVoidPtr(a[1]);
    const int64_t A = PyLong_AsLongLong(a[2]);
    const double alpha = PyFloat_AsDouble(a[8]);
    const at::Tensor *obs, *u;
    int64_t b;
    void *stream;
    if (not_for_us()) Py_RETURN_NONE;
    const at::Tensor *select = cuda_tensor(a[7], at::kFloat);
    if (!act_inputs(a[3], a[5], a[6], &obs, &u, &b) || !select || select->numel() != b ||
        !stream_of(a[9], obs->device().index(), &stream))
        Py_RETURN_NONE;
    at::Tensor logits = empty({b, A}, at::kFloat, *obs), actions = empty({b}, at::kInt, *obs),
               logp = empty({b}, at::kFloat, *obs), entropy = empty({b}, at::kFloat, *obs),
               use = empty({b}, at::kByte, *obs), value;
    if (a[4] == Py_True) value = empty({b}, at::kFloat, *obs);
    const void *obs_p = obs->data_ptr();
    const float *u_p = (const float *)u->data_ptr(), *sel_p = (const float *)select->data_ptr();
    float *value_p = value.defined() ? (float *)value.data_ptr() : nullptr;
    const accerl_status st = without_gil([&] {
        return accerl_policy_act_mixed((accerl_policy *)smaller, (accerl_policy *)original, obs_p, u_p, sel_p,
                                       (float)alpha, (int32_t)b, (float *)logits.data_ptr(),
                                       (int32_t *)actions.data_ptr(), (float *)logp.data_ptr(), value_p,
                                       (float *)entropy.data_ptr(), (uint8_t *)use.data_ptr(), stream);
    });
    if (st != ACCERL_OK) return PyLong_FromLong(st);
    PyObject *d = PyDict_New();
    if (!d) return nullptr;
    put(d, names.logits, std::move(logits));
    put(d, names.actions, std::move(actions));
    put(d, names.logp, std::move(logp));
    put(d, names.entropy, std::move(entropy));
    put(d, names.use_smaller, std::move(use));
    if (value.defined()) put(d, names.value, std::move(value));
    return d;
}

// kl(logits_original, logits_smaller, stream) -> (kl, mean_max)
PyObject *py_kl(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 3) return Py_BuildValue("");
    const at::Tensor *zo = cuda_tensor(a[0], at::kFloat), *zs = cuda_tensor(a[1], at::kFloat);
    void *stream;
    if (!zo || !zs || zo->dim() != 2 || zo->sizes() != zs->sizes() || zo->size(0) > INT32_MAX ||
        zo->size(1) > INT32_MAX || !stream_of(a[2], zo->device().index(), &stream))
        Py_RETURN_NONE;
    at::Tensor out = empty({zo->size(0)}, at::kFloat, *zo), stats = empty({2}, at::kFloat, *zo);
    const float *zo_p = (const float *)zo->data_ptr(), *zs_p = (const float *)zs->data_ptr();
    const int32_t b = (int32_t)zo->size(0), A = (int32_t)zo->size(1);
    const accerl_status st = without_gil([&] {
        return accerl_policy_kl(zo_p, zs_p, b, A, (float *)out.data_ptr(), (float *)stats.data_ptr(), stream);
    });
    if (st != ACCERL_OK) return PyLong_FromLong(st);
    return Py_BuildValue("(NN)", wrapped(std::move(out)), wrapped(std::move(stats)));
}

// vtrace(logp_smaller, logp_original, rewards, values, bootstrap, discounts, gamma, rho_hat, c_hat, stream)
// -> (vs, adv)
PyObject *py_vtrace(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 10) return Py_BuildValue("");
    const at::Tensor *in[6] = {};
    for (int i = 0; i < 6; ++i) {
        if (i == 5 && a[5] == Py_None) break;
        in[i] = cuda_tensor(a[i], at::kFloat);
        if (!in[i]) Py_RETURN_NONE;
        if (i == 4 ? in[4]->dim() != 1 || in[4]->size(0) != in[0]->size(1)
                   : in[i]->dim() != 2 || in[i]->sizes() != in[0]->sizes())
            Py_RETURN_NONE;
    }
    void *stream;
    if (in[0]->size(0) > INT32_MAX || in[0]->size(1) > INT32_MAX || !stream_of(a[9], in[0]->device().index(), &stream))
        Py_RETURN_NONE;
    const double gamma = PyFloat_AsDouble(a[6]), rho = PyFloat_AsDouble(a[7]), c = PyFloat_AsDouble(a[8]);
    if (not_for_us()) Py_RETURN_NONE;
    at::Tensor vs = empty(in[0]->sizes(), at::kFloat, *in[0]), adv = empty(in[0]->sizes(), at::kFloat, *in[0]);
    const float *p[6];
    for (int i = 0; i < 6; ++i) p[i] = in[i] ? (const float *)in[i]->data_ptr() : nullptr;
    const int32_t steps = (int32_t)in[0]->size(0), b = (int32_t)in[0]->size(1);
    const accerl_status st = without_gil([&] {
        return accerl_vtrace(p[0], p[1], p[2], p[3], p[4], p[5], steps, b, (float)gamma, (float)rho, (float)c,
                             (float *)vs.data_ptr(), (float *)adv.data_ptr(), stream);
    });
    if (st != ACCERL_OK) return PyLong_FromLong(st);
    return Py_BuildValue("(NN)", wrapped(std::move(vs)), wrapped(std::move(adv)));
}

// act_noalloc(handle, obs, uniforms, batch, logits, actions, logp, stream): raw addresses -> status, or None for
// arguments that are no plain integers (ctypes pointers, numpy integers: binding.py passes those through ctypes)
PyObject *py_act_noalloc(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 8) return Py_BuildValue("");
    void *p[8] = {};
    for (int i = 0; i < 8; ++i) {
        if (i == 3 || a[i] == Py_None) continue;
        if (!PyLong_Check(a[i])) Py_RETURN_NONE;
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (!p[i] && not_for_us()) Py_RETURN_NONE;
    }
    if (!PyLong_Check(a[3])) Py_RETURN_NONE;
    const long batch = PyLong_AsLong(a[3]);
    if (batch == -1 && not_for_us()) Py_RETURN_NONE;
    const accerl_status st = without_gil([&] {
        return accerl_policy_act_noalloc((accerl_policy *)p[0], p[1], (const float *)p[2], (int32_t)batch, (float *)p[4],
                                         (int32_t *)p[5], (float *)p[6], p[7]);
    });
    return PyLong_FromLong(st);
}

// C++ exceptions (a failed allocation among them) become the Python exceptions torch raises for them
template <PyObject *(*F)(PyObject *, PyObject *const *, Py_ssize_t)>
PyObject *guarded(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    return F(self, a, n);
    END_HANDLE_TH_ERRORS
}

#define FAST(f) (PyCFunction)(void (*)(void))guarded<f>, METH_FASTCALL
PyMethodDef methods[] = {{"act", FAST(py_act), nullptr},
                         {"act_ex", FAST(py_act_ex), nullptr},
                         {"act_mixed", FAST(py_act_mixed), nullptr},
                         {"act_noalloc", FAST(py_act_noalloc), nullptr},
                         {"kl", FAST(py_kl), nullptr},
                         {"vtrace", FAST(py_vtrace), nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void)
{
    names.logits = PyUnicode_InternFromString("logits");
    names.actions = PyUnicode_InternFromString("actions");
    names.logp = PyUnicode_InternFromString("logp");
    names.entropy = PyUnicode_InternFromString("entropy");
    names.value = PyUnicode_InternFromString("value");
    names.use_smaller = PyUnicode_InternFromString("use_smaller");
    return PyModule_Create(&module);
}
