// Python calls of the C ABI without ctypes: a step hands over some twenty tensors, and per call the marshalling in Python and
// ctypes took longer than the kernels' launches (26-node greedy step called one by one 15.9 -> 14.5 us; the first pass of a draft
// phase of six calls on new buffers 106 -> 67 us on one box).  What each argument has to be follows from the prototypes in fspad.h: a
// pointer to fspad_bf16, float, int32_t, uint64_t is a contiguous tensor of that type on the GPU (of the host entry point: in
// host memory, the cache apart) or None, a void pointer a uint8 tensor, an address or None, everything else a number.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <tuple>
#include <utility>

#include "fspad.h"

namespace {

template <typename T> struct Wanted;
template <> struct Wanted<fspad_bf16> { static constexpr at::ScalarType type = at::kBFloat16; static constexpr const char *name = "torch.bfloat16"; };
template <> struct Wanted<float> { static constexpr at::ScalarType type = at::kFloat; static constexpr const char *name = "torch.float32"; };
template <> struct Wanted<int32_t> { static constexpr at::ScalarType type = at::kInt; static constexpr const char *name = "torch.int32"; };
template <> struct Wanted<uint64_t> { static constexpr at::ScalarType type = at::kLong; static constexpr const char *name = "torch.int64"; };
template <> struct Wanted<void> { static constexpr at::ScalarType type = at::kByte; static constexpr const char *name = "torch.uint8"; };

// Address of a tensor's data; a Python error is set and false returned where it is not what the call takes.
template <typename T>
bool tensor_address(PyObject *o, bool on_gpu, void **out)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a tensor of %s, got %R", Wanted<T>::name, (PyObject *)Py_TYPE(o));
        return false;
    }
    const at::Tensor &t = THPVariable_Unpack(o);
    if (t.scalar_type() != Wanted<T>::type) {
        PyObject *is = PyObject_GetAttrString(o, "dtype");
        if (is != nullptr) PyErr_Format(PyExc_TypeError, "expected %s, got %S", Wanted<T>::name, is);
        Py_XDECREF(is);
        return false;
    }
    if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "tensor must be contiguous");
        return false;
    }
    if (on_gpu ? !t.is_cuda() : !t.is_cpu()) {
        PyErr_Format(PyExc_ValueError, "tensor must live on %s, not %s", on_gpu ? "cuda" : "cpu", t.device().str().c_str());
        return false;
    }
    *out = t.data_ptr();
    return true;
}

template <typename A>
bool convert(PyObject *o, bool on_gpu, A *out)
{
    if constexpr (std::is_pointer_v<A>) {
        using T = std::remove_cv_t<std::remove_pointer_t<A>>;
        void *p = nullptr;
        if (o == Py_None) {
        } else if constexpr (std::is_same_v<T, fspad_ctx> || std::is_same_v<T, void>) {
            if (PyLong_Check(o)) {
                p = PyLong_AsVoidPtr(o);
                if (p == nullptr && PyErr_Occurred()) return false;
            } else if constexpr (std::is_same_v<T, void>) {
                if (!tensor_address<T>(o, on_gpu, &p)) return false;
            } else {
                PyErr_SetString(PyExc_TypeError, "expected a context's address");
                return false;
            }
        } else if (!tensor_address<T>(o, on_gpu, &p)) {
            return false;
        }
        *out = static_cast<A>(p);
        return true;
    } else {
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) return false;
        if (static_cast<long long>(static_cast<A>(v)) != v) {
            PyErr_SetString(PyExc_OverflowError, "number does not fit");
            return false;
        }
        *out = static_cast<A>(v);
        return true;
    }
}

// host_from: the first argument whose tensors lie in host memory.  A tensor may throw when it is asked for its strides or its address
// (one inside vmap or grad, for instance): by torch's own translation that becomes the Python exception.
template <typename... A, size_t... I>
PyObject *invoke(int (*fn)(A...), PyObject *const *args, Py_ssize_t n, size_t host_from, std::index_sequence<I...>)
{
    if (n != (Py_ssize_t)sizeof...(A)) {
        PyErr_Format(PyExc_TypeError, "%zd arguments, not %zd", (Py_ssize_t)sizeof...(A), n);
        return nullptr;
    }
    std::tuple<A...> a{};
    try {
        if (!(convert(args[I], I < host_from, &std::get<I>(a)) && ...)) return nullptr;
    } catch (...) {
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(std::get<I>(a)...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
template <typename... A>
PyObject *invoke(int (*fn)(A...), PyObject *const *args, Py_ssize_t n, size_t host_from = 99)
{
    return invoke(fn, args, n, host_from, std::index_sequence_for<A...>());
}

#define FSPAD_CALL(name, ...) \
    PyObject *call_##name(PyObject *, PyObject *const *args, Py_ssize_t n) { return invoke(fspad_##name, args, n, ##__VA_ARGS__); }
FSPAD_CALL(tree_attn)
FSPAD_CALL(tree_attn_paged)
FSPAD_CALL(tree_accept)
FSPAD_CALL(kv_compact)
FSPAD_CALL(kv_compact_paged)
FSPAD_CALL(kv_append)
FSPAD_CALL(lm_head_accept)
FSPAD_CALL(feature_sampler)
FSPAD_CALL(tree_build)
FSPAD_CALL(draft_expand)
FSPAD_CALL(verify_step)
FSPAD_CALL(verify_step_host, 2)
#undef FSPAD_CALL

#define FSPAD_ENTRY(name) {#name, (PyCFunction)(void (*)(void))call_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FSPAD_ENTRY(tree_attn), FSPAD_ENTRY(tree_attn_paged), FSPAD_ENTRY(tree_accept), FSPAD_ENTRY(kv_compact),
                         FSPAD_ENTRY(kv_compact_paged), FSPAD_ENTRY(kv_append), FSPAD_ENTRY(lm_head_accept),
                         FSPAD_ENTRY(feature_sampler), FSPAD_ENTRY(tree_build), FSPAD_ENTRY(draft_expand),
                         FSPAD_ENTRY(verify_step), FSPAD_ENTRY(verify_step_host), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pycall() { return PyModule_Create(&module); }
