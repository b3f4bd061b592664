// Native half of the Python binding: argument marshalling for the C entry points, without ctypes.
//
// A small layer's launches take the GPU a few microseconds, and the interpreter took longer than that
// to issue them: per call 3.2 us to look up the current stream, 0.2 us per tensor for checks and
// pointer, 2.4 us per allocated result, about a microsecond of argument conversion (forward and
// backward of a layer with an activation: 33 us of host time for three launches). Here a call costs
// its launches and about a microsecond. The functions take what the Python functions of the same name
// take, in order and by position (paper: The stack under test: bindings compose training from the C ABI).
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "nb_linear.h"

namespace {

// given by the Python side: NbError, and what turns the rarer kinds of arguments into addresses
PyObject *g_error = nullptr, *g_pointer_of = nullptr, *g_stream_of = nullptr;

// Raises NbError(code, text) and returns null.
PyObject *raise(int rc)
{
    PyObject *e = g_error ? PyObject_CallFunction(g_error, "is", rc, nb_last_error()) : nullptr;
    if (e) {
        PyErr_SetObject(reinterpret_cast<PyObject *>(Py_TYPE(e)), e);
        Py_DECREF(e);
    } else if (!PyErr_Occurred()) {
        PyErr_Format(PyExc_RuntimeError, "nb_linear error %d: %s", rc, nb_last_error());
    }
    return nullptr;
}

void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

bool to_address(PyObject *o, void *&p)  // None or an int
{
    p = o == Py_None ? nullptr : PyLong_AsVoidPtr(o);
    return !(p == nullptr && PyErr_Occurred());
}
bool by_python(PyObject *convert, PyObject *o, void *&p)
{
    if (!convert) return PyErr_Format(PyExc_TypeError, "a tensor, an address or None is wanted, not %.100s", Py_TYPE(o)->tp_name), false;
    PyObject *a = PyObject_CallOneArg(convert, o);
    if (!a) return false;
    const bool ok = to_address(a, p);
    Py_DECREF(a);
    return ok;
}

// A device pointer from None, an address, a contiguous CUDA tensor, or (by Python) what behaves like one.
bool to_pointer(PyObject *o, void *&p)
{
    if (THPVariable_Check(o)) {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device tensors must be contiguous CUDA tensors");
            return false;
        }
        p = t.data_ptr();
        return true;
    }
    if (o == Py_None || PyLong_Check(o)) return to_address(o, p);
    return by_python(g_pointer_of, o, p);
}
// A stream from an address or (by Python) a stream object.
bool to_stream(PyObject *o, void *&p) { return PyLong_Check(o) ? to_address(o, p) : by_python(g_stream_of, o, p); }

template <class T>
bool convert(PyObject *o, T &v)
{
    if constexpr (std::is_pointer_v<T>) {
        void *p = nullptr;
        if (!to_pointer(o, p)) return false;
        v = p;
    } else if constexpr (std::is_floating_point_v<T>) {
        v = static_cast<T>(PyFloat_AsDouble(o));
        if (PyErr_Occurred()) return false;
    } else {
        const long long x = PyLong_AsLongLong(o);
        if (x == -1 && PyErr_Occurred()) return false;
        v = static_cast<T>(x);
        if (static_cast<long long>(v) != x) {
            PyErr_SetString(PyExc_OverflowError, "argument out of range");
            return false;
        }
    }
    return true;
}

// fn(args..., stream): the last argument may be left out or None, for the current stream.
template <class... A, size_t... I>
PyObject *call(int (*fn)(A...), PyObject *const *args, Py_ssize_t n, std::index_sequence<I...>)
{
    constexpr Py_ssize_t N = sizeof...(A);
    static_assert(std::is_same_v<std::tuple_element_t<N - 1, std::tuple<A...>>, void *>, "the last argument is the stream");
    if (n != N && n != N - 1) {
        PyErr_Format(PyExc_TypeError, "%zd or %zd arguments are wanted, not %zd", N - 1, N, n);
        return nullptr;
    }
    std::tuple<A...> v;
    auto one = [&](auto &dst, size_t i) {
        if constexpr (std::is_same_v<std::decay_t<decltype(dst)>, void *>)
            if (static_cast<Py_ssize_t>(i) == N - 1) {
                if (n < N || args[i] == Py_None) return dst = current_stream(), true;
                return to_stream(args[i], dst);
            }
        return convert(args[i], dst);
    };
    if (!(one(std::get<I>(v), I) && ...)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = std::apply(fn, v);
    Py_END_ALLOW_THREADS
    if (rc != NB_OK) return raise(rc);
    Py_RETURN_NONE;
}

template <auto fn>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    return [&]<class... A>(int (*f)(A...)) {
        return call(f, args, n, std::index_sequence_for<A...>{});
    }(fn);
    END_HANDLE_TH_ERRORS
}

bool to_tensor(PyObject *o, at::Tensor &t)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "a tensor is wanted, not %.100s", Py_TYPE(o)->tp_name);
        return false;
    }
    t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
        PyErr_SetString(PyExc_AssertionError, "device tensors must be contiguous CUDA tensors");
        return false;
    }
    return true;
}
bool dims(const at::Tensor &t, bool ok, const char *name)
{
    if (!ok) PyErr_Format(PyExc_ValueError, "%s has %lld dimensions", name, static_cast<long long>(t.dim()));
    return ok;
}
void *ptr(const at::Tensor &t) { return t.defined() ? t.data_ptr() : nullptr; }
PyObject *wrap(at::Tensor t)
{
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(std::move(t));
}

// linear_forward(inp, weight, bias, act) -> (out, pre_act or None)
PyObject *linear_forward(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    at::Tensor inp, weight;
    void *pb = nullptr;
    int act = 0;
    if (n != 4) return PyErr_Format(PyExc_TypeError, "4 arguments are wanted");
    if (!to_tensor(args[0], inp) || !to_tensor(args[1], weight) || !to_pointer(args[2], pb) || !convert(args[3], act))
        return nullptr;
    // of the weight only the number of rows is taken: it may have its columns in more than one dimension
    if (!dims(inp, inp.dim() == 2, "inp") || !dims(weight, weight.dim() >= 1, "weight")) return nullptr;
    const int64_t BT = inp.size(0), C = inp.size(1), OC = weight.size(0);
    const auto opt = inp.options().dtype(at::kBFloat16);
    at::Tensor out = at::empty({BT, act == NB_ACT_SWIGLU ? OC / 2 : OC}, opt), pre;
    if (act != NB_ACT_NONE) pre = at::empty({BT, OC}, opt);
    // whatever of torch can throw comes before the interpreter's lock is given up
    void *const po = ptr(out), *const pp = ptr(pre), *const pi = ptr(inp), *const pw = ptr(weight);
    void *const stream = current_stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = nb_linear_forward_ex(po, pp, pi, pw, pb, BT, C, OC, act, stream);
    Py_END_ALLOW_THREADS
    if (rc != NB_OK) return raise(rc);
    return Py_BuildValue("NN", wrap(std::move(out)), wrap(std::move(pre)));
    END_HANDLE_TH_ERRORS
}

// linear_backward(dout, inp, weight, pre_act, inp_pre_act, act, dweight, dbias, accumulate, need_dinp,
//                 need_dweight, need_dbias) -> (dinp, dweight, dbias)
PyObject *linear_backward(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    at::Tensor dout, weight, dinp, new_dw, new_db;
    void *pi = nullptr, *pp = nullptr, *pe = nullptr, *pdw = nullptr, *pdb = nullptr;
    int act = 0;
    if (n != 12) return PyErr_Format(PyExc_TypeError, "12 arguments are wanted");
    int flag[4];  // accumulate, need_dinp, need_dweight, need_dbias
    for (int i = 0; i < 4; ++i)
        if ((flag[i] = PyObject_IsTrue(args[8 + i])) < 0) return nullptr;
    // a gradient that is not asked for goes back as it came, whatever it is
    if (!to_tensor(args[0], dout) || !to_pointer(args[1], pi) || !to_tensor(args[2], weight) || !to_pointer(args[3], pp) ||
        !to_pointer(args[4], pe) || !convert(args[5], act) || (flag[2] && !to_pointer(args[6], pdw)) ||
        (flag[3] && !to_pointer(args[7], pdb)))
        return nullptr;
    // of dout only the number of rows is taken
    if (!dims(dout, dout.dim() >= 1, "dout") || !dims(weight, weight.dim() == 2, "weight")) return nullptr;
    const int64_t BT = dout.size(0), OC = weight.size(0), C = weight.size(1);
    const auto opt = dout.options();
    if (flag[1]) dinp = at::empty({BT, C}, opt.dtype(at::kBFloat16));
    if (flag[2] && args[6] == Py_None) pdw = ptr(new_dw = at::empty({OC, C}, opt.dtype(at::kFloat)));
    if (flag[3] && args[7] == Py_None) pdb = ptr(new_db = at::empty({OC}, opt.dtype(at::kFloat)));
    // whatever of torch can throw comes before the interpreter's lock is given up
    void *const px = ptr(dinp), *const pd = ptr(dout), *const pw = ptr(weight), *const stream = current_stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = nb_linear_backward_ex(px, pdw, pdb, pd, pi, pw, pp, pe, BT, C, OC, act, flag[0], NB_DTYPE_F32, stream);
    Py_END_ALLOW_THREADS
    if (rc != NB_OK) return raise(rc);
    auto given = [](PyObject *o, at::Tensor &t) { return t.defined() ? wrap(std::move(t)) : Py_NewRef(o); };
    return Py_BuildValue("NNN", wrap(std::move(dinp)), given(args[6], new_dw), given(args[7], new_db));
    END_HANDLE_TH_ERRORS
}

// set_python(NbError, pointer_of, stream_of)
PyObject *set_python(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != 3) return PyErr_Format(PyExc_TypeError, "3 arguments are wanted");
    Py_XSETREF(g_error, Py_NewRef(args[0]));
    Py_XSETREF(g_pointer_of, Py_NewRef(args[1]));
    Py_XSETREF(g_stream_of, Py_NewRef(args[2]));
    Py_RETURN_NONE;
}

#define NB_ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(&entry<name>)), METH_FASTCALL, nullptr}
#define NB_FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(&name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    NB_ENTRY(nb_linear_forward_ex),
    NB_ENTRY(nb_linear_backward_ex),
    NB_ENTRY(nb_gelu_dbias_noalloc),
    NB_ENTRY(nb_lora_linear_forward),
    NB_ENTRY(nb_lora_linear_backward),
    NB_ENTRY(nb_lora_down_stacked),
    NB_ENTRY(nb_lora_linear_forward_stacked),
    NB_ENTRY(nb_lora_linear_backward_stacked),
    NB_ENTRY(nb_lora_da_stacked),
    NB_ENTRY(nb_lm_head_ce_forward),
    NB_ENTRY(nb_ce_backward),
    NB_ENTRY(nb_cast_f32_to_bf16),
    NB_FAST(linear_forward),
    NB_FAST(linear_backward),
    NB_FAST(set_python),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling for the nb_linear C ABI.", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&g_module); }
