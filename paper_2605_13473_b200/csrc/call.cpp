// Argument marshalling of the hot calls (python module _osdn_call): torch tensors -> device pointers, the
// current stream of the current device, one call into libosdn.so.
//
// A decode step of one sequence is 2.7 us of GPU work, so the host side is what its caller waits for.  Built
// from Python objects (ctypes conversions, one method call per tensor property) that side took 10.9 us, with
// plain integers through ctypes 6.7 us; here the conversions take a few nanoseconds per tensor.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/osdn.h"

namespace {

enum Call { FWD, BWD, KDA_FWD, KDA_BWD, PRECOND, RATIO, DECODE, FWD_STATIC };
// tensor arguments of each call, the workspace (an own pair of pointer and size in the ABI) included
constexpr int kTensors[] = {12, 20, 12, 20, 6, 7, 9, 11};

bool pointer_of(PyObject* o, void** out, size_t* bytes)
{
    if (o == Py_None) {
        *out = nullptr;
        return true;
    }
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "the OSDN library takes torch tensors (or None)");
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "tensors passed to the OSDN library must be contiguous");
        return false;
    }
    *out = t.data_ptr();
    if (bytes) *bytes = t.nbytes();
    return true;
}

template <typename F> int with_workspace(F fn, const osdn_params* p, void** x, size_t bytes, void* st);
using Fwd = decltype(&osdn_fwd);
using Bwd = decltype(&osdn_bwd);
template <> int with_workspace<Fwd>(Fwd fn, const osdn_params* p, void** x, size_t bytes, void* st)
{
    auto f = [&](int i) { return static_cast<float*>(x[i]); };
    return fn(p, x[0], x[1], x[2], f(3), f(4), f(5), f(6), f(7), x[8], f(9), f(10), x[11], bytes, st);
}
template <> int with_workspace<Bwd>(Bwd fn, const osdn_params* p, void** x, size_t bytes, void* st)
{
    auto f = [&](int i) { return static_cast<float*>(x[i]); };
    return fn(p, x[0], x[1], x[2], f(3), f(4), f(5), f(6), f(7), x[8], f(9), f(10), x[11], x[12], x[13], f(14), f(15),
              f(16), f(17), f(18), x[19], bytes, st);
}

struct GilReleased {   // taken back on every way out
    PyThreadState* state = PyEval_SaveThread();
    ~GilReleased() { PyEval_RestoreThread(state); }
};

PyObject* g_params_type = nullptr;   // binding.OsdnParams

// register(type): the class of call's params
PyObject* register_params(PyObject*, PyObject* type)
{
    Py_INCREF(type);
    Py_XSETREF(g_params_type, type);
    Py_RETURN_NONE;
}

// call(which, params, *tensors) -> status code of the library
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    if (n < 2) {
        PyErr_SetString(PyExc_TypeError, "call(which, params, *tensors)");
        return nullptr;
    }
    const long which = PyLong_AsLong(args[0]);
    if (which == -1 && PyErr_Occurred()) return nullptr;
    if (which < FWD || which > FWD_STATIC || n - 2 != kTensors[which]) {
        PyErr_SetString(PyExc_TypeError, "unknown call, or a wrong number of tensors");
        return nullptr;
    }
    const int known = g_params_type ? PyObject_IsInstance(args[1], g_params_type) : 0;
    if (known < 0) return nullptr;
    if (!known) {
        PyErr_SetString(PyExc_TypeError, "params: not an OsdnParams");
        return nullptr;
    }
    Py_buffer view;   // the ctypes structure's own memory
    if (PyObject_GetBuffer(args[1], &view, PyBUF_SIMPLE) != 0) return nullptr;
    PyObject* result = nullptr;
    void* x[20];
    size_t bytes = 0;
    bool ok = view.len >= (Py_ssize_t)sizeof(osdn_params);
    if (!ok) PyErr_SetString(PyExc_TypeError, "params: not an OsdnParams");
    // torch throws where a tensor has no memory of its own (under vmap or grad) or there is no device: nothing may leave
    // through the C entry, it would end the process
    try {
        for (Py_ssize_t i = 0; ok && i < n - 2; ++i) ok = pointer_of(args[2 + i], &x[i], &bytes);   // the workspace is the last
        if (ok) {
            void* st = c10::cuda::getCurrentCUDAStream().stream();
            const osdn_params* p = static_cast<const osdn_params*>(view.buf);
            auto f = [&](int i) { return static_cast<float*>(x[i]); };
            int rc = 0;
            {
                const GilReleased released;   // a launch may wait for room in the stream
                switch (which) {
                    case FWD: rc = with_workspace<Fwd>(&osdn_fwd, p, x, bytes, st); break;
                    case KDA_FWD: rc = with_workspace<Fwd>(&osdn_kda_fwd, p, x, bytes, st); break;
                    case BWD: rc = with_workspace<Bwd>(&osdn_bwd, p, x, bytes, st); break;
                    case KDA_BWD: rc = with_workspace<Bwd>(&osdn_kda_bwd, p, x, bytes, st); break;
                    case PRECOND: rc = osdn_precond_update(p, x[0], f(1), f(2), f(3), x[4], f(5), st); break;
                    case RATIO: rc = osdn_residual_ratio(p, x[0], f(1), f(2), f(3), f(4), f(5), f(6), st); break;
                    case DECODE: rc = osdn_decode_step(p, x[0], x[1], x[2], f(3), f(4), f(5), f(6), f(7), x[8], st); break;
                    case FWD_STATIC:
                        rc = osdn_fwd_static(p, x[0], x[1], x[2], f(3), f(4), f(5), f(6), f(7), x[8], f(9), f(10), st);
                        break;
                }
            }
            result = PyLong_FromLong(rc);
        }
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    } catch (...) {
        PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
    }
    PyBuffer_Release(&view);
    return result;
}

PyMethodDef methods[] = {{"call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call)), METH_FASTCALL,
                          "call(which, params, *tensors) -> status code"},
                         {"register", register_params, METH_O, "register(type): the class of call's params"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_osdn_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__osdn_call() { return PyModule_Create(&module); }
