// Native argument marshalling of the two decode calls for Python (see api.py, which works without it).
//
// A decode step of one stream takes the GPU 4 us; from Python the checks and pointers of nine tensors, the output's allocation and
// the foreign call took the host 10 us a call, which is what a serving loop then saw.  Here the same checks and the same call run in
// one C function: 5.3 us.  It handles the plain case only - CUDA tensors, contiguous - and returns None for anything else: the Python
// path then raises or converts as ever.  Nothing is kept between calls.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using StepFn = int (*)(void *plan, int32_t Bdec, const void *q, const void *k, const void *v, const float *log_decay, const float *beta,
                       const float *lq, const float *lk, float *state, void *o, void *stream);
using StepsFn = int (*)(void *plan, int32_t Bdec, int32_t n_tokens, const void *q, const void *k, const void *v, const float *log_decay,
                        const float *beta, const float *lq, const float *lk, float *state, void *o, void *stream);

// The interpreter's lock is given up for as long as this lives (and is back before an exception reaches a handler).
struct Unlocked {
    PyThreadState *state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};

// Is obj None, or exactly a torch.Tensor (no subclass) on a CUDA device and contiguous?  Then its data goes to *p.
bool pointer(PyObject *obj, void **p) {
    *p = nullptr;
    if (obj == Py_None) return true;
    if (!THPVariable_CheckExact(obj)) return false;
    const at::Tensor &t = THPVariable_Unpack(obj);
    if (!t.is_cuda() || !t.is_contiguous()) return false;
    *p = t.data_ptr();
    return true;
}

// args: address of sla_decode_step or sla_decode_steps, plan, heads, width_v, bf16, several (0/1), q, k, v, log_decay, gq_logits, gk_logits,
// state, beta, o.  Returns (status, o), or None where the Python path has to take over.
PyObject *decode(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (n != 15) {
        PyErr_SetString(PyExc_TypeError, "decode takes 15 arguments");
        return nullptr;
    }
    try {
        void *fn = PyLong_AsVoidPtr(a[0]), *plan = PyLong_AsVoidPtr(a[1]);
        const long H = PyLong_AsLong(a[2]), dv = PyLong_AsLong(a[3]), bf16 = PyLong_AsLong(a[4]), several = PyLong_AsLong(a[5]);
        if (PyErr_Occurred()) return nullptr;
        if (!fn || a[6] == Py_None || !THPVariable_CheckExact(a[6])) Py_RETURN_NONE;
        const at::Tensor &q = THPVariable_Unpack(a[6]);
        if (q.dim() < (several ? 2 : 1)) Py_RETURN_NONE;
        void *p[9];                                     // q, k, v, log_decay, gq_logits, gk_logits, state, beta, o
        for (int i = 0; i < 9; ++i)
            if (!pointer(a[6 + i], &p[i])) Py_RETURN_NONE;
        PyObject *o = a[14];
        at::Tensor out;
        if (o == Py_None) {
            const auto opt = q.options().dtype(bf16 ? at::kBFloat16 : at::kFloat).requires_grad(false);
            out = several ? at::empty({q.size(0), q.size(1), H, dv}, opt) : at::empty({q.size(0), H, dv}, opt);
            p[8] = out.data_ptr();
        }
        const int32_t B = (int32_t)q.size(0);
        void *stream = (void *)c10::cuda::getCurrentCUDAStream(c10::cuda::current_device()).stream();
        int status;
        {
            Unlocked unlocked;              // (a launch waits where the stream's queue is full)
            if (several)
                status = reinterpret_cast<StepsFn>(fn)(plan, B, (int32_t)q.size(1), p[0], p[1], p[2], (const float *)p[3], (const float *)p[7],
                                                       (const float *)p[4], (const float *)p[5], (float *)p[6], p[8], stream);
            else
                status = reinterpret_cast<StepFn>(fn)(plan, B, p[0], p[1], p[2], (const float *)p[3], (const float *)p[7], (const float *)p[4],
                                                      (const float *)p[5], (float *)p[6], p[8], stream);
        }
        if (o == Py_None) o = THPVariable_Wrap(out);
        else Py_INCREF(o);
        if (!o) return nullptr;
        PyObject *code = PyLong_FromLong(status), *res = PyTuple_New(2);
        if (!code || !res) {
            Py_DECREF(o);
            Py_XDECREF(code);
            Py_XDECREF(res);
            return nullptr;
        }
        PyTuple_SET_ITEM(res, 0, code);
        PyTuple_SET_ITEM(res, 1, o);
        return res;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    } catch (...) {
        PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
        return nullptr;
    }
}

PyMethodDef methods[] = {{"decode", (PyCFunction)(void (*)(void))decode, METH_FASTCALL, "sla_decode_step(s) on torch tensors"}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_sla_fast", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sla_fast() { return PyModule_Create(&module); }
