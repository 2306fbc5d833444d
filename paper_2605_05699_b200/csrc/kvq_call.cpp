// The host side of the compute calls of binding.py in native code: tensors in, one C ABI call out.
//
// A small call is bound by the host: of 5.7 us per kvq_append of 64 vectors (D = 128), calls one after another, the kernel takes 3.2,
// which run under the host's work for the next call, and half of that work went into a score of attribute reads on the tensors and a
// ctypes call of twelve converted arguments.  So: 5.7 -> 3.3 us; window flush of 64 x 16 rows 6.1 -> 5.2; one pass of either after
// which the GPU is waited for 21 -> 14 and 24 -> 16 us.  The
// functions here take plain torch tensors and plain ints on the current stream and read the same properties in C++; what they do not
// take (other objects, a stream argument, a device that is not the current one, values that do not fit) they leave untouched and return
// kNotTaken, and binding.py goes its general way, which also raises whatever there is to raise.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/kvq.h"

namespace {

constexpr long kNotTaken = -1;

struct {
    decltype(&kvq_encode) encode;
    decltype(&kvq_decode) decode;
    decltype(&kvq_append) append;
    decltype(&kvq_append_at) append_at;
    decltype(&kvq_flush_block) flush_block;
} abi;

// A tensor argument: torch.Tensor itself or a Parameter, contiguous and on a CUDA device; null otherwise.
inline const at::Tensor *tensor(PyObject *o)
{
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor &t = THPVariable_Unpack(o);
    return t.is_cuda() && t.is_contiguous() ? &t : nullptr;
}

inline bool integer(PyObject *o, int64_t *v)
{
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    *v = PyLong_AsLongLongAndOverflow(o, &overflow);
    return overflow == 0;
}

// What every call has: the plan, the half-precision tensor that gives D, the row count, the type and the device, and the lambda rows
struct Common {
    kvq_plan_t *plan;
    kvq_dtype_t dtype;
    int64_t D, rows, n_lambda;
    void *stream;
};

bool common(PyObject *plan, const at::Tensor *x, const at::Tensor *lam, Common *c)
{
    int64_t handle;
    if (!integer(plan, &handle) || !x || !lam || x->dim() < 1) return false;
    c->plan = reinterpret_cast<kvq_plan_t *>(handle);
    if (x->scalar_type() == at::kHalf) c->dtype = KVQ_F16;
    else if (x->scalar_type() == at::kBFloat16) c->dtype = KVQ_BF16;
    else return false;
    c->D = x->size(-1);
    if (c->D < 1) return false;
    c->rows = x->numel() / c->D;
    c->n_lambda = lam->numel() / c->D;
    const c10::DeviceIndex dev = x->get_device();
    if (dev != c10::cuda::current_device()) return false;
    c->stream = c10::cuda::getCurrentCUDAStream(dev).stream();
    return true;
}

template <class F>
PyObject *status(F &&f)
{
    long st;
    Py_BEGIN_ALLOW_THREADS
    st = (long)f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

// (plan, x, lam, packed, scales, rows_per_lambda)
PyObject *call_encode(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    Common c;
    int64_t rpl;
    if (n != 6) return PyLong_FromLong(kNotTaken);
    const at::Tensor *x = tensor(a[1]), *lam = tensor(a[2]), *packed = tensor(a[3]), *scales = tensor(a[4]);
    if (!packed || !scales || !integer(a[5], &rpl) || !common(a[0], x, lam, &c)) return PyLong_FromLong(kNotTaken);
    const void *xp = x->data_ptr(), *lp = lam->data_ptr();
    void *pp = packed->data_ptr(), *sp = scales->data_ptr();
    return status([&] { return abi.encode(c.plan, xp, c.dtype, c.rows, (const float *)lp, c.n_lambda, rpl, (uint8_t *)pp, sp, c.stream); });
    END_HANDLE_TH_ERRORS
}

// (plan, packed, scales, lam, out, rows_per_lambda)
PyObject *call_decode(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    Common c;
    int64_t rpl;
    if (n != 6) return PyLong_FromLong(kNotTaken);
    const at::Tensor *packed = tensor(a[1]), *scales = tensor(a[2]), *lam = tensor(a[3]), *out = tensor(a[4]);
    if (!packed || !scales || !integer(a[5], &rpl) || !common(a[0], out, lam, &c)) return PyLong_FromLong(kNotTaken);
    const void *pp = packed->data_ptr(), *sp = scales->data_ptr(), *lp = lam->data_ptr();
    void *op = out->data_ptr();
    return status([&] { return abi.decode(c.plan, (const uint8_t *)pp, sp, c.rows, (const float *)lp, c.n_lambda, rpl, op, c.dtype, c.stream); });
    END_HANDLE_TH_ERRORS
}

// (plan, x_new, lam, packed_cache, scales_cache, pos, streams_per_lambda); pos: an int (append), one int64 on the device (append_at)
template <bool AT>
PyObject *call_append(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    Common c;
    int64_t pos = 0, spl;
    if (n != 7) return PyLong_FromLong(kNotTaken);
    const at::Tensor *x = tensor(a[1]), *lam = tensor(a[2]), *packed = tensor(a[3]), *scales = tensor(a[4]), *pos_dev = nullptr;
    if (!packed || !scales || packed->dim() < 2 || !integer(a[6], &spl)) return PyLong_FromLong(kNotTaken);
    if constexpr (AT) {
        pos_dev = tensor(a[5]);
        if (!pos_dev || pos_dev->scalar_type() != at::kLong || pos_dev->numel() != 1) return PyLong_FromLong(kNotTaken);
    } else if (!integer(a[5], &pos)) {
        return PyLong_FromLong(kNotTaken);
    }
    if (!common(a[0], x, lam, &c)) return PyLong_FromLong(kNotTaken);
    const int64_t t_max = packed->size(-2);
    const void *xp = x->data_ptr(), *lp = lam->data_ptr(), *at_dev = AT ? pos_dev->data_ptr() : nullptr;
    void *pp = packed->data_ptr(), *sp = scales->data_ptr();
    return status([&] {
        return AT ? abi.append_at(c.plan, xp, c.dtype, c.rows, (const float *)lp, c.n_lambda, spl, (uint8_t *)pp, sp, t_max, (const int64_t *)at_dev, c.stream)
                       : abi.append(c.plan, xp, c.dtype, c.rows, (const float *)lp, c.n_lambda, spl, (uint8_t *)pp, sp, t_max, pos, c.stream);
    });
    END_HANDLE_TH_ERRORS
}

// (plan, x_block [S, rows, D], lam, packed_cache, scales_cache, dq_cache, pos0, streams_per_lambda)
PyObject *call_flush_block(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    Common c;
    int64_t pos, spl;
    if (n != 8) return PyLong_FromLong(kNotTaken);
    const at::Tensor *x = tensor(a[1]), *lam = tensor(a[2]), *packed = tensor(a[3]), *scales = tensor(a[4]), *dq = tensor(a[5]);
    if (!packed || !scales || !dq || packed->dim() < 2 || !integer(a[6], &pos) || !integer(a[7], &spl) || !common(a[0], x, lam, &c) || x->dim() != 3)
        return PyLong_FromLong(kNotTaken);
    const int64_t S = x->size(0), rows = x->size(1), t_max = packed->size(-2);
    const void *xp = x->data_ptr(), *lp = lam->data_ptr();
    void *pp = packed->data_ptr(), *sp = scales->data_ptr(), *dp = dq->data_ptr();
    return status([&] {
        return abi.flush_block(c.plan, xp, c.dtype, S, rows, (const float *)lp, c.n_lambda, spl, (uint8_t *)pp, sp, dp, t_max, pos, c.stream);
    });
    END_HANDLE_TH_ERRORS
}

// bind(addresses of kvq_encode, kvq_decode, kvq_append, kvq_append_at, kvq_flush_block) of the library that binding.py has loaded
PyObject *bind(PyObject *, PyObject *args)
{
    unsigned long long f[5];
    if (!PyArg_ParseTuple(args, "KKKKK", &f[0], &f[1], &f[2], &f[3], &f[4])) return nullptr;
    abi.encode = reinterpret_cast<decltype(abi.encode)>(f[0]);
    abi.decode = reinterpret_cast<decltype(abi.decode)>(f[1]);
    abi.append = reinterpret_cast<decltype(abi.append)>(f[2]);
    abi.append_at = reinterpret_cast<decltype(abi.append_at)>(f[3]);
    abi.flush_block = reinterpret_cast<decltype(abi.flush_block)>(f[4]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"encode", (PyCFunction)(void (*)())call_encode, METH_FASTCALL, nullptr},
    {"decode", (PyCFunction)(void (*)())call_decode, METH_FASTCALL, nullptr},
    {"append", (PyCFunction)(void (*)())call_append<false>, METH_FASTCALL, nullptr},
    {"append_at", (PyCFunction)(void (*)())call_append<true>, METH_FASTCALL, nullptr},
    {"flush_block", (PyCFunction)(void (*)())call_flush_block, METH_FASTCALL, nullptr},
    {"bind", bind, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "kvq_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// torch_version: the torch whose class layouts are compiled in; binding.py takes the module under no other.
PyMODINIT_FUNC PyInit_kvq_call()
{
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "torch_version", KVQ_TORCH) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
