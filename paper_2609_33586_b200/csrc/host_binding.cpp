// The per-call host work of binding.attn_fwd as a CPython function: argument checks, the two output tensors, the current
// stream and the call through the C interface.  Written natively because this work, not the GPU, sets the time of small
// forwards: as Python and ctypes it took 19.7 us a call, of which the C interface itself is 3.5.
// No arithmetic of the method is here; the library is reached through the addresses of its C functions.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/Context.h>
#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/attn.h"

namespace {

struct Entries {
    decltype(&attn_fwd) fwd = nullptr;
    decltype(&attn_fwd_tau) tau = nullptr;
    decltype(&attn_fwd_pot) pot = nullptr;
    decltype(&attn_fwd_exact_emulated) emulated = nullptr;
} g_entries;

// set_entries(attn_fwd, attn_fwd_tau, attn_fwd_pot, attn_fwd_exact_emulated): addresses in the loaded library
PyObject* set_entries(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 4) {
        PyErr_SetString(PyExc_TypeError, "set_entries takes four addresses");
        return nullptr;
    }
    void* a[4];
    for (int i = 0; i < 4; ++i) {
        a[i] = PyLong_AsVoidPtr(args[i]);
        if (a[i] == nullptr) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address");
            return nullptr;
        }
    }
    g_entries.fwd = reinterpret_cast<decltype(&attn_fwd)>(a[0]);
    g_entries.tau = reinterpret_cast<decltype(&attn_fwd_tau)>(a[1]);
    g_entries.pot = reinterpret_cast<decltype(&attn_fwd_pot)>(a[2]);
    g_entries.emulated = reinterpret_cast<decltype(&attn_fwd_exact_emulated)>(a[3]);
    Py_RETURN_NONE;
}

int in_type(const at::Tensor& t) {
    switch (t.scalar_type()) {
        case at::kBFloat16: return ATTN_IN_BF16;
        case at::kFloat8_e4m3fn: return ATTN_IN_FP8_E4M3;
        case at::kHalf: return ATTN_IN_FP16;
        default: return -1;
    }
}

const at::Tensor* as_tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor");
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

// As ctypes takes an int argument: an integer (anything with __index__), of which the low bits count.  With `convert`
// whatever int() takes.
int as_int(PyObject* o, bool convert = false) {
    if (PyErr_Occurred()) return 0;
    PyObject* i = convert ? PyNumber_Long(o) : PyNumber_Index(o);
    if (i == nullptr) return 0;
    const unsigned long bits = PyLong_AsUnsignedLongMask(i);
    Py_DECREF(i);
    return static_cast<int>(static_cast<unsigned int>(bits));
}

float as_float(PyObject* o) { return PyErr_Occurred() ? 0.0f : static_cast<float>(PyFloat_AsDouble(o)); }

// Address of a tensor's data, or of whatever else has a data_ptr().
void* data_of(PyObject* o) {
    if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
    PyObject* address = PyObject_CallMethod(o, "data_ptr", nullptr);
    if (address == nullptr) return nullptr;
    void* p = PyLong_AsVoidPtr(address);
    Py_DECREF(address);
    return p;
}

// An output tensor.  The allocation goes past the dispatcher (0.25 us a tensor) unless somebody there would see or change it: a
// dispatch mode, or the fill of deterministic mode.
at::Tensor new_output(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& q) {
    if (c10::impl::TorchDispatchModeTLS::any_modes_set() || at::globalContext().deterministicAlgorithms())
        return at::empty(sizes, q.options().dtype(type));
    return at::detail::empty_cuda(sizes, type, q.device(), std::nullopt);
}

// forward(q, k, v, out | None, lse | None, return_lse, causal, softmax_scale, weight_mode, q_descale, k_descale, v_descale,
//         kind, option, option2, stream | None) -> (out, lse | None), or the status code of a call that failed.
// kind: 0 attn_fwd, 1 attn_fwd_tau (option = threshold), 2 attn_fwd_pot (option = K_max, option2 = drop_tail),
// 3 attn_fwd_exact_emulated (option = share in eighths).  `causal`, K_max and the share go through int(), weight_mode must be an
// integer, truth decides return_lse and drop_tail.
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 16) {
        PyErr_SetString(PyExc_TypeError, "forward takes 16 arguments");
        return nullptr;
    }
    const at::Tensor* t[3];
    for (int i = 0; i < 3; ++i) {
        t[i] = as_tensor(a[i]);
        if (t[i] == nullptr) return nullptr;
    }
    const at::Tensor &q = *t[0], &k = *t[1], &v = *t[2];
    for (const at::Tensor* x : t) {
        if (!x->is_cuda() || !x->is_contiguous()) {
            PyErr_SetString(PyExc_ValueError, "q, k, v must be contiguous CUDA tensors");
            return nullptr;
        }
    }
    const int dt = in_type(q);
    if (dt < 0) {
        PyErr_SetString(PyExc_TypeError, "unsupported storage dtype");
        return nullptr;
    }
    if (in_type(k) != dt || in_type(v) != dt) {
        PyErr_SetString(PyExc_TypeError, "q, k, v must share one storage dtype");
        return nullptr;
    }
    if (q.dim() != 4 || k.dim() != 4 || v.sizes() != k.sizes() || k.size(0) != q.size(0) || k.size(3) != q.size(3)) {
        PyErr_SetString(PyExc_ValueError, "shape mismatch between q, k, v");
        return nullptr;
    }
    const int64_t B = q.size(0), Sq = q.size(1), Hq = q.size(2), D = q.size(3), Sk = k.size(1), Hkv = k.size(2);
    for (int64_t x : {B, Sq, Hq, D, Sk, Hkv}) {
        if (x > INT_MAX) {
            PyErr_SetString(PyExc_ValueError, "a dimension does not fit the C interface");
            return nullptr;
        }
    }
    const int return_lse = PyObject_IsTrue(a[5]);
    const int causal = a[6] == Py_True ? 1 : a[6] == Py_False ? 0 : as_int(a[6], true);
    const float scale = as_float(a[7]);
    const int mode = as_int(a[8]);
    const float dq = as_float(a[9]), dk = as_float(a[10]), dv = as_float(a[11]);
    const int kind = as_int(a[12]);
    const float tau = kind == 1 ? as_float(a[13]) : 0.0f;
    const int option = kind >= 2 ? as_int(a[13], true) : 0;
    const int option2 = PyObject_IsTrue(a[14]);
    if (PyErr_Occurred()) return nullptr;
    void* stream;
    if (a[15] == Py_None) {
        stream = c10::cuda::getCurrentCUDAStream().stream();
    } else {
        stream = PyLong_AsVoidPtr(a[15]);
        if (PyErr_Occurred()) return nullptr;
    }

    at::Tensor out, lse;
    void *op, *lp = nullptr;
    if (a[3] == Py_None) {
        out = new_output({B, Sq, Hq, D}, at::kBFloat16, q);
        op = out.data_ptr();
    } else {
        op = data_of(a[3]);
    }
    if (a[4] != Py_None) {
        lp = data_of(a[4]);
    } else if (return_lse) {
        lse = new_output({B, Hq, Sq}, at::kFloat, q);
        lp = lse.data_ptr();
    }
    if (PyErr_Occurred()) return nullptr;
    const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr();
    float* lsep = static_cast<float*>(lp);
    const int b = static_cast<int>(B), hq = static_cast<int>(Hq), hkv = static_cast<int>(Hkv), sq = static_cast<int>(Sq),
              sk = static_cast<int>(Sk), d = static_cast<int>(D);
    int rc;
    Py_BEGIN_ALLOW_THREADS
    switch (kind) {
        case 1: rc = g_entries.tau(qp, kp, vp, op, lsep, b, hq, hkv, sq, sk, d, causal, scale, mode, dt, dq, dk, dv, tau, stream); break;
        case 2: rc = g_entries.pot(qp, kp, vp, op, lsep, b, hq, hkv, sq, sk, d, causal, scale, dt, dq, dk, dv, option, option2, stream); break;
        case 3: rc = g_entries.emulated(qp, kp, vp, op, lsep, b, hq, hkv, sq, sk, d, causal, scale, dt, dq, dk, dv, option, stream); break;
        default: rc = g_entries.fwd(qp, kp, vp, op, lsep, b, hq, hkv, sq, sk, d, causal, scale, mode, dt, dq, dk, dv, stream); break;
    }
    Py_END_ALLOW_THREADS
    if (rc != 0) return PyLong_FromLong(rc);
    PyObject* pair = PyTuple_New(2);
    if (pair == nullptr) return nullptr;
    PyObject* o;
    if (a[3] == Py_None) o = THPVariable_Wrap(std::move(out));
    else { o = a[3]; Py_INCREF(o); }
    PyObject* l;
    if (a[4] != Py_None) { l = a[4]; Py_INCREF(l); }
    else if (return_lse) l = THPVariable_Wrap(std::move(lse));
    else { l = Py_None; Py_INCREF(l); }
    PyTuple_SET_ITEM(pair, 0, o);
    PyTuple_SET_ITEM(pair, 1, l);
    if (o == nullptr || l == nullptr) {
        Py_DECREF(pair);
        return nullptr;
    }
    return pair;
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"set_entries", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(set_entries)), METH_FASTCALL, nullptr},
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
// build.py looks for this text to tell which torch the module was built for
constexpr char kBuiltFor[] = "host module for torch " ROWMAX_TORCH;
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_host", kBuiltFor, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host() {
    PyObject* m = PyModule_Create(&module_def);
    if (m != nullptr && PyModule_AddStringConstant(m, "torch_version", ROWMAX_TORCH) != 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
