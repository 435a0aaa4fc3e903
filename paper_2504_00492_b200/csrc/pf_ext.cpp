// The Python entry points' call path in native code: argument checks, outputs, current stream and the call through the C
// ABI, in one extension call.  (Marshalled in Python through ctypes the same took 20 - 25 us per call, several times the
// kernel time of a decoded token; here it takes about 3 us.)  Only the ordinary case is handled: anything that does not
// fit -- wrong types or shapes, tensors on the wrong device -- returns None, and the Python code next to the caller finds
// out what is wrong and raises.
#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <limits.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "pf.h"

namespace {

int (*g_forward)(const pf_params*) = nullptr;      // pf_deltanet_fwd_ex of the loaded libpf.so

// a dense CUDA tensor of this type on `dev`
bool fits(const at::Tensor& t, at::ScalarType type, c10::Device dev) {
    return t.scalar_type() == type && t.device() == dev && t.layout() == at::kStrided && t.is_contiguous();
}
bool get_tensor(PyObject* o, const at::Tensor** out) {
    if (!THPVariable_Check(o)) return false;
    *out = &THPVariable_Unpack(o);
    return true;
}

// forward(q, k, v, beta, S0, chunk, O, S_final, stream, want_state, f32, impl, mode, step)
//   -> (O, S_final), or the library's status (int) if it is not 0, or None: not the ordinary case
// What torch throws on the way (no memory for the outputs, no device, a tensor without storage such as a traced one) becomes the
// Python exception that torch gives it.
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 14 || !g_forward) Py_RETURN_NONE;
    const at::Tensor *q, *k, *v, *beta, *s0 = nullptr;
    if (!get_tensor(a[0], &q) || !get_tensor(a[1], &k) || !get_tensor(a[2], &v) || !get_tensor(a[3], &beta)) Py_RETURN_NONE;
    if (a[4] != Py_None && !get_tensor(a[4], &s0)) Py_RETURN_NONE;
    if (!PyLong_CheckExact(a[5]) || a[8] != Py_None) Py_RETURN_NONE;
    const bool f32 = a[10] == Py_True, want_state = PyObject_IsTrue(a[9]) == 1;
    const at::ScalarType type = f32 ? at::kFloat : at::kBFloat16;
    if (!q->is_cuda() || k->dim() != 5 || q->dim() != 4 || v->dim() != 5 || beta->dim() != 4) Py_RETURN_NONE;
    const c10::Device dev = q->device();
    if (!fits(*q, type, dev) || !fits(*k, type, dev) || !fits(*v, type, dev) || !fits(*beta, type, dev)) Py_RETURN_NONE;
    const int64_t B = k->size(0), H = k->size(1), L = k->size(2), r = k->size(3), dk = k->size(4), dv = v->size(4);
    auto is4 = [](const at::Tensor& t, int64_t x, int64_t y, int64_t z, int64_t w) {
        return t.size(0) == x && t.size(1) == y && t.size(2) == z && t.size(3) == w;
    };
    if (!is4(*q, B, H, L, dk) || !is4(*beta, B, H, L, r) || !is4(*v, B, H, L, r)) Py_RETURN_NONE;
    if (B > INT_MAX || H > INT_MAX || L > INT_MAX) Py_RETURN_NONE;
    if (s0 && (!fits(*s0, at::kFloat, dev) || s0->dim() != 4 || !is4(*s0, B, H, dk, dv))) Py_RETURN_NONE;
    const int chunk = (int)PyLong_AsLong(a[5]), impl = (int)PyLong_AsLong(a[11]), mode = (int)PyLong_AsLong(a[12]),
              step = (int)PyLong_AsLong(a[13]);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    const at::Tensor *o_in = nullptr, *s_in = nullptr;
    if (a[6] != Py_None && !get_tensor(a[6], &o_in)) Py_RETURN_NONE;
    if (a[7] != Py_None && !get_tensor(a[7], &s_in)) Py_RETURN_NONE;

    // (the stream is the current one of the tensors' device, whatever device is current)
    c10::cuda::OptionalCUDAGuard guard;
    if (c10::cuda::current_device() != dev.index()) guard.set_device(dev);
    const cudaStream_t stream = c10::cuda::getCurrentCUDAStream(dev.index()).stream();
    at::Tensor O, S;
    if (!o_in) O = at::Tensor(at::detail::empty_cuda({B, H, L, dv}, at::kFloat, dev, std::nullopt));
    if (!s_in && want_state) S = at::Tensor(at::detail::empty_cuda({B, H, dk, dv}, at::kFloat, dev, std::nullopt));
    pf_params p{};
    p.q = q->const_data_ptr();
    p.k = k->const_data_ptr();
    p.v = v->const_data_ptr();
    p.beta = beta->const_data_ptr();
    p.S0 = s0 ? (const float*)s0->const_data_ptr() : nullptr;
    p.B = (int)B; p.H = (int)H; p.L = (int)L; p.d_k = (int)dk; p.d_v = (int)dv; p.r = (int)r; p.chunk = chunk;
    p.O = (float*)(o_in ? *o_in : O).mutable_data_ptr();
    if (s_in || want_state) p.S_final = (float*)(s_in ? *s_in : S).mutable_data_ptr();
    p.in_dtype = f32 ? PF_DTYPE_F32 : PF_DTYPE_BF16;
    p.impl = impl; p.mode = mode; p.step = step;
    p.stream = stream;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = g_forward(&p);
    Py_END_ALLOW_THREADS
    if (st != PF_OK) return PyLong_FromLong(st);
    PyObject* out = PyTuple_New(2);
    if (!out) return nullptr;
    auto put = [&](int i, PyObject* given, at::Tensor& made) {
        if (given != Py_None || !made.defined()) {
            Py_INCREF(given);
            PyTuple_SET_ITEM(out, i, given);
        } else {
            PyTuple_SET_ITEM(out, i, THPVariable_Wrap(std::move(made)));
        }
    };
    put(0, a[6], O);
    put(1, a[7], S);
    return out;
    END_HANDLE_TH_ERRORS
}

// bind(address of pf_deltanet_fwd_ex)
PyObject* bind(PyObject*, PyObject* addr) {
    void* p = PyLong_AsVoidPtr(addr);
    if (!p && PyErr_Occurred()) return nullptr;
    g_forward = (int (*)(const pf_params*))p;
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"forward", (PyCFunction)(void (*)(void))forward, METH_FASTCALL, nullptr},
                         {"bind", bind, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pf_ext", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pf_ext(void) { return PyModule_Create(&module); }
