// Argument marshalling of the device entry points for Python: torch tensors in, C ABI calls out.
//
// A small layer's kernels take 3 to 6 us, so what a call costs on the host decides how fast layers follow
// one another.  Marshalling the same arguments in Python through ctypes took 9 us (decode) to 12 us (product)
// per call; here it takes well under one, the rest is the kernel launch itself.
//
// The module holds no arithmetic and no state beyond the addresses of the C functions, which the Python
// side hands over once (so that an alternative build of the library can be loaded in its place).
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "sqnn.h"

namespace {

decltype(&sqnn_decode) f_decode = nullptr;
decltype(&sqnn_decode_matmul) f_matmul = nullptr;
decltype(&sqnn_decode_matmul_static) f_matmul_static = nullptr;

PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t nargs)
{
    if (nargs != 3) { PyErr_SetString(PyExc_TypeError, "bind takes three addresses"); return nullptr; }
    void *p[3];
    for (int i = 0; i < 3; ++i) {
        p[i] = PyLong_AsVoidPtr(args[i]);
        if (PyErr_Occurred()) return nullptr;
    }
    f_decode = reinterpret_cast<decltype(f_decode)>(p[0]);
    f_matmul = reinterpret_cast<decltype(f_matmul)>(p[1]);
    f_matmul_static = reinterpret_cast<decltype(f_matmul_static)>(p[2]);
    Py_RETURN_NONE;
}

// The descriptor lives in a ctypes structure, which exports its memory through the buffer protocol.
struct DescArg {
    Py_buffer view{};
    bool held = false;
    const sqnn_desc *get(PyObject *o)
    {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return nullptr;
        held = true;
        if (view.len != (Py_ssize_t)sizeof(sqnn_desc)) {
            PyErr_SetString(PyExc_TypeError, "descriptor of the wrong size");
            return nullptr;
        }
        return static_cast<const sqnn_desc *>(view.buf);
    }
    ~DescArg() { if (held) PyBuffer_Release(&view); }
};

// A tensor argument; None stands for a null pointer.
bool tensor_arg(PyObject *o, const at::Tensor **t)
{
    if (o == Py_None) { *t = nullptr; return true; }
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor or None"); return false; }
    *t = &THPVariable_Unpack(o);
    return true;
}
template <typename T>
T *ptr(const at::Tensor *t) { return t ? static_cast<T *>(t->data_ptr()) : nullptr; }
size_t bytes_of(const at::Tensor *t) { return t ? (size_t)t->numel() * t->element_size() : 0; }

// None = torch's current stream of the current device, else an object with a cuda_stream attribute.
bool stream_arg(PyObject *o, void **st)
{
    if (o == Py_None) { *st = c10::cuda::getCurrentCUDAStream().stream(); return true; }
    PyObject *a = PyObject_GetAttrString(o, "cuda_stream");
    if (!a) return false;
    *st = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
    return !PyErr_Occurred();
}

bool enough(Py_ssize_t nargs, Py_ssize_t want)
{
    if (nargs == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
    return false;
}

// Other Python threads run while a C function is under way: a launch waits when the stream's queue is full, and in
// checked mode the call waits for its stream.  Everything a call needs has been read out of its Python
// arguments before; the caller's references keep them alive until it returns.
class Unlocked {
  public:
    Unlocked() : state_(PyEval_SaveThread()) {}
    ~Unlocked() { PyEval_RestoreThread(state_); }
    Unlocked(const Unlocked &) = delete;
    Unlocked &operator=(const Unlocked &) = delete;

  private:
    PyThreadState *state_;
};

// C++ exceptions of torch (a tensor without storage, for instance) must not cross into C.
template <typename F>
PyObject *guarded(F &&f)
{
    try {
        return f();
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// decode(desc, blob, mask, alpha, mode, out, status, stream) -> status code
PyObject *decode(PyObject *, PyObject *const *a, Py_ssize_t nargs)
{
    return guarded([&]() -> PyObject * {
        if (!enough(nargs, 8)) return nullptr;
        DescArg desc;
        const sqnn_desc *d = desc.get(a[0]);
        const at::Tensor *blob, *mask, *alpha, *out, *status;
        void *st;
        if (!d || !tensor_arg(a[1], &blob) || !tensor_arg(a[2], &mask) || !tensor_arg(a[3], &alpha) ||
            !tensor_arg(a[5], &out) || !tensor_arg(a[6], &status) || !stream_arg(a[7], &st))
            return nullptr;
        const long mode = PyLong_AsLong(a[4]);
        if (mode == -1 && PyErr_Occurred()) return nullptr;
        void *const p_blob = ptr<void>(blob), *const p_out = ptr<void>(out);
        const uint64_t *const p_mask = ptr<uint64_t>(mask);
        const float *const p_alpha = ptr<float>(alpha);
        uint32_t *const p_status = ptr<uint32_t>(status);
        const size_t out_bytes = bytes_of(out);
        int rc;
        {
            Unlocked u;
            rc = f_decode(d, p_blob, p_mask, p_alpha, (sqnn_out_mode)mode, p_out, out_bytes, p_status, st);
        }
        return PyLong_FromLong(rc);
    });
}

bool product_shapes(const at::Tensor *x, const at::Tensor *y)
{
    if (x && y && x->dim() == 2 && y->dim() == 2 && x->stride(1) == 1 && y->stride(1) == 1) return true;
    PyErr_SetString(PyExc_ValueError, "X and Y must be 2-D with unit inner stride");
    return false;
}

// What both products take out of their tensors.
struct Operands {
    void *blob, *x;
    uint64_t *mask;
    float *alpha, *y;
    uint32_t *status;
    uint32_t batch;
    int64_t ldx, ldy;
    Operands(const at::Tensor *blob_, const at::Tensor *mask_, const at::Tensor *alpha_, const at::Tensor *x_, const at::Tensor *y_,
             const at::Tensor *status_)
        : blob(ptr<void>(blob_)), x(ptr<void>(x_)), mask(ptr<uint64_t>(mask_)), alpha(ptr<float>(alpha_)), y(ptr<float>(y_)),
          status(ptr<uint32_t>(status_)), batch((uint32_t)x_->size(0)), ldx(x_->stride(0)), ldy(y_->stride(0)) {}
};

// matmul(desc, blob, mask, alpha, x, y, workspace, status, stream) -> status code
PyObject *matmul(PyObject *, PyObject *const *a, Py_ssize_t nargs)
{
    return guarded([&]() -> PyObject * {
        if (!enough(nargs, 9)) return nullptr;
        DescArg desc;
        const sqnn_desc *d = desc.get(a[0]);
        const at::Tensor *blob, *mask, *alpha, *x, *y, *ws, *status;
        void *st;
        if (!d || !tensor_arg(a[1], &blob) || !tensor_arg(a[2], &mask) || !tensor_arg(a[3], &alpha) ||
            !tensor_arg(a[4], &x) || !tensor_arg(a[5], &y) || !tensor_arg(a[6], &ws) || !tensor_arg(a[7], &status) ||
            !product_shapes(x, y))
            return nullptr;
        int xdt;
        if (x->scalar_type() == at::kFloat) xdt = SQNN_X_F32;
        else if (x->scalar_type() == at::kBFloat16) xdt = SQNN_X_BF16;
        else { PyErr_SetString(PyExc_ValueError, "X must be float32 or bfloat16"); return nullptr; }
        if (y->scalar_type() != at::kFloat) { PyErr_SetString(PyExc_ValueError, "Y must be float32"); return nullptr; }
        if (!stream_arg(a[8], &st)) return nullptr;
        const Operands o(blob, mask, alpha, x, y, status);
        void *const p_ws = ptr<void>(ws);
        const size_t ws_bytes = bytes_of(ws);
        int rc;
        {
            Unlocked u;
            rc = f_matmul(d, o.blob, o.mask, o.alpha, o.x, xdt, o.batch, o.ldx, o.y, o.ldy, p_ws, ws_bytes, o.status, st);
        }
        return PyLong_FromLong(rc);
    });
}

// matmul_static(desc, blob, mask, alpha, x, y, status, stream) -> status code
PyObject *matmul_static(PyObject *, PyObject *const *a, Py_ssize_t nargs)
{
    return guarded([&]() -> PyObject * {
        if (!enough(nargs, 8)) return nullptr;
        DescArg desc;
        const sqnn_desc *d = desc.get(a[0]);
        const at::Tensor *blob, *mask, *alpha, *x, *y, *status;
        void *st;
        if (!d || !tensor_arg(a[1], &blob) || !tensor_arg(a[2], &mask) || !tensor_arg(a[3], &alpha) ||
            !tensor_arg(a[4], &x) || !tensor_arg(a[5], &y) || !tensor_arg(a[6], &status) || !product_shapes(x, y))
            return nullptr;
        if (x->scalar_type() != at::kBFloat16 || y->scalar_type() != at::kFloat) {
            PyErr_SetString(PyExc_ValueError, "X must be bfloat16 and Y float32");
            return nullptr;
        }
        if (!stream_arg(a[7], &st)) return nullptr;
        const Operands o(blob, mask, alpha, x, y, status);
        int rc;
        {
            Unlocked u;
            rc = f_matmul_static(d, o.blob, o.mask, o.alpha, o.x, SQNN_X_BF16, o.batch, o.ldx, o.y, o.ldy, o.status, st);
        }
        return PyLong_FromLong(rc);
    });
}

PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, "addresses of the C functions"},
    {"decode", (PyCFunction)(void (*)(void))decode, METH_FASTCALL, "sqnn_decode"},
    {"matmul", (PyCFunction)(void (*)(void))matmul, METH_FASTCALL, "sqnn_decode_matmul"},
    {"matmul_static", (PyCFunction)(void (*)(void))matmul_static, METH_FASTCALL, "sqnn_decode_matmul_static"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_sqnn_python", "torch tensors to the C ABI of libsqnn", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sqnn_python(void) { return PyModule_Create(&module_def); }
