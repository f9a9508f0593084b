// Native call path of the Python binding: what Plan's methods do per call -- check the tensors, allocate the outputs,
// look up the current stream, call the C ABI -- in one C function each.
//
// A call on a few rows is bound by the host: the kernel takes 3 us, and the same steps in Python took 17.5 us per call
// (two torch.empty at 2.3 us, torch.cuda.current_stream at 3.3 us, argument checks, ctypes marshalling at 0.8 us and the
// launch itself at 2.7 us).
//
// Every function here handles the regular call only and returns None for anything else (a tensor of another type or
// device, a shape or stride that needs a view, an output that is too small, a non-zero status): the caller then takes
// the Python path, which raises the error or makes the view.  Nothing is enqueued before the checks have passed.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include "gbs.h"

namespace {

// -1: not a type the library takes
int dtype_code(at::ScalarType t)
{
    return t == at::kFloat ? GBS_DTYPE_F32 : (t == at::kBFloat16 ? GBS_DTYPE_BF16 : -1);
}

bool plan_of(PyObject* o, const gbs_plan_t** plan, gbs_plan_info_t* info)
{
    if (!PyLong_Check(o)) return false;
    *plan = static_cast<const gbs_plan_t*>(PyLong_AsVoidPtr(o));
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return gbs_plan_info(*plan, info) == GBS_OK;
}

// None: the current stream of the current device; else a stream object with a `cuda_stream` handle
bool stream_of(PyObject* o, void** stream)
{
    if (o == Py_None) {
        *stream = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (h) {
        *stream = PyLong_AsVoidPtr(h);
        Py_DECREF(h);
    }
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return true;
}

const at::Tensor* cuda_tensor(PyObject* o)
{
    if (!THPVariable_Check(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    return t.defined() && t.is_cuda() && t.layout() == at::kStrided ? &t : nullptr;
}

// rows [.., d]: two-dimensional with contiguous rows, or contiguous of any other rank
bool rows_of(const at::Tensor* t, int d, int64_t* n_rows, int64_t* stride)
{
    const int64_t r = t->dim();
    if (r < 1 || t->size(r - 1) != d || t->stride(r - 1) != 1) return false;
    if (r == 2) {
        *n_rows = t->size(0);
        *stride = *n_rows > 1 ? t->stride(0) : (t->stride(0) > d ? t->stride(0) : d);
        return true;
    }
    if (!t->is_contiguous()) return false;
    *n_rows = t->numel() / d;
    *stride = d;
    return true;
}

bool buffer_ok(const at::Tensor* t, const at::Device& device, int64_t min_numel)
{
    return t && t->device() == device && t->is_contiguous() && t->numel() >= min_numel;
}

at::Tensor empty2(int64_t r, int64_t c, at::ScalarType dtype, const at::Device& device)
{
    return at::detail::empty_cuda({r, c}, dtype, device, std::nullopt);
}

#define GBS_BEGIN try {
#define GBS_END } catch (...) { PyErr_Clear(); } Py_RETURN_NONE;

// rotate_quantize(plan, x, want_y, out, stream) -> (codes, scales, y) or None
PyObject* rotate_quantize(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GBS_BEGIN
    const gbs_plan_t* plan;
    gbs_plan_info_t info;
    void* stream;
    int64_t rows, stride;
    if (n != 5 || !plan_of(a[0], &plan, &info)) Py_RETURN_NONE;
    const at::Tensor* x = cuda_tensor(a[1]);
    if (!x || !rows_of(x, info.d, &rows, &stride) || !stream_of(a[4], &stream)) Py_RETURN_NONE;
    const int dt = dtype_code(x->scalar_type());
    if (dt < 0) Py_RETURN_NONE;
    const at::Device device = x->device();
    if (a[3] != Py_None) {
        if (!PyTuple_Check(a[3]) || PyTuple_GET_SIZE(a[3]) != 3) Py_RETURN_NONE;
        PyObject *oc = PyTuple_GET_ITEM(a[3], 0), *os = PyTuple_GET_ITEM(a[3], 1), *oy = PyTuple_GET_ITEM(a[3], 2);
        const at::Tensor *codes = cuda_tensor(oc), *scales = cuda_tensor(os), *y = oy == Py_None ? nullptr : cuda_tensor(oy);
        if (!buffer_ok(codes, device, rows * info.code_bytes_per_row) || codes->scalar_type() != at::kByte ||
            !buffer_ok(scales, device, rows * info.scale_floats_per_row) || scales->scalar_type() != at::kFloat ||
            (oy != Py_None && (!buffer_ok(y, device, rows * info.d_pad) || y->scalar_type() != at::kFloat)))
            Py_RETURN_NONE;
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = gbs_rotate_quantize(plan, x->data_ptr(), dt, rows, stride, codes->data_ptr(), static_cast<float*>(scales->data_ptr()),
                                 y ? static_cast<float*>(y->data_ptr()) : nullptr, stream);
        Py_END_ALLOW_THREADS
        if (rc != GBS_OK) Py_RETURN_NONE;
        Py_INCREF(a[3]);
        return a[3];
    }
    const int want_y = PyObject_IsTrue(a[2]);
    if (want_y < 0) { PyErr_Clear(); Py_RETURN_NONE; }
    at::Tensor codes = empty2(rows, info.code_bytes_per_row, at::kByte, device);
    at::Tensor scales = empty2(rows, info.scale_floats_per_row, at::kFloat, device);
    at::Tensor y;
    if (want_y) y = empty2(rows, info.d_pad, at::kFloat, device);
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = gbs_rotate_quantize(plan, x->data_ptr(), dt, rows, stride, codes.data_ptr(), static_cast<float*>(scales.data_ptr()),
                             want_y ? static_cast<float*>(y.data_ptr()) : nullptr, stream);
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    PyObject* out = PyTuple_New(3);
    if (!out) return nullptr;
    PyTuple_SET_ITEM(out, 0, THPVariable_Wrap(std::move(codes)));
    PyTuple_SET_ITEM(out, 1, THPVariable_Wrap(std::move(scales)));
    if (want_y) PyTuple_SET_ITEM(out, 2, THPVariable_Wrap(std::move(y)));
    else PyTuple_SET_ITEM(out, 2, Py_NewRef(Py_None));
    return out;
    GBS_END
}

// an output the caller passed, or a new one [r, c] of the dtype asked for; false: not the regular call
bool output_of(PyObject* o, PyObject* dtype, int64_t r, int64_t c, const at::Device& device, at::Tensor* out, int* dt)
{
    if (o != Py_None) {
        const at::Tensor* t = cuda_tensor(o);
        if (!buffer_ok(t, device, r * c)) return false;
        *out = *t;
    } else {
        if (!THPDtype_Check(dtype)) return false;
        const at::ScalarType st = reinterpret_cast<THPDtype*>(dtype)->scalar_type;
        if (dtype_code(st) < 0) return false;
        *out = empty2(r, c, st, device);
    }
    *dt = dtype_code(out->scalar_type());
    return *dt >= 0;
}

// dequantize(plan, codes, scales, inverse, dtype, out, stream) -> tensor or None
PyObject* dequantize(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GBS_BEGIN
    const gbs_plan_t* plan;
    gbs_plan_info_t info;
    void* stream;
    if (n != 7 || !plan_of(a[0], &plan, &info)) Py_RETURN_NONE;
    const at::Tensor *codes = cuda_tensor(a[1]), *scales = cuda_tensor(a[2]);
    if (!codes || codes->dim() < 1) Py_RETURN_NONE;
    const int64_t rows = codes->size(0);
    const at::Device device = codes->device();
    const int inverse = PyObject_IsTrue(a[3]);
    if (inverse < 0) { PyErr_Clear(); Py_RETURN_NONE; }
    if (codes->scalar_type() != at::kByte || !buffer_ok(codes, device, rows * info.code_bytes_per_row) ||
        !buffer_ok(scales, device, rows * info.scale_floats_per_row) || scales->scalar_type() != at::kFloat ||
        !stream_of(a[6], &stream))
        Py_RETURN_NONE;
    at::Tensor out;
    int dt;
    if (!output_of(a[5], a[4], rows, inverse ? info.d : info.d_pad, device, &out, &dt)) Py_RETURN_NONE;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = gbs_dequantize(plan, codes->data_ptr(), static_cast<const float*>(scales->data_ptr()), rows, out.data_ptr(), dt,
                        inverse ? GBS_INVERSE_ROTATE : 0, stream);
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    if (a[5] != Py_None) return Py_NewRef(a[5]);
    return THPVariable_Wrap(std::move(out));
    GBS_END
}

// quantized_matmul(plan_x, codes_x, scales_x, plan_w, codes_w, scales_w, dtype, out, stream) -> tensor or None
PyObject* quantized_matmul(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GBS_BEGIN
    const gbs_plan_t *px, *pw;
    gbs_plan_info_t ix, iw;
    void* stream;
    if (n != 9 || !plan_of(a[0], &px, &ix) || !plan_of(a[3], &pw, &iw)) Py_RETURN_NONE;
    const at::Tensor *cx = cuda_tensor(a[1]), *sx = cuda_tensor(a[2]), *cw = cuda_tensor(a[4]), *sw = cuda_tensor(a[5]);
    if (!cx || !cw || cx->dim() < 1 || cw->dim() < 1) Py_RETURN_NONE;
    const int64_t n_tok = cx->size(0), n_out = cw->size(0);
    const at::Device device = cx->device();
    if (cx->scalar_type() != at::kByte || !buffer_ok(cx, device, n_tok * ix.code_bytes_per_row) ||
        !buffer_ok(sx, device, n_tok * ix.scale_floats_per_row) || sx->scalar_type() != at::kFloat ||
        cw->scalar_type() != at::kByte || !buffer_ok(cw, device, n_out * iw.code_bytes_per_row) ||
        !buffer_ok(sw, device, n_out * iw.scale_floats_per_row) || sw->scalar_type() != at::kFloat || !stream_of(a[8], &stream))
        Py_RETURN_NONE;
    at::Tensor out;
    int dt;
    // a caller's `out` may have any row stride: that form keeps the Python path's checks
    if (a[7] != Py_None) {
        const at::Tensor* t = cuda_tensor(a[7]);
        if (!t || t->dim() != 2 || t->size(0) != n_tok || t->size(1) != n_out) Py_RETURN_NONE;
    }
    if (!output_of(a[7], a[6], n_tok, n_out, device, &out, &dt)) Py_RETURN_NONE;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = gbs_quantized_matmul(px, cx->data_ptr(), static_cast<const float*>(sx->data_ptr()), n_tok, pw, cw->data_ptr(),
                              static_cast<const float*>(sw->data_ptr()), n_out, out.data_ptr(), dt, n_out, stream);
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    if (a[7] != Py_None) return Py_NewRef(a[7]);
    return THPVariable_Wrap(std::move(out));
    GBS_END
}

// clip_error(plan, x, alphas, stream) -> a new tensor of the K error sums, or None
PyObject* clip_error(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    GBS_BEGIN
    const gbs_plan_t* plan;
    gbs_plan_info_t info;
    void* stream;
    int64_t rows, stride;
    if (n != 4 || !plan_of(a[0], &plan, &info)) Py_RETURN_NONE;
    const at::Tensor* x = cuda_tensor(a[1]);
    if (!x || !rows_of(x, info.d, &rows, &stride) || !stream_of(a[3], &stream)) Py_RETURN_NONE;
    const int dt = dtype_code(x->scalar_type());
    if (dt < 0 || !PySequence_Check(a[2])) Py_RETURN_NONE;
    const Py_ssize_t K = PySequence_Size(a[2]);
    if (K < 1 || K > GBS_MAX_CANDIDATES) { PyErr_Clear(); Py_RETURN_NONE; }
    float alphas[GBS_MAX_CANDIDATES];
    for (Py_ssize_t i = 0; i < K; ++i) {
        PyObject* v = PySequence_GetItem(a[2], i);
        if (v) {
            alphas[i] = static_cast<float>(PyFloat_AsDouble(v));
            Py_DECREF(v);
        }
        if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
        if (!(alphas[i] > 0.f) || !(alphas[i] <= 1.f)) Py_RETURN_NONE;
    }
    // the sums are zeroed on the stream that adds to them
    at::Tensor err = at::detail::empty_cuda({static_cast<int64_t>(K)}, at::kDouble, x->device(), std::nullopt);
    int rc = GBS_ERR_CUDA;
    Py_BEGIN_ALLOW_THREADS
    if (cudaMemsetAsync(err.data_ptr(), 0, sizeof(double) * static_cast<size_t>(K), static_cast<cudaStream_t>(stream)) == cudaSuccess)
        rc = gbs_clip_error(plan, x->data_ptr(), dt, rows, stride, alphas, static_cast<int>(K), static_cast<double*>(err.data_ptr()),
                            nullptr, stream);
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    return THPVariable_Wrap(std::move(err));
    GBS_END
}

#define FAST(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(rotate_quantize), FAST(dequantize), FAST(quantized_matmul), FAST(clip_error), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
