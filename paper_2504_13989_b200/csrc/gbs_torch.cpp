// Native call path of the Python binding: what Plan's methods do per call -- check the tensors, allocate the outputs,
// look up the current stream, call the C ABI -- in one C function each.
//
// A call on a few rows is bound by the host: the kernel takes 3 us, and the same steps in Python took 17.5 us per call
// (two torch.empty at 2.3 us, torch.cuda.current_stream at 3.3 us, argument checks, ctypes marshalling at 0.8 us and the
// launch itself at 2 us).
//
// Every function here handles the regular call only and answers None for anything else (a tensor of another type or
// device, a shape or stride that needs a view, an output that is too small, a non-zero status): that call then takes
// the Python path, which raises the error or makes the view.  Nothing is enqueued before the checks have passed.
//
// Two ways in: the module's functions, for a caller that has the plan's handle alone, and method objects that stand in the class
// under the names of Plan's methods, over the Python functions they were.  A method object binds like a function, so that a
// bound method keeps its plan, a subclass may override it and a class attribute may be replaced; it finds the plan's handle in the
// Calls object of the instance.  It saves the Python frame around each call (0.9 of 5.3 us for 16 rows); what it does not handle it
// passes to the function it wraps.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <string.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include "gbs.h"

namespace {

// -1: not a type the library takes
int dtype_code(at::ScalarType t)
{
    return t == at::kFloat ? GBS_DTYPE_F32 : (t == at::kBFloat16 ? GBS_DTYPE_BF16 : -1);
}

struct PlanRef {
    const gbs_plan_t* plan;
    gbs_plan_info_t info;
};

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

// A C++ exception (an allocation that fails, a tensor without memory of its own) makes the call an irregular one.  Whatever can throw
// stands before the GIL is released: a tensor's pointer, in particular, is asked for before.
#define GBS_BEGIN try {
#define GBS_END } catch (...) { PyErr_Clear(); } Py_RETURN_NONE;

// rotate_quantize(plan, x, want_y, out, stream) -> (codes, scales, y) or None
// (a[0] is not looked at: the plan comes as `ref`)
PyObject* do_rotate_quantize(const PlanRef& ref, PyObject* const* a)
{
    GBS_BEGIN
    const gbs_plan_t* plan = ref.plan;
    const gbs_plan_info_t& info = ref.info;
    void* stream;
    int64_t rows, stride;
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
        void *xp = x->data_ptr(), *cp = codes->data_ptr(), *sp = scales->data_ptr(), *yp = y ? y->data_ptr() : nullptr;
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = gbs_rotate_quantize(plan, xp, dt, rows, stride, cp, static_cast<float*>(sp), static_cast<float*>(yp), stream);
        Py_END_ALLOW_THREADS
        if (rc != GBS_OK) Py_RETURN_NONE;
        Py_INCREF(a[3]);
        return a[3];
    }
    const int want_y = PyObject_IsTrue(a[2]);
    if (want_y < 0) { PyErr_Clear(); Py_RETURN_NONE; }
    // two allocations (0.5 us each): outputs that shared one would be saved, kept and freed together
    at::Tensor codes = empty2(rows, info.code_bytes_per_row, at::kByte, device);
    at::Tensor scales = empty2(rows, info.scale_floats_per_row, at::kFloat, device), y;
    if (want_y) y = empty2(rows, info.d_pad, at::kFloat, device);
    void *xp = x->data_ptr(), *cp = codes.data_ptr(), *sp = scales.data_ptr(), *yp = want_y ? y.data_ptr() : nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = gbs_rotate_quantize(plan, xp, dt, rows, stride, cp, static_cast<float*>(sp), static_cast<float*>(yp), stream);
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
        if (dtype && !THPDtype_Check(dtype)) return false;
        const at::ScalarType st = dtype ? reinterpret_cast<THPDtype*>(dtype)->scalar_type : at::kFloat;      // null: not given
        if (dtype_code(st) < 0) return false;
        *out = empty2(r, c, st, device);
    }
    *dt = dtype_code(out->scalar_type());
    return *dt >= 0;
}

// dequantize(plan, codes, scales, inverse, dtype, out, stream) -> tensor or None
PyObject* do_dequantize(const PlanRef& ref, PyObject* const* a)
{
    GBS_BEGIN
    const gbs_plan_t* plan = ref.plan;
    const gbs_plan_info_t& info = ref.info;
    void* stream;
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
    void *cp = codes->data_ptr(), *sp = scales->data_ptr(), *op = out.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = gbs_dequantize(plan, cp, static_cast<const float*>(sp), rows, op, dt, inverse ? GBS_INVERSE_ROTATE : 0, stream);
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    if (a[5] != Py_None) return Py_NewRef(a[5]);
    return THPVariable_Wrap(std::move(out));
    GBS_END
}

// quantized_matmul(plan_x, codes_x, scales_x, plan_w, codes_w, scales_w, dtype, out, stream) -> tensor or None
PyObject* do_quantized_matmul(const PlanRef& ref, PyObject* const* a)
{
    GBS_BEGIN
    const gbs_plan_t *px = ref.plan, *pw;
    const gbs_plan_info_t& ix = ref.info;
    gbs_plan_info_t iw;
    void* stream;
    if (!plan_of(a[3], &pw, &iw)) Py_RETURN_NONE;
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
    void *cxp = cx->data_ptr(), *sxp = sx->data_ptr(), *cwp = cw->data_ptr(), *swp = sw->data_ptr(), *op = out.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = gbs_quantized_matmul(px, cxp, static_cast<const float*>(sxp), n_tok, pw, cwp, static_cast<const float*>(swp), n_out, op, dt, n_out,
                              stream);
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    if (a[7] != Py_None) return Py_NewRef(a[7]);
    return THPVariable_Wrap(std::move(out));
    GBS_END
}

// clip_error(plan, x, alphas, stream) -> a new tensor of the K error sums, or None
PyObject* do_clip_error(const PlanRef& ref, PyObject* const* a)
{
    GBS_BEGIN
    const gbs_plan_t* plan = ref.plan;
    const gbs_plan_info_t& info = ref.info;
    void* stream;
    int64_t rows, stride;
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
    void *xp = x->data_ptr(), *ep = err.data_ptr();
    int rc = GBS_ERR_CUDA;
    Py_BEGIN_ALLOW_THREADS
    if (cudaMemsetAsync(ep, 0, sizeof(double) * static_cast<size_t>(K), static_cast<cudaStream_t>(stream)) == cudaSuccess)
        rc = gbs_clip_error(plan, xp, dt, rows, stride, alphas, static_cast<int>(K), static_cast<double*>(ep), nullptr, stream);
    else
        cudaGetLastError();                               // the Python path reports it; later launches of others must not
    Py_END_ALLOW_THREADS
    if (rc != GBS_OK) Py_RETURN_NONE;
    return THPVariable_Wrap(std::move(err));
    GBS_END
}

// ---- the module's functions: the plan's handle first
template <PyObject* (*F)(const PlanRef&, PyObject* const*), int N>
PyObject* with_handle(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    PlanRef ref;
    if (n != N || !plan_of(a[0], &ref.plan, &ref.info)) Py_RETURN_NONE;
    return F(ref, a);
}

// ---- Calls(handle): the plan's handle and sizes for the methods below, until clear()
struct Calls {
    PyObject_HEAD
    PlanRef ref;              // ref.plan is null once the plan is closed
};
PyTypeObject* calls_type = nullptr;

int calls_init(PyObject* self, PyObject* args, PyObject*)
{
    Calls* c = reinterpret_cast<Calls*>(self);
    PyObject *handle, *unused;
    if (!PyArg_ParseTuple(args, "O|O", &handle, &unused)) return -1;
    if (!plan_of(handle, &c->ref.plan, &c->ref.info)) {
        c->ref.plan = nullptr;
        PyErr_SetString(PyExc_ValueError, "gbs: not a plan handle");
        return -1;
    }
    return 0;
}
void calls_dealloc(PyObject* self)
{
    PyTypeObject* type = Py_TYPE(self);
    type->tp_free(self);
    Py_DECREF(type);
}
PyObject* calls_clear(PyObject* self, PyObject*)
{
    reinterpret_cast<Calls*>(self)->ref.plan = nullptr;
    Py_RETURN_NONE;
}

// A method: the names of its arguments in Plan's order, how many must be given, and what to do with them.
struct Method {
    const char* name;
    int count, required;
    const char* args[8];
    PyObject* (*call)(const PlanRef&, PyObject* const* given);
};

PyObject* or_none(PyObject* o) { return o ? o : Py_None; }

constexpr Method ROTATE = {"rotate_quantize", 4, 1, {"x", "want_y", "out", "stream"}, [](const PlanRef& r, PyObject* const* g) {
    PyObject* a[5] = {nullptr, g[0], g[1] ? g[1] : Py_False, or_none(g[2]), or_none(g[3])};
    return do_rotate_quantize(r, a);
}};
constexpr Method DEQUANTIZE = {"dequantize", 6, 2, {"codes", "scales", "inverse", "dtype", "out", "stream"}, [](const PlanRef& r, PyObject* const* g) {
    PyObject* a[7] = {nullptr, g[0], g[1], g[2] ? g[2] : Py_False, g[3], or_none(g[4]), or_none(g[5])};
    return do_dequantize(r, a);
}};
constexpr Method MATMUL = {"quantized_matmul", 8, 5, {"codes_x", "scales_x", "plan_w", "codes_w", "scales_w", "dtype", "out", "stream"},
                           [](const PlanRef& r, PyObject* const* g) -> PyObject* {
    PyObject* handle = PyObject_GetAttrString(g[2], "handle");
    if (!handle) { PyErr_Clear(); Py_RETURN_NONE; }
    PyObject* a[9] = {nullptr, g[0], g[1], handle, g[3], g[4], g[5], or_none(g[6]), or_none(g[7])};
    PyObject* out = do_quantized_matmul(r, a);
    Py_DECREF(handle);
    return out;
}};
constexpr Method CLIP = {"clip_error", 5, 2, {"x", "alphas", "want_rows", "err_sum", "stream"}, [](const PlanRef& r, PyObject* const* g) -> PyObject* {
    if ((g[2] && g[2] != Py_False) || (g[3] && g[3] != Py_None)) Py_RETURN_NONE;
    PyObject* a[4] = {nullptr, g[0], g[1], or_none(g[4])};
    return do_clip_error(r, a);
}};

// ---- method(name, function, alloc_outputs): a function of Plan with the regular call in front of it
struct MethodObject {
    PyObject_HEAD
    vectorcallfunc vectorcall;
    const Method* method;
    PyObject* wrapped;
    PyObject* alloc;          // Plan.alloc_outputs, or null where the call allocates without it
};
PyObject *name_calls = nullptr, *name_alloc = nullptr;

// whether the plan's outputs come from Plan's own alloc_outputs (a subclass or an instance may have another)
bool own_alloc(PyObject* plan, PyObject* alloc)
{
    PyObject* f = PyObject_GetAttr(plan, name_alloc);
    if (!f) { PyErr_Clear(); return false; }
    const bool own = PyMethod_Check(f) && PyMethod_GET_FUNCTION(f) == alloc;
    Py_DECREF(f);
    return own;
}

PyObject* method_call(PyObject* self, PyObject* const* args, size_t nargsf, PyObject* kwnames)
{
    const MethodObject* o = reinterpret_cast<MethodObject*>(self);
    const Method& M = *o->method;
    const Py_ssize_t n = PyVectorcall_NARGS(nargsf) - 1, nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    PyObject* calls = n >= 0 ? PyObject_GetAttr(args[0], name_calls) : nullptr;
    if (!calls) PyErr_Clear();
    PyObject* given[8] = {nullptr};
    bool regular = calls && Py_TYPE(calls) == calls_type && reinterpret_cast<Calls*>(calls)->ref.plan && n <= M.count;
    for (Py_ssize_t i = 0; regular && i < n; ++i) given[i] = args[1 + i];
    for (Py_ssize_t k = 0; regular && k < nk; ++k) {
        int at = -1;
        for (int i = 0; i < M.count && at < 0; ++i)
            if (PyUnicode_CompareWithASCIIString(PyTuple_GET_ITEM(kwnames, k), M.args[i]) == 0) at = i;
        regular = at >= 0 && !given[at];
        if (regular) given[at] = args[1 + n + k];
    }
    for (int i = 0; regular && i < M.required; ++i) regular = given[i] != nullptr;
    if (regular && o->alloc) regular = own_alloc(args[0], o->alloc);
    PyObject* out = nullptr;
    if (regular) {
        const PlanRef ref = reinterpret_cast<Calls*>(calls)->ref;      // the caller's argument keeps the plan
        out = M.call(ref, given);
        if (out == Py_None) { Py_DECREF(out); regular = false; }
    }
    Py_XDECREF(calls);
    return regular ? out : PyObject_Vectorcall(o->wrapped, args, nargsf, kwnames);
}


PyObject* method_get(PyObject* self, PyObject* obj, PyObject*) { return obj ? PyMethod_New(self, obj) : Py_NewRef(self); }
// name, documentation, signature, module: the wrapped function's
PyObject* method_getattro(PyObject* self, PyObject* name)
{
    PyObject* wrapped = reinterpret_cast<MethodObject*>(self)->wrapped;
    if (PyUnicode_CompareWithASCIIString(name, "__wrapped__") == 0) return Py_NewRef(wrapped);
    if (PyUnicode_CompareWithASCIIString(name, "__class__") == 0 || PyUnicode_CompareWithASCIIString(name, "__call__") == 0)
        return PyObject_GenericGetAttr(self, name);
    return PyObject_GetAttr(wrapped, name);
}
int method_traverse(PyObject* self, visitproc visit, void* arg)
{
    MethodObject* o = reinterpret_cast<MethodObject*>(self);
    Py_VISIT(Py_TYPE(self));
    Py_VISIT(o->wrapped);
    Py_VISIT(o->alloc);
    return 0;
}
int method_clear(PyObject* self)
{
    MethodObject* o = reinterpret_cast<MethodObject*>(self);
    Py_CLEAR(o->wrapped);
    Py_CLEAR(o->alloc);
    return 0;
}
void method_dealloc(PyObject* self)
{
    PyTypeObject* type = Py_TYPE(self);
    PyObject_GC_UnTrack(self);
    method_clear(self);
    type->tp_free(self);
    Py_DECREF(type);
}
PyTypeObject* method_type = nullptr;
const Method* const METHODS[] = {&ROTATE, &DEQUANTIZE, &MATMUL, &CLIP};

PyObject* make_method(PyObject*, PyObject* args)
{
    const char* name;
    PyObject *wrapped, *alloc;
    if (!PyArg_ParseTuple(args, "sOO", &name, &wrapped, &alloc)) return nullptr;
    const Method* m = nullptr;
    for (const Method* c : METHODS)
        if (strcmp(name, c->name) == 0) m = c;
    if (!m) { PyErr_Format(PyExc_ValueError, "gbs: no native method '%s'", name); return nullptr; }
    MethodObject* o = reinterpret_cast<MethodObject*>(method_type->tp_alloc(method_type, 0));
    if (!o) return nullptr;
    o->vectorcall = method_call;
    o->method = m;
    o->wrapped = Py_NewRef(wrapped);
    o->alloc = alloc == Py_None ? nullptr : Py_NewRef(alloc);
    return reinterpret_cast<PyObject*>(o);
}

template <class F> PyCFunction cfunc(F f) { return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)); }

PyMethodDef calls_methods[] = {{"clear", calls_clear, METH_NOARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyType_Slot calls_slots[] = {{Py_tp_init, reinterpret_cast<void*>(calls_init)}, {Py_tp_dealloc, reinterpret_cast<void*>(calls_dealloc)},
                             {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)}, {Py_tp_methods, calls_methods}, {0, nullptr}};
PyType_Spec calls_spec = {"paper_2504_13989_b200._native.Calls", sizeof(Calls), 0, Py_TPFLAGS_DEFAULT, calls_slots};

PyMemberDef method_members[] = {{"__vectorcalloffset__", Py_T_PYSSIZET, offsetof(MethodObject, vectorcall), Py_READONLY, nullptr},
                                {nullptr, 0, 0, 0, nullptr}};
PyType_Slot method_slots[] = {{Py_tp_dealloc, reinterpret_cast<void*>(method_dealloc)}, {Py_tp_traverse, reinterpret_cast<void*>(method_traverse)},
                              {Py_tp_clear, reinterpret_cast<void*>(method_clear)}, {Py_tp_call, reinterpret_cast<void*>(PyVectorcall_Call)},
                              {Py_tp_descr_get, reinterpret_cast<void*>(method_get)}, {Py_tp_getattro, reinterpret_cast<void*>(method_getattro)},
                              {Py_tp_members, method_members}, {0, nullptr}};
PyType_Spec method_spec = {"paper_2504_13989_b200._native.Method", sizeof(MethodObject), 0,
                           Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_GC | Py_TPFLAGS_HAVE_VECTORCALL | Py_TPFLAGS_METHOD_DESCRIPTOR |
                               Py_TPFLAGS_DISALLOW_INSTANTIATION, method_slots};

PyMethodDef methods[] = {{ROTATE.name, cfunc(with_handle<do_rotate_quantize, 5>), METH_FASTCALL, nullptr},
                         {DEQUANTIZE.name, cfunc(with_handle<do_dequantize, 7>), METH_FASTCALL, nullptr},
                         {MATMUL.name, cfunc(with_handle<do_quantized_matmul, 9>), METH_FASTCALL, nullptr},
                         {CLIP.name, cfunc(with_handle<do_clip_error, 4>), METH_FASTCALL, nullptr},
                         {"method", make_method, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    name_calls = PyUnicode_InternFromString("_calls");
    name_alloc = PyUnicode_InternFromString("alloc_outputs");
    calls_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&calls_spec));
    method_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&method_spec));
    PyObject* m = PyModule_Create(&module);
    if (!name_calls || !name_alloc || !calls_type || !method_type || !m ||
        PyModule_AddObjectRef(m, "Calls", reinterpret_cast<PyObject*>(calls_type)) < 0) {
        Py_XDECREF(m);
        return nullptr;
    }
    return m;
}
