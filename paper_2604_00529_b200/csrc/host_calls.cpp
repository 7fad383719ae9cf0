// The plain case of the binding's per-tensor calls as native code (module _mxq_host): arguments that are ordinary
// contiguous CUDA tensors, on the current stream.  One call checks them, allocates the outputs that were not
// given and calls the C ABI; through Python attribute calls and ctypes the same took 2 - 3 times the launch itself.
//
// Every function returns None -- having enqueued nothing -- for anything else: other types and devices, tensor
// subclasses, tensors without storage (vmap, grad and functionalization wrappers), active torch modes, a stream
// argument, a status other than MXQ_OK (a failed launch of slice_scale_multi, which may follow others, is raised at
// once).  The caller in binding.py then takes its general path, which handles the case or raises the error it
// always raised.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/jit/frontend/tracer.h>

#include "../../include/mxq.h"

namespace {

// ---- the C ABI of the loaded library (addresses from the binding, see bind) -----------------------------

struct Api {
    decltype(&mxq_quantize) quantize;
    decltype(&mxq_slice_scale) slice_scale;
    decltype(&mxq_slice_scale_multi) slice_scale_multi;
    decltype(&mxq_dequantize) dequantize;
    decltype(&mxq_tiled_scales_bytes) tiled_scales_bytes;
    decltype(&mxq_quantize_tiled) quantize_tiled;
    decltype(&mxq_slice_scale_tiled) slice_scale_tiled;
    decltype(&mxq_fake_quant) fake_quant;
    decltype(&mxq_fake_quant_bwd) fake_quant_bwd;
    decltype(&mxq_codes_bytes) codes_bytes;
} api;

PyObject* formats = nullptr;          // the binding's name -> id dict
PyTypeObject* parameter = nullptr;    // torch.nn.Parameter
PyObject* mxq_error = nullptr;        // the binding's MxqError(status, what)

// ---- arguments ------------------------------------------------------------------------------------------

bool modes_active()
{
    return c10::impl::TorchDispatchModeTLS::any_modes_set() || at::impl::torch_function_mode_enabled();
}

// An ordinary contiguous CUDA tensor with storage, or null.
const at::Tensor* plain(PyObject* o)
{
    if (!THPVariable_CheckExact(o) && Py_TYPE(o) != parameter) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.unsafeGetTensorImpl()->is_python_dispatch() || !t.has_storage() ||
        t.layout() != at::kStrided || !t.is_contiguous())
        return nullptr;
    return &t;
}

bool dtype_id(at::ScalarType t, int* id)
{
    if (t == at::kFloat) *id = MXQ_F32;
    else if (t == at::kBFloat16) *id = MXQ_BF16;
    else return false;
    return true;
}

bool dtype_id(const at::Tensor& t, int* id) { return dtype_id(t.scalar_type(), id); }

bool as_int(PyObject* o, int* v)
{
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    const long x = PyLong_AsLongAndOverflow(o, &overflow);
    if (overflow || x != (int)x) return false;
    *v = (int)x;
    return true;
}

bool as_count(PyObject* o, int64_t* v)
{
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    *v = PyLong_AsLongLongAndOverflow(o, &overflow);
    return !overflow && *v >= 0;
}

bool format_id(PyObject* o, int* v)
{
    if (!PyUnicode_CheckExact(o)) return false;
    PyObject* id = PyDict_GetItemWithError(formats, o);      // borrowed
    if (!id) {
        PyErr_Clear();
        return false;
    }
    return as_int(id, v);
}

mxq_stream current_stream() { return static_cast<mxq_stream>(c10::cuda::getCurrentCUDAStream().stream()); }

// The interpreter's lock is released while a call allocates and enqueues: a launch waits when the queue is full, an
// allocation may wait for the device, and other Python threads (or a host callback that the queue itself waits for)
// have to run meanwhile.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    Unlocked() = default;
    Unlocked(const Unlocked&) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};

// What `fn` returns, run without the lock.
template <class FN>
int unlocked(FN&& fn)
{
    Unlocked u;
    return fn();
}

// An output argument: the given tensor, or a new one when it is None.
struct Output {
    const at::Tensor* tensor = nullptr;
    at::Tensor made;

    bool take(PyObject* o) { return o == Py_None || (tensor = plain(o)); }
    void make(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like)
    {
        if (!tensor) tensor = &(made = at::empty(sizes, at::TensorOptions().dtype(type).device(like.device())));
    }
    void make_like(const at::Tensor& like)
    {
        if (!tensor) tensor = &(made = at::empty_like(like));
    }
    void* data() const { return tensor->data_ptr(); }
    uint8_t* bytes() const { return static_cast<uint8_t*>(tensor->data_ptr()); }
    PyObject* result(PyObject* given) const
    {
        if (given == Py_None) return THPVariable_Wrap(made);
        Py_INCREF(given);
        return given;
    }
};

PyObject* pair(PyObject* a, PyObject* b)
{
    PyObject* t = a && b ? PyTuple_New(2) : nullptr;
    if (!t) {
        Py_XDECREF(a);
        Py_XDECREF(b);
        return nullptr;
    }
    PyTuple_SET_ITEM(t, 0, a);
    PyTuple_SET_ITEM(t, 1, b);
    return t;
}

uint8_t* bytes(const at::Tensor& t) { return static_cast<uint8_t*>(t.data_ptr()); }

// Sets MxqError(rc, what) as the Python error.
PyObject* raise_mxq_error(int rc, const char* what)
{
    if (PyObject* e = PyObject_CallFunction(mxq_error, "is", rc, what)) {
        PyErr_SetObject(mxq_error, e);
        Py_DECREF(e);
    }
    return nullptr;
}

#define GENERAL_UNLESS(cond) \
    if (!(cond)) Py_RETURN_NONE

// ---- the calls ------------------------------------------------------------------------------------------

// quantize(src, fmt, block, codes, scales, stream)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int fmt, block, dt;
    GENERAL_UNLESS(nargs == 6 && a[5] == Py_None && format_id(a[1], &fmt) && as_int(a[2], &block) && block > 0 && !modes_active());
    const at::Tensor* src = plain(a[0]);
    Output codes, scales;
    GENERAL_UNLESS(src && dtype_id(*src, &dt) && codes.take(a[3]) && scales.take(a[4]));
    const int rc = unlocked([&] {
        const int64_t n = src->numel();
        codes.make({(int64_t)api.codes_bytes((size_t)n, fmt)}, at::kByte, *src);
        scales.make({n / block}, at::kByte, *src);
        return api.quantize(src->data_ptr(), dt, (size_t)n, fmt, block, codes.data(), scales.bytes(), current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return pair(codes.result(a[3]), scales.result(a[4]));
    END_HANDLE_TH_ERRORS
}

// slice_scale(codes, scales, n, src_fmt, dst_fmt, block, out_codes, out_scales, stream)
PyObject* slice_scale(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int src_fmt, dst_fmt, block;
    int64_t n;
    GENERAL_UNLESS(nargs == 9 && a[8] == Py_None && as_count(a[2], &n) && format_id(a[3], &src_fmt) && format_id(a[4], &dst_fmt) &&
                   as_int(a[5], &block) && block > 0 && !modes_active());
    const at::Tensor *codes = plain(a[0]), *scales = plain(a[1]);
    Output oc, os;
    GENERAL_UNLESS(codes && scales && oc.take(a[6]) && os.take(a[7]));
    const int rc = unlocked([&] {
        oc.make({(int64_t)api.codes_bytes((size_t)n, dst_fmt)}, at::kByte, *codes);
        os.make({n / block}, at::kByte, *codes);
        return api.slice_scale(codes->data_ptr(), bytes(*scales), (size_t)n, block, src_fmt, dst_fmt, oc.data(), os.bytes(),
                               current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return pair(oc.result(a[6]), os.result(a[7]));
    END_HANDLE_TH_ERRORS
}

// slice_scale_multi(codes, scales, n, src_fmt, dst_fmts, block, outs, stream), outs None
PyObject* slice_scale_multi(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int src_fmt, block;
    int64_t n;
    GENERAL_UNLESS(nargs == 8 && a[6] == Py_None && a[7] == Py_None && as_count(a[2], &n) && format_id(a[3], &src_fmt) &&
                   as_int(a[5], &block) && block > 0 && !modes_active());
    GENERAL_UNLESS(PyList_CheckExact(a[4]) || PyTuple_CheckExact(a[4]));
    const Py_ssize_t k = PySequence_Fast_GET_SIZE(a[4]);
    GENERAL_UNLESS(k <= MXQ_MULTI_TARGETS_MAX);
    const at::Tensor *codes = plain(a[0]), *scales = plain(a[1]);
    GENERAL_UNLESS(codes && scales);
    int fmts[MXQ_MULTI_TARGETS_MAX];
    for (Py_ssize_t t = 0; t < k; ++t) GENERAL_UNLESS(format_id(PySequence_Fast_GET_ITEM(a[4], t), &fmts[t]));
    Output oc[MXQ_MULTI_TARGETS_MAX], os[MXQ_MULTI_TARGETS_MAX];
    const int rc = unlocked([&] {
        void* pc[MXQ_MULTI_TARGETS_MAX];
        uint8_t* ps[MXQ_MULTI_TARGETS_MAX];
        for (Py_ssize_t t = 0; t < k; ++t) {
            oc[t].make({(int64_t)api.codes_bytes((size_t)n, fmts[t])}, at::kByte, *codes);
            os[t].make({n / block}, at::kByte, *codes);
            pc[t] = oc[t].data();
            ps[t] = os[t].bytes();
        }
        return api.slice_scale_multi(codes->data_ptr(), bytes(*scales), (size_t)n, block, src_fmt, (int)k, fmts, pc, ps,
                                     current_stream());
    });
    // (other launches of the call may precede the one that failed: the general path would enqueue them again)
    if (rc == MXQ_ERR_CUDA) return raise_mxq_error(rc, "mxq_slice_scale_multi");
    GENERAL_UNLESS(rc == MXQ_OK);
    PyObject* list = PyList_New(k);
    if (!list) return nullptr;
    for (Py_ssize_t t = 0; t < k; ++t) {
        PyObject* p = pair(oc[t].result(Py_None), os[t].result(Py_None));
        if (!p) {
            Py_DECREF(list);
            return nullptr;
        }
        PyList_SET_ITEM(list, t, p);
    }
    return list;
    END_HANDLE_TH_ERRORS
}

// dequantize(codes, scales, n, fmt, block, dtype, dst, stream)
PyObject* dequantize(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int fmt, block, dt;
    int64_t n;
    GENERAL_UNLESS(nargs == 8 && a[7] == Py_None && as_count(a[2], &n) && format_id(a[3], &fmt) && as_int(a[4], &block) &&
                   !modes_active());
    const at::Tensor *codes = plain(a[0]), *scales = plain(a[1]);
    Output dst;
    GENERAL_UNLESS(codes && scales && dst.take(a[6]));
    at::ScalarType type = at::kFloat;
    if (dst.tensor) {
        GENERAL_UNLESS(dtype_id(*dst.tensor, &dt));
    } else {
        GENERAL_UNLESS(THPDtype_Check(a[5]));
        type = reinterpret_cast<THPDtype*>(a[5])->scalar_type;
        GENERAL_UNLESS(dtype_id(type, &dt));
    }
    const int rc = unlocked([&] {
        dst.make({n}, type, *codes);
        return api.dequantize(codes->data_ptr(), bytes(*scales), (size_t)n, fmt, block, dst.data(), dt, current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return dst.result(a[6]);
    END_HANDLE_TH_ERRORS
}

// quantize_tiled(src, fmt, block, codes, tiled_scales, stream)
PyObject* quantize_tiled(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int fmt, block, dt;
    GENERAL_UNLESS(nargs == 6 && a[5] == Py_None && format_id(a[1], &fmt) && as_int(a[2], &block) && !modes_active());
    const at::Tensor* src = plain(a[0]);
    Output codes, scales;
    GENERAL_UNLESS(src && dtype_id(*src, &dt) && src->dim() == 2 && codes.take(a[3]) && scales.take(a[4]));
    const int rc = unlocked([&] {
        const int64_t rows = src->size(0), cols = src->size(1);
        codes.make({(int64_t)api.codes_bytes((size_t)(rows * cols), fmt)}, at::kByte, *src);
        scales.make({(int64_t)api.tiled_scales_bytes((size_t)rows, (size_t)(cols / 32))}, at::kByte, *src);
        return api.quantize_tiled(src->data_ptr(), dt, (size_t)rows, (size_t)cols, fmt, block, codes.data(), scales.bytes(),
                                  current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return pair(codes.result(a[3]), scales.result(a[4]));
    END_HANDLE_TH_ERRORS
}

// slice_scale_tiled(codes, scales, rows, cols, src_fmt, dst_fmt, block, out_codes, out_tiled_scales, stream)
PyObject* slice_scale_tiled(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int src_fmt, dst_fmt, block;
    int64_t rows, cols;
    GENERAL_UNLESS(nargs == 10 && a[9] == Py_None && as_count(a[2], &rows) && as_count(a[3], &cols) && rows < (1ll << 31) &&
                   cols < (1ll << 31) && format_id(a[4], &src_fmt) && format_id(a[5], &dst_fmt) && as_int(a[6], &block) &&
                   !modes_active());
    const at::Tensor *codes = plain(a[0]), *scales = plain(a[1]);
    Output oc, os;
    GENERAL_UNLESS(codes && scales && oc.take(a[7]) && os.take(a[8]));
    const int rc = unlocked([&] {
        oc.make({(int64_t)api.codes_bytes((size_t)(rows * cols), dst_fmt)}, at::kByte, *codes);
        os.make({(int64_t)api.tiled_scales_bytes((size_t)rows, (size_t)(cols / 32))}, at::kByte, *codes);
        return api.slice_scale_tiled(codes->data_ptr(), bytes(*scales), (size_t)rows, (size_t)cols, block, src_fmt, dst_fmt, oc.data(),
                                     os.bytes(), current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return pair(oc.result(a[7]), os.result(a[8]));
    END_HANDLE_TH_ERRORS
}

// fake_quant(src, fmt, block, mode, dst, stream)
PyObject* fake_quant(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int fmt, block, mode, dt;
    GENERAL_UNLESS(nargs == 6 && a[5] == Py_None && format_id(a[1], &fmt) && as_int(a[2], &block) && as_int(a[3], &mode) &&
                   !modes_active());
    const at::Tensor* src = plain(a[0]);
    Output dst;
    GENERAL_UNLESS(src && dtype_id(*src, &dt) && dst.take(a[4]));
    const int rc = unlocked([&] {
        dst.make_like(*src);
        return api.fake_quant(src->data_ptr(), dt, (size_t)src->numel(), fmt, block, mode, dst.data(), current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return dst.result(a[4]);
    END_HANDLE_TH_ERRORS
}

// fake_quant_bwd(grad_out, grad_in, stream)
PyObject* fake_quant_bwd(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int dt;
    GENERAL_UNLESS(nargs == 3 && a[2] == Py_None && !modes_active());
    const at::Tensor* g = plain(a[0]);
    Output dst;
    GENERAL_UNLESS(g && dtype_id(*g, &dt) && dst.take(a[1]));
    const int rc = unlocked([&] {
        dst.make_like(*g);
        return api.fake_quant_bwd(g->data_ptr(), dt, (size_t)g->numel(), dst.data(), current_stream());
    });
    GENERAL_UNLESS(rc == MXQ_OK);
    return dst.result(a[1]);
    END_HANDLE_TH_ERRORS
}

// ---- calls with all arguments marshalled beforehand --------------------------------------------------------

// run_prepared(kind, arguments as a bytes object of int64s): the status.  (PreparedCall in binding.py; kinds in its
// _PREPARED.)
PyObject* run_prepared(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    if (nargs != 2 || !PyLong_CheckExact(a[0]) || !PyBytes_CheckExact(a[1]) || PyBytes_GET_SIZE(a[1]) < 9 * (Py_ssize_t)sizeof(int64_t)) {
        PyErr_SetString(PyExc_TypeError, "run_prepared(kind, arguments)");
        return nullptr;
    }
    int64_t v[9];
    memcpy(v, PyBytes_AS_STRING(a[1]), sizeof(v));
    auto ptr = [&](int i) { return reinterpret_cast<void*>(v[i]); };
    auto u8 = [&](int i) { return reinterpret_cast<uint8_t*>(v[i]); };
    auto num = [&](int i) { return (int)v[i]; };
    const long kind = PyLong_AsLong(a[0]);
    const int rc = unlocked([&] {
        const mxq_stream s = current_stream();
        switch (kind) {
        case 0: return api.quantize(ptr(0), num(1), (size_t)v[2], num(3), num(4), ptr(5), u8(6), s);
        case 1: return api.slice_scale(ptr(0), u8(1), (size_t)v[2], num(3), num(4), num(5), ptr(6), u8(7), s);
        case 2: return api.dequantize(ptr(0), u8(1), (size_t)v[2], num(3), num(4), ptr(5), num(6), s);
        case 3: return api.fake_quant(ptr(0), num(1), (size_t)v[2], num(3), num(4), num(5), ptr(6), s);
        case 4: return api.fake_quant_bwd(ptr(0), num(1), (size_t)v[2], ptr(3), s);
        default: return (int)MXQ_ERR_FORMAT;
        }
    });
    return PyLong_FromLong(rc);
    END_HANDLE_TH_ERRORS
}

// ---- the straight-through estimator as an autograd node -----------------------------------------------------

struct NotPlain {};                    // the launch was refused: the general path raises the error

// MxqError(rc, what) out of a backward pass, which runs without the interpreter's lock and on a thread of its own.
[[noreturn]] void throw_mxq_error(int rc, const char* what)
{
    pybind11::gil_scoped_acquire lock;
    raise_mxq_error(rc, what);
    python_error raised;
    raised.persist();
    throw python_error(std::move(raised));
}

struct FakeQuantSTE : torch::autograd::Function<FakeQuantSTE> {
    static at::Tensor forward(torch::autograd::AutogradContext* ctx, const at::Tensor& x, int64_t fmt, int64_t block, int64_t mode,
                              bool copy_grad)
    {
        ctx->saved_data["copy_grad"] = copy_grad;
        int dt = 0;
        dtype_id(x, &dt);
        at::Tensor y = at::empty_like(x);
        if (api.fake_quant(x.data_ptr(), dt, (size_t)x.numel(), (int)fmt, (int)block, (int)mode, y.data_ptr(), current_stream()) != MXQ_OK)
            throw NotPlain{};
        return y;
    }

    static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, torch::autograd::variable_list grads)
    {
        at::Tensor g = grads[0];       // identity: the incoming gradient itself, or a copy of it
        if (ctx->saved_data["copy_grad"].toBool()) {
            const at::Tensor src = g.contiguous();
            int dt = 0;
            TORCH_CHECK_TYPE(dtype_id(src, &dt), "mxq tensors are float32 or bfloat16, got ", src.scalar_type());
            TORCH_CHECK_VALUE(src.is_cuda(), "grad_out must be a CUDA tensor (libmxq has no CPU path)");
            at::NoGradGuard no_grad;
            at::Tensor copy = at::empty_like(src);
            const int rc = api.fake_quant_bwd(src.data_ptr(), dt, (size_t)src.numel(), copy.data_ptr(), current_stream());
            if (rc != MXQ_OK) throw_mxq_error(rc, "mxq_fake_quant_bwd");
            g = copy;
        }
        return {g, at::Tensor(), at::Tensor(), at::Tensor(), at::Tensor()};
    }
};

// fake_quant_ste(x, fmt, block, mode, copy_grad)
PyObject* fake_quant_ste(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    int fmt, block, mode, dt;
    GENERAL_UNLESS(nargs == 5 && format_id(a[1], &fmt) && as_int(a[2], &block) && as_int(a[3], &mode) && PyBool_Check(a[4]) &&
                   !modes_active() && !torch::jit::tracer::isTracing());
    const at::Tensor* x = plain(a[0]);
    // (forward-mode AD and functorch transforms: the Python function says what it supports)
    const bool transforms = c10::impl::tls_is_dispatch_key_included(c10::DispatchKey::FuncTorchDynamicLayerFrontMode);
    GENERAL_UNLESS(x && dtype_id(*x, &dt) && !x->_fw_grad(0).defined() && !transforms);
    at::Tensor y;
    try {
        Unlocked u;
        y = FakeQuantSTE::apply(*x, (int64_t)fmt, (int64_t)block, (int64_t)mode, a[4] == Py_True);
    } catch (const NotPlain&) {
        Py_RETURN_NONE;
    }
    return THPVariable_Wrap(y);
    END_HANDLE_TH_ERRORS
}

// bind(addresses by name, formats, torch.nn.Parameter, MxqError)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    if (nargs != 4 || !PyDict_Check(a[0]) || !PyDict_Check(a[1]) || !PyType_Check(a[2]) || !PyType_Check(a[3])) {
        PyErr_SetString(PyExc_TypeError, "bind(addresses, formats, parameter type, error type)");
        return nullptr;
    }
    bool ok = true;
    auto take = [&](const char* name, auto& fn) {
        PyObject* v = PyDict_GetItemString(a[0], name);
        void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
        if (!p) ok = false;
        fn = reinterpret_cast<std::decay_t<decltype(fn)>>(p);
    };
    Api n{};
    take("mxq_quantize", n.quantize);
    take("mxq_slice_scale", n.slice_scale);
    take("mxq_slice_scale_multi", n.slice_scale_multi);
    take("mxq_dequantize", n.dequantize);
    take("mxq_tiled_scales_bytes", n.tiled_scales_bytes);
    take("mxq_quantize_tiled", n.quantize_tiled);
    take("mxq_slice_scale_tiled", n.slice_scale_tiled);
    take("mxq_fake_quant", n.fake_quant);
    take("mxq_fake_quant_bwd", n.fake_quant_bwd);
    take("mxq_codes_bytes", n.codes_bytes);
    if (!ok) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, "an entry point has no address");
        return nullptr;
    }
    api = n;
    Py_INCREF(a[1]);
    Py_INCREF(a[2]);
    Py_INCREF(a[3]);
    Py_XSETREF(mxq_error, a[3]);
    Py_XSETREF(formats, a[1]);
    Py_XSETREF(parameter, reinterpret_cast<PyTypeObject*>(a[2]));
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(bind),           FAST(quantize),          FAST(slice_scale), FAST(slice_scale_multi),
                         FAST(dequantize),     FAST(quantize_tiled),    FAST(slice_scale_tiled), FAST(fake_quant),
                         FAST(fake_quant_bwd), FAST(run_prepared),      FAST(fake_quant_ste), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mxq_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mxq_host() { return PyModule_Create(&module); }
