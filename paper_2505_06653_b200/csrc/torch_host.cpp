// Native half of the Python binding: turns torch CUDA tensors into device pointers, allocates the
// outputs from torch's caching allocator and calls the C ABI of libbof4.so on the current stream.
//
// A call on a small tensor is bound by the host: the same marshalling in Python (device context,
// stream object, torch.empty, ctypes conversion of ten to eighteen arguments) took 16 ... 20 us a
// call against 2 ... 7 us of device time.  Here it is a few hundred nanoseconds beside the
// allocations and the launches.  Plain CPython entry points (positional vector call); binding.py keeps the
// signatures and their documentation.
//
// Other Python threads run while the library enqueues (a launch waits where the stream's queue is full) and while
// memory is allocated (which may synchronise): what such a stretch uses is owned by this call, not borrowed
// from a list that another thread may change.
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime.h>
#include <torch/csrc/Device.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "../../include/bof4.h"

// The torch and Python this module is built for: the binding looks for it in the file before it loads the module.
__attribute__((used)) static const char g_built_for[] = BOF4_HOST_TAG;

namespace {

struct PySet {};  // a Python exception has been set

[[noreturn]] void fail(PyObject* type, const char* msg)
{
    PyErr_SetString(type, msg);
    throw PySet{};
}
template <class... A>
[[noreturn]] void failf(PyObject* type, const char* fmt, A... a)
{
    PyErr_Format(type, fmt, a...);
    throw PySet{};
}

// Python objects of binding.py used on rare paths.
PyObject* g_error = nullptr;      // Bof4Error(code, message)
PyObject* g_codebook = nullptr;   // levels of any array-like -> tensor
PyObject* g_allocator = nullptr;  // fn(numel, dtype, device, zero), or NULL

void check(int rc)
{
    if (rc == BOF4_OK) return;
    if (PyObject* e = PyObject_CallFunction(g_error, "is", rc, bof4_last_error())) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw PySet{};
}

struct NoGil {  // other Python threads run during its lifetime
    PyThreadState* state = PyEval_SaveThread();
    NoGil() = default;
    NoGil(const NoGil&) = delete;
    NoGil& operator=(const NoGil&) = delete;
    ~NoGil() { PyEval_RestoreThread(state); }
};

// A call of the library; the arguments are already plain pointers and numbers.
template <class... P, class... A>
void call(int (*fn)(P...), A... args)
{
    int rc;
    {
        const NoGil others;
        rc = fn(args...);
    }
    check(rc);
}

struct Ref {  // owned reference
    PyObject* p;
    explicit Ref(PyObject* q) : p(q)
    {
        if (!q) throw PySet{};
    }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
    ~Ref() { Py_XDECREF(p); }
    PyObject* release()
    {
        PyObject* q = p;
        p = nullptr;
        return q;
    }
};

const at::Tensor& tensor(PyObject* o, const char* name)
{
    if (!THPVariable_Check(o)) failf(PyExc_TypeError, "%s must be a torch tensor", name);
    return THPVariable_Unpack(o);
}
// A contiguous CUDA tensor.
const at::Tensor& dev(PyObject* o, const char* name)
{
    const at::Tensor& t = tensor(o, name);
    if (!t.is_cuda()) failf(PyExc_ValueError, "%s must be a CUDA tensor (there is no CPU path)", name);
    if (!t.is_contiguous()) failf(PyExc_ValueError, "%s must be contiguous", name);
    return t;
}
int dtype_code(const at::Tensor& t)
{
    if (t.scalar_type() == at::kFloat) return BOF4_F32;
    if (t.scalar_type() == at::kBFloat16) return BOF4_BF16;
    failf(PyExc_TypeError, "weights must be float32 or bfloat16, got %s", c10::toString(t.scalar_type()));
}
at::ScalarType torch_dtype(int code) { return code == BOF4_F32 ? at::kFloat : at::kBFloat16; }

int64_t integer(PyObject* o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v != -1 || !PyErr_Occurred()) return v;
    PyErr_Clear();  // numpy integers and the like
    Ref i(PyNumber_Index(o));
    const long long u = PyLong_AsLongLong(i.p);
    if (u == -1 && PyErr_Occurred()) throw PySet{};
    return u;
}
double real(PyObject* o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PySet{};
    return v;
}
bool none(PyObject* o) { return o == Py_None; }

// k uninitialised buffers, then fn(), a call of the library that may use them.
struct Spec {
    int64_t numel;
    at::ScalarType dt;
};
template <class F>
void make_and_call(at::Tensor* out, const Spec* spec, size_t k, at::Device d, F&& fn)
{
    if (g_allocator) {
        for (size_t i = 0; i < k; ++i) {
            Ref device(THPDevice_New(d));
            Ref r(PyObject_CallFunction(g_allocator, "LOOO", (long long)(spec[i].numel < 0 ? 0 : spec[i].numel),
                                        (PyObject*)torch::getTHPDtype(spec[i].dt), device.p, Py_False));
            out[i] = tensor(r.p, "the allocator's result");
        }
        k = 0;
    }
    int rc;
    {
        const NoGil others;
        for (size_t i = 0; i < k; ++i)
            out[i] = at::detail::empty_cuda({spec[i].numel < 0 ? 0 : spec[i].numel}, spec[i].dt, d, std::nullopt);
        rc = fn();
    }
    check(rc);
}
void make(at::Tensor* out, const Spec* spec, size_t k, at::Device d)
{
    make_and_call(out, spec, k, d, [] { return BOF4_OK; });
}
at::Tensor make(int64_t numel, at::ScalarType dt, at::Device d, bool zero = false)
{
    at::Tensor t;
    const Spec spec{numel, dt};
    make(&t, &spec, 1, d);
    if (zero) {
        const NoGil others;
        t.zero_();
    }
    return t;
}
PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

// The 16 levels as a device tensor fp32 (the caller's own tensor where it already is one).
at::Tensor codebook(PyObject* o, at::Device d)
{
    if (THPVariable_Check(o)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.scalar_type() == at::kFloat && t.device() == d && t.is_contiguous()) {
            if (t.numel() != BOF4_LEVELS) fail(PyExc_ValueError, "a codebook has 16 levels");
            return t;
        }
    }
    Ref device(THPDevice_New(d));
    Ref r(PyObject_CallFunctionObjArgs(g_codebook, o, device.p, nullptr));
    return tensor(r.p, "levels");
}
const float* levels_ptr(const at::Tensor& t) { return t.const_data_ptr<float>(); }

void* stream_of(at::Device d) { return c10::cuda::getCurrentCUDAStream(d.index()).stream(); }

// The workspace given, or a new one of the bytes a size query returned (0: it refused the arguments).
at::Tensor workspace(PyObject* given, size_t bytes, at::Device d)
{
    if (!none(given)) return tensor(given, "workspace");
    if (bytes == 0) {
        if (PyObject* e = PyObject_CallFunction(g_error, "is", -2, "the workspace size query rejected the arguments")) {
            PyErr_SetObject(g_error, e);
            Py_DECREF(e);
        }
        throw PySet{};
    }
    return make((int64_t)bytes, at::kByte, d);  // torch allocations are 512-byte aligned
}

// An outlier list (idx, val, n_out) or None.
struct Outliers {
    const int32_t* idx = nullptr;
    const void* val = nullptr;
    const int64_t* cnt = nullptr;
    int64_t cap = 0;
    at::Tensor own[3];
    explicit Outliers(PyObject* o)
    {
        if (none(o)) return;
        Ref f(PySequence_Fast(o, "outliers must be (idx, val, n_out)"));
        if (PySequence_Fast_GET_SIZE(f.p) != 3) fail(PyExc_ValueError, "outliers must be (idx, val, n_out)");
        PyObject** v = PySequence_Fast_ITEMS(f.p);
        for (int k = 0; k < 3; ++k) own[k] = dev(v[k], "outliers");
        idx = static_cast<const int32_t*>(own[0].const_data_ptr());
        val = own[1].const_data_ptr();
        cnt = static_cast<const int64_t*>(own[2].const_data_ptr());
        cap = own[0].numel();
    }
};

// The items of a sequence as a tuple (a new reference), or NULL with a TypeError.
PyObject* items(PyObject* o, const char* msg)
{
    PyObject* t = PySequence_Tuple(o);
    if (!t && PyErr_ExceptionMatches(PyExc_TypeError)) PyErr_SetString(PyExc_TypeError, msg);
    return t;
}

// A list of tensors (or one tensor) of one dtype: pointers and sizes.
struct List {
    Ref own;  // the tensor, or a tuple of the list's
    std::vector<const void*> ptr;
    std::vector<int64_t> n;
    int64_t total = 0;
    int dt = 0;
    at::Device d = at::kCUDA;
    explicit List(PyObject* o) : own(THPVariable_Check(o) ? Py_NewRef(o) : items(o, "weights must be a tensor or a list of tensors"))
    {
        if (THPVariable_Check(o)) {
            add(o);
        } else {
            const Py_ssize_t k = PyTuple_GET_SIZE(own.p);
            if (k == 0) fail(PyExc_ValueError, "empty tensor list");
            ptr.reserve(k);
            n.reserve(k);
            for (Py_ssize_t i = 0; i < k; ++i) add(PyTuple_GET_ITEM(own.p, i));
        }
    }
    void add(PyObject* o)
    {
        const at::Tensor& t = ::dev(o, "weights");
        const int c = dtype_code(t);
        if (ptr.empty()) {
            dt = c;
            d = t.device();
        } else if (c != dt) {
            fail(PyExc_TypeError, "all tensors of one call must share a dtype");
        }
        ptr.push_back(t.const_data_ptr());
        n.push_back(t.numel());
        total += t.numel();
    }
};

int64_t blocks_of(int64_t n, int64_t block)
{
    if (block < 1) block = 1;
    return (n + block - 1) / block;
}

// ---------------------------------------------------------------- entry points
//
// Every function takes the positional arguments of the binding.py function of the same name.

PyObject* set_hooks(PyObject* const* a)
{
    Py_INCREF(a[0]);
    Py_XSETREF(g_error, a[0]);
    Py_INCREF(a[1]);
    Py_XSETREF(g_codebook, a[1]);
    Py_RETURN_NONE;
}

PyObject* set_allocator(PyObject* const* a)
{
    if (none(a[0])) {
        Py_CLEAR(g_allocator);
    } else {
        Py_INCREF(a[0]);
        Py_XSETREF(g_allocator, a[0]);
    }
    Py_RETURN_NONE;
}

// (w, block_size, norm, levels, scale_dtype, out)
PyObject* quantize(PyObject* const* a)
{
    const at::Tensor& w = dev(a[0], "w");
    const int64_t n = w.numel(), block = integer(a[1]);
    const int dt = dtype_code(w), sd = none(a[4]) ? dt : (int)integer(a[4]);
    const c10::cuda::CUDAGuard guard(w.device());
    const at::Tensor cb = codebook(a[3], w.device());
    if (none(a[5])) {
        at::Tensor made[2];
        const Spec spec[2] = {{(n + 1) / 2, at::kByte}, {blocks_of(n, block), torch_dtype(sd)}};
        const int norm = (int)integer(a[2]);
        make_and_call(made, spec, 2, w.device(), [&] {
            return bof4_quantize(w.const_data_ptr(), dt, n, (int)block, norm, levels_ptr(cb), static_cast<uint8_t*>(made[0].data_ptr()),
                                 made[1].data_ptr(), sd, stream_of(w.device()));
        });
        Ref c(wrap(made[0])), s(wrap(made[1]));
        return PyTuple_Pack(2, c.p, s.p);
    }
    Ref out(PySequence_Tuple(a[5]));
    if (PyTuple_GET_SIZE(out.p) != 2) fail(PyExc_ValueError, "out must be (codes, scales)");
    call(bof4_quantize, w.const_data_ptr(), dt, n, (int)block, (int)integer(a[2]), levels_ptr(cb),
         static_cast<uint8_t*>(tensor(PyTuple_GET_ITEM(out.p, 0), "codes").data_ptr()),
         tensor(PyTuple_GET_ITEM(out.p, 1), "scales").data_ptr(), sd, stream_of(w.device()));
    return out.release();
}

// (codes, scales, block_size, levels, out_dtype, outliers, out, n)
PyObject* dequantize(PyObject* const* a)
{
    const at::Tensor &codes = dev(a[0], "codes"), &scales = dev(a[1], "scales");
    const int64_t n = none(a[7]) ? codes.numel() * 2 : integer(a[7]);
    if ((n + 1) / 2 != codes.numel()) fail(PyExc_ValueError, "codes must hold (n + 1) // 2 bytes");
    const c10::cuda::CUDAGuard guard(codes.device());
    const at::Tensor cb = codebook(a[3], codes.device());
    const int od = (int)integer(a[4]);
    const Outliers o(a[5]);
    const int sd = dtype_code(scales), block = (int)integer(a[2]);
    at::Tensor out;
    const Spec spec{n, torch_dtype(od)};
    if (!none(a[6])) out = tensor(a[6], "out");
    make_and_call(&out, &spec, none(a[6]) ? 1 : 0, codes.device(), [&] {
        return bof4_dequantize(static_cast<const uint8_t*>(codes.const_data_ptr()), scales.const_data_ptr(), sd, n, block, levels_ptr(cb),
                               o.idx, o.val, o.cnt, o.cap, out.data_ptr(), od, stream_of(codes.device()));
    });
    if (!none(a[6])) {
        Py_INCREF(a[6]);
        return a[6];
    }
    return wrap(out);
}

// (codes, scales, rows, cols, block_size, levels, x, outliers, out)
PyObject* gemv(PyObject* const* a)
{
    const at::Tensor &codes = dev(a[0], "codes"), &scales = dev(a[1], "scales"), &x = dev(a[6], "x");
    const int64_t rows = integer(a[2]), cols = integer(a[3]);
    if (codes.numel() * 2 != rows * cols || x.numel() != cols)
        fail(PyExc_ValueError, "codes must hold rows * cols weights and x cols values");
    const c10::cuda::CUDAGuard guard(codes.device());
    const at::Tensor cb = codebook(a[5], codes.device());
    const Outliers o(a[7]);
    const int sd = dtype_code(scales), xd = dtype_code(x), block = (int)integer(a[4]);
    at::Tensor out;
    const Spec spec{rows, at::kFloat};
    if (!none(a[8])) out = tensor(a[8], "out");
    make_and_call(&out, &spec, none(a[8]) ? 1 : 0, codes.device(), [&] {
        return bof4_gemv(static_cast<const uint8_t*>(codes.const_data_ptr()), scales.const_data_ptr(), sd, rows, cols, block, levels_ptr(cb),
                         x.const_data_ptr(), xd, o.idx, o.val, o.cnt, o.cap, static_cast<float*>(out.data_ptr()), stream_of(codes.device()));
    });
    if (!none(a[8])) {
        Py_INCREF(a[8]);
        return a[8];
    }
    return wrap(out);
}

// (codes, scales, rows, cols, block_size, levels, x, workspace, split, outliers)
PyObject* gemm_tc(PyObject* const* a)
{
    const at::Tensor &codes = dev(a[0], "codes"), &scales = dev(a[1], "scales"), &x = dev(a[6], "x");
    const int64_t rows = integer(a[2]), cols = integer(a[3]);
    if (x.scalar_type() != at::kBFloat16 || x.dim() != 2 || x.size(1) != cols || codes.numel() * 2 != rows * cols)
        fail(PyExc_ValueError, "x must be bf16 [n_rhs, cols] and codes must hold rows * cols weights");
    const int64_t n_rhs = x.size(0);
    const at::Device d = codes.device();
    const c10::cuda::CUDAGuard guard(d);
    const at::Tensor cb = codebook(a[5], d);
    const Outliers o(a[9]);
    const int sd = dtype_code(scales), block = (int)integer(a[4]);
    at::Tensor made[3];  // the product, its status (written by the call), the workspace: tickets and two parts of tiles per SM
    const Spec spec[3] = {{rows * n_rhs, at::kFloat}, {1, at::kInt}, {rows / 16 + 256 + 148 * 2 * 128 * 4 * n_rhs, at::kByte}};
    const bool split = none(a[7]) && PyObject_IsTrue(a[8]);
    if (!none(a[7])) made[2] = tensor(a[7], "workspace");
    make_and_call(made, spec, split ? 3 : 2, d, [&] {
        if (rows == 0) made[1].zero_();  // nothing to do
        const at::Tensor& ws = made[2];
        return bof4_gemm_tc(static_cast<const uint8_t*>(codes.const_data_ptr()), scales.const_data_ptr(), sd, rows, cols, block,
                            levels_ptr(cb), x.const_data_ptr(), (int)n_rhs, o.idx, o.val, o.cnt, o.cap,
                            static_cast<float*>(made[0].data_ptr()), static_cast<int*>(made[1].data_ptr()),
                            ws.defined() ? ws.data_ptr() : nullptr, ws.defined() ? (size_t)ws.numel() : 0, stream_of(d));
    });
    const at::Tensor y = made[0].view({rows, n_rhs}), &status = made[1];
    Ref ry(wrap(y)), rs(wrap(status));
    return PyTuple_Pack(2, ry.p, rs.p);
}

// (w, block_size, norm, levels, tau, capacity, scale_dtype, workspace, out)
PyObject* quantize_opq(PyObject* const* a)
{
    const at::Tensor& w = dev(a[0], "w");
    const at::Device d = w.device();
    const int64_t n = w.numel(), block = integer(a[1]), cap = integer(a[5]);
    const int dt = dtype_code(w), sd = none(a[6]) ? dt : (int)integer(a[6]);
    const c10::cuda::CUDAGuard guard(d);
    const at::Tensor cb = codebook(a[3], d);
    const at::Tensor ws = workspace(a[7], bof4_workspace_bytes(BOF4_OP_OPQ, n, (int)block, 0), d);
    Ref out(none(a[8]) ? PyTuple_New(5) : PySequence_Tuple(a[8]));
    if (none(a[8])) {
        at::Tensor t[5];
        const Spec spec[5] = {{(n + 1) / 2, at::kByte}, {blocks_of(n, block), torch_dtype(sd)}, {cap, at::kInt}, {cap, at::kBFloat16}, {1, at::kLong}};
        make(t, spec, 5, d);
        for (int k = 0; k < 5; ++k) PyTuple_SET_ITEM(out.p, k, wrap(t[k]));
    }
    if (PyTuple_GET_SIZE(out.p) != 5) fail(PyExc_ValueError, "out must be (codes, scales, idx, val, n_out)");
    auto ptr = [&](int k) { return tensor(PyTuple_GET_ITEM(out.p, k), "out").data_ptr(); };
    call(bof4_quantize_opq, w.const_data_ptr(), dt, n, (int)block, (int)integer(a[2]), levels_ptr(cb), (float)real(a[4]),
         static_cast<uint8_t*>(ptr(0)), ptr(1), sd, static_cast<int32_t*>(ptr(2)), ptr(3), cap,
         static_cast<int64_t*>(ptr(4)), ws.data_ptr(), (size_t)ws.numel(), stream_of(d));
    return out.release();
}

// (n_out, capacity)
PyObject* outlier_count(PyObject* const* a)
{
    const at::Tensor& n_out = dev(a[0], "n_out");
    if (n_out.scalar_type() != at::kLong || n_out.numel() != 1)
        fail(PyExc_ValueError, "n_out must be the int64[1] count tensor of an OPQ call");
    const c10::cuda::CUDAGuard guard(n_out.device());
    const int64_t cap = integer(a[1]);
    int64_t host = 0;
    call(bof4_outlier_count, static_cast<const int64_t*>(n_out.const_data_ptr()), cap, &host, stream_of(n_out.device()));
    return PyLong_FromLongLong(host);
}

// (weights, block_size, norm, levels, scale_dtype, out)
PyObject* quantize_batch(PyObject* const* a)
{
    const List w(a[0]);
    const int64_t block = integer(a[1]);
    const int sd = none(a[4]) ? w.dt : (int)integer(a[4]);
    const size_t k = w.ptr.size();
    const c10::cuda::CUDAGuard guard(w.d);
    const at::Tensor cb = codebook(a[3], w.d);
    std::vector<uint8_t*> codes(k);
    std::vector<void*> scales(k);
    std::vector<at::Tensor> made;
    if (none(a[5])) {
        std::vector<Spec> spec;
        spec.reserve(2 * k);
        for (size_t t = 0; t < k; ++t) {
            spec.push_back({(w.n[t] + 1) / 2, at::kByte});
            spec.push_back({blocks_of(w.n[t], block), torch_dtype(sd)});
        }
        made.resize(2 * k);
        make(made.data(), spec.data(), 2 * k, w.d);
    }
    PyObject *lc, *ls;
    if (none(a[5])) {
        lc = PyList_New((Py_ssize_t)k);
        ls = PyList_New((Py_ssize_t)k);
    } else {
        Ref out(PySequence_Tuple(a[5]));
        if (PyTuple_GET_SIZE(out.p) != 2) fail(PyExc_ValueError, "out must be (codes, scales)");
        lc = PySequence_List(PyTuple_GET_ITEM(out.p, 0));
        ls = PySequence_List(PyTuple_GET_ITEM(out.p, 1));
    }
    Ref rc_(lc), rs_(ls);
    if ((size_t)PyList_GET_SIZE(lc) != k || (size_t)PyList_GET_SIZE(ls) != k)
        fail(PyExc_ValueError, "out buffers do not match the tensors");
    for (size_t t = 0; t < k; ++t) {
        const int64_t nc = (w.n[t] + 1) / 2, ns = blocks_of(w.n[t], block);
        if (none(a[5])) {
            const at::Tensor &c = made[2 * t], &s = made[2 * t + 1];
            codes[t] = static_cast<uint8_t*>(c.data_ptr());
            scales[t] = s.data_ptr();
            PyList_SET_ITEM(lc, (Py_ssize_t)t, wrap(c));
            PyList_SET_ITEM(ls, (Py_ssize_t)t, wrap(s));
        } else {
            const at::Tensor &c = dev(PyList_GET_ITEM(lc, (Py_ssize_t)t), "codes"), &s = dev(PyList_GET_ITEM(ls, (Py_ssize_t)t), "scales");
            if (c.numel() != nc || s.numel() != ns || dtype_code(s) != sd)
                fail(PyExc_ValueError, "out buffers do not match the tensors");
            codes[t] = static_cast<uint8_t*>(c.data_ptr());
            scales[t] = s.data_ptr();
        }
    }
    call(bof4_quantize_batch, w.ptr.data(), w.n.data(), (int)k, w.dt, (int)block, (int)integer(a[2]), levels_ptr(cb), codes.data(),
         scales.data(), sd, stream_of(w.d));
    return PyTuple_Pack(2, lc, ls);
}

// (codes, scales, sizes, block_size, levels, out_dtype, out)
PyObject* dequantize_batch(PyObject* const* a)
{
    Ref fc(items(a[0], "codes must be a list of tensors")), fs(items(a[1], "scales must be a list of tensors")),
        fn(items(a[2], "sizes must be a list"));
    const size_t k = (size_t)PyTuple_GET_SIZE(fc.p);
    if (k == 0) fail(PyExc_ValueError, "empty tensor list");
    const int64_t block = integer(a[3]);
    const int od = (int)integer(a[5]);
    Ref lo(none(a[6]) ? PyList_New((Py_ssize_t)k) : PySequence_List(a[6]));
    if ((size_t)PyTuple_GET_SIZE(fs.p) != k || (size_t)PyTuple_GET_SIZE(fn.p) != k || (size_t)PyList_GET_SIZE(lo.p) != k)
        fail(PyExc_ValueError, "buffers do not match the sizes");
    const at::Device d = dev(PyTuple_GET_ITEM(fc.p, 0), "codes").device();
    const c10::cuda::CUDAGuard guard(d);
    const at::Tensor cb = codebook(a[4], d);
    std::vector<const uint8_t*> codes(k);
    std::vector<const void*> scales(k);
    std::vector<void*> outs(k);
    std::vector<int64_t> ns(k);
    int sd = 0;
    for (size_t t = 0; t < k; ++t) {
        const Py_ssize_t i = (Py_ssize_t)t;
        const at::Tensor &c = dev(PyTuple_GET_ITEM(fc.p, i), "codes"), &s = dev(PyTuple_GET_ITEM(fs.p, i), "scales");
        const int64_t n = ns[t] = integer(PyTuple_GET_ITEM(fn.p, i));
        if (t == 0) sd = dtype_code(s);
        if (c.numel() != (n + 1) / 2 || s.numel() != blocks_of(n, block) || dtype_code(s) != sd)
            fail(PyExc_ValueError, "buffers do not match the sizes");
        codes[t] = static_cast<const uint8_t*>(c.const_data_ptr());
        scales[t] = s.const_data_ptr();
        if (none(a[6])) {
            const at::Tensor o = make(n, torch_dtype(od), d);
            outs[t] = o.data_ptr();
            PyList_SET_ITEM(lo.p, i, wrap(o));
        } else {
            const at::Tensor& o = dev(PyList_GET_ITEM(lo.p, i), "out");
            if (o.numel() != n || dtype_code(o) != od) fail(PyExc_ValueError, "buffers do not match the sizes");
            outs[t] = o.data_ptr();
        }
    }
    call(bof4_dequantize_batch, codes.data(), scales.data(), sd, ns.data(), (int)k, (int)block, levels_ptr(cb), outs.data(), od,
         stream_of(d));
    return lo.release();
}

// (scales, norm)
PyObject* scales_compress(PyObject* const* a)
{
    const at::Tensor& scales = dev(a[0], "scales");
    const at::Device d = scales.device();
    const int64_t b = scales.numel();
    const int norm = (int)integer(a[1]);
    const c10::cuda::CUDAGuard guard(d);
    at::Tensor made[3];  // q, group, sign (signed normalisation)
    const Spec spec[3] = {{b, at::kByte}, {(b + 255) / 256, at::kFloat}, {(b + 7) / 8, at::kByte}};
    const int sd = dtype_code(scales);
    const at::Tensor &q = made[0], &g = made[1], &sign = made[2];
    make_and_call(made, spec, norm == BOF4_NORM_SIGNED ? 3 : 2, d, [&] {
        return bof4_scales_compress(scales.const_data_ptr(), sd, b, norm, static_cast<uint8_t*>(q.data_ptr()), static_cast<float*>(g.data_ptr()),
                                    sign.defined() ? static_cast<uint8_t*>(sign.data_ptr()) : nullptr, stream_of(d));
    });
    Ref rq(wrap(q)), rg(wrap(g));
    if (!sign.defined()) return PyTuple_Pack(3, rq.p, rg.p, Py_None);
    Ref rs(wrap(sign));
    return PyTuple_Pack(3, rq.p, rg.p, rs.p);
}

// (q, group, sign)
PyObject* scales_expand(PyObject* const* a)
{
    const at::Tensor &q = dev(a[0], "q"), &g = dev(a[1], "group");
    const uint8_t* sign = none(a[2]) ? nullptr : static_cast<const uint8_t*>(dev(a[2], "sign").const_data_ptr());
    const c10::cuda::CUDAGuard guard(q.device());
    at::Tensor out;
    const Spec spec{q.numel(), at::kFloat};
    make_and_call(&out, &spec, 1, q.device(), [&] {
        return bof4_scales_expand(static_cast<const uint8_t*>(q.const_data_ptr()), static_cast<const float*>(g.const_data_ptr()), sign,
                                  q.numel(), static_cast<float*>(out.data_ptr()), stream_of(q.device()));
    });
    return wrap(out);
}

// (weights, block_size, norm, metric, levels, fixed_mask, iters, workspace, sync, out)
PyObject* fit_codebook(PyObject* const* a)
{
    const List w(a[0]);
    const int block = (int)integer(a[1]), norm = (int)integer(a[2]), metric = (int)integer(a[3]);
    const int64_t iters = integer(a[6]);
    const c10::cuda::CUDAGuard guard(w.d);
    void* const st = stream_of(w.d);
    at::Tensor cb, log;
    if (!none(a[9])) {
        Ref out(PySequence_Tuple(a[9]));
        if (PyTuple_GET_SIZE(out.p) < 2) fail(PyExc_ValueError, "out must be (float32[16], float64[>= iters])");
        cb = dev(PyTuple_GET_ITEM(out.p, 0), "out[0]");
        log = dev(PyTuple_GET_ITEM(out.p, 1), "out[1]");
        if (cb.scalar_type() != at::kFloat || cb.numel() != BOF4_LEVELS || log.scalar_type() != at::kDouble || log.numel() < iters)
            fail(PyExc_ValueError, "out must be (float32[16], float64[>= iters])");
        const at::Tensor src = codebook(a[4], w.d);
        const NoGil others;
        if (src.data_ptr() != cb.data_ptr()) cb.copy_(src);  // levels may be the output buffer itself: continue in place
    } else {
        Py_buffer view;
        bool done = false;
        if (!THPVariable_Check(a[4]) && PyObject_CheckBuffer(a[4]) &&
            PyObject_GetBuffer(a[4], &view, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) == 0) {
            // 16 fp32 levels of a host array: straight into the result's buffer
            if (view.len == BOF4_LEVELS * 4 && view.format && view.format[0] == 'f' && view.format[1] == 0) {
                // through a tensor: a copy from pageable memory of this size is staged before the call returns
                const NoGil others;
                cb = at::detail::empty_cuda({BOF4_LEVELS}, at::kFloat, w.d, std::nullopt);
                done = cudaMemcpyAsync(cb.data_ptr(), view.buf, (size_t)view.len, cudaMemcpyHostToDevice,
                                       static_cast<cudaStream_t>(st)) == cudaSuccess;
            }
            PyBuffer_Release(&view);
        } else {
            PyErr_Clear();
        }
        if (!done) {
            const at::Tensor src = codebook(a[4], w.d);
            const NoGil others;
            cb = src.clone();
        }
        log = make(iters > 1 ? iters : 1, at::kDouble, w.d, iters < 1);  // the fit writes every entry
    }
    const at::Tensor ws = workspace(a[7], bof4_fit_workspace_bytes(w.total, w.dt, block, metric, (int)iters), w.d);
    call(bof4_fit_codebook, w.ptr.data(), w.n.data(), (int)w.ptr.size(), w.dt, block, norm, metric,
         static_cast<float*>(cb.data_ptr()), (uint32_t)integer(a[5]), (int)iters,
         static_cast<double*>(log.data_ptr()), ws.data_ptr(), (size_t)ws.numel(), st);
    if (PyObject_IsTrue(a[8])) {
        cudaError_t e;
        {
            const NoGil others;
            e = cudaStreamSynchronize(static_cast<cudaStream_t>(st));
        }
        if (e != cudaSuccess) failf(PyExc_RuntimeError, "CUDA error: %s", cudaGetErrorString(e));
    }
    Ref rc(wrap(cb)), rl(wrap(log.narrow(0, 0, iters < 0 ? 0 : iters)));
    return PyTuple_Pack(2, rc.p, rl.p);
}

template <PyObject* (*F)(PyObject* const*), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    try {
        if (n != N) failf(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
        return F(args);
    } catch (const PySet&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

#define BOF4_ENTRY(name, n) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<name, n>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    BOF4_ENTRY(set_hooks, 2), BOF4_ENTRY(set_allocator, 1), BOF4_ENTRY(quantize, 6), BOF4_ENTRY(dequantize, 8),
    BOF4_ENTRY(gemv, 9), BOF4_ENTRY(gemm_tc, 10), BOF4_ENTRY(quantize_opq, 9), BOF4_ENTRY(outlier_count, 2),
    BOF4_ENTRY(quantize_batch, 6), BOF4_ENTRY(dequantize_batch, 7), BOF4_ENTRY(scales_compress, 2), BOF4_ENTRY(scales_expand, 3),
    BOF4_ENTRY(fit_codebook, 10), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_bof4_torch", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__bof4_torch(void) { return PyModule_Create(&g_module); }
