// The calls a program makes per layer or per token, as a CPython module over the C ABI: torch tensors in, C
// structs and pointers out.  Argument marshalling only, like the ctypes face (binding.py), whose functions
// forward their arguments here.  Marshalling a decode call through ctypes took 14 us of host time, twice what
// the GPU needs for it; from here it takes about as long as the launch itself.
//
// Every function takes its arguments by position.  A failing call raises the exception class given to
// set_error(status, message); broken preconditions raise AssertionError as the Python asserts did.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/core/DefaultDtype.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Device.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/device_lazy_init.h>

#include "powerattn.h"

namespace {

PyObject *g_error = nullptr;  // the binding's PaError

struct Raised {};  // a Python exception has been set

[[noreturn]] void raise(PyObject *type, const char *msg)
{
    PyErr_SetString(type, msg);
    throw Raised();
}
void expect(bool ok, const char *msg)
{
    if (!ok) raise(PyExc_AssertionError, msg);
}

const at::Tensor &tensor(PyObject *o)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch.Tensor");
    return THPVariable_Unpack(o);
}
int64_t integer(PyObject *o)
{
    const int64_t v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return v;
}
int32_t integer32(PyObject *o)
{
    const int64_t v = integer(o);
    if (v != (int32_t)v) raise(PyExc_OverflowError, "value does not fit in 32 bits");
    return (int32_t)v;
}
float number(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised();
    return (float)v;
}
at::ScalarType dtype(PyObject *o)
{
    if (o == Py_None) return c10::get_default_dtype_as_scalartype();  // (as in torch.empty)
    if (!THPDtype_Check(o)) raise(PyExc_TypeError, "expected a torch.dtype");
    return reinterpret_cast<THPDtype *>(o)->scalar_type;
}
bool is_int32(const at::Tensor &t) { return t.scalar_type() == at::kInt; }
pa_dtype out_dtype(at::ScalarType t) { return t == at::kFloat ? PA_F32 : PA_BF16; }

pa_strides strides4(const at::Tensor &t)
{
    expect(t.dim() == 4 && t.stride(3) == 1, "expected [batch, seq, head, head_dim] with contiguous head_dim");
    return {t.stride(0), t.stride(1), t.stride(2)};
}

struct WithoutGil {
    PyThreadState *state = PyEval_SaveThread();
    ~WithoutGil() { PyEval_RestoreThread(state); }
};

// As torch.empty: the device's Python side is set up first, and the allocation, which may wait for the device or another
// thread, goes without the interpreter lock.
at::Tensor empty(at::IntArrayRef size, const at::TensorOptions &options)
{
    torch::utils::maybe_initialize_device(options);
    const WithoutGil released;
    return at::empty(size, options);
}

// An output or scratch tensor: the caller's, or one allocated here.
struct Out {
    at::Tensor t;
    PyObject *given = nullptr;
    template <typename Make>
    Out(PyObject *o, Make make)
    {
        if (o == Py_None) {
            t = make();
        } else {
            t = tensor(o);
            given = o;
        }
    }
    PyObject *object() const { return given ? Py_NewRef(given) : THPVariable_Wrap(t); }
    void *ptr() const { return t.data_ptr(); }
};
at::Tensor make(const at::Tensor &like, at::IntArrayRef size, at::ScalarType type)
{
    return empty(size, like.options().dtype(type));
}
at::Tensor make_bytes(const at::Tensor &like, size_t n)
{
    return make(like, {(int64_t)(n < 16 ? 16 : n)}, at::kByte);
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Runs a library call without the interpreter lock; raises on a status other than PA_OK.
template <typename Call>
void run(Call call)
{
    const pa_status s = [&] {
        const WithoutGil released;
        return call();
    }();
    if (s == PA_OK) return;
    if (PyObject *e = PyObject_CallFunction(g_error, "is", (int)s, pa_last_error_message())) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Raised();
}

template <typename... O>
PyObject *tuple(const O &...outs)
{
    return Py_BuildValue(sizeof...(O) == 3 ? "(NNN)" : "(NNNN)", outs.object()...);
}

pa_prefill_params prefill_params(const at::Tensor &q, const at::Tensor &k, const at::Tensor &v, const at::Tensor &o,
                                 PyObject *block, PyObject *scale)
{
    const pa_strides sq = strides4(q), sk = strides4(k), sv = strides4(v), so = strides4(o);
    return {(int32_t)q.size(0), (int32_t)q.size(2), (int32_t)k.size(2), (int32_t)q.size(3), q.size(1), integer32(block),
            number(scale), sq, sk, sv, so, out_dtype(o.scalar_type())};
}

// q, k, v, row_ptr, col_idx, o, lse, workspace, block, softmax_scale, o_dtype, nnz
PyObject *prefill(PyObject *const *x)
{
    const at::Tensor &q = tensor(x[0]), &k = tensor(x[1]), &v = tensor(x[2]), &row_ptr = tensor(x[3]), &col_idx = tensor(x[4]);
    expect(q.dim() == 4 && k.dim() == 4, "expected [batch, seq, head, head_dim]");
    const Out o(x[5], [&] { return make(q, q.sizes(), dtype(x[10])); });
    const Out lse(x[6], [&] { return make(q, {q.size(0), q.size(2), q.size(1)}, at::kFloat); });
    const pa_prefill_params p = prefill_params(q, k, v, o.t, x[8], x[9]);
    const Out ws(x[7], [&] { return make_bytes(q, pa_prefill_workspace_bytes(&p)); });
    const int64_t nnz = x[11] == Py_None ? col_idx.numel() : integer(x[11]);
    run([&] {
        return pa_prefill(&p, q.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)row_ptr.data_ptr(),
                          (const int32_t *)col_idx.data_ptr(), nnz, o.ptr(), (float *)lse.ptr(), ws.ptr(),
                          (size_t)ws.t.numel(), stream());
    });
    return tuple(o, lse, ws);
}

// q, k, v, cu_seqlens, max_seq_len, row_ptr, col_idx, o, lse, workspace, block, softmax_scale, o_dtype
PyObject *prefill_varlen(PyObject *const *x)
{
    const at::Tensor &q = tensor(x[0]), &k = tensor(x[1]), &v = tensor(x[2]), &cu = tensor(x[3]), &row_ptr = tensor(x[5]),
                     &col_idx = tensor(x[6]);
    expect(q.dim() == 3 && k.dim() == 3 && v.dim() == 3 && q.stride(2) == 1 && k.stride(2) == 1 && v.stride(2) == 1 &&
               is_int32(cu),
           "expected [total, head, head_dim] tensors with contiguous head_dim and int32 cu_seqlens");
    const Out o(x[7], [&] { return make(q, q.sizes(), dtype(x[12])); });
    const Out lse(x[8], [&] { return make(q, {q.size(1), q.size(0)}, at::kFloat); });
    auto st = [](const at::Tensor &t) { return pa_strides{0, t.stride(0), t.stride(1)}; };
    const pa_prefill_params p = {(int32_t)(cu.numel() - 1), (int32_t)q.size(1), (int32_t)k.size(1), (int32_t)q.size(2),
                                 integer(x[4]), integer32(x[10]), number(x[11]), st(q), st(k), st(v), st(o.t),
                                 out_dtype(o.t.scalar_type())};
    const Out ws(x[9], [&] { return make_bytes(q, pa_prefill_workspace_bytes(&p)); });
    run([&] {
        return pa_prefill_varlen(&p, q.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)cu.data_ptr(), q.size(0),
                                 (const int32_t *)row_ptr.data_ptr(), (const int32_t *)col_idx.data_ptr(), col_idx.numel(),
                                 o.ptr(), (float *)lse.ptr(), ws.ptr(), (size_t)ws.t.numel(), stream());
    });
    return tuple(o, lse, ws);
}

// q, k, v, o, lse, d_o, row_ptr, col_idx, dq, dk, dv, workspace, block, softmax_scale
PyObject *prefill_backward(PyObject *const *x)
{
    const at::Tensor &q = tensor(x[0]), &k = tensor(x[1]), &v = tensor(x[2]), &o = tensor(x[3]), &lse = tensor(x[4]),
                     &d_o = tensor(x[5]), &row_ptr = tensor(x[6]), &col_idx = tensor(x[7]);
    expect(d_o.strides() == o.strides() && o.scalar_type() == at::kBFloat16 && d_o.scalar_type() == at::kBFloat16,
           "o and d_o are bfloat16 of the same strides");
    const pa_prefill_params p = prefill_params(q, k, v, o, x[12], x[13]);
    const at::IntArrayRef q_size = q.sizes();
    const int64_t kv_size[4] = {q.size(0), q.size(1), k.size(2), q.size(3)};
    const Out dq(x[8], [&] { return make(q, q_size, at::kFloat); });
    const Out dk(x[9], [&] { return make(q, kv_size, at::kFloat); });
    const Out dv(x[10], [&] { return make(q, kv_size, at::kFloat); });
    const int64_t nnz = col_idx.numel();
    const Out ws(x[11], [&] { return make_bytes(q, pa_prefill_backward_workspace_bytes(&p, nnz) + 256); });
    const uintptr_t at0 = (uintptr_t)ws.ptr(), at = (at0 + 255) & ~(uintptr_t)255;
    const int64_t left = ws.t.numel() - (int64_t)(at - at0);
    run([&] {
        return pa_prefill_backward(&p, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), (const float *)lse.data_ptr(),
                                   d_o.data_ptr(), (const int32_t *)row_ptr.data_ptr(), (const int32_t *)col_idx.data_ptr(),
                                   nnz, (float *)dq.ptr(), (float *)dk.ptr(), (float *)dv.ptr(), (void *)at,
                                   (size_t)(left > 0 ? left : 0), stream());
    });
    return tuple(dq, dk, dv, ws);
}

pa_decode_params decode_params(const at::Tensor &q, const at::Tensor &k, const at::Tensor &v, PyObject *window, PyObject *sink,
                               PyObject *block, PyObject *scale, at::ScalarType o_type)
{
    expect(q.dim() == 3, "expected q [batch, head, head_dim]");
    const pa_strides sk = strides4(k), sv = strides4(v);
    return {(int32_t)q.size(0), (int32_t)q.size(1), (int32_t)k.size(2), (int32_t)q.size(2), integer32(block), integer32(window),
            integer32(sink), k.size(1), number(scale), sk, sv, out_dtype(o_type)};
}
void check_decode(const at::Tensor &lens, const at::Tensor &q, const at::Tensor &o)
{
    expect(is_int32(lens) && q.is_contiguous() && o.is_contiguous(), "cache_lens is int32, q and o are contiguous");
}

// q, k_cache, v_cache, cache_lens, window_blocks, sink_blocks, o, lse, workspace, block, softmax_scale, o_dtype
PyObject *decode(PyObject *const *x)
{
    const at::Tensor &q = tensor(x[0]), &k = tensor(x[1]), &v = tensor(x[2]), &lens = tensor(x[3]);
    expect(q.dim() == 3, "expected q [batch, head, head_dim]");
    const Out o(x[6], [&] { return make(q, q.sizes(), dtype(x[11])); });
    const Out lse(x[7], [&] { return make(q, {q.size(0), q.size(1)}, at::kFloat); });
    const pa_decode_params p = decode_params(q, k, v, x[4], x[5], x[9], x[10], o.t.scalar_type());
    const Out ws(x[8], [&] { return make_bytes(q, pa_decode_workspace_bytes(&p)); });
    check_decode(lens, q, o.t);
    run([&] {
        return pa_decode(&p, q.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)lens.data_ptr(), o.ptr(),
                         (float *)lse.ptr(), ws.ptr(), (size_t)ws.t.numel(), stream());
    });
    return tuple(o, lse, ws);
}

// q, k_cache, v_cache, cache_lens, window_blocks, sink_blocks, o, lse, block, softmax_scale
PyObject *decode_static(PyObject *const *x)
{
    const at::Tensor &q = tensor(x[0]), &k = tensor(x[1]), &v = tensor(x[2]), &lens = tensor(x[3]), &o = tensor(x[6]),
                     &lse = tensor(x[7]);
    check_decode(lens, q, o);
    const pa_decode_params p = decode_params(q, k, v, x[4], x[5], x[8], x[9], o.scalar_type());
    run([&] {
        return pa_decode_static(&p, q.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)lens.data_ptr(), o.data_ptr(),
                                (float *)lse.data_ptr(), stream());
    });
    Py_RETURN_NONE;
}

pa_paged_params paged_params(int64_t batch, int64_t hq, int64_t hkv, int64_t d, const at::Tensor &k, const at::Tensor &v,
                             const at::Tensor &table, int32_t block, int32_t window, int32_t sink, float scale, pa_dtype o_type)
{
    const pa_strides sk = strides4(k), sv = strides4(v);
    expect(table.dim() == 2, "expected a block table [batch, max_blocks]");
    return {(int32_t)batch, (int32_t)hq, (int32_t)hkv, (int32_t)d, block, window, sink, (int32_t)k.size(0),
            (int32_t)table.size(1), scale, sk, sv, o_type};
}

// q, k_pool, v_pool, block_table, cache_lens, window_blocks, sink_blocks, o, lse, workspace, block, softmax_scale, o_dtype
PyObject *decode_paged(PyObject *const *x)
{
    const at::Tensor &q = tensor(x[0]), &k = tensor(x[1]), &v = tensor(x[2]), &table = tensor(x[3]), &lens = tensor(x[4]);
    expect(q.dim() == 3 && k.dim() == 4, "expected q [batch, head, head_dim] and pools [n_pages, block, head, head_dim]");
    const Out o(x[7], [&] { return make(q, q.sizes(), dtype(x[12])); });
    const Out lse(x[8], [&] { return make(q, {q.size(0), q.size(1)}, at::kFloat); });
    const int32_t block = integer32(x[10]);
    expect(k.size(1) == block && is_int32(table) && table.is_contiguous(),
           "pages hold `block` tokens, the table is contiguous int32");
    const pa_paged_params p = paged_params(q.size(0), q.size(1), k.size(2), q.size(2), k, v, table, block, integer32(x[5]),
                                           integer32(x[6]), number(x[11]), out_dtype(o.t.scalar_type()));
    const Out ws(x[9], [&] { return make_bytes(q, pa_decode_paged_workspace_bytes(&p)); });
    check_decode(lens, q, o.t);
    run([&] {
        return pa_decode_paged(&p, q.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)table.data_ptr(),
                               (const int32_t *)lens.data_ptr(), o.ptr(), (float *)lse.ptr(), ws.ptr(), (size_t)ws.t.numel(),
                               stream());
    });
    return tuple(o, lse, ws);
}

// k_new, v_new, k_pool, v_pool, block_table, cache_lens, block
PyObject *kv_append(PyObject *const *x)
{
    const at::Tensor &kn = tensor(x[0]), &vn = tensor(x[1]), &k = tensor(x[2]), &v = tensor(x[3]), &table = tensor(x[4]),
                     &lens = tensor(x[5]);
    expect(kn.dim() == 3 && kn.is_contiguous() && vn.is_contiguous() && is_int32(lens),
           "k_new and v_new [batch, head, head_dim] are contiguous, cache_lens is int32");
    const pa_paged_params p = paged_params(kn.size(0), kn.size(1), kn.size(1), kn.size(2), k, v, table, integer32(x[6]), 0, 0,
                                           0.f, PA_BF16);
    run([&] {
        return pa_kv_append(&p, kn.data_ptr(), vn.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)table.data_ptr(),
                            (int32_t *)lens.data_ptr(), stream());
    });
    Py_RETURN_NONE;
}

// seq_len, block, window_blocks, sink_blocks, tile, row_ptr, col_idx, device; tile None: pa_build_layout, 0:
// pa_build_window_layout, else pa_build_tile_layout
PyObject *build_layout(PyObject *const *x)
{
    const int64_t seq_len = integer(x[0]);
    const int32_t block = integer32(x[1]), window = integer32(x[2]), sink = integer32(x[3]);
    const int32_t tile = x[4] == Py_None ? -1 : integer32(x[4]);
    int32_t rows = 0;
    int64_t nnz = 0;
    run([&] {
        return tile < 0    ? pa_layout_size(seq_len, block, window, sink, &rows, &nnz)
               : tile == 0 ? pa_window_layout_size(seq_len, block, window, sink, &rows, &nnz)
                           : pa_tile_layout_size(seq_len, block, window, sink, tile, &rows, &nnz);
    });
    auto fresh = [&](int64_t n) {
        if (!THPDevice_Check(x[7])) raise(PyExc_TypeError, "expected a torch.device");
        const c10::Device device = reinterpret_cast<THPDevice *>(x[7])->device;
        return empty({n}, at::TensorOptions().dtype(at::kInt).device(device));
    };
    const Out row_ptr(x[5], [&] { return fresh((int64_t)rows + 1); });
    const Out col_idx(x[6], [&] { return fresh(nnz); });
    expect(is_int32(row_ptr.t) && is_int32(col_idx.t) && row_ptr.t.numel() >= (int64_t)rows + 1,
           "row_ptr and col_idx are int32, row_ptr has a row more than the layout");
    run([&] {
        int32_t *rp = (int32_t *)row_ptr.ptr(), *ci = (int32_t *)col_idx.ptr();
        const int64_t room = col_idx.t.numel();
        return tile < 0    ? pa_build_layout(seq_len, block, window, sink, rp, ci, room, stream())
               : tile == 0 ? pa_build_window_layout(seq_len, block, window, sink, rp, ci, room, stream())
                           : pa_build_tile_layout(seq_len, block, window, sink, tile, rp, ci, room, stream());
    });
    return Py_BuildValue("(NN)", row_ptr.object(), col_idx.object());
}

// Wraps a function of N positional arguments.
template <int N, PyObject *(*F)(PyObject *const *)>
PyObject *call(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Raised &) {
    } catch (const std::exception &) {  // (as torch's own functions raise it: OutOfMemoryError and so on)
        torch::translate_exception_to_python(std::current_exception());
    }
    return nullptr;
}

PyObject *set_error(PyObject *, PyObject *type)
{
    Py_XSETREF(g_error, Py_NewRef(type));
    Py_RETURN_NONE;
}

#define PA_METHOD(name, n) {#name, (PyCFunction)(void (*)())call<n, name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"set_error", set_error, METH_O, nullptr}, PA_METHOD(prefill, 12),       PA_METHOD(prefill_varlen, 13),
    PA_METHOD(prefill_backward, 14),           PA_METHOD(decode, 12),        PA_METHOD(decode_static, 10),
    PA_METHOD(decode_paged, 13),               PA_METHOD(kv_append, 7),
    PA_METHOD(build_layout, 8),                {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls()
{
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "torch_version", PA_TORCH_VERSION) < 0) Py_CLEAR(m);
    return m;
}
