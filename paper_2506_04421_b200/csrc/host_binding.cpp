// The Python side of the calls, in native code: checks of the tensors, allocation of the results, the stream and the call
// of the C entry point.  In Python (tensor attributes, allocations through the interpreter, a ctypes call of a dozen
// arguments) a call of a small scale was host time only: 9.0 us for a step and 7.2 to 7.8 for the sampler's two calls.
// Here the host needs 5.1 us for a step without LSE, 6.1 with it, 3.7 where both outputs are given (an allocation is 1.3
// and the rest mostly the launch), 2.8 for an accumulation; the GPU needs 3.4 to 3.8 in a graph, and takes plain
// launches in a row every 5.2 to 6.2.
//
// The module holds no reference to the library: bind() takes the handle of the one the package loaded.  Every function
// returns its results, or the entry point's status as an int where that is not HMAR_OK.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <c10/util/SmallVector.h>
#include <dlfcn.h>

#include "../../include/hmar.h"

namespace py = pybind11;

namespace {

struct Entry {
#define HMAR_ENTRIES(X)                                                                                                          \
    X(hmar_attn_fwd) X(hmar_attn_fwd_f32) X(hmar_attn_fwd_window) X(hmar_attn_fwd_window_f32) X(hmar_attn_fwd_packed)            \
    X(hmar_attn_bwd) X(hmar_attn_bwd_f32) X(hmar_attn_bwd_window) X(hmar_attn_bwd_window_f32) X(hmar_attn_bwd_packed)            \
    X(hmar_attn_bwd_workspace_bytes) X(hmar_attn_scale_step) X(hmar_attn_scale_step_f32) X(hmar_attn_scale_step_strided)         \
    X(hmar_recon_accumulate) X(hmar_recon_downsample)
#define X(name) decltype(&::name) name = nullptr;
    HMAR_ENTRIES(X)
#undef X
} entry;

// A tensor argument; None is an undefined tensor.
const at::Tensor& tensor(PyObject* o) {
    static const at::Tensor none;
    if (o == Py_None) return none;
    if (!THPVariable_Check(o)) TORCH_CHECK_TYPE(false, "expected a tensor, got ", Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}

void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }

template <typename... T>
void need(const T&... t) {
    if (!((!t.defined() || (t.is_cuda() && t.is_contiguous())) && ...)) TORCH_CHECK_VALUE(false, "tensors must be contiguous CUDA tensors");
}

void need_dims(const at::Tensor& t, int64_t n) {
    if (!t.defined() || t.dim() != n) TORCH_CHECK_VALUE(false, "expected a tensor of ", n, " dimensions");
}

bool is_f32(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return true;
    if (t.scalar_type() == at::kBFloat16) return false;
    TORCH_CHECK_TYPE(false, "tensors must be bfloat16 or float32");
}

long long integer(PyObject* o) {
    if (PyLong_Check(o)) {
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) throw py::error_already_set();
        return v;
    }
    const py::object number = py::reinterpret_steal<py::object>(PyNumber_Long(o));
    if (!number) throw py::error_already_set();
    const long long v = PyLong_AsLongLong(number.ptr());
    if (v == -1 && PyErr_Occurred()) throw py::error_already_set();
    return v;
}

// An integer or an integer type (numpy's, a tensor of one); floats are refused.
long long index(PyObject* o) {
    if (PyLong_Check(o)) return integer(o);
    const py::object number = py::reinterpret_steal<py::object>(PyNumber_Index(o));
    if (!number) throw py::error_already_set();
    return integer(number.ptr());
}

// An integer, or something equal to one (4.0); other numbers and text are refused.
long long whole(PyObject* o) {
    if (PyLong_Check(o)) return integer(o);
    const py::object number = py::reinterpret_steal<py::object>(PyNumber_Long(o));
    if (!number) throw py::error_already_set();
    const int equal = PyObject_RichCompareBool(o, number.ptr(), Py_EQ);
    if (equal < 0) throw py::error_already_set();
    if (equal == 0) TORCH_CHECK_VALUE(false, "expected a whole number");
    return integer(number.ptr());
}

float real(PyObject* o) {
    if (PyFloat_Check(o)) return (float)PyFloat_AS_DOUBLE(o);
    const py::object number = py::reinterpret_steal<py::object>(PyNumber_Float(o));
    if (!number) throw py::error_already_set();
    return (float)PyFloat_AS_DOUBLE(number.ptr());
}

bool truth(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw py::error_already_set();
    return v != 0;
}

using Sides = c10::SmallVector<int, HMAR_MAX_SCALES>;

Sides sides_of(PyObject* o) {
    if (PyObject_Size(o) < 0) throw py::error_already_set();
    const py::object items = py::reinterpret_steal<py::object>(PySequence_Fast(o, "side_lens must be a sequence"));
    if (!items) throw py::error_already_set();
    Sides s;
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(items.ptr()); ++i) s.push_back((int)integer(PySequence_Fast_GET_ITEM(items.ptr(), i)));
    return s;
}

// None: torch's current stream on the current device; otherwise the stream's handle as an int.
void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    void* s = PyLong_AsVoidPtr(o);
    if (s == nullptr && PyErr_Occurred()) throw py::error_already_set();
    return s;
}

at::Tensor or_empty(const at::Tensor& given, const at::Tensor& like, at::IntArrayRef shape, at::ScalarType type) {
    return given.defined() ? given : at::empty(shape, like.options().dtype(type));
}

// The caller's object where it gave one, a new one otherwise.
PyObject* wrap(PyObject* given, const at::Tensor& t) {
    if (given != Py_None) return Py_NewRef(given);
    return THPVariable_Wrap(t);
}

template <typename... T>
PyObject* results(T... o) {
    PyObject* objects[] = {o...};
    PyObject* tuple = PyTuple_New(sizeof...(o));
    Py_ssize_t i = 0;
    bool ok = tuple != nullptr;
    for (PyObject* x : objects) ok = ok && x != nullptr;
    for (PyObject* x : objects) {
        if (ok) PyTuple_SET_ITEM(tuple, i++, x);
        else Py_XDECREF(x);
    }
    if (!ok) Py_CLEAR(tuple);
    return tuple;
}

// The entry points run without the interpreter's lock: a launch waits where the queue of launches is full.  What is checked,
// converted or asked for is so in statements before the call, in the order of the checks: the order in which a call's
// arguments are evaluated is the compiler's.
template <typename F, typename... A>
int call(F f, A... a) {
    py::gil_scoped_release no_lock;
    return f(a...);
}

void need_args(Py_ssize_t n, Py_ssize_t expected) {
    if (n != expected) TORCH_CHECK_TYPE(false, "wrong number of arguments");
    if (entry.hmar_attn_fwd == nullptr) TORCH_CHECK_VALUE(false, "the library is not bound");
}

// fwd(q, k, v, out, lse, side_lens, softmax_scale, stream, window)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 9);
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]);
    need(q, k, v, tensor(a[3]), tensor(a[4]));
    need_dims(q, 4);
    const bool f32 = is_f32(q);
    const int B = (int)q.size(0), H = (int)q.size(1), D = (int)q.size(3);
    const at::Tensor out = or_empty(tensor(a[3]), q, q.sizes(), q.scalar_type());
    const at::Tensor lse = or_empty(tensor(a[4]), q, q.sizes().slice(0, 3), at::kFloat);
    const Sides sides = sides_of(a[5]);
    const float scale = real(a[6]);
    void* stream = stream_of(a[7]);
    const int window = (int)integer(a[8]);
    float* l = (float*)ptr(lse);
    int status;
    if (window != HMAR_WINDOW_MARKOV)
        status = f32 ? call(entry.hmar_attn_fwd_window_f32, (const float*)ptr(q), (const float*)ptr(k), (const float*)ptr(v), (float*)ptr(out), l, B, H, D, (int)sides.size(), sides.data(), window, scale, stream)
                     : call(entry.hmar_attn_fwd_window, ptr(q), ptr(k), ptr(v), ptr(out), l, B, H, D, (int)sides.size(), sides.data(), window, scale, stream);
    else
        status = f32 ? call(entry.hmar_attn_fwd_f32, (const float*)ptr(q), (const float*)ptr(k), (const float*)ptr(v), (float*)ptr(out), l, B, H, D, (int)sides.size(), sides.data(), scale, stream)
                     : call(entry.hmar_attn_fwd, ptr(q), ptr(k), ptr(v), ptr(out), l, B, H, D, (int)sides.size(), sides.data(), scale, stream);
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return results(wrap(a[3], out), wrap(a[4], lse));
    END_HANDLE_TH_ERRORS
}

// bwd(q, k, v, out, lse, dout, side_lens, softmax_scale, dq, dk, dv, workspace, stream, window)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 14);
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]), &out = tensor(a[3]), &lse = tensor(a[4]), &dout = tensor(a[5]);
    need(q, k, v, out, lse, dout, tensor(a[8]), tensor(a[9]), tensor(a[10]), tensor(a[11]));
    need_dims(q, 4);
    const bool f32 = is_f32(q);
    const int B = (int)q.size(0), H = (int)q.size(1), D = (int)q.size(3);
    const at::Tensor dq = or_empty(tensor(a[8]), q, q.sizes(), q.scalar_type());
    const at::Tensor dk = or_empty(tensor(a[9]), q, q.sizes(), q.scalar_type());
    const at::Tensor dv = or_empty(tensor(a[10]), q, q.sizes(), q.scalar_type());
    const Sides sides = sides_of(a[6]);
    const int n_sides = (int)sides.size();
    at::Tensor ws = tensor(a[11]);
    if (!ws.defined()) ws = at::empty({(int64_t)entry.hmar_attn_bwd_workspace_bytes(B, H, D, n_sides, sides.data())}, q.options().dtype(at::kByte));
    const float scale = real(a[7]);
    void* stream = stream_of(a[12]);
    const int window = (int)integer(a[13]);
    const float* l = (const float*)ptr(lse);
    int status;
    if (f32) {
        const float *fq = (const float*)ptr(q), *fk = (const float*)ptr(k), *fv = (const float*)ptr(v), *fo = (const float*)ptr(out), *fg = (const float*)ptr(dout);
        float *gq = (float*)ptr(dq), *gk = (float*)ptr(dk), *gv = (float*)ptr(dv);
        status = window != HMAR_WINDOW_MARKOV
                     ? call(entry.hmar_attn_bwd_window_f32, fq, fk, fv, fo, l, fg, gq, gk, gv, ptr(ws), ws.nbytes(), B, H, D, n_sides, sides.data(), window, scale, stream)
                     : call(entry.hmar_attn_bwd_f32, fq, fk, fv, fo, l, fg, gq, gk, gv, ptr(ws), ws.nbytes(), B, H, D, n_sides, sides.data(), scale, stream);
    } else {
        status = window != HMAR_WINDOW_MARKOV
                     ? call(entry.hmar_attn_bwd_window, ptr(q), ptr(k), ptr(v), ptr(out), l, ptr(dout), ptr(dq), ptr(dk), ptr(dv), ptr(ws), ws.nbytes(), B, H, D, n_sides, sides.data(), window, scale, stream)
                     : call(entry.hmar_attn_bwd, ptr(q), ptr(k), ptr(v), ptr(out), l, ptr(dout), ptr(dq), ptr(dk), ptr(dv), ptr(ws), ws.nbytes(), B, H, D, n_sides, sides.data(), scale, stream);
    }
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return results(wrap(a[8], dq), wrap(a[9], dk), wrap(a[10], dv));
    END_HANDLE_TH_ERRORS
}

// fwd_packed(qkv, out, lse, side_lens, softmax_scale, stream)
PyObject* fwd_packed(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 6);
    const at::Tensor& qkv = tensor(a[0]);
    need(qkv, tensor(a[1]), tensor(a[2]));
    need_dims(qkv, 5);
    const int64_t B = qkv.size(0), L = qkv.size(1), H = qkv.size(3), D = qkv.size(4);
    if (qkv.size(2) != 3 || is_f32(qkv)) TORCH_CHECK_VALUE(false, "qkv must be bfloat16 [B, L, 3, H, D]");
    const at::Tensor out = or_empty(tensor(a[1]), qkv, {B, L, H, D}, qkv.scalar_type());
    const at::Tensor lse = or_empty(tensor(a[2]), qkv, {B, H, L}, at::kFloat);
    const Sides sides = sides_of(a[3]);
    const float scale = real(a[4]);
    void* stream = stream_of(a[5]);
    const int status = call(entry.hmar_attn_fwd_packed, ptr(qkv), ptr(out), (float*)ptr(lse), (int)B, (int)H, (int)D, (int)sides.size(), sides.data(), scale, stream);
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return results(wrap(a[1], out), wrap(a[2], lse));
    END_HANDLE_TH_ERRORS
}

// bwd_packed(qkv, out, lse, dout, side_lens, softmax_scale, dqkv, workspace, stream)
PyObject* bwd_packed(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 9);
    const at::Tensor &qkv = tensor(a[0]), &out = tensor(a[1]), &lse = tensor(a[2]), &dout = tensor(a[3]);
    need(qkv, out, lse, dout, tensor(a[6]), tensor(a[7]));
    need_dims(qkv, 5);
    if (qkv.size(2) != 3 || is_f32(qkv)) TORCH_CHECK_VALUE(false, "qkv must be bfloat16 [B, L, 3, H, D]");
    const int B = (int)qkv.size(0), H = (int)qkv.size(3), D = (int)qkv.size(4);
    const at::Tensor dqkv = or_empty(tensor(a[6]), qkv, qkv.sizes(), qkv.scalar_type());
    const Sides sides = sides_of(a[4]);
    at::Tensor ws = tensor(a[7]);
    if (!ws.defined()) ws = at::empty({(int64_t)entry.hmar_attn_bwd_workspace_bytes(B, H, D, (int)sides.size(), sides.data())}, qkv.options().dtype(at::kByte));
    const float scale = real(a[5]);
    void* stream = stream_of(a[8]);
    const int status = call(entry.hmar_attn_bwd_packed, ptr(qkv), ptr(out), (const float*)ptr(lse), ptr(dout), ptr(dqkv), ptr(ws), ws.nbytes(), B, H, D, (int)sides.size(), sides.data(), scale, stream);
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return wrap(a[6], dqkv);
    END_HANDLE_TH_ERRORS
}

// scale_step(q, k_prev, v_prev, k_cur, v_cur, side_prev, side_cur, softmax_scale, out, lse, want_lse, stream)
PyObject* scale_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 12);
    const at::Tensor &q = tensor(a[0]), &kp = tensor(a[1]), &vp = tensor(a[2]), &kc = tensor(a[3]), &vc = tensor(a[4]);
    need(q, kp, vp, kc, vc, tensor(a[8]), tensor(a[9]));
    need_dims(q, 4);
    const bool f32 = is_f32(q);
    const int B = (int)q.size(0), H = (int)q.size(1), D = (int)q.size(3), prev = (int)integer(a[5]), cur = (int)integer(a[6]);
    const at::Tensor out = or_empty(tensor(a[8]), q, q.sizes(), q.scalar_type());
    at::Tensor lse = tensor(a[9]);
    const bool new_lse = !lse.defined() && truth(a[10]);
    if (new_lse) lse = at::empty(q.sizes().slice(0, 3), q.options().dtype(at::kFloat));
    const float scale = real(a[7]);
    void* stream = stream_of(a[11]);
    const int status = f32 ? call(entry.hmar_attn_scale_step_f32, (const float*)ptr(q), (const float*)ptr(kp), (const float*)ptr(vp), (const float*)ptr(kc), (const float*)ptr(vc), (float*)ptr(out), (float*)ptr(lse), B, H, D, prev, cur, scale, stream)
                           : call(entry.hmar_attn_scale_step, ptr(q), ptr(kp), ptr(vp), ptr(kc), ptr(vc), ptr(out), (float*)ptr(lse), B, H, D, prev, cur, scale, stream);
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return results(wrap(a[8], out), new_lse ? THPVariable_Wrap(lse) : Py_NewRef(a[9]));
    END_HANDLE_TH_ERRORS
}

// Distance between the heads of a [B,H,rows,D] view with contiguous rows and evenly spaced heads.
long long head_stride(const at::Tensor& t, long long H) {
    if (!t.defined()) return 0;
    need_dims(t, 4);
    const long long b = t.size(0), h = t.size(1), rows = t.size(2), D = t.size(3);
    if (!t.is_cuda() || t.stride(3) != 1 || t.stride(2) != D || (h > 1 && b > 1 && t.stride(0) != H * t.stride(1)))
        TORCH_CHECK_VALUE(false, "views must have contiguous rows and evenly spaced heads");
    return h > 1 ? t.stride(1) : (b > 1 ? t.stride(0) : rows * D);
}

// scale_step_strided(q, k_prev, v_prev, k_cur, v_cur, side_prev, side_cur, softmax_scale, out, lse, want_lse, stream)
PyObject* scale_step_strided(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 12);
    const at::Tensor &q = tensor(a[0]), &kp = tensor(a[1]), &vp = tensor(a[2]), &kc = tensor(a[3]), &vc = tensor(a[4]);
    need_dims(q, 4);
    if (is_f32(q)) TORCH_CHECK_TYPE(false, "hmar_attn_scale_step_strided takes bfloat16 tensors");
    const int B = (int)q.size(0), H = (int)q.size(1), D = (int)q.size(3), prev = (int)integer(a[5]), cur = (int)integer(a[6]);
    const at::Tensor out = or_empty(tensor(a[8]), q, q.sizes(), q.scalar_type());
    at::Tensor lse = tensor(a[9]);
    const bool new_lse = !lse.defined() && truth(a[10]);
    if (new_lse) lse = at::empty(q.sizes().slice(0, 3), q.options().dtype(at::kFloat));
    const long long q_stride = head_stride(q, H), prev_stride = head_stride(kp, H), cur_stride = head_stride(kc, H), out_stride = head_stride(out, H);
    const float scale = real(a[7]);
    void* stream = stream_of(a[11]);
    const int status = call(entry.hmar_attn_scale_step_strided, ptr(q), ptr(kp), ptr(vp), ptr(kc), ptr(vc), ptr(out), (float*)ptr(lse), B, H, D, prev, cur, q_stride, prev_stride, cur_stride, out_stride, scale, stream);
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return results(wrap(a[8], out), new_lse ? THPVariable_Wrap(lse) : Py_NewRef(a[9]));
    END_HANDLE_TH_ERRORS
}

// recon_accumulate(xhat, codebook, tokens_new, tokens_old, mask, tokens_out, stream)
PyObject* recon_accumulate(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 7);
    const at::Tensor &xhat = tensor(a[0]), &codebook = tensor(a[1]), &fresh = tensor(a[2]), &old = tensor(a[3]), &mask = tensor(a[4]), &chosen = tensor(a[5]);
    need(xhat, codebook, fresh, old, mask, chosen);
    need_dims(xhat, 4);
    if (!codebook.defined() || !fresh.defined() || xhat.scalar_type() != at::kFloat || codebook.scalar_type() != at::kFloat || fresh.scalar_type() != at::kInt)
        TORCH_CHECK_TYPE(false, "xhat and codebook must be float32, tokens int32");
    if (mask.defined() && mask.scalar_type() != at::kByte) TORCH_CHECK_TYPE(false, "mask must be uint8");
    const int status = call(entry.hmar_recon_accumulate, (float*)ptr(xhat), (const float*)ptr(codebook), (const int*)ptr(old), (const int*)ptr(fresh), (const unsigned char*)ptr(mask), (int*)ptr(chosen),
                            (int)xhat.size(0), (int)xhat.size(1), (int)codebook.size(0), (int)fresh.size(1), (int)xhat.size(2), stream_of(a[6]));
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return Py_NewRef(a[0]);
    END_HANDLE_TH_ERRORS
}

// recon_downsample(xhat, out_side, out, stream)
PyObject* recon_downsample(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    need_args(n, 4);
    const at::Tensor& xhat = tensor(a[0]);
    need(xhat, tensor(a[2]));
    need_dims(xhat, 4);
    if (xhat.scalar_type() != at::kFloat) TORCH_CHECK_TYPE(false, "xhat must be float32");
    const int64_t B = xhat.size(0), C = xhat.size(1), side = a[2] == Py_None ? index(a[1]) : whole(a[1]);
    const at::Tensor out = or_empty(tensor(a[2]), xhat, {B, C, side, side}, at::kFloat);
    if (out.scalar_type() != at::kFloat || out.sizes() != at::IntArrayRef({B, C, side, side})) TORCH_CHECK_VALUE(false, "out must be float32 [B, C, out_side, out_side]");
    const int status = call(entry.hmar_recon_downsample, (const float*)ptr(xhat), (float*)ptr(out), (int)B, (int)C, (int)xhat.size(2), (int)side, stream_of(a[3]));
    if (status != HMAR_OK) return PyLong_FromLong(status);
    return wrap(a[2], out);
    END_HANDLE_TH_ERRORS
}

// bind(handle): looks the entry points up in the loaded library.
PyObject* bind(PyObject*, PyObject* handle) {
    HANDLE_TH_ERRORS
    void* lib = PyLong_AsVoidPtr(handle);
    if (lib == nullptr) TORCH_CHECK_VALUE(false, "not the handle of a library");
#define X(name)                                                                        \
    entry.name = reinterpret_cast<decltype(entry.name)>(dlsym(lib, #name));            \
    if (entry.name == nullptr) TORCH_CHECK_VALUE(false, "the library has no " #name);
    HMAR_ENTRIES(X)
#undef X
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    FAST(fwd), FAST(bwd), FAST(fwd_packed), FAST(bwd_packed), FAST(scale_step), FAST(scale_step_strided), FAST(recon_accumulate), FAST(recon_downsample),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_hmar_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__hmar_host() { return PyModule_Create(&module); }
