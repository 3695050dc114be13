// Native half of the Python binding: argument checks, output allocation and the call into the C ABI, without the interpreter.
//
// A decode step of one sequence runs for about 3 us on the device; marshalled in Python (descriptor fields through ctypes,
// device and stream context managers, a dozen attribute reads) the call took 16 us of host time, which was then also what a
// batch of 64 sequences took (8.6 us on the device).  Semantics are those of binding.py's docstrings: CUDA, contiguous tensors
// (ValueError), dtypes (TypeError), KlaError for a non-zero status, the current stream of q's device, outputs allocated from
// torch's caching allocator.  No arithmetic happens here.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <ATen/ops/zeros.h>
#include <c10/cuda/CUDAException.h>
#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include "kla.h"

namespace {

PyObject *g_kla_error = nullptr;   // binding.KlaError
PyObject *g_status_for = nullptr;  // binding._status_for: the binding's own status word of a device

struct Failed {};   // a Python exception has been set

[[noreturn]] void fail(PyObject *type, const char *msg, const char *name = nullptr)
{
    if (name) PyErr_Format(type, "%s %s", name, msg);
    else PyErr_SetString(type, msg);
    throw Failed();
}

const at::Tensor *opt_tensor(PyObject *o, const char *name)
{
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) fail(PyExc_ValueError, "must be a contiguous CUDA tensor", name);
    return &THPVariable_Unpack(o);
}
const at::Tensor &tensor(PyObject *o, const char *name)
{
    const at::Tensor *t = opt_tensor(o, name);
    if (!t) fail(PyExc_ValueError, "must be a tensor", name);
    return *t;
}
// device address of a contiguous CUDA tensor (null for none), as binding._dev
void *addr(const at::Tensor *t, const char *name)
{
    if (!t) return nullptr;
    if (!t->is_cuda() || !t->is_contiguous()) fail(PyExc_ValueError, "must be a contiguous CUDA tensor", name);
    return t->data_ptr();
}
float *addr_f32(const at::Tensor *t, const char *name)
{
    void *p = addr(t, name);
    if (t && t->scalar_type() != at::kFloat) fail(PyExc_TypeError, "must be torch.float32", name);
    return static_cast<float *>(p);
}
int32_t kla_dtype_of(const at::Tensor &t)
{
    if (t.scalar_type() == at::kFloat) return KLA_F32;
    if (t.scalar_type() == at::kBFloat16) return KLA_BF16;
    fail(PyExc_TypeError, "q, k, v, out must be float32 or bfloat16");
}
at::ScalarType dtype_arg(PyObject *o, const at::Tensor &like)
{
    if (o == Py_None) return like.scalar_type();
    if (!THPDtype_Check(o)) fail(PyExc_TypeError, "out_dtype must be a torch.dtype");
    return reinterpret_cast<THPDtype *>(o)->scalar_type;
}
double number(PyObject *o)
{
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) throw Failed();
    return x;
}
long integer(PyObject *o)
{
    const long x = PyLong_AsLong(o);
    if (x == -1 && PyErr_Occurred()) throw Failed();
    return x;
}
// Larger buffers than a call needs are the caller's business; smaller ones would be read or written past their end.
void holds(const at::Tensor *t, int64_t n, const char *name)
{
    if (t && t->numel() < n) fail(PyExc_ValueError, "holds fewer elements than the call takes", name);
}
void one_dtype(const at::Tensor &q, const at::Tensor &k, const at::Tensor &v)
{
    if (k.scalar_type() != q.scalar_type() || v.scalar_type() != q.scalar_type()) fail(PyExc_TypeError, "q, k, v must share one dtype");
}
// Packed input: the host copy of the offsets, contiguous, and the number of sequences.
at::Tensor offsets(const at::Tensor &cu, PyObject *host_seqlens, int64_t *n_seq)
{
    if (cu.scalar_type() != at::kInt) fail(PyExc_TypeError, "cu_seqlens must be int32");
    const at::Tensor &host = tensor(host_seqlens, "host_seqlens");
    if (host.is_cuda() || host.scalar_type() != at::kInt) fail(PyExc_TypeError, "host_seqlens must be a CPU int32 tensor");
    *n_seq = cu.numel() - 1;
    holds(&host, *n_seq + 1, "host_seqlens");
    return host.contiguous();
}
bool has_shape(const at::Tensor &t, at::IntArrayRef shape) { return t.sizes() == shape; }

// The status word of a call: the caller's, else the binding's own of the device (kept alive by the binding).
int32_t *status_word(PyObject *given, c10::Device device)
{
    PyObject *o = given;   // borrowed
    if (o == Py_None) {
        PyObject *dev = PyLong_FromLong(device.index());
        o = dev ? PyObject_CallOneArg(g_status_for, dev) : nullptr;
        Py_XDECREF(dev);
        if (!o) throw Failed();
        Py_DECREF(o);
    }
    const at::Tensor &t = tensor(o, "status_word");
    void *p = addr(&t, "status_word");
    if (t.scalar_type() != at::kInt) fail(PyExc_TypeError, "must be torch.int32", "status_word");
    return static_cast<int32_t *>(p);
}

void check(kla_status st)
{
    if (st == KLA_OK) return;
    PyObject *e = PyObject_CallFunction(g_kla_error, "is", (int)st, kla_status_str(st));
    if (e) {
        PyErr_SetObject(g_kla_error, e);
        Py_DECREF(e);
    }
    throw Failed();
}

// kla_decode_step / kla_decode_steps / kla_dg_decode_step:
// (q, k, v, log_alpha, eta, eps, state_inout, out, out_dtype, flags, kind)   kind 0: one step, 1: steps, 2: diagonal gates
PyObject *decode(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 11) {
        PyErr_SetString(PyExc_TypeError, "decode: 11 arguments");
        return nullptr;
    }
    try {
        const at::Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
        const at::Tensor &la = tensor(a[3], "log_alpha"), &eta = tensor(a[4], "eta"), &state = tensor(a[6], "state_inout");
        const float eps = (float)number(a[5]);
        const long kind = integer(a[10]);
        const int lead = kind == 1 ? 1 : 0;
        if (q.dim() != 3 + lead || v.dim() < 1) fail(PyExc_ValueError, lead ? "q must be [n, B, H, d_k]" : "q must be [B, H, d_k]");
        const int64_t steps = lead ? q.size(0) : 1, B = q.size(lead), H = q.size(lead + 1), d_k = q.size(-1), d_v = v.size(-1);
        const at::Tensor *given = opt_tensor(a[7], "out");
        one_dtype(q, k, v);
        const int64_t units = steps * B * H;
        holds(&k, units * d_k, "k");
        holds(&v, units * d_v, "v");
        holds(&la, kind == 2 ? units * d_k : units, "log_alpha");
        holds(&eta, units, "eta");
        holds(&state, B * H * d_k * d_v, "state_inout");
        holds(given, units * d_v, "out");
        void *qa = addr(&q, "q");
        const c10::cuda::OptionalCUDAGuard guard(q.device());
        at::Tensor out;
        if (given) out = *given;
        else if (lead) out = at::empty({steps, B, H, d_v}, q.options().dtype(dtype_arg(a[8], q)));
        else out = at::empty({B, H, d_v}, q.options().dtype(dtype_arg(a[8], q)));
        kla_desc d = {};
        d.B = d.n_seq = (int32_t)B;
        d.T = 1;
        d.H = (int32_t)H;
        d.d_k = (int32_t)d_k;
        d.d_v = (int32_t)d_v;
        d.io_dtype = kla_dtype_of(q);
        d.out_dtype = kla_dtype_of(out);
        d.flags = (int32_t)integer(a[9]);
        d.stream = c10::cuda::getCurrentCUDAStream(q.device().index()).stream();
        void *ka = addr(&k, "k"), *va = addr(&v, "v"), *oa = addr(&out, "out");
        float *laa = addr_f32(&la, "log_alpha"), *ea = addr_f32(&eta, "eta"), *sa = addr_f32(&state, "state_inout");
        kla_status st;
        Py_BEGIN_ALLOW_THREADS
        st = kind == 2 ? kla_dg_decode_step(&d, qa, ka, va, laa, ea, eps, sa, oa) : kla_decode_steps(&d, (int32_t)steps, qa, ka, va, laa, ea, eps, sa, oa);
        Py_END_ALLOW_THREADS
        check(st);
        if (given) {
            Py_INCREF(a[7]);
            return a[7];
        }
        return THPVariable_Wrap(std::move(out));
    } catch (const Failed &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// kla_chunk_fwd (dg = 0) and kla_dg_fwd (dg = 1), without the measurement aids of binding.kla_chunk_fwd:
// (q, k, v, log_alpha, eta, eps, chunk, init_state, out, final_state, cu_seqlens, host_seqlens, out_dtype, flags,
//  want_final_state, status_word, dg) -> (out, final_state)
PyObject *forward(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 17) {
        PyErr_SetString(PyExc_TypeError, "forward: 17 arguments");
        return nullptr;
    }
    try {
        const at::Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
        const at::Tensor &la = tensor(a[3], "log_alpha"), &eta = tensor(a[4], "eta");
        const float eps = (float)number(a[5]);
        const int32_t chunk = (int32_t)integer(a[6]);
        const bool dg = integer(a[16]) != 0;
        if (q.dim() != 4 || v.dim() < 1) fail(PyExc_ValueError, "q must be [B, T, H, d_k]");
        const int64_t B = q.size(0), T = q.size(1), H = q.size(2), d_k = q.size(3), d_v = v.size(-1);
        if (!has_shape(k, q.sizes()) || !has_shape(v, {B, T, H, d_v})) fail(PyExc_ValueError, "q, k, v shapes disagree");
        if (!has_shape(eta, {B, T, H}) || !(dg ? has_shape(la, {B, T, H, d_k}) : has_shape(la, {B, T, H})))
            fail(PyExc_ValueError, dg ? "log_alpha must be [B, T, H, d_k] and eta [B, T, H]" : "log_alpha, eta must be [B, T, H]");
        one_dtype(q, k, v);
        int64_t n_seq = B;
        const at::Tensor *cu = opt_tensor(a[10], "cu_seqlens");
        at::Tensor host;
        if (cu) host = offsets(*cu, a[11], &n_seq);
        const at::Tensor *out_given = opt_tensor(a[8], "out"), *fin_given = opt_tensor(a[9], "final_state"), *init = opt_tensor(a[7], "init_state");
        holds(out_given, B * T * H * d_v, "out");
        holds(fin_given, n_seq * H * d_k * d_v, "final_state");
        void *qa = addr(&q, "q");
        const c10::cuda::OptionalCUDAGuard guard(q.device());
        at::Tensor out, fin, ws;
        if (out_given) out = *out_given;
        else out = at::empty({B, T, H, d_v}, q.options().dtype(dtype_arg(a[12], q)));
        if (fin_given) fin = *fin_given;
        else if (integer(a[14])) fin = at::empty({n_seq, H, d_k, d_v}, q.options().dtype(at::kFloat));
        if (init && !has_shape(*init, {n_seq, H, d_k, d_v})) fail(PyExc_ValueError, "init_state must be [n_seq, H, d_k, d_v]");
        kla_desc d = {};
        d.B = (int32_t)B;
        d.T = (int32_t)T;
        d.H = (int32_t)H;
        d.d_k = (int32_t)d_k;
        d.d_v = (int32_t)d_v;
        d.n_seq = (int32_t)n_seq;
        d.cu_seqlens = static_cast<const int32_t *>(addr(cu, "cu_seqlens"));
        d.host_seqlens = cu ? static_cast<const int32_t *>(host.data_ptr()) : nullptr;
        d.io_dtype = kla_dtype_of(q);
        d.out_dtype = kla_dtype_of(out);
        d.flags = (int32_t)integer(a[13]);
        d.stream = c10::cuda::getCurrentCUDAStream(q.device().index()).stream();
        if (!dg) d.status_word = status_word(a[15], q.device());   // (kernels of diagonal gates wait for nothing)
        if (!dg) {
            if (const size_t need = kla_chunk_fwd_workspace_bytes(&d, chunk)) {
                ws = at::empty({(int64_t)need}, q.options().dtype(at::kByte));
                d.workspace = ws.data_ptr();
                d.workspace_bytes = need;
            }
        }
        void *ka = addr(&k, "k"), *va = addr(&v, "v"), *oa = addr(&out, "out");
        float *laa = addr_f32(&la, "log_alpha"), *ea = addr_f32(&eta, "eta"), *ia = addr_f32(init, "init_state");
        float *fa = fin.defined() ? addr_f32(&fin, "final_state") : nullptr;
        kla_status st;
        Py_BEGIN_ALLOW_THREADS
        st = dg ? kla_dg_fwd(&d, qa, ka, va, laa, ea, eps, ia, oa, fa) : kla_chunk_fwd(&d, qa, ka, va, laa, ea, eps, chunk, ia, oa, fa);
        Py_END_ALLOW_THREADS
        check(st);
        PyObject *po, *pf;
        if (out_given) Py_INCREF(po = a[8]);
        else po = THPVariable_Wrap(std::move(out));
        if (fin_given || !fin.defined()) Py_INCREF(pf = a[9]);   // (None when no final state is wanted)
        else pf = THPVariable_Wrap(std::move(fin));
        if (!po || !pf) {
            Py_XDECREF(po);
            Py_XDECREF(pf);
            return nullptr;
        }
        PyObject *r = PyTuple_New(2);
        PyTuple_SET_ITEM(r, 0, po);
        PyTuple_SET_ITEM(r, 1, pf);
        return r;
    } catch (const Failed &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// kla_bwd: (q, k, v, log_alpha, eta, eps, d_out, init_state, d_final_state, cu_seqlens, host_seqlens, flags, want_dinit_state,
// workspace, status_word) -> dict
PyObject *backward(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 15) {
        PyErr_SetString(PyExc_TypeError, "backward: 15 arguments");
        return nullptr;
    }
    try {
        const at::Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
        const at::Tensor &la = tensor(a[3], "log_alpha"), &eta = tensor(a[4], "eta"), &d_out = tensor(a[6], "d_out");
        const float eps = (float)number(a[5]);
        if (q.dim() != 4 || v.dim() < 1) fail(PyExc_ValueError, "q must be [B, T, H, d_k]");
        const int64_t B = q.size(0), T = q.size(1), H = q.size(2), d_k = q.size(3), d_v = v.size(-1);
        if (!has_shape(d_out, {B, T, H, d_v}) || d_out.scalar_type() != q.scalar_type())
            fail(PyExc_ValueError, "d_out must be [B, T, H, d_v] with the dtype of q");
        one_dtype(q, k, v);
        int64_t n_seq = B;
        const at::Tensor *cu = opt_tensor(a[9], "cu_seqlens"), *init = opt_tensor(a[7], "init_state"), *dfin = opt_tensor(a[8], "d_final_state");
        const at::Tensor *given = opt_tensor(a[13], "workspace");
        at::Tensor host;
        if (cu) host = offsets(*cu, a[10], &n_seq);
        holds(&k, q.numel(), "k");
        holds(&v, B * T * H * d_v, "v");
        holds(&la, B * T * H, "log_alpha");
        holds(&eta, B * T * H, "eta");
        holds(init, n_seq * H * d_k * d_v, "init_state");
        holds(dfin, n_seq * H * d_k * d_v, "d_final_state");
        void *qa = addr(&q, "q");
        const c10::cuda::OptionalCUDAGuard guard(q.device());
        kla_desc d = {};
        d.B = (int32_t)B;
        d.T = (int32_t)T;
        d.H = (int32_t)H;
        d.d_k = (int32_t)d_k;
        d.d_v = (int32_t)d_v;
        d.n_seq = (int32_t)n_seq;
        d.cu_seqlens = static_cast<const int32_t *>(addr(cu, "cu_seqlens"));
        d.host_seqlens = cu ? static_cast<const int32_t *>(host.data_ptr()) : nullptr;
        d.io_dtype = kla_dtype_of(q);
        d.out_dtype = KLA_F32;
        d.flags = (int32_t)integer(a[11]);
        d.stream = c10::cuda::getCurrentCUDAStream(q.device().index()).stream();
        d.status_word = status_word(a[14], q.device());
        const auto f32 = q.options().dtype(at::kFloat);
        const bool want = PyObject_IsTrue(a[12]) == 1;
        at::Tensor g[6] = {at::empty({B, T, H, d_k}, f32), at::empty({B, T, H, d_k}, f32), at::empty({B, T, H, d_v}, f32),
                           at::empty({B, T, H}, f32), at::empty({B, T, H}, f32), want ? at::empty({n_seq, H, d_k, d_v}, f32) : at::Tensor()};
        at::Tensor ws;
        if (given) ws = *given;
        else if (const size_t need = kla_bwd_workspace_bytes(&d)) ws = at::empty({(int64_t)need}, q.options().dtype(at::kByte));
        if (ws.defined()) {
            d.workspace = addr(&ws, "workspace");
            d.workspace_bytes = (size_t)ws.numel() * ws.element_size();
        }
        void *ka = addr(&k, "k"), *va = addr(&v, "v"), *da = addr(&d_out, "d_out");
        float *laa = addr_f32(&la, "log_alpha"), *ea = addr_f32(&eta, "eta"), *ia = addr_f32(init, "init_state"), *fa = addr_f32(dfin, "d_final_state");
        float *ga[6];
        for (int i = 0; i < 6; ++i) ga[i] = g[i].defined() ? static_cast<float *>(g[i].data_ptr()) : nullptr;
        kla_status st;
        Py_BEGIN_ALLOW_THREADS
        st = kla_bwd(&d, qa, ka, va, laa, ea, eps, ia, da, fa, ga[0], ga[1], ga[2], ga[3], ga[4], ga[5]);
        Py_END_ALLOW_THREADS
        check(st);
        static const char *const names[6] = {"dq", "dk", "dv", "dlog_alpha", "deta", "dinit_state"};
        PyObject *r = PyDict_New();
        for (int i = 0; r && i < 6; ++i) {
            PyObject *o = g[i].defined() ? THPVariable_Wrap(std::move(g[i])) : (Py_INCREF(Py_None), Py_None);
            if (!o || PyDict_SetItemString(r, names[i], o) != 0) Py_CLEAR(r);
            Py_XDECREF(o);
        }
        return r;
    } catch (const Failed &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// new_status_word(device index) -> int32[1], zero.  Made on a stream of its own and complete on return: on the current stream, if that is
// being captured, the word would belong to the graph, whose every replay would clear it.
PyObject *new_status_word(PyObject *, PyObject *index)
{
    try {
        const c10::Device device(c10::kCUDA, (c10::DeviceIndex)integer(index));
        const c10::cuda::CUDAGuard guard(device);
        const c10::cuda::CUDAStreamCaptureModeGuard relaxed(cudaStreamCaptureModeRelaxed);   // (of this thread, for a moment)
        cudaStream_t own;
        C10_CUDA_CHECK(cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking));
        at::Tensor word;
        {
            const c10::cuda::CUDAStreamGuard on(c10::cuda::getStreamFromExternal(own, device.index()));
            word = at::zeros({1}, at::TensorOptions().device(device).dtype(at::kInt));
        }
        C10_CUDA_CHECK(cudaStreamSynchronize(own));
        C10_CUDA_CHECK(cudaStreamDestroy(own));
        return THPVariable_Wrap(std::move(word));
    } catch (const Failed &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

PyObject *init(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 2) {
        PyErr_SetString(PyExc_TypeError, "init: 2 arguments");
        return nullptr;
    }
    Py_INCREF(g_kla_error = a[0]);
    Py_INCREF(g_status_for = a[1]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"init", (PyCFunction)(void (*)())init, METH_FASTCALL, nullptr},
                         {"decode", (PyCFunction)(void (*)())decode, METH_FASTCALL, nullptr},
                         {"forward", (PyCFunction)(void (*)())forward, METH_FASTCALL, nullptr},
                         {"new_status_word", new_status_word, METH_O, nullptr},
                         {"backward", (PyCFunction)(void (*)())backward, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host(void) { return PyModule_Create(&module); }
