// The Python binding's hot calls in native code: tensor checks, descriptor, workspace, output allocation and the C call.
//
// What bounds it: the smallest passes of a serving engine are two calls whose kernels take 3-10 us each, and marshalling
// one call in Python (about sixty interpreted operations: ctypes structures and pointers, per-tensor checks, stream and
// workspace look-up) took 25 us, so the GPU waited for the host.  Here the same work reads the tensors' C++ objects.
// One request with a 37-token suffix (state copy + Mamba-2 scan): 53.3 -> 16.4 us per pass; one 8K Mamba-2 request
// (composition of 8 chunks + 1024-token scan): 55.2 -> 35.6 us.  With today's kernels 11 and 29 us: the second is paced by the GPU, the
// first by the host again (10.3-11.2 us, 3.6 of them for three new tensors; 8.9 us from a graph).
//
// The functions mirror the Python wrappers of binding.py one to one (same arguments, results, checks and exceptions);
// binding.py keeps the signatures, the constants and everything that is not on the request path.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <mutex>

#include "../../include/lkv.h"

namespace {

// handed over once by binding.py
PyObject *g_error = nullptr;      // LkvError(status, where)
PyObject *g_workspace = nullptr;  // workspace(device, nbytes, raw stream): makes and caches a workspace
PyObject *g_ws_cache = nullptr;   // its cache: {(device index, raw stream): tensor}
PyObject *g_host_i32 = nullptr;   // any index sequence -> contiguous int32 numpy array

struct Failed {};   // a Python exception is set

[[noreturn]] void fail(PyObject *type, const char *msg) {
    PyErr_SetString(type, msg);
    throw Failed{};
}

const at::Tensor &tensor_of(PyObject *o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch.Tensor");
    return THPVariable_Unpack(o);
}

int dtype_code(const at::Tensor &t) {
    const auto st = t.scalar_type();
    if (st == at::kFloat) return LKV_DTYPE_F32;
    if (st == at::kBFloat16) return LKV_DTYPE_BF16;
    PyErr_Format(PyExc_TypeError, "unsupported dtype %s", c10::toString(st));
    throw Failed{};
}

// device pointer of a tensor argument; None = NULL
void *ptr_of(PyObject *o) {
    if (o == Py_None) return nullptr;
    const at::Tensor &t = tensor_of(o);
    if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_ValueError, "device buffers must be contiguous CUDA tensors");
    return t.data_ptr();
}

// Host int32 index array: an int32 buffer is read in place, anything else goes through binding._host_i32.
class HostInts {
public:
    explicit HostInts(PyObject *o) {
        if (o == Py_None) return;
        if (!take(o)) {
            PyErr_Clear();
            conv_ = PyObject_CallOneArg(g_host_i32, o);
            if (!conv_) throw Failed{};
            if (!take(conv_)) {
                Py_CLEAR(conv_);
                throw Failed{};
            }
        }
    }
    ~HostInts() {
        if (held_) PyBuffer_Release(&view_);
        Py_XDECREF(conv_);
    }
    HostInts(const HostInts &) = delete;
    HostInts &operator=(const HostInts &) = delete;
    const int32_t *data() const { return data_; }
    int size() const { return n_; }

private:
    bool take(PyObject *o) {
        if (THPVariable_Check(o) || !PyObject_CheckBuffer(o)) return false;
        if (PyObject_GetBuffer(o, &view_, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS) != 0) return false;
        if (view_.itemsize != 4 || !view_.format || view_.format[0] != 'i' || view_.format[1] != 0) {
            PyBuffer_Release(&view_);
            return false;
        }
        held_ = true;
        n_ = static_cast<int>(view_.len / 4);
        static int32_t none;   // an empty list is a valid pointer to nothing, as numpy's is
        data_ = view_.buf ? static_cast<const int32_t *>(view_.buf) : &none;
        return true;
    }
    Py_buffer view_{};
    bool held_ = false;
    PyObject *conv_ = nullptr;
    const int32_t *data_ = nullptr;
    int n_ = 0;
};

void *stream_of(PyObject *o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *raw = PyObject_GetAttrString(o, "cuda_stream");
    if (!raw) throw Failed{};
    void *s = PyLong_AsVoidPtr(raw);
    Py_DECREF(raw);
    if (!s && PyErr_Occurred()) throw Failed{};
    return s;
}

// The caller's workspace tensor, or the cached one of this device and the call's stream (binding.workspace).
template <typename Desc>
void set_workspace(Desc &d, PyObject *given, const at::Tensor &like, void *stream, int which, int n_units, int n_index) {
    if (given != Py_None) {
        const at::Tensor &t = tensor_of(given);
        d.workspace = t.data_ptr();
        d.workspace_bytes = static_cast<size_t>(t.numel());
        return;
    }
    const size_t need = lkv_workspace_bytes(which, &d, n_units, n_index);
    const int dev = like.device().index();
    const auto raw = static_cast<unsigned long long>(reinterpret_cast<uintptr_t>(stream));
    PyObject *key = Py_BuildValue("(iK)", dev, raw);
    if (!key) throw Failed{};
    PyObject *hit = PyDict_GetItemWithError(g_ws_cache, key);   // borrowed; the cache keeps it
    Py_DECREF(key);
    if (hit) {
        const at::Tensor &t = tensor_of(hit);
        if (static_cast<size_t>(t.numel()) >= need) {
            d.workspace = t.data_ptr();
            d.workspace_bytes = static_cast<size_t>(t.numel());
            return;
        }
    } else if (PyErr_Occurred()) {
        throw Failed{};
    }
    PyObject *made = PyObject_CallFunction(g_workspace, "inK", dev, static_cast<Py_ssize_t>(need), raw);
    if (!made) throw Failed{};
    const at::Tensor &t = tensor_of(made);
    d.workspace = t.data_ptr();
    d.workspace_bytes = static_cast<size_t>(t.numel());
    Py_DECREF(made);   // the cache holds it
}

void check(int st, const char *where) {
    if (st == LKV_OK) return;
    PyObject *e = PyObject_CallFunction(g_error, "is", st, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Failed{};
}

// The C call with the interpreter lock released, as ctypes does it: a launch into a full stream queue blocks, and so does the copy
// of a long index list; the engine's other threads run on meanwhile.  The arguments are plain C values by then, what they
// point to is held by the caller's frame.  A call may be several launches that pass data through the workspace, and threads that
// share a stream share its workspace: calls on one workspace take turns (the lock is picked by the workspace's address).
std::mutex g_turns[64];
template <typename... P, typename... A>
void call(const char *where, const void *workspace, int (*f)(P...), A... args) {
    int st;
    {
        struct Released {
            PyThreadState *state = PyEval_SaveThread();
            ~Released() { PyEval_RestoreThread(state); }
        } released;
        std::lock_guard<std::mutex> turn(g_turns[(reinterpret_cast<uintptr_t>(workspace) >> 9) % 64]);
        st = f(args...);
    }
    check(st, where);
}

int to_int(PyObject *o) {
    PyObject *i = PyNumber_Long(o);
    if (!i) throw Failed{};
    const long v = PyLong_AsLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    if (v != static_cast<int>(v)) fail(PyExc_OverflowError, "value does not fit an int32");
    return static_cast<int>(v);
}

at::Tensor new_tensor(at::IntArrayRef shape, at::ScalarType st, const at::Tensor &like) {
    return at::empty(shape, at::TensorOptions().dtype(st).device(like.device()));
}

// The output tensor passed by the caller (a new reference), or a new one when it is wanted; nullptr = none.
struct Output {
    PyObject *obj = nullptr;
    void *ptr = nullptr;
    Output() = default;
    Output(const Output &) = delete;
    Output &operator=(const Output &) = delete;
    ~Output() { Py_XDECREF(obj); }
    void given(PyObject *o) {
        ptr = ptr_of(o);
        Py_INCREF(o);
        obj = o;
    }
    void make(at::Tensor t) {
        ptr = t.data_ptr();
        obj = THPVariable_Wrap(std::move(t));
        if (!obj) throw Failed{};
    }
    PyObject *take() {
        PyObject *o = obj;
        obj = nullptr;
        if (!o) Py_RETURN_NONE;
        return o;
    }
};

PyObject *pair(Output &x, Output &y) {
    PyObject *t = PyTuple_New(2);
    if (!t) throw Failed{};
    PyTuple_SET_ITEM(t, 0, x.take());
    PyTuple_SET_ITEM(t, 1, y.take());
    return t;
}

template <typename F>
PyObject *guarded(F f) {
    HANDLE_TH_ERRORS   // exceptions of at::empty (out of memory and the like) become torch's own Python exceptions
    try {
        return f();
    } catch (const Failed &) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

at::ScalarType scalar_type_of(PyObject *o) {
    if (!THPDtype_Check(o)) fail(PyExc_TypeError, "expected a torch.dtype");
    return reinterpret_cast<THPDtype *>(o)->scalar_type;
}

void need_dim(const at::Tensor &t, int dim) {
    if (t.dim() != dim) fail(PyExc_ValueError, "a tensor has the wrong number of dimensions");
}

void need_args(Py_ssize_t n, Py_ssize_t want) {
    if (n != want) fail(PyExc_TypeError, "wrong number of arguments");
}

lkv_init_desc init_desc(const at::Tensor &states, PyObject *family, PyObject *compute) {
    need_dim(states, 4);
    lkv_init_desc d{};
    d.family = to_int(family);
    d.compute = to_int(compute);
    d.n_chunks = static_cast<int32_t>(states.size(0));
    d.H = static_cast<int32_t>(states.size(1));
    d.d_k = static_cast<int32_t>(states.size(2));
    d.d_v = static_cast<int32_t>(states.size(3));
    d.state_dtype = dtype_code(states);
    return d;
}

// (states, transitions, K, mode, S0, family, chunk_ids, sel_index, compute, workspace_t, stream) -> S0
PyObject *init_state(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 11);
        const at::Tensor &states = tensor_of(a[0]);
        lkv_init_desc d = init_desc(states, a[5], a[8]);
        const int K = to_int(a[2]);
        HostInts ids(a[6]);
        d.sel_index = to_int(a[7]);
        d.chunk_ids = ids.data();
        void *stream = stream_of(a[10]);
        const int mode = to_int(a[3]);
        set_workspace(d, a[9], states, stream, mode == LKV_INIT_EXACT ? LKV_WS_INIT : LKV_WS_INIT_LIST, 1, K);
        Output S0;
        if (a[4] != Py_None) S0.given(a[4]);
        else S0.make(new_tensor(states.sizes().slice(1), at::kFloat, states));
        call("lkv_init_state", d.workspace, lkv_init_state, ptr_of(a[0]), ptr_of(a[1]), K, mode, S0.ptr, &d,
             stream);
        return S0.take();
    });
}

// (states, transitions, chunk_ids, cu_k, n_req, mode, sel_index, S0, family, compute, workspace_t, stream) -> S0
PyObject *init_state_batched(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 12);
        const at::Tensor &states = tensor_of(a[0]);
        lkv_init_desc d = init_desc(states, a[8], a[9]);
        HostInts ids(a[2]), cu(a[3]), sel(a[6]);
        const int n_req = to_int(a[4]);
        void *stream = stream_of(a[11]);
        set_workspace(d, a[10], states, stream, LKV_WS_INIT_LIST, n_req, ids.size());
        Output S0;
        if (a[7] != Py_None) S0.given(a[7]);
        else S0.make(new_tensor({n_req, states.size(1), states.size(2), states.size(3)}, at::kFloat, states));
        call("lkv_init_state_batched", d.workspace, lkv_init_state_batched, ptr_of(a[0]), ptr_of(a[1]), ids.data(), cu.data(),
             n_req, to_int(a[5]), sel.data(), S0.ptr, &d, stream);
        return S0.take();
    });
}

// Descriptor of a GDN call over tokens of k [T, H_k, d_k]; the caller sets io_dtype.
lkv_gdn_desc gdn_desc(const at::Tensor &k, int64_t H_v, int64_t d_v, const HostInts &cu, PyObject *compute) {
    need_dim(k, 3);
    lkv_gdn_desc d{};
    d.T_total = static_cast<int32_t>(k.size(0));
    d.n_seq = cu.data() ? cu.size() - 1 : 1;
    d.cu_seqlens = cu.data();
    d.H_k = static_cast<int32_t>(k.size(1));
    d.d_k = static_cast<int32_t>(k.size(2));
    d.H_v = static_cast<int32_t>(H_v);
    d.d_v = static_cast<int32_t>(d_v);
    d.compute = to_int(compute);
    return d;
}

// (q, k, v, g, beta, S0, o, S_T, cu_seqlens, scale, compute, want_final_state, want_outputs, state_dtype, workspace_t,
//  stream) -> (o, S_T)
PyObject *gdn_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 16);
        const at::Tensor &v = tensor_of(a[2]);
        need_dim(v, 3);
        HostInts cu(a[8]);
        lkv_gdn_desc d = gdn_desc(tensor_of(a[0]), v.size(1), v.size(2), cu, a[10]);
        d.io_dtype = dtype_code(v);
        d.scale = static_cast<float>(PyFloat_AsDouble(a[9]));
        if (PyErr_Occurred()) throw Failed{};
        void *stream = stream_of(a[15]);
        set_workspace(d, a[14], v, stream, LKV_WS_GDN, d.n_seq, 0);
        Output o, S_T;
        if (a[6] != Py_None) o.given(a[6]);
        else if (PyObject_IsTrue(a[12]) == 1) o.make(new_tensor(v.sizes(), v.scalar_type(), v));
        if (a[7] != Py_None) S_T.given(a[7]);
        else if (PyObject_IsTrue(a[11]) == 1) S_T.make(new_tensor({d.n_seq, d.H_v, d.d_k, d.d_v}, scalar_type_of(a[13]), v));
        if (S_T.obj) d.state_dtype = dtype_code(THPVariable_Unpack(S_T.obj));
        call("lkv_gdn_fwd", d.workspace, lkv_gdn_fwd, ptr_of(a[0]), ptr_of(a[1]), ptr_of(a[2]),
             static_cast<float *>(ptr_of(a[3])), static_cast<float *>(ptr_of(a[4])), static_cast<float *>(ptr_of(a[5])), o.ptr,
             S_T.ptr, &d, stream);
        return pair(o, S_T);
    });
}

// (k, v, g, beta, states, transitions, cu_seqlens, compute, workspace_t, stream) -> (states, transitions)
PyObject *gdn_chunk_artifacts(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 10);
        const at::Tensor &k = tensor_of(a[0]), &v = tensor_of(a[1]);
        need_dim(v, 3);
        HostInts cu(a[6]);
        lkv_gdn_desc d = gdn_desc(k, v.size(1), v.size(2), cu, a[7]);
        d.io_dtype = dtype_code(k);
        void *stream = stream_of(a[9]);
        set_workspace(d, a[8], k, stream, LKV_WS_GDN, 2 * d.n_seq, 0);
        Output S, T;
        if (a[4] != Py_None) S.given(a[4]);
        else S.make(new_tensor({d.n_seq, d.H_v, d.d_k, d.d_v}, at::kFloat, k));
        if (a[5] != Py_None) T.given(a[5]);
        else T.make(new_tensor({d.n_seq, d.H_v, d.d_k, d.d_k}, at::kFloat, k));
        call("lkv_gdn_chunk_artifacts", d.workspace, lkv_gdn_chunk_artifacts, ptr_of(a[0]), ptr_of(a[1]),
             static_cast<float *>(ptr_of(a[2])), static_cast<float *>(ptr_of(a[3])), static_cast<float *>(S.ptr),
             static_cast<float *>(T.ptr), &d, stream);
        return pair(S, T);
    });
}

// (x, dt, A, B, C, S0, y, S_T, cu_seqlens, compute, want_final_state, want_outputs, state_dtype, workspace_t, stream) -> (y, S_T)
PyObject *ssd_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 15);
        const at::Tensor &x = tensor_of(a[0]), &B = tensor_of(a[3]);
        need_dim(x, 3);
        need_dim(B, 3);
        HostInts cu(a[8]);
        lkv_ssd_desc d{};
        d.T_total = static_cast<int32_t>(x.size(0));
        d.n_seq = cu.data() ? cu.size() - 1 : 1;
        d.cu_seqlens = cu.data();
        d.H = static_cast<int32_t>(x.size(1));
        d.P = static_cast<int32_t>(x.size(2));
        d.G = static_cast<int32_t>(B.size(1));
        d.N = static_cast<int32_t>(B.size(2));
        d.io_dtype = dtype_code(x);
        d.compute = to_int(a[9]);
        void *stream = stream_of(a[14]);
        set_workspace(d, a[13], x, stream, LKV_WS_SSD, d.n_seq, 0);
        Output y, S_T;
        if (a[6] != Py_None) y.given(a[6]);
        else if (PyObject_IsTrue(a[11]) == 1) y.make(new_tensor(x.sizes(), x.scalar_type(), x));
        if (a[7] != Py_None) S_T.given(a[7]);
        else if (PyObject_IsTrue(a[10]) == 1) S_T.make(new_tensor({d.n_seq, d.H, d.N, d.P}, scalar_type_of(a[12]), x));
        if (S_T.obj) d.state_dtype = dtype_code(THPVariable_Unpack(S_T.obj));
        call("lkv_ssd_fwd", d.workspace, lkv_ssd_fwd, ptr_of(a[0]), static_cast<float *>(ptr_of(a[1])),
             static_cast<float *>(ptr_of(a[2])), ptr_of(a[3]), ptr_of(a[4]), static_cast<float *>(ptr_of(a[5])), y.ptr,
             S_T.ptr, &d, stream);
        return pair(y, S_T);
    });
}

// (dt, A, logdecay, cu_seqlens, workspace_t, stream) -> logdecay
PyObject *mamba_chunk_logdecay(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 6);
        const at::Tensor &dt = tensor_of(a[0]);
        need_dim(dt, 2);
        HostInts cu(a[3]);
        lkv_ssd_desc d{};
        d.T_total = static_cast<int32_t>(dt.size(0));
        d.n_seq = cu.data() ? cu.size() - 1 : 1;
        d.cu_seqlens = cu.data();
        d.H = static_cast<int32_t>(dt.size(1));
        d.P = d.N = d.G = 1;
        void *stream = stream_of(a[5]);
        set_workspace(d, a[4], dt, stream, LKV_WS_SSD, d.n_seq, 0);
        Output out;
        if (a[2] != Py_None) out.given(a[2]);
        else out.make(new_tensor({d.n_seq, d.H}, at::kFloat, dt));
        call("lkv_mamba_chunk_logdecay", d.workspace, lkv_mamba_chunk_logdecay, static_cast<float *>(ptr_of(a[0])),
             static_cast<float *>(ptr_of(a[1])), static_cast<float *>(out.ptr), &d, stream);
        return out.take();
    });
}

// setup(LkvError, workspace, workspace cache, host_i32)
PyObject *setup(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        need_args(n, 4);
        PyObject **to[4] = {&g_error, &g_workspace, &g_ws_cache, &g_host_i32};
        for (int i = 0; i < 4; ++i) {
            Py_INCREF(a[i]);
            Py_XSETREF(*to[i], a[i]);
        }
        Py_RETURN_NONE;
    });
}

#define LKV_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {LKV_METHOD(setup), LKV_METHOD(init_state), LKV_METHOD(init_state_batched), LKV_METHOD(gdn_fwd),
                         LKV_METHOD(gdn_chunk_artifacts), LKV_METHOD(ssd_fwd), LKV_METHOD(mamba_chunk_logdecay),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lkv_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__lkv_calls(void) { return PyModule_Create(&module); }
