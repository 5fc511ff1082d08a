// Python <-> C ABI marshalling of the entry points that run once per layer or per step: tensors are unpacked, checked
// and handed to libentropycache here instead of attribute by attribute in the interpreter.
//
// What bounds it: nothing but host instructions.  A partial step of a 32-layer model is 34 calls of 9 to 20 us on the
// GPU; marshalled through ctypes a call took 12 to 15 us of host time, of which the launch itself is 3, so at short
// contexts the GPU waited for the host.  Unpacking a tensor here is a pointer read (about 10 ns against 0.3 us for
// is_cuda, is_contiguous, data_ptr and a c_void_p).  The interpreter lock is released around every library call: a
// launch can block on a full queue.
//
// Each function returns the library's status (the Python wrapper raises) or, for the gates, (status, outputs...).
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <stdexcept>
#include <string>

#include "entropycache.h"

namespace {

struct PyRaised : std::exception {};   // a Python exception is set

[[noreturn]] void raise(PyObject* type, const std::string& what) {
    PyErr_SetString(type, what.c_str());
    throw PyRaised();
}

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string(name) + " must be a torch.Tensor");
    return THPVariable_Unpack(o);
}

// device pointer of a dense CUDA tensor; nullptr for None
void* dev(PyObject* o, const char* name) {
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o, name);
    if (!t.is_cuda()) raise(PyExc_ValueError, std::string(name) + " must be a CUDA tensor (the library has no host path)");
    if (!t.is_contiguous()) raise(PyExc_ValueError, std::string(name) + " must be contiguous");
    return t.data_ptr();
}
template <class T>
T* dev_as(PyObject* o, const char* name) { return static_cast<T*>(dev(o, name)); }

size_t bytes_of(PyObject* o) { return o == Py_None ? 0 : THPVariable_Unpack(o).nbytes(); }

int32_t dtype_code(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return EC_F32;
    if (t.scalar_type() == at::kBFloat16) return EC_BF16;
    raise(PyExc_TypeError, std::string("unsupported element type ") + c10::toString(t.scalar_type()));
}

long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyRaised();
    return v;
}
int32_t int32(PyObject* o) {
    const long long v = integer(o);
    if (v < INT32_MIN || v > INT32_MAX) raise(PyExc_OverflowError, "value does not fit 32 bits");
    return (int32_t)v;
}
float real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyRaised();
    return (float)v;
}

// the stream object's handle, or PyTorch's current stream for None
void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw PyRaised();
    void* s = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!s && PyErr_Occurred()) throw PyRaised();
    return s;
}

// a copy of the ctypes structure's bytes
ec_attn_desc desc_of(PyObject* o) {
    Py_buffer v;
    if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) != 0) throw PyRaised();
    ec_attn_desc d;
    const bool ok = v.len == (Py_ssize_t)sizeof d;
    if (ok) d = *static_cast<const ec_attn_desc*>(v.buf);
    PyBuffer_Release(&v);
    if (!ok) raise(PyExc_TypeError, "desc must be an ec_attn_desc");
    return d;
}

template <class F>
ec_status without_gil(F f) {
    ec_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return st;
}

template <class F>
PyObject* guarded(F f) {
    try {
        return f();
    } catch (const PyRaised&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

void want(Py_ssize_t n, Py_ssize_t expected) {
    if (n != expected) raise(PyExc_TypeError, "wrong number of arguments");
}

// ---- attention -----------------------------------------------------------------------------------------------------
// (desc, k_cache, v_cache, k_new, v_new, active_idx, stream)
PyObject* kv_refresh(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 7);
        const ec_attn_desc d = desc_of(a[0]);
        void *kc = dev(a[1], "k_cache"), *vc = dev(a[2], "v_cache"), *kn = dev(a[3], "k_new"), *vn = dev(a[4], "v_new");
        const int32_t* idx = dev_as<int32_t>(a[5], "active_idx");
        const int32_t n_active = (int32_t)tensor(a[3], "k_new").size(1);
        void* s = stream_of(a[6]);
        return PyLong_FromLong(without_gil([&] { return ec_kv_refresh(&d, kc, vc, kn, vn, idx, n_active, s); }));
    });
}

// (desc, q, k_new, v_new, k_cache, v_cache, active_idx, out, workspace, dev_status, stream)
PyObject* attend(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 11);
        const ec_attn_desc d = desc_of(a[0]);
        void *q = dev(a[1], "q"), *kn = dev(a[2], "k_new"), *vn = dev(a[3], "v_new"), *kc = dev(a[4], "k_cache"),
             *vc = dev(a[5], "v_cache");
        const int32_t* idx = dev_as<int32_t>(a[6], "active_idx");
        void *out = dev(a[7], "out"), *ws = dev(a[8], "workspace");
        const size_t ws_bytes = bytes_of(a[8]);
        int32_t* status = dev_as<int32_t>(a[9], "dev_status");
        const int32_t n_active = (int32_t)tensor(a[1], "q").size(1);
        void* s = stream_of(a[10]);
        return PyLong_FromLong(
            without_gil([&] { return ec_attend(&d, q, kn, vn, kc, vc, idx, n_active, out, ws, ws_bytes, status, s); }));
    });
}

// ---- gate ----------------------------------------------------------------------------------------------------------
// The outputs a gate call returns: the caller's tensors, and slices of ONE allocation for those that were not given
// (seven allocations cost more host time than the kernel takes at a small vocabulary).
class Outputs {
public:
    explicit Outputs(const at::Tensor& like) : like_(like) {}
    // `given` is None: an output of n elements of this type, to be carved from the common allocation
    void add(PyObject* given, const char* name, int64_t n, at::ScalarType type) {
        Item& it = items_[count_++];
        it = Item{given, name, n, type, total_};
        if (given != Py_None) return;
        total_ += (n * (int64_t)c10::elementSize(type) + 15) & ~15ll;
        any_ = true;
    }
    void skip() { items_[count_++] = Item{nullptr, "", 0, at::kFloat, 0}; }   // not wanted: NULL, None
    void allocate() {
        if (any_) blob_ = at::empty({total_}, like_.options().dtype(at::kByte));
        for (int i = 0; i < count_; ++i) {
            Item& it = items_[i];
            if (!it.given) continue;
            if (it.given != Py_None) {
                it.ptr = dev(it.given, it.name);
                continue;
            }
            auto impl = c10::make_intrusive<c10::TensorImpl>(c10::Storage(blob_.storage()), blob_.key_set(),
                                                             c10::scalarTypeToTypeMeta(it.type));
            impl->set_storage_offset(it.off / (int64_t)c10::elementSize(it.type));
            impl->set_sizes_contiguous({it.n});
            it.made = at::Tensor(std::move(impl));
            it.ptr = static_cast<char*>(blob_.data_ptr()) + it.off;
        }
    }
    template <class T>
    T* ptr(int i) const { return static_cast<T*>(items_[i].ptr); }
    // (status, output 0, output 1, ...)
    PyObject* result(ec_status st) {
        PyObject* t = PyTuple_New(count_ + 1);
        if (!t) throw PyRaised();
        PyTuple_SET_ITEM(t, 0, PyLong_FromLong(st));
        for (int i = 0; i < count_; ++i) {
            Item& it = items_[i];
            PyObject* o = it.made.defined() ? THPVariable_Wrap(std::move(it.made))
                                            : Py_NewRef(it.given ? it.given : Py_None);
            PyTuple_SET_ITEM(t, i + 1, o);
        }
        return t;
    }

private:
    struct Item {
        PyObject* given = nullptr;
        const char* name = "";
        int64_t n = 0;
        at::ScalarType type = at::kFloat;
        int64_t off = 0;
        void* ptr = nullptr;
        at::Tensor made = {};
    };
    const at::Tensor& like_;
    at::Tensor blob_;
    Item items_[8];
    int count_ = 0;
    int64_t total_ = 0;
    bool any_ = false;   // some output is to be made; total_ may still be 0 (a call without rows)
};

struct Logits {
    const at::Tensor& t;
    int32_t dtype, rows, rows_per_seq, n_seq, vocab;
    int64_t stride;
    void* ptr;
};
// dense: the entry point takes contiguous logits only; otherwise rows of any stride
Logits logits_of(PyObject* o, PyObject* vocab, PyObject* rows_per_seq, bool dense) {
    const at::Tensor& t = tensor(o, "logits");
    if (t.dim() != 2) raise(PyExc_ValueError, "logits must be a 2-D CUDA tensor [n_rows, row_stride]");
    void* p = nullptr;
    int64_t stride = t.size(1);
    if (dense) {
        p = dev(o, "logits");
    } else {
        if (!t.is_cuda()) raise(PyExc_ValueError, "logits must be a 2-D CUDA tensor [n_rows, row_stride]");
        if (t.stride(1) != 1) raise(PyExc_ValueError, "logits rows must be contiguous");
        p = t.data_ptr();
        stride = t.stride(0);
    }
    const int32_t rps = int32(rows_per_seq), rows = (int32_t)t.size(0);
    return Logits{t, dtype_code(t), rows, rps, rps > 0 ? rows / rps : 0, int32(vocab), stride, p};
}

// (logits, vocab, rows_per_seq, decoded_flags, tau, argmax, conf, entropy, max_entropy, decision, workspace, want_rows,
//  stream) -> (status, argmax, conf, entropy, max_entropy, decision)
PyObject* gate(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 13);
        const Logits lg = logits_of(a[0], a[1], a[2], false);
        const uint8_t* flags = dev_as<uint8_t>(a[3], "decoded_flags");
        const float tau = real(a[4]);
        Outputs o(lg.t);
        const bool rows = PyObject_IsTrue(a[11]) == 1;
        const auto row_out = [&](PyObject* g, const char* name, at::ScalarType t) {
            if (rows || g != Py_None) o.add(g, name, lg.rows, t); else o.skip();
        };
        row_out(a[5], "argmax_out", at::kInt);
        row_out(a[6], "conf_out", at::kFloat);
        row_out(a[7], "entropy_out", at::kFloat);
        o.add(a[8], "max_entropy_out", lg.n_seq, at::kFloat);
        o.add(a[9], "decision_out", lg.n_seq, at::kInt);
        void* ws = dev(a[10], "workspace");
        const size_t ws_bytes = bytes_of(a[10]);
        o.allocate();
        void* s = stream_of(a[12]);
        return o.result(without_gil([&] {
            return ec_entropy_gate(lg.ptr, lg.dtype, lg.rows, lg.vocab, lg.stride, lg.rows_per_seq, flags, tau,
                                   o.ptr<int32_t>(0), o.ptr<float>(1), o.ptr<float>(2), o.ptr<float>(3),
                                   o.ptr<int32_t>(4), ws, ws_bytes, s);
        }));
    });
}

// (logits, vocab, rows_per_seq, masked, conf_threshold, tau, tokens, decoded, argmax, conf, entropy, max_entropy,
//  decision, workspace, want_rows, stream) -> (status, decoded, argmax, conf, entropy, max_entropy, decision)
PyObject* gate_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 16);
        const Logits lg = logits_of(a[0], a[1], a[2], true);
        const at::Tensor &m = tensor(a[3], "masked"), &tk = tensor(a[6], "tokens");
        if (m.scalar_type() != at::kByte || tk.scalar_type() != at::kInt || m.numel() != lg.rows || tk.numel() != lg.rows)
            raise(PyExc_ValueError, "masked must be uint8 [n_rows], tokens int32 [n_rows]");
        uint8_t* masked = dev_as<uint8_t>(a[3], "masked");
        int32_t* tokens = dev_as<int32_t>(a[6], "tokens");
        const float thr = real(a[4]), tau = real(a[5]);
        Outputs o(lg.t);
        const bool rows = PyObject_IsTrue(a[14]) == 1;
        const auto row_out = [&](PyObject* g, const char* name, at::ScalarType t) {
            if (rows || g != Py_None) o.add(g, name, lg.rows, t); else o.skip();
        };
        o.add(a[7], "decoded_out", lg.rows, at::kByte);
        row_out(a[8], "argmax_out", at::kInt);
        row_out(a[9], "conf_out", at::kFloat);
        row_out(a[10], "entropy_out", at::kFloat);
        o.add(a[11], "max_entropy_out", lg.n_seq, at::kFloat);
        o.add(a[12], "decision_out", lg.n_seq, at::kInt);
        void* ws = dev(a[13], "workspace");
        const size_t ws_bytes = bytes_of(a[13]);
        o.allocate();
        void* s = stream_of(a[15]);
        return o.result(without_gil([&] {
            return ec_entropy_gate_decode(lg.ptr, lg.dtype, lg.rows, lg.vocab, lg.stride, lg.rows_per_seq, masked, thr, tau,
                                          o.ptr<uint8_t>(0), tokens, o.ptr<int32_t>(1), o.ptr<float>(2), o.ptr<float>(3),
                                          o.ptr<float>(4), o.ptr<int32_t>(5), ws, ws_bytes, s);
        }));
    });
}

// (logits, vocab, rows_per_seq, decoded_flags, tau, workspace, stream)
//   -> (status, argmax, conf, entropy, max_entropy, decision, entropy_sum, max_conf)
PyObject* gate_metrics(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 7);
        const Logits lg = logits_of(a[0], a[1], a[2], true);
        const uint8_t* flags = dev_as<uint8_t>(a[3], "decoded_flags");
        const float tau = real(a[4]);
        Outputs o(lg.t);
        o.add(Py_None, "argmax", lg.rows, at::kInt);
        o.add(Py_None, "conf", lg.rows, at::kFloat);
        o.add(Py_None, "entropy", lg.rows, at::kFloat);
        o.add(Py_None, "max_entropy", lg.n_seq, at::kFloat);
        o.add(Py_None, "decision", lg.n_seq, at::kInt);
        o.add(Py_None, "entropy_sum", lg.n_seq, at::kFloat);
        o.add(Py_None, "max_conf", lg.n_seq, at::kFloat);
        void* ws = dev(a[5], "workspace");
        const size_t ws_bytes = bytes_of(a[5]);
        o.allocate();
        void* s = stream_of(a[6]);
        return o.result(without_gil([&] {
            return ec_entropy_gate_metrics(lg.ptr, lg.dtype, lg.rows, lg.vocab, lg.stride, lg.rows_per_seq, flags, tau,
                                           o.ptr<int32_t>(0), o.ptr<float>(1), o.ptr<float>(2), o.ptr<float>(3),
                                           o.ptr<int32_t>(4), o.ptr<float>(5), o.ptr<float>(6), ws, ws_bytes, s);
        }));
    });
}

// ---- selection -----------------------------------------------------------------------------------------------------
void check(bool ok, PyObject* type, const char* what) {
    if (!ok) raise(type, what);
}
bool is(PyObject* o, const char* name, at::ScalarType t) { return tensor(o, name).scalar_type() == t; }

// (history, state, decoded_flags, window_start, block, decision, k, active_idx, stream)
PyObject* select_recent(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 9);
        const at::Tensor &h = tensor(a[0], "history"), &st = tensor(a[1], "state"), &idx = tensor(a[7], "active_idx");
        check(h.dim() == 2 && st.dim() == 2 && idx.dim() == 2, PyExc_ValueError,
              "history must be [B, L], state [B, 4], active_idx [B, n_cap]");
        check(h.scalar_type() == at::kInt && st.scalar_type() == at::kInt && idx.scalar_type() == at::kInt, PyExc_TypeError,
              "history, state and active_idx must be int32");
        check(is(a[2], "decoded_flags", at::kByte) && is(a[3], "window_start", at::kInt) && is(a[5], "decision", at::kInt),
              PyExc_TypeError, "decoded_flags must be uint8, window_start and decision int32");
        const int64_t batch = h.size(0);
        const int32_t block = int32(a[4]), k = int32(a[6]);
        check(st.size(0) == batch && st.size(1) == 4 && idx.size(0) == batch && tensor(a[2], "").numel() == batch * block,
              PyExc_ValueError, "state must be [B, 4], active_idx [B, n_cap], decoded_flags [B * block]");
        check(tensor(a[3], "").numel() == batch && tensor(a[5], "").numel() == batch, PyExc_ValueError,
              "window_start and decision must hold one entry per sequence");
        int32_t* hp = dev_as<int32_t>(a[0], "history");
        auto* sp = dev_as<ec_step_state>(a[1], "state");
        const uint8_t* fp = dev_as<uint8_t>(a[2], "decoded_flags");
        const int32_t *wp = dev_as<int32_t>(a[3], "window_start"), *dp = dev_as<int32_t>(a[5], "decision");
        int32_t* ip = dev_as<int32_t>(a[7], "active_idx");
        const int32_t L = (int32_t)h.size(1), cap = (int32_t)idx.size(1);
        void* s = stream_of(a[8]);
        return PyLong_FromLong(
            without_gil([&] { return ec_select_recent(hp, L, (int32_t)batch, sp, fp, wp, block, dp, k, ip, cap, s); }));
    });
}

// (history, state, masked, decoded_flags, window, decision, k, active_idx, stream)
PyObject* select_recent_sliding(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&] {
        want(n, 9);
        const at::Tensor &h = tensor(a[0], "history"), &st = tensor(a[1], "state"), &m = tensor(a[2], "masked"),
                         &idx = tensor(a[7], "active_idx");
        check(h.dim() == 2 && st.dim() == 2 && m.dim() == 2 && idx.dim() == 2, PyExc_ValueError,
              "masked must be [B, L], state [B, 4], active_idx [B, n_cap]");
        check(h.scalar_type() == at::kInt && st.scalar_type() == at::kInt && idx.scalar_type() == at::kInt, PyExc_TypeError,
              "history, state and active_idx must be int32");
        check(m.scalar_type() == at::kByte && is(a[3], "decoded_flags", at::kByte) && is(a[5], "decision", at::kInt),
              PyExc_TypeError, "masked and decoded_flags must be uint8, decision int32");
        const int64_t batch = h.size(0), ctx = h.size(1);
        const int32_t window = int32(a[4]), k = int32(a[6]);
        check(m.size(0) == batch && m.size(1) == ctx && st.size(0) == batch && st.size(1) == 4 && idx.size(0) == batch,
              PyExc_ValueError, "masked must be [B, L], state [B, 4], active_idx [B, n_cap]");
        check(tensor(a[3], "").numel() == batch * window && tensor(a[5], "").numel() == batch, PyExc_ValueError,
              "decoded_flags must be [B * window], decision [B]");
        int32_t* hp = dev_as<int32_t>(a[0], "history");
        auto* sp = dev_as<ec_step_state>(a[1], "state");
        uint8_t* mp = dev_as<uint8_t>(a[2], "masked");
        const uint8_t* fp = dev_as<uint8_t>(a[3], "decoded_flags");
        const int32_t* dp = dev_as<int32_t>(a[5], "decision");
        int32_t* ip = dev_as<int32_t>(a[7], "active_idx");
        const int32_t cap = (int32_t)idx.size(1);
        void* s = stream_of(a[8]);
        return PyLong_FromLong(without_gil([&] {
            return ec_select_recent_sliding(hp, (int32_t)ctx, (int32_t)batch, sp, mp, fp, window, dp, k, ip, cap, s);
        }));
    });
}

#define EC_FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {EC_FAST(kv_refresh),   EC_FAST(attend),        EC_FAST(gate),
                         EC_FAST(gate_decode),  EC_FAST(gate_metrics),  EC_FAST(select_recent),
                         EC_FAST(select_recent_sliding), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_ec_python", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ec_python() { return PyModule_Create(&module_def); }
