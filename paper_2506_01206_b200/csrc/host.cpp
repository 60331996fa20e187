// Argument marshalling between torch and the C ABI (include/mdraft.h), as a CPython extension.
//
// A launch of this library takes the GPU a few microseconds, and turning its 30 arguments into C values in the interpreter
// took 12-15 us of host time per call, which is what bounded single-layer calls.  Here a call's tensors are read through torch's
// C++ interface and handed straight to the library; nothing is cached between calls, so a layer or a cache whose tensors are
// replaced is seen as it is.  The functions take the entry points as a table of addresses: the table belongs to the loaded
// library the caller chose, which need not be the default one.  The interpreter lock is released around the library calls.
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include <c10/cuda/CUDAStream.h>

#include <string>
#include <vector>

#include "../../include/mdraft.h"

namespace {

// The order in which binding.py lists the addresses.
struct Entry {
    decltype(&mdraft_conv_scan_prefill) prefill;
    decltype(&mdraft_conv_scan_prefill_noalloc) prefill_noalloc;
    decltype(&mdraft_tree_step) tree_step;
    decltype(&mdraft_tree_step_proj) tree_step_proj;
    decltype(&mdraft_state_commit) commit;
    decltype(&mdraft_ssd_prefill) ssd_prefill;
    decltype(&mdraft_ssd_tree_step) ssd_tree_step;
    decltype(&mdraft_conv_scan_prefill_stack) prefill_stack;
    decltype(&mdraft_tree_step_stack) tree_step_stack;
    decltype(&mdraft_block_generation) block_generation;
};

struct Failed {};  // a Python exception is set

[[noreturn]] void fail(PyObject* type, const std::string& text) {
    PyErr_SetString(type, text.c_str());
    throw Failed();
}

// Attribute names, interned once.
struct Names {
    PyObject *A, *D, *conv_w, *conv_b, *dt_bias, *act, *flags, *d_inner, *d_state, *d_conv, *headdim, *ssm, *conv, *n_layers, *n_slots, *cuda_stream, *cuda_event;
};
Names N;

// An owned reference that goes away with the scope.
struct Ref {
    PyObject* p;
    explicit Ref(PyObject* o) : p(o) { if (!p) throw Failed(); }
    Ref(const Ref&) = delete;
    ~Ref() { Py_DECREF(p); }
};

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, std::string(name) + ": must be a tensor");
    return THPVariable_Unpack(o);
}
const void* data(PyObject* o, const char* name) { return o == Py_None ? nullptr : tensor(o, name).const_data_ptr(); }
void* mutable_data(PyObject* o, const char* name) { return const_cast<void*>(data(o, name)); }

// Address of a tensor attribute; the owner keeps the tensor alive for the length of the call.
const void* attr_data(PyObject* owner, PyObject* name) {
    Ref r(PyObject_GetAttr(owner, name));
    return data(r.p, PyUnicode_AsUTF8(name));
}
int64_t as_int(PyObject* o) {
    if (PyLong_Check(o)) {
        const int64_t v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) throw Failed();
        return v;
    }
    Ref i(PyNumber_Long(o));
    const int64_t v = PyLong_AsLongLong(i.p);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return v;
}
int64_t attr_int(PyObject* owner, PyObject* name) {
    Ref r(PyObject_GetAttr(owner, name));
    return as_int(r.p);
}
int act_of(PyObject* owner) {
    Ref r(PyObject_GetAttr(owner, N.act));
    if (THPDtype_Check(r.p)) {
        const at::ScalarType t = reinterpret_cast<THPDtype*>(r.p)->scalar_type;
        if (t == at::kFloat) return MDRAFT_F32;
        if (t == at::kBFloat16) return MDRAFT_BF16;
    }
    fail(PyExc_TypeError, "activation dtype must be float32 or bfloat16");
}

// (pointer, row stride in elements) of a 2-D tensor whose last dim is contiguous; None = absent.
struct Matrix {
    const void* p = nullptr;
    int64_t ld = 0, rows = 0;
    Matrix(PyObject* o, const char* name) {
        if (o == Py_None) return;
        const at::Tensor& t = tensor(o, name);
        if (t.dim() != 2 || (t.size(1) > 1 && t.stride(1) != 1))
            fail(PyExc_ValueError, std::string(name) + ": need a 2-D tensor with unit stride along the last dim");
        if (!t.is_cuda()) fail(PyExc_ValueError, std::string(name) + ": must be a CUDA tensor");
        p = t.const_data_ptr();
        ld = t.stride(0);
        rows = t.size(0);
    }
    void* out() const { return const_cast<void*>(p); }
};

// int32 indices with one entry per sequence or node; None = absent.
const int32_t* indices(PyObject* o, int64_t n, const char* type_text, const char* size_text, PyObject* size_error) {
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o, "slot indices");
    if (t.scalar_type() != at::kInt) fail(PyExc_TypeError, type_text);
    if (n >= 0 && t.numel() != n) fail(size_error, size_text);
    return static_cast<const int32_t*>(t.const_data_ptr());
}

void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyObject* s = PyObject_GetAttr(o, N.cuda_stream)) {
        Ref r(s);
        return reinterpret_cast<void*>(as_int(s));
    }
    PyErr_Clear();
    return reinterpret_cast<void*>(as_int(o));
}

mdraft_layer layer_of(PyObject* o, PyObject* flags) {
    mdraft_layer l;
    l.d_inner = (int32_t)attr_int(o, N.d_inner); l.d_state = (int32_t)attr_int(o, N.d_state); l.d_conv = (int32_t)attr_int(o, N.d_conv);
    l.act = act_of(o);
    l.flags = (uint32_t)(flags == Py_None ? attr_int(o, N.flags) : as_int(flags));
    l.reserved = 0;
    l.A = static_cast<const float*>(attr_data(o, N.A)); l.D = static_cast<const float*>(attr_data(o, N.D));
    l.conv_w = static_cast<const float*>(attr_data(o, N.conv_w)); l.conv_b = static_cast<const float*>(attr_data(o, N.conv_b));
    l.dt_bias = static_cast<const float*>(attr_data(o, N.dt_bias));
    return l;
}

mdraft_ssd_layer ssd_layer_of(PyObject* o, PyObject* flags) {
    mdraft_ssd_layer l;
    l.d_inner = (int32_t)attr_int(o, N.d_inner); l.headdim = (int32_t)attr_int(o, N.headdim);
    l.d_state = (int32_t)attr_int(o, N.d_state); l.d_conv = (int32_t)attr_int(o, N.d_conv);
    l.act = MDRAFT_BF16;
    l.flags = (uint32_t)(flags == Py_None ? attr_int(o, N.flags) : as_int(flags));
    l.A = static_cast<const float*>(attr_data(o, N.A)); l.D = static_cast<const float*>(attr_data(o, N.D));
    l.conv_w = static_cast<const float*>(attr_data(o, N.conv_w)); l.conv_b = static_cast<const float*>(attr_data(o, N.conv_b));
    l.dt_bias = static_cast<const float*>(attr_data(o, N.dt_bias));
    return l;
}

// A state pool; `present` is false for None.
struct Cache {
    mdraft_cache c;
    bool present;
    explicit Cache(PyObject* o) : present(o != Py_None) {
        if (!present) return;
        Ref s(PyObject_GetAttr(o, N.ssm)), v(PyObject_GetAttr(o, N.conv));
        const at::Tensor &ssm = tensor(s.p, "ssm"), &conv = tensor(v.p, "conv");
        c.ssm = static_cast<float*>(ssm.data_ptr());
        c.ssm_layer_stride = ssm.stride(0); c.ssm_slot_stride = ssm.stride(1);
        c.conv = conv.data_ptr();
        c.conv_layer_stride = conv.stride(0); c.conv_slot_stride = conv.stride(1);
        c.n_layers = (int32_t)attr_int(o, N.n_layers); c.n_slots = (int32_t)attr_int(o, N.n_slots);
    }
    const mdraft_cache* get() const { return present ? &c : nullptr; }
};

// chunk_len: tokens per chunk (0 or None: the library's plan), or a pair (tokens, channels per block); events: None or two events
// to record.
struct Opts {
    mdraft_prefill_opts o = {};
    bool present = false;
    Opts(PyObject* chunk, PyObject* events) {
        if (PyTuple_Check(chunk) || PyList_Check(chunk)) {
            Ref f(PySequence_Fast(chunk, "chunk_len"));
            if (PySequence_Fast_GET_SIZE(f.p) != 2) fail(PyExc_ValueError, "chunk_len: an int or a pair (chunk_len, block_channels)");
            o.chunk_len = (int32_t)as_int(PySequence_Fast_GET_ITEM(f.p, 0));
            o.block_channels = (int32_t)as_int(PySequence_Fast_GET_ITEM(f.p, 1));
        } else if (chunk != Py_None) {
            o.chunk_len = (int32_t)as_int(chunk);
        }
        present = o.chunk_len || o.block_channels || events != Py_None;
        if (events != Py_None) {
            Ref a(PySequence_GetItem(events, 0)), b(PySequence_GetItem(events, 1));
            Ref ha(PyObject_GetAttr(a.p, N.cuda_event)), hb(PyObject_GetAttr(b.p, N.cuda_event));
            o.event_after_chunk_state = reinterpret_cast<void*>(as_int(ha.p));
            o.event_after_carry_scan = reinterpret_cast<void*>(as_int(hb.p));
        }
    }
    const mdraft_prefill_opts* get() const { return present ? &o : nullptr; }
};

// The offsets of a packed batch and the slots of its sequences.
struct Sequences {
    int64_t n_seq = 1;
    const int32_t *cu = nullptr, *init = nullptr, *fin = nullptr;
    Sequences(PyObject* offsets, PyObject* init_slot, PyObject* final_slot) {
        if (offsets != Py_None) {
            const at::Tensor& t = tensor(offsets, "cu_seqlens");
            if (t.scalar_type() != at::kInt) fail(PyExc_TypeError, "cu_seqlens must be int32");
            n_seq = t.numel() - 1;
            cu = static_cast<const int32_t*>(t.const_data_ptr());
        }
        init = indices(init_slot, n_seq, "init_slot must be int32 with one entry per sequence", "init_slot must be int32 with one entry per sequence", PyExc_TypeError);
        fin = indices(final_slot, n_seq, "final_slot must be int32 with one entry per sequence", "final_slot must be int32 with one entry per sequence", PyExc_TypeError);
    }
};

// Level boundaries of a tree call (None: one level).
struct Levels {
    std::vector<int32_t> v;
    explicit Levels(PyObject* o) {
        if (o == Py_None) return;
        Ref f(PySequence_Fast(o, "level_offsets must be a sequence"));
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(f.p);
        v.resize((size_t)n);
        for (Py_ssize_t i = 0; i < n; ++i) v[(size_t)i] = (int32_t)as_int(PySequence_Fast_GET_ITEM(f.p, i));
        if (n == 0) fail(PyExc_ValueError, "level_offsets must not be empty");
    }
    int32_t count() const { return v.empty() ? 1 : (int32_t)v.size() - 1; }
    const int32_t* get() const { return v.empty() ? nullptr : v.data(); }
};

struct Workspace {
    void* p = nullptr;
    size_t bytes = 0;
    explicit Workspace(PyObject* o) {
        if (o == Py_None) return;
        const at::Tensor& t = tensor(o, "workspace");
        p = t.data_ptr();
        bytes = (size_t)t.numel() * t.element_size();
    }
};

const Entry& entry(PyObject* o) {
    void* p = PyCapsule_GetPointer(o, "mdraft.entry");
    if (!p) throw Failed();
    return *static_cast<const Entry*>(p);
}

// Runs `call` without the interpreter lock and returns its status as a Python int.
template <typename F>
PyObject* released(F&& call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// Every function below takes exactly kArgs arguments, which it reads without asking for their number again; C++ exceptions
// become Python exceptions.
template <PyObject* (*body)(PyObject* const*), int kArgs>
PyObject* guarded(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != kArgs) return PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", kArgs, n);
    try {
        return body(a);
    } catch (const Failed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// (addresses) -> table for the calls below
PyObject* table(PyObject* const* a) {
    Ref f(PySequence_Fast(a[0], "addresses"));
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(f.p);
    if (n * sizeof(void*) != sizeof(Entry)) fail(PyExc_ValueError, "wrong number of entry points");
    void** t = static_cast<void**>(PyMem_Malloc(sizeof(Entry)));
    if (!t) { PyErr_NoMemory(); throw Failed(); }
    for (Py_ssize_t i = 0; i < n; ++i) t[i] = reinterpret_cast<void*>(as_int(PySequence_Fast_GET_ITEM(f.p, i)));
    return PyCapsule_New(t, "mdraft.entry", [](PyObject* c) { PyMem_Free(PyCapsule_GetPointer(c, "mdraft.entry")); });
}

// (table, layer, cache, layer_index, x, z, dt, B, C, out, cu_seqlens, max_seqlen, init_slot, final_slot, workspace, chunk_len,
//  dev_status, stream, flags, phase_events)
PyObject* prefill(PyObject* const* a) {
    const mdraft_layer l = layer_of(a[1], a[18]);
    const Cache c(a[2]);
    const int32_t li = (int32_t)as_int(a[3]), longest = (int32_t)as_int(a[11]);
    const Matrix x(a[4], "x"), z(a[5], "z"), dt(a[6], "dt"), B(a[7], "B"), C(a[8], "C"), o(a[9], "out");
    const Sequences s(a[10], a[12], a[13]);
    const Workspace ws(a[14]);
    const Opts opts(a[15], a[19]);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[16], "dev_status"));
    void* stream = stream_of(a[17]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.prefill(&l, c.get(), li, x.p, x.ld, z.p, z.ld, dt.p, dt.ld, B.p, B.ld, C.p, C.ld, o.out(), o.ld, (int32_t)x.rows,
                         (int32_t)s.n_seq, longest, s.cu, s.init, s.fin, ws.p, ws.bytes, opts.get(), st, stream);
    });
}

// As prefill without the workspace and the events.
PyObject* prefill_noalloc(PyObject* const* a) {
    const mdraft_layer l = layer_of(a[1], a[17]);
    const Cache c(a[2]);
    const int32_t li = (int32_t)as_int(a[3]), longest = (int32_t)as_int(a[11]);
    const Matrix x(a[4], "x"), z(a[5], "z"), dt(a[6], "dt"), B(a[7], "B"), C(a[8], "C"), o(a[9], "out");
    const Sequences s(a[10], a[12], a[13]);
    const Opts opts(a[14], Py_None);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[15], "dev_status"));
    void* stream = stream_of(a[16]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.prefill_noalloc(&l, c.get(), li, x.p, x.ld, z.p, z.ld, dt.p, dt.ld, B.p, B.ld, C.p, C.ld, o.out(), o.ld, (int32_t)x.rows,
                                 (int32_t)s.n_seq, longest, s.cu, s.init, s.fin, opts.get(), st, stream);
    });
}

struct Nodes {
    const int32_t *parent, *node;
    Nodes(PyObject* p, PyObject* n, int64_t m) {
        const char *type = "slot index arrays must be int32", *size = "one parent slot and one node slot per node";
        parent = indices(p, m, type, size, PyExc_ValueError);
        node = indices(n, m, type, size, PyExc_ValueError);
    }
};

// (table, layer, cache, layer_index, x, z, dt, B, C, out, parent_slot, node_slot, level_offsets, dev_status, stream, flags)
PyObject* tree_step(PyObject* const* a) {
    const mdraft_layer l = layer_of(a[1], a[15]);
    const Cache c(a[2]);
    const int32_t li = (int32_t)as_int(a[3]);
    const Matrix x(a[4], "x"), z(a[5], "z"), dt(a[6], "dt"), B(a[7], "B"), C(a[8], "C"), o(a[9], "out");
    const Nodes n(a[10], a[11], x.rows);
    const Levels lv(a[12]);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[13], "dev_status"));
    void* stream = stream_of(a[14]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.tree_step(&l, c.get(), li, x.p, x.ld, z.p, z.ld, dt.p, dt.ld, B.p, B.ld, C.p, C.ld, o.out(), o.ld, (int32_t)x.rows,
                           n.parent, n.node, lv.count(), lv.get(), st, stream);
    });
}

// (table, layer, cache, layer_index, W_x, W_dt, x, z, out, parent_slot, node_slot, dev_status, stream, flags, nodes_per_cluster)
PyObject* tree_step_proj(PyObject* const* a) {
    const mdraft_layer l = layer_of(a[1], a[13]);
    const Cache c(a[2]);
    const int32_t li = (int32_t)as_int(a[3]);
    const Matrix x(a[6], "x"), z(a[7], "z"), o(a[8], "out");
    const Nodes n(a[9], a[10], x.rows);
    const at::Tensor &wx = tensor(a[4], "W_x"), &wdt = tensor(a[5], "W_dt");
    const at::ScalarType act = tensor(a[6], "x").scalar_type();
    if (wx.scalar_type() != act || wdt.scalar_type() != act || !wx.is_contiguous() || !wdt.is_contiguous())
        fail(PyExc_TypeError, "W_x and W_dt must be contiguous and of the activation dtype");
    const int64_t R = wdt.dim() == 2 ? wdt.size(1) : -1;
    if (wdt.dim() != 2 || wx.dim() != 2 || wdt.size(0) != l.d_inner || wx.size(0) != R + 2 * l.d_state || wx.size(1) != l.d_inner)
        fail(PyExc_ValueError, "W_x must be (dt_rank + 2 d_state, d_inner) and W_dt (d_inner, dt_rank)");
    const mdraft_select_proj pr = {wx.const_data_ptr(), wdt.const_data_ptr(), (int32_t)R, (int32_t)as_int(a[14])};
    int32_t* st = static_cast<int32_t*>(mutable_data(a[11], "dev_status"));
    void* stream = stream_of(a[12]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.tree_step_proj(&l, c.get(), li, &pr, x.p, x.ld, z.p, z.ld, o.out(), o.ld, (int32_t)x.rows, n.parent, n.node, st, stream);
    });
}

// (table, cache, src_slot, dst_slot, dev_status, stream)
PyObject* commit(PyObject* const* a) {
    const Cache c(a[1]);
    if (!c.present) fail(PyExc_TypeError, "cache must not be None");
    const int32_t d = (int32_t)attr_int(a[1], N.d_inner), n = (int32_t)attr_int(a[1], N.d_state), w = (int32_t)attr_int(a[1], N.d_conv);
    const int act = act_of(a[1]);
    const char* text = "src_slot / dst_slot must be int32 arrays of equal length";
    const int64_t m = tensor(a[2], "src_slot").numel();
    const int32_t *src = indices(a[2], m, text, text, PyExc_TypeError), *dst = indices(a[3], m, text, text, PyExc_TypeError);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[4], "dev_status"));
    void* stream = stream_of(a[5]);
    const Entry& e = entry(a[0]);
    return released([&] { return e.commit(c.get(), d, n, w, act, (int32_t)m, src, dst, st, stream); });
}

// (table, layer, cache, layer_index, x, z, dt, B, C, out, cu_seqlens, init_slot, final_slot, workspace, dev_status, stream, flags)
PyObject* ssd_prefill(PyObject* const* a) {
    const mdraft_ssd_layer l = ssd_layer_of(a[1], a[16]);
    const Cache c(a[2]);
    const int32_t li = (int32_t)as_int(a[3]);
    const Matrix x(a[4], "x"), z(a[5], "z"), dt(a[6], "dt"), B(a[7], "B"), C(a[8], "C"), o(a[9], "out");
    const Sequences s(a[10], a[11], a[12]);
    const Workspace ws(a[13]);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[14], "dev_status"));
    void* stream = stream_of(a[15]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.ssd_prefill(&l, c.get(), li, x.p, x.ld, z.p, z.ld, dt.p, dt.ld, B.p, B.ld, C.p, C.ld, o.out(), o.ld, (int32_t)x.rows,
                             (int32_t)s.n_seq, s.cu, s.init, s.fin, ws.p, ws.bytes, st, stream);
    });
}

// (table, layer, cache, layer_index, x, z, dt, B, C, out, parent_slot, node_slot, level_offsets, dev_status, stream, flags)
PyObject* ssd_tree_step(PyObject* const* a) {
    const mdraft_ssd_layer l = ssd_layer_of(a[1], a[15]);
    const Cache c(a[2]);
    const int32_t li = (int32_t)as_int(a[3]);
    const Matrix x(a[4], "x"), z(a[5], "z"), dt(a[6], "dt"), B(a[7], "B"), C(a[8], "C"), o(a[9], "out");
    const Nodes n(a[10], a[11], x.rows);
    const Levels lv(a[12]);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[13], "dev_status"));
    void* stream = stream_of(a[14]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.ssd_tree_step(&l, c.get(), li, x.p, x.ld, z.p, z.ld, dt.p, dt.ld, B.p, B.ld, C.p, C.ld, o.out(), o.ld, (int32_t)x.rows,
                               n.parent, n.node, lv.count(), lv.get(), st, stream);
    });
}

// The layers of a stack call, gathered; `apart` says whether they may run side by side.
struct Stack {
    std::vector<mdraft_layer> layers;
    std::vector<int32_t> index;
    std::vector<mdraft_io> io;
    int64_t rows = 0;
    bool apart = true;

    struct Span { uintptr_t lo, hi; };
    static Span span(const Matrix& m, int64_t cols, int64_t es) {
        const uintptr_t p = reinterpret_cast<uintptr_t>(m.p);
        return m.p && m.rows > 0 ? Span{p, p + (uintptr_t)(((m.rows - 1) * m.ld + cols) * es)} : Span{0, 0};
    }
    static bool meet(const Span& a, const Span& b) { return a.lo < b.hi && b.lo < a.hi; }

    Stack(PyObject* layer_list, PyObject* which, PyObject* inputs, PyObject* outs) {
        Ref w(PySequence_Fast(which, "layers to run"));
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(w.p);
        std::vector<Span> in, out;
        for (Py_ssize_t k = 0; k < n; ++k) {
            const int64_t l = as_int(PySequence_Fast_GET_ITEM(w.p, k));
            Ref lay(PySequence_GetItem(layer_list, l)), ins(PySequence_GetItem(inputs, l)), o(PySequence_GetItem(outs, l));
            Ref f(PySequence_Fast(ins.p, "a layer's inputs are (x, z, dt, B, C)"));
            if (PySequence_Fast_GET_SIZE(f.p) != 5) fail(PyExc_ValueError, "a layer's inputs are (x, z, dt, B, C)");
            layers.push_back(layer_of(lay.p, Py_None));
            index.push_back((int32_t)(l < 0 ? -1 : l));
            const Matrix x(PySequence_Fast_GET_ITEM(f.p, 0), "x"), z(PySequence_Fast_GET_ITEM(f.p, 1), "z"), dt(PySequence_Fast_GET_ITEM(f.p, 2), "dt"),
                B(PySequence_Fast_GET_ITEM(f.p, 3), "B"), C(PySequence_Fast_GET_ITEM(f.p, 4), "C"), y(o.p, "out");
            io.push_back({x.p, z.p, dt.p, B.p, C.p, y.out(), x.ld, z.ld, dt.ld, B.ld, C.ld, y.ld});
            const mdraft_layer& L = layers.back();
            const int64_t es = L.act == MDRAFT_BF16 ? 2 : 4;
            for (const Matrix* m : {&x, &z, &dt}) in.push_back(span(*m, L.d_inner, es));
            in.push_back(span(B, L.d_state, es));
            in.push_back(span(C, L.d_state, es));
            out.push_back(span(y, L.d_inner, es));
            if (k == 0) rows = x.rows;
            apart = apart && x.rows == rows && l >= 0 && L.d_inner == layers[0].d_inner && L.act == layers[0].act;
        }
        // A layer that reads what another writes, or two that write the same rows or states, have to run one after another.
        for (Py_ssize_t a = 0; a < n && apart; ++a)
            for (Py_ssize_t b = 0; b < n && apart; ++b) {
                if (a == b) continue;
                apart = index[a] != index[b] && !meet(out[a], out[b]);
                for (int i = 0; i < 5 && apart; ++i) apart = !meet(out[a], in[5 * b + i]);
            }
    }
};

// (table, layers, which, cache, inputs, outs, cu_seqlens, max_seqlen, init_slot, final_slot, workspace, dev_status, stream)
// -> status, or None when the layers have to run one after another
PyObject* prefill_stack(PyObject* const* a) {
    const Stack k(a[1], a[2], a[4], a[5]);
    if (!k.apart || k.layers.size() < 2) Py_RETURN_NONE;
    const Cache c(a[3]);
    const Sequences s(a[6], a[8], a[9]);
    const int32_t longest = (int32_t)as_int(a[7]);
    const Workspace ws(a[10]);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[11], "dev_status"));
    void* stream = stream_of(a[12]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.prefill_stack((int32_t)k.layers.size(), k.layers.data(), c.get(), k.index.data(), k.io.data(), (int32_t)k.rows, (int32_t)s.n_seq,
                               longest, s.cu, s.init, s.fin, ws.p, ws.bytes, nullptr, st, stream);
    });
}

// (table, layers, which, cache, inputs, outs, parent_slot, node_slot, level_offsets, dev_status, stream) -> status or None, as above
PyObject* tree_step_stack(PyObject* const* a) {
    const Stack k(a[1], a[2], a[4], a[5]);
    if (!k.apart || k.layers.size() < 2) Py_RETURN_NONE;
    const Cache c(a[3]);
    const Nodes n(a[6], a[7], k.rows);
    const Levels lv(a[8]);
    int32_t* st = static_cast<int32_t*>(mutable_data(a[9], "dev_status"));
    void* stream = stream_of(a[10]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.tree_step_stack((int32_t)k.layers.size(), k.layers.data(), c.get(), k.index.data(), k.io.data(), (int32_t)k.rows, n.parent, n.node,
                                 lv.count(), lv.get(), st, stream);
    });
}

// A list of dense bf16 matrices of one shape, as addresses.
std::vector<const void*> dense(PyObject* list, const char* name, int64_t rows, int64_t cols) {
    Ref f(PySequence_Fast(list, name));
    std::vector<const void*> v;
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(f.p); ++i) {
        const at::Tensor& t = tensor(PySequence_Fast_GET_ITEM(f.p, i), name);
        if (t.scalar_type() != at::kBFloat16 || t.dim() != 2 || t.size(0) != rows || t.size(1) != cols || !t.is_contiguous() || !t.is_cuda())
            fail(PyExc_ValueError, std::string(name) + ": need contiguous bf16 CUDA matrices of " + std::to_string(rows) + " x " + std::to_string(cols));
        v.push_back(t.const_data_ptr());
    }
    return v;
}
void* scratch(PyObject* o, const char* name, int64_t rows, int64_t cols) {
    const at::Tensor& t = tensor(o, name);
    if (t.scalar_type() != at::kBFloat16 || t.dim() != 2 || t.size(0) < rows || t.size(1) != cols || !t.is_contiguous())
        fail(PyExc_ValueError, std::string(name) + ": need a contiguous bf16 matrix with " + std::to_string(cols) + " columns and a row per node");
    return t.data_ptr();
}

// (table, layers, (W_in, W_x, W_dt, W_out, embed, W_lm), cache, tokens, parent_slot, node_slot, h, xz, y, logits, dev_status,
//  stream, flags, eps)
PyObject* block_generation(PyObject* const* a) {
    Ref ls(PySequence_Fast(a[1], "layers")), w(PySequence_Fast(a[2], "weights"));
    if (PySequence_Fast_GET_SIZE(w.p) != 6) fail(PyExc_ValueError, "weights are (W_in, W_x, W_dt, W_out, embed, W_lm)");
    std::vector<mdraft_layer> layers;
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(ls.p); ++i) layers.push_back(layer_of(PySequence_Fast_GET_ITEM(ls.p, i), a[13]));
    if (layers.empty()) fail(PyExc_ValueError, "no layers");
    const at::Tensor &embed = tensor(PySequence_Fast_GET_ITEM(w.p, 4), "embed"), &lm = tensor(PySequence_Fast_GET_ITEM(w.p, 5), "W_lm");
    Ref dts(PySequence_Fast(PySequence_Fast_GET_ITEM(w.p, 2), "W_dt"));
    if (PySequence_Fast_GET_SIZE(dts.p) < 1) fail(PyExc_ValueError, "no W_dt");
    const at::Tensor& wdt = tensor(PySequence_Fast_GET_ITEM(dts.p, 0), "W_dt");
    if (embed.dim() != 2 || lm.dim() != 2 || wdt.dim() != 2 || embed.scalar_type() != at::kBFloat16 || lm.scalar_type() != at::kBFloat16 ||
        !embed.is_contiguous() || !lm.is_contiguous() || embed.size(0) != lm.size(1) || embed.size(1) != lm.size(0))
        fail(PyExc_ValueError, "embed (vocab, d_model) and W_lm (d_model, vocab) must be contiguous bf16 matrices");
    const int64_t D = layers[0].d_inner, M = embed.size(1), V = embed.size(0), R = wdt.size(1);
    const auto W_in = dense(PySequence_Fast_GET_ITEM(w.p, 0), "W_in", M, 2 * D), W_x = dense(PySequence_Fast_GET_ITEM(w.p, 1), "W_x", R + 2 * layers[0].d_state, D),
               W_dt = dense(dts.p, "W_dt", D, R), W_out = dense(PySequence_Fast_GET_ITEM(w.p, 3), "W_out", D, M);
    const size_t n = layers.size();
    if (W_in.size() != n || W_x.size() != n || W_dt.size() != n || W_out.size() != n) fail(PyExc_ValueError, "one matrix of each kind per layer");
    const mdraft_block_stack stack = {(int32_t)n, (int32_t)M, (int32_t)R, (int32_t)V, layers.data(), W_in.data(), W_x.data(), W_dt.data(), W_out.data(),
                                      embed.const_data_ptr(), lm.const_data_ptr(), (float)PyFloat_AsDouble(a[14])};
    if (PyErr_Occurred()) throw Failed();
    const Cache c(a[3]);
    const at::Tensor& tok = tensor(a[4], "tokens");
    if (tok.scalar_type() != at::kLong || !tok.is_contiguous()) fail(PyExc_TypeError, "tokens must be contiguous int64");
    const int64_t m = tok.numel();
    const Nodes nodes(a[5], a[6], m);
    void *h = scratch(a[7], "h", m, M), *xz = scratch(a[8], "xz", m, 2 * D), *y = scratch(a[9], "y", m, D);
    const Matrix logits(a[10], "logits");
    if (logits.rows != m || tensor(a[10], "logits").scalar_type() != at::kBFloat16) fail(PyExc_ValueError, "logits: one bf16 row per node");
    int32_t* st = static_cast<int32_t*>(mutable_data(a[11], "dev_status"));
    void* stream = stream_of(a[12]);
    const Entry& e = entry(a[0]);
    return released([&] {
        return e.block_generation(&stack, c.get(), static_cast<const int64_t*>(tok.const_data_ptr()), (int32_t)m, nodes.parent, nodes.node, h, xz, y,
                                  logits.out(), logits.ld, st, stream);
    });
}

#define ENTRY(name, args) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&guarded<name, args>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(table, 1), ENTRY(prefill, 20), ENTRY(prefill_noalloc, 18), ENTRY(tree_step, 16), ENTRY(tree_step_proj, 15),
                         ENTRY(commit, 6), ENTRY(ssd_prefill, 17), ENTRY(ssd_tree_step, 16), ENTRY(prefill_stack, 13),
                         ENTRY(tree_step_stack, 11), ENTRY(block_generation, 15), {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_host", "argument marshalling for libmdraft.so", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host() {
    struct { PyObject** to; const char* text; } all[] = {
        {&N.A, "A"}, {&N.D, "D"}, {&N.conv_w, "conv_w"}, {&N.conv_b, "conv_b"}, {&N.dt_bias, "dt_bias"}, {&N.act, "act"}, {&N.flags, "flags"},
        {&N.d_inner, "d_inner"}, {&N.d_state, "d_state"}, {&N.d_conv, "d_conv"}, {&N.headdim, "headdim"}, {&N.ssm, "ssm"}, {&N.conv, "conv"},
        {&N.n_layers, "n_layers"}, {&N.n_slots, "n_slots"}, {&N.cuda_stream, "cuda_stream"}, {&N.cuda_event, "cuda_event"}};
    for (auto& n : all)
        if (!(*n.to = PyUnicode_InternFromString(n.text))) return nullptr;
    return PyModule_Create(&module_def);
}
