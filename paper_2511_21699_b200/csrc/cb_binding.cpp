// The host side of the calls that a decoding loop makes once a step: argument checks, device pointers and the current stream in one
// C++ call each.  A launch costs the host 2 to 3 us; checked and marshalled in Python (nine tensors a call, an object for the
// stream, ctypes' conversions) a call took 10 to 13 us, longer than the kernels of a small batch run: acceptance of one sequence over 32 k
// tokens 11.4 us a call that way and 5 to 6 this way, a prompt of 300 tokens with reset and first draft (three calls) 24 and 19 us.
//
// The entry points of the C library come as addresses from _lib.load() (set_library), so that this module calls the build of the library
// that was loaded.  What a check refuses raises CachebackError with the text that it has in api.py; torch's own exceptions
// (a stride of a tensor without dimensions, a tensor without memory) pass through as they do there.
#include <Python.h>

#include <algorithm>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "cacheback.h"

namespace {

PyObject* g_error = nullptr;                                 // CachebackError
PyObject *s_cuda_stream, *s_tokens, *s_parent, *s_depth, *s_mask, *s_n_nodes, *s_n_accept, *s_accept_nodes, *s_out_tokens, *s_target_ids;

struct Library {
    decltype(&cb_reset) reset;
    decltype(&cb_update) update;
    decltype(&cb_update_bulk) update_bulk;
    decltype(&cb_draft_tree) draft_tree;
    decltype(&cb_update_draft_tree) update_draft_tree;
    decltype(&cb_tree_attn) tree_attn;
    decltype(&cb_accept) accept;
    decltype(&cb_accept_update_draft_tree) accept_update_draft_tree;
    decltype(&cb_kv_commit) kv_commit;
    decltype(&cb_status_str) status_str;
} g_lib;

struct Refused {};                                           // a Python exception is set

[[noreturn]] void refuse(const char* text) {
    PyErr_SetString(g_error, text);
    throw Refused();
}

const at::Tensor& tensor_of(PyObject* o) {
    if (!THPVariable_Check(o)) refuse("expected a contiguous CUDA tensor");
    return THPVariable_Unpack(o);
}

const char* type_name(at::ScalarType t) { return t == at::kInt ? "torch.int32" : t == at::kFloat ? "torch.float32" : "torch.bfloat16"; }

// The device pointer of a contiguous CUDA tensor of the given type; None: a null pointer.
template <typename T = int32_t>
T* ptr(PyObject* o, at::ScalarType want = at::kInt) {
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor_of(o);
    if (!t.is_cuda() || !t.is_contiguous()) refuse("expected a contiguous CUDA tensor");
    if (t.scalar_type() != want) {
        PyObject* d = PyObject_GetAttrString(o, "dtype");
        if (d) { PyErr_Format(g_error, "expected dtype %s, got %S", type_name(want), d); Py_DECREF(d); }
        throw Refused();
    }
    return static_cast<T*>(t.data_ptr());
}

struct Ref {                                                 // an owned reference
    PyObject* o;
    explicit Ref(PyObject* x) : o(x) { if (!x) throw Refused(); }
    Ref(const Ref&) = delete;
    ~Ref() { Py_DECREF(o); }
};
template <typename T = int32_t>
T* item(PyObject* mapping, PyObject* key) {
    Ref r(PyObject_GetItem(mapping, key));
    return ptr<T>(r.o);
}

void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    Ref r(PyObject_GetAttr(o, s_cuda_stream));
    void* p = PyLong_AsVoidPtr(r.o);
    if (!p && PyErr_Occurred()) throw Refused();
    return p;
}

cb_ctx* ctx_of(PyObject* o) {
    if (o == Py_None) return nullptr;                         // a closed context: the library refuses it
    Ref r(PyObject_GetAttrString(o, "value"));
    if (r.o == Py_None) return nullptr;
    void* p = PyLong_AsVoidPtr(r.o);
    if (!p && PyErr_Occurred()) throw Refused();
    return static_cast<cb_ctx*>(p);
}

// The logits of all nodes: [batch, max_nodes, vocab] with one stride from row to row.
const void* logits_of(PyObject* o, int32_t* dtype, int64_t* stride) {
    const at::Tensor& t = tensor_of(o);
    if (t.scalar_type() == at::kFloat) *dtype = CB_DTYPE_F32;
    else if (t.scalar_type() == at::kBFloat16) *dtype = CB_DTYPE_BF16;
    else refuse("logits must be float32 or bfloat16");
    if (!(t.is_cuda() && t.dim() == 3 && t.stride(2) == 1 && t.stride(0) == t.size(1) * t.stride(1)))
        refuse("logits must be [batch, max_nodes, vocab] with a uniform row stride");
    *stride = t.stride(1);
    return t.data_ptr();
}

int64_t long_of(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Refused();
    return v;
}

template <typename F>
void call(const char* what, F&& f) {
    cb_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    if (st != CB_OK) {
        PyErr_Format(g_error, "%s failed: %s", what, g_lib.status_str(st));
        throw Refused();
    }
}

// Python's entry: the number of arguments is fixed (api.py fills in the defaults)
template <int N, void (*F)(PyObject* const*)>
PyObject* entry(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != N) { PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n); return nullptr; }
    try {
        F(a);
    } catch (const Refused&) {
        return nullptr;
    }
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// The token history [batch, columns]: its pointer and the columns that a row has.  The stride of a dimension of size one says nothing:
// the transpose of a [columns, 1] tensor is contiguous with a stride of 1.
template <typename T = int32_t>
T* history_of(PyObject* o, int64_t* row_stride) {
    T* p = ptr<T>(o);
    const at::Tensor& t = tensor_of(o);
    *row_stride = t.stride(0);
    if (t.dim() > 1 && t.size(0) == 1) *row_stride = std::max(*row_stride, t.numel());
    return p;
}

// handle, seq_mask, stream
void do_reset(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    const int32_t* m = ptr(a[1]);
    void* st = stream_of(a[2]);
    call("cb_reset", [&] { return g_lib.reset(c, m, st); });
}
// handle, tokens, n_old, n_new, stream
template <bool BULK>
void do_update(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    int64_t rs;
    const int32_t* tok = history_of(a[1], &rs);
    const int32_t *n0 = ptr(a[2]), *n1 = ptr(a[3]);
    void* st = stream_of(a[4]);
    call(BULK ? "cb_update_bulk" : "cb_update", [&] { return (BULK ? g_lib.update_bulk : g_lib.update)(c, tok, rs, n0, n1, st); });
}
struct Tree { int32_t *tok, *par, *dep; uint32_t* mask; int32_t* n; };
Tree tree_of(PyObject* t, bool mask) {
    Tree r;
    r.tok = item(t, s_tokens); r.par = item(t, s_parent); r.dep = item(t, s_depth);
    r.mask = mask ? item<uint32_t>(t, s_mask) : nullptr;
    r.n = item(t, s_n_nodes);
    return r;
}
// handle, tokens, seq_len, tree, stream
void do_draft(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    int64_t rs;
    const int32_t* tok = history_of(a[1], &rs);
    const int32_t* n = ptr(a[2]);
    const Tree t = tree_of(a[3], true);
    void* st = stream_of(a[4]);
    call("cb_draft_tree", [&] { return g_lib.draft_tree(c, tok, rs, n, t.tok, t.par, t.dep, t.mask, t.n, st); });
}
// handle, tokens, n_old, n_new, tree, stream
void do_update_draft(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    int64_t rs;
    const int32_t* tok = history_of(a[1], &rs);
    const int32_t *n0 = ptr(a[2]), *n1 = ptr(a[3]);
    const Tree t = tree_of(a[4], true);
    void* st = stream_of(a[5]);
    call("cb_update_draft_tree", [&] { return g_lib.update_draft_tree(c, tok, rs, n0, n1, t.tok, t.par, t.dep, t.mask, t.n, st); });
}
// handle, tree, logits, target_ids, res, stream
void do_accept(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    int32_t dtype = 0;
    int64_t rs = 0;
    const void* lg = a[2] == Py_None ? nullptr : logits_of(a[2], &dtype, &rs);
    const Tree t = tree_of(a[1], false);
    const int32_t* ids = ptr(a[3]);
    int32_t *na = item(a[4], s_n_accept), *an = item(a[4], s_accept_nodes), *ot = item(a[4], s_out_tokens), *ti = item(a[4], s_target_ids);
    void* st = stream_of(a[5]);
    call("cb_accept", [&] { return g_lib.accept(c, t.tok, t.par, t.dep, t.n, lg, dtype, rs, ids, na, an, ot, ti, st); });
}
// handle, tree, logits, tokens, seq_len, next_tree, res, stream
void do_accept_update_draft(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    cb_accept_draft_args x = {};
    x.logits = logits_of(a[2], &x.logits_dtype, &x.logits_row_stride);
    const Tree t = tree_of(a[1], false);
    x.tree_tokens = t.tok; x.tree_parent = t.par; x.tree_depth = t.dep; x.n_nodes = t.n;
    x.n_accept = item(a[6], s_n_accept); x.accept_nodes = item(a[6], s_accept_nodes);
    x.out_tokens = item(a[6], s_out_tokens); x.target_ids_out = item(a[6], s_target_ids);
    x.tokens = history_of(a[3], &x.row_stride);
    x.seq_len = ptr(a[4]);
    const Tree n = tree_of(a[5], true);
    x.next_tokens = n.tok; x.next_parent = n.par; x.next_depth = n.dep; x.next_mask = n.mask; x.next_n_nodes = n.n;
    void* st = stream_of(a[7]);
    call("cb_accept_update_draft_tree", [&] { return g_lib.accept_update_draft_tree(c, &x, st); });
}
// handle, q, k_pool, v_pool, block_table, ctx_len, k_tree, v_tree, tree_mask, n_nodes, out, lse, max_ctx, scale, stream
void do_attn(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    cb_attn_args x = {};
    const auto bf = at::kBFloat16;
    x.q = ptr<void>(a[1], bf); x.k_pool = ptr<void>(a[2], bf); x.v_pool = ptr<void>(a[3], bf);
    x.block_table = ptr(a[4]); x.ctx_len = ptr(a[5]);
    x.k_tree = ptr<void>(a[6], bf); x.v_tree = ptr<void>(a[7], bf);
    x.tree_mask = ptr<uint32_t>(a[8]); x.n_nodes = ptr(a[9]);
    x.out = ptr<void>(a[10], bf); x.lse = ptr<float>(a[11], at::kFloat);
    x.max_pages = (int32_t)tensor_of(a[4]).size(1);
    x.num_pages = (int32_t)tensor_of(a[2]).size(0);
    x.max_ctx = (int32_t)long_of(a[12]);
    const double sc = PyFloat_AsDouble(a[13]);
    if (sc == -1.0 && PyErr_Occurred()) throw Refused();
    x.scale = (float)sc;
    void* st = stream_of(a[14]);
    call("cb_tree_attn", [&] { return g_lib.tree_attn(c, &x, st); });
}
// handle, k_pool, v_pool, block_table, ctx_len, k_tree, v_tree, n_accept, accept_nodes, stream
void do_kv_commit(PyObject* const* a) {
    cb_ctx* c = ctx_of(a[0]);
    cb_kv_commit_args x = {};
    const auto bf = at::kBFloat16;
    x.k_pool = ptr<void>(a[1], bf); x.v_pool = ptr<void>(a[2], bf);
    x.block_table = ptr(a[3]); x.ctx_len = ptr(a[4]);
    x.k_tree = ptr<void>(a[5], bf); x.v_tree = ptr<void>(a[6], bf);
    x.n_accept = ptr(a[7]); x.accept_nodes = ptr(a[8]);
    x.max_pages = (int32_t)tensor_of(a[3]).size(1);
    x.num_pages = (int32_t)tensor_of(a[1]).size(0);
    void* st = stream_of(a[9]);
    call("cb_kv_commit", [&] { return g_lib.kv_commit(c, &x, st); });
}

// set_library(CachebackError, {name: address})
PyObject* set_library(PyObject*, PyObject* args) {
    PyObject *err, *addr;
    if (!PyArg_ParseTuple(args, "OO!", &err, &PyDict_Type, &addr)) return nullptr;
    auto take = [&](const char* name, auto* f) {
        PyObject* o = PyDict_GetItemString(addr, name);
        if (!o) { PyErr_Format(PyExc_KeyError, "%s", name); return false; }
        void* p = PyLong_AsVoidPtr(o);
        if (!p) { if (!PyErr_Occurred()) PyErr_Format(PyExc_ValueError, "no address for %s", name); return false; }
        *f = reinterpret_cast<std::remove_reference_t<decltype(*f)>>(p);
        return true;
    };
    Library l;
    if (!(take("cb_reset", &l.reset) && take("cb_update", &l.update) && take("cb_update_bulk", &l.update_bulk) && take("cb_draft_tree", &l.draft_tree) &&
          take("cb_update_draft_tree", &l.update_draft_tree) && take("cb_tree_attn", &l.tree_attn) && take("cb_accept", &l.accept) &&
          take("cb_accept_update_draft_tree", &l.accept_update_draft_tree) && take("cb_kv_commit", &l.kv_commit) && take("cb_status_str", &l.status_str)))
        return nullptr;
    g_lib = l;
    Py_INCREF(err);
    Py_XSETREF(g_error, err);
    Py_RETURN_NONE;
}

#define CB_FAST(name, n, f) {name, (PyCFunction)(void (*)(void))(entry<n, f>), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    {"set_library", set_library, METH_VARARGS, nullptr},
    CB_FAST("reset", 3, do_reset), CB_FAST("update", 5, do_update<false>), CB_FAST("update_bulk", 5, do_update<true>), CB_FAST("draft_tree", 5, do_draft),
    CB_FAST("update_draft_tree", 6, do_update_draft), CB_FAST("accept", 6, do_accept), CB_FAST("accept_update_draft_tree", 8, do_accept_update_draft),
    CB_FAST("tree_attn", 15, do_attn), CB_FAST("kv_commit", 10, do_kv_commit), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
    struct { PyObject** at; const char* text; } names[] = {
        {&s_cuda_stream, "cuda_stream"}, {&s_tokens, "tokens"}, {&s_parent, "parent"}, {&s_depth, "depth"}, {&s_mask, "mask"}, {&s_n_nodes, "n_nodes"},
        {&s_n_accept, "n_accept"}, {&s_accept_nodes, "accept_nodes"}, {&s_out_tokens, "out_tokens"}, {&s_target_ids, "target_ids"}};
    for (auto& n : names)
        if (!(*n.at = PyUnicode_InternFromString(n.text))) return nullptr;
    return PyModule_Create(&g_module);
}
