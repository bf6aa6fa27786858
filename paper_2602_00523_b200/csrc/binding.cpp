// Marshalling of the library's calls for Python: takes torch tensors, checks what the Python side used to
// check (device, contiguity, element type), and calls the C entry points of libsage.so (include/sage.h)
// with raw pointers, sizes and the stream.  A call through ctypes spent 18 to 33 us on this, more than
// most of the kernels run (a round's small calls last 2 to 20 us on the GPU); here it is about one.
//
// Every function takes its arguments by position and returns the entry point's code; None means that `out` lacks
// a tensor (the Python wrapper then allocates and calls again).  The GIL is released around the C call.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "sage.h"

namespace {

struct Failed {};                                   // a Python exception has been set

[[noreturn]] void fail(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw Failed{};
}
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a torch tensor is expected");
    return THPVariable_Unpack(o);
}
// Address of a tensor, nullptr for None.
template <typename T = void>
T* ptr(PyObject* o) {
    if (o == nullptr || o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o);
    if (!t.is_cuda()) fail(PyExc_ValueError, "device tensors only");
    if (!t.is_contiguous()) fail(PyExc_ValueError, "contiguous tensors only");
    return static_cast<T*>(t.data_ptr());
}
int64_t length(PyObject* o) { return (o == nullptr || o == Py_None) ? 0 : tensor(o).numel(); }
int integer(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    if (v > INT32_MAX || v < INT32_MIN) fail(PyExc_OverflowError, "integer argument out of range");
    return static_cast<int>(v);
}
int size32(int64_t v) {
    if (v > INT32_MAX) fail(PyExc_OverflowError, "size out of range");
    return static_cast<int>(v);
}
void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    static PyObject* name = PyUnicode_InternFromString("cuda_stream");
    PyObject* v = PyObject_GetAttr(o, name);
    if (v == nullptr) throw Failed{};
    void* s = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw Failed{};
    return s;
}
// A ctypes structure's bytes.
template <typename T>
T structure(PyObject* o) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Failed{};
    const bool fits = view.len == static_cast<Py_ssize_t>(sizeof(T));
    T v{};
    if (fits) v = *static_cast<const T*>(view.buf);
    PyBuffer_Release(&view);
    if (!fits) fail(PyExc_TypeError, "unexpected policy structure");
    return v;
}

// Names of dict entries.
struct Names {
    PyObject *topk_idx, *topk_logprob, *entropy_full, *entropy_topk, *alpha, *lse, *draft_token, *template_id, *depth_cont,
        *width_cont, *next_parent, *next_rank, *next_node_offsets, *parent, *rank, *depth, *token, *cum_logprob, *n_nodes,
        *frontier_begin, *path, *path_len, *bonus_token;
} N;

struct Missing {};                                  // `out` lacks an entry
// A dict, or any other mapping, of tensors; what another mapping hands out is held until the call has been made.
class Tensors {
public:
    explicit Tensors(PyObject* o) : o_(o), dict_(PyDict_Check(o)) {
        if (!dict_ && !PyMapping_Check(o)) fail(PyExc_TypeError, "a dict of tensors is expected");
    }
    ~Tensors() {
        for (int i = 0; i < n_held_; ++i) Py_DECREF(held_[i]);
    }
    Tensors(const Tensors&) = delete;
    Tensors& operator=(const Tensors&) = delete;
    PyObject* get(PyObject* name) {                 // nullptr where there is none
        if (dict_) {
            PyObject* v = PyDict_GetItemWithError(o_, name);
            if (v == nullptr && PyErr_Occurred()) throw Failed{};
            return v;
        }
        PyObject* v = PyObject_GetItem(o_, name);
        if (v == nullptr) {
            if (!PyErr_ExceptionMatches(PyExc_KeyError)) throw Failed{};
            PyErr_Clear();
            return nullptr;
        }
        return held_[n_held_++] = v;
    }
    PyObject* operator[](PyObject* name) {
        PyObject* v = get(name);
        if (v == nullptr) throw Missing{};
        return v;
    }

private:
    PyObject* o_;
    bool dict_;
    int n_held_ = 0;
    PyObject* held_[8];                             // (no call asks for more)
};

template <typename F>
PyObject* guarded(Py_ssize_t n_args, Py_ssize_t want, F body) {
    if (n_args != want) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    try {
        return PyLong_FromLong(body());
    } catch (const Failed&) {
        return nullptr;
    } catch (const Missing&) {
        Py_RETURN_NONE;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename F>
int without_gil(F call) {
    int code;
    Py_BEGIN_ALLOW_THREADS
    code = call();
    Py_END_ALLOW_THREADS
    return code;
}

// logits, k, k_entropy, parent, rank, node_offsets, root_token, out, ws (None: the static variant), status, stream, static?
PyObject* expand_topk(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 12, [&]() -> int {
        const at::Tensor& lg = tensor(a[0]);
        if (lg.scalar_type() != at::kFloat || lg.dim() != 2 || lg.stride(1) != 1)
            fail(PyExc_AssertionError, "logits: fp32 [rows, vocab] with contiguous rows");
        Tensors o(a[7]);
        const int k = integer(a[1]), ke = integer(a[2]);
        const bool tree = a[3] != Py_None, is_static = a[11] == Py_True;
        int32_t* idx = ptr<int32_t>(o[N.topk_idx]);
        float *lp = ptr<float>(o[N.topk_logprob]), *hf = ptr<float>(o[N.entropy_full]),
              *ht = ptr<float>(o[N.entropy_topk]), *al = ptr<float>(o[N.alpha]), *ls = ptr<float>(o[N.lse]);
        int32_t* tok = ptr<int32_t>(tree ? o[N.draft_token] : o.get(N.draft_token));
        if (!is_static && a[8] == Py_None) throw Missing{};
        const int batch = tree ? size32(length(a[5]) - 1) : 0;
        const int32_t *parent = ptr<int32_t>(a[3]), *rank = ptr<int32_t>(a[4]), *offs = ptr<int32_t>(a[5]), *root = ptr<int32_t>(a[6]);
        void* ws = is_static ? nullptr : ptr(a[8]);
        const size_t ws_bytes = is_static ? 0 : static_cast<size_t>(length(a[8]));
        int32_t* status = ptr<int32_t>(a[9]);
        void* stream = stream_of(a[10]);
        const float* x = static_cast<const float*>(lg.data_ptr());
        const int rows = size32(lg.size(0)), vocab = size32(lg.size(1));
        const int64_t stride = lg.stride(0);
        return without_gil([&] {
            return is_static ? sage_expand_topk_static(x, rows, vocab, stride, k, ke, idx, lp, hf, ht, al, ls, parent, rank, offs,
                                                       batch, root, tok, status, stream)
                             : sage_expand_topk(x, rows, vocab, stride, k, ke, idx, lp, hf, ht, al, ls, parent, rank, offs, batch,
                                                root, tok, ws, ws_bytes, status, stream);
        });
    });
}

// alpha, alpha_row, batch, policy, out, bank_parent, bank_rank, bank_n_nodes, handover?, status, stream
PyObject* select_tree(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 11, [&]() -> int {
        Tensors o(a[4]);
        const sage_tree_policy pol = structure<sage_tree_policy>(a[3]);
        const bool handover = PyObject_IsTrue(a[8]) == 1;
        int32_t* id = ptr<int32_t>(o[N.template_id]);
        float *d = ptr<float>(o[N.depth_cont]), *w = ptr<float>(o[N.width_cont]);
        int32_t* np = ptr<int32_t>(handover ? o[N.next_parent] : o.get(N.next_parent));
        int32_t* nr = ptr<int32_t>(handover ? o[N.next_rank] : o.get(N.next_rank));
        int32_t* no = ptr<int32_t>(handover ? o[N.next_node_offsets] : o.get(N.next_node_offsets));
        const float* alpha = ptr<float>(a[0]);
        const int32_t *row = ptr<int32_t>(a[1]), *bp = ptr<int32_t>(a[5]), *br = ptr<int32_t>(a[6]), *bn = ptr<int32_t>(a[7]);
        const int batch = a[2] != Py_None ? integer(a[2]) : size32(a[1] != Py_None ? length(a[1]) : length(a[0]));
        int32_t* status = ptr<int32_t>(a[9]);
        void* stream = stream_of(a[10]);
        return without_gil([&] { return sage_select_tree(alpha, row, batch, &pol, id, d, w, bp, br, bn, np, nr, no, status, stream); });
    });
}

// topk_idx, topk_logprob, alpha, policy, tree, alpha_row, n_max, d_max_seq, status, stream
PyObject* grow_tree(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&]() -> int {
        Tensors t(a[4]);
        const sage_tree_policy pol = structure<sage_tree_policy>(a[3]);
        const at::Tensor& idx = tensor(a[0]);
        if (idx.dim() != 2) fail(PyExc_AssertionError, "topk_idx: [slots, k]");
        PyObject* nn = t[N.n_nodes];
        const int batch = size32(length(nn)), k = size32(idx.size(1)), n_max = integer(a[6]);
        const int32_t* ix = ptr<int32_t>(a[0]);
        const float *lp = ptr<float>(a[1]), *alpha = ptr<float>(a[2]), *dm = ptr<float>(a[7]);
        const int32_t* row = ptr<int32_t>(a[5]);
        int32_t *parent = ptr<int32_t>(t[N.parent]), *rank = ptr<int32_t>(t[N.rank]),
                *depth = ptr<int32_t>(t[N.depth]), *token = ptr<int32_t>(t[N.token]);
        float* cum = ptr<float>(t[N.cum_logprob]);
        int32_t *nodes = ptr<int32_t>(nn), *fb = ptr<int32_t>(t[N.frontier_begin]), *status = ptr<int32_t>(a[8]);
        void* stream = stream_of(a[9]);
        return without_gil([&] {
            return sage_grow_tree(ix, lp, k, alpha, row, batch, &pol, n_max, parent, rank, depth, token, cum, nodes, fb, dm, status, stream);
        });
    });
}

// path_len, policy, window_buf, count, d_max, status, stream
PyObject* update_history(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 7, [&]() -> int {
        const sage_history_policy pol = structure<sage_history_policy>(a[1]);
        const int32_t* pl = ptr<int32_t>(a[0]);
        const int batch = size32(length(a[0]));
        int32_t *win = ptr<int32_t>(a[2]), *count = ptr<int32_t>(a[3]), *status = ptr<int32_t>(a[5]);
        float* d = ptr<float>(a[4]);
        void* stream = stream_of(a[6]);
        return without_gil([&] { return sage_update_history(pl, batch, &pol, win, count, d, status, stream); });
    });
}

// parent, node_offsets, out, status, stream
PyObject* build_ancestor_mask(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 5, [&]() -> int {
        const int32_t *parent = ptr<int32_t>(a[0]), *offs = ptr<int32_t>(a[1]);
        const int batch = size32(length(a[1]) - 1);
        uint64_t* anc = ptr<uint64_t>(a[2]);
        int32_t* status = ptr<int32_t>(a[3]);
        void* stream = stream_of(a[4]);
        return without_gil([&] { return sage_build_ancestor_mask(parent, offs, batch, anc, status, stream); });
    });
}

// Shapes of the two pools ([layers, pages, kv heads, page, head dim], layers at the same distance in both).
struct Pools {
    void *k, *v;
    int64_t layer_stride;
    int layers, pages, kv_heads, page, dim;
};
Pools pools_of(PyObject* ko, PyObject* vo) {
    const at::Tensor &k = tensor(ko), &v = tensor(vo);
    if (k.dim() != 5) fail(PyExc_ValueError, "pools: [layers, pages, kv heads, page, head dim]");
    Pools p{k.data_ptr(), v.data_ptr(), 0, size32(k.size(0)), size32(k.size(1)), size32(k.size(2)), size32(k.size(3)), size32(k.size(4))};
    p.layer_stride = p.layers > 1 ? k.stride(0) : static_cast<int64_t>(p.pages) * p.kv_heads * p.page * p.dim;
    return p;
}

// q, k_pool, v_pool, page_table, seq_len, parent, node_offsets, sm_scale, out, ws, status, stream
PyObject* tree_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 12, [&]() -> int {
        const at::Tensor &q = tensor(a[0]), &kt = tensor(a[1]), &vt = tensor(a[2]), &pt = tensor(a[3]);
        if (q.scalar_type() != at::kBFloat16 || kt.scalar_type() != at::kBFloat16 || vt.scalar_type() != at::kBFloat16)
            fail(PyExc_AssertionError, "q and the pools are bf16");
        if (q.dim() != 4 || pt.dim() != 2) fail(PyExc_ValueError, "q: [layers, nodes, heads, head dim]; page_table: [batch, pages]");
        const Pools p = pools_of(a[1], a[2]);
        const int layers = size32(q.size(0));
        const int64_t stride = layers > 1 ? kt.stride(0) : static_cast<int64_t>(p.pages) * p.kv_heads * p.page * p.dim;
        if (!vt.sizes().equals(kt.sizes()) || (layers > 1 && vt.stride(0) != stride))
            fail(PyExc_AssertionError, "the pools have one shape and one distance between layers");
        const double scale = PyFloat_AsDouble(a[7]);
        if (scale == -1.0 && PyErr_Occurred()) throw Failed{};
        const int nodes = size32(q.size(1)), heads = size32(q.size(2)), dim = size32(q.size(3));
        const int batch = size32(pt.size(0)), max_pages = size32(pt.size(1));
        const void* qp = ptr(a[0]);
        const int32_t *table = ptr<int32_t>(a[3]), *len = ptr<int32_t>(a[4]), *parent = ptr<int32_t>(a[5]), *offs = ptr<int32_t>(a[6]);
        void *out = ptr(a[8]), *ws = ptr(a[9]);
        const size_t ws_bytes = static_cast<size_t>(length(a[9]));
        int32_t* status = ptr<int32_t>(a[10]);
        void* stream = stream_of(a[11]);
        return without_gil([&] {
            return sage_tree_attention(qp, p.k, p.v, stride, layers, p.pages, table, max_pages, len, parent, offs, batch, nodes, heads,
                                       p.kv_heads, dim, p.page, static_cast<float>(scale), out, ws, ws_bytes, status, stream);
        });
    });
}

// parent, draft_token, target_argmax, node_offsets, max_path, out, status, stream
PyObject* accept(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&]() -> int {
        Tensors o(a[5]);
        int32_t *path = ptr<int32_t>(o[N.path]), *pl = ptr<int32_t>(o[N.path_len]),
                *bonus = ptr<int32_t>(o[N.bonus_token]);
        const int32_t *parent = ptr<int32_t>(a[0]), *draft = ptr<int32_t>(a[1]), *target = ptr<int32_t>(a[2]), *offs = ptr<int32_t>(a[3]);
        const int batch = size32(length(a[3]) - 1), max_path = integer(a[4]);
        int32_t* status = ptr<int32_t>(a[6]);
        void* stream = stream_of(a[7]);
        return without_gil([&] { return sage_accept(parent, draft, target, offs, batch, max_path, path, pl, bonus, status, stream); });
    });
}

// k_pool, v_pool, page_table, seq_len, path, path_len, status, stream
PyObject* compact_kv(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&]() -> int {
        const Pools p = pools_of(a[0], a[1]);
        const at::Tensor &pt = tensor(a[2]), &path_t = tensor(a[4]);
        if (pt.dim() != 2 || path_t.dim() != 2) fail(PyExc_ValueError, "page_table: [batch, pages]; path: [batch, max_path]");
        const int batch = size32(pt.size(0)), max_pages = size32(pt.size(1)), max_path = size32(path_t.size(1));
        const int32_t* table = ptr<int32_t>(a[2]);
        int32_t* len = ptr<int32_t>(a[3]);
        const int32_t *path = ptr<int32_t>(a[4]), *pl = ptr<int32_t>(a[5]);
        int32_t* status = ptr<int32_t>(a[6]);
        void* stream = stream_of(a[7]);
        return without_gil([&] {
            return sage_compact_kv(p.k, p.v, p.layer_stride, p.layers, p.pages, table, max_pages, len, path, pl, batch, max_path,
                                   p.kv_heads, p.dim, p.page, status, stream);
        });
    });
}

#define ENTRY(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(f)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {ENTRY(expand_topk), ENTRY(select_tree), ENTRY(grow_tree), ENTRY(update_history),
                          ENTRY(build_ancestor_mask), ENTRY(tree_attention), ENTRY(accept), ENTRY(compact_kv),
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", "Marshalling of libsage.so's calls.", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
#define NAME(x) N.x = PyUnicode_InternFromString(#x)
    NAME(topk_idx); NAME(topk_logprob); NAME(entropy_full); NAME(entropy_topk); NAME(alpha); NAME(lse); NAME(draft_token);
    NAME(template_id); NAME(depth_cont); NAME(width_cont); NAME(next_parent); NAME(next_rank); NAME(next_node_offsets);
    NAME(parent); NAME(rank); NAME(depth); NAME(token); NAME(cum_logprob); NAME(n_nodes); NAME(frontier_begin);
    NAME(path); NAME(path_len); NAME(bonus_token);
#undef NAME
    return PyModule_Create(&kModule);
}
