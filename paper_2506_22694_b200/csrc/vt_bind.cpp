// Argument marshalling of the calls that a drafting loop or a vocabulary build makes, as a CPython extension: the checks, the outputs'
// allocation and the call into libvocabtrim.so, without Python in between.  A drafting step is 9 to 40 us on the device, and
// Python marshalling added 4 us to a call on the host (us, Python / here: a head 12.9 / 8.5, a rerank 9.9 / 5.8); nothing of the method
// happens here.  The functions of the library are registered by address (`use`), so that the library can be another build.
//
// Every function returns its outputs, or the library's status as an int when that is not VT_OK.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ops/empty.h>

#include <cstdint>

#include "vocabtrim.h"

namespace {

decltype(&vt_draft_head) g_head, g_head_overlapped, g_head_host;
decltype(&vt_draft_head_expand) g_expand;
decltype(&vt_tree_rerank) g_rerank;
decltype(&vt_verify_greedy) g_verify;
decltype(&vt_build_vocab) g_build;
decltype(&vt_trim_head) g_trim;
PyObject *g_make_ws, *g_raw_stream, *g_device;       // (op, shape, like) -> Workspace; torch's raw current stream of a device; its current device
PyObject *s_ptr, *s_nbytes;

struct Ref {                                         // an owned reference
    PyObject* p;
    explicit Ref(PyObject* o = nullptr) : p(o) {}
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
};

// thrown with a Python exception set
[[noreturn]] void raise() { throw python_error(); }
template <class... A>
[[noreturn]] void raise(PyObject* type, const char* format, A... a) {
    PyErr_Format(type, format, a...);
    raise();
}

const at::Tensor& tensor(PyObject* o, const char* attribute = "is_cuda") {
    if (!THPVariable_Check(o)) raise(PyExc_AttributeError, "'%s' object has no attribute '%s'", Py_TYPE(o)->tp_name, attribute);
    return THPVariable_Unpack(o);
}

const at::Tensor& dev(PyObject* o, at::ScalarType dtype, const char* name) {
    const at::Tensor& t = tensor(o);
    if (!(t.is_cuda() && t.scalar_type() == dtype && t.is_contiguous()))
        raise(PyExc_TypeError, "%s must be a contiguous CUDA tensor of dtype torch.%s", name,
              dtype == at::kInt ? "int32" : dtype == at::kLong ? "int64" : dtype == at::kFloat ? "float32" : "bfloat16");
    return t;
}

template <class T>
T* data(const at::Tensor& t) { return reinterpret_cast<T*>(t.data_ptr()); }
template <class T>
T* data_of(PyObject* o) { return o == Py_None ? nullptr : data<T>(tensor(o, "data_ptr")); }

int64_t integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) raise();
    return v;
}

void* pointer(PyObject* o) {
    if (o == Py_None) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) raise();
    return p;
}

void* stream() {
    Ref d(PyObject_CallNoArgs(g_device));
    if (!d.p) raise();
    Ref s(PyObject_CallOneArg(g_raw_stream, d.p));
    if (!s.p) raise();
    return pointer(s.p);
}

void expect_args(Py_ssize_t n, Py_ssize_t want) {
    if (n != want) raise(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
}

// The interpreter's lock given up for a scope (an exception that leaves it has the lock again).
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    Unlocked() = default;
    Unlocked(const Unlocked&) = delete;
    Unlocked& operator=(const Unlocked&) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};

// A call into the library without the lock.  Its arguments are plain pointers and numbers, all of them made before the lock is given
// up: a tensor may refuse its data pointer, which raises.
template <class F, class... A>
int call(F* function, A... arguments) {
    const Unlocked u;
    return function(arguments...);
}

// the parts of a tuple or list, checked for their number as Python's unpacking does, and kept (a list may lose them meanwhile)
struct Parts {
    Ref own[3];
    PyObject* at[3];
    Parts(PyObject* o, Py_ssize_t want) {
        const Ref seq(PySequence_Fast(o, "cannot unpack non-iterable object"));
        if (!seq.p) raise();
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq.p);
        if (n < want) raise(PyExc_ValueError, "not enough values to unpack (expected %zd, got %zd)", want, n);
        if (n > want) raise(PyExc_ValueError, "too many values to unpack (expected %zd)", want);
        for (Py_ssize_t i = 0; i < want; ++i) Py_INCREF(own[i].p = at[i] = PySequence_Fast_GET_ITEM(seq.p, i));
    }
};

// the caller's workspace, or one made for the call
struct Space {
    Ref made;
    void* ptr;
    size_t bytes;
    Space(PyObject* ws, int op, PyObject* like, int64_t n, int64_t V, int64_t K, int64_t d, int64_t B, int64_t topk) {
        if (ws == Py_None) {
            made.p = PyObject_CallFunction(g_make_ws, "iLLLLLLO", op, (long long)n, (long long)V, (long long)K, (long long)d, (long long)B,
                                           (long long)topk, like);
            if (!made.p) raise();
            ws = made.p;
        }
        Ref p(PyObject_GetAttr(ws, s_ptr));
        if (!p.p) raise();
        Ref b(PyObject_GetAttr(ws, s_nbytes));
        if (!b.p) raise();
        ptr = pointer(p.p);
        bytes = (size_t)integer(b.p);
    }
};

// (without the lock, as torch.empty: an allocation may wait for the device)
at::Tensor make(const at::Tensor& like, at::ScalarType dtype, at::IntArrayRef shape) {
    const at::TensorOptions options = like.options().dtype(dtype).requires_grad(false);
    const Unlocked u;
    return at::empty(shape, options);
}

// what a head call takes, checked
struct Head {
    const at::Tensor &h, &W, &temp;
    const int32_t* map = nullptr;
    const float* u = nullptr;
    int64_t B, d, K, topk;
    Head(PyObject* ph, PyObject* pW, PyObject* pmap, PyObject* ptemp, PyObject* ptopk, PyObject* pu)
        : h(dev(ph, at::kBFloat16, "h")), W(dev(pW, at::kBFloat16, "W_trim")), temp(dev(ptemp, at::kFloat, "temp")) {
        if (h.dim() != 2) raise(PyExc_ValueError, "h must be [B,d]");
        if (W.dim() < 2) raise(PyExc_IndexError, "tuple index out of range");
        B = h.size(0);
        d = h.size(1);
        K = W.size(0);
        if (W.size(1) != d || temp.numel() != B) raise(PyExc_ValueError, "shape mismatch between h, W_trim and temp");
        if (pmap != Py_None) {
            const at::Tensor& m = dev(pmap, at::kInt, "map");
            if (m.numel() != K) raise(PyExc_ValueError, "map must have K entries");
            map = data<int32_t>(m);
        }
        if (pu != Py_None) {
            const at::Tensor& t = dev(pu, at::kFloat, "uniforms");
            if (t.dim() != 2 || t.size(0) != B || t.size(1) != K) raise(PyExc_ValueError, "uniforms must be [B,K]");
            u = data<float>(t);
        }
        topk = integer(ptopk);
    }
};

// the caller's (ids, log-probabilities), or new ones
struct Outs {
    Ref ids, lps;
    Outs(PyObject* out, const Head& a) {
        if (out == Py_None) {
            ids.p = THPVariable_Wrap(make(a.h, at::kInt, {a.B, 1 + a.topk}));
            lps.p = THPVariable_Wrap(make(a.h, at::kFloat, {a.B, 1 + a.topk}));
            if (!ids.p || !lps.p) raise();
        } else {
            Parts p(out, 2);
            Py_INCREF(ids.p = p.at[0]);
            Py_INCREF(lps.p = p.at[1]);
        }
    }
};

struct Pool {
    Parts parts;
    const at::Tensor &token, &parent, &score;
    int64_t capacity;
    explicit Pool(PyObject* o)
        : parts(o, 3), token(dev(parts.at[0], at::kInt, "pool token")), parent(dev(parts.at[1], at::kInt, "pool parent")),
          score(dev(parts.at[2], at::kFloat, "pool score")) {
        capacity = std::min(std::min(token.numel(), parent.numel()), score.numel());
    }
};

// (h, W_trim, map, temp, topk, uniforms, ws, out, overlapped)
PyObject* draft_head(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 9);
    const Head in(a[0], a[1], a[2], a[3], a[4], a[5]);
    Outs out(a[7], in);
    int32_t* ids = data_of<int32_t>(out.ids.p);
    float* lps = data_of<float>(out.lps.p);
    const Space ws(a[6], VT_OP_DRAFT_HEAD, a[0], 0, 0, in.K, in.d, in.B, in.topk);
    const int overlapped = PyObject_IsTrue(a[8]);
    if (overlapped < 0) raise();
    void* s = stream();
    const int status = call(overlapped ? g_head_overlapped : g_head, data<uint16_t>(in.h), data<uint16_t>(in.W), in.map, (int32_t)in.B, (int32_t)in.K,
                                                              (int32_t)in.d, data<float>(in.temp), (int32_t)in.topk, in.u, ids, lps,
                                                              ws.ptr, ws.bytes, s);
    if (status != VT_OK) return PyLong_FromLong(status);
    return PyTuple_Pack(2, out.ids.p, out.lps.p);
    END_HANDLE_TH_ERRORS
}

// (h, W_trim, map, temp, topk, uniforms, frontier, pool, pool_base, n_front, ws, out)
PyObject* draft_head_expand(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 12);
    const Head in(a[0], a[1], a[2], a[3], a[4], a[5]);
    if (a[6] != Py_None && dev(a[6], at::kInt, "frontier_nodes").numel() != in.B)
        raise(PyExc_ValueError, "frontier_nodes must have B entries");
    const Pool pool(a[7]);
    Outs out(a[11], in);
    const int64_t base = integer(a[8]), n_front = integer(a[9]);
    const at::Tensor next = make(pool.token, at::kInt, {n_front});
    int32_t* ids = data_of<int32_t>(out.ids.p);
    float* lps = data_of<float>(out.lps.p);
    const Space ws(a[10], VT_OP_DRAFT_HEAD, a[0], 0, 0, in.K, in.d, in.B, in.topk);
    const int32_t* frontier = data_of<int32_t>(a[6]);
    void* s = stream();
    const int status = call(g_expand, data<uint16_t>(in.h), data<uint16_t>(in.W), in.map, (int32_t)in.B, (int32_t)in.K, (int32_t)in.d,
                             data<float>(in.temp), (int32_t)in.topk, in.u, ids, lps, frontier, data<int32_t>(pool.token),
                             data<int32_t>(pool.parent), data<float>(pool.score), (int32_t)base, (int32_t)pool.capacity, (int32_t)n_front,
                             data<int32_t>(next), ws.ptr, ws.bytes, s);
    if (status != VT_OK) return PyLong_FromLong(status);
    Ref nx(THPVariable_Wrap(next));
    if (!nx.p) raise();
    return PyTuple_Pack(3, out.ids.p, out.lps.p, nx.p);
    END_HANDLE_TH_ERRORS
}

// (h, W_trim, map, B, K, d, temp, topk, uniforms, ids, lps, ws)
PyObject* draft_head_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 12);
    const Space ws(a[11], VT_OP_DRAFT_HEAD_HOST, a[0], 0, 0, 0, 0, 0, 0);
    const uint16_t *h = data_of<uint16_t>(a[0]), *W = data_of<uint16_t>(a[1]);
    const int32_t* map = data_of<int32_t>(a[2]);
    const int32_t B = (int32_t)integer(a[3]), K = (int32_t)integer(a[4]), d = (int32_t)integer(a[5]), topk = (int32_t)integer(a[7]);
    const float *temp = data_of<float>(a[6]), *u = data_of<float>(a[8]);
    int32_t* ids = data_of<int32_t>(a[9]);
    float* lps = data_of<float>(a[10]);
    void* s = stream();
    const int status = call(g_head_host, h, W, map, B, K, d, temp, topk, u, ids, lps, ws.ptr, ws.bytes, s);
    return PyLong_FromLong(status);
    END_HANDLE_TH_ERRORS
}

// (pool, n, budget)
PyObject* tree_rerank(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 3);
    const Pool pool(a[0]);
    const int64_t nodes = integer(a[1]), budget = integer(a[2]);
    if (nodes > pool.capacity) raise(PyExc_ValueError, "n exceeds the pool");
    at::Tensor t[3];
    for (at::Tensor& x : t) x = make(pool.token, at::kInt, {budget});
    void* s = stream();
    const int status = call(g_rerank, data<int32_t>(pool.token), data<int32_t>(pool.parent), data<float>(pool.score), (int32_t)nodes, (int32_t)budget,
                             data<int32_t>(t[0]), data<int32_t>(t[1]), data<int32_t>(t[2]), s);
    if (status != VT_OK) return PyLong_FromLong(status);
    Ref r0(THPVariable_Wrap(t[0])), r1(THPVariable_Wrap(t[1])), r2(THPVariable_Wrap(t[2]));
    if (!r0.p || !r1.p || !r2.p) raise();
    return PyTuple_Pack(3, r0.p, r1.p, r2.p);
    END_HANDLE_TH_ERRORS
}

// (token, parent, target, tokens_total)
PyObject* verify_greedy(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 4);
    const at::Tensor &token = dev(a[0], at::kInt, "token"), &target = dev(a[2], at::kInt, "target");
    if (token.dim() != 2) raise(PyExc_ValueError, "token must be [S, N]");
    const int64_t S = token.size(0), N = token.size(1);
    if (target.dim() != 2 || target.size(0) != S || target.size(1) != N + 1) raise(PyExc_ValueError, "target must be [S, N+1]");
    if (a[1] != Py_None) {
        const at::Tensor& p = dev(a[1], at::kInt, "parent");
        if (p.dim() != 2 || p.size(0) != S || p.size(1) != N) raise(PyExc_ValueError, "parent must be [S, N]");
    }
    if (a[3] != Py_None) dev(a[3], at::kLong, "tokens_total");
    const at::Tensor n_accept = make(token, at::kInt, {S}), path = make(token, at::kInt, {S, N}), emitted = make(token, at::kInt, {S, N + 1});
    const int32_t* parent = data_of<int32_t>(a[1]);
    uint64_t* total = data_of<uint64_t>(a[3]);
    void* s = stream();
    const int status = call(g_verify, data<int32_t>(token), parent, data<int32_t>(target), (int32_t)S, (int32_t)N, data<int32_t>(n_accept),
                             data<int32_t>(path), data<int32_t>(emitted), total, s);
    if (status != VT_OK) return PyLong_FromLong(status);
    Ref r0(THPVariable_Wrap(n_accept)), r1(THPVariable_Wrap(path)), r2(THPVariable_Wrap(emitted));
    if (!r0.p || !r1.p || !r2.p) raise();
    return PyTuple_Pack(3, r0.p, r1.p, r2.p);
    END_HANDLE_TH_ERRORS
}

// (ids, V, K, ws)
PyObject* build_vocab(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 4);
    const at::Tensor& ids = dev(a[0], at::kInt, "ids");
    const int64_t V = integer(a[1]), K = integer(a[2]), count = ids.numel();
    const at::Tensor map = make(ids, at::kInt, {K}), inv = make(ids, at::kInt, {V});
    const Space ws(a[3], VT_OP_BUILD_VOCAB, a[0], count, V, K, 0, 0, 0);
    void* s = stream();
    const int status = call(g_build, data<int32_t>(ids), count, (int32_t)V, (int32_t)K, data<int32_t>(map), data<int32_t>(inv), ws.ptr, ws.bytes, s);
    if (status != VT_OK) return PyLong_FromLong(status);
    Ref r0(THPVariable_Wrap(map)), r1(THPVariable_Wrap(inv));
    if (!r0.p || !r1.p) raise();
    return PyTuple_Pack(2, r0.p, r1.p);
    END_HANDLE_TH_ERRORS
}

// (W_full, map, W_trim or None, ws or None)
PyObject* trim_head(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 4);
    const at::Tensor &W = dev(a[0], at::kBFloat16, "W_full"), &map = dev(a[1], at::kInt, "map");
    if (W.dim() != 2) raise(PyExc_ValueError, "W_full must be [V,d]");
    const int64_t V = W.size(0), d = W.size(1), K = map.numel();
    Ref out;
    if (a[2] == Py_None) out.p = THPVariable_Wrap(make(W, at::kBFloat16, {K, d}));
    else Py_INCREF(out.p = a[2]);
    if (!out.p) raise();
    const at::Tensor& trim = dev(out.p, at::kBFloat16, "W_trim");
    void* ws = nullptr;
    const int given = PyObject_IsTrue(a[3]);
    if (given < 0) raise();
    if (given) {
        Ref p(PyObject_GetAttr(a[3], s_ptr));
        if (!p.p) raise();
        ws = pointer(p.p);
    }
    void* s = stream();
    const int status = call(g_trim, data<uint16_t>(W), data<int32_t>(map), data<uint16_t>(trim), (int32_t)V, (int32_t)K, (int32_t)d, ws, s);
    if (status != VT_OK) return PyLong_FromLong(status);
    Py_INCREF(out.p);
    return out.p;
    END_HANDLE_TH_ERRORS
}

// (addresses of the library's functions by name, make_ws, raw_stream, current_device)
PyObject* use(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    expect_args(n, 4);
    auto at = [&](const char* name) {
        PyObject* o = PyDict_GetItemString(a[0], name);
        if (!o) raise(PyExc_KeyError, "%s", name);
        return pointer(o);
    };
    g_head = reinterpret_cast<decltype(g_head)>(at("vt_draft_head"));
    g_head_overlapped = reinterpret_cast<decltype(g_head)>(at("vt_draft_head_overlapped"));
    g_head_host = reinterpret_cast<decltype(g_head)>(at("vt_draft_head_host"));
    g_expand = reinterpret_cast<decltype(g_expand)>(at("vt_draft_head_expand"));
    g_rerank = reinterpret_cast<decltype(g_rerank)>(at("vt_tree_rerank"));
    g_verify = reinterpret_cast<decltype(g_verify)>(at("vt_verify_greedy"));
    g_build = reinterpret_cast<decltype(g_build)>(at("vt_build_vocab"));
    g_trim = reinterpret_cast<decltype(g_trim)>(at("vt_trim_head"));
    PyObject** kept[] = {&g_make_ws, &g_raw_stream, &g_device};
    for (int i = 0; i < 3; ++i) {
        Py_INCREF(a[1 + i]);
        Py_XDECREF(*kept[i]);
        *kept[i] = a[1 + i];
    }
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

#define VT_FN(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {VT_FN(draft_head), VT_FN(draft_head_expand), VT_FN(draft_head_host), VT_FN(tree_rerank), VT_FN(verify_greedy),
                           VT_FN(build_vocab), VT_FN(trim_head), VT_FN(use), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_vt_bind", "Argument marshalling for libvocabtrim.so", -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// What the module was compiled for: its view of torch's and Python's objects is theirs only.  (VT_BIND_FOR comes from build.py, which also
// looks for this text in the file to know whether it is up to date.)
static const char kFor[] = "_vt_bind for " VT_BIND_FOR;

static bool fits() {
    Ref torch(PyImport_ImportModule("torch")), sys(PyImport_ImportModule("sys"));
    Ref core(torch.p ? PyObject_GetAttrString(torch.p, "_C") : nullptr), impl(sys.p ? PyObject_GetAttrString(sys.p, "implementation") : nullptr);
    if (!core.p || !impl.p) return false;
    Ref tag(PyObject_GetAttrString(impl.p, "cache_tag")), version(PyObject_GetAttrString(torch.p, "__version__"));
    Ref abi(PyObject_GetAttrString(core.p, "_GLIBCXX_USE_CXX11_ABI"));
    if (!tag.p || !version.p || !abi.p) return false;
    Ref now(PyUnicode_FromFormat("_vt_bind for %S, torch %S, C++ ABI %d", tag.p, version.p, PyObject_IsTrue(abi.p)));
    if (!now.p) return false;
    if (PyUnicode_CompareWithASCIIString(now.p, kFor) == 0) return true;
    PyErr_Format(PyExc_ImportError, "built as %s, this is %U", kFor, now.p);
    return false;
}

PyMODINIT_FUNC PyInit__vt_bind() {
    if (!fits()) return nullptr;
    s_ptr = PyUnicode_InternFromString("ptr");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    return s_ptr && s_nbytes ? PyModule_Create(&g_module) : nullptr;
}
