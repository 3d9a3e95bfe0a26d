// Argument marshalling of the Python binding, in native code: dtype / device / shape checks of torch tensors, output
// and workspace allocation, and the call of the C entry point of the same name.
//
// The calls of a step on few sequences are shorter on the GPU (10 - 20 us) than ctypes marshalling was on the host
// (25 us per attention call: a dozen ctypes objects, as many tensor attribute look-ups, numpy conversions of the two
// host arrays), so the host paced the GPU.  The same checks cost about a microsecond here.  The library is not linked: its entry
// points are handed over by address (attach), so that the binding can load another build of it.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <stdarg.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <exception>
#include <utility>
#include <vector>

#include "../../include/specroll.h"

namespace {

struct Raised {};  // a Python exception has been set

PyObject *g_error = nullptr;     // SpecrollError
PyObject *g_host_i32 = nullptr;  // binding._host_i32: anything array-like -> contiguous int32 numpy array
PyObject *g_alloc = nullptr;     // replacement of torch.empty as f(shape, dtype code, device index), or nullptr

constexpr at::ScalarType BF16 = at::kBFloat16, F32 = at::kFloat, I32 = at::kInt, U8 = at::kByte;

[[noreturn]] void fail(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    PyObject *msg = PyUnicode_FromFormatV(fmt, ap);
    va_end(ap);
    if (msg) {
        PyErr_SetObject(g_error ? g_error : PyExc_RuntimeError, msg);
        Py_DECREF(msg);
    }
    throw Raised();
}

// The library's entry points, by address.
#define SPECROLL_ENTRIES(X)                                                                                          \
    X(specroll_strerror) X(specroll_propose_workspace_bytes) X(specroll_propose) X(specroll_tree_draw)               \
    X(specroll_tree_attn_workspace_bytes) X(specroll_tree_attn) X(specroll_tree_attn_paged_workspace_bytes)          \
    X(specroll_tree_attn_paged) X(specroll_commit_path) X(specroll_commit_path_layers) X(specroll_gather_hidden)                             \
    X(specroll_verify_workspace_bytes) X(specroll_verify) X(specroll_verify_static)                                  \
    X(specroll_verify_nucleus_workspace_bytes)                                                                       \
    X(specroll_verify_nucleus) X(specroll_reflex_feedback_workspace_bytes) X(specroll_reflex_feedback_ex)            \
    X(specroll_reflex_sketch) X(specroll_reflex_gate) X(specroll_target_head_stats_workspace_bytes)                  \
    X(specroll_target_head_stats) X(specroll_target_head_rows) X(specroll_verify_want_ids)                           \
    X(specroll_target_head_tile_mass_bytes)                                                                          \
    X(specroll_target_head_stats_tiles) X(specroll_verify_hidden)
struct Entries {
#define X(name) decltype(&::name) name;
    SPECROLL_ENTRIES(X)
#undef X
} lib;

void check(int rc, const char *what) {
    if (rc != SPECROLL_OK) fail("%s: %s (code %d)", what, lib.specroll_strerror(rc), rc);
}

// ---- arguments
const at::Tensor *tensor(PyObject *o, const char *name) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) fail("%s must be a CUDA tensor", name);
    return &THPVariable_Unpack(o);
}
const at::Tensor &need(PyObject *o, const char *name, int dim) {
    const at::Tensor *t = tensor(o, name);
    if (!t || t->dim() != dim) fail("%s must be a tensor of %d dimensions", name, dim);
    return *t;
}
const at::Tensor &need(PyObject *o, const char *name) {  // (of any shape)
    const at::Tensor *t = tensor(o, name);
    if (!t) fail("%s must be a CUDA tensor", name);
    return *t;
}
void *dev(const at::Tensor *t, at::ScalarType dtype, const char *name) {
    if (!t) return nullptr;
    if (!t->is_cuda()) fail("%s must be a CUDA tensor", name);
    if (t->scalar_type() != dtype) fail("%s must have dtype %s, got %s", name, c10::toString(dtype), c10::toString(t->scalar_type()));
    if (!t->is_contiguous()) fail("%s must be contiguous", name);
    return t->mutable_data_ptr();  // (as Tensor.data_ptr(): a lazily cloned tensor gets storage of its own)
}
void *dev(const at::Tensor &t, at::ScalarType dtype, const char *name) { return dev(&t, dtype, name); }
void *dev(PyObject *o, at::ScalarType dtype, const char *name) { return dev(tensor(o, name), dtype, name); }

bool shape(const at::Tensor &t, std::initializer_list<int64_t> want) { return t.sizes() == at::IntArrayRef(want); }

long integer(PyObject *o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return v;
}
float number(PyObject *o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised();
    return (float)v;
}

// A one-dimensional int32 host array for the length of a call: numpy arrays of that type as they are, anything else
// through the binding's converter.
class HostI32 {
  public:
    HostI32(PyObject *o, const char *name) {
        if (!view(o)) {
            made_ = PyObject_CallFunction(g_host_i32, "Os", o, name);
            if (!made_) throw Raised();
            if (!view(made_)) {
                Py_DECREF(made_);
                fail("%s must be one-dimensional", name);
            }
        }
    }
    ~HostI32() {
        PyBuffer_Release(&buf_);
        Py_XDECREF(made_);
    }
    HostI32(const HostI32 &) = delete;
    HostI32 &operator=(const HostI32 &) = delete;
    const int32_t *data() const { return static_cast<const int32_t *>(buf_.buf); }
    int64_t size() const { return buf_.len / 4; }
    int32_t last() const { return size() ? data()[size() - 1] : 0; }

  private:
    bool view(PyObject *o) {
        if (!PyObject_CheckBuffer(o)) return false;
        if (PyObject_GetBuffer(o, &buf_, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
            PyErr_Clear();
            return false;
        }
        if (buf_.ndim == 1 && buf_.itemsize == 4 && buf_.format && buf_.format[0] == 'i' && !buf_.format[1]) return true;
        PyBuffer_Release(&buf_);
        return false;
    }
    Py_buffer buf_{};
    PyObject *made_ = nullptr;
};

// A reference held for the length of a call.
struct Ref {
    PyObject *o;
    explicit Ref(PyObject *o_) : o(o_) {
        if (!o) throw Raised();
    }
    Ref(Ref &&r) noexcept : o(std::exchange(r.o, nullptr)) {}
    ~Ref() { Py_XDECREF(o); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

// ---- results
at::Tensor alloc(std::initializer_list<int64_t> size, at::ScalarType dtype, const at::Tensor &like) {
    if (!g_alloc) return at::empty(at::IntArrayRef(size), at::TensorOptions().dtype(dtype).device(like.device()));
    PyObject *shp = PyTuple_New((Py_ssize_t)size.size());
    Py_ssize_t i = 0;
    for (int64_t s : size) PyTuple_SET_ITEM(shp, i++, PyLong_FromLongLong(s));
    PyObject *r = PyObject_CallFunction(g_alloc, "Nii", shp, (int)dtype, like.is_cuda() ? (int)like.get_device() : -1);
    if (!r) throw Raised();
    if (!THPVariable_Check(r)) {
        Py_DECREF(r);
        fail("the allocator must return a tensor");
    }
    at::Tensor t = THPVariable_Unpack(r);
    Py_DECREF(r);
    return t;
}
at::Tensor alloc_bytes(size_t n, const at::Tensor &like) {
    return alloc({(int64_t)(n < 256 ? 256 : n)}, U8, like);
}
// The workspace of a call: the caller's, or a new one of `n` bytes.
at::Tensor workspace(PyObject *o, size_t n, const at::Tensor &like) {
    const at::Tensor *t = tensor(o, "workspace");
    return t ? *t : alloc_bytes(n, like);
}
void *ptr(const at::Tensor &t) { return t.mutable_data_ptr(); }
size_t bytes_of(const at::Tensor &t) { return (size_t)t.numel(); }

// The outputs by name: the caller's mapping, or a new dict that new tensors go into.
class Out {
  public:
    explicit Out(PyObject *given) : given_(given && given != Py_None ? given : nullptr) {
        dict_ = given_ ? Py_NewRef(given_) : PyDict_New();
        if (!dict_) throw Raised();
    }
    ~Out() { Py_XDECREF(dict_); }
    void *get(const char *name, std::initializer_list<int64_t> size, at::ScalarType dtype, const at::Tensor &like, bool optional = false) {
        if (!given_) return put(name, alloc(size, dtype, like));
        if (!PyDict_CheckExact(given_)) {
            const Ref o(optional ? PyObject_CallMethod(given_, "get", "s", name) : PyMapping_GetItemString(given_, name));
            return dev(o.o, dtype, name);
        }
        PyObject *o = PyDict_GetItemString(given_, name);
        if (!o) {
            if (optional) return nullptr;
            PyErr_SetString(PyExc_KeyError, name);
            throw Raised();
        }
        return dev(o, dtype, name);
    }
    void *put(const char *name, const at::Tensor &t) {
        PyObject *o = THPVariable_Wrap(t);
        if (!o || PyDict_SetItemString(dict_, name, o) != 0) {
            Py_XDECREF(o);
            throw Raised();
        }
        Py_DECREF(o);
        return ptr(t);
    }
    PyObject *release() { return std::exchange(dict_, nullptr); }
    PyObject *peek() const { return dict_; }

  private:
    PyObject *given_, *dict_;
};

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The C call itself runs without the interpreter lock, as a ctypes call does.  Its arguments are evaluated before the lock is
// given up (they may raise, or turn Python objects into numbers), and it is taken back however the call ends.
struct Unlocked {
    PyThreadState *state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <class F, class... Args>
int call_unlocked(F *entry, Args... args) {
    Unlocked u;
    return entry(args...);
}
#define CALL(name, ...) check(call_unlocked(lib.name, __VA_ARGS__, stream()), #name)

// ------------------------------------------------------------------------------ proposal

PyObject *propose(PyObject *const *a) {
    const at::Tensor &h = need(a[0], "h", 2), &A = need(a[2], "A", 3), &bias = need(a[3], "bias", 2), &W = need(a[4], "W", 2);
    const at::Tensor *m = tensor(a[5], "m"), *alpha = tensor(a[6], "alpha");
    HostI32 parent(a[7], "parent");
    const at::Tensor &anchor = need(a[1], "anchor", 1), &u = need(a[8], "u_draw", 2);
    const int64_t B = h.size(0), d = h.size(1), K = A.size(0), V = W.size(0), N = parent.size(), k = integer(a[9]);
    const int flags = (int)integer(a[18]);
    if (!shape(A, {K, d, d}) || !shape(bias, {K, d}) || W.size(1) != d) fail("propose: inconsistent weight shapes");
    if (!shape(u, {B, N}) || anchor.size(0) != B) fail("propose: inconsistent u_draw / anchor shapes");
    if (flags & SPECROLL_REFLEX_PRE_HEAD) {
        if (m && !shape(*m, {B, d})) fail("propose: with REFLEX_PRE_HEAD m must be [B,d]");
        if (alpha && !shape(*alpha, {B})) fail("propose: with REFLEX_PRE_HEAD alpha must be [B]");
    } else {
        if (m && !shape(*m, {B, K, d})) fail("propose: m must be [B,K,d]");
        if (alpha && !shape(*alpha, {B, K})) fail("propose: alpha must be [B,K]");
    }
    const specroll_propose_desc D = {(int32_t)B, (int32_t)N, (int32_t)K, (int32_t)k, (int32_t)d, (int32_t)V,
                                     number(a[10]), number(a[11]), number(a[12]), number(a[13]), flags};
    Out out(a[17]);
    auto *ci = (int32_t *)out.get("cand_id", {B, K, k}, I32, h);
    auto *cl = (float *)out.get("cand_logit", {B, K, k}, F32, h);
    auto *tt = (int32_t *)out.get("tree_tok", {B, N}, I32, h);
    auto *tc = (uint8_t *)out.get("tree_cand", {B, N}, U8, h);
    auto *sq = (float *)out.get("slot_q", {B, N}, F32, h);
    const at::Tensor ws = workspace(a[16], lib.specroll_propose_workspace_bytes(&D), h);
    const void *ph = dev(h, BF16, "h"), *pA = dev(A, BF16, "A"), *pb = dev(bias, BF16, "bias"), *pW = dev(W, BF16, "W");
    const void *pg = dev(a[14], BF16, "ln_gamma"), *pbt = dev(a[15], BF16, "ln_beta");
    const auto *pan = (const int32_t *)dev(anchor, I32, "anchor");
    const auto *pm = (const float *)dev(m, F32, "m"), *pal = (const float *)dev(alpha, F32, "alpha"), *pu = (const float *)dev(u, F32, "u_draw");
    CALL(specroll_propose, &D, ph, pan, pA, pb, pg, pbt, pW, pm, pal, parent.data(), pu, ci, cl, tt, tc, sq, ptr(ws), bytes_of(ws));
    return Py_BuildValue("NN", out.release(), THPVariable_Wrap(ws));
}

PyObject *tree_draw(PyObject *const *a) {
    HostI32 parent(a[0], "parent");
    const at::Tensor &ci = need(a[2], "cand_id", 3);
    const int64_t B = ci.size(0), K = ci.size(1), k = ci.size(2), N = parent.size();
    Out out(nullptr);
    auto *tt = (int32_t *)out.get("tree_tok", {B, N}, I32, ci);
    auto *tc = (uint8_t *)out.get("tree_cand", {B, N}, U8, ci);
    auto *sq = (float *)out.get("slot_q", {B, N}, F32, ci);
    const auto *pa = (const int32_t *)dev(a[1], I32, "anchor"), *pc = (const int32_t *)dev(ci, I32, "cand_id");
    const auto *pl = (const float *)dev(a[3], F32, "cand_logit"), *pu = (const float *)dev(a[4], F32, "u_draw");
    CALL(specroll_tree_draw, (int32_t)B, (int32_t)N, (int32_t)K, (int32_t)k, number(a[5]), parent.data(), pa, pc, pl, pu, tt, tc, sq);
    return out.release();
}

// ------------------------------------------------------------------------------ attention

float attn_scale(PyObject *o, int64_t D) { return o == Py_None ? (float)(1.0 / std::sqrt((double)D)) : number(o); }

// (out, lse, workspace) of an attention call
PyObject *attn_result(const at::Tensor &O, const at::Tensor &lse, const at::Tensor &ws) {
    return Py_BuildValue("NNN", THPVariable_Wrap(O), lse.defined() ? THPVariable_Wrap(lse) : Py_NewRef(Py_None), THPVariable_Wrap(ws));
}

PyObject *tree_attn(PyObject *const *a) {
    const at::Tensor &Q = need(a[0], "Q", 4), &Kc = need(a[1], "Kc", 3), &Vc = need(a[2], "Vc", 3), &Kt = need(a[5], "Kt", 4), &Vt = need(a[6], "Vt", 4);
    HostI32 ip(a[4], "kv_indptr_host"), parent(a[7], "parent");
    const int64_t B = Q.size(0), N = Q.size(1), Hq = Q.size(2), D = Q.size(3), Hkv = Kt.size(2);
    if (ip.size() != B + 1 || !shape(Kt, {B, N, Hkv, D}) || !shape(Vt, {B, N, Hkv, D}) || parent.size() < N)
        fail("tree_attn: inconsistent shapes");
    if (!shape(Kc, {ip.last(), Hkv, D}) || Vc.sizes() != Kc.sizes()) fail("tree_attn: cache shape does not match kv_indptr");
    const specroll_attn_desc desc = {(int32_t)B, (int32_t)N, (int32_t)Hq, (int32_t)Hkv, (int32_t)D, attn_scale(a[8], D), (int32_t)integer(a[13])};
    const at::Tensor O = a[11] != Py_None ? *tensor(a[11], "O") : alloc({B, N, Hq, D}, BF16, Q);
    at::Tensor lse;
    if (a[12] != Py_None) lse = *tensor(a[12], "lse");
    else if (PyObject_IsTrue(a[9])) lse = alloc({B, N, Hq}, F32, Q);
    const at::Tensor ws = workspace(a[10], a[10] == Py_None ? lib.specroll_tree_attn_workspace_bytes(&desc, ip.data()) : 0, Q);
    const void *pq = dev(Q, BF16, "Q"), *pk = dev(Kc, BF16, "Kc"), *pv = dev(Vc, BF16, "Vc"), *pkt = dev(Kt, BF16, "Kt"), *pvt = dev(Vt, BF16, "Vt");
    const auto *pi = (const int32_t *)dev(a[3], I32, "kv_indptr_dev");
    void *po = dev(O, BF16, "O");
    auto *pl = lse.defined() ? (float *)dev(lse, F32, "lse") : nullptr;
    CALL(specroll_tree_attn, &desc, pq, pk, pv, pi, ip.data(), pkt, pvt, parent.data(), po, pl, ptr(ws), bytes_of(ws));
    return attn_result(O, lse, ws);
}

PyObject *tree_attn_paged(PyObject *const *a) {
    const at::Tensor &Q = need(a[0], "Q", 4), &Kp = need(a[1], "Kp", 4), &Vp = need(a[2], "Vp", 4), &Kt = need(a[7], "Kt", 4), &Vt = need(a[8], "Vt", 4);
    const at::Tensor &pi = need(a[4], "page_indptr"), &kl = need(a[5], "kv_len_dev");
    HostI32 len(a[6], "kv_len_host"), parent(a[9], "parent");
    const int64_t B = Q.size(0), N = Q.size(1), Hq = Q.size(2), D = Q.size(3), Hkv = Kt.size(2);
    if (len.size() != B || !shape(Kt, {B, N, Hkv, D}) || !shape(Vt, {B, N, Hkv, D}) || parent.size() < N)
        fail("tree_attn_paged: inconsistent shapes");
    if (!shape(Kp, {Kp.size(0), SPECROLL_PAGE_TOKENS, Hkv, D}) || Vp.sizes() != Kp.sizes())
        fail("tree_attn_paged: page pool must be [n_pages, 128, Hkv, D]");
    if (pi.numel() != B + 1 || kl.numel() != B) fail("tree_attn_paged: page_indptr / kv_len_dev sizes");
    const specroll_attn_desc desc = {(int32_t)B, (int32_t)N, (int32_t)Hq, (int32_t)Hkv, (int32_t)D, attn_scale(a[10], D), (int32_t)integer(a[15])};
    const at::Tensor O = a[13] != Py_None ? *tensor(a[13], "O") : alloc({B, N, Hq, D}, BF16, Q);
    at::Tensor lse;
    if (a[14] != Py_None) lse = *tensor(a[14], "lse");
    else if (PyObject_IsTrue(a[11])) lse = alloc({B, N, Hq}, F32, Q);
    const at::Tensor ws = workspace(a[12], a[12] == Py_None ? lib.specroll_tree_attn_paged_workspace_bytes(&desc, len.data()) : 0, Q);
    const void *pq = dev(Q, BF16, "Q"), *pk = dev(Kp, BF16, "Kp"), *pv = dev(Vp, BF16, "Vp"), *pkt = dev(Kt, BF16, "Kt"), *pvt = dev(Vt, BF16, "Vt");
    const auto *pt = (const int32_t *)dev(a[3], I32, "page_table"), *pip = (const int32_t *)dev(pi, I32, "page_indptr"), *pkl = (const int32_t *)dev(kl, I32, "kv_len_dev");
    void *po = dev(O, BF16, "O");
    auto *pl = lse.defined() ? (float *)dev(lse, F32, "lse") : nullptr;
    CALL(specroll_tree_attn_paged, &desc, pq, pk, pv, (int64_t)Kp.size(0), pt, pip, pkl, len.data(), pkt, pvt, parent.data(), po, pl, ptr(ws), bytes_of(ws));
    return attn_result(O, lse, ws);
}

// ------------------------------------------------------------------------------ between two rounds

PyObject *commit_path(PyObject *const *a) {
    // Kt, Vt, path_node, n_acc, Kp, Vp, page_table, page_indptr, kv_len, kv_len_out, status
    const at::Tensor &Kt = need(a[0], "Kt", 4), &path = need(a[2], "path_node"), &Kp = need(a[4], "Kp");
    const int64_t B = Kt.size(0), N = Kt.size(1), Hkv = Kt.size(2), D = Kt.size(3), K = path.size(1) - 1, n_pages = Kp.size(0);
    const void *pkt = dev(Kt, BF16, "Kt"), *pvt = dev(a[1], BF16, "Vt");
    void *pk = dev(Kp, BF16, "Kp"), *pv = dev(a[5], BF16, "Vp");
    const auto *pp = (const int32_t *)dev(path, I32, "path_node"), *pn = (const int32_t *)dev(a[3], I32, "n_acc");
    const auto *pt = (const int32_t *)dev(a[6], I32, "page_table"), *pi = (const int32_t *)dev(a[7], I32, "page_indptr"), *pl = (const int32_t *)dev(a[8], I32, "kv_len");
    auto *po = (int32_t *)dev(a[9], I32, "kv_len_out"), *ps = (int32_t *)dev(a[10], I32, "status");
    CALL(specroll_commit_path, (int32_t)B, (int32_t)N, (int32_t)K, (int32_t)Hkv, (int32_t)D, pkt, pvt, pp, pn, pk, pv, n_pages, pt, pi, pl, po, ps);
    return Py_NewRef(Py_None);
}

PyObject *commit_path_layers(PyObject *const *a) {
    // four sequences of tensors, one per layer (lists, tuples, or a tensor whose first dimension is the layer)
    static const char *const names[4] = {"Kt", "Vt", "Kp", "Vp"};
    PyObject *const src[4] = {a[0], a[1], a[4], a[5]};
    std::vector<Ref> seqs;  // (hold the items of a sequence that makes them on the way)
    std::vector<void *> ptrs[4];
    const at::Tensor *first[4] = {};
    Py_ssize_t n = -1;
    for (int i = 0; i < 4; ++i) {
        const Py_ssize_t len = PyObject_Size(src[i]);
        if (len < 0) throw Raised();
        if (n < 0) n = len;
        if (len != n || n == 0) fail("commit_path_layers: one tensor per layer in each list");
        seqs.emplace_back(PySequence_Fast(src[i], "commit_path_layers: one tensor per layer in each list"));
        if (PySequence_Fast_GET_SIZE(seqs.back().o) != n) fail("commit_path_layers: one tensor per layer in each list");
        ptrs[i].reserve((size_t)n);
        for (Py_ssize_t l = 0; l < n; ++l) {
            PyObject *o = PySequence_Fast_GET_ITEM(seqs.back().o, l);
            const at::Tensor &t = i < 2 ? need(o, names[i], 4) : need(o, names[i]);
            if (l == 0) first[i] = &t;
            if (i < 2 && t.sizes() != first[0]->sizes()) fail("commit_path_layers: tree K/V shapes differ between layers");
            if (i >= 2 && t.sizes() != first[2]->sizes()) fail("commit_path_layers: page pools differ between layers");
            ptrs[i].push_back(dev(t, BF16, names[i]));
        }
    }
    const at::Tensor &path = need(a[2], "path_node");
    const int64_t B = first[0]->size(0), N = first[0]->size(1), Hkv = first[0]->size(2), D = first[0]->size(3), K = path.size(1) - 1;
    const auto *pp = (const int32_t *)dev(path, I32, "path_node"), *pn = (const int32_t *)dev(a[3], I32, "n_acc");
    const auto *pt = (const int32_t *)dev(a[6], I32, "page_table"), *pi = (const int32_t *)dev(a[7], I32, "page_indptr"), *pl = (const int32_t *)dev(a[8], I32, "kv_len");
    auto *po = (int32_t *)dev(a[9], I32, "kv_len_out"), *ps = (int32_t *)dev(a[10], I32, "status");
    CALL(specroll_commit_path_layers, (int32_t)B, (int32_t)N, (int32_t)K, (int32_t)Hkv, (int32_t)D, (int32_t)n, ptrs[0].data(), ptrs[1].data(), pp, pn,
         ptrs[2].data(), ptrs[3].data(), first[2]->size(0), pt, pi, pl, po, ps);
    return Py_NewRef(Py_None);
}

at::Tensor gather_hidden_t(const at::Tensor &hidden, const at::Tensor *node, PyObject *out) {
    const int64_t B = hidden.size(0), N = hidden.size(1), d = hidden.size(2);
    const at::Tensor o = out && out != Py_None ? *tensor(out, "h_next") : alloc({B, d}, BF16, hidden);
    const void *ph = dev(hidden, BF16, "hidden");
    const auto *pn = (const int32_t *)dev(node, I32, "term_node");
    void *po = dev(o, BF16, "h_next");
    CALL(specroll_gather_hidden, (int32_t)B, (int32_t)N, (int32_t)d, ph, pn, po);
    return o;
}
PyObject *gather_hidden(PyObject *const *a) {
    return THPVariable_Wrap(gather_hidden_t(need(a[0], "hidden", 3), tensor(a[1], "term_node"), a[2]));
}

// ------------------------------------------------------------------------------ verification

// The arguments that every form shares, and its outputs.
struct VerifyArgs {
    int64_t B, N, K, k, V;
    const int32_t *tree_tok, *cand_id;
    const uint8_t *tree_cand;
    const float *cand_logit, *u_acc, *u_fin;
    VerifyArgs(const char *what, int64_t B_, int64_t N_, int64_t V_, const HostI32 &parent, PyObject *const *a, bool flat = false)
        : B(B_), N(N_), V(V_) {
        // a: tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin
        const at::Tensor &tok = need(a[0], "tree_tok"), &id = need(a[2], "cand_id", 3), &ua = need(a[4], "u_acc");
        K = id.size(1);
        k = id.size(2);
        // flat: the arrays of any shape that holds enough (verification from hidden states)
        if (flat ? parent.size() < N || tok.numel() < B * N || ua.numel() < B * N
                 : parent.size() != N || !shape(tok, {B, N}) || !shape(ua, {B, N}))
            fail("%s: inconsistent shapes", what);
        tree_tok = (const int32_t *)dev(tok, I32, "tree_tok");
        tree_cand = (const uint8_t *)dev(a[1], U8, "tree_cand");
        cand_id = (const int32_t *)dev(id, I32, "cand_id");
        cand_logit = (const float *)dev(a[3], F32, "cand_logit");
        u_acc = (const float *)dev(ua, F32, "u_acc");
        u_fin = (const float *)dev(a[5], F32, "u_fin");
    }
};
struct VerifyOut {
    int32_t *n_acc, *path_node, *out_tok, *term_node, *term_kind;
    float *row_max, *row_sum, *min_margin;
    VerifyOut(Out &o, const VerifyArgs &v, const at::Tensor &like, bool rows = true) {
        n_acc = (int32_t *)o.get("n_acc", {v.B}, I32, like);
        path_node = (int32_t *)o.get("path_node", {v.B, v.K + 1}, I32, like);
        out_tok = (int32_t *)o.get("out_tok", {v.B, v.K + 1}, I32, like);
        term_node = (int32_t *)o.get("term_node", {v.B}, I32, like);
        term_kind = (int32_t *)o.get("term_kind", {v.B}, I32, like);
        if (rows) {
            row_max = (float *)o.get("row_max", {v.B, v.N}, F32, like);
            row_sum = (float *)o.get("row_sum", {v.B, v.N}, F32, like);
        }
        min_margin = (float *)o.get("min_margin", {v.B}, F32, like, true);
    }
};

PyObject *verify(PyObject *const *a) {
    // logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature, workspace, out, flags
    HostI32 parent(a[1], "parent");
    const at::Tensor &lg = need(a[0], "logits", 3);
    const VerifyArgs v("verify", lg.size(0), lg.size(1), lg.size(2), parent, a + 2);
    const specroll_verify_desc D = {(int32_t)v.B, (int32_t)v.N, (int32_t)v.K, (int32_t)v.k, (int32_t)v.V, number(a[8]), (int32_t)integer(a[11])};
    Out out(a[10]);
    const VerifyOut o(out, v, lg);
    const at::Tensor ws = workspace(a[9], lib.specroll_verify_workspace_bytes(&D), lg);
    const void *pl = dev(lg, BF16, "logits");
    CALL(specroll_verify, &D, pl, parent.data(), v.tree_tok, v.tree_cand, v.cand_id, v.cand_logit, v.u_acc, v.u_fin, o.n_acc, o.path_node, o.out_tok,
         o.term_node, o.term_kind, o.row_max, o.row_sum, o.min_margin, ptr(ws), bytes_of(ws));
    return out.release();
}

PyObject *verify_static(PyObject *const *a) {
    // logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature, out
    HostI32 parent(a[1], "parent");
    const at::Tensor &lg = need(a[0], "logits", 3);
    const VerifyArgs v("verify_static", lg.size(0), lg.size(1), lg.size(2), parent, a + 2);
    const specroll_verify_desc D = {(int32_t)v.B, (int32_t)v.N, (int32_t)v.K, (int32_t)v.k, (int32_t)v.V, number(a[8]), 0};
    Out out(a[9]);
    const VerifyOut o(out, v, lg);
    const void *pl = dev(lg, BF16, "logits");
    CALL(specroll_verify_static, &D, pl, parent.data(), v.tree_tok, v.tree_cand, v.cand_id, v.cand_logit, v.u_acc, v.u_fin, o.n_acc, o.path_node,
         o.out_tok, o.term_node, o.term_kind, o.row_max, o.row_sum, o.min_margin);
    return out.release();
}

PyObject *verify_nucleus(PyObject *const *a) {
    // logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, top_p, temperature, workspace, out, flags
    HostI32 parent(a[1], "parent");
    const at::Tensor &lg = need(a[0], "logits", 3);
    const VerifyArgs v("verify_nucleus", lg.size(0), lg.size(1), lg.size(2), parent, a + 2);
    const specroll_verify_desc D = {(int32_t)v.B, (int32_t)v.N, (int32_t)v.K, (int32_t)v.k, (int32_t)v.V, number(a[9]), (int32_t)integer(a[12])};
    Out out(a[11]);
    const VerifyOut o(out, v, lg);
    auto *thr = (float *)out.get("nucleus_thr", {v.B, v.N}, F32, lg, true);
    auto *sum = (float *)out.get("nucleus_sum", {v.B, v.N}, F32, lg, true);
    const at::Tensor ws = workspace(a[10], lib.specroll_verify_nucleus_workspace_bytes(&D), lg);
    const void *pl = dev(lg, BF16, "logits");
    CALL(specroll_verify_nucleus, &D, number(a[8]), pl, parent.data(), v.tree_tok, v.tree_cand, v.cand_id, v.cand_logit, v.u_acc, v.u_fin, o.n_acc,
         o.path_node, o.out_tok, o.term_node, o.term_kind, o.row_max, o.row_sum, o.min_margin, thr, sum, ptr(ws), bytes_of(ws));
    return out.release();
}

void target_head_stats_into(const at::Tensor &H, const at::Tensor &W, const at::Tensor *want, float T, PyObject *ws_, Out &out) {
    const int64_t R = H.size(0), d = H.size(1), V = W.size(0), kw = want ? want->size(1) : 0;
    auto *rm = (float *)out.get("row_max", {R}, F32, H);
    auto *rs = (float *)out.get("row_sum", {R}, F32, H);
    void *wl = out.get("want_logit", {R, kw}, BF16, H);
    const size_t need_ws = lib.specroll_target_head_stats_workspace_bytes((int32_t)R, (int32_t)d, (int32_t)V);
    if (need_ws == 0) fail("target_head_stats: invalid shape");
    const at::Tensor ws = workspace(ws_, need_ws, H);
    const void *ph = dev(H, BF16, "H"), *pw = dev(W, BF16, "W");
    const auto *pi = kw ? (const int32_t *)dev(want, I32, "want_id") : nullptr;
    CALL(specroll_target_head_stats, (int32_t)R, (int32_t)d, (int32_t)V, T, ph, pw, pi, (int32_t)kw, rm, rs, kw ? wl : nullptr, ptr(ws), bytes_of(ws));
}
PyObject *target_head_stats(PyObject *const *a) {  // H, W, want_id, temperature, workspace
    const at::Tensor *want = tensor(a[2], "want_id");
    Out out(nullptr);
    target_head_stats_into(need(a[0], "H", 2), need(a[1], "W", 2), want, number(a[3]), a[4], out);
    return out.release();
}

at::Tensor target_head_rows_t(const at::Tensor &H, const at::Tensor &W, PyObject *out) {
    const int64_t R = H.size(0), d = H.size(1), V = W.size(0);
    const at::Tensor o = out && out != Py_None ? *tensor(out, "logits") : alloc({R, V}, BF16, H);
    const at::Tensor status = alloc({1}, I32, H);  // (the call clears it)
    const void *ph = dev(H, BF16, "H"), *pw = dev(W, BF16, "W");
    void *po = dev(o, BF16, "logits");
    CALL(specroll_target_head_rows, (int32_t)R, (int32_t)d, (int32_t)V, ph, pw, po, (int32_t *)ptr(status));
    return o;
}
PyObject *target_head_rows(PyObject *const *a) {
    return THPVariable_Wrap(target_head_rows_t(need(a[0], "H", 2), need(a[1], "W", 2), a[2]));
}

PyObject *verify_fused(PyObject *const *a) {
    // hidden, W, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature
    HostI32 parent(a[2], "parent");
    const at::Tensor &hidden = need(a[0], "hidden", 3), &W = need(a[1], "W", 2);
    const int64_t B = hidden.size(0), N = hidden.size(1), d = hidden.size(2);
    const VerifyArgs v("verify_fused", B, N, W.size(0), parent, a + 3, true);
    const float T = number(a[9]);
    const specroll_verify_desc D = {(int32_t)B, (int32_t)N, (int32_t)v.K, (int32_t)v.k, (int32_t)v.V, T, 0};
    const at::Tensor want = alloc({B * N, v.k}, I32, hidden);
    CALL(specroll_verify_want_ids, &D, parent.data(), v.cand_id, (int32_t *)ptr(want));
    const at::Tensor row_max = alloc({B, N}, F32, hidden), row_sum = alloc({B, N}, F32, hidden);
    const at::Tensor want_logit = alloc({B * N, v.k}, BF16, hidden);
    const size_t need_ws = lib.specroll_target_head_stats_workspace_bytes((int32_t)(B * N), (int32_t)d, (int32_t)v.V);
    if (need_ws == 0) fail("target_head_stats: invalid shape");
    const at::Tensor ws_head = alloc_bytes(need_ws, hidden);
    const void *ph = dev(hidden, BF16, "H"), *pw = dev(W, BF16, "W");
    const at::Tensor tiles = alloc_bytes(lib.specroll_target_head_tile_mass_bytes((int32_t)(B * N), (int32_t)v.V), hidden);
    CALL(specroll_target_head_stats_tiles, (int32_t)(B * N), (int32_t)d, (int32_t)v.V, T, ph, pw, (const int32_t *)ptr(want), (int32_t)v.k,
         (float *)ptr(row_max), (float *)ptr(row_sum), ptr(want_logit), ptr(tiles), ptr(ws_head), bytes_of(ws_head));
    Out out(nullptr);
    const VerifyOut o(out, v, hidden, false);
    out.put("row_max", row_max);
    out.put("row_sum", row_sum);
    CALL(specroll_verify_hidden, &D, (int32_t)d, ph, pw, ptr(want_logit), ptr(tiles), (const float *)ptr(row_max), (const float *)ptr(row_sum),
         parent.data(), v.tree_tok, v.tree_cand, v.cand_id, v.cand_logit, v.u_acc, v.u_fin, o.n_acc, o.path_node, o.out_tok, o.term_node,
         o.term_kind, o.min_margin);
    return out.release();
}

// ------------------------------------------------------------------------------ feedback, sketches, gate

PyObject *reflex_feedback(PyObject *const *a) {
    // logits, rec_row, row_max, row_sum, cand_id, cand_logit, y_star, W, rho, rec_mem, m, k_support, temperature, eps, workspace, severity_min, want_e
    const at::Tensor *lgp = tensor(a[0], "logits");
    const at::Tensor &ci = need(a[4], "cand_id", 2), &W = need(a[7], "W", 2);
    if (!lgp || lgp->dim() < 1) fail("logits must be a CUDA tensor");
    const int64_t R = ci.size(0), k = ci.size(1), d = W.size(1), V = lgp->size(-1);
    const bool weighted = a[15] != Py_None, want_e = PyObject_IsTrue(a[16]) == 1;
    const specroll_feedback_desc D = {(int32_t)R, (int32_t)k, (int32_t)integer(a[11]), (int32_t)d, (int32_t)V, number(a[12]), number(a[13]),
                                      weighted ? SPECROLL_FEEDBACK_SEVERITY : 0, weighted ? number(a[15]) : 0.f};
    Out out(nullptr);
    auto *dd = (float *)out.get("d_dist", {R}, F32, *lgp);
    auto *dc = (float *)out.get("d_cov", {R}, F32, *lgp);
    auto *tv = (float *)out.get("tv", {R}, F32, *lgp);
    auto *sv = (float *)out.get("severity", {R}, F32, *lgp);
    auto *e = want_e ? (float *)out.get("e", {R, d}, F32, *lgp) : nullptr;
    const size_t need_ws = lib.specroll_reflex_feedback_workspace_bytes(&D);
    if (need_ws == 0) fail("reflex_feedback: invalid descriptor");
    const at::Tensor ws = workspace(a[14], need_ws, *lgp);
    const void *pl = dev(lgp, BF16, "logits"), *pw = dev(W, BF16, "W");
    const auto *rr = (const int32_t *)dev(a[1], I32, "rec_row"), *ys = (const int32_t *)dev(a[6], I32, "y_star"), *rmem = (const int32_t *)dev(a[9], I32, "rec_mem");
    const auto *rm = (const float *)dev(a[2], F32, "row_max"), *rs = (const float *)dev(a[3], F32, "row_sum"), *cl = (const float *)dev(a[5], F32, "cand_logit");
    const auto *id = (const int32_t *)dev(ci, I32, "cand_id");
    const auto *rho = (const float *)dev(a[8], F32, "rho");
    auto *m = (float *)dev(a[10], F32, "m");
    CALL(specroll_reflex_feedback_ex, &D, pl, rr, rm, rs, id, cl, ys, pw, rho, rmem, m, dd, dc, tv, sv, e, ptr(ws), bytes_of(ws));
    return out.release();
}

PyObject *reflex_sketch(PyObject *const *a) {  // X, Pi, rows
    const at::Tensor *X = tensor(a[0], "X"), *rows = tensor(a[2], "rows");
    const at::Tensor &Pi = need(a[1], "Pi", 2);
    if (!X || X->dim() < 1) fail("X must be a CUDA tensor");
    const int64_t rank = Pi.size(0), d = Pi.size(1), R = rows ? rows->size(0) : X->size(0);
    const at::Tensor out = alloc({R, rank}, F32, *X);
    const auto *px = (const float *)dev(X, F32, "X"), *pp = (const float *)dev(Pi, F32, "Pi");
    const auto *pr = (const int32_t *)dev(rows, I32, "rows");
    CALL(specroll_reflex_sketch, (int32_t)R, (int32_t)d, (int32_t)rank, px, pr, pp, (float *)dev(out, F32, "sketch"));
    return THPVariable_Wrap(out);
}

PyObject *reflex_gate(PyObject *const *a) {
    // s, xi, slot, keep, n, mean, M2, n_fb, m, horizon, n_align_min, n_fb_min, alpha_lo, alpha_hi, z_delta, mem_eps
    const at::Tensor &s = need(a[0], "s", 2), &m = need(a[8], "m", 2), &am = need(a[10], "n_align_min");
    const int64_t R = s.size(0), S = m.size(0);
    const specroll_gate_desc D = {(int32_t)R, (int32_t)S, (int32_t)m.size(1), (int32_t)s.size(1), (int32_t)am.size(0), number(a[14]), number(a[15]), 0};
    Out out(nullptr);
    const at::Tensor al = alloc({R > 0 ? R : 1}, F32, m);
    out.put("a", R > 0 ? al : al.slice(0, 0, 0));
    auto *rel = (float *)out.get("rel", {S}, F32, m);
    auto *alpha = (float *)out.get("alpha", {S}, F32, m);
    const auto *ps = (const float *)dev(s, F32, "s"), *px = (const float *)dev(a[1], F32, "xi"), *pm = (const float *)dev(m, F32, "m");
    const auto *slot = (const int32_t *)dev(a[2], I32, "slot"), *hor = (const int32_t *)dev(a[9], I32, "horizon");
    const auto *keep = (const uint8_t *)dev(a[3], U8, "keep");
    auto *n = (int32_t *)dev(a[4], I32, "n"), *nf = (int32_t *)dev(a[7], I32, "n_fb");
    auto *mean = (float *)dev(a[5], F32, "mean"), *M2 = (float *)dev(a[6], F32, "M2");
    const auto *pa = (const int32_t *)dev(am, I32, "n_align_min"), *pf = (const int32_t *)dev(a[11], I32, "n_fb_min");
    const auto *lo = (const float *)dev(a[12], F32, "alpha_lo"), *hi = (const float *)dev(a[13], F32, "alpha_hi");
    CALL(specroll_reflex_gate, &D, ps, px, slot, keep, n, mean, M2, nf, pm, hor, pa, pf, lo, hi, (float *)ptr(al), rel, alpha);
    return out.release();
}

// ------------------------------------------------------------------------------ module

// attach(SpecrollError, _host_i32, {entry name: address})
PyObject *attach(PyObject *const *a) {
    auto addr = [&](const char *name) -> void * {
        PyObject *o = PyDict_GetItemString(a[2], name);
        if (!o) fail("the library has no %s", name);
        return PyLong_AsVoidPtr(o);
    };
#define X(name) lib.name = reinterpret_cast<decltype(&::name)>(addr(#name));
    SPECROLL_ENTRIES(X)
#undef X
    Py_XSETREF(g_error, Py_NewRef(a[0]));
    Py_XSETREF(g_host_i32, Py_NewRef(a[1]));
    return Py_NewRef(Py_None);
}
PyObject *set_alloc(PyObject *const *a) {
    Py_XSETREF(g_alloc, a[0] == Py_None ? nullptr : Py_NewRef(a[0]));
    return Py_NewRef(Py_None);
}

template <PyObject *(*F)(PyObject *const *), int NARGS>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != NARGS) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", NARGS, n);
        return nullptr;
    }
    if (!lib.specroll_strerror && F != &attach && F != &set_alloc) {
        PyErr_SetString(PyExc_RuntimeError, "attach() has not been called");
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Raised &) {
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
#define METHOD(name, nargs) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<&name, nargs>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(attach, 3),
                         METHOD(set_alloc, 1),
                         METHOD(propose, 19),
                         METHOD(tree_draw, 6),
                         METHOD(tree_attn, 14),
                         METHOD(tree_attn_paged, 16),
                         METHOD(commit_path, 11),
                         METHOD(commit_path_layers, 11),
                         METHOD(gather_hidden, 3),
                         METHOD(verify, 12),
                         METHOD(verify_static, 10),
                         METHOD(verify_nucleus, 13),
                         METHOD(verify_fused, 10),
                         METHOD(target_head_stats, 5),
                         METHOD(target_head_rows, 3),
                         METHOD(reflex_feedback, 17),
                         METHOD(reflex_sketch, 3),
                         METHOD(reflex_gate, 16),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of the binding.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
