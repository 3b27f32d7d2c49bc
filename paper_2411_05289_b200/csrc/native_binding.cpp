// CPython binding of the entry points a decoding iteration calls: argument checks, descriptors and
// output tensors for include/spechub.h.  (A call costs 5-8 us of host time, most of it the output tensors
// and the launches; the same marshalling in Python cost 20-30 us, more than the kernels of a small batch.)
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <initializer_list>
#include <string>

#include "spechub.h"

namespace {

using at::Tensor;

PyObject *g_error = nullptr;  // the package's SpecHubError

struct PyFail {};             // a Python exception is set
[[noreturn]] void value_error(const char *msg) {
    PyErr_SetString(PyExc_ValueError, msg);
    throw PyFail{};
}
[[noreturn]] void fail() { throw PyFail{}; }

struct Ref {  // an owned reference
    PyObject *o;
    explicit Ref(PyObject *p) : o(p) {}
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
    ~Ref() { Py_XDECREF(o); }
    PyObject *release() { PyObject *p = o; o = nullptr; return p; }
};

struct Names {  // interned attribute and key names
    PyObject *levels, *child, *node_kind, *k, *cuda_stream, *record_stream;
    PyObject *tokens, *hub, *prob, *status, *stats;
    PyObject *accept_idx, *token, *beta, *rate, *n_accepted, *n_emitted, *path_nodes, *path_tokens;
    PyObject *spechub, *rrs, *rrsw;
} N;

// Without the interpreter's lock: other Python threads run while a call waits for a place in a full launch queue or for
// memory.  (Among them may be the callback that the queue waits for.)
struct Unlocked {
    PyThreadState *state = PyEval_SaveThread();
    Unlocked() = default;
    Unlocked(const Unlocked &) = delete;
    Unlocked &operator=(const Unlocked &) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};

void check(int code) {
    if (code == SPECHUB_OK) return;
    Ref e(PyObject_CallFunction(g_error, "is", code, spechub_status_string(code)));
    if (e.o) PyErr_SetObject(g_error, e.o);
    fail();
}

const Tensor &tensor(PyObject *o, const char *msg) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, msg);
        fail();
    }
    return THPVariable_Unpack(o);
}

Tensor make(at::IntArrayRef sizes, at::ScalarType t, const at::Device &dev) {
    if (dev.is_cuda()) return at::detail::empty_cuda(sizes, t, dev, c10::nullopt);
    return at::empty(sizes, at::TensorOptions().dtype(t).device(dev));
}
void put(PyObject *dict, PyObject *key, const Tensor &t) {
    Ref v(THPVariable_Wrap(t));
    if (!v.o || PyDict_SetItem(dict, key, v.o) < 0) fail();
}

struct TreeView {
    long levels, k;
    Ref child, node_kind;
    explicit TreeView(PyObject *tree)
        : child(PyObject_GetAttr(tree, N.child)), node_kind(PyObject_GetAttr(tree, N.node_kind)) {
        Ref l(PyObject_GetAttr(tree, N.levels)), kk(PyObject_GetAttr(tree, N.k));
        if (!child.o || !node_kind.o || !l.o || !kk.o) fail();
        levels = PyLong_AsLong(l.o);
        k = PyLong_AsLong(kk.o);
        if (PyErr_Occurred()) fail();
    }
};

void need_k2(const TreeView &t) {
    if (t.k != 2) value_error("SpecHub takes exactly two drafts per node");
}

struct Desc {
    spechub_desc d;
    Tensor temperature;  // keeps a converted temperature vector alive until the launch is enqueued
    int64_t B, Nn, V;
    at::Device dev{at::kCPU};

    Desc(const Tensor &x, const TreeView &tree, PyObject *temp, unsigned flags) {
        if (x.dim() != 3 || x.stride(2) != 1)
            value_error("logits must be [batch][nodes][vocab] with a contiguous vocabulary axis");
        if (!x.is_cuda()) value_error("logits must live on a CUDA device");
        const auto st = x.scalar_type();
        if (st != at::kFloat && st != at::kBFloat16) value_error("logits must be float32 or bfloat16");
        B = x.size(0); Nn = x.size(1); V = x.size(2);
        dev = x.device();
        d = {};
        d.struct_size = sizeof(spechub_desc);
        d.version = SPECHUB_ABI_VERSION;
        d.batch = static_cast<int32_t>(B); d.nodes = static_cast<int32_t>(Nn); d.vocab = static_cast<int32_t>(V);
        d.k = static_cast<int32_t>(tree.k);
        d.dtype = st == at::kFloat ? SPECHUB_F32 : SPECHUB_BF16;
        d.levels = static_cast<int32_t>(tree.levels);
        const int64_t s0 = x.stride(0), s1 = x.stride(1);
        d.stride_seq = B > 1 ? s0 : std::max(s0, (Nn - 1) * s1 + V);
        d.stride_node = Nn > 1 ? s1 : std::max(s1, V);
        if (THPVariable_Check(temp)) {
            temperature = THPVariable_Unpack(temp);
            {
                Unlocked u;
                if (temperature.device() != dev || temperature.scalar_type() != at::kFloat)
                    temperature = temperature.to(dev, at::kFloat);
                temperature = temperature.contiguous();
            }
            if (temperature.dim() != 1 || temperature.size(0) != B) value_error("temperature tensor must be [batch]");
            d.temperature = 1.0f;
            d.temperature_per_seq = temperature.const_data_ptr<float>();
        } else {
            const Ref f(PyNumber_Float(temp));   // whatever float() takes
            if (!f.o) fail();
            d.temperature = static_cast<float>(PyFloat_AS_DOUBLE(f.o));
        }
        if (tree.child.o != Py_None) {
            const Tensor &c = tensor(tree.child.o, "child must be a tensor");
            if (c.scalar_type() != at::kInt || c.dim() != 2 || c.size(0) != Nn || c.size(1) != tree.k || !c.is_contiguous())
                value_error("child must be a contiguous int32 [nodes][k] tensor");
            d.child = static_cast<const int32_t *>(c.const_data_ptr());
        }
        if (tree.node_kind.o != Py_None) {
            const Tensor &kd = tensor(tree.node_kind.o, "node_kind must be a tensor");
            if (kd.scalar_type() != at::kByte || kd.dim() != 1 || kd.size(0) != Nn)
                value_error("node_kind must be a uint8 [nodes] tensor");
            d.node_kind = static_cast<const uint8_t *>(kd.const_data_ptr());
        }
        d.flags = flags;  // SPECHUB_FLAG_SPLIT_n has the value n
    }
};

const float *uniforms_of(PyObject *o, const Desc &d) {
    const Tensor &u = tensor(o, "uniforms must be a tensor");
    if (u.scalar_type() != at::kFloat || u.dim() != 3 || u.size(0) != d.B || u.size(1) != d.Nn ||
        u.size(2) != 2 * d.d.k + 1 || !u.is_contiguous() || u.device() != d.dev)
        value_error("uniforms must be a contiguous float32 [batch][nodes][2k+1] tensor on the logits' device");
    return static_cast<const float *>(u.const_data_ptr());
}

void same_layout(const Tensor &a, const Tensor &b) {
    if (a.sizes() != b.sizes() || a.scalar_type() != b.scalar_type() || a.strides() != b.strides() || a.device() != b.device())
        value_error("target and draft logits must share shape, dtype, strides and device");
}

const int32_t *tokens_of(PyObject *o, const Desc &d, const char *msg) {
    const Tensor &t = tensor(o, msg);
    if (t.scalar_type() != at::kInt || t.dim() != 3 || t.size(0) != d.B || t.size(1) != d.Nn || t.size(2) != d.d.k ||
        !t.is_contiguous() || t.device() != d.dev)
        value_error(msg);
    return static_cast<const int32_t *>(t.const_data_ptr());
}

const void *stats_of(PyObject *o, const Desc &d) {
    const char *msg = "stats must be the tensor a *_draft_sample_stats call returned for this shape";
    if (o == Py_None || !THPVariable_Check(o)) value_error(msg);
    const Tensor &s = THPVariable_Unpack(o);
    if (s.scalar_type() != at::kInt || !s.is_contiguous() || s.device() != d.dev ||
        static_cast<size_t>(s.numel()) * 4 < spechub_draft_stats_bytes(&d.d))
        value_error(msg);
    return s.const_data_ptr();
}

Tensor make_stats(const Desc &d) {
    const size_t n = spechub_draft_stats_bytes(&d.d);
    return make({static_cast<int64_t>(std::max<size_t>(n, 16) / 4)}, at::kInt, d.dev);
}

void *stream_of(PyObject *stream) {
    if (stream == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    Ref p(PyObject_GetAttr(stream, N.cuda_stream));
    if (!p.o) fail();
    void *s = PyLong_AsVoidPtr(p.o);
    if (PyErr_Occurred()) fail();
    return s;
}

// Tensors that may be freed when the Python call returns, while the kernels may still be queued.  On the current
// stream torch's allocator orders the reuse after them; on any other stream it has to be told.
void hold(PyObject *stream, const Tensor &t) {
    if (stream == Py_None || !t.defined()) return;
    Ref w(THPVariable_Wrap(t));
    if (!w.o) fail();
    Ref r(PyObject_CallMethodOneArg(w.o, N.record_stream, stream));
    if (!r.o) fail();
}
void hold(PyObject *stream, PyObject *t) {
    if (stream == Py_None || t == Py_None) return;
    Ref r(PyObject_CallMethodOneArg(t, N.record_stream, stream));
    if (!r.o) fail();
}
void hold_values(PyObject *stream, PyObject *mapping) {
    if (stream == Py_None) return;
    Ref vals(PyMapping_Values(mapping));
    if (!vals.o) fail();
    for (Py_ssize_t i = 0; i < PyList_GET_SIZE(vals.o); ++i) hold(stream, PyList_GET_ITEM(vals.o, i));
}

// ---- outputs of a verify call --------------------------------------------------------------------
struct NewOutputs {
    Tensor accept_idx, token, hub, beta, rate, status, n_accepted, n_emitted, path_nodes, path_tokens;
    void allocate(const Desc &d, int64_t levels, int64_t k, bool probabilities, spechub_node_out &no, spechub_seq_out &so) {
        for (Tensor *t : {&accept_idx, &token, &hub, &status}) *t = make({d.B, d.Nn}, at::kInt, d.dev);
        beta = make({d.B, d.Nn, k}, at::kFloat, d.dev);
        rate = make({d.B, d.Nn, k + 1}, at::kFloat, d.dev);
        for (Tensor *t : {&n_accepted, &n_emitted}) *t = make({d.B}, at::kInt, d.dev);
        for (Tensor *t : {&path_nodes, &path_tokens}) *t = make({d.B, levels}, at::kInt, d.dev);
        no = {};
        no.accept_idx = static_cast<int32_t *>(accept_idx.data_ptr());
        no.token = static_cast<int32_t *>(token.data_ptr());
        no.hub = static_cast<int32_t *>(hub.data_ptr());
        if (probabilities) {
            no.beta = static_cast<float *>(beta.data_ptr());
            no.rate = static_cast<float *>(rate.data_ptr());
        }
        no.status = static_cast<uint32_t *>(status.data_ptr());
        so.n_accepted = static_cast<int32_t *>(n_accepted.data_ptr());
        so.n_emitted = static_cast<int32_t *>(n_emitted.data_ptr());
        so.path_nodes = static_cast<int32_t *>(path_nodes.data_ptr());
        so.path_tokens = static_cast<int32_t *>(path_tokens.data_ptr());
    }
    PyObject *dict() const {
        Ref o(PyDict_New());
        if (!o.o) fail();
        put(o.o, N.accept_idx, accept_idx);
        put(o.o, N.token, token);
        put(o.o, N.hub, hub);
        put(o.o, N.beta, beta);
        put(o.o, N.rate, rate);
        put(o.o, N.status, status);
        put(o.o, N.n_accepted, n_accepted);
        put(o.o, N.n_emitted, n_emitted);
        put(o.o, N.path_nodes, path_nodes);
        put(o.o, N.path_tokens, path_tokens);
        return o.release();
    }
};

template <class T>
T *field(PyObject *out, PyObject *key) {
    Ref v(PyObject_GetItem(out, key));
    if (!v.o) fail();
    return static_cast<T *>(tensor(v.o, "output buffers must be tensors").data_ptr());
}
void output_pointers(PyObject *out, bool probabilities, spechub_node_out &no, spechub_seq_out &so) {
    no = {};
    no.accept_idx = field<int32_t>(out, N.accept_idx);
    no.token = field<int32_t>(out, N.token);
    no.hub = field<int32_t>(out, N.hub);
    if (probabilities) {
        no.beta = field<float>(out, N.beta);
        no.rate = field<float>(out, N.rate);
    }
    no.status = field<uint32_t>(out, N.status);
    so.n_accepted = field<int32_t>(out, N.n_accepted);
    so.n_emitted = field<int32_t>(out, N.n_emitted);
    so.path_nodes = field<int32_t>(out, N.path_nodes);
    so.path_tokens = field<int32_t>(out, N.path_tokens);
}

bool truth(PyObject *o) {
    const int t = PyObject_IsTrue(o);
    if (t < 0) fail();
    return t != 0;
}

}  // namespace

namespace {

enum { kSpecHub = 0, kRRS = 1, kRRSw = 2 };

unsigned flags_of(PyObject *o) {
    const unsigned long f = PyLong_AsUnsignedLong(o);
    if (PyErr_Occurred()) fail();
    return static_cast<unsigned>(f);
}
int method_of(PyObject *o) {
    const long m = PyLong_AsLong(o);
    if (PyErr_Occurred()) fail();
    return static_cast<int>(m);
}
void need_args(Py_ssize_t n, Py_ssize_t want) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
        fail();
    }
}

// (method, draft_logits, uniforms, tree, temperature, stream, flags, with_stats)
PyObject *draft_impl(PyObject *const *a, Py_ssize_t n) {
    need_args(n, 8);
    const int method = method_of(a[0]);
    const Tensor &x = tensor(a[1], "draft_logits must be a tensor");
    const TreeView tree(a[3]);
    if (method == kSpecHub) need_k2(tree);
    const Desc d(x, tree, a[4], flags_of(a[6]));
    const float *un = uniforms_of(a[2], d);
    const bool with_stats = truth(a[7]);
    void *s = stream_of(a[5]);
    Tensor tokens, status, hub, prob, stats;
    const void *xp = x.const_data_ptr();
    int rc;
    {
        Unlocked u;
        tokens = make({d.B, d.Nn, tree.k}, at::kInt, d.dev);
        status = make({d.B, d.Nn}, at::kInt, d.dev);
        if (with_stats) stats = make_stats(d);
        void *stp = with_stats ? stats.data_ptr() : nullptr;
        int32_t *tp = static_cast<int32_t *>(tokens.data_ptr());
        uint32_t *sp = static_cast<uint32_t *>(status.data_ptr());
        if (method == kSpecHub) {
            hub = make({d.B, d.Nn}, at::kInt, d.dev);
            prob = make({d.B, d.Nn, 2}, at::kFloat, d.dev);
            int32_t *hp = static_cast<int32_t *>(hub.data_ptr());
            float *pp = static_cast<float *>(prob.data_ptr());
            rc = with_stats ? spechub_draft_sample_stats(&d.d, xp, un, tp, hp, pp, sp, stp, s)
                            : spechub_draft_sample(&d.d, xp, un, tp, hp, pp, sp, s);
        } else {
            const int wo = method == kRRSw;
            rc = with_stats ? rrs_draft_sample_stats(&d.d, xp, un, wo, tp, sp, stp, s)
                            : rrs_draft_sample(&d.d, xp, un, wo, tp, sp, s);
        }
    }
    check(rc);
    Ref out(PyDict_New());
    if (!out.o) fail();
    put(out.o, N.tokens, tokens);
    if (method == kSpecHub) {
        put(out.o, N.hub, hub);
        put(out.o, N.prob, prob);
    }
    put(out.o, N.status, status);
    if (with_stats) put(out.o, N.stats, stats);
    hold(a[5], d.temperature);
    hold_values(a[5], out.o);
    return out.release();
}

Tensor make_workspace(const Desc &d, size_t &bytes) {
    bytes = spechub_workspace_bytes(&d.d);
    return bytes ? make({static_cast<int64_t>(bytes)}, at::kByte, d.dev) : Tensor();
}

// (method, target_logits, draft_logits, stats, draft_tokens, uniforms, tree, temperature, stream, out,
//  probabilities, flags, with_stats)
PyObject *verify_impl(PyObject *const *a, Py_ssize_t n) {
    need_args(n, 13);
    const int method = method_of(a[0]);
    const Tensor &tl = tensor(a[1], "target_logits must be a tensor"), &dl = tensor(a[2], "draft_logits must be a tensor");
    same_layout(tl, dl);
    const TreeView tree(a[6]);
    const Desc d(tl, tree, a[7], flags_of(a[11]));
    if (method == kSpecHub) need_k2(tree);
    const float *un = uniforms_of(a[5], d);
    const int32_t *tok = tokens_of(a[4], d, "draft_tokens must be a contiguous int32 [batch][nodes][k] tensor");
    Ref out(a[9] == Py_None ? nullptr : Py_NewRef(a[9]));
    const bool probabilities = truth(a[10]), with_stats = truth(a[12]);
    spechub_node_out no;
    spechub_seq_out so;
    if (out.o) output_pointers(out.o, probabilities, no, so);
    const void *st = with_stats ? stats_of(a[3], d) : nullptr;
    void *s = stream_of(a[8]);
    const void *tp = tl.const_data_ptr(), *dp = dl.const_data_ptr();
    NewOutputs fresh;
    Tensor ws;
    int rc;
    {
        Unlocked u;
        if (!out.o) fresh.allocate(d, tree.levels, tree.k, probabilities, no, so);
        size_t wsb;
        ws = make_workspace(d, wsb);
        void *wp = wsb ? ws.data_ptr() : nullptr;
        if (with_stats)
            rc = method == kSpecHub ? spechub_verify_tree_stats(&d.d, tp, dp, st, tok, un, &no, &so, wp, wsb, s)
                                    : rrs_verify_tree_stats(&d.d, tp, dp, st, tok, un, method == kRRSw, &no, &so, wp, wsb, s);
        else
            rc = method == kSpecHub ? spechub_verify_tree(&d.d, tp, dp, tok, un, &no, &so, wp, wsb, s)
                                    : rrs_verify_tree(&d.d, tp, dp, tok, un, method == kRRSw, &no, &so, wp, wsb, s);
    }
    check(rc);
    if (!out.o) out.o = fresh.dict();
    hold(a[8], d.temperature);
    hold(a[8], ws);
    hold(a[8], a[3]);
    hold_values(a[8], out.o);
    return out.release();
}

// (draft_logits, uniforms, tree, temperature, stream, flags, with_stats)
PyObject *compare_draft_impl(PyObject *const *a, Py_ssize_t n) {
    need_args(n, 7);
    const Tensor &x = tensor(a[0], "draft_logits must be a tensor");
    const TreeView tree(a[2]);
    need_k2(tree);
    const Desc d(x, tree, a[3], flags_of(a[5]));
    const float *un = uniforms_of(a[1], d);
    const bool with_stats = truth(a[6]);
    void *s = stream_of(a[4]);
    Tensor tokens[3], status[3], stats, hub, prob;
    const void *xp = x.const_data_ptr();
    int rc;
    {
        Unlocked u;
        int32_t *tp[3];
        uint32_t *sp[3];
        for (int m = 0; m < 3; ++m) {
            tokens[m] = make({d.B, d.Nn, 2}, at::kInt, d.dev);
            status[m] = make({d.B, d.Nn}, at::kInt, d.dev);
            tp[m] = static_cast<int32_t *>(tokens[m].data_ptr());
            sp[m] = static_cast<uint32_t *>(status[m].data_ptr());
        }
        hub = make({d.B, d.Nn}, at::kInt, d.dev);
        prob = make({d.B, d.Nn, 2}, at::kFloat, d.dev);
        if (with_stats) stats = make_stats(d);
        int32_t *hp = static_cast<int32_t *>(hub.data_ptr());
        float *pp = static_cast<float *>(prob.data_ptr());
        rc = with_stats ? mdsd_compare_draft_sample_stats(&d.d, xp, un, tp, hp, pp, sp, stats.data_ptr(), s)
                        : mdsd_compare_draft_sample(&d.d, xp, un, tp, hp, pp, sp, s);
    }
    check(rc);
    Ref out(PyDict_New());
    if (!out.o) fail();
    PyObject *names[3] = {N.spechub, N.rrs, N.rrsw};
    for (int m = 0; m < 3; ++m) {
        Ref one(PyDict_New());
        if (!one.o) fail();
        put(one.o, N.tokens, tokens[m]);
        if (m == kSpecHub) {
            put(one.o, N.hub, hub);
            put(one.o, N.prob, prob);
        }
        put(one.o, N.status, status[m]);
        hold_values(a[4], one.o);
        if (PyDict_SetItem(out.o, names[m], one.o) < 0) fail();
    }
    if (with_stats) put(out.o, N.stats, stats);
    hold(a[4], d.temperature);
    hold(a[4], stats);
    return out.release();
}

// (target_logits, draft_logits, stats, draft_tokens, uniforms, tree, temperature, stream, out, probabilities,
//  flags, with_stats); draft_tokens and out keyed by method name
PyObject *compare_verify_impl(PyObject *const *a, Py_ssize_t n) {
    need_args(n, 12);
    const Tensor &tl = tensor(a[0], "target_logits must be a tensor"), &dl = tensor(a[1], "draft_logits must be a tensor");
    const TreeView tree(a[5]);
    need_k2(tree);
    same_layout(tl, dl);
    const Desc d(tl, tree, a[6], flags_of(a[10]));
    const float *un = uniforms_of(a[4], d);
    PyObject *names[3] = {N.spechub, N.rrs, N.rrsw};
    const int32_t *tok[3];
    for (int m = 0; m < 3; ++m) {
        Ref t(PyObject_GetItem(a[3], names[m]));
        if (!t.o) fail();
        const std::string msg = std::string("draft_tokens[") + PyUnicode_AsUTF8(names[m]) +
                                "] must be a contiguous int32 [batch][nodes][2] tensor";
        tok[m] = tokens_of(t.o, d, msg.c_str());
    }
    Ref out(a[8] == Py_None ? nullptr : Py_NewRef(a[8]));
    spechub_node_out no[3];
    spechub_seq_out so[3];
    const bool probabilities = truth(a[9]), with_stats = truth(a[11]);
    for (int m = 0; m < 3 && out.o; ++m) {
        Ref one(PyObject_GetItem(out.o, names[m]));
        if (!one.o) fail();
        output_pointers(one.o, probabilities, no[m], so[m]);
    }
    const void *st = with_stats ? stats_of(a[2], d) : nullptr;
    void *s = stream_of(a[7]);
    const void *tp = tl.const_data_ptr(), *dp = dl.const_data_ptr();
    NewOutputs fresh[3];
    Tensor ws;
    int rc;
    {
        Unlocked u;
        for (int m = 0; m < 3 && !out.o; ++m) fresh[m].allocate(d, tree.levels, 2, probabilities, no[m], so[m]);
        size_t wsb;
        ws = make_workspace(d, wsb);
        void *wp = wsb ? ws.data_ptr() : nullptr;
        rc = with_stats ? mdsd_compare_verify_tree_stats(&d.d, tp, dp, st, tok, un, no, so, wp, wsb, s)
                        : mdsd_compare_verify_tree(&d.d, tp, dp, tok, un, no, so, wp, wsb, s);
    }
    check(rc);
    if (!out.o) {
        out.o = PyDict_New();
        if (!out.o) fail();
        for (int m = 0; m < 3; ++m) {
            Ref one(fresh[m].dict());
            if (PyDict_SetItem(out.o, names[m], one.o) < 0) fail();
        }
    }
    hold(a[7], d.temperature);
    hold(a[7], ws);
    hold(a[7], a[2]);
    if (a[7] != Py_None)
        for (int m = 0; m < 3; ++m) {
            Ref one(PyObject_GetItem(out.o, names[m]));
            if (!one.o) fail();
            hold_values(a[7], one.o);
        }
    return out.release();
}

// (target_logits, draft_logits, draft_tokens, uniforms, tree, temperature, stream, out, flags)
PyObject *verify_static_impl(PyObject *const *a, Py_ssize_t n) {
    need_args(n, 9);
    const Tensor &tl = tensor(a[0], "target_logits must be a tensor"), &dl = tensor(a[1], "draft_logits must be a tensor");
    const TreeView tree(a[4]);
    need_k2(tree);
    same_layout(tl, dl);
    const Desc d(tl, tree, a[5], flags_of(a[8]));
    const float *un = uniforms_of(a[3], d);
    const int32_t *tok = tokens_of(a[2], d, "draft_tokens must be a contiguous int32 [batch][nodes][2] tensor");
    Ref out(a[7] == Py_None ? nullptr : Py_NewRef(a[7]));
    spechub_node_out no;
    spechub_seq_out so;
    if (out.o) output_pointers(out.o, true, no, so);
    void *s = stream_of(a[6]);
    const void *tp = tl.const_data_ptr(), *dp = dl.const_data_ptr();
    NewOutputs fresh;
    int rc;
    {
        Unlocked u;
        if (!out.o) fresh.allocate(d, tree.levels, 2, true, no, so);
        rc = spechub_verify_tree_static(&d.d, tp, dp, tok, un, &no, &so, s);
    }
    check(rc);
    if (!out.o) out.o = fresh.dict();
    hold(a[6], d.temperature);
    hold_values(a[6], out.o);
    return out.release();
}

template <PyObject *(*IMPL)(PyObject *const *, Py_ssize_t)>
PyObject *guarded(PyObject *, PyObject *const *a, Py_ssize_t n) {
    try {
        return IMPL(a, n);
    } catch (const PyFail &) {
        return nullptr;
    } catch (...) {   // torch's, as torch's own functions raise them (OutOfMemoryError and the like)
        if (!PyErr_Occurred()) torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}

PyObject *set_error(PyObject *, PyObject *cls) {
    Py_XDECREF(g_error);
    g_error = Py_NewRef(cls);
    Py_RETURN_NONE;
}

#define FAST(name, impl) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&guarded<impl>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("draft", draft_impl),
    FAST("verify", verify_impl),
    FAST("compare_draft", compare_draft_impl),
    FAST("compare_verify", compare_verify_impl),
    FAST("verify_static", verify_static_impl),
    {"set_error", set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_spechub_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__spechub_native() {
    const std::initializer_list<std::pair<PyObject **, const char *>> names = {
        {&N.levels, "levels"}, {&N.child, "child"}, {&N.node_kind, "node_kind"}, {&N.k, "k"},
        {&N.cuda_stream, "cuda_stream"}, {&N.record_stream, "record_stream"},
        {&N.tokens, "tokens"}, {&N.hub, "hub"}, {&N.prob, "prob"}, {&N.status, "status"}, {&N.stats, "stats"},
        {&N.accept_idx, "accept_idx"}, {&N.token, "token"}, {&N.beta, "beta"}, {&N.rate, "rate"},
        {&N.n_accepted, "n_accepted"}, {&N.n_emitted, "n_emitted"}, {&N.path_nodes, "path_nodes"}, {&N.path_tokens, "path_tokens"},
        {&N.spechub, "spechub"}, {&N.rrs, "rrs"}, {&N.rrsw, "rrsw"},
    };
    for (const auto &p : names)
        if (!(*p.first = PyUnicode_InternFromString(p.second))) return nullptr;
    return PyModule_Create(&module);
}
