// Python side of the C ABI for the calls that a decode loop makes on every pass: takes torch tensors, reads their
// addresses and strides, calls libtsd.  A call through ctypes costs 10-17 us of interpreter time (argument
// conversion, torch.cuda.current_stream()), as much as the kernels of a small pass; here it costs about 2 us plus
// the launches.  Only the CPython API is used: tensors are asked for data_ptr(), stride(), shape and nbytes.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include "../../include/tsd.h"

namespace {

PyObject *n_data_ptr, *n_stride, *n_shape, *n_nbytes, *n_dtype, *n_cuda_stream, *n_is_contiguous;
PyObject *get_device, *get_raw_stream, *dtype_f32, *dtype_bf16, *error_type;  // set by setup()

struct Failed {};  // a Python exception is set

struct Ref {  // owned reference
  PyObject* p;
  explicit Ref(PyObject* o) : p(o) { if (!o) throw Failed{}; }
  Ref(const Ref&) = delete;
  ~Ref() { Py_DECREF(p); }
};

int64_t to_int(PyObject* o) {
  const int64_t v = PyLong_AsLongLong(o);
  if (v != -1 || !PyErr_Occurred()) return v;
  PyErr_Clear();
  Ref i(PyNumber_Long(o));  // anything int() takes
  const int64_t w = PyLong_AsLongLong(i.p);
  if (w == -1 && PyErr_Occurred()) throw Failed{};
  return w;
}
int32_t to_i32(PyObject* o) { return (int32_t)to_int(o); }
float to_float(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Failed{};
  return (float)v;
}
// device address of a tensor; None = NULL
template <typename T = void>
T* ptr(PyObject* t, int64_t offset_bytes = 0) {
  if (t == Py_None) return nullptr;
  Ref a(PyObject_CallMethodNoArgs(t, n_data_ptr));
  void* p = PyLong_AsVoidPtr(a.p);
  if (!p && PyErr_Occurred()) throw Failed{};
  return reinterpret_cast<T*>(static_cast<char*>(p) + offset_bytes);
}
size_t nbytes(PyObject* t) {
  if (t == Py_None) return 0;
  Ref n(PyObject_GetAttr(t, n_nbytes));
  return (size_t)to_int(n.p);
}
int read_tuple(const Ref& t, int64_t* v, int most) {
  if (!PyTuple_Check(t.p)) { PyErr_SetString(PyExc_TypeError, "a tensor is wanted"); throw Failed{}; }
  const int n = (int)PyTuple_GET_SIZE(t.p);
  for (int i = 0; i < n && i < most; ++i) v[i] = to_int(PyTuple_GET_ITEM(t.p, i));
  return n;
}
int64_t last_size(PyObject* t) {
  Ref s(PyObject_GetAttr(t, n_shape));
  Ref last(PySequence_GetItem(s.p, -1));
  return to_int(last.p);
}
int shape(PyObject* t, int64_t (&v)[4]) { return read_tuple(Ref(PyObject_GetAttr(t, n_shape)), v, 4); }
int strides(PyObject* t, int64_t (&v)[4]) { return read_tuple(Ref(PyObject_CallMethodNoArgs(t, n_stride)), v, 4); }
bool contiguous(PyObject* t) {  // as torch has it: the stride of a dimension of size 1 does not matter
  Ref c(PyObject_CallMethodNoArgs(t, n_is_contiguous));
  return c.p == Py_True;
}
void want(bool ok, const char* what) {
  if (ok) return;
  PyErr_SetString(PyExc_AssertionError, what);
  throw Failed{};
}
// [batch, rows, heads, dim], dim contiguous -> (batch, row, head) strides in elements
void strides3(PyObject* t, int64_t (&v)[4]) {
  want(strides(t, v) == 4 && v[3] == 1, "head_dim must be contiguous");
}
void same_strides(const int64_t (&a)[4], PyObject* t) {
  int64_t b[4];
  want(strides(t, b) == 4 && a[0] == b[0] && a[1] == b[1] && a[2] == b[2] && a[3] == b[3], "K and V strides differ");
}
[[noreturn]] void raise_error(int rc, const char* where) {
  PyObject* e = PyObject_CallFunction(error_type, "is", rc, where);
  if (e) {
    PyErr_SetObject(error_type, e);
    Py_DECREF(e);
  }
  throw Failed{};
}
int32_t dtype_code(PyObject* t) {
  Ref d(PyObject_GetAttr(t, n_dtype));
  if (d.p == dtype_f32) return TSD_F32;
  if (d.p == dtype_bf16) return TSD_BF16;
  Ref text(PyObject_Str(d.p));
  Ref where(PyUnicode_FromFormat("dtype %U", text.p));
  raise_error(TSD_ERR_UNSUPPORTED, PyUnicode_AsUTF8(where.p));
}
// None = torch's current stream of the current device
tsd_stream_t stream_of(PyObject* s) {
  if (s == Py_None) {
    Ref dev(PyObject_CallNoArgs(get_device));
    Ref raw(PyObject_CallOneArg(get_raw_stream, dev.p));
    return reinterpret_cast<tsd_stream_t>((uintptr_t)to_int(raw.p));
  }
  PyObject* raw = PyObject_GetAttr(s, n_cuda_stream);
  if (raw) {
    Ref r(raw);
    return reinterpret_cast<tsd_stream_t>((uintptr_t)to_int(r.p));
  }
  PyErr_Clear();
  return reinterpret_cast<tsd_stream_t>((uintptr_t)to_int(s));
}
struct Layout {  // a ctypes structure, read through the buffer protocol
  Py_buffer b;
  explicit Layout(PyObject* o) {
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) throw Failed{};
    if (b.len != (Py_ssize_t)sizeof(tsd_layout)) {
      PyBuffer_Release(&b);
      PyErr_SetString(PyExc_TypeError, "a tsd_layout is wanted");
      throw Failed{};
    }
  }
  ~Layout() { PyBuffer_Release(&b); }
  const tsd_layout* get() const { return static_cast<const tsd_layout*>(b.buf); }
};
// the call itself runs without the interpreter lock
template <typename... P, typename... A>
int call(int (*f)(P...), A... args) {
  PyThreadState* state = PyEval_SaveThread();
  const int rc = f(static_cast<P>(args)...);
  PyEval_RestoreThread(state);
  return rc;
}
PyObject* done(int rc, const char* where) {
  if (rc != TSD_OK) raise_error(rc, where);
  Py_RETURN_NONE;
}

using Args = PyObject* const*;

PyObject* setup(Args a) {
  PyObject** to[] = {&get_device, &get_raw_stream, &dtype_f32, &dtype_bf16, &error_type};
  for (int i = 0; i < 5; ++i) {
    Py_INCREF(a[i]);
    Py_XSETREF(*to[i], a[i]);
  }
  Py_RETURN_NONE;
}

struct AttnViews {
  int64_t q[4], c[4] = {0, 0, 0, 1}, d[4], o[4];
  AttnViews(const tsd_layout* L, PyObject* q_, PyObject* kc, PyObject* vc, PyObject* kd, PyObject* vd, PyObject* out) {
    if (kc != Py_None) {
      strides3(kc, c);
      if (vc != Py_None) same_strides(c, vc);
    } else {
      want(vc == Py_None, "V rows of the cache without K rows");
      c[2] = L->head_dim;
    }
    strides3(kd, d);
    same_strides(d, vd);
    strides3(q_, q);
    strides3(out, o);
  }
};

// layout, mask, q, k_cache, v_cache, k_draft, v_draft, out, lse, sm_scale, workspace, flags, status, stream
PyObject* verify_attention(Args a) {
  Layout L(a[0]);
  const AttnViews v(L.get(), a[2], a[3], a[4], a[5], a[6], a[7]);
  return done(call(tsd_verify_attention, L.get(), ptr(a[1]), ptr(a[2]), v.q[0], v.q[1], v.q[2], ptr(a[3]), ptr(a[4]), v.c[0], v.c[1],
                                   v.c[2], ptr(a[5]), ptr(a[6]), v.d[0], v.d[1], v.d[2], ptr(a[7]), v.o[0], v.o[1], v.o[2],
                                   ptr<float>(a[8]), to_float(a[9]), ptr(a[10]), nbytes(a[10]), (uint32_t)to_int(a[11]),
                                   ptr<uint32_t>(a[12]), stream_of(a[13])),
              "tsd_verify_attention");
}

// layout, mask, q, k_codes, v_codes, k_scale, v_scale, k_draft, v_draft, out, workspace, lse, sm_scale, flags, status, stream
PyObject* verify_attention_fp8(Args a) {
  Layout L(a[0]);
  const AttnViews v(L.get(), a[2], a[3], a[4], a[7], a[8], a[9]);
  want(a[10] != Py_None, "a workspace is wanted");
  return done(call(tsd_verify_attention_fp8_cache, L.get(), ptr(a[1]), ptr(a[2]), v.q[0], v.q[1], v.q[2], ptr<uint8_t>(a[3]), ptr<uint8_t>(a[4]), v.c[0], v.c[1],
                  v.c[2], ptr<float>(a[5]), ptr<float>(a[6]), ptr(a[7]), ptr(a[8]), v.d[0], v.d[1], v.d[2], ptr(a[9]), v.o[0],
                  v.o[1], v.o[2], ptr<float>(a[11]), to_float(a[12]), ptr(a[10]), nbytes(a[10]), (uint32_t)to_int(a[13]),
                  ptr<uint32_t>(a[14]), stream_of(a[15])),
              "tsd_verify_attention_fp8_cache");
}

struct Logits {
  int64_t n, pitch;
  int32_t vocab, dtype;
  explicit Logits(PyObject* t) {
    int64_t s[4], st[4];
    want(shape(t, s) == 2 && strides(t, st) == 2 && st[1] == 1, "logits are [rows, vocab], contiguous in the vocabulary");
    n = s[0];
    vocab = (int32_t)s[1];
    pitch = st[0];
    dtype = dtype_code(t);
  }
};

// logits, k, conf, topk_idx, topk_prob, lse, workspace, status, stream
PyObject* confidence_topk(Args a) {
  const Logits x(a[0]);
  return done(call(tsd_confidence_topk, ptr(a[0]), x.dtype, x.n, x.vocab, x.pitch, to_i32(a[1]), ptr<float>(a[2]), ptr<int32_t>(a[3]),
                                  ptr<float>(a[4]), ptr<float>(a[5]), ptr(a[6]), nbytes(a[6]), ptr<uint32_t>(a[7]),
                                  stream_of(a[8])),
              "tsd_confidence_topk");
}

void shape3(PyObject* t, int64_t (&v)[4]) {
  if (shape(t, v) == 3) return;
  PyErr_SetString(PyExc_ValueError, "state is [sequences, branches, rows]");
  throw Failed{};
}

// parent, state, n_cur (None = one tree), mask_id, conf, top1, top1_stride, tau, rule, search, edge_valid, prefix_len,
// accepted_node, accepted_len, n_new_tokens, unmask_flag, unmask_tok, status, stream
PyObject* accept(Args a) {
  int64_t s[4];
  shape3(a[1], s);
  const bool one = a[2] == Py_None;
  return done(call(tsd_accept_joint_trees, (int32_t)s[0], (int32_t)s[1], one ? (int32_t)s[1] : to_i32(a[2]), (int32_t)s[2],
                                     ptr<int32_t>(a[0]), ptr<int32_t>(a[1]), to_i32(a[3]), ptr<float>(a[4]), ptr<int32_t>(a[5]),
                                     to_i32(a[6]), to_float(a[7]), to_i32(a[8]), to_i32(a[9]), ptr<uint8_t>(a[10]),
                                     ptr<int32_t>(a[11]), ptr<int32_t>(a[12]), ptr<int32_t>(a[13]), ptr<int32_t>(a[14]),
                                     ptr<uint8_t>(a[15]), ptr<int32_t>(a[16]), ptr<uint32_t>(a[17]), stream_of(a[18])),
              one ? "tsd_accept_trajectories" : "tsd_accept_joint_trees");
}

// parent, state, n_cur, mask_id, conf, topk_idx, topk_m, logits, lse, tau, rule, search, edge_valid, prefix_len,
// accepted_node, accepted_len, n_new_tokens, unmask_flag, unmask_tok, draft_prob, status, stream
PyObject* accept_relaxed(Args a) {
  int64_t s[4], c[4];
  shape3(a[1], s);
  const int n_cand = shape(a[5], c) == 4 ? (int)c[3] : 1;
  int32_t dtype = 0;
  int64_t vocab = 0, pitch = 0;
  if (a[7] != Py_None) {
    const Logits x(a[7]);
    want(x.n == s[0] * s[1] * s[2], "logits have a row for every (sequence, branch, row)");
    dtype = x.dtype;
    vocab = x.vocab;
    pitch = x.pitch;
  }
  return done(call(tsd_accept_relaxed, (int32_t)s[0], (int32_t)s[1], to_i32(a[2]), (int32_t)s[2], ptr<int32_t>(a[0]), ptr<int32_t>(a[1]),
                                 to_i32(a[3]), ptr<float>(a[4]), ptr<int32_t>(a[5]), n_cand, to_i32(a[6]), ptr(a[7]), dtype, vocab,
                                 pitch, ptr<float>(a[8]), to_float(a[9]), to_i32(a[10]), to_i32(a[11]), ptr<uint8_t>(a[12]),
                                 ptr<int32_t>(a[13]), ptr<int32_t>(a[14]), ptr<int32_t>(a[15]), ptr<int32_t>(a[16]),
                                 ptr<uint8_t>(a[17]), ptr<int32_t>(a[18]), ptr<float>(a[19]), ptr<uint32_t>(a[20]),
                                 stream_of(a[21])),
              "tsd_accept_relaxed");
}

// parent, state, accepted_node, unmask_flag, unmask_tok, mask_id, tokens, block_start, root_out, fill_step, step_base,
// n_masked, status, stream, tree_root
PyObject* commit(Args a) {
  int64_t s[4], st[4] = {0, 0, 0, 0};
  shape3(a[1], s);
  if (a[6] != Py_None) want(strides(a[6], st) == 2 && st[1] == 1, "tokens are [sequences, length], contiguous");
  return done(call(tsd_commit_accepted, (int32_t)s[0], (int32_t)s[1], (int32_t)s[2], to_i32(a[14]), ptr<int32_t>(a[0]),
                                  ptr<int32_t>(a[1]), ptr<int32_t>(a[2]), ptr<uint8_t>(a[3]), ptr<int32_t>(a[4]), to_i32(a[5]),
                                  ptr<int32_t>(a[6]), st[0], ptr<int32_t>(a[7]), ptr<int32_t>(a[8]), ptr<int32_t>(a[9]),
                                  ptr<int32_t>(a[10]), ptr<int32_t>(a[11]), ptr<uint32_t>(a[12]), stream_of(a[13])),
              "tsd_commit_accepted");
}

// prev_state, accepted_node, unmask_flag, unmask_tok, mask_id, topk_idx, topk_prob, width, depth, parent, state, node_prob,
// n_nodes, status, stream, first, max_nodes (None = the rest), enable
PyObject* build_tree(Args a) {
  int64_t s[4], o[4];
  shape3(a[0], s);
  const int64_t k = last_size(a[5]);
  shape3(a[10], o);
  const int64_t first = to_int(a[15]), B = o[1], max_nodes = a[16] == Py_None ? B - first : to_int(a[16]);
  want(0 <= first && first + max_nodes <= B, "the tree fits the output arrays");
  return done(call(tsd_build_draft_tree, (int32_t)s[0], (int32_t)s[1], (int32_t)s[2], (int32_t)k, ptr<int32_t>(a[0]),
                                   ptr<int32_t>(a[1]), ptr<uint8_t>(a[2]), ptr<int32_t>(a[3]), to_i32(a[4]), ptr<int32_t>(a[5]),
                                   ptr<float>(a[6]), to_i32(a[7]), to_i32(a[8]), (int32_t)max_nodes, (int32_t)B, (int32_t)first,
                                   ptr<uint8_t>(a[17]), ptr<int32_t>(a[9], first * 4), ptr<int32_t>(a[10], first * o[2] * 4),
                                   ptr<float>(a[11], first * 4), ptr<int32_t>(a[12]), ptr<uint32_t>(a[13]), stream_of(a[14])),
              "tsd_build_draft_tree");
}

// layout, vis, cache_lens, mask_out, dense_out, stream
PyObject* build_mask(Args a) {
  Layout L(a[0]);
  return done(call(tsd_build_branch_mask, L.get(), ptr<uint64_t>(a[1]), ptr<int32_t>(a[2]), ptr(a[3]), nbytes(a[3]), ptr<uint8_t>(a[4]),
                                    stream_of(a[5])),
              "tsd_build_branch_mask");
}

// n_cur, vis, stream
PyObject* interblock_vis(Args a) {
  int64_t s[4];
  want(shape(a[1], s) == 3 && s[2] == (s[1] + 63) / 64 && contiguous(a[1]) && (int64_t)nbytes(a[1]) == 8 * s[0] * s[1] * s[2],
       "vis is a contiguous 64-bit [sequences, branches, words]");
  return done(call(tsd_build_interblock_vis, (int32_t)s[0], (int32_t)s[1], to_i32(a[0]), ptr<uint64_t>(a[1]), stream_of(a[2])),
              "tsd_build_interblock_vis");
}

// state, conf, node_cur, node_next, mask_id, tau, trigger, top_conf, status, stream
PyObject* interblock_trigger(Args a) {
  int64_t s[4];
  shape3(a[0], s);
  return done(call(tsd_interblock_trigger, (int32_t)s[0], (int32_t)s[1], (int32_t)s[2], ptr<int32_t>(a[0]), ptr<float>(a[1]),
                   ptr<int32_t>(a[2]), to_i32(a[3]), to_i32(a[4]), to_float(a[5]), ptr<uint8_t>(a[6]), ptr<float>(a[7]),
                   ptr<uint32_t>(a[8]), stream_of(a[9])),
              "tsd_interblock_trigger");
}

// layout, mask, q, k_cache, v_cache, k_draft, v_draft, out, attn_lse, sm_scale, attn_workspace, flags, logits, k, conf,
// topk_idx, topk_prob, lse, topk_workspace, parent, state, mask_id, tau, rule, search, edge_valid, prefix_len,
// accepted_node, accepted_len, n_new_tokens, unmask_flag, unmask_tok, status, stream
PyObject* verify_step(Args a) {
  Layout L(a[0]);
  const AttnViews v(L.get(), a[2], a[3], a[4], a[5], a[6], a[7]);
  const Logits x(a[12]);
  tsd_step_args t = {};
  t.layout = L.get();
  t.mask = ptr(a[1]);
  t.q = ptr(a[2]); t.k_cache = ptr(a[3]); t.v_cache = ptr(a[4]); t.k_draft = ptr(a[5]); t.v_draft = ptr(a[6]); t.out = ptr(a[7]);
  for (int i = 0; i < 3; ++i) { t.q_stride[i] = v.q[i]; t.c_stride[i] = v.c[i]; t.d_stride[i] = v.d[i]; t.o_stride[i] = v.o[i]; }
  t.attn_lse = ptr<float>(a[8]);
  t.sm_scale = to_float(a[9]);
  t.attn_workspace = ptr(a[10]);
  t.attn_workspace_bytes = nbytes(a[10]);
  t.flags = (uint32_t)to_int(a[11]);
  t.logits = ptr(a[12]);
  t.n_rows = x.n; t.row_stride = x.pitch; t.logits_dtype = x.dtype; t.vocab = x.vocab;
  t.k = to_i32(a[13]);
  t.conf = ptr<float>(a[14]); t.topk_idx = ptr<int32_t>(a[15]); t.topk_prob = ptr<float>(a[16]); t.lse = ptr<float>(a[17]);
  t.topk_workspace = ptr(a[18]);
  t.topk_workspace_bytes = nbytes(a[18]);
  t.parent = ptr<int32_t>(a[19]); t.state = ptr<int32_t>(a[20]);
  t.mask_id = to_i32(a[21]);
  t.tau = to_float(a[22]);
  t.rule = to_i32(a[23]);
  t.search = to_i32(a[24]);
  t.edge_valid = ptr<uint8_t>(a[25]); t.prefix_len = ptr<int32_t>(a[26]); t.accepted_node = ptr<int32_t>(a[27]);
  t.accepted_len = ptr<int32_t>(a[28]); t.n_new_tokens = ptr<int32_t>(a[29]); t.unmask_flag = ptr<uint8_t>(a[30]);
  t.unmask_tok = ptr<int32_t>(a[31]); t.status = ptr<uint32_t>(a[32]);
  return done(call(tsd_verify_step, &t, stream_of(a[33])), "tsd_verify_step");
}

// root_state [S, R], mask_id, parent, state, n_nodes, root_out, fill_step, step_base, n_masked, report, ticket, status, stream
PyObject* begin_block(Args a) {
  int64_t s[4];
  shape3(a[3], s);
  return done(call(tsd_begin_block, (int32_t)s[0], (int32_t)s[1], (int32_t)s[2], to_i32(a[1]), ptr<int32_t>(a[0]), ptr<int32_t>(a[2]),
                   ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), ptr<int32_t>(a[5]), ptr<int32_t>(a[6]), ptr<int32_t>(a[7]),
                   ptr<int32_t>(a[8]), ptr<uint64_t>(a[9]), (uint32_t)to_int(a[10]), ptr<uint32_t>(a[11]), stream_of(a[12])),
              "tsd_begin_block");
}

// logits, k, conf, topk_idx, topk_prob, lse, topk_workspace, parent, state, mask_id, tau, rule, search, edge_valid, prefix_len,
// accepted_node, accepted_len, n_new_tokens, unmask_flag, unmask_tok, draft_prob, tokens, block_start, root_out, fill_step,
// step_base, n_masked, width, depth, next_parent, next_state, next_prob, next_n, report, ticket, status, stream, done
PyObject* advance_block(Args a) {
  int64_t s[4], st[4] = {0, 0, 0, 0};
  shape3(a[8], s);
  const Logits x(a[0]);
  want(to_i32(a[11]) == TSD_ACCEPT_PROB ? x.n == s[0] * s[1] * s[2] : x.n <= s[0] * s[1] * s[2],
       "logits have a row for every (sequence, branch, row)");
  if (a[21] != Py_None) want(strides(a[21], st) == 2 && st[1] == 1, "tokens are [sequences, length], contiguous");
  tsd_advance_args t = {};
  t.batch = (int32_t)s[0]; t.n_branches = (int32_t)s[1]; t.rows_per_branch = (int32_t)s[2];
  t.logits = ptr(a[0]);
  t.n_rows = x.n; t.row_stride = x.pitch; t.logits_dtype = x.dtype; t.vocab = x.vocab;
  t.k = to_i32(a[1]);
  t.conf = ptr<float>(a[2]); t.topk_idx = ptr<int32_t>(a[3]); t.topk_prob = ptr<float>(a[4]); t.lse = ptr<float>(a[5]);
  t.topk_workspace = ptr(a[6]);
  t.topk_workspace_bytes = nbytes(a[6]);
  t.parent = ptr<int32_t>(a[7]); t.state = ptr<int32_t>(a[8]);
  t.mask_id = to_i32(a[9]);
  t.tau = to_float(a[10]);
  t.rule = to_i32(a[11]);
  t.search = to_i32(a[12]);
  t.edge_valid = ptr<uint8_t>(a[13]); t.prefix_len = ptr<int32_t>(a[14]); t.accepted_node = ptr<int32_t>(a[15]);
  t.accepted_len = ptr<int32_t>(a[16]); t.n_new_tokens = ptr<int32_t>(a[17]); t.unmask_flag = ptr<uint8_t>(a[18]);
  t.unmask_tok = ptr<int32_t>(a[19]); t.draft_prob = ptr<float>(a[20]);
  t.tokens = ptr<int32_t>(a[21]);
  t.seq_stride = st[0];
  t.block_start = ptr<int32_t>(a[22]);
  t.root_out = ptr<int32_t>(a[23]); t.fill_step = ptr<int32_t>(a[24]); t.step_base = ptr<int32_t>(a[25]); t.n_masked = ptr<int32_t>(a[26]);
  t.width = to_i32(a[27]); t.depth = to_i32(a[28]);
  t.next_parent = ptr<int32_t>(a[29]); t.next_state = ptr<int32_t>(a[30]); t.next_prob = ptr<float>(a[31]); t.next_n = ptr<int32_t>(a[32]);
  t.report = ptr<uint64_t>(a[33]);
  t.done = ptr<uint64_t>(a[37]);
  t.ticket = (uint32_t)to_int(a[34]);
  t.status = ptr<uint32_t>(a[35]);
  return done(call(tsd_advance_block, &t, stream_of(a[36])), "tsd_advance_block");
}

// n_masked [S], status, report, ticket, stream
PyObject* report_block(Args a) {
  int64_t s[4];
  want(shape(a[0], s) == 1, "n_masked is [sequences]");
  return done(call(tsd_report_block, (int32_t)s[0], ptr<int32_t>(a[0]), ptr<uint32_t>(a[1]), ptr<uint64_t>(a[2]), (uint32_t)to_int(a[3]),
                   stream_of(a[4])),
              "tsd_report_block");
}

// report [S], ticket, stream -> (largest count of masked rows, status bits)
PyObject* wait_block(Args a) {
  int64_t s[4];
  want(shape(a[0], s) == 1, "report is [sequences]");
  int32_t masked = 0;
  uint32_t bits = 0;
  const int rc = call(tsd_wait_block, (int32_t)s[0], ptr<uint64_t>(a[0]), (uint32_t)to_int(a[1]), &masked, &bits, stream_of(a[2]));
  if (rc != TSD_OK) raise_error(rc, "tsd_wait_block");
  return Py_BuildValue("iI", masked, bits);
}

// METH_FASTCALL entry: argument count, then C++ to Python errors
template <PyObject* (*F)(Args), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "%d arguments are wanted, got %zd", N, n);
    return nullptr;
  }
  try {
    return F(args);
  } catch (Failed&) {
    return nullptr;
  }
}

#define TSD_METHOD(f, n) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<f, n>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {TSD_METHOD(setup, 5),           TSD_METHOD(verify_attention, 14), TSD_METHOD(verify_attention_fp8, 16),
                         TSD_METHOD(confidence_topk, 9), TSD_METHOD(accept, 19),           TSD_METHOD(accept_relaxed, 22),
                         TSD_METHOD(commit, 15),         TSD_METHOD(build_tree, 18),       TSD_METHOD(build_mask, 6),
                         TSD_METHOD(verify_step, 34),    TSD_METHOD(interblock_vis, 3),    TSD_METHOD(interblock_trigger, 10),
                         TSD_METHOD(begin_block, 13),    TSD_METHOD(advance_block, 38),    TSD_METHOD(report_block, 5),
                         TSD_METHOD(wait_block, 3),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tsd_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tsd_native(void) {
  n_data_ptr = PyUnicode_InternFromString("data_ptr");
  n_stride = PyUnicode_InternFromString("stride");
  n_shape = PyUnicode_InternFromString("shape");
  n_nbytes = PyUnicode_InternFromString("nbytes");
  n_dtype = PyUnicode_InternFromString("dtype");
  n_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  n_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  return PyModule_Create(&module);
}
