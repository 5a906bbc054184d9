/* CPython entry points of the C ABI: argument marshalling of the calls a decoding loop makes per step.  A call through
 * ctypes costs 6-10 us of host time (two structures, ~15 attribute calls, the current-stream object); the small
 * calls of this library run 2-10 us on the GPU, so the host decided their time.  Here a call fills the C
 * structures straight from the keyword arguments. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stddef.h>
#include <string.h>

#include "vvs.h"

static PyObject *g_error, *g_raw_stream, *g_get_device;   /* VvsError; torch's current raw stream and device */
static PyObject *s_data_ptr, *s_shape, *s_cuda_stream;

/* tensor (or integer address, or None) -> address; -1 with an exception set on failure */
static int to_ptr(PyObject* o, void** out) {
  if (o == Py_None) { *out = NULL; return 0; }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return PyErr_Occurred() ? -1 : 0;
  }
  PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}
static int to_int(PyObject* o, int32_t* out) {
  PyObject* v = PyNumber_Long(o);
  if (!v) return -1;
  const long x = PyLong_AsLong(v);
  Py_DECREF(v);
  if (x == -1 && PyErr_Occurred()) return -1;
  *out = (int32_t)x;
  return 0;
}
static int to_float(PyObject* o, float* out) {
  const double x = PyFloat_AsDouble(o);
  if (x == -1.0 && PyErr_Occurred()) return -1;
  *out = (float)x;
  return 0;
}
/* the stream of a call: None = torch's current stream of the current device */
static int to_stream(PyObject* o, void** out) {
  PyObject* v;
  if (!o || o == Py_None) {
    PyObject* dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return -1;
    v = PyObject_CallOneArg(g_raw_stream, dev);
    Py_DECREF(dev);
  } else if (PyLong_Check(o)) {
    v = Py_NewRef(o);
  } else {
    v = PyObject_GetAttr(o, s_cuda_stream);
    if (!v && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      v = PyNumber_Long(o);
    }
  }
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

/* One parameter of an entry point: where it goes and what it is. */
typedef struct {
  const char* name;
  char kind;          /* p tensor / address, i int32, f float, b truth value, c context, s stream, o object */
  char required;
  size_t off;         /* byte offset in the call's frame */
  PyObject* key;      /* interned name */
} Param;
#define MAX_PARAMS 40

static int put(const Param* q, PyObject* v, char* frame) {
  void* at = frame + q->off;
  switch (q->kind) {
    case 'p': return to_ptr(v, (void**)at);
    case 'i': return to_int(v, (int32_t*)at);
    case 'f': return to_float(v, (float*)at);
    case 'b': return to_int(v, (int32_t*)at);
    case 'c': *(void**)at = v == Py_None ? NULL : PyLong_AsVoidPtr(v); return PyErr_Occurred() ? -1 : 0;
    case 's': return to_stream(v, (void**)at);
    default: *(PyObject**)at = v; return 0;
  }
}

/* Fills `frame` from the call; positional arguments take the parameters in order (at most `n_pos` of them). */
static int parse(const char* fn, const Param* ps, int n, int n_pos, void* frame, PyObject* const* args, Py_ssize_t nargs,
                 PyObject* kwnames) {
  unsigned char seen[MAX_PARAMS] = {0};
  if (nargs > n_pos) {
    PyErr_Format(PyExc_TypeError, "%s() takes %d positional arguments but %zd were given", fn, n_pos, nargs);
    return -1;
  }
  for (Py_ssize_t i = 0; i < nargs; ++i) {
    if (put(&ps[i], args[i], frame) < 0) return -1;
    seen[i] = 1;
  }
  const Py_ssize_t nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  int hint = (int)nargs;
  for (Py_ssize_t k = 0; k < nk; ++k) {
    PyObject* key = PyTuple_GET_ITEM(kwnames, k);
    int j = -1;
    for (int t = 0; t < n && j < 0; ++t) {           /* callers keep their order: start behind the previous match */
      const int c = hint + t < n ? hint + t : hint + t - n;
      if (ps[c].key == key) j = c;
    }
    for (int c = 0; j < 0 && c < n; ++c)
      if (PyUnicode_Compare(ps[c].key, key) == 0) j = c;
    if (j < 0) {
      PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", fn, key);
      return -1;
    }
    if (seen[j]) {
      PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", fn, ps[j].name);
      return -1;
    }
    if (put(&ps[j], args[nargs + k], frame) < 0) return -1;
    seen[j] = 1;
    hint = j + 1 < n ? j + 1 : 0;
  }
  for (int i = 0; i < n; ++i) {
    if (seen[i]) continue;
    if (ps[i].required) {
      PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", fn, ps[i].name);
      return -1;
    }
    if (ps[i].kind == 's' && to_stream(NULL, (void**)((char*)frame + ps[i].off)) < 0) return -1;
  }
  return 0;
}

static PyObject* done(int status, const char* where) {
  if (status == VVS_OK) Py_RETURN_NONE;
  PyObject* e = PyObject_CallFunction(g_error, "is", status, where);
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  return NULL;
}
/* The library call runs without the interpreter lock (a first call captures a graph: milliseconds). */
#define CALL(name, expr)        \
  do {                          \
    int rc;                     \
    Py_BEGIN_ALLOW_THREADS      \
    rc = (expr);                \
    Py_END_ALLOW_THREADS        \
    return done(rc, name);      \
  } while (0)

/* ---- the decision-making calls: one frame for all of them ------------------------------------------------------ */
typedef struct {
  vvs_ctx* ctx;
  vvs_verify_args a;
  vvs_verify_out o;
  void* stream;
  void *hidden_in, *drafts, *target_probs, *nbr_row_ptr, *nbr_col, *status_bits;
  int32_t n_rows_per_seq, first_row, vocab, vocab_offset;
} Frame;
#define A(f) offsetof(Frame, a) + offsetof(vvs_verify_args, f)
#define O(f) offsetof(Frame, o) + offsetof(vvs_verify_out, f)
#define F(f) offsetof(Frame, f)

static void frame_init(Frame* f) {
  memset(f, 0, sizeof(*f));
  f->a.n_cfg = f->a.n_forced = f->a.nbr_k = 1;
  f->a.cfg_scale = f->a.temperature = 1.f;
  f->a.delta = Py_HUGE_VAL;
}

#define DECISION_PARAMS                                                                                              \
  {"draft_probs", 'p', 1, A(draft_probs)}, {"uniforms", 'p', 1, A(uniforms)}, {"accept_len", 'p', 1, O(accept_len)}, \
      {"next_token", 'p', 1, O(next_token)}, {"n_draft", 'p', 0, A(n_draft)}, {"mode", 'i', 0, A(mode)},             \
      {"nbr_k", 'i', 0, A(nbr_k)}, {"delta", 'f', 0, A(delta)}, {"accept_mask", 'p', 0, O(accept_mask)},             \
      {"margins", 'p', 0, O(margins)}, {"adjusted_residual", 'b', 0, A(adjusted_residual)}, {"stream", 's', 0, F(stream)}

static Param verify_params[] = {
    {"ctx", 'c', 1, F(ctx)}, {"n_images", 'i', 1, A(n_images)}, {"n_cfg", 'i', 1, A(n_cfg)}, {"n_forced", 'i', 1, A(n_forced)},
    {"n_draft_max", 'i', 1, A(n_draft_max)}, {"block", 'p', 1, A(block)}, {"kv_k", 'p', 1, A(kv_k)}, {"kv_v", 'p', 1, A(kv_v)},
    {"kv_rows", 'i', 1, A(kv_rows)}, {"cache_len", 'p', 1, A(cache_len)}, {"new_len", 'p', 1, O(new_len)},
    {"cache_len_host", 'p', 0, A(cache_len_host)}, {"cfg_scale", 'f', 0, A(cfg_scale)}, {"temperature", 'f', 0, A(temperature)},
    {"n_commit", 'p', 0, O(n_commit)}, {"target_probs", 'p', 0, O(target_probs)}, {"hidden", 'p', 0, O(hidden)},
    {"tree_parent", 'p', 0, A(tree_parent)}, {"accept_path", 'p', 0, O(accept_path)}, DECISION_PARAMS};
static Param epilogue_params[] = {
    {"ctx", 'c', 1, F(ctx)}, {"hidden_in", 'p', 1, F(hidden_in)}, {"n_rows_per_seq", 'i', 1, F(n_rows_per_seq)},
    {"first_row", 'i', 1, F(first_row)}, {"drafts", 'p', 1, F(drafts)}, {"n_images", 'i', 1, A(n_images)},
    {"n_cfg", 'i', 1, A(n_cfg)}, {"n_draft_max", 'i', 1, A(n_draft_max)}, {"cfg_scale", 'f', 0, A(cfg_scale)},
    {"temperature", 'f', 0, A(temperature)}, {"target_probs", 'p', 0, O(target_probs)}, DECISION_PARAMS};
static Param decide_params[] = {
    {"ctx", 'c', 1, F(ctx)}, {"target_probs", 'p', 1, F(target_probs)}, {"n_rows_per_seq", 'i', 1, F(n_rows_per_seq)},
    {"first_row", 'i', 1, F(first_row)}, {"drafts", 'p', 1, F(drafts)}, {"n_images", 'i', 1, A(n_images)},
    {"n_draft_max", 'i', 1, A(n_draft_max)}, {"tree_parent", 'p', 0, A(tree_parent)}, {"accept_path", 'p', 0, O(accept_path)},
    DECISION_PARAMS};
static Param noalloc_params[] = {
    {"target_probs", 'p', 1, F(target_probs)}, {"vocab", 'i', 1, F(vocab)}, {"vocab_offset", 'i', 1, F(vocab_offset)},
    {"n_rows_per_seq", 'i', 1, F(n_rows_per_seq)}, {"first_row", 'i', 1, F(first_row)}, {"drafts", 'p', 1, F(drafts)},
    {"n_images", 'i', 1, A(n_images)}, {"n_draft_max", 'i', 1, A(n_draft_max)}, {"nbr_row_ptr", 'p', 0, F(nbr_row_ptr)},
    {"nbr_col", 'p', 0, F(nbr_col)}, {"status_bits", 'p', 0, F(status_bits)}, {"tree_parent", 'p', 0, A(tree_parent)},
    {"accept_path", 'p', 0, O(accept_path)}, DECISION_PARAMS};
#define N(ps) (int)(sizeof(ps) / sizeof(ps[0]))
#define FAST PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames
#define PARSE(name, ps, n_pos) parse(name, ps, N(ps), n_pos, &f, args, nargs, kwnames)

static PyObject* py_verify(FAST) {
  (void)self;
  Frame f;
  frame_init(&f);
  if (PARSE("vvs_verify", verify_params, 1) < 0) return NULL;
  CALL("vvs_verify", vvs_verify(f.ctx, &f.a, &f.o, f.stream));
}
static PyObject* py_epilogue(FAST) {
  (void)self;
  Frame f;
  frame_init(&f);
  if (PARSE("vvs_epilogue", epilogue_params, 1) < 0) return NULL;
  CALL("vvs_epilogue", vvs_epilogue(f.ctx, f.hidden_in, f.n_rows_per_seq, f.first_row, f.drafts, &f.a, &f.o, f.stream));
}
static PyObject* py_decide(FAST) {
  (void)self;
  Frame f;
  frame_init(&f);
  if (PARSE("vvs_decide", decide_params, 1) < 0) return NULL;
  CALL("vvs_decide", vvs_decide(f.ctx, f.target_probs, f.n_rows_per_seq, f.first_row, f.drafts, &f.a, &f.o, f.stream));
}
static PyObject* py_decide_noalloc(FAST) {
  (void)self;
  Frame f;
  frame_init(&f);
  if (PARSE("vvs_decide_noalloc", noalloc_params, 0) < 0) return NULL;
  CALL("vvs_decide_noalloc", vvs_decide_noalloc(f.target_probs, f.vocab, f.vocab_offset, f.n_rows_per_seq, f.first_row, f.drafts,
                                                f.nbr_row_ptr, f.nbr_col, &f.a, &f.o, f.status_bits, f.stream));
}

/* ---- feature cache and the verification-free step -------------------------------------------------------------- */
typedef struct {
  vvs_ctx* ctx;
  PyObject *fc, *paths, *codebook;
  void *hidden, *base_pos, *n_store, *skip_mask, *gamma, *out, *out_pos, *stream;
  void *path_len, *last_verified, *decision, *similarity, *uniforms, *out_path, *out_gamma, *out_tokens;
  int32_t n_rows_per_seq, n_images, gamma_max, staleness, stride;
  float alpha, threshold;
} Frame2;
#define G(f) offsetof(Frame2, f)
static Param reset_params[] = {{"ctx", 'c', 1, G(ctx)}, {"fc", 'o', 1, G(fc)}, {"stream", 's', 0, G(stream)}};
static Param store_params[] = {
    {"ctx", 'c', 1, G(ctx)}, {"fc", 'o', 1, G(fc)}, {"hidden", 'p', 1, G(hidden)}, {"n_rows_per_seq", 'i', 1, G(n_rows_per_seq)},
    {"base_pos", 'p', 1, G(base_pos)}, {"n_store", 'p', 1, G(n_store)}, {"stream", 's', 0, G(stream)}};
static Param fetch_params[] = {
    {"ctx", 'c', 1, G(ctx)}, {"fc", 'o', 1, G(fc)}, {"skip_mask", 'p', 1, G(skip_mask)}, {"n_images", 'i', 1, G(n_images)},
    {"gamma", 'p', 1, G(gamma)}, {"gamma_max", 'i', 1, G(gamma_max)}, {"staleness", 'i', 1, G(staleness)}, {"out", 'p', 1, G(out)},
    {"out_pos", 'p', 1, G(out_pos)}, {"stream", 's', 0, G(stream)}};
static Param skip_params[] = {
    {"ctx", 'c', 1, G(ctx)}, {"paths", 'o', 1, G(paths)}, {"path_len", 'p', 1, G(path_len)}, {"codebook", 'o', 1, G(codebook)},
    {"last_verified", 'p', 1, G(last_verified)}, {"stride", 'i', 1, G(stride)}, {"alpha", 'f', 1, G(alpha)},
    {"threshold", 'f', 1, G(threshold)}, {"decision", 'p', 1, G(decision)}, {"similarity", 'p', 1, G(similarity)},
    {"stream", 's', 0, G(stream)}};
static Param select_params[] = {
    {"ctx", 'c', 1, G(ctx)}, {"paths", 'o', 1, G(paths)}, {"path_len", 'p', 1, G(path_len)}, {"uniforms", 'p', 1, G(uniforms)},
    {"out_path", 'p', 1, G(out_path)}, {"out_gamma", 'p', 1, G(out_gamma)}, {"out_tokens", 'p', 1, G(out_tokens)},
    {"stream", 's', 0, G(stream)}};

static int shape_of(PyObject* t, int want, int32_t* dims) {
  PyObject* sh = PyObject_GetAttr(t, s_shape);
  if (!sh) return -1;
  int rc = -1;
  if (!PyTuple_Check(sh) || PyTuple_GET_SIZE(sh) != want) {
    PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions", want);
  } else {
    rc = 0;
    for (int i = 0; i < want && rc == 0; ++i) rc = to_int(PyTuple_GET_ITEM(sh, i), &dims[i]);
  }
  Py_DECREF(sh);
  return rc;
}
/* the structure behind a ctypes vvs_fcache */
static int fcache_of(PyObject* o, vvs_fcache* out) {
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) < 0) return -1;
  const int ok = b.len == (Py_ssize_t)sizeof(*out);
  if (ok) memcpy(out, b.buf, sizeof(*out));
  PyBuffer_Release(&b);
  if (!ok) PyErr_SetString(PyExc_TypeError, "expected a vvs_fcache");
  return ok ? 0 : -1;
}

static PyObject* py_reset(FAST) {
  (void)self;
  Frame2 f = {0};
  vvs_fcache fc;
  if (PARSE("vvs_feature_cache_reset", reset_params, N(reset_params)) < 0 || fcache_of(f.fc, &fc) < 0) return NULL;
  CALL("vvs_feature_cache_reset", vvs_feature_cache_reset(f.ctx, &fc, f.stream));
}
static PyObject* py_store(FAST) {
  (void)self;
  Frame2 f = {0};
  vvs_fcache fc;
  if (PARSE("vvs_feature_cache_store", store_params, N(store_params)) < 0 || fcache_of(f.fc, &fc) < 0) return NULL;
  CALL("vvs_feature_cache_store", vvs_feature_cache_store(f.ctx, &fc, f.hidden, f.n_rows_per_seq, f.base_pos, f.n_store, f.stream));
}
static PyObject* py_fetch(FAST) {
  (void)self;
  Frame2 f = {0};
  vvs_fcache fc;
  if (PARSE("vvs_feature_cache_fetch", fetch_params, N(fetch_params)) < 0 || fcache_of(f.fc, &fc) < 0) return NULL;
  CALL("vvs_feature_cache_fetch", vvs_feature_cache_fetch(f.ctx, &fc, f.skip_mask, f.n_images, f.gamma, f.gamma_max, f.staleness,
                                                          f.out, f.out_pos, f.stream));
}
static PyObject* py_skip(FAST) {
  (void)self;
  Frame2 f = {0};
  int32_t d[3], e[2];
  void *paths, *codebook;
  if (PARSE("vvs_skip_decide", skip_params, N(skip_params)) < 0 || shape_of(f.paths, 3, d) < 0 || shape_of(f.codebook, 2, e) < 0 ||
      to_ptr(f.paths, &paths) < 0 || to_ptr(f.codebook, &codebook) < 0)
    return NULL;
  CALL("vvs_skip_decide", vvs_skip_decide(f.ctx, paths, f.path_len, d[0], d[1], d[2], codebook, e[0], e[1], f.last_verified,
                                          f.stride, f.alpha, f.threshold, f.decision, f.similarity, f.stream));
}
static PyObject* py_select(FAST) {
  (void)self;
  Frame2 f = {0};
  int32_t d[3];
  void* paths;
  if (PARSE("vvs_select_unverified", select_params, N(select_params)) < 0 || shape_of(f.paths, 3, d) < 0 ||
      to_ptr(f.paths, &paths) < 0)
    return NULL;
  CALL("vvs_select_unverified", vvs_select_unverified(f.ctx, paths, f.path_len, d[0], d[1], d[2], f.uniforms, f.out_path,
                                                      f.out_gamma, f.out_tokens, f.stream));
}

/* setup(VvsError, current_raw_stream, current_device) */
static PyObject* py_setup(PyObject* self, PyObject* args) {
  (void)self;
  PyObject *e, *r, *d;
  if (!PyArg_ParseTuple(args, "OOO", &e, &r, &d)) return NULL;
  Py_XSETREF(g_error, Py_NewRef(e));
  Py_XSETREF(g_raw_stream, Py_NewRef(r));
  Py_XSETREF(g_get_device, Py_NewRef(d));
  Py_RETURN_NONE;
}

#define FN(name, f, doc) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL | METH_KEYWORDS, doc}
static PyMethodDef methods[] = {
    {"setup", py_setup, METH_VARARGS, NULL},
    FN("vvs_verify", py_verify, "vvs_verify(ctx, **fields of vvs_verify_args and vvs_verify_out, stream=None): one verification step."),
    FN("vvs_epilogue", py_epilogue, "LM head and decisions on given features."),
    FN("vvs_decide", py_decide, "Decisions on given target probabilities."),
    FN("vvs_decide_noalloc", py_decide_noalloc,
       "vvs_decide for callers that must not allocate device memory: no context (limits: 64 images, 16 drafts, 64 "
       "neighbours, vocab 65536; chains only: tree_parent / accept_path are refused)."),
    FN("vvs_feature_cache_reset", py_reset, "vvs_feature_cache_reset(ctx, fc, stream=None)"),
    FN("vvs_feature_cache_store", py_store, "vvs_feature_cache_store(ctx, fc, hidden, n_rows_per_seq, base_pos, n_store, stream=None)"),
    FN("vvs_feature_cache_fetch", py_fetch,
       "vvs_feature_cache_fetch(ctx, fc, skip_mask, n_images, gamma, gamma_max, staleness, out, out_pos, stream=None)"),
    FN("vvs_skip_decide", py_skip,
       "Alg. 1 / Eq. 2 of the paper: vvs_skip_decide(ctx, paths, path_len, codebook, last_verified, stride, alpha, threshold, "
       "decision, similarity, stream=None); paths int32 [B, N, L], path_len int32 [B, N] or None, codebook float32 [V, dim], "
       "last_verified uint8 [B] or None -> decision uint8 [B], similarity float32 [B]."),
    FN("vvs_select_unverified", py_select,
       "Sec. 4.2 / Eq. 3: uniform draw of one candidate path per image, cut to gamma tokens: vvs_select_unverified(ctx, paths, "
       "path_len, uniforms, out_path, out_gamma, out_tokens, stream=None)."),
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

static int intern(Param* ps, int n) {
  for (int i = 0; i < n; ++i)
    if (!(ps[i].key = PyUnicode_InternFromString(ps[i].name))) return -1;
  return 0;
}
PyMODINIT_FUNC PyInit__native(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_shape = PyUnicode_InternFromString("shape");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
#define I(ps) intern(ps, N(ps)) < 0
  if (!s_data_ptr || !s_shape || !s_cuda_stream || I(verify_params) || I(epilogue_params) || I(decide_params) || I(noalloc_params) ||
      I(reset_params) || I(store_params) || I(fetch_params) || I(skip_params) || I(select_params))
    return NULL;
  return PyModule_Create(&module);
}
