/* CPython module behind paper_2605_14877_b200/sweep.py: issues the C-ABI calls of a generation in order.  Pure call
 * sequencing, as the Python it replaces: a call cost 9 us from Python through ctypes (3.5 of them the launch), which bound
 * small images; from here 5. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <limits.h>

#include "heatkv.h"

static PyObject *s_data_ptr, *s_stride;

/* Interned callables of the process: (heatkv._check, torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream). */
typedef struct {
  PyObject *check, *device, *raw_stream;
} Hooks;
static Hooks hooks;

static int fail(int rc, const char* where) {
  PyObject* r = PyObject_CallFunction(hooks.check, "is", rc, where);      /* raises HeatKVError */
  Py_XDECREF(r);
  if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, where);
  return -1;
}

static int current_stream(void** out) {
  if (!hooks.check) {
    PyErr_SetString(PyExc_RuntimeError, "set_hooks has not been called");
    return -1;
  }
  PyObject* dev = PyObject_CallNoArgs(hooks.device);
  if (!dev) return -1;
  PyObject* st = PyObject_CallOneArg(hooks.raw_stream, dev);
  Py_DECREF(dev);
  if (!st) return -1;
  *out = PyLong_AsVoidPtr(st);
  Py_DECREF(st);
  return PyErr_Occurred() ? -1 : 0;
}

/* device address of a tensor (or the address itself) */
static int data_ptr(PyObject* t, char** out) {
  PyObject* v = PyLong_Check(t) ? Py_NewRef(t) : PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

/* the first three strides of a [n_seq, H, tokens, d] tensor whose d axis is contiguous */
static int strides(PyObject* t, int64_t* seq, int64_t* head, int64_t* tok) {
  PyObject* v = PyObject_CallMethodNoArgs(t, s_stride);
  if (!v) return -1;
  int ok = PyTuple_Check(v) && PyTuple_GET_SIZE(v) == 4;
  if (ok) {
    *seq = PyLong_AsLongLong(PyTuple_GET_ITEM(v, 0));
    *head = PyLong_AsLongLong(PyTuple_GET_ITEM(v, 1));
    *tok = PyLong_AsLongLong(PyTuple_GET_ITEM(v, 2));
    ok = PyLong_AsLongLong(PyTuple_GET_ITEM(v, 3)) == 1;
  }
  Py_DECREF(v);
  if (PyErr_Occurred()) return -1;
  if (!ok) PyErr_SetString(PyExc_AssertionError, "activations are [n_seq, H, tokens, d] with d contiguous");
  return ok ? 0 : -1;
}

/* Attention of one layer at one step and its cache update; `lo` = first token of the step on the token axis. */
static int layer_step(heatkv_ctx* ctx, const int* ids, int n_seq, int layer, int step, int64_t lo, PyObject* q, PyObject* k,
                      PyObject* v, PyObject* out, PyObject* bias, int fused) {
  heatkv_strides st;
  char *qp, *kp, *vp, *op, *bp = NULL;
  void* stream;
  if (strides(q, &st.q_seq, &st.q_head, &st.q_tok) || strides(k, &st.kv_seq, &st.kv_head, &st.kv_tok) ||
      strides(out, &st.o_seq, &st.o_head, &st.o_tok) || data_ptr(q, &qp) || data_ptr(k, &kp) || data_ptr(v, &vp) ||
      data_ptr(out, &op) || (bias != Py_None && data_ptr(bias, &bp)) || current_stream(&stream))
    return -1;
  qp += 2 * lo * st.q_tok;
  kp += 2 * lo * st.kv_tok;
  vp += 2 * lo * st.kv_tok;
  op += 2 * lo * st.o_tok;
  int rc;
  const char* where;
  Py_BEGIN_ALLOW_THREADS
  if (fused) {
    where = "heatkv_attention_append";
    rc = heatkv_attention_append(ctx, ids, n_seq, layer, step, qp, kp, vp, &st, (const float*)bp, op, stream);
  } else {
    where = "heatkv_scale_attention";
    rc = heatkv_scale_attention(ctx, ids, n_seq, layer, step, qp, kp, vp, &st, (const float*)bp, op, stream);
    if (rc == HEATKV_OK) {
      where = "heatkv_append_compact";
      rc = heatkv_append_compact(ctx, ids, n_seq, layer, step, kp, vp, &st, stream);
    }
  }
  Py_END_ALLOW_THREADS
  return rc == HEATKV_OK ? 0 : fail(rc, where);
}

/* a context handle: None (a closed session) is the library's to refuse */
static int parse_ctx(PyObject* v, void* out) {
  void* p = v == Py_None ? NULL : PyLong_AsVoidPtr(v);
  if (PyErr_Occurred()) return 0;
  *(heatkv_ctx**)out = (heatkv_ctx*)p;
  return 1;
}

/* sequence ids of a call, anything int() takes; a batch past the limit keeps its length and is the library's to refuse */
static int parse_ids(PyObject* seq, int* ids, int* n) {
  PyObject* f = PySequence_Fast(seq, "seq_ids must be a sequence");
  if (!f) return -1;
  const Py_ssize_t m = PySequence_Fast_GET_SIZE(f);
  for (Py_ssize_t i = 0; i < m && i < HEATKV_MAX_BATCH; ++i) {
    PyObject* v = PyNumber_Long(PySequence_Fast_GET_ITEM(f, i));
    if (!v) break;
    ids[i] = (int)PyLong_AsLong(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) break;
  }
  Py_DECREF(f);
  *n = m < INT_MAX ? (int)m : INT_MAX;
  return PyErr_Occurred() ? -1 : 0;
}

static PyObject* py_run_layer_step(PyObject* self, PyObject* args) {
  heatkv_ctx* ctx;
  int layer, step, fused, n;
  long long lo;
  PyObject *seq, *q, *k, *v, *out, *bias;
  int ids[HEATKV_MAX_BATCH];
  if (!PyArg_ParseTuple(args, "O&OiiLOOOOOp", parse_ctx, &ctx, &seq, &layer, &step, &lo, &q, &k, &v, &out, &bias, &fused)) return NULL;
  if (parse_ids(seq, ids, &n) || layer_step(ctx, ids, n, layer, step, lo, q, k, v, out, bias, fused))
    return NULL;
  Py_RETURN_NONE;
}

static PyObject* py_generate(PyObject* self, PyObject* args) {
  heatkv_ctx* c;
  int L, fused, n;
  PyObject *seq, *begins, *qkv_of, *out_of, *bias_of, *after;
  int ids[HEATKV_MAX_BATCH];
  if (!PyArg_ParseTuple(args, "O&OO!iOOOOp", parse_ctx, &c, &seq, &PyTuple_Type, &begins, &L, &qkv_of, &out_of, &bias_of, &after, &fused))
    return NULL;
  if (parse_ids(seq, ids, &n)) return NULL;
  const int K = (int)PyTuple_GET_SIZE(begins);
  for (int step = 0; step < K; ++step) {
    const int64_t lo = PyLong_AsLongLong(PyTuple_GET_ITEM(begins, step));
    void* stream;
    if (PyErr_Occurred() || current_stream(&stream)) return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = heatkv_append_compact(c, ids, n, -1, step, NULL, NULL, NULL, stream);
    Py_END_ALLOW_THREADS
    if (rc != HEATKV_OK) {
      fail(rc, "heatkv_append_compact");
      return NULL;
    }
    PyObject* py_step = PyLong_FromLong(step);
    if (!py_step) return NULL;
    for (int layer = 0; layer < L; ++layer) {
      int bad = 1;
      PyObject *py_layer = PyLong_FromLong(layer), *qkv = NULL, *fast = NULL, *out = NULL, *bias = NULL;
      if (py_layer && (qkv = PyObject_CallOneArg(qkv_of, py_layer)) &&
          (fast = PySequence_Fast(qkv, "qkv_of_layer returns (q, k, v)"))) {
        if (PySequence_Fast_GET_SIZE(fast) != 3) {
          PyErr_SetString(PyExc_ValueError, "qkv_of_layer returns (q, k, v)");
        } else {
          PyObject* lc[2] = {py_layer, py_step};
          if (bias_of == Py_None) {
            bias = Py_None;
            Py_INCREF(bias);
          } else {
            bias = PyObject_Vectorcall(bias_of, lc, 2, NULL);
          }
          if (bias && (out = PyObject_CallOneArg(out_of, py_layer)))
            bad = layer_step(c, ids, n, layer, step, lo, PySequence_Fast_GET_ITEM(fast, 0), PySequence_Fast_GET_ITEM(fast, 1),
                             PySequence_Fast_GET_ITEM(fast, 2), out, bias, fused);
          if (!bad && after != Py_None) {
            PyObject* sl[2] = {py_step, py_layer};
            PyObject* r = PyObject_Vectorcall(after, sl, 2, NULL);
            bad = r == NULL;
            Py_XDECREF(r);
          }
        }
      }
      Py_XDECREF(bias);
      Py_XDECREF(out);
      Py_XDECREF(fast);
      Py_XDECREF(qkv);
      Py_XDECREF(py_layer);
      if (bad) {
        Py_DECREF(py_step);
        return NULL;
      }
    }
    Py_DECREF(py_step);
  }
  Py_RETURN_NONE;
}

static PyObject* py_set_hooks(PyObject* self, PyObject* args) {
  Hooks h;
  if (!PyArg_ParseTuple(args, "OOO", &h.check, &h.device, &h.raw_stream)) return NULL;
  Py_INCREF(h.check);
  Py_INCREF(h.device);
  Py_INCREF(h.raw_stream);
  Py_XDECREF(hooks.check);
  Py_XDECREF(hooks.device);
  Py_XDECREF(hooks.raw_stream);
  hooks = h;
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"run_layer_step", py_run_layer_step, METH_VARARGS,
     "(ctx, seq_ids, layer, step, first_token, q, k, v, out, seg_bias | None, fused): one layer at one step"},
    {"generate", py_generate, METH_VARARGS,
     "(ctx, seq_ids, first_token_of_step, L, qkv_of_layer, out_of_layer, bias_of | None, after | None, fused): a whole sweep"},
    {"set_hooks", py_set_hooks, METH_VARARGS, "(check, current_device, raw_stream)"},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_stride = PyUnicode_InternFromString("stride");
  if (!s_data_ptr || !s_stride) return NULL;
  return PyModule_Create(&module);
}
