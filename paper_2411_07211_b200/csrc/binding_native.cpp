// Python entry points of the library: one callable object per routine.
//
// A call of a small problem is bound by the host: the kernel takes 1-2 us and its launch 2 us, while
// marshalling the arguments in Python (f-strings, ctypes conversions, torch.cuda.current_stream,
// a fresh context structure) took 6-7 us.  Here the arguments go from the interpreter's vector
// straight into the C call: converters are generated from the prototypes of b2blas.h, tensors give
// up their address, type and device without a Python-level call, the context structure is
// assembled from the fields of the Context object.  Measured at n = 65536 in float, nine level-1
// calls: 87 us before, 22-24 us now, 2.0 us of each call being the kernel launch.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <structmember.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <functional>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

#include "b2blas.h"

namespace {

constexpr int kMaxParams = 16;
PyObject* g_error_class = nullptr;   // B2Error
PyObject* g_ensure_loaded = nullptr; // binding.lib: loads the library or raises
PyObject* g_signature = nullptr;     // binding._signature: parameter names -> inspect.Signature
PyObject* g_lookup = nullptr;        // binding._routine: name -> callable (how a routine is pickled)
std::string g_lib_path;
void* g_lib = nullptr;

// ---- Context: the fields of b2_ctx that do not change from call to call ---------------------
struct ContextObject {
  PyObject_HEAD
  PyObject* status;  // int32 tensor
  unsigned long long ws_ptr, ws_bytes, wait_limit;
  int device;        // index of the device whose current stream the calls use
};

void context_dealloc(PyObject* self) {
  PyTypeObject* tp = Py_TYPE(self);
  PyObject_GC_UnTrack(self);
  Py_CLEAR(reinterpret_cast<ContextObject*>(self)->status);
  tp->tp_free(self);
  Py_DECREF(tp);
}
int context_traverse(PyObject* self, visitproc visit, void* arg) {
  Py_VISIT(reinterpret_cast<ContextObject*>(self)->status);
  Py_VISIT(Py_TYPE(self));
  return 0;
}
int context_clear(PyObject* self) {
  Py_CLEAR(reinterpret_cast<ContextObject*>(self)->status);
  return 0;
}
PyMemberDef context_members[] = {
    {"status", T_OBJECT_EX, offsetof(ContextObject, status), 0, nullptr},
    {"_ws_ptr", T_ULONGLONG, offsetof(ContextObject, ws_ptr), 0, nullptr},
    {"_ws_bytes", T_ULONGLONG, offsetof(ContextObject, ws_bytes), 0, nullptr},
    {"wait_limit", T_ULONGLONG, offsetof(ContextObject, wait_limit), 0, nullptr},
    {"_device_index", T_INT, offsetof(ContextObject, device), 0, nullptr},
    {nullptr, 0, 0, 0, nullptr}};
PyType_Slot context_slots[] = {{Py_tp_dealloc, (void*)context_dealloc},
                               {Py_tp_traverse, (void*)context_traverse},
                               {Py_tp_clear, (void*)context_clear},
                               {Py_tp_members, context_members},
                               {0, nullptr}};
PyType_Spec context_spec = {"paper_2411_07211_b200._binding.ContextBase", sizeof(ContextObject), 0,
                            Py_TPFLAGS_DEFAULT | Py_TPFLAGS_BASETYPE | Py_TPFLAGS_HAVE_GC, context_slots};
PyTypeObject* g_context_type = nullptr;

bool fill_ctx(PyObject* o, b2_ctx* c) {
  if (!PyObject_TypeCheck(o, g_context_type)) {
    PyErr_Format(PyExc_TypeError, "the first argument is a Context, got %.100s", Py_TYPE(o)->tp_name);
    return false;
  }
  const ContextObject* s = reinterpret_cast<ContextObject*>(o);
  if (s->status == nullptr || !THPVariable_Check(s->status)) {
    PyErr_SetString(PyExc_AttributeError, "the Context has no status tensor");
    return false;
  }
  c->stream = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)s->device).stream();
  c->workspace = reinterpret_cast<void*>(s->ws_ptr);
  c->workspace_bytes = (size_t)s->ws_bytes;
  c->device_status = static_cast<int*>(THPVariable_Unpack(s->status).data_ptr());
  c->wait_limit = s->wait_limit;
  return true;
}

// ---- argument converters --------------------------------------------------------------------
bool convert(PyObject* o, int64_t* v) {
  *v = PyLong_AsLongLong(o);
  return !(*v == -1 && PyErr_Occurred());
}
bool convert(PyObject* o, int* v) {
  const long t = PyLong_AsLong(o);
  *v = (int)t;
  return !(t == -1 && PyErr_Occurred());
}
bool convert(PyObject* o, double* v) {
  *v = PyFloat_AsDouble(o);
  return !(*v == -1.0 && PyErr_Occurred());
}
bool convert(PyObject* o, float* v) {
  const double t = PyFloat_AsDouble(o);
  *v = (float)t;
  return !(t == -1.0 && PyErr_Occurred());
}
// Tensors (their first element), None (a null pointer) or an address.
template <typename P>
bool convert(PyObject* o, P** v) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda()) {
      PyErr_SetString(PyExc_AssertionError, "b2blas routines take device tensors");
      return false;
    }
    *v = static_cast<P*>(t.data_ptr());
    return true;
  }
  if (o == Py_None) {
    *v = nullptr;
    return true;
  }
  *v = static_cast<P*>(PyLong_AsVoidPtr(o));
  return !(*v == nullptr && PyErr_Occurred());
}

// ---- calls ----------------------------------------------------------------------------------
// Calls recorded by prepare(): function, context and arguments as they were marshalled then, and
// the Python objects that own host memory among the arguments.
using Thunk = std::function<int()>;
struct Recording {
  std::vector<Thunk> calls;
  std::vector<PyObject*> keep;
  ~Recording() {
    for (PyObject* o : keep) Py_DECREF(o);
  }
};
// The recording that the calls of this thread go to.  (One per thread: prepare() runs Python code, other threads run in
// between, and their calls, or a second recording of theirs, are not this one's.)
thread_local Recording* t_recording = nullptr;

// args[0] is the context, args[1..] the arguments of the C function in order.  Returns false with
// a Python error set when an argument does not convert.
template <class... A, size_t... I>
bool call_typed(void* sym, PyObject* const* args, int* st, std::index_sequence<I...>) {
  using Fn = int (*)(const b2_ctx*, A...);
  const Fn fn = reinterpret_cast<Fn>(sym);
  b2_ctx c;
  if (!fill_ctx(args[0], &c)) return false;
  std::tuple<A...> a;
  if (!(convert(args[1 + I], &std::get<I>(a)) && ...)) return false;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = fn(&c, std::get<I>(a)...);
  Py_END_ALLOW_THREADS
  *st = rc;
  if (t_recording) t_recording->calls.emplace_back([fn, c, a]() { return fn(&c, std::get<I>(a)...); });
  return true;
}
template <class... A>
bool invoke(int (*)(const b2_ctx*, A...), void* sym, PyObject* const* args, int* st) {
  return call_typed<A...>(sym, args, st, std::index_sequence_for<A...>{});
}

// A routine of the table: parameter names (the context first), the parameter whose type picks the
// s or d symbol (-1: one symbol only), and the two symbols with their invokers.
struct RoutineDef {
  const char* name;
  const char* sym[2];
  bool (*run[2])(void*, PyObject* const*, int*);
  int type_of;
  const char* params;  // space-separated
  const char* doc;
};
#define B2_INVOKER(FN) +[](void* s, PyObject* const* a, int* st) { return invoke(static_cast<decltype(&FN)>(nullptr), s, a, st); }
#define B2_PAIR(S, D) {#S, #D}, {B2_INVOKER(S), B2_INVOKER(D)}
#define B2_ONE(S) {#S, nullptr}, {B2_INVOKER(S), nullptr}

const RoutineDef kRoutines[] = {
    {"axpy", B2_PAIR(b2_saxpy, b2_daxpy), 3, "ctx n alpha x incx y incy",
     "y <- alpha*x + y."},
    {"scal", B2_PAIR(b2_sscal, b2_dscal), 3, "ctx n alpha x incx",
     "x <- alpha*x."},
    {"copy", B2_PAIR(b2_scopy, b2_dcopy), 2, "ctx n x incx y incy",
     "y <- x."},
    {"swap", B2_PAIR(b2_sswap, b2_dswap), 2, "ctx n x incx y incy",
     "x <-> y."},
    {"rot", B2_PAIR(b2_srot, b2_drot), 2, "ctx n x incx y incy c s",
     "(x, y) <- (c*x + s*y, c*y - s*x)."},
    {"rotm", B2_PAIR(b2_srotm, b2_drotm), 2, "ctx n x incx y incy param",
     "Modified Givens rotation; param: the address of 5 host values."},
    {"dot", B2_PAIR(b2_sdot, b2_ddot), 2, "ctx n x incx y incy result",
     "result[0] <- sum of x*y."},
    {"dsdot", B2_ONE(b2_dsdot), -1, "ctx n x incx y incy result",
     "result[0] <- sum of x*y in double: float32 vectors, float64 device result."},
    {"sdsdot", B2_ONE(b2_sdsdot), -1, "ctx n sb x incx y incy result",
     "result[0] <- sb + sum of x*y, accumulated in double: float32 vectors and result."},
    {"asum", B2_PAIR(b2_sasum, b2_dasum), 2, "ctx n x incx result",
     "result[0] <- sum of |x|."},
    {"nrm2", B2_PAIR(b2_snrm2, b2_dnrm2), 2, "ctx n x incx result",
     "result[0] <- square root of the sum of x*x."},
    {"iamax", B2_PAIR(b2_isamax, b2_idamax), 2, "ctx n x incx result",
     "result[0] (int64) <- the first index, from 0, of the largest |x|."},
    {"gemv", B2_PAIR(b2_sgemv, b2_dgemv), 6, "ctx order trans m n alpha a lda x incx beta y incy",
     "y <- alpha*op(A)*x + beta*y, A m x n."},
    {"ger", B2_PAIR(b2_sger, b2_dger), 9, "ctx order m n alpha x incx y incy a lda",
     "A <- alpha*x*y^T + A, A m x n."},
    {"syr", B2_PAIR(b2_ssyr, b2_dsyr), 7, "ctx order uplo n alpha x incx a lda",
     "A <- alpha*x*x^T + A on the uplo triangle."},
    {"syr2", B2_PAIR(b2_ssyr2, b2_dsyr2), 9, "ctx order uplo n alpha x incx y incy a lda",
     "A <- alpha*(x*y^T + y*x^T) + A on the uplo triangle."},
    {"symv", B2_PAIR(b2_ssymv, b2_dsymv), 5, "ctx order uplo n alpha a lda x incx beta y incy",
     "y <- alpha*A*x + beta*y, A symmetric, its uplo triangle stored."},
    {"trmv", B2_PAIR(b2_strmv, b2_dtrmv), 6, "ctx order uplo trans diag n a lda x incx",
     "x <- op(A)*x, A triangular."},
    {"trsv", B2_PAIR(b2_strsv, b2_dtrsv), 6, "ctx order uplo trans diag n a lda x incx",
     "x <- the solution of op(A)*x = b, A triangular; b is passed in x."},
};

struct RoutineObject {
  PyObject_HEAD
  vectorcallfunc vectorcall;
  const RoutineDef* def;
  int nparams;                  // without `check`
  PyObject* names[kMaxParams];  // interned; `check` last
  void* fn[2];
};

bool resolve(RoutineObject* r) {
  if (g_lib == nullptr) {
    PyObject* ok = PyObject_CallNoArgs(g_ensure_loaded);
    if (ok == nullptr) return false;
    Py_DECREF(ok);
    g_lib = dlopen(g_lib_path.c_str(), RTLD_NOW | RTLD_LOCAL);
    if (g_lib == nullptr) {
      PyErr_Format(PyExc_ImportError, "%s: %s", g_lib_path.c_str(), dlerror());
      return false;
    }
  }
  for (int k = 0; k < 2; ++k)
    if (r->def->sym[k] != nullptr && (r->fn[k] = dlsym(g_lib, r->def->sym[k])) == nullptr) {
      PyErr_Format(PyExc_ImportError, "%s has no symbol %s", g_lib_path.c_str(), r->def->sym[k]);
      return false;
    }
  return true;
}

PyObject* raise_status(const char* name, int st) {
  PyObject* e = PyObject_CallFunction(g_error_class, "si", name, st);
  if (e != nullptr) {
    PyErr_SetObject(g_error_class, e);
    Py_DECREF(e);
  }
  return nullptr;
}

PyObject* routine_call(PyObject* self, PyObject* const* args, size_t nargsf, PyObject* kwnames) {
  RoutineObject* r = reinterpret_cast<RoutineObject*>(self);
  const int np = r->nparams;
  const Py_ssize_t npos = PyVectorcall_NARGS(nargsf);
  PyObject* v[kMaxParams + 1];
  if (npos > np + 1) {
    PyErr_Format(PyExc_TypeError, "%s() takes %d arguments, %zd were given", r->def->name, np + 1, npos);
    return nullptr;
  }
  for (Py_ssize_t i = 0; i < npos; ++i) v[i] = args[i];
  for (Py_ssize_t i = npos; i <= np; ++i) v[i] = nullptr;
  if (kwnames != nullptr) {
    const Py_ssize_t nk = PyTuple_GET_SIZE(kwnames);
    for (Py_ssize_t k = 0; k < nk; ++k) {
      PyObject* name = PyTuple_GET_ITEM(kwnames, k);
      int at = -1;
      for (int i = 0; i <= np && at < 0; ++i)
        if (r->names[i] == name) at = i;
      for (int i = 0; i <= np && at < 0; ++i)
        if (PyUnicode_Compare(r->names[i], name) == 0) at = i;
      if (at < 0 || v[at] != nullptr) {
        if (at < 0) PyErr_Format(PyExc_TypeError, "%s() got an unexpected argument '%U'", r->def->name, name);
        else PyErr_Format(PyExc_TypeError, "%s() got two values for '%U'", r->def->name, name);
        return nullptr;
      }
      v[at] = args[npos + k];
    }
  }
  for (int i = 0; i < np; ++i)
    if (v[i] == nullptr) {
      PyErr_Format(PyExc_TypeError, "%s() misses argument '%U'", r->def->name, r->names[i]);
      return nullptr;
    }
  int which = 0;
  if (r->def->type_of >= 0) {
    PyObject* t = v[r->def->type_of];
    if (!THPVariable_Check(t)) {
      PyErr_Format(PyExc_TypeError, "%s(): '%U' is a tensor", r->def->name, r->names[r->def->type_of]);
      return nullptr;
    }
    const at::ScalarType st = THPVariable_Unpack(t).scalar_type();
    if (st == at::kDouble) which = 1;
    else if (st != at::kFloat) {
      PyErr_Format(PyExc_TypeError, "b2blas supports float32/float64, got torch.%s", c10::toString(st));
      return nullptr;
    }
  }
  if (r->fn[which] == nullptr && !resolve(r)) return nullptr;
  int st = 0;
  try {
    if (!r->def->run[which](r->fn[which], v, &st)) return nullptr;
  } catch (const std::exception& e) {  // (a tensor without storage, no CUDA device)
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
  if (st != 0) {
    const int check = v[np] == nullptr ? 1 : PyObject_IsTrue(v[np]);
    if (check < 0) return nullptr;
    if (check) return raise_status(r->def->sym[which], st);
  }
  return PyLong_FromLong(st);
}

PyObject* routine_repr(PyObject* self) {
  const RoutineDef* d = reinterpret_cast<RoutineObject*>(self)->def;
  return PyUnicode_FromFormat("<b2blas routine %s(%s check=True)>", d->name, d->params);
}
void routine_dealloc(PyObject* self) {
  RoutineObject* r = reinterpret_cast<RoutineObject*>(self);
  for (int i = 0; i <= r->nparams; ++i) Py_CLEAR(r->names[i]);
  PyTypeObject* tp = Py_TYPE(self);
  tp->tp_free(self);
  Py_DECREF(tp);
}
// What a Python function has: name, module, docstring, signature, pickling by name.
PyObject* routine_doc(PyObject* self, void*) {
  const RoutineDef* d = reinterpret_cast<RoutineObject*>(self)->def;
  std::string head = std::string(d->name) + "(" + d->params + " check=True)";
  for (size_t i = 0; i < head.size(); ++i)
    if (head[i] == ' ') head.insert(i++, ",");
  return PyUnicode_FromFormat("%s\n\n%s  check: raise B2Error on a non-zero status instead of returning it.", head.c_str(), d->doc);
}
PyObject* routine_signature(PyObject* self, void*) { return PyObject_CallFunction(g_signature, "s", reinterpret_cast<RoutineObject*>(self)->def->params); }
PyObject* routine_reduce(PyObject* self, PyObject*) { return Py_BuildValue("O(s)", g_lookup, reinterpret_cast<RoutineObject*>(self)->def->name); }
PyMethodDef routine_methods[] = {{"__reduce__", routine_reduce, METH_NOARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyObject* routine_name(PyObject* self, void*) { return PyUnicode_FromString(reinterpret_cast<RoutineObject*>(self)->def->name); }
PyMemberDef routine_members[] = {{"__vectorcalloffset__", T_PYSSIZET, offsetof(RoutineObject, vectorcall), READONLY, nullptr},
                                 {nullptr, 0, 0, 0, nullptr}};
PyGetSetDef routine_getset[] = {{"__name__", routine_name, nullptr, nullptr, nullptr},
                                {"__qualname__", routine_name, nullptr, nullptr, nullptr},
                                {"__doc__", routine_doc, nullptr, nullptr, nullptr},
                                {"__signature__", routine_signature, nullptr, nullptr, nullptr},
                                {nullptr, nullptr, nullptr, nullptr, nullptr}};
PyType_Slot routine_slots[] = {{Py_tp_dealloc, (void*)routine_dealloc},
                               {Py_tp_call, (void*)PyVectorcall_Call},
                               {Py_tp_repr, (void*)routine_repr},
                               {Py_tp_members, routine_members},
                               {Py_tp_methods, routine_methods},
                               {Py_tp_getset, routine_getset},
                               {0, nullptr}};
PyType_Spec routine_spec = {"paper_2411_07211_b200._binding.Routine", sizeof(RoutineObject), 0,
                            Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL, routine_slots};
PyTypeObject* g_routine_type = nullptr;

// ---- prepare(): recorded calls --------------------------------------------------------------
struct ReplayObject {
  PyObject_HEAD
  vectorcallfunc vectorcall;
  Recording* rec;
};
PyObject* replay_call(PyObject* self, PyObject* const*, size_t, PyObject*) {
  int st = 0;
  const std::vector<Thunk>& calls = reinterpret_cast<ReplayObject*>(self)->rec->calls;
  Py_BEGIN_ALLOW_THREADS
  for (const Thunk& t : calls) st = t();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}
void replay_dealloc(PyObject* self) {
  delete reinterpret_cast<ReplayObject*>(self)->rec;
  PyTypeObject* tp = Py_TYPE(self);
  tp->tp_free(self);
  Py_DECREF(tp);
}
PyMemberDef replay_members[] = {{"__vectorcalloffset__", T_PYSSIZET, offsetof(ReplayObject, vectorcall), READONLY, nullptr},
                                {nullptr, 0, 0, 0, nullptr}};
PyType_Slot replay_slots[] = {{Py_tp_dealloc, (void*)replay_dealloc},
                              {Py_tp_call, (void*)PyVectorcall_Call},
                              {Py_tp_members, replay_members},
                              {0, nullptr}};
PyType_Spec replay_spec = {"paper_2411_07211_b200._binding.Replay", sizeof(ReplayObject), 0,
                           Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL, replay_slots};
PyTypeObject* g_replay_type = nullptr;

PyObject* record(PyObject*, PyObject* thunk) {
  Recording* const outer = t_recording;
  Recording* rec = new Recording();
  t_recording = rec;
  PyObject* r = PyObject_CallNoArgs(thunk);
  t_recording = outer;
  ReplayObject* o = r == nullptr ? nullptr : PyObject_New(ReplayObject, g_replay_type);
  Py_XDECREF(r);
  if (o == nullptr) {
    delete rec;
    return nullptr;
  }
  o->vectorcall = replay_call;
  o->rec = rec;
  return reinterpret_cast<PyObject*>(o);
}

// keep(obj): while a recording runs, obj lives as long as its replay (host memory that a recorded
// call points into).
PyObject* keep(PyObject*, PyObject* obj) {
  if (t_recording) t_recording->keep.push_back(Py_NewRef(obj));
  Py_RETURN_NONE;
}

// routines(lib_path, error_class, ensure_loaded, signature, lookup) -> {name: callable}
PyObject* routines(PyObject*, PyObject* args) {
  const char* path;
  PyObject *err, *ensure, *signature, *lookup;
  if (!PyArg_ParseTuple(args, "sOOOO", &path, &err, &ensure, &signature, &lookup)) return nullptr;
  g_lib_path = path;
  Py_XSETREF(g_error_class, Py_NewRef(err));
  Py_XSETREF(g_ensure_loaded, Py_NewRef(ensure));
  Py_XSETREF(g_signature, Py_NewRef(signature));
  Py_XSETREF(g_lookup, Py_NewRef(lookup));
  PyObject* out = PyDict_New();
  for (const RoutineDef& d : kRoutines) {
    RoutineObject* r = PyObject_New(RoutineObject, g_routine_type);
    if (r == nullptr) return nullptr;
    r->vectorcall = routine_call;
    r->def = &d;
    r->nparams = 0;
    r->fn[0] = r->fn[1] = nullptr;
    const char* p = d.params;
    while (*p) {
      const char* e = strchr(p, ' ');
      const size_t len = e ? (size_t)(e - p) : strlen(p);
      PyObject* s = PyUnicode_FromStringAndSize(p, (Py_ssize_t)len);
      PyUnicode_InternInPlace(&s);
      r->names[r->nparams++] = s;
      p += len + (e ? 1 : 0);
    }
    r->names[r->nparams] = PyUnicode_InternFromString("check");
    PyDict_SetItemString(out, d.name, reinterpret_cast<PyObject*>(r));
    Py_DECREF(r);
  }
  return out;
}

PyMethodDef methods[] = {{"routines", routines, METH_VARARGS, nullptr}, {"record", record, METH_O, nullptr},
                         {"keep", keep, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  g_context_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&context_spec));
  g_routine_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&routine_spec));
  g_replay_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&replay_spec));
  if (!g_context_type || !g_routine_type || !g_replay_type) return nullptr;
  PyObject* m = PyModule_Create(&module);
  if (m != nullptr) PyModule_AddObjectRef(m, "ContextBase", reinterpret_cast<PyObject*>(g_context_type));
  return m;
}
