// Python side of epara_collect without ctypes.  A serving loop asks once per request, so that a step of forty small requests
// spends as long in the foreign-function call (0.8 us an answer) as in everything else it does on the host; here an answer is
// 0.4 us, the library's own work included.  (Two small MLPs, 8 + 32 requests: 72 us a step through ctypes, 52 like this.)
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>

namespace {

struct Collect {
  int (*fn)(void* ctx, uint64_t ticket, void* out);
  int (*ready)(void* ctx, uint64_t ticket, void* out);   // the same for answers that are there already
  int pending;           // its answer for the others
  PyObject* out_type;    // the ctypes structure that an answer is returned in
  PyObject* general;     // the same method through ctypes, for calls of any other form
  PyObject* handle;      // name of the attribute that holds the context's address as an int
};

void free_collect(PyObject* capsule) {
  Collect* c = static_cast<Collect*>(PyCapsule_GetPointer(capsule, nullptr));
  if (!c) return;
  Py_XDECREF(c->out_type);
  Py_XDECREF(c->general);
  Py_XDECREF(c->handle);
  PyMem_Free(c);
}

// (status, Output) = self.epara_collect(ticket)
PyObject* collect(PyObject* capsule, PyObject* const* args, Py_ssize_t n, PyObject* names) {
  Collect* c = static_cast<Collect*>(PyCapsule_GetPointer(capsule, nullptr));
  if (!c) return nullptr;
  if (n != 2 || names || !PyLong_CheckExact(args[1])) return PyObject_Vectorcall(c->general, args, n, names);
  PyObject* h = PyObject_GetAttr(args[0], c->handle);
  if (!h) return nullptr;
  const uint64_t ctx = PyLong_AsUnsignedLongLong(h);
  Py_DECREF(h);
  if (ctx == (uint64_t)-1 && PyErr_Occurred()) return nullptr;
  const uint64_t ticket = PyLong_AsUnsignedLongLongMask(args[1]);
  if (ticket == (uint64_t)-1 && PyErr_Occurred()) return nullptr;
  PyObject* out = PyObject_CallNoArgs(c->out_type);
  if (!out) return nullptr;
  Py_buffer view;
  if (PyObject_GetBuffer(out, &view, PyBUF_WRITABLE) < 0) { Py_DECREF(out); return nullptr; }
  // An answer that is there already is a look into a table.  For the others, usually a step's first, the library asks the CUDA driver
  // whether the step is through, and the driver's own lock can be held by another thread's launches: without the interpreter lock
  // then, as ctypes does it.  (Letting it go for every answer: two small MLPs 38.3 -> 40.7 us a step.)
  int status = c->ready(reinterpret_cast<void*>(static_cast<uintptr_t>(ctx)), ticket, view.buf);
  if (status == c->pending) {
    Py_BEGIN_ALLOW_THREADS
    status = c->fn(reinterpret_cast<void*>(static_cast<uintptr_t>(ctx)), ticket, view.buf);
    Py_END_ALLOW_THREADS
  }
  PyBuffer_Release(&view);
  PyObject* s = PyLong_FromLong(status);
  PyObject* r = s ? PyTuple_New(2) : nullptr;
  if (!r) { Py_XDECREF(s); Py_DECREF(out); return nullptr; }
  PyTuple_SET_ITEM(r, 0, s);
  PyTuple_SET_ITEM(r, 1, out);
  return r;
}

PyMethodDef collect_def = {"epara_collect", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(collect)), METH_FASTCALL | METH_KEYWORDS,
                           "(status, Output) of a ticket"};

// collect_method(addresses of epara_collect and epara_collect_ready, EPARA_PENDING, Output, general, name of the handle's attribute)
// -> method for the context class
PyObject* collect_method(PyObject*, PyObject* args) {
  unsigned long long fn, ready;
  int pending;
  PyObject *out_type, *general, *handle;
  if (!PyArg_ParseTuple(args, "KKiOOU", &fn, &ready, &pending, &out_type, &general, &handle)) return nullptr;
  Collect* c = static_cast<Collect*>(PyMem_Malloc(sizeof(Collect)));
  if (!c) return PyErr_NoMemory();
  c->fn = reinterpret_cast<int (*)(void*, uint64_t, void*)>(static_cast<uintptr_t>(fn));
  c->ready = reinterpret_cast<int (*)(void*, uint64_t, void*)>(static_cast<uintptr_t>(ready));
  c->pending = pending;
  c->out_type = Py_NewRef(out_type);
  c->general = Py_NewRef(general);
  c->handle = Py_NewRef(handle);
  PyObject* capsule = PyCapsule_New(c, nullptr, free_collect);
  if (!capsule) { Py_DECREF(out_type); Py_DECREF(general); Py_DECREF(handle); PyMem_Free(c); return nullptr; }
  PyObject* f = PyCFunction_New(&collect_def, capsule);
  Py_DECREF(capsule);
  if (!f) return nullptr;
  PyObject* m = PyInstanceMethod_New(f);          // (a builtin does not bind to the instance by itself)
  Py_DECREF(f);
  return m;
}

PyMethodDef methods[] = {{"collect_method", collect_method, METH_VARARGS, "epara_collect as a method of the context class"}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall(void) { return PyModule_Create(&module); }
