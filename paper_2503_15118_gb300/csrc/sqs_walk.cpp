// Walks a gate list (workloads.py's tuples) and issues each gate through the C
// ABI, in native code: State.run() of a 200-gate circuit on a small state spent
// 2.5 us a gate on tuple unpacking and ctypes marshalling against about 0.5 us
// on the call itself.
//
// Only plain values are taken here -- exact ints, floats, tuples or lists of
// them, tables already on the device.  Anything else (a numpy integer, a matrix,
// a table's first use, a malformed gate) is left to the binding's Python code,
// which converts it, or refuses it, as it always did: run() returns its index.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstring>

#include "../../include/sqs.h"

namespace {

// One gate's arguments; `ok` turns false at the first value not taken here.
struct Args {
  PyObject* g;
  Py_ssize_t n;
  bool ok = true;

  PyObject* at(Py_ssize_t i) {
    if (i < n) return PyTuple_GET_ITEM(g, i);
    ok = false;
    return nullptr;
  }
  bool integer(PyObject* o, long long& v) {
    if (!ok || !o || !PyLong_CheckExact(o)) return ok = false;
    int over = 0;
    v = PyLong_AsLongLongAndOverflow(o, &over);
    return ok = over == 0;
  }
  uint32_t u32(Py_ssize_t i) {
    long long v = 0;
    integer(at(i), v);
    return (uint32_t)v;  // as ctypes converts it
  }
  uint64_t u64(Py_ssize_t i) {
    PyObject* o = at(i);
    if (!ok || !PyLong_CheckExact(o)) {
      ok = false;
      return 0;
    }
    return PyLong_AsUnsignedLongLongMask(o);
  }
  double real(Py_ssize_t i) {
    PyObject* o = at(i);
    if (!ok || !PyFloat_Check(o)) {
      ok = false;
      return 0.0;
    }
    return PyFloat_AS_DOUBLE(o);
  }
  // Controls or predicates: at most `most` of them into c; their number.
  uint32_t ctrls(Py_ssize_t i, sqs_ctrl* c, Py_ssize_t most) {
    PyObject* o = at(i);
    if (!ok || !(PyTuple_CheckExact(o) || PyList_CheckExact(o))) {
      ok = false;
      return 0;
    }
    const Py_ssize_t m = PySequence_Fast_GET_SIZE(o);
    if (m > most) {
      ok = false;
      return 0;
    }
    for (Py_ssize_t k = 0; k < m; ++k) {
      PyObject* t = PySequence_Fast_GET_ITEM(o, k);
      if (!PyTuple_CheckExact(t) || PyTuple_GET_SIZE(t) < 2) {
        ok = false;
        return 0;
      }
      long long v[3] = {0, 0, 1};
      const Py_ssize_t w = PyTuple_GET_SIZE(t) > 2 ? 3 : 2;
      for (Py_ssize_t q = 0; q < w; ++q)
        if (!integer(PyTuple_GET_ITEM(t, q), v[q])) return 0;
      c[k].reg = (uint32_t)v[0];
      c[k].bit = (uint32_t)v[1];
      c[k].value = (uint32_t)v[2];
    }
    return (uint32_t)m;
  }
};

// The library may wait for the device, and its allocator calls back into
// Python: the interpreter lock is released around every call.
template <class F>
sqs_status call(F f) {
  sqs_status s;
  Py_BEGIN_ALLOW_THREADS
  s = f();
  Py_END_ALLOW_THREADS
  return s;
}

// Issues one gate; false when it is not taken here.
bool issue(sqs_state* st, PyObject* g, PyObject* tables, sqs_status& s) {
  if (!PyTuple_CheckExact(g) || PyTuple_GET_SIZE(g) < 1) return false;
  Args a{g, PyTuple_GET_SIZE(g)};
  PyObject* name = PyTuple_GET_ITEM(g, 0);
  if (!PyUnicode_CheckExact(name)) return false;
  const char* op = PyUnicode_AsUTF8(name);
  if (!op) {
    PyErr_Clear();
    return false;
  }
  auto is = [&](const char* x) { return std::strcmp(op, x) == 0; };
  sqs_ctrl c[SQS_MAX_PRED];
  sqs_perm_op p;
  std::memset(&p, 0, sizeof(p));
  bool perm = false;
  if (is("h")) {
    const uint32_t r = a.u32(1), b = a.u32(2), n = a.ctrls(3, c, SQS_MAX_PRED);
    if (!a.ok) return false;
    s = call([&] { return sqs_apply_h(st, r, b, c, n); });
  } else if (is("ry")) {
    const uint32_t r = a.u32(1), b = a.u32(2);
    const double th = a.real(3);
    const uint32_t n = a.ctrls(4, c, SQS_MAX_PRED);
    if (!a.ok) return false;
    s = call([&] { return sqs_apply_ry(st, r, b, th, c, n); });
  } else if (is("ry_reg")) {
    const uint32_t r = a.u32(1), b = a.u32(2), ang = a.u32(3);
    const double scale = a.real(4), offset = a.real(5);
    const uint32_t n = a.ctrls(6, c, SQS_MAX_PRED);
    if (!a.ok) return false;
    s = call([&] { return sqs_apply_ry_reg(st, r, b, ang, scale, offset, c, n); });
  } else if (is("phase")) {
    const uint32_t n = a.ctrls(1, c, SQS_MAX_PRED);
    const double phi = a.real(2);
    if (!a.ok) return false;
    s = call([&] { return sqs_apply_phase(st, c, n, phi); });
  } else if (is("x")) {
    perm = true;
    p.kind = SQS_PERM_X;
    p.reg = a.u32(1);
    p.bit = a.u32(2);
    p.n_ctrl = a.ctrls(3, p.ctrl, SQS_MAX_CTRL);
  } else if (is("add") || is("sub")) {
    perm = true;
    p.reg = a.u32(1);
    long long src = 0;
    if (!a.integer(a.at(2), src)) return false;
    if (src >= 0) {
      p.kind = op[0] == 'a' ? SQS_PERM_ADD_REG : SQS_PERM_SUB_REG;
      p.src_reg = (uint32_t)src;
    } else {
      p.kind = op[0] == 'a' ? SQS_PERM_ADD_CONST : SQS_PERM_SUB_CONST;
      p.constant = a.u64(3);
    }
    p.n_ctrl = a.ctrls(4, p.ctrl, SQS_MAX_CTRL);
  } else if (is("swap")) {
    perm = true;
    p.kind = SQS_PERM_SWAP;
    p.reg = a.u32(1);
    p.src_reg = a.u32(2);
    p.n_ctrl = a.ctrls(3, p.ctrl, SQS_MAX_CTRL);
  } else if (is("muladd") || is("divxor")) {
    perm = true;
    p.kind = op[0] == 'm' ? SQS_PERM_MUL_ADD : SQS_PERM_DIV_XOR;
    p.reg = a.u32(1);
    p.src_reg = a.u32(2);
    p.src2_reg = a.u32(3);
    p.n_ctrl = a.ctrls(4, p.ctrl, SQS_MAX_CTRL);
  } else if (is("mulc")) {
    perm = true;
    p.kind = SQS_PERM_MUL_CONST;
    p.reg = a.u32(1);
    p.constant = a.u64(2);
    p.n_ctrl = a.ctrls(3, p.ctrl, SQS_MAX_CTRL);
  } else if (is("qload") || is("qunload")) {
    const bool load = op[1] == 'l';
    PyObject* addr = a.at(1);
    const uint32_t data = a.u32(2);
    long long first = 0, count = 1, ti = 0;
    if (!a.ok || !a.integer(a.at(3), ti)) return false;
    const bool span = PyTuple_CheckExact(addr);
    if (span) {
      if (PyTuple_GET_SIZE(addr) != 2 || !a.integer(PyTuple_GET_ITEM(addr, 0), first) ||
          !a.integer(PyTuple_GET_ITEM(addr, 1), count))
        return false;
    } else if (!a.integer(addr, first)) {
      return false;
    }
    if (ti < 0 || ti >= PyList_GET_SIZE(tables)) return false;
    PyObject* h = PyList_GET_ITEM(tables, (Py_ssize_t)ti);
    if (!PyLong_CheckExact(h)) return false;  // not on the device yet
    const sqs_table* t = (const sqs_table*)PyLong_AsVoidPtr(h);
    s = call([&] {
      if (span)
        return load ? sqs_qram_load_span(st, (uint32_t)first, (uint32_t)count, data, t)
                    : sqs_qram_unload_span(st, (uint32_t)first, (uint32_t)count, data, t);
      return load ? sqs_qram_load(st, (uint32_t)first, data, t)
                  : sqs_qram_unload(st, (uint32_t)first, data, t);
    });
  } else if (is("prune")) {
    const double eps = a.real(1);
    if (!a.ok) return false;
    s = call([&] { return sqs_prune(st, eps, nullptr); });
  } else {
    return false;
  }
  if (perm) {
    if (!a.ok) return false;
    s = call([&] { return sqs_apply_perm(st, &p, 1); });
  }
  return true;
}

// run(handle, gates, first, tables) -> (index, status): issues gates[first:]
// until one is not taken here or fails; index is that gate's (len(gates) when
// all were issued), status the failing call's (0 otherwise).  gates: a list or
// tuple; tables: a list of device table handles, None where there is none yet.
PyObject* run(PyObject*, PyObject* args) {
  unsigned long long handle;
  PyObject *gates, *tables;
  Py_ssize_t first;
  if (!PyArg_ParseTuple(args, "KOnO!", &handle, &gates, &first, &PyList_Type, &tables))
    return nullptr;
  if (!PyList_CheckExact(gates) && !PyTuple_CheckExact(gates)) {
    PyErr_SetString(PyExc_TypeError, "gates: a list or a tuple");
    return nullptr;
  }
  sqs_state* const st = (sqs_state*)(uintptr_t)handle;
  Py_ssize_t i = first;
  sqs_status s = SQS_OK;
  // The list may change while the lock is released: its length is read anew.
  for (; i < PySequence_Fast_GET_SIZE(gates); ++i) {
    PyObject* g = PySequence_Fast_GET_ITEM(gates, i);
    Py_INCREF(g);
    const bool taken = issue(st, g, tables, s);
    Py_DECREF(g);
    if (!taken || s != SQS_OK) break;
    if ((i & 255) == 255 && PyErr_CheckSignals() < 0) return nullptr;
  }
  return Py_BuildValue("(ni)", i, (int)s);
}

PyMethodDef kMethods[] = {{"run", run, METH_VARARGS, "Issues a gate list (see the source)."},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "sqs_walk", nullptr, -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_sqs_walk(void) { return PyModule_Create(&kModule); }
