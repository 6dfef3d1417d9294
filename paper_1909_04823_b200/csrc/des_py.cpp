// Argument marshalling for the calls of a step, in native code: Python tensors in, C ABI structs out.  Nothing is
// computed here.  (Through ctypes a call spends 6-10 us building structs and pointer objects, more than
// the small kernels behind it take; here it is about 1 us.)
//
// The C ABI is resolved from an already built library by path, so that the product and the checking library
// can be used side by side: open(path, batch class) -> capsule, then every function takes (capsule, table handle, ...).
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <string.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "des.h"

namespace {

struct Lib {
  decltype(&des_find_or_insert) find_or_insert;
  decltype(&des_forward_partials) forward_partials;
  decltype(&des_aggregate) aggregate;
  decltype(&des_forward_fused) forward_fused;
  decltype(&des_backward_update) backward_update;
  decltype(&des_head) head;
  decltype(&des_table_read_rows) read_rows;
  decltype(&des_table_write_rows) write_rows;
  decltype(&des_step_host) step_host;
  decltype(&des_step_host_submit) step_host_submit;
  decltype(&des_step_host_wait) step_host_wait;
  decltype(&des_dense1_get) dense1_get;
  decltype(&des_cross_forward) cross_forward;
  decltype(&des_cross_backward) cross_backward;
  decltype(&des_cross_workspace_floats) cross_workspace_floats;
  void* dl;
};

struct BadArgs {};                                     // thrown with the Python error already set

Lib* lib_of(PyObject* capsule) {
  Lib* l = (Lib*)PyCapsule_GetPointer(capsule, "des_lib");
  if (!l) throw BadArgs();
  return l;
}

void need(Py_ssize_t got, Py_ssize_t want) {
  if (got != want) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got); throw BadArgs(); }
}

long long as_int(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw BadArgs();
  return v;
}

float as_float(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw BadArgs();
  return (float)v;
}

des_table_t* table_of(PyObject* o) {                   // None: a closed table (the library answers INVALID_ARG)
  return o == Py_None ? nullptr : (des_table_t*)(uintptr_t)PyLong_AsUnsignedLongLong(o);
}

const at::Tensor& tensor_of(PyObject* o) {
  if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a tensor"); throw BadArgs(); }
  return THPVariable_Unpack(o);
}

const at::Tensor& matrix_of(PyObject* o) {              // as `B, d = x.shape` has it
  const at::Tensor& x = tensor_of(o);
  if (x.dim() != 2) { PyErr_Format(PyExc_ValueError, "expected a matrix, got %lld dimension(s)", (long long)x.dim()); throw BadArgs(); }
  return x;
}

long long method_int(PyObject* o, const char* name) {
  PyObject* v = PyObject_CallMethod(o, name, nullptr);
  if (!v) throw BadArgs();
  const unsigned long long r = PyLong_AsUnsignedLongLong(v);
  Py_DECREF(v);
  if (r == ~0ull && PyErr_Occurred()) throw BadArgs();
  return (long long)r;
}

// Memory is anything with data_ptr(): a tensor, a subclass that has its own idea of it, a storage, a caller's own class.
template <typename T>
T* ptr(PyObject* o) {
  if (o == Py_None) return nullptr;
  return THPVariable_CheckExact(o) ? (T*)THPVariable_Unpack(o).data_ptr() : (T*)(uintptr_t)method_int(o, "data_ptr");
}
int64_t numel_of(PyObject* o) { return THPVariable_CheckExact(o) ? THPVariable_Unpack(o).numel() : method_int(o, "numel"); }

void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

PyObject *s_batch, *s_nnz, *s_offsets, *s_ids, *s_vals, *s_rows, *s_shards, *s_uidx, *s_uniq_rows, *s_n_uniq;

template <typename T>
T* attr_ptr(PyObject* o, PyObject* name) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) throw BadArgs();
  T* p = nullptr;
  try { p = ptr<T>(v); } catch (...) { Py_DECREF(v); throw; }
  Py_DECREF(v);                                        // (the batch object keeps the tensor)
  return p;
}

long long attr_int(PyObject* o, PyObject* name) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) throw BadArgs();
  const long long r = PyLong_AsLongLong(v);
  Py_DECREF(v);
  if (r == -1 && PyErr_Occurred()) throw BadArgs();
  return r;
}

PyObject* batch_type;                                  // binding.DeviceBatch

// A batch of the binding's own class is read by its attributes; one of any other class builds its struct itself (c(), a
// ctypes structure: 3 us).
des_batch_t batch_of(PyObject* o) {
  des_batch_t b;
  if ((PyObject*)Py_TYPE(o) != batch_type) {
    PyObject* c = PyObject_CallMethod(o, "c", nullptr);
    if (!c) throw BadArgs();
    Py_buffer v;
    const bool ok = PyObject_GetBuffer(c, &v, PyBUF_SIMPLE) == 0;
    const bool whole = ok && v.len == (Py_ssize_t)sizeof(b);
    if (whole) memcpy(&b, v.buf, sizeof(b));
    if (ok) PyBuffer_Release(&v);
    Py_DECREF(c);
    if (ok && !whole) PyErr_SetString(PyExc_TypeError, "c() is not a des_batch_t");
    if (!whole) throw BadArgs();
    return b;
  }
  b.batch = (int32_t)attr_int(o, s_batch);
  b.nnz = attr_int(o, s_nnz);
  b.offsets = attr_ptr<int32_t>(o, s_offsets);
  b.ids = attr_ptr<uint64_t>(o, s_ids);
  b.vals = attr_ptr<float>(o, s_vals);
  b.rows = attr_ptr<uint32_t>(o, s_rows);
  b.shards = attr_ptr<uint8_t>(o, s_shards);
  b.uidx = attr_ptr<uint32_t>(o, s_uidx);
  b.uniq_rows = attr_ptr<uint32_t>(o, s_uniq_rows);
  b.n_uniq = attr_ptr<uint32_t>(o, s_n_uniq);
  return b;
}

template <typename F>
int unlocked(F&& call) {                               // a call of the library, without the interpreter lock
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = (int)call();
  Py_END_ALLOW_THREADS
  return rc;
}
template <typename F>
PyObject* status(F&& call) { return PyLong_FromLong(unlocked(call)); }

template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* a, Py_ssize_t n) {
  try {
    HANDLE_TH_ERRORS                                   // (torch's exceptions keep their types: torch.OutOfMemoryError, ...)
    return F(a, n);
    END_HANDLE_TH_ERRORS
  } catch (const BadArgs&) {
    return nullptr;
  }
}

PyObject* py_open(PyObject* const* a, Py_ssize_t n) {
  need(n, 2);                                          // (path, class of the binding's batches)
  const char* path = PyUnicode_AsUTF8(a[0]);
  if (!path) throw BadArgs();
  void* h = dlopen(path, RTLD_NOW | RTLD_LOCAL);
  if (!h) { PyErr_SetString(PyExc_OSError, dlerror()); throw BadArgs(); }
  Lib* l = new Lib();
  l->dl = h;
  bool ok = true;
#define SYM(field, name) ok &= (l->field = (decltype(l->field))dlsym(h, name)) != nullptr
  SYM(find_or_insert, "des_find_or_insert"); SYM(forward_partials, "des_forward_partials");
  SYM(aggregate, "des_aggregate"); SYM(forward_fused, "des_forward_fused");
  SYM(backward_update, "des_backward_update"); SYM(head, "des_head"); SYM(read_rows, "des_table_read_rows");
  SYM(write_rows, "des_table_write_rows"); SYM(step_host, "des_step_host");
  SYM(step_host_submit, "des_step_host_submit"); SYM(step_host_wait, "des_step_host_wait");
  SYM(dense1_get, "des_dense1_get"); SYM(cross_forward, "des_cross_forward");
  SYM(cross_backward, "des_cross_backward"); SYM(cross_workspace_floats, "des_cross_workspace_floats");
#undef SYM
  if (!ok) { delete l; PyErr_SetString(PyExc_OSError, "library lacks a symbol of the C ABI"); throw BadArgs(); }
  Py_INCREF(a[1]);
  Py_XSETREF(batch_type, a[1]);
  return PyCapsule_New(l, "des_lib", nullptr);         // lives as long as the process, like the library
}

// (lib, table, batch, insert)
PyObject* py_find_or_insert(PyObject* const* a, Py_ssize_t n) {
  need(n, 4);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const des_batch_t b = batch_of(a[2]);
  const int insert = PyObject_IsTrue(a[3]);
  if (insert < 0) throw BadArgs();
  void* st = stream();
  return status([&] { return l->find_or_insert(t, &b, insert, st); });
}

// (lib, table, ops, batch, part_small, pooled, part_pooled, part_dense)
PyObject* py_forward_partials(PyObject* const* a, Py_ssize_t n) {
  need(n, 8);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t ops = (uint32_t)as_int(a[2]);
  const des_batch_t b = batch_of(a[3]);
  const des_partials_t p = {ptr<float>(a[4]), ptr<float>(a[5]), ptr<float>(a[6]), ptr<float>(a[7])};
  void* st = stream();
  return status([&] { return l->forward_partials(t, ops, &b, &p, st); });
}

// (lib, table, ops, batch, part_small, pooled, part_pooled, part_dense, out_small, out_pooled, Z)
PyObject* py_aggregate(PyObject* const* a, Py_ssize_t n) {
  need(n, 11);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t ops = (uint32_t)as_int(a[2]);
  const des_batch_t b = batch_of(a[3]);
  const des_partials_t p = {ptr<float>(a[4]), ptr<float>(a[5]), ptr<float>(a[6]), ptr<float>(a[7])};
  const des_outputs_t o = {ptr<float>(a[8]), ptr<float>(a[9]), ptr<float>(a[10])};
  void* st = stream();
  return status([&] { return l->aggregate(t, ops, &b, &p, &o, st); });
}

// (lib, table, ops, batch, part_small, pooled, out_small, Z)
PyObject* py_forward_fused(PyObject* const* a, Py_ssize_t n) {
  need(n, 8);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t ops = (uint32_t)as_int(a[2]);
  const des_batch_t b = batch_of(a[3]);
  const des_partials_t p = {ptr<float>(a[4]), ptr<float>(a[5]), nullptr, nullptr};
  const des_outputs_t o = {ptr<float>(a[6]), ptr<float>(a[5]), ptr<float>(a[7])};
  void* st = stream();
  return status([&] { return l->forward_fused(t, ops, &b, &p, &o, st); });
}

// (lib, table, ops, batch, out_small, pooled, Z, gL, gF, gE, gZ, gE_work)
PyObject* py_backward_update(PyObject* const* a, Py_ssize_t n) {
  need(n, 12);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t ops = (uint32_t)as_int(a[2]);
  const des_batch_t b = batch_of(a[3]);
  const des_outputs_t o = {ptr<float>(a[4]), ptr<float>(a[5]), ptr<float>(a[6])};
  const des_grads_t g = {ptr<float>(a[7]), ptr<float>(a[8]), ptr<float>(a[9]), ptr<float>(a[10]), ptr<float>(a[11])};
  void* st = stream();
  return status([&] { return l->backward_update(t, ops, &b, &o, &g, st); });
}

// (lib, table, ops, batch size, b0, c_lr, c_fm, u, b1, q, d, out_small, pooled, Z, xdense, y, logit, loss, gL, gF, gE, gZ)
PyObject* py_head(PyObject* const* a, Py_ssize_t n) {
  need(n, 22);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t ops = (uint32_t)as_int(a[2]);
  const int32_t B = (int32_t)as_int(a[3]);
  des_head_t h;
  h.b0 = as_float(a[4]); h.c_lr = as_float(a[5]); h.c_fm = as_float(a[6]);
  h.u = ptr<float>(a[7]); h.b1 = ptr<float>(a[8]); h.q = ptr<float>(a[9]); h.d = ptr<float>(a[10]);
  h.n_dense = a[10] == Py_None ? 0 : (int32_t)numel_of(a[10]);
  const des_outputs_t o = {ptr<float>(a[11]), ptr<float>(a[12]), ptr<float>(a[13])};
  const float *xd = ptr<float>(a[14]), *y = ptr<float>(a[15]);
  float *logit = ptr<float>(a[16]), *loss = ptr<float>(a[17]);
  const des_head_grads_t g = {ptr<float>(a[18]), ptr<float>(a[19]), ptr<float>(a[20]), ptr<float>(a[21])};
  void* st = stream();
  return status([&] { return l->head(t, ops, B, &h, &o, xd, y, logit, loss, &g, st); });
}

// (lib, table, rows, k) -> (status, emb, lin, acc_emb, acc_lin)
PyObject* py_read_rows(PyObject* const* a, Py_ssize_t n) {
  need(n, 4);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t* r = ptr<uint32_t>(a[2]);
  const int64_t m = numel_of(a[2]), k = as_int(a[3]);
  const auto opt = at::TensorOptions().dtype(at::kFloat).device(at::kCUDA);
  at::Tensor emb = at::empty({m, k}, opt), lin = at::empty({m}, opt), ae = at::empty({m, k}, opt), al = at::empty({m}, opt);
  void* st = stream();
  float *pe = (float*)emb.data_ptr(), *pl = (float*)lin.data_ptr(), *pae = (float*)ae.data_ptr(), *pal = (float*)al.data_ptr();
  const int rc = unlocked([&] { return l->read_rows(t, r, m, pe, pl, pae, pal, st); });
  return Py_BuildValue("(iNNNN)", rc, THPVariable_Wrap(emb), THPVariable_Wrap(lin), THPVariable_Wrap(ae), THPVariable_Wrap(al));
}

// (lib, table, rows, emb, lin, acc_emb, acc_lin)
PyObject* py_write_rows(PyObject* const* a, Py_ssize_t n) {
  need(n, 7);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const uint32_t* r = ptr<uint32_t>(a[2]);
  const int64_t m = numel_of(a[2]);
  const float *emb = ptr<float>(a[3]), *lin = ptr<float>(a[4]), *ae = ptr<float>(a[5]), *al = ptr<float>(a[6]);
  void* st = stream();
  return status([&] { return l->write_rows(t, r, m, emb, lin, ae, al, st); });
}

struct HostStep {
  uint32_t ops; int32_t batch; int64_t nnz;
  const int32_t* offsets; const uint64_t* ids; const float* vals;
  float *out, *pooled, *Z;
  des_grads_t g;
};
// a[0..14]: ops, batch size, nnz, offsets, ids, vals, out_small, pooled, Z, gL, gF, gE, gZ, gE_work
HostStep host_step_of(PyObject* const* a) {
  HostStep s;
  s.ops = (uint32_t)as_int(a[0]); s.batch = (int32_t)as_int(a[1]); s.nnz = as_int(a[2]);
  s.offsets = ptr<int32_t>(a[3]); s.ids = ptr<uint64_t>(a[4]); s.vals = ptr<float>(a[5]);
  s.out = ptr<float>(a[6]); s.pooled = ptr<float>(a[7]); s.Z = ptr<float>(a[8]);
  s.g = {ptr<float>(a[9]), ptr<float>(a[10]), ptr<float>(a[11]), ptr<float>(a[12]), ptr<float>(a[13])};
  return s;
}

// (lib, table, <host step>)
PyObject* py_step_host(PyObject* const* a, Py_ssize_t n) {
  need(n, 16);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const HostStep s = host_step_of(a + 2);
  void* st = stream();
  return status([&] { return l->step_host(t, s.ops, s.batch, s.nnz, s.offsets, s.ids, s.vals, &s.g, s.pooled, s.Z, s.out, st); });
}

// (lib, table, <host step>) -> (status, ticket)
PyObject* py_step_host_submit(PyObject* const* a, Py_ssize_t n) {
  need(n, 16);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const HostStep s = host_step_of(a + 2);
  void* st = stream();
  int32_t ticket = -1;
  const int rc = unlocked([&] {
    return l->step_host_submit(t, s.ops, s.batch, s.nnz, s.offsets, s.ids, s.vals, &s.g, s.pooled, s.Z, s.out, st, &ticket);
  });
  return Py_BuildValue("(ii)", rc, (int)ticket);
}

// (lib, table, ticket)
PyObject* py_step_host_wait(PyObject* const* a, Py_ssize_t n) {
  need(n, 3);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  const int32_t ticket = (int32_t)as_int(a[2]);
  return status([&] { return l->step_host_wait(t, ticket); });
}

// (lib, table, F * k, H) -> (status, W1)
PyObject* py_dense1_get(PyObject* const* a, Py_ssize_t n) {
  need(n, 4);
  Lib* l = lib_of(a[0]);
  des_table_t* t = table_of(a[1]);
  at::Tensor w = at::empty({as_int(a[2]), as_int(a[3])}, at::TensorOptions().dtype(at::kFloat).device(at::kCUDA));
  float* pw = (float*)w.data_ptr();
  void* st = stream();
  const int rc = unlocked([&] { return l->dense1_get(t, pw, st); });
  return Py_BuildValue("(iN)", rc, THPVariable_Wrap(w));
}

// (lib, x0, x, w, b, shards, want_part) -> (status, y, P, part or None)
PyObject* py_cross_forward(PyObject* const* a, Py_ssize_t n) {
  need(n, 7);
  Lib* l = lib_of(a[0]);
  const at::Tensor& x = matrix_of(a[2]);
  const int64_t B = x.size(0), d = x.size(1), S = as_int(a[5]);
  const auto opt = at::TensorOptions().dtype(at::kFloat).device(x.device());
  at::Tensor y = at::empty_like(x), P = at::empty({B}, opt), part;
  const int want = PyObject_IsTrue(a[6]);
  if (want < 0) throw BadArgs();
  if (want) part = at::empty({S, B}, opt);
  const float *x0 = ptr<float>(a[1]), *px = ptr<float>(a[2]), *pw = ptr<float>(a[3]), *pb = ptr<float>(a[4]);
  float *pp = want ? (float*)part.data_ptr() : nullptr, *pP = (float*)P.data_ptr(), *py = (float*)y.data_ptr();
  void* st = stream();
  const int rc = unlocked([&] { return l->cross_forward((int32_t)B, (int32_t)d, (int32_t)S, x0, px, pw, pb, pp, pP, py, st); });
  if (want) return Py_BuildValue("(iNNN)", rc, THPVariable_Wrap(y), THPVariable_Wrap(P), THPVariable_Wrap(part));
  return Py_BuildValue("(iNNO)", rc, THPVariable_Wrap(y), THPVariable_Wrap(P), Py_None);
}

// (lib, x0, x, w, P, gY) -> (status, gx0, gx, gw, gb)
PyObject* py_cross_backward(PyObject* const* a, Py_ssize_t n) {
  need(n, 6);
  Lib* l = lib_of(a[0]);
  const at::Tensor& x = matrix_of(a[2]);
  const int64_t B = x.size(0), d = x.size(1);
  const auto opt = at::TensorOptions().dtype(at::kFloat).device(x.device());
  at::Tensor gx0 = at::empty_like(x), gx = at::empty_like(x), gw = at::empty({d}, opt), gb = at::empty({d}, opt);
  at::Tensor ws = at::empty({l->cross_workspace_floats((int32_t)B, (int32_t)d)}, opt);
  const float *x0 = ptr<float>(a[1]), *px = ptr<float>(a[2]), *pw = ptr<float>(a[3]), *pP = ptr<float>(a[4]), *pY = ptr<float>(a[5]);
  float *p0 = (float*)gx0.data_ptr(), *p1 = (float*)gx.data_ptr(), *p2 = (float*)gw.data_ptr(), *p3 = (float*)gb.data_ptr(),
        *p4 = (float*)ws.data_ptr();
  void* st = stream();
  const int rc = unlocked([&] { return l->cross_backward((int32_t)B, (int32_t)d, x0, px, pw, pP, pY, p0, p1, p2, p3, p4, st); });
  return Py_BuildValue("(iNNNN)", rc, THPVariable_Wrap(gx0), THPVariable_Wrap(gx), THPVariable_Wrap(gw), THPVariable_Wrap(gb));
}

#define FN(name) {#name, (PyCFunction)(void (*)(void))guarded<py_##name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FN(open), FN(find_or_insert), FN(forward_partials), FN(aggregate), FN(forward_fused),
                         FN(backward_update), FN(head), FN(read_rows), FN(write_rows), FN(step_host), FN(step_host_submit),
                         FN(step_host_wait), FN(dense1_get), FN(cross_forward), FN(cross_backward),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) {
  s_batch = PyUnicode_InternFromString("batch"); s_nnz = PyUnicode_InternFromString("nnz");
  s_offsets = PyUnicode_InternFromString("offsets"); s_ids = PyUnicode_InternFromString("ids");
  s_vals = PyUnicode_InternFromString("vals"); s_rows = PyUnicode_InternFromString("rows");
  s_shards = PyUnicode_InternFromString("shards"); s_uidx = PyUnicode_InternFromString("uidx");
  s_uniq_rows = PyUnicode_InternFromString("uniq_rows"); s_n_uniq = PyUnicode_InternFromString("n_uniq");
  return PyModule_Create(&module_def);
}
