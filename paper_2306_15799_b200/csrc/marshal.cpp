// Argument marshalling of the calls that short problems repeat: flurka_forward and flurka_backward on torch tensors.
//
// A short call's time is host time, and binding.py takes its tensors apart attribute by attribute and hands fifteen values to
// ctypes.  This module makes the same checks on the tensors themselves.  Calls in a loop, with the shared-memory limits raised
// once: forward, 2 heads x N = 1024, 32.6 -> 23.5 us; backward, RNN, 2 heads x N = 512, 45.0 -> 33.4 us.
// Whatever it does not recognise as a plain call (anything but exact torch tensors that fit together) it leaves to binding.py:
// it returns None, and the Python path accepts or refuses the call as it always has.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

typedef int (*ForwardFn)(const void*, const void*, const void*, const void*, const void*, const void*, int, int, int, int,
                         int, int, int, void*, void*);
typedef int (*BackwardFn)(const void*, const void*, const void*, const void*, const void*, const void*, const void*, int,
                          int, int, int, int, int, int, void*, void*, void*, void*, void*, void*);
ForwardFn g_forward = nullptr;
BackwardFn g_backward = nullptr;

constexpr int kPerformer = 0, kRnn = 1, kFp32 = 0x100, kBnhd = 0x200, kPerHead = 0x400;

struct Problem {
  const at::Tensor *Q, *K, *V, *E, *F, *W, *dO;
  int variant, B, H, N, d, k, m;
};

// What of a call may throw (addresses, the stream) is taken while the interpreter is held: an exception that left a block
// without it would be caught by code that uses the interpreter.
class WithoutInterpreter {
 public:
  WithoutInterpreter() : state_(PyEval_SaveThread()) {}
  ~WithoutInterpreter() { PyEval_RestoreThread(state_); }
  WithoutInterpreter(const WithoutInterpreter&) = delete;
  WithoutInterpreter& operator=(const WithoutInterpreter&) = delete;

 private:
  PyThreadState* state_;
};

// the tensor of an exact torch.Tensor on the device that Q is like: contiguous, on CUDA, of Q's type, with memory of its own
// (the wrapped tensors of torch.func's transforms have the type, device and strides of what they wrap, but no memory)
const at::Tensor* plain(PyObject* o, const at::Tensor* like) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.has_storage() || !t.is_cuda() || t.layout() != at::kStrided || !t.is_contiguous()) return nullptr;
  if (like && t.scalar_type() != like->scalar_type()) return nullptr;
  return &t;
}

// args: Q, K, V, E, F, W or None, variant (an int), bnhd (True or False)
bool parse(PyObject* const* a, Problem* p) {
  p->Q = plain(a[0], nullptr);
  if (!p->Q) return false;
  const at::Tensor& Q = *p->Q;
  if (!(p->K = plain(a[1], p->Q)) || !(p->V = plain(a[2], p->Q)) || !(p->E = plain(a[3], p->Q)) || !(p->F = plain(a[4], p->Q)))
    return false;
  const bool fp32 = Q.scalar_type() == at::kFloat;
  if (!fp32 && Q.scalar_type() != at::kBFloat16) return false;
  if (!PyLong_CheckExact(a[6])) return false;
  const long variant = PyLong_AsLong(a[6]);
  if (variant != kPerformer && variant != kRnn) { PyErr_Clear(); return false; }
  const bool bnhd = a[7] == Py_True;
  if (Q.dim() != 4 || p->K->sizes() != Q.sizes() || p->V->sizes() != Q.sizes() || p->F->sizes() != p->E->sizes()) return false;
  for (int64_t s : Q.sizes())
    if (s > INT32_MAX) return false;
  const int64_t H = Q.size(bnhd ? 2 : 1), N = Q.size(bnhd ? 1 : 2);
  const int64_t ed = p->E->dim();
  if (!(ed == 2 || (ed == 3 && p->E->size(0) == H)) || p->E->size(ed - 1) != N || p->E->size(ed - 2) > INT32_MAX) return false;
  p->B = (int)Q.size(0);
  p->H = (int)H;
  p->N = (int)N;
  p->d = (int)Q.size(3);
  p->k = (int)p->E->size(ed - 2);
  p->W = nullptr;
  p->m = 0;
  if (variant == kPerformer) {
    if (!(p->W = plain(a[5], p->Q)) || p->W->dim() != 2 || p->W->size(1) != p->d || p->W->size(0) > INT32_MAX) return false;
    p->m = (int)p->W->size(0);
  } else if (a[5] != Py_None) {
    if (!THPVariable_CheckExact(a[5])) return false;      // (its address goes along, as binding.py has it)
    p->W = &THPVariable_Unpack(a[5]);
  }
  p->variant = (int)variant | (fp32 ? kFp32 : 0) | (bnhd ? kBnhd : 0) | (ed == 3 ? kPerHead : 0);
  return true;
}

const void* address(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
void* stream_of_current_device() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

// init(address of flurka_forward, address of flurka_backward)
PyObject* init(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 2) { PyErr_SetString(PyExc_TypeError, "init takes two addresses"); return nullptr; }
  g_forward = (ForwardFn)PyLong_AsVoidPtr(a[0]);
  g_backward = (BackwardFn)PyLong_AsVoidPtr(a[1]);
  if (PyErr_Occurred()) return nullptr;
  Py_RETURN_NONE;
}

// forward(Q, K, V, E, F, W, variant, bnhd) -> (status, out) on the current stream, or None: not a plain call
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Problem p;
  try {
    if (n != 8 || !g_forward || !parse(a, &p)) Py_RETURN_NONE;
    at::Tensor out = at::empty_like(*p.Q);
    if (out.sizes() != p.Q->sizes() || !out.is_contiguous()) Py_RETURN_NONE;
    const void* const in[6] = {address(p.Q), address(p.K), address(p.V), address(p.E), address(p.F), address(p.W)};
    void* const to = out.data_ptr();
    void* const stream = stream_of_current_device();
    int rc;
    {
      WithoutInterpreter released;
      rc = g_forward(in[0], in[1], in[2], in[3], in[4], in[5], p.variant, p.B, p.H, p.N, p.d, p.k, p.m, to, stream);
    }
    return Py_BuildValue("(iN)", rc, THPVariable_Wrap(std::move(out)));
  } catch (...) {
    Py_RETURN_NONE;                                        // (out of memory and the like: the Python path says so)
  }
}

// backward(Q, K, V, E, F, W, variant, bnhd, dO) -> (status, dQ, dK, dV, dE, dF), or None: not a plain call
PyObject* backward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Problem p;
  try {
    if (n != 9 || !g_backward || !parse(a, &p)) Py_RETURN_NONE;
    if (!(p.dO = plain(a[8], p.Q)) || p.dO->sizes() != p.Q->sizes()) Py_RETURN_NONE;
    const at::Tensor* like[5] = {p.Q, p.K, p.V, p.E, p.F};
    at::Tensor g[5];
    void* to[5];
    for (int i = 0; i < 5; ++i) {
      g[i] = at::empty_like(*like[i]);
      if (!g[i].is_contiguous()) Py_RETURN_NONE;
      to[i] = g[i].data_ptr();
    }
    const void* const in[7] = {address(p.Q), address(p.K), address(p.V), address(p.E), address(p.F), address(p.W), address(p.dO)};
    void* const stream = stream_of_current_device();
    int rc;
    {
      WithoutInterpreter released;
      rc = g_backward(in[0], in[1], in[2], in[3], in[4], in[5], in[6], p.variant, p.B, p.H, p.N, p.d, p.k, p.m, to[0], to[1],
                      to[2], to[3], to[4], stream);
    }
    return Py_BuildValue("(iNNNNN)", rc, THPVariable_Wrap(std::move(g[0])), THPVariable_Wrap(std::move(g[1])),
                         THPVariable_Wrap(std::move(g[2])), THPVariable_Wrap(std::move(g[3])), THPVariable_Wrap(std::move(g[4])));
  } catch (...) {
    Py_RETURN_NONE;
  }
}

PyMethodDef kMethods[] = {
    {"init", (PyCFunction)(void*)init, METH_FASTCALL, "init(flurka_forward, flurka_backward): addresses in libflurka.so"},
    {"forward", (PyCFunction)(void*)forward, METH_FASTCALL, "forward(Q, K, V, E, F, W, variant, bnhd)"},
    {"backward", (PyCFunction)(void*)backward, METH_FASTCALL, "backward(Q, K, V, E, F, W, variant, bnhd, dO)"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", FLURKA_MARSHAL_TAG, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) { return PyModule_Create(&kModule); }
