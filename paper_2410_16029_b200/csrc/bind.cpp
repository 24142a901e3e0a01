// The pointers of a step's tensors, checked and collected in one call: statement by statement the interpreter takes 0.95 us a
// matrix for it, 90 us for 102 of them (so 2 us), and a set of many small matrices waited for its host: 102 matrices of 192
// columns and more, r = 12, 106 us a step whose kernels take 35.
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>
#include <torch/version.h>

namespace {

enum Mode { kUnchecked = 0, kDevice = 1, kHost = 2 };

struct Fast {
  PyObject* o;
  explicit Fast(PyObject* s) : o(PySequence_Fast(s, "a sequence of tensors")) {}
  ~Fast() { Py_XDECREF(o); }
};

const at::Tensor* plain_tensor(PyObject* o) { return THPVariable_CheckExact(o) ? &THPVariable_Unpack(o) : nullptr; }

bool device_ok(const at::Tensor& t, at::ScalarType dtype, const int64_t* shape) {
  return t.is_cuda() && t.scalar_type() == dtype && t.dim() == 2 && t.size(0) == shape[0] && t.size(1) == shape[1] && t.is_contiguous();
}

// A buffer that a step on host memory reads and writes as rows x cols floats or bf16 values, whatever its shape: it has to hold that many.
// (Gradients may come as the bits of their values.)
bool host_ok(const at::Tensor& t, bool weights, const int64_t* shape) {
  const at::ScalarType type = t.scalar_type();
  const bool typed = weights ? type == at::kFloat : type == at::kBFloat16 || type == at::kShort || type == at::kUInt16;
  return t.is_cpu() && typed && t.is_contiguous() && t.numel() >= shape[0] * shape[1];
}

// collect(W, G, n, shapes, W_out, G_out, mode): shapes, W_out and G_out are addresses (2 n int64, n pointers each).  True: the pointers are
// there.  False: something else than n plain tensors each, which the caller has to look at itself.  AssertionError: a tensor that
// is not what a step takes.
PyObject* collect(PyObject*, PyObject* args) {
  PyObject *w_seq, *g_seq;
  Py_ssize_t n;
  unsigned long long shapes_at, w_at, g_at;
  int mode;
  if (!PyArg_ParseTuple(args, "OOnKKKi", &w_seq, &g_seq, &n, &shapes_at, &w_at, &g_at, &mode)) return nullptr;
  if (!(PyList_Check(w_seq) || PyTuple_Check(w_seq)) || !(PyList_Check(g_seq) || PyTuple_Check(g_seq))) Py_RETURN_FALSE;
  const Fast w_fast(w_seq), g_fast(g_seq);
  if (w_fast.o == nullptr || g_fast.o == nullptr) return nullptr;
  if (PySequence_Fast_GET_SIZE(w_fast.o) != n || PySequence_Fast_GET_SIZE(g_fast.o) != n) Py_RETURN_FALSE;
  const int64_t* shapes = reinterpret_cast<const int64_t*>(shapes_at);
  void **w_out = reinterpret_cast<void**>(w_at), **g_out = reinterpret_cast<void**>(g_at);
  try {
    for (Py_ssize_t i = 0; i < n; ++i) {
      const at::Tensor *w = plain_tensor(PySequence_Fast_GET_ITEM(w_fast.o, i)), *g = plain_tensor(PySequence_Fast_GET_ITEM(g_fast.o, i));
      if (w == nullptr || g == nullptr) Py_RETURN_FALSE;
      if (mode == kDevice && !(device_ok(*w, at::kFloat, shapes + 2 * i) && device_ok(*g, at::kBFloat16, shapes + 2 * i))) {
        PyErr_Format(PyExc_AssertionError, "matrix %zd: a step takes contiguous CUDA tensors of its shape, W float32 and G bfloat16", i);
        return nullptr;
      }
      if (mode == kHost && !(host_ok(*w, true, shapes + 2 * i) && host_ok(*g, false, shapes + 2 * i))) {
        PyErr_Format(PyExc_AssertionError, "matrix %zd: a step on host buffers takes contiguous CPU tensors of its size, W float32 and G bfloat16", i);
        return nullptr;
      }
      w_out[i] = w->data_ptr();
      g_out[i] = g->data_ptr();
    }
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
  Py_RETURN_TRUE;
}

PyMethodDef methods[] = {{"collect", collect, METH_VARARGS, "Checks and collects the pointers of a step's tensors."}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_bind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (built_for: the tensor's layout that is compiled in belongs to one torch and one Python, see ngalore.py)
PyMODINIT_FUNC PyInit__bind() {
  PyObject* m = PyModule_Create(&module);
  if (m != nullptr && PyModule_AddObject(m, "built_for", Py_BuildValue("(sii)", TORCH_VERSION, PY_MAJOR_VERSION, PY_MINOR_VERSION)) != 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
