// Native call path of the stand-alone acceptance step for torch tensors: argument checks, output allocation and the library
// call in one C++ function.  The step itself takes about 12 us on the GPU for one sequence; the same marshalling in Python
// (a dozen attribute checks, four allocations, the stream object, a ctypes call with 15 arguments) took 20 us.
#include <Python.h>

#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/torch.h>

#include <map>
#include <utility>

#include "../../include/sdd.h"

namespace {

bool fail(const char* what) {
  PyErr_SetString(PyExc_AssertionError, what);
  return false;
}

struct Problem {
  at::Tensor lp, lq, ids;
  int rows, gamma, V;
};

bool want_tensor(PyObject* o, at::Tensor* t, at::ScalarType type, const char* what) {
  if (!THPVariable_Check(o)) return fail(what);
  *t = THPVariable_Unpack(o);
  return (t->is_cuda() && t->is_contiguous() && t->scalar_type() == type) || fail(what);
}

bool parse_problem(PyObject* const* a, Problem* p) {
  if (!want_tensor(a[0], &p->lp, at::kFloat, "logits_p: contiguous fp32 CUDA tensor") ||
      !want_tensor(a[1], &p->lq, at::kFloat, "logits_q: contiguous fp32 CUDA tensor") ||
      !want_tensor(a[2], &p->ids, at::kInt, "draft_ids: contiguous int32 CUDA tensor"))
    return false;
  if (p->lp.dim() != 3 || p->lq.dim() != 3 || p->ids.dim() != 2) return fail("logits_p, logits_q: 3 dimensions, draft_ids: 2");
  const int64_t rows = p->lp.size(0), gamma = p->lp.size(1) - 1, V = p->lp.size(2);
  if (p->lq.size(0) != rows || p->lq.size(1) != gamma || p->lq.size(2) != V || p->ids.size(0) != rows || p->ids.size(1) != gamma)
    return fail("logits_q [rows, gamma, V], draft_ids [rows, gamma]");
  if (rows > INT32_MAX || gamma > INT32_MAX || V > INT32_MAX) return fail("sizes of 32 bits");
  p->rows = (int)rows;
  p->gamma = (int)gamma;
  p->V = (int)V;
  return true;
}

// temp_p, temp_q, seed, round
bool parse_numbers(PyObject* const* a, float* tp, float* tq, uint64_t* seed, uint64_t* rnd) {
  *tp = (float)PyFloat_AsDouble(a[0]);
  *tq = (float)PyFloat_AsDouble(a[1]);
  *seed = PyLong_AsUnsignedLongLongMask(a[2]);
  *rnd = PyLong_AsUnsignedLongLongMask(a[3]);
  return !PyErr_Occurred();
}

bool parse_stream(PyObject* o, const at::Tensor& t, cudaStream_t* st) {
  if (o == Py_None) {
    *st = c10::cuda::getCurrentCUDAStream(t.device().index()).stream();
    return true;
  }
  *st = (cudaStream_t)PyLong_AsUnsignedLongLongMask(o);
  return !PyErr_Occurred();
}

// One scratch per device and stream, kept between calls (calls on one stream follow one another on the device).  A call that is
// being captured gets its own: the graph may be replayed beside the stream it was captured on.
at::Tensor scratch_for(const at::Tensor& like, cudaStream_t st, uint64_t bytes) {
  static auto* kept = new std::map<std::pair<int, cudaStream_t>, at::Tensor>();   // never destroyed: the allocator may go first
  const auto opt = like.options().dtype(at::kByte);
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) return at::empty({(int64_t)bytes}, opt);
  at::Tensor& t = (*kept)[{like.device().index(), st}];
  if (!t.defined() || (uint64_t)t.numel() < bytes) t = at::empty({(int64_t)bytes}, opt);
  return t;
}

// (logits_p, logits_q, draft_ids, temp_p, temp_q, seed, round, scratch or None, stream handle or None)
// -> (status, n_accept, out_ids, accept_prob)
PyObject* accept_logits(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 9) { PyErr_SetString(PyExc_TypeError, "9 arguments"); return nullptr; }
  try {
    Problem p;
    float tp, tq;
    uint64_t seed, rnd;
    cudaStream_t st;
    if (!parse_problem(a, &p) || !parse_numbers(a + 3, &tp, &tq, &seed, &rnd) || !parse_stream(a[8], p.lp, &st)) return nullptr;
    at::Tensor scratch;
    const uint64_t need = sdd_accept_scratch_bytes(p.rows, p.gamma, p.V);
    if (a[7] != Py_None) {
      if (!THPVariable_Check(a[7])) { fail("scratch: tensor"); return nullptr; }
      scratch = THPVariable_Unpack(a[7]);
    } else {
      scratch = scratch_for(p.lp, st, need);
    }
    const auto ints = p.ids.options();
    at::Tensor n_accept = at::empty({p.rows}, ints), out_ids = at::empty({p.rows, p.gamma + 1}, ints);
    at::Tensor prob = at::empty({p.rows, p.gamma}, p.lp.options());
    const int32_t s = sdd_accept_logits(p.lp.const_data_ptr<float>(), p.lq.const_data_ptr<float>(), p.ids.const_data_ptr<int32_t>(), p.rows,
                                        p.gamma, p.V, tp, tq, seed, rnd, n_accept.mutable_data_ptr<int32_t>(),
                                        out_ids.mutable_data_ptr<int32_t>(), prob.mutable_data_ptr<float>(), scratch.data_ptr(), st);
    PyObject* r = PyTuple_New(4);
    PyTuple_SET_ITEM(r, 0, PyLong_FromLong(s));
    PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(n_accept)));
    PyTuple_SET_ITEM(r, 2, THPVariable_Wrap(std::move(out_ids)));
    PyTuple_SET_ITEM(r, 3, THPVariable_Wrap(std::move(prob)));
    return r;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// (logits_p, logits_q, draft_ids, n_accept, out_ids, accept_prob, temp_p, temp_q, seed, round, stream handle or None) -> status
PyObject* accept_logits_static(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 11) { PyErr_SetString(PyExc_TypeError, "11 arguments"); return nullptr; }
  try {
    Problem p;
    at::Tensor na, out, prob;
    float tp, tq;
    uint64_t seed, rnd;
    cudaStream_t st;
    if (!parse_problem(a, &p) || !want_tensor(a[3], &na, at::kInt, "n_accept: contiguous int32 CUDA tensor") ||
        !want_tensor(a[4], &out, at::kInt, "out_ids: contiguous int32 CUDA tensor") ||
        !want_tensor(a[5], &prob, at::kFloat, "accept_prob: contiguous fp32 CUDA tensor") ||
        !parse_numbers(a + 6, &tp, &tq, &seed, &rnd) || !parse_stream(a[10], p.lp, &st))
      return nullptr;
    if (na.dim() != 1 || na.size(0) != p.rows || out.dim() != 2 || out.size(0) != p.rows || out.size(1) != p.gamma + 1 || prob.dim() != 2 ||
        prob.size(0) != p.rows || prob.size(1) != p.gamma) {
      fail("n_accept [rows], out_ids [rows, gamma + 1], accept_prob [rows, gamma]");
      return nullptr;
    }
    return PyLong_FromLong(sdd_accept_logits_static(p.lp.const_data_ptr<float>(), p.lq.const_data_ptr<float>(), p.ids.const_data_ptr<int32_t>(),
                                                    p.rows, p.gamma, p.V, tp, tq, seed, rnd, na.mutable_data_ptr<int32_t>(),
                                                    out.mutable_data_ptr<int32_t>(), prob.mutable_data_ptr<float>(), st));
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {
    {"accept_logits", (PyCFunction)(void (*)(void))accept_logits, METH_FASTCALL, nullptr},
    {"accept_logits_static", (PyCFunction)(void (*)(void))accept_logits_static, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_sdd_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sdd_torch(void) { return PyModule_Create(&module); }
