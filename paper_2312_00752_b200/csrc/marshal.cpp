// Argument marshalling of the Python binding: torch tensors to the pointers of the C ABI (include/ssm_scan.h,
// include/ssm_conv1d.h), output and workspace allocation.  A CPython module, because the same work in Python (about twelve
// tensors of a call checked attribute by attribute, the ctypes conversions) cost 12 to 40 us a call, more than a decoding
// step or a short prompt takes on the GPU.  Nothing of the method is here: the library is loaded by path at import and
// every call ends in one call of the C ABI.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include <map>
#include <mutex>
#include <string>
#include <utility>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "ssm_conv1d.h"
#include "ssm_scan.h"

namespace {

PyObject* g_error = nullptr;           // SsmScanError
PyObject* g_out_of_memory = nullptr;   // torch.OutOfMemoryError

// the entry points, resolved from the library the binding chose
#define SSM_ENTRY_POINTS(X)                                                                                       \
  X(ssm_scan_fwd_state) X(ssm_scan_fwd_fused_dt) X(ssm_scan_fwd_static) X(ssm_scan_bwd) X(ssm_scan_bwd_state)     \
  X(ssm_scan_bwd_fused_dt) X(ssm_scan_bwd_fused_dt_state) X(ssm_step) X(ssm_scan_fwd_workspace_bytes)             \
  X(ssm_scan_bwd_workspace_bytes) X(ssm_scan_saved_state_bytes) X(ssm_status_string) X(ssm_conv1d_fwd)            \
  X(ssm_conv1d_bwd) X(ssm_conv1d_bwd_workspace_bytes)
struct Api {
#define X(name) decltype(&::name) name;
  SSM_ENTRY_POINTS(X)
#undef X
} api;

struct Raised {};   // a Python exception is set

[[noreturn]] void raise(const std::string& what) {
  PyErr_SetString(g_error, what.c_str());
  throw Raised{};
}

std::string dtype_name(at::ScalarType t) {
  switch (t) {
    case at::kFloat: return "torch.float32";
    case at::kBFloat16: return "torch.bfloat16";
    case at::kHalf: return "torch.float16";
    case at::kDouble: return "torch.float64";
    default: return c10::toString(t);
  }
}

std::string shape_text(at::IntArrayRef s) {
  std::string r = "(";
  for (size_t i = 0; i < s.size(); ++i) r += (i ? ", " : "") + std::to_string(s[i]);
  return r + (s.size() == 1 ? ",)" : ")");
}

const at::Tensor* tensor(PyObject* o, const char* name) {
  if (o == Py_None) return nullptr;
  if (!THPVariable_Check(o)) raise(std::string(name) + " must be a torch.Tensor");
  return &THPVariable_Unpack(o);
}

// device pointer of a contiguous CUDA tensor (null for None)
void* pointer(const at::Tensor* t, const char* name) {
  if (t == nullptr) return nullptr;
  if (!t->is_cuda()) raise(std::string(name) + " must be a CUDA tensor");
  if (!t->is_contiguous()) raise(std::string(name) + " must be contiguous");
  return t->data_ptr();
}
void* pointer(const at::Tensor* t, const char* name, at::IntArrayRef shape, at::ScalarType dtype) {
  void* p = pointer(t, name);
  if (t == nullptr) return p;
  if (t->sizes() != shape) raise(std::string(name) + " has shape " + shape_text(t->sizes()) + ", expected " + shape_text(shape));
  if (t->scalar_type() != dtype)
    raise(std::string(name) + " has dtype " + dtype_name(t->scalar_type()) + ", expected " + dtype_name(dtype));
  return p;
}
void* pointer(PyObject* o, const char* name, at::IntArrayRef shape, at::ScalarType dtype) {
  return pointer(tensor(o, name), name, shape, dtype);
}

int io_dtype(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return SSM_F32;
  if (t.scalar_type() == at::kBFloat16) return SSM_BF16;
  raise("io dtype must be float32 or bfloat16, got " + dtype_name(t.scalar_type()));
}

at::Tensor empty(at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor& like) {
  if (!like.is_cuda()) raise("x must be a CUDA tensor");
  return at::detail::empty_cuda(shape, dtype, like.device(), std::nullopt);
}

void* stream_of(PyObject* stream, const at::Tensor& x) {
  if (!x.is_cuda()) raise("x must be a CUDA tensor");
  if (stream == Py_None) return c10::cuda::getCurrentCUDAStream(x.device().index()).stream();
  PyObject* v = PyObject_GetAttrString(stream, "cuda_stream");
  if (v == nullptr) throw Raised{};
  void* s = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (s == nullptr && PyErr_Occurred()) throw Raised{};
  return s;
}

// A new result of a call on `stream`.  It is a block of the current stream; where that is another one the allocator is told, so
// that a result that is dropped early is not given to other tensors while the call still writes to it.
at::Tensor result(at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor& like, void* stream) {
  at::Tensor t = empty(shape, dtype, like);
  const auto s = static_cast<cudaStream_t>(stream);
  const c10::DeviceIndex dev = like.device().index();
  if (c10::cuda::getCurrentCUDAStream(dev).stream() != s)
    c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), c10::cuda::getStreamFromExternal(s, dev));
  return t;
}

// A buffer for work on `stream`, which need not be the current one: a block of that stream's own, so that the allocator takes
// it from nobody whose work on another stream still uses it, and gives it back to nobody else.
at::Tensor scratch_buffer(size_t bytes, const at::Tensor& x, void* stream) {
  const auto s = c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(stream), x.device().index());
  const c10::cuda::CUDAStreamGuard on(s);
  return empty({(int64_t)bytes}, at::kByte, x);
}

// Scratch of one (device, stream): a buffer that only grows (calls on different streams never share scratch memory), and a lock
// that a call on it holds while it enqueues.  A call is several launches that hand results to each other through the buffer,
// and the interpreter lock is not held meanwhile: without this one the launches of two threads on one stream would mix.
// (The table is guarded by the interpreter lock; never destroyed, because the allocator may be gone by the time statics are.)
struct Scratch {
  at::Tensor buffer;
  std::mutex enqueue;
};
std::map<std::pair<int, void*>, Scratch>& workspaces() {
  static auto* m = new std::map<std::pair<int, void*>, Scratch>();
  return *m;
}
// What a call uses of it: a reference to the buffer of its own (another thread may put a larger one in its place), and the lock.
struct Workspace {
  at::Tensor buffer;
  std::mutex* enqueue = nullptr;
};
Workspace workspace(size_t bytes, const at::Tensor& x, void* stream) {
  if (bytes == 0) return {};
  // A call that is being captured gets a buffer of its own, from the graph's memory: the graph keeps its address, while the
  // buffer kept here may be given back when a larger one takes its place.
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(static_cast<cudaStream_t>(stream), &capture) != cudaSuccess) (void)cudaGetLastError();
  if (capture != cudaStreamCaptureStatusNone) return {scratch_buffer(bytes, x, stream), nullptr};
  Scratch& scratch = workspaces()[{x.device().index(), stream}];
  at::Tensor& ws = scratch.buffer;
  // (the old buffer is a block of the same stream: whoever gets its memory is enqueued behind the kernels that use it)
  if (!ws.defined() || (size_t)ws.numel() < bytes) ws = scratch_buffer(bytes, x, stream);
  return {ws, &scratch.enqueue};
}

// Calls a function of the library with the interpreter lock released (a full launch queue blocks), raises its error.
// `enqueue`: the lock of the scratch the call works in, if it does; taken without the interpreter lock, so that a thread
// that waits for the one never holds the other.
template <typename F>
void call(const char* what, std::mutex* enqueue, F&& f) {
  PyThreadState* const t = PyEval_SaveThread();
  ssm_status_t st;
  {
    const auto hold = enqueue != nullptr ? std::unique_lock<std::mutex>(*enqueue) : std::unique_lock<std::mutex>();
    st = f();
  }
  PyEval_RestoreThread(t);
  if (st != SSM_OK) raise(std::string(what) + ": " + api.ssm_status_string(st));
}

bool truth(PyObject* o) {
  const int t = PyObject_IsTrue(o);
  if (t < 0) throw Raised{};
  return t != 0;
}

PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

// shapes and element types of the arguments of a scan
struct Problem {
  ssm_problem_t p;
  at::ScalarType io;
  c10::SmallVector<int64_t, 4> a, b, c, h, rows;
  at::ScalarType bt, ct;
};
Problem problem(const at::Tensor& x, const at::Tensor* B, bool step, uint32_t flags) {
  if (B == nullptr) raise("B must be a CUDA tensor");
  const bool cplx = flags & SSM_FLAG_COMPLEX, sb = flags & SSM_FLAG_STATIC_B, sc = flags & SSM_FLAG_STATIC_C;
  if (x.dim() != (step ? 2 : 3)) raise(std::string("x must have ") + (step ? "2" : "3") + " dimensions");
  if (B->dim() < (cplx ? 2 : 1)) raise("B has too few dimensions");
  Problem r;
  const int64_t batch = x.size(0), L = step ? 1 : x.size(1), D = x.size(-1), N = B->size(cplx ? -2 : -1);
  r.io = x.scalar_type();
  r.p = ssm_problem_t{(int32_t)batch, (int32_t)L, (int32_t)D, (int32_t)N, io_dtype(x), flags};
  r.rows.assign(x.sizes().begin(), x.sizes().end());
  r.a = {D, N};
  r.b = step ? c10::SmallVector<int64_t, 4>{batch, N} : c10::SmallVector<int64_t, 4>{batch, L, N};
  r.h = {batch, D, N};
  if (cplx) {
    r.a.push_back(2);
    r.b.push_back(2);
    r.h.push_back(2);
  }
  r.c = r.b;
  r.bt = r.ct = r.io;
  if (sb) {
    r.b = {D, N};
    r.bt = at::kFloat;
  }
  if (sc) {
    r.c = {D, N};
    r.ct = at::kFloat;
  }
  return r;
}

uint32_t scan_flags(PyObject* z, PyObject* dskip, PyObject* general, PyObject* zoh, PyObject* sb, PyObject* sc, PyObject* cplx) {
  return (z != Py_None ? SSM_FLAG_HAS_Z : 0u) | (dskip != Py_None ? SSM_FLAG_HAS_DSKIP : 0u) |
         (truth(general) ? SSM_FLAG_GENERAL_A : 0u) | (truth(zoh) ? SSM_FLAG_ZOH_BBAR : 0u) |
         (truth(sb) ? SSM_FLAG_STATIC_B : 0u) | (truth(sc) ? SSM_FLAG_STATIC_C : 0u) |
         (truth(cplx) ? SSM_FLAG_COMPLEX : 0u);
}

template <typename F>
PyObject* guarded(F&& f) {
  try {
    return f();
  } catch (const Raised&) {
    return nullptr;
  } catch (const c10::OutOfMemoryError& e) {
    PyErr_SetString(g_out_of_memory, e.what_without_backtrace());
    return nullptr;
  } catch (const c10::Error& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// fwd(x, delta, delta_bias, A, B, C, D_skip, z, h0, out, h_last, saved_states, workspace, stream, save_states, general_A,
//     zoh, static_B, static_C, complex_state, softplus, entry) -> out or (out, saved_states)
// entry: 0 ssm_scan_fwd_state, 1 ssm_scan_fwd_fused_dt, 2 ssm_scan_fwd_static
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 22) return PyErr_Format(PyExc_TypeError, "fwd: 22 arguments");
  return guarded([&]() -> PyObject* {
    const bool save = truth(a[14]);
    const long entry = PyLong_AsLong(a[21]);
    const at::Tensor* xp = tensor(a[0], "x");
    if (xp == nullptr) raise("x must be a CUDA tensor");
    const at::Tensor& x = *xp;
    const at::Tensor* B = tensor(a[4], "B");
    uint32_t flags = scan_flags(a[7], a[6], a[15], a[16], a[17], a[18], a[19]) | (save ? SSM_FLAG_SAVE_STATES : 0u);
    if (truth(a[20])) flags |= SSM_FLAG_DELTA_SOFTPLUS;
    Problem pr = problem(x, B, false, flags);
    const int64_t D = pr.p.D;
    void* stream = stream_of(a[13], x);
    const at::Tensor* given = tensor(a[9], "out");
    at::Tensor out = given != nullptr ? *given : result(pr.rows, pr.io, x, stream);
    const at::Tensor* sgiven = save ? tensor(a[11], "saved_states") : nullptr;
    at::Tensor saved;
    if (save) saved = sgiven != nullptr ? *sgiven : result({(int64_t)(api.ssm_scan_saved_state_bytes(&pr.p) / 4)}, at::kFloat, x, stream);
    const at::Tensor* ws = tensor(a[12], "workspace");
    Workspace own;
    if (ws == nullptr && entry != 2) own = workspace(api.ssm_scan_fwd_workspace_bytes(&pr.p), x, stream);
    if (own.buffer.defined()) ws = &own.buffer;
    void* wp = pointer(ws, "workspace");
    const size_t wbytes = ws == nullptr ? 0 : (size_t)ws->numel() * ws->element_size();
    void* px = pointer(&x, "x", pr.rows, pr.io);
    void* pd = pointer(a[1], entry == 1 ? "delta_pre" : "delta", pr.rows, pr.io);
    auto* pA = static_cast<float*>(pointer(a[3], "A", pr.a, at::kFloat));
    void* pB = pointer(B, "B", pr.b, pr.bt);
    void* pC = pointer(a[5], "C", pr.c, pr.ct);
    auto* pD = static_cast<float*>(pointer(a[6], "D_skip", {D}, at::kFloat));
    void* pz = pointer(a[7], "z", pr.rows, pr.io);
    auto* ph = static_cast<float*>(pointer(a[8], "h0", pr.h, at::kFloat));
    void* po = pointer(&out, "out", pr.rows, pr.io);
    auto* pl = static_cast<float*>(pointer(a[10], "h_last", pr.h, at::kFloat));
    void* ps = save ? pointer(&saved, "saved_states") : nullptr;
    if (entry == 2) {
      call("ssm_scan_fwd_static", nullptr, [&] {
        return api.ssm_scan_fwd_static(&pr.p, px, pd, pA, pB, pC, pD, pz, po, ps, stream);
      });
    } else if (entry == 1) {
      auto* pb = static_cast<float*>(pointer(a[2], "delta_bias", {D}, at::kFloat));
      call("ssm_scan_fwd_fused_dt", own.enqueue, [&] {
        return api.ssm_scan_fwd_fused_dt(&pr.p, px, pd, pb, pA, pB, pC, pD, pz, ph, po, pl, ps, wp, wbytes, stream);
      });
    } else {
      call("ssm_scan_fwd_state", own.enqueue, [&] {
        return api.ssm_scan_fwd_state(&pr.p, px, pd, pA, pB, pC, pD, pz, ph, po, pl, ps, wp, wbytes, stream);
      });
    }
    if (!save) return wrap(out);
    PyObject* o = wrap(out);
    PyObject* sv = wrap(saved);
    PyObject* r = PyTuple_Pack(2, o, sv);
    Py_DECREF(o);
    Py_DECREF(sv);
    return r;
  });
}

// an output of a backward call: the tensor of `outputs` under that name, or a new one, which is put there
at::Tensor output(PyObject* outputs, const char* name, at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor& like,
                  void* stream) {
  PyObject* have = PyDict_GetItemString(outputs, name);
  if (have != nullptr && have != Py_None) {
    const at::Tensor* t = tensor(have, name);
    pointer(t, name, shape, dtype);
    return *t;
  }
  at::Tensor t = result(shape, dtype, like, stream);
  PyObject* o = wrap(t);
  const int rc = PyDict_SetItemString(outputs, name, o);
  Py_DECREF(o);
  if (rc != 0) throw Raised{};
  return t;
}
void no_output(PyObject* outputs, const char* name) {
  if (PyDict_SetItemString(outputs, name, Py_None) != 0) throw Raised{};
}

// bwd(x, delta, delta_bias, A, B, C, D_skip, z, dout, saved_states, h0, dh_last, workspace, stream, outputs, general_A,
//     zoh, static_B, static_C, complex_state, softplus, fused, want_dh0, extra_flags): fills and returns `outputs`
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 24) return PyErr_Format(PyExc_TypeError, "bwd: 24 arguments");
  return guarded([&]() -> PyObject* {
    const at::Tensor* xp = tensor(a[0], "x");
    if (xp == nullptr) raise("x must be a CUDA tensor");
    const at::Tensor& x = *xp;
    const at::Tensor* B = tensor(a[4], "B");
    uint32_t flags = scan_flags(a[7], a[6], a[15], a[16], a[17], a[18], a[19]) | (uint32_t)PyLong_AsLong(a[23]);
    if (truth(a[20])) flags |= SSM_FLAG_DELTA_SOFTPLUS;
    const bool fused = truth(a[21]), want_dh0 = truth(a[22]);
    const bool state = a[10] != Py_None || a[11] != Py_None || want_dh0;
    Problem pr = problem(x, B, false, flags);
    const int64_t D = pr.p.D;
    PyObject* o = a[14];
    void* stream = stream_of(a[13], x);
    const at::Tensor* ws = tensor(a[12], "workspace");
    Workspace own;
    if (ws == nullptr) own = workspace(api.ssm_scan_bwd_workspace_bytes(&pr.p), x, stream);
    if (own.buffer.defined()) ws = &own.buffer;
    void* wp = pointer(ws, "workspace");
    const size_t wbytes = ws == nullptr ? 0 : (size_t)ws->numel() * ws->element_size();
    void* px = pointer(&x, "x", pr.rows, pr.io);
    void* pd = pointer(a[1], fused ? "delta_pre" : "delta", pr.rows, pr.io);
    auto* pA = static_cast<float*>(pointer(a[3], "A", pr.a, at::kFloat));
    void* pB = pointer(B, "B", pr.b, pr.bt);
    void* pC = pointer(a[5], "C", pr.c, pr.ct);
    auto* pD = static_cast<float*>(pointer(a[6], "D_skip", {D}, at::kFloat));
    void* pz = pointer(a[7], "z", pr.rows, pr.io);
    void* pg = pointer(a[8], "dout", pr.rows, pr.io);
    void* ps = pointer(tensor(a[9], "saved_states"), "saved_states");
    auto* ph = static_cast<float*>(pointer(a[10], "h0", pr.h, at::kFloat));
    auto* pm = static_cast<float*>(pointer(a[11], "dh_last", pr.h, at::kFloat));
    at::Tensor dx = output(o, "dx", pr.rows, pr.io, x, stream), dd = output(o, "ddelta", pr.rows, pr.io, x, stream);
    at::Tensor dA = output(o, "dA", pr.a, at::kFloat, x, stream), dB = output(o, "dB", pr.b, pr.bt, x, stream), dC = output(o, "dC", pr.c, pr.ct, x, stream);
    at::Tensor dD, dz, dbias, dh0;
    if (pD != nullptr) dD = output(o, "dD", {D}, at::kFloat, x, stream);
    else no_output(o, "dD");
    if (pz != nullptr) dz = output(o, "dz", pr.rows, pr.io, x, stream);
    else no_output(o, "dz");
    if (fused) dbias = output(o, "ddelta_bias", {D}, at::kFloat, x, stream);
    if (want_dh0) dh0 = output(o, "dh0", pr.h, at::kFloat, x, stream);
    auto data = [](const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; };
    auto fdata = [](const at::Tensor& t) { return t.defined() ? static_cast<float*>(t.data_ptr()) : nullptr; };
    if (fused) {
      auto* pb = static_cast<float*>(pointer(a[2], "delta_bias", {D}, at::kFloat));
      if (state)
        call("ssm_scan_bwd_fused_dt_state", own.enqueue, [&] {
        return api.ssm_scan_bwd_fused_dt_state(&pr.p, px, pd, pb, pA, pB, pC, pD, pz, pg, ph, pm, ps, data(dx), data(dd), fdata(dbias),
        fdata(dA), data(dB), data(dC), fdata(dD), data(dz), fdata(dh0), wp, wbytes, stream);
      });
      else
        call("ssm_scan_bwd_fused_dt", own.enqueue, [&] {
        return api.ssm_scan_bwd_fused_dt(&pr.p, px, pd, pb, pA, pB, pC, pD, pz, pg, ps, data(dx), data(dd), fdata(dbias), fdata(dA),
        data(dB), data(dC), fdata(dD), data(dz), wp, wbytes, stream);
      });
    } else if (state) {
      call("ssm_scan_bwd_state", own.enqueue, [&] {
        return api.ssm_scan_bwd_state(&pr.p, px, pd, pA, pB, pC, pD, pz, pg, ph, pm, ps, data(dx), data(dd), fdata(dA), data(dB), data(dC),
        fdata(dD), data(dz), fdata(dh0), wp, wbytes, stream);
      });
    } else {
      call("ssm_scan_bwd", own.enqueue, [&] {
        return api.ssm_scan_bwd(&pr.p, px, pd, pA, pB, pC, pD, pz, pg, ps, data(dx), data(dd), fdata(dA), data(dB), data(dC), fdata(dD),
        data(dz), wp, wbytes, stream);
      });
    }
    Py_INCREF(o);
    return o;
  });
}

// step(x, delta, A, B, C, D_skip, z, h, out, stream, zoh, static_B, static_C, complex_state) -> out
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 14) return PyErr_Format(PyExc_TypeError, "step: 14 arguments");
  return guarded([&]() -> PyObject* {
    const at::Tensor* xp = tensor(a[0], "x");
    if (xp == nullptr) raise("x must be a CUDA tensor");
    const at::Tensor& x = *xp;
    const at::Tensor* B = tensor(a[3], "B");
    Problem pr = problem(x, B, true, scan_flags(a[6], a[5], Py_False, a[10], a[11], a[12], a[13]));
    const at::Tensor* given = tensor(a[8], "out");
    void* px = pointer(&x, "x", pr.rows, pr.io);
    void* pd = pointer(a[1], "delta", pr.rows, pr.io);
    auto* pA = static_cast<float*>(pointer(a[2], "A", pr.a, at::kFloat));
    void* pB = pointer(B, "B", pr.b, pr.bt);
    void* pC = pointer(a[4], "C", pr.c, pr.ct);
    auto* pD = static_cast<float*>(pointer(a[5], "D_skip", {(int64_t)pr.p.D}, at::kFloat));
    void* pz = pointer(a[6], "z", pr.rows, pr.io);
    auto* ph = static_cast<float*>(pointer(a[7], "h", pr.h, at::kFloat));
    void* stream = stream_of(a[9], x);
    at::Tensor out = given != nullptr ? *given : result(pr.rows, pr.io, x, stream);
    void* po = pointer(&out, "out", pr.rows, pr.io);
    call("ssm_step", nullptr, [&] {
        return api.ssm_step(&pr.p, px, pd, pA, pB, pC, pD, pz, ph, po, stream);
      });
    return wrap(out);
  });
}

ssm_conv_problem_t conv_problem(const at::Tensor& x, const at::Tensor* w, bool silu, bool bias) {
  if (w == nullptr || w->dim() != 2) raise("w must be a (D, W) tensor");
  if (x.dim() != 3) raise("x must have 3 dimensions");
  return ssm_conv_problem_t{(int32_t)x.size(0), (int32_t)x.size(1), (int32_t)x.size(2), (int32_t)w->size(1), io_dtype(x),
                            (silu ? SSM_CONV_FLAG_SILU : 0u) | (bias ? SSM_CONV_FLAG_HAS_BIAS : 0u)};
}

// conv_fwd(x, w, bias, x_prev, out, stream, silu) -> y
PyObject* conv_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7) return PyErr_Format(PyExc_TypeError, "conv_fwd: 7 arguments");
  return guarded([&]() -> PyObject* {
    const at::Tensor* xp = tensor(a[0], "x");
    if (xp == nullptr) raise("x must be a CUDA tensor");
    const at::Tensor& x = *xp;
    const at::Tensor* w = tensor(a[1], "w");
    const ssm_conv_problem_t p = conv_problem(x, w, truth(a[6]), a[2] != Py_None);
    const at::ScalarType io = x.scalar_type();
    const int64_t D = p.D, W = p.width;
    void* px = pointer(&x, "x", x.sizes(), io);
    auto* pw = static_cast<float*>(pointer(w, "w", {D, W}, at::kFloat));
    auto* pb = static_cast<float*>(pointer(a[2], "bias", {D}, at::kFloat));
    void* pp = pointer(a[3], "x_prev", {(int64_t)p.batch, W - 1, D}, io);
    const at::Tensor* given = tensor(a[4], "y");
    void* stream = stream_of(a[5], x);
    at::Tensor y = given != nullptr ? *given : result(x.sizes(), io, x, stream);
    void* py = pointer(&y, "y", x.sizes(), io);
    call("ssm_conv1d_fwd", nullptr, [&] {
        return api.ssm_conv1d_fwd(&p, px, pw, pb, pp, py, stream);
      });
    return wrap(y);
  });
}

// conv_bwd(x, w, bias, x_prev, dy, stream, outputs, silu, want_dx_prev): fills and returns `outputs`
PyObject* conv_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 9) return PyErr_Format(PyExc_TypeError, "conv_bwd: 9 arguments");
  return guarded([&]() -> PyObject* {
    const at::Tensor* xp = tensor(a[0], "x");
    if (xp == nullptr) raise("x must be a CUDA tensor");
    const at::Tensor& x = *xp;
    const at::Tensor* w = tensor(a[1], "w");
    const ssm_conv_problem_t p = conv_problem(x, w, truth(a[7]), a[2] != Py_None);
    const at::ScalarType io = x.scalar_type();
    const int64_t D = p.D, W = p.width;
    PyObject* o = a[6];
    void* stream = stream_of(a[5], x);
    void* px = pointer(&x, "x", x.sizes(), io);
    auto* pw = static_cast<float*>(pointer(w, "w", {D, W}, at::kFloat));
    auto* pb = static_cast<float*>(pointer(a[2], "bias", {D}, at::kFloat));
    void* pp = pointer(a[3], "x_prev", {(int64_t)p.batch, W - 1, D}, io);
    void* pg = pointer(a[4], "dy", x.sizes(), io);
    at::Tensor dx = output(o, "dx", x.sizes(), io, x, stream), dw = output(o, "dw", {D, W}, at::kFloat, x, stream), db, dp;
    if (pb != nullptr) db = output(o, "dbias", {D}, at::kFloat, x, stream);
    else no_output(o, "dbias");
    if (truth(a[8]) && W > 1) dp = output(o, "dx_prev", {(int64_t)p.batch, W - 1, D}, io, x, stream);
    const Workspace own = workspace(api.ssm_conv1d_bwd_workspace_bytes(&p), x, stream);
    const at::Tensor& ws = own.buffer;
    call("ssm_conv1d_bwd", own.enqueue, [&] {
        return api.ssm_conv1d_bwd(&p, px, pw, pb, pp, pg, dx.data_ptr(), static_cast<float*>(dw.data_ptr()),
        db.defined() ? static_cast<float*>(db.data_ptr()) : nullptr, dp.defined() ? dp.data_ptr() : nullptr,
        ws.defined() ? ws.data_ptr() : nullptr, ws.defined() ? (size_t)ws.numel() : 0, stream);
      });
    Py_INCREF(o);
    return o;
  });
}

// workspace(device index, stream) -> the cached scratch tensor or None
PyObject* cached_workspace(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 2) return PyErr_Format(PyExc_TypeError, "workspace: 2 arguments");
  return guarded([&]() -> PyObject* {
    const int dev = (int)PyLong_AsLong(a[0]);
    void* s = PyLong_AsVoidPtr(a[1]);
    if (PyErr_Occurred()) throw Raised{};
    auto it = workspaces().find({dev, s});
    if (it == workspaces().end() || !it->second.buffer.defined()) Py_RETURN_NONE;
    return wrap(it->second.buffer);
  });
}

// init(path of the library, error class, torch's out-of-memory class)
PyObject* init(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 3) return PyErr_Format(PyExc_TypeError, "init: 3 arguments");
  const char* path = PyUnicode_AsUTF8(a[0]);
  if (path == nullptr) return nullptr;
  void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
  if (lib == nullptr) return PyErr_Format(PyExc_OSError, "%s", dlerror());
#define X(name)                                                                        \
  api.name = reinterpret_cast<decltype(api.name)>(dlsym(lib, #name));                  \
  if (api.name == nullptr) return PyErr_Format(PyExc_OSError, "%s: no symbol " #name, path);
  SSM_ENTRY_POINTS(X)
#undef X
  Py_INCREF(a[1]);
  Py_XDECREF(g_error);
  g_error = a[1];
  Py_INCREF(a[2]);
  Py_XDECREF(g_out_of_memory);
  g_out_of_memory = a[2];
  Py_RETURN_NONE;
}

#define METHOD(name, f) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD("init", init),         METHOD("fwd", fwd),           METHOD("bwd", bwd),
                         METHOD("step", step),         METHOD("conv_fwd", conv_fwd), METHOD("conv_bwd", conv_bwd),
                         METHOD("workspace", cached_workspace), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
