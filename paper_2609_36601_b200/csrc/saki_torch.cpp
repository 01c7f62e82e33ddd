// The tensor side of the Python binding: argument checks, output tensors, argument records and the call into the C ABI
// for the entry points whose kernels take no longer than that work takes in Python (a forward call on eight rows: 34 us of
// host time through ctypes and fifteen torch.empty calls, against 25 us on the GPU).  No arithmetic: binding.py holds the
// signatures and documentation, libsaki.so the library, whose functions are handed over by address (bind).
#include <Python.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/cuda/CUDAEvent.h>
#include <ATen/ops/empty_native.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <string>
#include <vector>
#include "../../include/saki.h"

namespace {

struct Lib {
  decltype(&saki_route_fwd) route_fwd;
  decltype(&saki_route_fwd_bwd) route_fwd_bwd;
  decltype(&saki_route_fwd_bwd_noalloc) route_fwd_bwd_noalloc;
  decltype(&saki_route_bwd_from_meta) route_bwd_from_meta;
  decltype(&saki_select_tm) select_tm;
  decltype(&saki_spec_verify) spec_verify;
  decltype(&saki_sample_proposal) sample_proposal;
  decltype(&saki_vshard_stage) vshard_stage;
  decltype(&saki_last_error) last_error;
};
Lib lib = {};
PyObject* saki_error = nullptr;     // the exception class

constexpr int N_FIELDS = 15;
// saki_out's members, in order
const char* const FIELD[N_FIELDS] = {"corrected", "token", "teacher_top1", "lambda", "kl", "tv", "accept_prob", "logp_x", "logq_x",
                                     "logT_x", "logp_y", "logq_y", "logT_y", "loss", "row_status"};
// ... and in the order in which the output dict lists them
const int DICT_ORDER[N_FIELDS] = {0, 1, 2, 14, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13};
PyObject* field_key[N_FIELDS];
PyObject *key_loss, *key_logp_tok, *key_row_status, *key_n_accept, *key_next_token, *key_next_is_correction, *key_per_pos;

struct Raised {};     // a Python exception is set
[[noreturn]] void raise_saki(int code, const char* text) {
  PyObject* e = PyObject_CallFunction(saki_error, "is", code, text);
  if (e) { PyErr_SetObject(saki_error, e); Py_DECREF(e); }
  throw Raised();
}
[[noreturn]] void raise_value(const std::string& text) {
  PyErr_SetString(PyExc_ValueError, text.c_str());
  throw Raised();
}
void check_rc(int rc) { if (rc != 0) raise_saki(rc, lib.last_error()); }

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a tensor, got %s", Py_TYPE(o)->tp_name);
    throw Raised();
  }
  return THPVariable_Unpack(o);
}
void* ptr_or_null(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
double number(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Raised();
  return v;
}
uint64_t word(PyObject* o) {       // as a 64-bit field takes an int: the low bits
  const uint64_t v = PyLong_AsUnsignedLongLongMask(o);
  if (v == (uint64_t)-1 && PyErr_Occurred()) throw Raised();
  return v;
}
int64_t integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw Raised();
  return v;
}
void* stream_of(PyObject* o) {     // None: torch's current stream; else the handle
  if (o == Py_None) return (void*)c10::cuda::getCurrentCUDAStream().stream();
  return (void*)word(o);
}
int dtype_code(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return SAKI_F32;
  if (t.scalar_type() == at::kBFloat16) return SAKI_BF16;
  raise_saki(1, (std::string("unsupported logits dtype ") + c10::toString(t.scalar_type())).c_str());
}
int64_t row_stride(const at::Tensor& t) { return t.size(0) > 1 ? t.stride(0) : t.size(1); }

at::Tensor empty(at::IntArrayRef sizes, at::ScalarType type, at::Device dev) {
  // on a GPU the function that the dispatcher would end up in: a call on eight rows, fifteen fields, is about as long as its
  // kernels (17.6 us) with it, 18.1 us, and takes 21.5 us through the dispatcher
  if (dev.is_cuda()) return at::native::empty_cuda(sizes, type, std::nullopt, dev, std::nullopt, std::nullopt);
  return at::empty(sizes, at::TensorOptions().dtype(type).device(dev));
}
at::ScalarType field_type(int k) { return k == 0 ? at::kByte : (k <= 2 || k == 14) ? at::kInt : at::kFloat; }

struct Owned {            // a reference of our own
  PyObject* p;
  explicit Owned(PyObject* o) : p(o) { if (!p) throw Raised(); }
  ~Owned() { Py_XDECREF(p); }
  Owned(const Owned&) = delete;
  PyObject* release() { PyObject* o = p; p = nullptr; return o; }
};
void put(PyObject* dict, PyObject* key, const at::Tensor& t) {
  Owned v(THPVariable_Wrap(t));
  if (PyDict_SetItem(dict, key, v.p) < 0) throw Raised();
}

// The per-position outputs as a dict of tensors, and their record (so may be NULL).  A tensor of its own per field, in the
// dict's order: pieces of one allocation would tie a field that a caller keeps to the fourteen others, could not be saved
// (torch.save refuses one storage under several types), and grow into one another where one is resized.
PyObject* alloc_outputs(int64_t n, at::Device dev, saki_out* so) {
  Owned d(PyDict_New());
  void** const m = (void**)so;
  for (int k : DICT_ORDER) {
    const at::Tensor f = empty({n}, field_type(k), dev);
    put(d.p, field_key[k], f);
    if (so) m[k] = f.data_ptr();
  }
  return d.release();
}
static_assert(sizeof(saki_out) == N_FIELDS * sizeof(void*), "saki_out is fifteen pointers in FIELD's order");

void out_record(PyObject* out, saki_out* so) {
  void** const m = (void**)so;
  for (int k = 0; k < N_FIELDS; ++k) {
    m[k] = nullptr;
    if (PyDict_Check(out)) {
      PyObject* const v = PyDict_GetItemWithError(out, field_key[k]);
      if (!v && PyErr_Occurred()) throw Raised();
      if (v) m[k] = ptr_or_null(v);
    } else {
      Owned v(PyObject_CallMethod(out, "get", "O", field_key[k]));
      m[k] = ptr_or_null(v.p);
    }
  }
}

struct Unlocked {      // without the interpreter lock while it lives, however its scope is left
  PyThreadState* const save = PyEval_SaveThread();
  Unlocked() = default;
  Unlocked(const Unlocked&) = delete;
  ~Unlocked() { PyEval_RestoreThread(save); }
};
template <typename F> auto unlocked(F&& call) {      // a call that may take long or wait
  const Unlocked u;
  return call();
}
template <typename F> PyObject* guarded(F&& body) {  // what torch raises becomes the Python exception that torch makes of it
  HANDLE_TH_ERRORS
  try { return body(); }
  catch (const Raised&) { return nullptr; }
  END_HANDLE_TH_ERRORS
}
void n_args(Py_ssize_t got, Py_ssize_t want) {
  if (got != want) { PyErr_Format(PyExc_TypeError, "%zd arguments, got %zd", want, got); throw Raised(); }
}

// bind(SakiError, address of each function of Lib in order)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    constexpr Py_ssize_t N_LIB = sizeof(Lib) / sizeof(void*);
    n_args(n, 1 + N_LIB);
    Py_INCREF(a[0]);
    Py_XSETREF(saki_error, a[0]);
    void** const f = (void**)&lib;
    for (Py_ssize_t k = 0; k < N_LIB; ++k) f[k] = (void*)word(a[1 + k]);
    Py_RETURN_NONE;
  });
}

// alloc_outputs(n, device)
PyObject* py_alloc_outputs(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 2);
    if (PyLong_Check(a[1])) return alloc_outputs(integer(a[0]), at::Device(at::kCUDA, (c10::DeviceIndex)integer(a[1])), nullptr);
    Owned text(PyObject_Str(a[1]));
    return alloc_outputs(integer(a[0]), at::Device(PyUnicode_AsUTF8(text.p)), nullptr);
  });
}

// route(mode, s, t, proposal, eps, temperature, seed, row_offset, mask, grad_scale, out, dlogits, stream)
// mode 0: saki_route_fwd -> out; 1: saki_route_fwd_bwd, 2: saki_route_fwd_bwd_noalloc -> (out, dlogits)
PyObject* py_route(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 13);
    const int64_t mode = integer(a[0]);
    const at::Tensor &s = tensor(a[1]), &t = tensor(a[2]);
    if (s.dim() != 2 || !t.sizes().equals(s.sizes()) || t.scalar_type() != s.scalar_type() || s.stride(1) != 1 || t.stride(1) != 1)
      raise_saki(1, "student/teacher logits must be [N,V] of the same dtype with unit stride along V");
    saki_in si = {};
    si.student_logits = s.data_ptr(); si.teacher_logits = t.data_ptr();
    si.ld_s = row_stride(s); si.ld_t = row_stride(t);
    si.N = s.size(0); si.V = (int32_t)s.size(1); si.dtype = dtype_code(s);
    si.proposal = (const int32_t*)tensor(a[3]).data_ptr();
    si.eps = (float)number(a[4]); si.temperature = (float)number(a[5]);
    si.seed = word(a[6]); si.row_offset = word(a[7]);
    si.mask = (const uint8_t*)ptr_or_null(a[8]);
    saki_out so;
    PyObject* out_obj = a[10];
    if (out_obj == Py_None) out_obj = alloc_outputs(si.N, s.device(), &so);
    else { Py_INCREF(out_obj); out_record(out_obj, &so); }
    Owned out(out_obj);
    void* const st = stream_of(a[12]);
    if (mode == 0) {
      check_rc(unlocked([&] { return lib.route_fwd(&si, &so, st); }));
      return out.release();
    }
    const float gs = (float)number(a[9]);
    at::Tensor g = a[11] == Py_None ? at::empty_like(s) : tensor(a[11]);
    const int64_t ld_g = row_stride(g);
    void* const gp = g.data_ptr();
    check_rc(unlocked([&] { return (mode == 1 ? lib.route_fwd_bwd : lib.route_fwd_bwd_noalloc)(&si, &so, gp, ld_g, gs, st); }));
    Owned go(a[11] == Py_None ? THPVariable_Wrap(g) : Py_NewRef(a[11]));
    return PyTuple_Pack(2, out.p, go.p);
  });
}

const void* vector(PyObject* o, at::ScalarType type, int64_t n, at::Device dev, const char* name) {
  const at::Tensor& v = tensor(o);
  if (v.scalar_type() != type || v.dim() != 1 || v.size(0) != n || v.device() != dev || !v.is_contiguous())
    raise_value(std::string(name) + " must be a contiguous " +
                (type == at::kByte ? "torch.uint8" : type == at::kInt ? "torch.int32" : "torch.float32") +
                " tensor of length N on the logits' device");
  return v.data_ptr();
}

// meta(s, corrected, proposal, teacher_top1, advantage, temperature, mask, rollout_status, grad_scale, dlogits, stream)
PyObject* py_meta(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 11);
    const at::Tensor& s = tensor(a[0]);
    if (s.dim() != 2 || s.stride(1) != 1) raise_value("logits must be [N,V] with unit stride along V");
    const int64_t N = s.size(0);
    const at::Device dev = s.device();
    at::Tensor g = a[9] == Py_None ? at::empty_like(s) : tensor(a[9]);
    saki_meta_in mi = {};
    mi.student_logits = s.data_ptr(); mi.ld_s = row_stride(s); mi.N = N; mi.V = (int32_t)s.size(1);
    mi.corrected = (const uint8_t*)vector(a[1], at::kByte, N, dev, "corrected");
    mi.proposal = (const int32_t*)vector(a[2], at::kInt, N, dev, "proposal");
    mi.teacher_top1 = (const int32_t*)vector(a[3], at::kInt, N, dev, "teacher_top1");
    mi.advantage = (const float*)vector(a[4], at::kFloat, N, dev, "advantage");
    mi.dtype = dtype_code(s);
    if (a[6] != Py_None) mi.mask = (const uint8_t*)vector(a[6], at::kByte, N, dev, "mask");
    if (a[7] != Py_None) mi.rollout_status = (const uint32_t*)vector(a[7], at::kInt, N, dev, "rollout_status");
    mi.temperature = (float)number(a[5]);
    const float gs = (float)number(a[8]);
    const at::Tensor loss = empty({N}, at::kFloat, dev), logp = empty({N}, at::kFloat, dev), status = empty({N}, at::kInt, dev);
    saki_meta_out mo = {(float*)loss.data_ptr(), (float*)logp.data_ptr(), (uint32_t*)status.data_ptr()};
    void* const st = stream_of(a[10]);
    void* const gp = g.data_ptr();
    const int64_t ld_g = row_stride(g);
    check_rc(unlocked([&] { return lib.route_bwd_from_meta(&mi, &mo, gp, ld_g, gs, st); }));
    Owned d(PyDict_New());
    put(d.p, key_loss, loss); put(d.p, key_logp_tok, logp); put(d.p, key_row_status, status);
    Owned go(a[9] == Py_None ? THPVariable_Wrap(g) : Py_NewRef(a[9]));
    return PyTuple_Pack(2, d.p, go.p);
  });
}

// select(seq_start, corrected, tv, mode, seed, row_offset, mask, rollout_status, stream)
PyObject* py_select(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 9);
    const at::Tensor &seq = tensor(a[0]), &corrected = tensor(a[1]);
    const at::Device dev = corrected.device();
    const int64_t N = corrected.size(0), B = seq.size(0) - 1;
    if (seq.scalar_type() != at::kLong || seq.device() != dev || !seq.is_contiguous())
      raise_value("seq_start must be a contiguous int64 tensor on the same device");
    saki_select_in si = {};
    si.N = N; si.B = B; si.seq_start = (const int64_t*)seq.data_ptr();
    si.corrected = (const uint8_t*)vector(a[1], at::kByte, N, dev, "corrected");
    if (a[2] != Py_None) si.tv = (const float*)vector(a[2], at::kFloat, N, dev, "tv");
    si.mode = (int32_t)integer(a[3]); si.seed = word(a[4]); si.row_offset = word(a[5]);
    if (a[6] != Py_None) si.mask = (const uint8_t*)vector(a[6], at::kByte, N, dev, "mask");
    if (a[7] != Py_None) si.rollout_status = (const uint32_t*)vector(a[7], at::kInt, N, dev, "rollout_status");
    const at::Tensor selected = empty({N}, at::kByte, dev), m = empty({std::max<int64_t>(B, 0)}, at::kInt, dev);
    void* const st = stream_of(a[8]);
    uint8_t* const sp = (uint8_t*)selected.data_ptr();
    int32_t* const mp = (int32_t*)m.data_ptr();
    check_rc(unlocked([&] { return lib.select_tm(&si, sp, mp, st); }));
    Owned x(THPVariable_Wrap(selected)), y(THPVariable_Wrap(m));
    return PyTuple_Pack(2, x.p, y.p);
  });
}

// spec(s, t, draft, eps, temperature, seed, seq_offset, stream)
PyObject* py_spec(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 8);
    const at::Tensor &s = tensor(a[0]), &t = tensor(a[1]), &draft = tensor(a[2]);
    if (s.dim() != 3 || !t.sizes().equals(s.sizes()) || t.scalar_type() != s.scalar_type() || s.stride(2) != 1 || t.stride(2) != 1)
      raise_saki(1, "logits must be [B,K+1,V] with unit stride along V");
    const int64_t B = s.size(0), K1 = s.size(1);
    const at::Device dev = s.device();
    saki_spec_out so = {};
    Owned per(alloc_outputs(B * K1, dev, &so.per_pos));
    const at::Tensor n_accept = empty({B}, at::kInt, dev), next_token = empty({B}, at::kInt, dev), is_corr = empty({B}, at::kByte, dev);
    saki_spec_in si = {};
    si.student_logits = s.data_ptr(); si.teacher_logits = t.data_ptr();
    si.ss_seq = s.stride(0); si.ss_pos = s.stride(1); si.ts_seq = t.stride(0); si.ts_pos = t.stride(1);
    si.B = B; si.K = (int32_t)(K1 - 1); si.V = (int32_t)s.size(2); si.dtype = dtype_code(s);
    si.draft = (const int32_t*)draft.data_ptr(); si.draft_ld = B > 1 ? draft.stride(0) : draft.size(1);
    si.eps = (float)number(a[3]); si.temperature = (float)number(a[4]); si.seed = word(a[5]); si.seq_offset = word(a[6]);
    so.n_accept = (int32_t*)n_accept.data_ptr(); so.next_token = (int32_t*)next_token.data_ptr(); so.next_is_correction = (uint8_t*)is_corr.data_ptr();
    void* const st = stream_of(a[7]);
    check_rc(unlocked([&] { return lib.spec_verify(&si, &so, st); }));
    Owned d(PyDict_New());
    put(d.p, key_n_accept, n_accept); put(d.p, key_next_token, next_token); put(d.p, key_next_is_correction, is_corr);
    if (PyDict_SetItem(d.p, key_per_pos, per.p) < 0) throw Raised();
    return d.release();
  });
}

// propose(s, temperature, seed, row_offset, stream)
PyObject* py_propose(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 5);
    const at::Tensor& s = tensor(a[0]);
    const at::Tensor out = empty({s.size(0)}, at::kInt, s.device());
    const float tau = (float)number(a[1]);
    const uint64_t seed = word(a[2]), off = word(a[3]);
    void* const st = stream_of(a[4]);
    const int code = dtype_code(s);
    int32_t* const op = (int32_t*)out.data_ptr();
    check_rc(unlocked([&] { return lib.sample_proposal(s.data_ptr(), row_stride(s), s.size(0), (int32_t)s.size(1), code, tau, seed, off, op, st); }));
    return THPVariable_Wrap(out);
  });
}

// vshard_local(slices, V, proposal, eps, temperature, seed, row_offset, mask, grad_scale, backward, stream, eager_waves,
// max_waves): the stages of all ranks' slices on one device -> (out, gradient slices, waves, state)
PyObject* py_vshard_local(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    n_args(n, 13);
    Owned seq(PySequence_Fast(a[0], "slices must be a sequence of (student, teacher, first column)"));
    const int world = (int)PySequence_Fast_GET_SIZE(seq.p);
    if (world < 1) raise_value("no slices");
    const bool backward = PyObject_IsTrue(a[9]) == 1;
    std::vector<saki_vshard_in> in((size_t)world);
    std::vector<void*> part((size_t)world), grad;
    std::vector<int64_t> ld_g;
    Owned gs(PyList_New(world));
    at::Device dev = at::kCPU;
    int64_t N = 0;
    for (int r = 0; r < world; ++r) {
      Owned item(PySequence_Fast(PySequence_Fast_GET_ITEM(seq.p, r), "a slice is (student, teacher, first column)"));
      if (PySequence_Fast_GET_SIZE(item.p) != 3) raise_value("a slice is (student, teacher, first column)");
      const at::Tensor &s = tensor(PySequence_Fast_GET_ITEM(item.p, 0)), &t = tensor(PySequence_Fast_GET_ITEM(item.p, 1));
      if (r == 0) { dev = s.device(); N = s.size(0); }
      saki_vshard_in& si = in[(size_t)r];
      si = saki_vshard_in{};
      si.student_logits = s.data_ptr(); si.teacher_logits = t.data_ptr();
      si.ld_s = s.size(0) > 1 ? s.stride(0) : std::max<int64_t>(1, s.size(1));
      si.ld_t = t.size(0) > 1 ? t.stride(0) : std::max<int64_t>(1, t.size(1));
      si.N = s.size(0); si.V_local = (int32_t)s.size(1); si.dtype = dtype_code(s);
      si.V = (int32_t)integer(a[1]); si.v0 = (int32_t)integer(PySequence_Fast_GET_ITEM(item.p, 2));
      si.proposal = (const int32_t*)tensor(a[2]).data_ptr();
      si.eps = (float)number(a[3]); si.temperature = (float)number(a[4]); si.seed = word(a[5]); si.row_offset = word(a[6]);
      si.mask = (const uint8_t*)ptr_or_null(a[7]);
      si.rank = r; si.world = world;
      if (backward) {
        const at::Tensor g = at::empty_like(s);
        grad.push_back(g.data_ptr());
        ld_g.push_back(g.size(0) > 1 ? g.stride(0) : std::max<int64_t>(1, g.size(1)));
        PyList_SET_ITEM(gs.p, r, THPVariable_Wrap(g));
      } else PyList_SET_ITEM(gs.p, r, Py_NewRef(Py_None));
    }
    // the slices' device is the current one from here on: without a stream from the caller, the stages, the zeroing and the reading
    // of the counters take one and the same stream of it
    c10::cuda::OptionalCUDAGuard on_device;
    if (dev.is_cuda()) on_device.set_device(dev);
    const float scale = (float)number(a[8]);
    void* const st = stream_of(a[10]);
    const int eager = (int)integer(a[11]), max_waves = (int)integer(a[12]);
    saki_out so;
    Owned out(alloc_outputs(N, dev, &so));
    // the caller's stream is torch's current one from here on: the counters are zeroed and read in the order of the stages,
    // and what is freed at the end of the call goes back to the allocator on the stream that used it
    c10::cuda::OptionalCUDAStreamGuard on_stream;
    if (a[10] != Py_None && dev.is_cuda()) on_stream.reset_stream(c10::cuda::getStreamFromExternal((cudaStream_t)st, dev.index()));
    const at::Tensor state = empty({N, SAKI_VSHARD_STATE}, at::kDouble, dev), gathered = empty({world, N, SAKI_VSHARD_PARTIALS}, at::kDouble, dev);
    const at::Tensor counts = at::zeros({eager + 1, 2}, at::TensorOptions().dtype(at::kInt).device(dev));
    double* const sp = (double*)state.data_ptr();
    double* const gp = (double*)gathered.data_ptr();
    uint32_t* const np = (uint32_t*)counts.data_ptr();
    for (int r = 0; r < world; ++r) part[(size_t)r] = gp + (int64_t)r * N * SAKI_VSHARD_PARTIALS;   // where the all-gather would put it
    auto stage = [&](int k, uint32_t* count, int flags) {
      check_rc(unlocked([&] {
        return lib.vshard_stage(in.data(), world, k, sp, (double* const*)part.data(), gp, k == 2 && backward ? (void* const*)grad.data() : nullptr,
                                ld_g.data(), scale, k == 3 ? &so : nullptr, count, flags, st);
      }));
    };
    // the rows still solving after stage 0 and after each wave, and those marked for float64 (page-locked: the device is idle
    // until the host has looked at them)
    const at::Tensor h = at::empty({eager + 1, 2}, at::TensorOptions().dtype(at::kInt).pinned_memory(dev.is_cuda()));
    at::cuda::CUDAEvent copied;
    auto read = [&] {
      return unlocked([&] {
        h.copy_(counts, true);
        if (dev.is_cuda()) { copied.record(c10::cuda::getCurrentCUDAStream(dev.index())); copied.synchronize(); }
        return (const int32_t*)h.data_ptr();
      });
    };
    int waves = 0;
    if (N > 0) {
      constexpr int NONE = SAKI_VSHARD_NONE_MARKED;
      stage(0, np, NONE);                                    // a wave's combine is the first that can mark a row
      for (int k = 0; k < eager; ++k) stage(1, np + 2 * (1 + k), k == 0 ? NONE : 0);
      const int32_t* c = read();
      while (waves < eager && c[2 * waves] > 0) ++waves;
      int32_t sum = c[2 * eager], left = sum, marked = 0;
      for (int k = 0; k < eager; ++k) marked += c[2 * k + 1];
      while (left > 0 && waves < max_waves) {
        stage(1, np + 2 * eager, 0);                         // (adds to the last pair)
        ++waves;
        c = read();
        left = c[2 * eager] - sum;
        sum = c[2 * eager];
      }
      marked += c[2 * eager + 1];
      stage(2, nullptr, marked ? 0 : NONE);
      stage(3, nullptr, marked ? 0 : NONE);
    }
    Owned w(PyLong_FromLong(waves)), sv(THPVariable_Wrap(state));
    return PyTuple_Pack(4, out.p, gs.p, w.p, sv.p);
  });
}

PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, nullptr},
    {"alloc_outputs", (PyCFunction)(void (*)(void))py_alloc_outputs, METH_FASTCALL, nullptr},
    {"route", (PyCFunction)(void (*)(void))py_route, METH_FASTCALL, nullptr},
    {"meta", (PyCFunction)(void (*)(void))py_meta, METH_FASTCALL, nullptr},
    {"select", (PyCFunction)(void (*)(void))py_select, METH_FASTCALL, nullptr},
    {"spec", (PyCFunction)(void (*)(void))py_spec, METH_FASTCALL, nullptr},
    {"propose", (PyCFunction)(void (*)(void))py_propose, METH_FASTCALL, nullptr},
    {"vshard_local", (PyCFunction)(void (*)(void))py_vshard_local, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_saki_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// the torch and the interpreter that this file was compiled against, to be found in the binary
extern "C" __attribute__((used, visibility("default"))) const char saki_built_for[] = SAKI_BUILT_FOR;

PyMODINIT_FUNC PyInit__saki_torch(void) {
  for (int k = 0; k < N_FIELDS; ++k) field_key[k] = PyUnicode_InternFromString(FIELD[k]);
  key_loss = PyUnicode_InternFromString("loss"); key_logp_tok = PyUnicode_InternFromString("logp_tok");
  key_row_status = PyUnicode_InternFromString("row_status"); key_n_accept = PyUnicode_InternFromString("n_accept");
  key_next_token = PyUnicode_InternFromString("next_token"); key_next_is_correction = PyUnicode_InternFromString("next_is_correction");
  key_per_pos = PyUnicode_InternFromString("per_pos");
  return PyModule_Create(&module);
}
