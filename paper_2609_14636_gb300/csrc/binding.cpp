// binding.cpp -- the Python module's calls into libstride.so: argument checks
// and marshalling in native code.
//
// A scoring call passes 10 to 20 arguments, most of them tensors.  Checking
// each in Python (type, device, dtype, contiguity, size) and converting them
// for ctypes took longer than the GPU needs for a small call: on the Grace
// host a decode step over 8 rows is issued every 19.7 us that way and every
// 5.0 us this way (which its kernel takes), a 512-row fp32 window of 32,000
// logits every 57 and every 25.5 us (its slices' Python included).
//
// Each function here takes its Python counterpart's arguments in order (None
// for what was not given), makes the same checks and calls the C ABI.  It
// answers with the status code, or with None, having called nothing, when an
// argument is anything but the plain form (an exact torch.Tensor that passes
// every check, an exact int, a float, ...): the caller's general code then
// takes the call, converts what can be converted and says what is wrong with
// the rest.  So what is accepted and what is refused is stated in one place,
// in Python.
#include <Python.h>

#include <string.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "stride.h"

namespace {

struct Entry {
  decltype(&stride_state_init) state_init;
  decltype(&stride_score_batch) score_batch;
  decltype(&stride_score_batch_noalloc) score_batch_noalloc;
  decltype(&stride_score_batch_multi_teacher) score_batch_multi_teacher;
  decltype(&stride_score_step) score_step;
  decltype(&stride_score_step_compact) score_step_compact;
  decltype(&stride_select_restart) select_restart;
  decltype(&stride_buffer_record) buffer_record;
  decltype(&stride_partial_lse) partial_lse;
  decltype(&stride_combine_partials) combine_partials;
  decltype(&stride_scan_logprobs) scan_logprobs;
} g_entry;

const char* const kRowOutputs[] = {"logp_s", "logp_t", "opd", "lse_s", "lse_t", "x_s", "x_t"};
constexpr int kNumRowOutputs = 7;
PyObject* g_row_output_names[kNumRowOutputs];  // interned

constexpr int64_t kStateBytes = sizeof(stride_scan_state);
constexpr int64_t kStatsBytes = sizeof(stride_turn_stats);

// Thrown (and caught in `call` below) when an argument is not of the plain form.
struct NotPlain {};

void need(bool ok) {
  if (!ok) throw NotPlain{};
}

const at::Tensor& tensor(PyObject* o) {
  need(THPVariable_CheckExact(o));
  const at::Tensor& t = THPVariable_Unpack(o);
  need(t.is_cuda() && t.has_storage());
  return t;
}

// A contiguous CUDA tensor of dtype dt and at least `numel` elements.
void* dev(PyObject* o, at::ScalarType dt, int64_t numel = 0) {
  const at::Tensor& t = tensor(o);
  need(t.scalar_type() == dt && t.is_contiguous() && t.numel() >= numel);
  return t.data_ptr();
}

void* dev_or_null(PyObject* o, at::ScalarType dt, int64_t numel = 0) { return o == Py_None ? nullptr : dev(o, dt, numel); }

template <typename T>
T* dev_as(PyObject* o, at::ScalarType dt, int64_t numel = 0) {
  return static_cast<T*>(dev(o, dt, numel));
}
template <typename T>
T* dev_or_null_as(PyObject* o, at::ScalarType dt, int64_t numel = 0) {
  return static_cast<T*>(dev_or_null(o, dt, numel));
}

int64_t integer(PyObject* o) {
  need(PyLong_CheckExact(o));
  int overflow = 0;
  const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
  need(overflow == 0);
  return v;
}

int32_t integer32(PyObject* o) {
  const int64_t v = integer(o);
  need(v >= INT32_MIN && v <= INT32_MAX);
  return (int32_t)v;
}

float real(PyObject* o) {
  need(PyFloat_Check(o) || PyLong_CheckExact(o));
  const double v = PyFloat_AsDouble(o);
  if (PyErr_Occurred()) {
    PyErr_Clear();
    throw NotPlain{};
  }
  return (float)v;
}

// A layout array's count of trajectories or turns.
int32_t count(PyObject* off) {
  const int64_t n = tensor(off).numel() - 1;
  need(n >= INT32_MIN && n <= INT32_MAX);
  return (int32_t)n;
}

void* stream(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  if (PyLong_CheckExact(o)) return reinterpret_cast<void*>((intptr_t)integer(o));
  PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) {
    PyErr_Clear();
    throw NotPlain{};
  }
  int overflow = 0;
  const long long v = PyLong_CheckExact(h) ? PyLong_AsLongLongAndOverflow(h, &overflow) : (overflow = 1, 0);
  Py_DECREF(h);
  need(overflow == 0);
  return reinterpret_cast<void*>((intptr_t)v);
}

int32_t logit_dtype(const at::Tensor& t) {
  need(t.dim() == 2 && t.stride(1) == 1);
  if (t.scalar_type() == at::kBFloat16) return STRIDE_DTYPE_BF16;
  need(t.scalar_type() == at::kFloat);
  return STRIDE_DTYPE_F32;
}

struct Logits {
  const void *S, *T;
  int32_t dtype;
  int64_t rows, ld, V;
  Logits(PyObject* s, PyObject* t, PyObject* v) {
    const at::Tensor &a = tensor(s), &b = tensor(t);
    dtype = logit_dtype(a);
    need(logit_dtype(b) == dtype && a.size(0) == b.size(0) && a.size(1) == b.size(1) && a.stride(0) == b.stride(0));
    S = a.data_ptr();
    T = b.data_ptr();
    rows = a.size(0);
    ld = a.stride(0);
    V = v == Py_None ? a.size(1) : integer(v);
  }
};

struct Lambda {
  const float* each = nullptr;
  float all = NAN;
  Lambda(PyObject* o, int64_t n) {
    if (THPVariable_CheckExact(o))
      each = dev_as<const float>(o, at::kFloat, n);
    else
      all = real(o);
  }
};

struct RowOutputs {
  stride_row_outputs o = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  bool any = false;
  RowOutputs(PyObject* d, int64_t rows) {
    if (d == Py_None) return;
    need(PyDict_CheckExact(d));
    float** const slot[kNumRowOutputs] = {&o.logp_s, &o.logp_t, &o.opd, &o.lse_s, &o.lse_t, &o.x_s, &o.x_t};
    PyObject *key, *value;
    for (Py_ssize_t at = 0; PyDict_Next(d, &at, &key, &value);) {
      need(PyUnicode_CheckExact(key));
      int k = 0;
      while (k < kNumRowOutputs && key != g_row_output_names[k]) ++k;
      if (k == kNumRowOutputs)
        for (k = 0; k < kNumRowOutputs && PyUnicode_CompareWithASCIIString(key, kRowOutputs[k]) != 0; ++k) {
        }
      need(k < kNumRowOutputs);
      *slot[k] = dev_as<float>(value, at::kFloat, rows);
      any = true;
    }
  }
  const stride_row_outputs* ptr() const { return any ? &o : nullptr; }
};

// The trajectory layout, the stop rule and what the scan writes: shared by
// the batch calls and the scan on log-probs.
struct Scan {
  const int64_t *traj_row, *turn_row;
  const int32_t* traj_turn;
  int32_t n_traj, n_turns;
  int64_t begin, end, rows;
  int32_t mode;
  Lambda lam;
  stride_scan_state* state;
  stride_turn_stats* stats;
  int32_t* status;
  double* profile;
  void* stream_;
  // a: traj_row_off, turn_row_off, traj_turn_off, row_begin, row_end, stop_mode, lam, state
  Scan(PyObject* const* a, PyObject* stats_, PyObject* status_, PyObject* profile_, PyObject* st)
      : traj_row(dev_as<const int64_t>(a[0], at::kLong)),
        turn_row(dev_as<const int64_t>(a[1], at::kLong)),
        traj_turn(dev_as<const int32_t>(a[2], at::kInt)),
        n_traj(count(a[0])),
        n_turns(count(a[1])),
        begin(integer(a[3])),
        end(integer(a[4])),
        rows((int64_t)((uint64_t)end - (uint64_t)begin)),
        mode(integer32(a[5])),
        lam(a[6], n_traj),
        state(dev_as<stride_scan_state>(a[7], at::kByte, n_traj * kStateBytes)),
        stats(dev_or_null_as<stride_turn_stats>(stats_, at::kByte, n_turns * kStatsBytes)),
        status(dev_or_null_as<int32_t>(status_, at::kInt, 1)),
        profile(dev_or_null_as<double>(profile_, at::kDouble, 3 * STRIDE_PROFILE_BINS)),
        stream_(stream(st)) {
    need(begin >= 0 && end >= 0);  // (so that `rows` cannot have overflowed)
  }
};

struct Workspace {
  void* p;
  size_t bytes = 0;
  explicit Workspace(PyObject* o) : p(dev_or_null(o, at::kByte)) {
    if (o != Py_None) bytes = (size_t)THPVariable_Unpack(o).numel();
  }
};

// Runs f with the interpreter's lock released, as a ctypes call does.
template <typename F>
int unlocked(F&& f) {
  int rc;
  Py_BEGIN_ALLOW_THREADS rc = f();
  Py_END_ALLOW_THREADS return rc;
}

// A function of N arguments as a Python callable: its status code, or None
// where an argument was not of the plain form.
template <int N, int (*F)(PyObject* const*)>
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", N, n);
    return nullptr;
  }
  try {
    return PyLong_FromLong(F(args));
  } catch (const NotPlain&) {
  } catch (const std::exception&) {  // what torch refuses, the general code meets again
  }
  Py_RETURN_NONE;
}

int state_init(PyObject* const* a) {
  const int64_t n = integer32(a[1]);
  auto* p = dev_as<stride_scan_state>(a[0], at::kByte, n * kStateBytes);
  void* s = stream(a[2]);
  return unlocked([&] { return g_entry.state_init(p, (int32_t)n, s); });
}

// S, T, tokens, traj_row_off, turn_row_off, traj_turn_off, row_begin, row_end, stop_mode, lam, state, out, turn_stats,
// dev_status, workspace, V, stream, profile
int score_batch(PyObject* const* a) {
  const Logits x(a[0], a[1], a[15]);
  const Scan s(a + 3, a[12], a[13], a[17], a[16]);
  const auto* tok = dev_as<const int32_t>(a[2], at::kInt, s.rows);
  const RowOutputs out(a[11], s.rows);
  const Workspace ws(a[14]);
  return unlocked([&] {
    return g_entry.score_batch(x.S, x.T, x.dtype, x.ld, x.V, tok, s.traj_row, s.turn_row, s.traj_turn, s.n_traj, s.n_turns,
                               s.begin, s.end, s.mode, s.lam.each, s.lam.all, s.state, out.ptr(), s.stats, s.profile,
                               s.status, ws.p, ws.bytes, s.stream_);
  });
}

// S, T, tokens, traj_row_off, turn_row_off, traj_turn_off, row_begin, row_end, stop_mode, lam, state, out, turn_stats,
// dev_status, V, stream, profile
int score_batch_noalloc(PyObject* const* a) {
  const Logits x(a[0], a[1], a[14]);
  const Scan s(a + 3, a[12], a[13], a[16], a[15]);
  const int64_t rows = s.rows > 0 ? s.rows : 0;
  const auto* tok = dev_as<const int32_t>(a[2], at::kInt, rows);
  const RowOutputs out(a[11], rows);
  return unlocked([&] {
    return g_entry.score_batch_noalloc(x.S, x.T, x.dtype, x.ld, x.V, tok, s.traj_row, s.turn_row, s.traj_turn, s.n_traj,
                                       s.n_turns, s.begin, s.end, s.mode, s.lam.each, s.lam.all, s.state, out.ptr(),
                                       s.stats, s.profile, s.status, s.stream_);
  });
}

// S, T_domains, traj_domain, traj_T_row0, tokens, traj_row_off, turn_row_off, traj_turn_off, row_begin, row_end,
// stop_mode, lam, state, out, turn_stats, dev_status, workspace, V, stream, profile
int score_batch_multi_teacher(PyObject* const* a) {
  constexpr int kMost = 8;  // the library refuses more; the general code passes any number on
  need(PyList_CheckExact(a[1]));
  const Py_ssize_t D = PyList_GET_SIZE(a[1]);
  need(D >= 1 && D <= kMost);
  const at::Tensor& S = tensor(a[0]);
  const int32_t dtype = logit_dtype(S);
  const void* base[kMost];
  int64_t domain_rows[kMost], ld_T = 0;
  for (Py_ssize_t i = 0; i < D; ++i) {
    const at::Tensor& t = tensor(PyList_GET_ITEM(a[1], i));
    need(logit_dtype(t) == dtype);
    if (i == 0) ld_T = t.stride(0);
    need(t.stride(0) == ld_T);
    base[i] = t.data_ptr();
    domain_rows[i] = t.size(0);
  }
  const Scan s(a + 5, a[14], a[15], a[19], a[18]);
  const auto* domain = dev_as<const uint8_t>(a[2], at::kByte, s.n_traj);
  const auto* row0 = dev_as<const int64_t>(a[3], at::kLong, s.n_traj);
  const auto* tok = dev_as<const int32_t>(a[4], at::kInt, s.rows);
  const RowOutputs out(a[13], s.rows);
  const Workspace ws(a[16]);
  const int64_t V = a[17] == Py_None ? S.size(1) : integer(a[17]), ld = S.stride(0);
  const void* const Sp = S.data_ptr();
  return unlocked([&] {
    return g_entry.score_batch_multi_teacher(Sp, base, domain_rows, (int32_t)D, ld_T, domain, row0, dtype, ld, V, tok,
                                             s.traj_row, s.turn_row, s.traj_turn, s.n_traj, s.n_turns, s.begin, s.end,
                                             s.mode, s.lam.each, s.lam.all, s.state, out.ptr(), s.stats, s.profile,
                                             s.status, ws.p, ws.bytes, s.stream_);
  });
}

// S, T, tokens, turn_end, stop_mode, lam, state, out, stopped_now, turn_out, dev_status, V, stream
int score_step(PyObject* const* a) {
  const Logits x(a[0], a[1], a[11]);
  const int64_t B = x.rows;
  need(B <= INT32_MAX);
  const auto* tok = dev_as<const int32_t>(a[2], at::kInt, B);
  const auto* end = dev_as<const uint8_t>(a[3], at::kByte, B);
  const int32_t mode = integer32(a[4]);
  const Lambda lam(a[5], B);
  auto* state = dev_as<stride_scan_state>(a[6], at::kByte, B * kStateBytes);
  const RowOutputs out(a[7], B);
  auto* now = dev_or_null_as<uint8_t>(a[8], at::kByte, B);
  auto* turn = dev_or_null_as<stride_turn_stats>(a[9], at::kByte, B * kStatsBytes);
  auto* status = dev_or_null_as<int32_t>(a[10], at::kInt, 1);
  void* st = stream(a[12]);
  return unlocked([&] {
    return g_entry.score_step(x.S, x.T, x.dtype, x.ld, x.V, tok, end, (int32_t)B, mode, lam.each, lam.all, state,
                              out.ptr(), now, turn, status, st);
  });
}

// S, T, tokens, turn_end, rollout_idx, stop_mode, lam, state, out, stopped_now, turn_out, dev_status, V, n_rows, stream
int score_step_compact(PyObject* const* a) {
  const Logits x(a[0], a[1], a[12]);
  const at::Tensor &ix = tensor(a[4]), &st_t = tensor(a[7]);
  need(ix.dim() >= 1);
  const int64_t n = a[13] == Py_None ? ix.size(0) : integer(a[13]);
  need(n <= x.rows && n <= INT32_MAX && n >= INT32_MIN);
  const auto* tok = dev_as<const int32_t>(a[2], at::kInt, n);
  const auto* end = dev_as<const uint8_t>(a[3], at::kByte, n);
  const auto* idx = dev_as<const int32_t>(a[4], at::kInt, n);
  const int32_t mode = integer32(a[5]);
  const int64_t n_state = st_t.numel() / kStateBytes;
  need(n_state <= INT32_MAX);
  const Lambda lam(a[6], n_state);
  auto* state = dev_as<stride_scan_state>(a[7], at::kByte);
  const RowOutputs out(a[8], n);
  auto* now = dev_or_null_as<uint8_t>(a[9], at::kByte, n);
  auto* turn = dev_or_null_as<stride_turn_stats>(a[10], at::kByte, n * kStatsBytes);
  auto* status = dev_or_null_as<int32_t>(a[11], at::kInt, 1);
  void* st = stream(a[14]);
  return unlocked([&] {
    return g_entry.score_step_compact(x.S, x.T, x.dtype, x.ld, x.V, tok, end, idx, (int32_t)n, (int32_t)n_state, mode,
                                      lam.each, lam.all, state, out.ptr(), now, turn, status, st);
  });
}

// turn_mean, n_turns, correct, alpha, k_star, k_max, stream
int select_restart(PyObject* const* a) {
  const at::Tensor& m = tensor(a[0]);
  need(m.dim() == 2 && m.size(0) <= INT32_MAX && m.size(1) <= INT32_MAX);
  const int64_t N = m.size(0), T = m.size(1);
  const auto* mean = dev_as<const float>(a[0], at::kFloat);
  const auto* n_turns = dev_as<const int32_t>(a[1], at::kInt, N);
  const auto* ok = dev_or_null_as<const uint8_t>(a[2], at::kByte, N * T);
  const float alpha = real(a[3]);
  auto* k_star = dev_as<int32_t>(a[4], at::kInt, N);
  auto* k_max = dev_as<int32_t>(a[5], at::kInt, N);
  void* st = stream(a[6]);
  return unlocked(
      [&] { return g_entry.select_restart(mean, n_turns, ok, alpha, (int32_t)N, (int32_t)T, k_star, k_max, st); });
}

// buf_mean, buf_n_turns, task_of_traj, k0_of_traj, turn_stats, traj_turn_off, dev_status, stream
int buffer_record(PyObject* const* a) {
  const at::Tensor& m = tensor(a[0]);
  need(m.dim() == 2 && m.size(0) <= INT32_MAX && m.size(1) <= INT32_MAX);
  const int64_t tasks = m.size(0), T = m.size(1);
  const int32_t n = count(a[5]);
  auto* mean = dev_as<float>(a[0], at::kFloat);
  auto* n_turns = dev_as<int32_t>(a[1], at::kInt, tasks);
  const auto* task = dev_as<const int32_t>(a[2], at::kInt, n);
  const auto* k0 = dev_or_null_as<const int32_t>(a[3], at::kInt, n);
  const auto* stats = dev_as<const stride_turn_stats>(a[4], at::kByte);
  const auto* off = dev_as<const int32_t>(a[5], at::kInt, (int64_t)n + 1);
  auto* status = dev_or_null_as<int32_t>(a[6], at::kInt, 1);
  void* st = stream(a[7]);
  return unlocked([&] {
    return g_entry.buffer_record(mean, n_turns, (int32_t)tasks, (int32_t)T, task, k0, stats, off, n, status, st);
  });
}

// S, T, tokens, col0, partials, dev_status, V_shard, stream
int partial_lse(PyObject* const* a) {
  const Logits x(a[0], a[1], a[6]);
  const auto* tok = dev_as<const int32_t>(a[2], at::kInt, x.rows);
  const int64_t col0 = integer(a[3]);
  auto* parts = dev_as<float>(a[4], at::kFloat, x.rows * 6);
  auto* status = dev_or_null_as<int32_t>(a[5], at::kInt, 1);
  void* st = stream(a[7]);
  return unlocked(
      [&] { return g_entry.partial_lse(x.S, x.T, x.dtype, x.ld, x.V, col0, tok, x.rows, parts, status, st); });
}

// partials, logp_s, logp_t, lse_s, lse_t, dev_status, stream
int combine_partials(PyObject* const* a) {
  const at::Tensor& q = tensor(a[0]);
  need(q.dim() == 3 && q.size(2) == 6 && q.size(0) <= INT32_MAX);
  const int64_t n = q.size(0), rows = q.size(1);
  const auto* parts = dev_as<const float>(a[0], at::kFloat);
  float* o[4];
  for (int i = 0; i < 4; ++i) o[i] = dev_or_null_as<float>(a[1 + i], at::kFloat, rows);
  auto* status = dev_or_null_as<int32_t>(a[5], at::kInt, 1);
  void* st = stream(a[6]);
  return unlocked(
      [&] { return g_entry.combine_partials(parts, (int32_t)n, rows, o[0], o[1], o[2], o[3], status, st); });
}

// logp_s, logp_t, traj_row_off, turn_row_off, traj_turn_off, row_begin, row_end, stop_mode, lam, state, opd,
// turn_stats, dev_status, workspace, stream, profile
int scan_logprobs(PyObject* const* a) {
  const Scan s(a + 2, a[11], a[12], a[15], a[14]);
  const auto* ls = dev_as<const float>(a[0], at::kFloat, s.rows);
  const auto* lt = dev_as<const float>(a[1], at::kFloat, s.rows);
  auto* opd = dev_or_null_as<float>(a[10], at::kFloat, s.rows);
  const Workspace ws(a[13]);
  return unlocked([&] {
    return g_entry.scan_logprobs(ls, lt, s.traj_row, s.turn_row, s.traj_turn, s.n_traj, s.n_turns, s.begin, s.end, s.mode,
                                 s.lam.each, s.lam.all, s.state, opd, s.stats, s.profile, s.status, ws.p, ws.bytes,
                                 s.stream_);
  });
}

// The addresses of the library's functions, from the handle that the Python
// module opened (in the order of Entry's members).
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
  constexpr Py_ssize_t kCount = sizeof(Entry) / sizeof(void*);
  if (n != kCount) {
    PyErr_Format(PyExc_TypeError, "%zd addresses expected, got %zd", kCount, n);
    return nullptr;
  }
  void* at[kCount];
  for (Py_ssize_t i = 0; i < n; ++i) {
    at[i] = PyLong_AsVoidPtr(args[i]);
    if (!at[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "a null address");
      return nullptr;
    }
  }
  memcpy(&g_entry, at, sizeof(g_entry));
  Py_RETURN_NONE;
}

#define STRIDE_METHOD(name, n) \
  {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call<n, name>)), METH_FASTCALL, nullptr}

PyMethodDef g_methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(bind)), METH_FASTCALL, nullptr},
    STRIDE_METHOD(state_init, 3),
    STRIDE_METHOD(score_batch, 18),
    STRIDE_METHOD(score_batch_noalloc, 17),
    STRIDE_METHOD(score_batch_multi_teacher, 20),
    STRIDE_METHOD(score_step, 13),
    STRIDE_METHOD(score_step_compact, 15),
    STRIDE_METHOD(select_restart, 7),
    STRIDE_METHOD(buffer_record, 8),
    STRIDE_METHOD(partial_lse, 8),
    STRIDE_METHOD(combine_partials, 7),
    STRIDE_METHOD(scan_logprobs, 16),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  for (int i = 0; i < kNumRowOutputs; ++i) {
    g_row_output_names[i] = PyUnicode_InternFromString(kRowOutputs[i]);
    if (!g_row_output_names[i]) return nullptr;
  }
  return PyModule_Create(&g_module);
}
