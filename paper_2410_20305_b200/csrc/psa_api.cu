// extern "C" entry points psa_fwd / psa_bwd / psa_step_host: argument validation, then the launchers.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <mutex>

#include "psa_internal.h"

namespace {
inline bool misaligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0; }
}  // namespace

namespace psa {
// The plan's device blob lives on the device that was current when it was uploaded; a launch
// from another device would hand the kernels pointers that mean nothing there.
bool plan_on_current_device(const psa_plan_t* plan) {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess && dev == plan->device;
}
}  // namespace psa

namespace psa {
namespace {
// Copy streams of psa_step_host.  A pair belongs to one caller's stream at a time: what is enqueued on it waits for that
// stream, so a call on another stream gets the pair only when both of its streams have run dry, and otherwise another
// pair or none (it then uses its own stream alone).  So no call waits for another one's stream.
struct HostPipe {
  cudaStream_t in = nullptr, out = nullptr;   // copies in, copies out
  cudaEvent_t event = nullptr;
  unsigned long long owner = 0;                // id of the stream of the last call
  bool taken = false;                          // a call is enqueueing
};
// Two pairs: steps on two streams overlap each within themselves, and a third one overlaps with them as a whole.
constexpr int kHostPipes = 2, kDevicesMax = 32;
std::mutex g_pipe_mutex;
HostPipe g_pipes[kDevicesMax][kHostPipes];
bool g_pipes_made[kDevicesMax];

// While it lives, a capture in another thread does not mind this thread's calls (none of them touches its streams).
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

bool run_dry(cudaStream_t s) {
  const cudaError_t e = cudaStreamQuery(s);
  if (e == cudaErrorNotReady) cudaGetLastError();   // (an answer, not an error of this call)
  return e == cudaSuccess;
}

// A pair for one call on `stream`, or null.
HostPipe* take_host_pipe(int device, cudaStream_t stream) {
  unsigned long long id = 0;   // (unlike a handle, never given to another stream)
  if (device >= kDevicesMax) return nullptr;
  if (cudaStreamGetId(stream, &id) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  RelaxedCapture relaxed;
  HostPipe* found = nullptr;
  for (HostPipe& p : g_pipes[device])
    if (p.event && p.owner == id) {
      if (p.taken) return nullptr;   // another thread enqueues on the same stream
      found = &p;
    }
  for (HostPipe& p : g_pipes[device])
    if (!found && p.event && !p.taken && run_dry(p.in) && run_dry(p.out)) found = &p;
  if (found) {
    found->owner = id;
    found->taken = true;
  }
  return found;
}

void give_host_pipe(HostPipe* p) {
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  p->taken = false;
}
}  // namespace

void make_host_pipes(int device) {
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  if (device < 0 || device >= kDevicesMax || g_pipes_made[device]) return;
  g_pipes_made[device] = true;
  RelaxedCapture relaxed;
  for (HostPipe& p : g_pipes[device]) {
    if (cudaStreamCreateWithFlags(&p.in, cudaStreamNonBlocking) == cudaSuccess &&
        cudaStreamCreateWithFlags(&p.out, cudaStreamNonBlocking) == cudaSuccess &&
        cudaEventCreateWithFlags(&p.event, cudaEventDisableTiming) == cudaSuccess)
      continue;
    cudaGetLastError();   // without a pair the calls use their own stream
    if (p.in) cudaStreamDestroy(p.in);
    if (p.out) cudaStreamDestroy(p.out);
    p = HostPipe{};
  }
}
}  // namespace psa

extern "C" psa_status_t psa_fwd(const psa_plan_t* plan, const void* q, const void* k, const void* v, void* o,
                                float* lse, int32_t* device_status, void* stream) {
  if (!plan) return PSA_ERR_INVALID_ARG;
  if (plan->T == 0) return PSA_OK;
  if (!plan->d_blob) return PSA_ERR_INVALID_ARG;  // host-only plan: upload it first
  if (!q || !k || !v || !o || !lse) return PSA_ERR_INVALID_ARG;
  if (misaligned(q, 16) || misaligned(k, 16) || misaligned(v, 16) || misaligned(o, 16) || misaligned(lse, 4))
    return PSA_ERR_ALIGNMENT;
  if (!psa::plan_on_current_device(plan)) return PSA_ERR_INVALID_ARG;
  psa::note_plan_use(plan, stream);
  return psa::launch_fwd(plan, plan->whole, q, k, v, o, lse, device_status, stream);
}

extern "C" psa_status_t psa_bwd(const psa_plan_t* plan, const void* d_o, const void* q, const void* k,
                                const void* v, const void* o, const float* lse, void* dq, void* dk, void* dv,
                                void* workspace, int32_t* device_status, void* stream) {
  if (!plan) return PSA_ERR_INVALID_ARG;
  if (plan->T == 0) return PSA_OK;
  if (!plan->d_blob) return PSA_ERR_INVALID_ARG;
  if (!d_o || !q || !k || !v || !o || !lse || !dq || !dk || !dv || !workspace) return PSA_ERR_INVALID_ARG;
  if (misaligned(d_o, 16) || misaligned(q, 16) || misaligned(k, 16) || misaligned(v, 16) || misaligned(o, 16) ||
      misaligned(dq, 16) || misaligned(dk, 16) || misaligned(dv, 16) || misaligned(lse, 4) ||
      misaligned(workspace, 256))
    return PSA_ERR_ALIGNMENT;
  if (!psa::plan_on_current_device(plan)) return PSA_ERR_INVALID_ARG;
  psa::note_plan_use(plan, stream);
  return psa::launch_bwd(plan, plan->whole, d_o, q, k, v, o, lse, dq, dk, dv, workspace, false, device_status, stream);
}

extern "C" psa_status_t psa_bwd_f32(const psa_plan_t* plan, const void* d_o, const void* q, const void* k,
                                    const void* v, const void* o, const float* lse, float* dq, float* dk,
                                    float* dv, void* workspace, int32_t* device_status, void* stream) {
  if (!plan) return PSA_ERR_INVALID_ARG;
  if (plan->T == 0) return PSA_OK;
  if (!plan->d_blob) return PSA_ERR_INVALID_ARG;
  if (!d_o || !q || !k || !v || !o || !lse || !dq || !dk || !dv || !workspace) return PSA_ERR_INVALID_ARG;
  if (misaligned(d_o, 16) || misaligned(q, 16) || misaligned(k, 16) || misaligned(v, 16) || misaligned(o, 16) ||
      misaligned(dq, 16) || misaligned(dk, 16) || misaligned(dv, 16) || misaligned(lse, 4) ||
      misaligned(workspace, 256))
    return PSA_ERR_ALIGNMENT;
  if (!psa::plan_on_current_device(plan)) return PSA_ERR_INVALID_ARG;
  psa::note_plan_use(plan, stream);
  return psa::launch_bwd(plan, plan->whole, d_o, q, k, v, o, lse, dq, dk, dv, workspace, true, device_status, stream);
}

namespace {
// Arena of psa_step_host: the nine tensors and the backward scratch, each 256-byte aligned.
struct StepArena {
  size_t q, k, v, d_o, o, lse, dq, dk, dv, ws, bytes;
};
StepArena step_arena_layout(const psa_plan_t* plan) {
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  const size_t nq = size_t(plan->T) * plan->Hq * plan->d * 2, nk = size_t(plan->T) * plan->Hkv * plan->d * 2;
  StepArena a;
  size_t off = 0;
  auto take = [&](size_t n) { const size_t at = off; off += up(n); return at; };
  a.q = take(nq); a.k = take(nk); a.v = take(nk); a.d_o = take(nq); a.o = take(nq);
  a.lse = take(size_t(plan->Hq) * plan->T * 4);
  a.dq = take(nq); a.dk = take(nk); a.dv = take(nk);
  a.ws = take(plan->bwd_workspace_bytes);
  a.bytes = off;
  return a;
}
}  // namespace

extern "C" size_t psa_step_host_arena_bytes(const psa_plan_t* plan) {
  return plan ? step_arena_layout(plan).bytes : 0;
}

extern "C" psa_status_t psa_step_host(const psa_plan_t* plan, const void* h_q, const void* h_k, const void* h_v,
                                      const void* h_do, void* h_o, float* h_lse, void* h_dq, void* h_dk,
                                      void* h_dv, void* arena, size_t arena_bytes, int32_t* device_status,
                                      void* stream) {
  if (!plan) return PSA_ERR_INVALID_ARG;
  if (plan->T == 0) return PSA_OK;
  if (!plan->d_blob) return PSA_ERR_INVALID_ARG;
  if (!h_q || !h_k || !h_v || !h_do || !h_o || !h_lse || !h_dq || !h_dk || !h_dv || !arena) return PSA_ERR_INVALID_ARG;
  const StepArena a = step_arena_layout(plan);
  if (arena_bytes < a.bytes) return PSA_ERR_INVALID_ARG;
  if (misaligned(arena, 256)) return PSA_ERR_ALIGNMENT;
  if (!psa::plan_on_current_device(plan)) return PSA_ERR_INVALID_ARG;
  psa::note_plan_use(plan, stream);
  char* base = static_cast<char*>(arena);
  const cudaStream_t st = cudaStream_t(stream);
  const size_t q_row = size_t(plan->Hq) * plan->d * 2, kv_row = size_t(plan->Hkv) * plan->d * 2, lse_row = size_t(plan->T) * 4;
  // Copies and kernels of one part of the pack.
  auto copy_in = [&](const psa::PlanPart& w, const void* src, size_t at, size_t row, cudaStream_t s) {
    return cudaMemcpyAsync(base + at + w.row0 * row, static_cast<const char*>(src) + w.row0 * row,
                           (w.row1 - w.row0) * row, cudaMemcpyHostToDevice, s) == cudaSuccess;
  };
  auto copy_in_qkv = [&](const psa::PlanPart& w, cudaStream_t s) {
    return copy_in(w, h_q, a.q, q_row, s) && copy_in(w, h_k, a.k, kv_row, s) && copy_in(w, h_v, a.v, kv_row, s);
  };
  auto copy_in_do = [&](const psa::PlanPart& w, cudaStream_t s) { return copy_in(w, h_do, a.d_o, q_row, s); };
  auto copy_out = [&](const psa::PlanPart& w, void* dst, size_t at, size_t row, cudaStream_t s) {
    return cudaMemcpyAsync(static_cast<char*>(dst) + w.row0 * row, base + at + w.row0 * row, (w.row1 - w.row0) * row,
                           cudaMemcpyDeviceToHost, s) == cudaSuccess;
  };
  auto copy_out_lse = [&](const psa::PlanPart& w, cudaStream_t s) {
    if (w.row0 == 0 && w.row1 == plan->T)
      return cudaMemcpyAsync(h_lse, base + a.lse, lse_row * plan->Hq, cudaMemcpyDeviceToHost, s) == cudaSuccess;
    return cudaMemcpy2DAsync(h_lse + w.row0, lse_row, base + a.lse + size_t(w.row0) * 4, lse_row,
                             size_t(w.row1 - w.row0) * 4, plan->Hq, cudaMemcpyDeviceToHost, s) == cudaSuccess;
  };
  auto forward = [&](const psa::PlanPart& w) {
    return psa::launch_fwd(plan, w, base + a.q, base + a.k, base + a.v, base + a.o, reinterpret_cast<float*>(base + a.lse),
                           device_status, stream);
  };
  auto backward = [&](const psa::PlanPart& w) {
    return psa::launch_bwd(plan, w, base + a.d_o, base + a.q, base + a.k, base + a.v, base + a.o,
                           reinterpret_cast<const float*>(base + a.lse), base + a.dq, base + a.dk, base + a.dv,
                           base + a.ws, false, device_status, stream);
  };

  // A captured call, and a pack that is not worth splitting, run in stream order on the caller's stream.
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  psa::HostPipe* pipe = nullptr;
  if (!plan->parts.empty() && cudaStreamIsCapturing(st, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone)
    pipe = psa::take_host_pipe(plan->device, st);
  if (!pipe) {
    const psa::PlanPart& w = plan->whole;
    if (!copy_in_qkv(w, st) || !copy_in_do(w, st)) return psa::check_last_cuda_error("psa_step_host copy in");
    psa_status_t rc = forward(w);
    if (rc != PSA_OK) return rc;
    // o and lse are final after the forward: their copies out can leave before the backward runs.
    if (!copy_out(w, h_o, a.o, q_row, st) || !copy_out_lse(w, st))
      return psa::check_last_cuda_error("psa_step_host copy out");
    rc = backward(w);
    if (rc != PSA_OK) return rc;
    if (!copy_out(w, h_dq, a.dq, q_row, st) || !copy_out(w, h_dk, a.dk, kv_row, st) || !copy_out(w, h_dv, a.dv, kv_row, st))
      return psa::check_last_cuda_error("psa_step_host copy out");
    return PSA_OK;
  }

  // The parts one after the other: copies in on one stream, kernels on the caller's, copies out on a third, so that
  // both directions of the link and the kernels work at the same time; within a part d_o arrives under the forward
  // and o leaves under the backward.  7727 tokens, 32/8 heads of 128 (158 MB in, 159 MB out): 6080 -> 4460 us, where
  // the link takes 2870 us for each direction alone and 3670 us for both at once; 3333 tokens of one sample, 8/2
  // heads: 1002 -> 800 us.
  // An event may be recorded again as soon as the wait for its previous recording has been enqueued.
  auto order = [&](cudaStream_t before, cudaStream_t after) {
    return cudaEventRecord(pipe->event, before) == cudaSuccess && cudaStreamWaitEvent(after, pipe->event, 0) == cudaSuccess;
  };
  psa_status_t rc = PSA_OK;
  bool ok = order(st, pipe->in) && copy_in_qkv(plan->parts[0], pipe->in);
  for (size_t i = 0; ok && i < plan->parts.size(); ++i) {
    const psa::PlanPart& w = plan->parts[i];
    ok = order(pipe->in, st) && copy_in_do(w, pipe->in);
    if (!ok || (rc = forward(w)) != PSA_OK) break;
    ok = order(st, pipe->out) && copy_out(w, h_o, a.o, q_row, pipe->out) && copy_out_lse(w, pipe->out) && order(pipe->in, st);
    if (ok && i + 1 < plan->parts.size()) ok = copy_in_qkv(plan->parts[i + 1], pipe->in);
    if (!ok || (rc = backward(w)) != PSA_OK) break;
    ok = order(st, pipe->out) && copy_out(w, h_dq, a.dq, q_row, pipe->out) && copy_out(w, h_dk, a.dk, kv_row, pipe->out) &&
         copy_out(w, h_dv, a.dv, kv_row, pipe->out);
  }
  // The caller's stream ends behind both, also where a part could not be enqueued.
  const bool joined_in = order(pipe->in, st), joined_out = order(pipe->out, st);
  psa::give_host_pipe(pipe);
  if (rc != PSA_OK) return rc;
  if (!ok || !joined_in || !joined_out) {
    const psa_status_t e = psa::check_last_cuda_error("psa_step_host");
    return e == PSA_OK ? PSA_ERR_CUDA : e;
  }
  return PSA_OK;
}

namespace psa {
psa_status_t check_last_cuda_error(const char* where) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return PSA_OK;
  if (std::getenv("PSA_DEBUG")) std::fprintf(stderr, "libpsa: %s: %s\n", where, cudaGetErrorString(e));
  return PSA_ERR_CUDA;
}

ProfileEvents g_profile[5] = {{nullptr, nullptr}, {nullptr, nullptr}, {nullptr, nullptr}, {nullptr, nullptr},
                              {nullptr, nullptr}};
ProfileScope::ProfileScope(int which, void* s) : ev(g_profile[which]), stream(s) {
  if (ev.start) cudaEventRecord(cudaEvent_t(ev.start), cudaStream_t(stream));
}
ProfileScope::~ProfileScope() {
  if (ev.stop) cudaEventRecord(cudaEvent_t(ev.stop), cudaStream_t(stream));
}
}  // namespace psa

extern "C" psa_status_t psa_profile_events(int32_t which, void* start, void* stop) {
  if (which < 0 || which > 4 || ((start == nullptr) != (stop == nullptr))) return PSA_ERR_INVALID_ARG;
  psa::g_profile[which] = psa::ProfileEvents{start, stop};
  return PSA_OK;
}
