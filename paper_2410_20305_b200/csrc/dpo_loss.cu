// dpo_loss / simpo_loss / orpo_loss / dpo_logp_bwd: the DPO loss of Eq. 1 (Section 2.1; the printed ratio of logs is
// read as  -log sigmoid(beta * [(lp_theta(c) - lp_ref(c)) - (lp_theta(r) - lp_ref(r))]),
// averaged over the samples) and its gradient back into the logits,
//     dlogits[t][v] = sum over labels (t, y, g) scored by row t of  coef[g] * (1[v == y] - softmax(logits[t])[v]).
// dpo_logp_bwd is HBM-bound: a live row is read for two sweeps, the second from shared memory (rows up to 96 KB: one
// read from DRAM) or from L2, where not all of it is left (1000 x 128256 bf16: 17 % of the live bytes come from DRAM a
// second time), and written once with streaming stores; rows that score nothing are only written (zeros).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "psa.h"
#include "psa_device.cuh"
#include "psa_internal.h"
#include "psa_launch.cuh"

namespace psa {
namespace {

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint4 ld_16(const uint4* p, uint64_t l2_policy) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(l2_policy));
  return v;
}
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

template <typename T>
struct Elem;
template <>
struct Elem<float> {
  static constexpr int kVec = 4;
  __device__ static void unpack(const uint4& v, float* x) {
    x[0] = __uint_as_float(v.x); x[1] = __uint_as_float(v.y); x[2] = __uint_as_float(v.z); x[3] = __uint_as_float(v.w);
  }
  __device__ static uint4 pack(const float* x) {
    return make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
  }
  __device__ static float load1(const float* p) { return *p; }
  __device__ static void store1(float* p, float x) { *p = x; }
};
template <>
struct Elem<__nv_bfloat16> {
  static constexpr int kVec = 8;
  __device__ static void unpack(const uint4& v, float* x) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[2 * i] = __uint_as_float(w[i] << 16);
      x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  __device__ static uint4 pack(const float* x) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat162 b = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
      w[i] = *reinterpret_cast<uint32_t*>(&b);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
  __device__ static float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  __device__ static void store1(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }
};

struct MaxSum {
  float m, s;
  __device__ void merge(float m2, float s2) {
    const float mn = fmaxf(m, m2);
    if (mn == -INFINITY) return;
    s = s * ex2_approx(m - mn) + s2 * ex2_approx(m2 - mn);
    m = mn;
  }
};

// One block; n_samples is small.
__global__ void dpo_loss_kernel(const float* pol, const float* ref, int n, float beta,
                                float* __restrict__ loss, float* __restrict__ coef) {
  __shared__ float part[32];
  behind_wait();
  float acc = 0.f;
  for (int s = threadIdx.x; s < n; s += blockDim.x) {
    const float z = beta * ((pol[2 * s] - ref[2 * s]) - (pol[2 * s + 1] - ref[2 * s + 1]));
    const float e = expf(-fabsf(z));
    acc += fmaxf(-z, 0.f) + log1pf(e);                   // -log sigmoid(z)
    const float sig_neg = expf(-fmaxf(z, 0.f)) / (1.f + e);   // sigmoid(-z)
    coef[2 * s] = -beta * sig_neg / float(n);
    coef[2 * s + 1] = beta * sig_neg / float(n);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) *loss = n > 0 ? t / float(n) : 0.f;
  }
}

// Length-normalised, reference-free variant (SimPO); one block.
__global__ void simpo_loss_kernel(const float* pol, const int32_t* len, int n, float beta,
                                  float gamma, float* __restrict__ loss, float* __restrict__ coef,
                                  int32_t* __restrict__ status) {
  __shared__ float part[32];
  behind_wait();
  float acc = 0.f;
  for (int s = threadIdx.x; s < n; s += blockDim.x) {
    const int lc = len[2 * s], lr = len[2 * s + 1];
    if (lc < 1 || lr < 1) {
      if (status) atomicOr(status, PSA_DEVSTAT_BAD_SEGMENT);
      coef[2 * s] = 0.f;
      coef[2 * s + 1] = 0.f;
      continue;
    }
    const float z = beta * (pol[2 * s] / float(lc) - pol[2 * s + 1] / float(lr)) - gamma;
    const float e = expf(-fabsf(z));
    acc += fmaxf(-z, 0.f) + log1pf(e);                   // -log sigmoid(z)
    const float sig_neg = expf(-fmaxf(z, 0.f)) / (1.f + e);   // sigmoid(-z)
    coef[2 * s] = -beta * sig_neg / (float(n) * float(lc));
    coef[2 * s + 1] = beta * sig_neg / (float(n) * float(lr));
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) *loss = n > 0 ? t / float(n) : 0.f;
  }
}

// Odds-ratio variant (ORPO); one block.
__global__ void orpo_loss_kernel(const float* pol, const int32_t* len, int n, float lam,
                                 float* __restrict__ loss, float* __restrict__ coef, int32_t* __restrict__ status) {
  __shared__ float part[32];
  behind_wait();
  float acc = 0.f;
  for (int s = threadIdx.x; s < n; s += blockDim.x) {
    const int lc = len[2 * s], lr = len[2 * s + 1];
    if (lc < 1 || lr < 1) {
      if (status) atomicOr(status, PSA_DEVSTAT_BAD_SEGMENT);
      coef[2 * s] = 0.f;
      coef[2 * s + 1] = 0.f;
      continue;
    }
    const float ac = pol[2 * s] / float(lc), ar = pol[2 * s + 1] / float(lr);
    const float qc = -expm1f(ac), qr = -expm1f(ar);          // 1 - P
    const float z = (ac - logf(qc)) - (ar - logf(qr));       // log odds ratio
    const float e = expf(-fabsf(z));
    acc += -ac + lam * (fmaxf(-z, 0.f) + log1pf(e));
    const float sig_neg = expf(-fmaxf(z, 0.f)) / (1.f + e);   // sigmoid(-z)
    coef[2 * s] = (-1.f - lam * sig_neg / qc) / (float(n) * float(lc));
    coef[2 * s + 1] = (lam * sig_neg / qr) / (float(n) * float(lr));
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) *loss = n > 0 ? t / float(n) : 0.f;
  }
}

// Labels scored by one row (its own and forks): (target, coefficient).
constexpr int kMaxLabels = 4;
struct RowLabels {
  int32_t y[kMaxLabels];
  float c[kMaxLabels];
  float csum = 0.f;
  int n = 0;
};

// The labels of `row`, the same in every thread; invalid ones are reported by the thread that is told to, and skipped.
__device__ __forceinline__ RowLabels row_labels(int64_t row, int64_t vocab, const int32_t* targets,
                                                const int32_t* segment_ids, const int32_t* fork_rows,
                                                const int32_t* fork_targets, const int32_t* fork_segments,
                                                int32_t n_forks, int32_t n_segments, const float* coef, bool report,
                                                int32_t* status) {
  RowLabels lab;
  auto add = [&](int32_t y, int32_t g) {
    if (g < 0) return;
    if (g >= n_segments) { if (status && report) atomicOr(status, PSA_DEVSTAT_BAD_SEGMENT); return; }
    if (y < 0 || y >= vocab) { if (status && report) atomicOr(status, PSA_DEVSTAT_BAD_TARGET); return; }
    if (lab.n < kMaxLabels) {
      const float c = coef[g];
#pragma unroll
      for (int a = 0; a < kMaxLabels; ++a)   // (kept in registers: no access by a variable index)
        if (a == lab.n) { lab.y[a] = y; lab.c[a] = c; }
      lab.csum += c;
      ++lab.n;
    }
  };
  add(targets[row], segment_ids[row]);
  bool forked = false;   // every warp looks through the whole fork list, one entry per lane
  for (int f = threadIdx.x & 31; f < n_forks; f += 32) forked |= fork_rows[f] == row;
  if (__any_sync(0xffffffffu, forked))
    for (int f = 0; f < n_forks; ++f)
      if (fork_rows[f] == row) add(fork_targets[f], fork_segments[f]);
  return lab;
}

// Adds one 16-byte vector of logits to a running (max, sum): one rescale of the sum per vector, one exponential per
// element.  A vector of -inf logits (banned or padded vocabulary entries) before anything finite takes its shift
// against 0 instead, so that (-inf) - (-inf) never forms; every term is 0.
template <typename T>
__device__ __forceinline__ void take_vector(MaxSum& acc, const uint4& v) {
  constexpr int E = Elem<T>::kVec;
  float y[E];
  Elem<T>::unpack(v, y);
  float mx = y[0];
#pragma unroll
  for (int j = 1; j < E; ++j) mx = fmaxf(mx, y[j]);
  mx *= kLog2e;
  const float mn = fmaxf(acc.m, mx);
  const float sh = (mn == -INFINITY) ? 0.f : mn;
  float s = acc.s * ex2_approx(acc.m - sh);
#pragma unroll
  for (int j = 0; j < E; ++j) s += ex2_approx(fmaf(y[j], kLog2e, -sh));
  acc.m = mn;
  acc.s = s;
}

// Gradient of one 16-byte vector where no label lies: -csum * softmax.
template <typename T>
__device__ __forceinline__ uint4 grad_vector(const uint4& v, float csum, float lse2) {
  constexpr int E = Elem<T>::kVec;
  float y[E];
  Elem<T>::unpack(v, y);
#pragma unroll
  for (int j = 0; j < E; ++j) y[j] = -csum * ex2_approx(fmaf(y[j], kLog2e, -lse2));
  return Elem<T>::pack(y);
}

// log2 sum_v 2^(x_v log2 e) of the block's running pairs; the same value in every thread.
template <int kThreads>
__device__ __forceinline__ float block_lse2(MaxSum acc, float2* s_part /* [kThreads / 32] */) {
  constexpr int kWarps = kThreads / 32;
  const int lane = threadIdx.x & 31;
  auto over_warp = [](MaxSum& t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, t.m, o);
      const float s2 = __shfl_xor_sync(0xffffffffu, t.s, o);
      t.merge(m2, s2);
    }
  };
  over_warp(acc);
  if (lane == 0) s_part[threadIdx.x >> 5] = make_float2(acc.m, acc.s);
  __syncthreads();
  MaxSum t{-INFINITY, 0.f};
  if (lane < kWarps) t = MaxSum{s_part[lane].x, s_part[lane].y};
  over_warp(t);
  return t.m + log2f(t.s);
}

// Both kernels: one CTA per row.  A dead row is written as zeros without being read; a live row takes a first sweep
// for its log-sum-exp and a second one for the gradient.  The element that a label names is written again by the
// thread that has written it before (its stores stay in order): testing every element for a label inside the sweep
// cost 45 % on 16215 x 128256 bf16 (1325 -> 1950 us), because the vector then lives in indexed local memory.
//
// kStaged: the row is kept in shared memory between the sweeps, brought in by bulk copies in kParts pieces (the first
// sweep starts on the first piece).  Many small CTAs per SM keep loads, exponentials and stores of different rows
// in flight at the same time.
// Otherwise the second sweep reads the row again, from L2: with kPerSm CTAs of 1024 threads per SM, 148 kPerSm rows are
// between their sweeps, loaded with an evict-last policy in the first and evict-first in the second.
template <typename T, int kThreads, bool kStaged, int kPerSm>
__global__ void __launch_bounds__(kThreads, kPerSm)
dpo_logp_bwd_kernel(const T* logits, int64_t vocab, int64_t row_stride, const int32_t* targets, const int32_t* segment_ids,
                    const int32_t* fork_rows, const int32_t* fork_targets, const int32_t* fork_segments,
                    int32_t n_forks, int32_t n_segments, const float* coef, T* __restrict__ dlogits,
                    int32_t* __restrict__ status) {
  constexpr int E = Elem<T>::kVec;
  constexpr int kParts = 4;
  extern __shared__ __align__(16) uint4 s_row[];   // kStaged: the whole vectors of the row
  __shared__ __align__(8) uint64_t s_bar[kParts];
  __shared__ float2 s_part[kThreads / 32];
  __shared__ int s_abort, s_late;
  const int64_t row = blockIdx.x;
  const int tid = threadIdx.x;
  const T* x = logits + row * row_stride;
  T* dx = dlogits + row * row_stride;
  const uint4* xv = reinterpret_cast<const uint4*>(x);
  uint4* dv = reinterpret_cast<uint4*>(dx);
  const int64_t n_vec = vocab / E;
  behind_wait();
  const RowLabels lab = row_labels(row, vocab, targets, segment_ids, fork_rows, fork_targets, fork_segments, n_forks,
                                   n_segments, coef, tid == 0, status);
  if (lab.n == 0) {
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = tid; i < n_vec; i += kThreads) st_stream(dv + i, z);
    for (int64_t j = n_vec * E + tid; j < vocab; j += kThreads) Elem<T>::store1(dx + j, 0.f);
    return;
  }

  MaxSum acc{-INFINITY, 0.f};
  uint64_t keep, last;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(last));
  if constexpr (kStaged) {
    const int n = int(n_vec);
    const int part = (n + kParts * kThreads - 1) / (kParts * kThreads) * kThreads;   // whole turns of the block
    const uint32_t bar0 = dev::smem_u32(s_bar);
    if (tid == 0) {
      s_abort = s_late = 0;
      for (int p = 0; p < kParts; ++p) dev::mbar_init(bar0 + 8 * p, 1);
      dev::fence_mbar_init();
      for (int p = 0; p < kParts; ++p) {
        const int lo = p * part, cnt = min(part, n - lo);
        if (cnt <= 0) break;
        dev::mbar_expect_tx(bar0 + 8 * p, uint32_t(cnt) * 16u);
        dev::bulk_load(dev::smem_u32(s_row + lo), xv + lo, uint32_t(cnt) * 16u, bar0 + 8 * p);
      }
    }
    __syncthreads();
    const dev::WaitCtx wctx{&s_abort, status, dev::kWaitLimitClocks};
    for (int p = 0; p < kParts; ++p) {
      const int lo = p * part, hi = min(lo + part, n);
      if (lo >= hi) break;
      dev::mbar_wait(bar0 + 8 * p, 0, wctx);
      for (int i = lo + tid; i < hi; i += kThreads) take_vector<T>(acc, s_row[i]);
    }
  } else {
    for (int64_t i = tid; i < n_vec; i += kThreads) take_vector<T>(acc, ld_16(xv + i, keep));
  }
  for (int64_t j = n_vec * E + tid; j < vocab; j += kThreads) acc.merge(Elem<T>::load1(x + j) * kLog2e, 1.f);
  const float lse2 = block_lse2<kThreads>(acc, s_part);
  if constexpr (kStaged) {
    if (*static_cast<volatile int*>(&s_abort)) {
      // A wait has expired (and said so): the row is not written, and the CTA stays until the copies into its shared
      // memory have ended, again for a limited time.
      const dev::WaitCtx again{&s_late, status, dev::kWaitLimitClocks};
      const int n = int(n_vec), part = (n + kParts * kThreads - 1) / (kParts * kThreads) * kThreads;
      for (int p = 0; tid == 0 && p < kParts && p * part < n; ++p) dev::mbar_wait(dev::smem_u32(s_bar) + 8 * p, 0, again);
      return;
    }
  }

  if constexpr (kStaged) {
    for (int i = tid; i < int(n_vec); i += kThreads) st_stream(dv + i, grad_vector<T>(s_row[i], lab.csum, lse2));
  } else {
    for (int64_t i = tid; i < n_vec; i += kThreads) st_stream(dv + i, grad_vector<T>(ld_16(xv + i, last), lab.csum, lse2));
  }
  for (int64_t j = n_vec * E + tid; j < vocab; j += kThreads)
    Elem<T>::store1(dx + j, -lab.csum * ex2_approx(fmaf(Elem<T>::load1(x + j), kLog2e, -lse2)));
#pragma unroll
  for (int a = 0; a < kMaxLabels; ++a) {
    if (a >= lab.n) break;
    const int64_t at = lab.y[a], vec = at / E;
    if (int(vec < n_vec ? vec % kThreads : (at - n_vec * E) % kThreads) != tid) continue;
    float add = 0.f;   // labels of this row that name the same token share one element
#pragma unroll
    for (int b = 0; b < kMaxLabels; ++b)
      if (b < lab.n && lab.y[b] == lab.y[a]) add += lab.c[b];
    Elem<T>::store1(dx + at, add - lab.csum * ex2_approx(fmaf(Elem<T>::load1(x + at), kLog2e, -lse2)));
  }
}

// Row size -> kernel (us of the whole call, 2/3 of the rows live; before: 1024 threads, one CTA per SM, two sweeps):
//   up to 32 KB   staged, 128 threads      12180 x 2429 bf16 172 -> 27, 8000 x 8192 bf16 152 -> 38
//   up to 96 KB   staged, 256 threads      2048 x 32000 bf16 68 -> 41 (128 threads: 44; two sweeps: 46 to 52)
//   up to 320 KB  two sweeps, two CTAs per SM   16215 x 128256 bf16 1325 -> 1238 (5.6 TB/s of one read of the live rows
//                 and one write), 4096 x 32000 fp32 184 -> 150 (staged: 175)
//   longer        two sweeps, one CTA per SM    3312 x 115288 fp32, 360 rows live: 264 as before (two per SM: 297, their
//                 296 rows of 461 KB are more than L2 holds)
// Clusters of 2 to 8 CTAs that share a staged row were slower (1538 and more on 16215 x 128256: barriers, and too few
// rows in flight), and so was, over the range, a persistent CTA that streams rows through a ring of bulk copies (1197
// there, but 265 against 247 on 4096 x 50257 fp32 and 94 against 86 on 1000 x 128256 bf16).
constexpr int64_t kStagedSmall = 32 * 1024, kStagedMost = 96 * 1024, kTwoPerSmMost = 320 * 1024;

template <typename T, int kThreads, bool kStaged, int kPerSm>
psa_status_t launch_logp_bwd(const T* logits, int64_t n_rows, int64_t vocab, int64_t row_stride, const int32_t* targets,
                             const int32_t* segment_ids, const int32_t* fork_rows, const int32_t* fork_targets,
                             const int32_t* fork_segments, int32_t n_forks, int32_t n_segments, const float* coef,
                             T* dlogits, int32_t* status, cudaStream_t stream) {
  auto kernel = dpo_logp_bwd_kernel<T, kThreads, kStaged, kPerSm>;
  // (One CTA per SM at kPerSm = 1 is the registers' doing: 1024 threads of more than 32.)
  const size_t smem = kStaged ? size_t(vocab / Elem<T>::kVec) * 16 : 0;
  if (smem > 40 * 1024 &&
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kStagedMost)) != cudaSuccess)
    return PSA_ERR_CUDA;
  // (us of log-probs, loss and gradient with every launch behind the one before: 1515 x 5592 bf16 15.0 -> 13.9, 436 x 2773
  // fp32 13.1 -> 12.1, 4486 x 4935 bf16 21.1 -> 19.9)
  launch_behind(true, kernel, dim3(unsigned(n_rows)), kThreads, smem, stream, logits, vocab, row_stride, targets, segment_ids,
                fork_rows, fork_targets, fork_segments, n_forks, n_segments, coef, dlogits, status);
  return check_last_cuda_error("dpo_logp_bwd launch");
}

template <typename T, typename... Args>
psa_status_t dispatch_logp_bwd(const T* logits, int64_t n_rows, int64_t vocab, Args... args) {
  const int64_t bytes = vocab / Elem<T>::kVec * 16;
  if (bytes <= kStagedSmall) return launch_logp_bwd<T, 128, true, 12>(logits, n_rows, vocab, args...);
  if (bytes <= kStagedMost) return launch_logp_bwd<T, 256, true, 6>(logits, n_rows, vocab, args...);
  if (bytes <= kTwoPerSmMost) return launch_logp_bwd<T, 1024, false, 2>(logits, n_rows, vocab, args...);
  return launch_logp_bwd<T, 1024, false, 1>(logits, n_rows, vocab, args...);
}

}  // namespace
}  // namespace psa

extern "C" psa_status_t dpo_loss(const float* policy_logps, const float* ref_logps, int32_t n_samples, float beta,
                                 float* loss, float* coef, void* stream) {
  if (n_samples < 0 || !loss || (n_samples > 0 && (!policy_logps || !ref_logps || !coef))) return PSA_ERR_INVALID_ARG;
  psa::launch_behind(true, psa::dpo_loss_kernel, dim3(1), 256, 0, cudaStream_t(stream), policy_logps, ref_logps, n_samples, beta, loss, coef);
  return psa::check_last_cuda_error("dpo_loss launch");
}

extern "C" psa_status_t simpo_loss(const float* policy_logps, const int32_t* lengths, int32_t n_samples, float beta,
                                   float gamma, float* loss, float* coef, int32_t* device_status, void* stream) {
  if (n_samples < 0 || !loss || (n_samples > 0 && (!policy_logps || !lengths || !coef))) return PSA_ERR_INVALID_ARG;
  psa::launch_behind(true, psa::simpo_loss_kernel, dim3(1), 256, 0, cudaStream_t(stream), policy_logps, lengths, n_samples, beta, gamma, loss, coef,
                                                             device_status);
  return psa::check_last_cuda_error("simpo_loss launch");
}

extern "C" psa_status_t orpo_loss(const float* policy_logps, const int32_t* lengths, int32_t n_samples, float lambda,
                                  float* loss, float* coef, int32_t* device_status, void* stream) {
  if (n_samples < 0 || !loss || (n_samples > 0 && (!policy_logps || !lengths || !coef))) return PSA_ERR_INVALID_ARG;
  psa::launch_behind(true, psa::orpo_loss_kernel, dim3(1), 256, 0, cudaStream_t(stream), policy_logps, lengths, n_samples, lambda, loss, coef,
                                                            device_status);
  return psa::check_last_cuda_error("orpo_loss launch");
}

extern "C" psa_status_t dpo_logp_bwd(const void* logits, int32_t logits_dtype, int64_t n_rows, int64_t vocab,
                                     int64_t row_stride, const int32_t* targets, const int32_t* segment_ids,
                                     const int32_t* fork_rows, const int32_t* fork_targets,
                                     const int32_t* fork_segments, int32_t n_forks, int32_t n_segments,
                                     const float* coef, void* dlogits, int32_t* device_status, void* stream) {
  if (n_rows < 0 || vocab <= 0 || row_stride < vocab || n_forks < 0 || n_segments < 0) return PSA_ERR_INVALID_ARG;
  if (n_rows > 0 && (!logits || !targets || !segment_ids || !dlogits)) return PSA_ERR_INVALID_ARG;
  if (n_segments > 0 && !coef) return PSA_ERR_INVALID_ARG;
  if (n_forks > 0 && (!fork_rows || !fork_targets || !fork_segments)) return PSA_ERR_INVALID_ARG;
  if (logits_dtype != PSA_DTYPE_F32 && logits_dtype != PSA_DTYPE_BF16) return PSA_ERR_INVALID_ARG;
  if (n_rows > 0x7fffffffLL) return PSA_ERR_UNSUPPORTED;
  const int64_t esz = logits_dtype == PSA_DTYPE_F32 ? 4 : 2;
  if ((reinterpret_cast<uintptr_t>(logits) & 15) || (reinterpret_cast<uintptr_t>(dlogits) & 15) ||
      (n_rows > 1 && ((row_stride * esz) & 15)))   // the stride is not used when there is a single row
    return PSA_ERR_ALIGNMENT;
  if (n_rows == 0) return PSA_OK;
  cudaStream_t st = cudaStream_t(stream);
  if (logits_dtype == PSA_DTYPE_F32)
    return psa::dispatch_logp_bwd(static_cast<const float*>(logits), n_rows, vocab, row_stride, targets, segment_ids,
                                  fork_rows, fork_targets, fork_segments, n_forks, n_segments, coef,
                                  static_cast<float*>(dlogits), device_status, st);
  return psa::dispatch_logp_bwd(static_cast<const __nv_bfloat16*>(logits), n_rows, vocab, row_stride, targets,
                                segment_ids, fork_rows, fork_targets, fork_segments, n_forks, n_segments, coef,
                                static_cast<__nv_bfloat16*>(dlogits), device_status, st);
}
