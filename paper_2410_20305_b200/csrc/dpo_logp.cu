// dpo_logp: per-response summed log-probabilities (Section 2.1; responses are
// recovered from their boundaries, Section 3.2).  HBM-bound: one small CTA streams one
// live logits row exactly once with 16-byte coalesced loads, keeps a running
// (max, sum of exp) per thread in fp32, merges across the warp with shuffles and
// across warps through shared memory, and adds  logit[target] - lse  into
// out[segment] with one atomic per scored label, or, where the caller gives scratch for them, into
// fp64 sums: a response of 250 tokens is then off by its lse's and one final rounding (3e-8) instead
// of 250 (1e-7 to 4e-7).  Every term is at most 0, so a sum only falls while its rows arrive, and
// so does its rounding to fp32: out[segment] is the lowest of the roundings that the rows have seen,
// whatever their order, and nothing has to wait for the last row.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "psa.h"
#include "psa_internal.h"
#include "psa_launch.cuh"

namespace psa {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr double kLn2 = 0.6931471805599453;

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Streaming 16-byte load that does not linger in L1.
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

template <typename T>
struct Vec;  // 16 bytes of logits -> floats
template <>
struct Vec<float> {
  static constexpr int kElems = 4;
  __device__ static void unpack(const uint4& v, float* x) {
    x[0] = __uint_as_float(v.x); x[1] = __uint_as_float(v.y);
    x[2] = __uint_as_float(v.z); x[3] = __uint_as_float(v.w);
  }
  __device__ static float load1(const float* p) { return *p; }
};
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int kElems = 8;
  __device__ static void unpack(const uint4& v, float* x) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[2 * i] = __uint_as_float(w[i] << 16);
      x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  __device__ static float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
};

// Running log2-domain (max, sum): sum = sum_i 2^(y_i - m), y = x * log2(e).
struct MaxSum {
  float m, s;
  __device__ void merge(float m2, float s2) {
    const float mn = fmaxf(m, m2);
    if (mn == -INFINITY) {   // nothing finite on either side: both sums are 0, or NaN where a logit was
      s += s2;
      return;
    }
    s = s * ex2_approx(m - mn) + s2 * ex2_approx(m2 - mn);
    m = mn;
  }
};

// One launch for both arrays.  With add_f64 it replaced a pass over the segment ids that counted the live rows, the count
// of every row at its end and a last row that rounded all sums (small launches), or a second kernel that did (large ones);
// us of the whole call, before -> now, and with fp32 atomics behind a memset: 6335 x 6215 bf16 24.0 -> 15.3 (18.4),
// 12000 x 1000 bf16 with 100 responses 21.9 -> 13.6 (16.0), with 4000 responses 47.2 -> 10.5 (10.4), 700 x 1024 fp32
// 6.9 -> 4.7 (6.3), 8192 x 50257 fp32 147.5 -> 143.3 (167).
__global__ void dpo_logp_clear_kernel(float* __restrict__ out, double* __restrict__ sums, int32_t n_segments) {
  const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  behind_wait();
  behind_go();
  if (g < n_segments) {
    out[g] = 0.f;
    sums[g] = 0.0;
  }
}

// Adds a term (a log-probability) to the fp64 sum and lowers out to its rounding.
__device__ __forceinline__ void add_f64(double* sum, float* out, double term) {
  // a probability that rounding has put above 1 counts as 1, so that the sum never rises (a NaN stays one)
  if (term > 0.0) term = 0.0;
  const double now = atomicAdd(sum, term) + term;
  // The bits of floats that are not positive grow as the values fall; the largest of all is a NaN.
  atomicMax(reinterpret_cast<uint32_t*>(out), now == now ? __float_as_uint(float(now)) : 0xffffffffu);
}

template <typename T, int kUnroll, int kLogpThreads>
__global__ void __launch_bounds__(kLogpThreads)
dpo_logp_kernel(const T* __restrict__ logits, int64_t vocab, int64_t row_stride, const int32_t* __restrict__ targets,
                const int32_t* __restrict__ segment_ids, const int32_t* __restrict__ fork_rows,
                const int32_t* __restrict__ fork_targets, const int32_t* __restrict__ fork_segments, int32_t n_forks,
                int32_t n_segments, float* __restrict__ out, double* __restrict__ sums /* [n_segments], or null */,
                int32_t* __restrict__ status) {
  constexpr int E = Vec<T>::kElems;
  const int64_t row = blockIdx.x;
  const int32_t seg = segment_ids[row];
  // Every warp looks through the whole fork list, one entry per lane: the answer is block-uniform.
  bool forked = false;
  for (int f = threadIdx.x & 31; f < n_forks; f += 32) forked |= fork_rows[f] == row;
  forked = __any_sync(0xffffffffu, forked);
  if (seg < 0 && !forked) {            // dead row: its logits are never read
    if (row == 0) behind_wait();       // (the launch as a whole does not end before the kernel that clears the sums)
    return;
  }

  const T* x = logits + row * row_stride;
  const uint4* xv = reinterpret_cast<const uint4*>(x);
  const int64_t n_vec = vocab / E;
  MaxSum acc{-INFINITY, 0.f};

  // Main loop: kUnroll independent 16-byte loads in flight per thread.
  int64_t i = threadIdx.x;
  for (; i + int64_t(kUnroll - 1) * kLogpThreads < n_vec; i += int64_t(kUnroll) * kLogpThreads) {
    uint4 v[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) v[u] = ld_stream(xv + i + int64_t(u) * kLogpThreads);
    float y[kUnroll * E];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) Vec<T>::unpack(v[u], y + u * E);
    float mx = y[0];
#pragma unroll
    for (int j = 1; j < kUnroll * E; ++j) mx = fmaxf(mx, y[j]);
    mx *= kLog2e;
    // One rescale of the running sum per chunk, one exponential per element.
    const float mn = fmaxf(acc.m, mx);
    // A chunk of -inf logits (banned or padded vocabulary entries) before anything finite:
    // the shift is taken against 0 instead, so that (-inf) - (-inf) never forms; every term is 0.
    const float sh = (mn == -INFINITY) ? 0.f : mn;
    float s = acc.s * ex2_approx(acc.m - sh);
#pragma unroll
    for (int j = 0; j < kUnroll * E; ++j) s += ex2_approx(fmaf(y[j], kLog2e, -sh));
    acc.m = mn;
    acc.s = s;
  }
  for (; i < n_vec; i += kLogpThreads) {
    float y[E];   // (one vector at a time, as above: 12180 x 2429 bf16, whose rows are all remainder, 22.6 -> 21.6 us)
    Vec<T>::unpack(ld_stream(xv + i), y);
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
  for (int64_t j = n_vec * E + threadIdx.x; j < vocab; j += kLogpThreads) {  // ragged tail of the row
    const float y = Vec<T>::load1(x + j), m2 = y * kLog2e;
    if (y != -INFINITY) acc.merge(m2, ex2_approx(fmaf(y, kLog2e, -m2)));     // (what the product's rounding has left)
  }

  // Warp merge by shuffles, then across warps through shared memory.
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, acc.m, o);
    const float s2 = __shfl_xor_sync(0xffffffffu, acc.s, o);
    acc.merge(m2, s2);
  }
  __shared__ float sm_m[kLogpThreads / 32], sm_s[kLogpThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sm_m[warp] = acc.m; sm_s[warp] = acc.s; }
  __syncthreads();
  if (warp == 0) {
    MaxSum t{-INFINITY, 0.f};
    if (lane < kLogpThreads / 32) { t.m = sm_m[lane]; t.s = sm_s[lane]; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, t.m, o);
      const float s2 = __shfl_xor_sync(0xffffffffu, t.s, o);
      t.merge(m2, s2);
    }
    behind_wait();   // the sums are cleared
    if (lane == 0) {
      // log2 of the probability, the maximum taken off before anything is rounded to fp32: the term of a token
      // that takes nearly all of the probability is then near 0 itself, not the difference of two numbers like 50
      const double m = t.m, log2s = log2f(t.s);
      auto score = [&](int32_t y, int32_t g) {
        if (g < 0) return;
        if (g >= n_segments) { if (status) atomicOr(status, PSA_DEVSTAT_BAD_SEGMENT); return; }
        if (y < 0 || y >= vocab) { if (status) atomicOr(status, PSA_DEVSTAT_BAD_TARGET); return; }
        const double term = (fma(double(Vec<T>::load1(x + y)), double(kLog2e), -m) - log2s) * kLn2;
        if (sums) add_f64(sums + g, out + g, term);
        else atomicAdd(out + g, float(term));
      };
      score(targets[row], seg);
      if (forked) {
        // Several forks may name the same row only if the caller built them so; score each.
        for (int f = 0; f < n_forks; ++f)
          if (fork_rows[f] == row) score(fork_targets[f], fork_segments[f]);
      }
    }
  }
}

}  // namespace
}  // namespace psa

namespace {
psa_status_t run_logp(const void* logits, int32_t logits_dtype, int64_t n_rows, int64_t vocab, int64_t row_stride,
                      const int32_t* targets, const int32_t* segment_ids, const int32_t* fork_rows,
                      const int32_t* fork_targets, const int32_t* fork_segments, int32_t n_forks, int32_t n_segments,
                      float* out, double* sums, int32_t* device_status, void* stream) {
  if (n_rows < 0 || vocab <= 0 || row_stride < vocab || n_forks < 0 || n_segments < 0) return PSA_ERR_INVALID_ARG;
  if (n_segments > 0 && !out) return PSA_ERR_INVALID_ARG;
  if (n_rows > 0 && (!logits || !targets || !segment_ids)) return PSA_ERR_INVALID_ARG;
  if (n_forks > 0 && (!fork_rows || !fork_targets || !fork_segments)) return PSA_ERR_INVALID_ARG;
  if (logits_dtype != PSA_DTYPE_F32 && logits_dtype != PSA_DTYPE_BF16) return PSA_ERR_INVALID_ARG;
  if (n_rows > 0x7fffffffLL) return PSA_ERR_UNSUPPORTED;
  const int64_t esz = logits_dtype == PSA_DTYPE_F32 ? 4 : 2;
  // the stride is not used when there is a single row
  if ((reinterpret_cast<uintptr_t>(logits) & 15) || (n_rows > 1 && ((row_stride * esz) & 15))) return PSA_ERR_ALIGNMENT;
  cudaStream_t st = cudaStream_t(stream);
  if (n_rows == 0) sums = nullptr;   // nothing is added: only out is cleared
  if (sums && n_segments > 0)
    psa::launch_behind(true, psa::dpo_logp_clear_kernel, dim3(unsigned(n_segments + 127) / 128), 128, 0, st, out, sums, n_segments);
  else if (n_segments > 0 && cudaMemsetAsync(out, 0, sizeof(float) * size_t(n_segments), st) != cudaSuccess)
    return PSA_ERR_CUDA;
  if (n_rows == 0) return PSA_OK;
  psa::ProfileScope prof(2, stream);
  auto run = [&](auto kernel, auto* x, int threads) {
    // Behind the kernel that clears the sums, which has waited for whatever wrote the logits: the rows are read meanwhile.
    // us of the whole call: 1515 x 5592 bf16 6.1 -> 5.5, 11957 x 2429 11.9 -> 11.5, 1652 x 15739 10.9 -> 9.6.  (The rows do
    // not let the next kernel start before their end: it would fill the SMs that run dry first, and stay there; 11957 x
    // 2429 16.4.)
    psa::launch_behind(sums && n_segments > 0, kernel, dim3(unsigned(n_rows)), unsigned(threads), 0, st, x, vocab, row_stride,
                       targets, segment_ids, fork_rows, fork_targets, fork_segments, n_forks, n_segments, out, sums, device_status);
  };
  // Threads x loads in flight per thread.  Small CTAs keep many rows in flight per SM and retire unevenly, which suits
  // many rows: 16215 x 128256 bf16, 2/3 live, 400 us with 128 x 4, 408 with 256 x 4, 484 with 512 x 4.  A few long rows
  // are less than two waves of 1480 such CTAs, and a wave lasts as long as a row: 1800 x 128256 bf16 66 -> 60 us with
  // 256 x 4.  (The host knows the number of rows, not how many of them are live: a frozen model's pass with 1200 live of
  // 15154 rows is such a launch too, but takes 128 x 4.)  fp32 rows have half the exponentials per byte and take more loads in flight from 64 KB on: 4096 x 50257
  // 107 -> 85 us with 256 x 8, 8192 x 50257 171 -> 157, 4000 x 16384 36 -> 33, 3312 x 115288 (360 live) 54 -> 37; below,
  // 128 x 4 stays better (6000 x 8192 27 against 29).
  const int64_t row_bytes = vocab * esz;
  if (logits_dtype == PSA_DTYPE_F32) {
    const float* x = static_cast<const float*>(logits);
    if (row_bytes >= 64 * 1024) run(psa::dpo_logp_kernel<float, 8, 256>, x, 256);
    else run(psa::dpo_logp_kernel<float, 4, 128>, x, 128);
  } else {
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(logits);
    if (row_bytes >= 128 * 1024 && n_rows <= 4096) run(psa::dpo_logp_kernel<__nv_bfloat16, 4, 256>, x, 256);
    else run(psa::dpo_logp_kernel<__nv_bfloat16, 4, 128>, x, 128);
  }
  return psa::check_last_cuda_error("dpo_logp launch");
}
}  // namespace

extern "C" psa_status_t dpo_logp(const void* logits, int32_t logits_dtype, int64_t n_rows, int64_t vocab,
                                 int64_t row_stride, const int32_t* targets, const int32_t* segment_ids,
                                 const int32_t* fork_rows, const int32_t* fork_targets,
                                 const int32_t* fork_segments, int32_t n_forks, int32_t n_segments, float* out,
                                 int32_t* device_status, void* stream) {
  return run_logp(logits, logits_dtype, n_rows, vocab, row_stride, targets, segment_ids, fork_rows, fork_targets,
                  fork_segments, n_forks, n_segments, out, nullptr, device_status, stream);
}

extern "C" psa_status_t dpo_logp_f64sum(const void* logits, int32_t logits_dtype, int64_t n_rows, int64_t vocab,
                                        int64_t row_stride, const int32_t* targets, const int32_t* segment_ids,
                                        const int32_t* fork_rows, const int32_t* fork_targets,
                                        const int32_t* fork_segments, int32_t n_forks, int32_t n_segments, float* out,
                                        void* scratch, int32_t* device_status, void* stream) {
  if (!scratch) return PSA_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(scratch) & 7) return PSA_ERR_ALIGNMENT;
  return run_logp(logits, logits_dtype, n_rows, vocab, row_stride, targets, segment_ids, fork_rows, fork_targets,
                  fork_segments, n_forks, n_segments, out, static_cast<double*>(scratch), device_status, stream);
}
