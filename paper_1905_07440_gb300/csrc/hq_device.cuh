// Device building blocks of the Holstein DQMC engine (one CTA per Markov chain): sums, bounded
// waits, random numbers, section counters.  Matrices are column-major n x n (element (r, c) at c*ld + r) in
// global memory (L1/L2 cached).  The FP64 pipe is narrow on GB300 (about 1/74 of the FP32 rate):
// contractions run on the tensor cores (hq_oz.cuh), panels in registers (hq_panel.cuh, hq_lu.cuh).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#define HQ_THREADS 256
#define HQ_WARPS (HQ_THREADS / 32)
#define HQ_FULL 0xffffffffu

namespace hq {

// Optional per-section cycle counters (compile with -DHQ_SECTION_TIMING): thread 0 of each
// CTA adds the clock64() span of a code section to a device array that
// hq_get_section_cycles() returns.  Off by default; no effect on results.
enum {
  SEC_DL = 0, SEC_KIN, SEC_PREPIVOT, SEC_QR, SEC_FORMQ, SEC_TUPD, SEC_LOGDET, SEC_MOVE, SEC_WAIT,
  SEC_PROP_PREP, SEC_PROP_SEQ, SEC_WRAP, SEC_RESTAB_PROD, SEC_RESTAB_QR, SEC_RESTAB_GREEN, SEC_MEASURE,
  SEC_FLUSH, SEC_COUNT
};
#ifdef HQ_SECTION_TIMING
static __device__ unsigned long long g_section_cycles[SEC_COUNT];  // per translation unit
#define HQ_TIC(name) const long long hq_tic_##name = clock64()
#define HQ_TOC(name, slot)                                                              \
  do {                                                                                \
    if (threadIdx.x == 0) atomicAdd(&g_section_cycles[slot], (unsigned long long)(clock64() - hq_tic_##name)); \
  } while (0)
#else
#define HQ_TIC(name) (void)0
#define HQ_TOC(name, slot) (void)0
#endif

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(HQ_FULL, v, o);
  return v;
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(HQ_FULL, v, o));
  return v;
}

// Sum over the CTA in a fixed order (deterministic); every thread gets the result.
// red: HQ_WARPS doubles of shared memory.
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < HQ_WARPS; ++w) s += red[w];
  return s;
}

__device__ __forceinline__ double block_max(double v, double* red) {
  v = warp_max(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = red[0];
#pragma unroll
  for (int w = 1; w < HQ_WARPS; ++w) s = fmax(s, red[w]);
  return s;
}

// ---------------------------------------------------------------- bounded waits
__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Spin (with growing sleeps) until *v >= target.  Gives up -- returns false -- when *abort_flag
// becomes non-zero or after limit_ns of global time, so a wait never hangs the GPU.
__device__ inline bool bounded_wait_geq(volatile int* v, int target, volatile int* abort_flag,
                                        unsigned long long limit_ns) {
  if (*v >= target) return true;
  const unsigned long long t0 = global_timer_ns();
  unsigned ns = 32;
  while (*v < target) {
    if (*abort_flag != 0 || global_timer_ns() - t0 > limit_ns) return false;
    __nanosleep(ns);
    if (ns < 2048) ns *= 2;
  }
  return true;
}

// ---------------------------------------------------------------- bfloat16
__device__ __forceinline__ float bf16_to_float(uint16_t h) { return __uint_as_float((uint32_t)h << 16); }

// round to nearest even (finite inputs)
__device__ __forceinline__ uint16_t float_to_bf16(float f) {
  const uint32_t u = __float_as_uint(f);
  return (uint16_t)((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
}

// ---------------------------------------------------------------- Philox4x32-10
// Salmon, Moraes, Dror, Shaw (SC'11): ten rounds of two 32x32->64 multiplies with the
// round constants, key bumped by the Weyl constants between rounds.
__device__ __forceinline__ void philox4x32_10(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3,
                                              uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
}

// 53-bit uniform in [0,1) from the 27 high bits of a and the 26 high bits of b.
__device__ __forceinline__ double uniform53(uint32_t a, uint32_t b) {
  return ((double)(a >> 5) * 67108864.0 + (double)(b >> 6)) * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ void proposal_uniforms(uint32_t key0, uint32_t key1, uint32_t event,
                                                  uint32_t sweep, uint32_t chain, uint32_t tag,
                                                  double& u1, double& u2) {
  uint32_t c0 = event, c1 = sweep, c2 = chain, c3 = tag;
  philox4x32_10(c0, c1, c2, c3, key0, key1);
  u1 = uniform53(c0, c1);
  u2 = uniform53(c2, c3);
}

// ----------------------------------------------------------------- small helpers

__device__ __forceinline__ void set_identity(double* A, int ld, int n) {
  for (int idx = threadIdx.x; idx < n * n; idx += HQ_THREADS) {
    const int r = idx % n, c = idx / n;
    A[(size_t)c * ld + r] = (r == c) ? 1.0 : 0.0;
  }
}

// B <- A (n x n, contiguous, n^2 a multiple of 16)
__device__ __forceinline__ void copy_mat(double* B, const double* A, int n) {
  const double2* a = reinterpret_cast<const double2*>(A);
  double2* b = reinterpret_cast<double2*>(B);
#pragma unroll 4
  for (int idx = threadIdx.x; idx < n * n / 2; idx += HQ_THREADS) b[idx] = a[idx];
}

// Sum over groups of G lanes (the warp's 32 lanes all take part).
template <int G>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(HQ_FULL, v, o);
  return v;
}

}  // namespace hq
