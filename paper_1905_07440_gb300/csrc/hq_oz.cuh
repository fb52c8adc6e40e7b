// FP64 matrix products on the tensor cores (error-free splitting into FP16 digits).
//
// GB300 issues about 1.65 DFMA per clock and SM, but 870 FP16 multiply-adds with FP32
// accumulation through mma.sync.m16n8k16 (measured: 550 TFLOP/s against 1.06).  So the
// contractions of the engine run as sums of exact digit products (the splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59 (2012), with fixed-point digits):
//
//   * An operand value a with |a| < 2^e (e shared by the line that one product sums over, i.e. a
//     row of the left and a column of the right factor) becomes the integer I = trunc(a 2^(P-e)),
//     |I| < 2^P, P = 58, in six signed base-1024 digits, I = sum_i q_i 1024^(5-i),
//     |q_i| <= 512.  Digits are exact in FP16.
//   * Per 16 terms of the sum, digit i of the left times digit j of the right factor, i + j <= 5,
//     are 21 MMAs into six FP32 accumulators S_(i+j).  A product of digits is at most 2^18, so
//     S_0 .. S_3 are integers below 2^24 and exact whatever the data; S_4 and S_5 reach 2^24 only
//     when all digits are extreme and then lose units that weigh 2^-58 of 2^(ea+eb).
//   * S_0 .. S_4 (+ S_5 / 1024) are added up in 64-bit integers, converted once and scaled by
//     the exponents.  The digit pairs left out (i + j > 5) and the last integer digit weigh about
//     2^-56 of the largest |a| |b| of the sum, against 2^-53 per operation of a DFMA chain.  Where a line's terms
//     differ in size and the other factor's make up for it, a DFMA chain keeps the small ones' bits and this does
//     not, unless the terms are scaled (oz_gemm's sk, oz_t_product).
//
// The splits run on the integer pipe (about 27 instructions per value), so a product costs about
// as much as its operands' splits plus 1/16 of the DFMA time.  tcgen05 is not used: operands
// are formed in registers, most products here have 16 columns or rows (the panel width), and
// staging their digits through shared-memory descriptors would cost more than the MMAs.
//
// Non-finite values: a line with a NaN or infinity gets the exponent kOzBad, and every result
// that uses it is NaN or infinite, so that the checks on G and log|det| see it.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include "hq_device.cuh"

namespace hq {

constexpr int kOzDigits = 6;
constexpr int kOzBad = 1 << 19;    // exponent of a line with a non-finite value
constexpr int kOzUnit = 1024;      // exponent bound of |a| <= 1 (below 2^(1024 - 1023))
constexpr int kOzP = 58;           // bits of an operand (59 would let the biased top digit leave its ten bits)

// Biased exponent bound E of a line from the largest high word (sign bit off): |a| < 2^(E - 1023).
// Lines below 2^-895 count as zero.
__device__ __forceinline__ int oz_bound(uint32_t hi) {
  const int e = (int)(hi >> 20) + 1;
  return e >= 2048 ? kOzBad : (e > 128 ? e : 128);
}

__device__ __forceinline__ uint32_t oz_abs_hi(double a) { return (uint32_t)__double2hiint(a) & 0x7fffffffu; }

// trunc(a 2^(P - (E - 1023))) plus the digit bias 512 sum_i 1024^i.
template <int P>
__device__ __forceinline__ unsigned long long oz_fix(double a, int E) {
  constexpr unsigned long long kBias = 512ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) + (1ull << 40) +
                                                 (1ull << 50));
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const int e = (int)((hi >> 20) & 0x7ffu);
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;  // a = +-m 2^(e - 1075)
  m = (m << (P - 53)) >> min((unsigned)(E - 1 - e), 63u);
  return (int)hi < 0 ? kBias - m : kBias + m;
}

// The six digits of two values as packed FP16 pairs (first value in the low half), top digit first.
__device__ __forceinline__ void oz_pack(unsigned long long u, unsigned long long v, uint32_t (&q)[kOzDigits]) {
  const uint32_t u0 = (uint32_t)u, v0 = (uint32_t)v, u1 = (uint32_t)(u >> 30), v1 = (uint32_t)(v >> 30);
  const __half2 off = __halves2half2(__ushort_as_half(0x6600), __ushort_as_half(0x6600));  // 1024 + 512
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    uint32_t a = (__byte_perm(u0 >> (10 * s), v0 >> (10 * s), 0x5410) & 0x03ff03ffu) | 0x64006400u;
    uint32_t b = (__byte_perm(u1 >> (10 * s), v1 >> (10 * s), 0x5410) & 0x03ff03ffu) | 0x64006400u;
    __half2 ha = __hsub2(*reinterpret_cast<__half2*>(&a), off), hb = __hsub2(*reinterpret_cast<__half2*>(&b), off);
    q[5 - s] = *reinterpret_cast<uint32_t*>(&ha);
    q[2 - s] = *reinterpret_cast<uint32_t*>(&hb);
  }
}

template <int P>
__device__ __forceinline__ void oz_split(double a, double b, int Ea, int Eb, uint32_t (&q)[kOzDigits]) {
  oz_pack(oz_fix<P>(a, Ea), oz_fix<P>(b, Eb), q);
}

__device__ __forceinline__ void oz_mma1(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}

// T += the 16-term products of a 16 x 8 tile: a[i][4] digit i of the left fragment, bf(j) digit j
// of the right one.  T counts units of 2^60 / 2^(2P).
template <class BF>
__device__ __forceinline__ void oz_mma(const uint32_t (&a)[4][kOzDigits], BF bf, long long (&T)[4]) {
  float s[6][4];
#pragma unroll
  for (int d = 0; d < 6; ++d)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[d][e] = 0.f;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const uint2 b = bf(j);
#pragma unroll
    for (int i = 0; i + j < 6; ++i) oz_mma1(s[i + j], a[0][i], a[1][i], a[2][i], a[3][i], b);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int i0 = __float2int_rn(s[0][e]), i1 = __float2int_rn(s[1][e]), i2 = __float2int_rn(s[2][e]),
              i3 = __float2int_rn(s[3][e]), i4 = __float2int_rn(fmaf(s[5][e], 1.f / 1024.f, s[4][e]));
    long long t = T[e] + i4;
    t += (long long)i3 * (1 << 10);
    t += (long long)i2 * (1 << 20);
    t += (long long)i1 * (1 << 30);
    T[e] = t + (long long)((unsigned long long)(unsigned)(i0 << 8) << 32);
  }
}

// The same with two accumulators per entry (sums of more than 64 terms, whose S_0 part would
// leave 64 bits): H counts units of 2^80, T units of 2^60.
template <class BF>
__device__ __forceinline__ void oz_mma_wide(const uint32_t (&a)[4][kOzDigits], BF bf, long long (&H)[4],
                                            long long (&T)[4]) {
  float s[6][4];
#pragma unroll
  for (int d = 0; d < 6; ++d)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[d][e] = 0.f;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const uint2 b = bf(j);
#pragma unroll
    for (int i = 0; i + j < 6; ++i) oz_mma1(s[i + j], a[0][i], a[1][i], a[2][i], a[3][i], b);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int i0 = __float2int_rn(s[0][e]), i1 = __float2int_rn(s[1][e]), i2 = __float2int_rn(s[2][e]),
              i3 = __float2int_rn(s[3][e]), i4 = __float2int_rn(fmaf(s[5][e], 1.f / 1024.f, s[4][e]));
    T[e] += (long long)i3 * (1 << 10) + i4;
    H[e] += (long long)i0 * (1 << 20) + ((long long)i1 * (1 << 10) + i2);
  }
}

// v 2^x for a finite v by an integer add to the exponent; zero below the normal range, NaN for a marked line.
__device__ __forceinline__ double oz_scale(double v, int x) {
  const int hi = __double2hiint(v), e0 = (hi >> 20) & 0x7ff, e = e0 + x;
  int nh = hi + (int)((unsigned)x << 20);
  int nl = __double2loint(v);
  if (e0 == 0 || e <= 0) nh = nl = 0;
  if (e >= 2047 && e0 != 0) { nh = (hi & (int)0x80000000) | 0x7ff00000; nl = 0; }
  if (x > (1 << 17)) { nh = 0x7ff80000; nl = 0; }
  return __hiloint2double(nh, nl);
}

// Exponent of a product's result: T 2^(60 - 2P) 2^(ea + eb).
template <int P>
__device__ __forceinline__ int oz_expo(int Ea, int Eb) { return Ea + Eb - 2 * 1023 + 60 - 2 * P; }

__device__ __forceinline__ double oz_wide_value(long long H, long long T) {
  return fma((double)H, 1048576.0, (double)T);
}

__device__ __forceinline__ uint32_t oz_trans8x8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(v));
  return r;
}

// --------------------------------------------------------------- line exponents
// e[r] = bound of line r (0 <= r < lines) over its K entries f(r, k).  along_k: consecutive k are consecutive
// in memory (a warp per line), else consecutive lines are (a thread per line, K shared out).  Ends with a
// barrier.
template <class F>
__device__ inline void oz_line_bounds(bool along_k, int lines, int K, int* e, F f) {
  if (along_k) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 1
    for (int r = warp; r < lines; r += HQ_WARPS) {
      uint32_t m = 0;
#pragma unroll 2
      for (int k = lane; k < K; k += 32) m = max(m, oz_abs_hi(f(r, k)));
      m = __reduce_max_sync(HQ_FULL, m);
      if (lane == 0) e[r] = oz_bound(m);
    }
    __syncthreads();
    return;
  }
  uint32_t* m = reinterpret_cast<uint32_t*>(e);
  for (int r = threadIdx.x; r < lines; r += HQ_THREADS) m[r] = 0;
  __syncthreads();
  const int parts = lines >= HQ_THREADS ? 1 : HQ_THREADS / lines;
  const int r = threadIdx.x % lines, p = threadIdx.x / lines;
  if (p < parts) {
    uint32_t b = 0;
#pragma unroll 4
    for (int k = p; k < K; k += parts) b = max(b, oz_abs_hi(f(r, k)));
    atomicMax(&m[r], b);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < lines; q += HQ_THREADS) e[q] = oz_bound(m[q]);
  __syncthreads();
}

// v 2^x, any v
__device__ __forceinline__ double oz_scale_any(double v, int x) {
  return oz_abs_hi(v) >= 0x7ff00000u ? v : oz_scale(v, x);
}

// -------------------------------------------------------------------- staging
// Exponents of the terms of a sum: term k of the left operand is taken times 2^sk(k), of the right one times 2^-sk(k),
// by moving the exponents of the splits (a bound below 128 would not shift a zero out).
struct OzNoShift {};
template <class SK>
__device__ __forceinline__ int oz_shift_at(const SK& sk, int k, int K) { return k < K ? sk(k) : 0; }
__device__ __forceinline__ int oz_shift_at(const OzNoShift&, int, int) { return 0; }
template <class SK>
__device__ __forceinline__ int oz_shifted(int E, int shift) { return std::is_same<SK, OzNoShift>::value ? E : max(E + shift, 128); }

// Right-operand fragments of nk k-steps x nt tiles of 8 lines: frag[((ks nt + tile) 6 + digit) 32 + lane],
// line = 8 tile + g, k = 16 ks + 2t (+1, +8, +9).  f(line, k): value; eb(line): bound of the values 2^sk(k), k < K.
template <int P, class F, class EB, class SK = OzNoShift>
__device__ __forceinline__ void oz_stage(uint2* frag, int k0, int nk, int nt, F f, EB eb, SK sk = SK(), int K = 0) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  for (int it = threadIdx.x >> 5; it < (nk - k0) * nt; it += HQ_WARPS) {
    const int ks = k0 + it / nt, tile = it % nt, line = 8 * tile + g, k = 16 * ks + 2 * t;
    const int E = eb(line);
    uint32_t x[kOzDigits], y[kOzDigits];
    auto e = [&](int kk) { return oz_shifted<SK>(E, -oz_shift_at(sk, kk, K)); };
    oz_split<P>(f(line, k), f(line, k + 1), e(k), e(k + 1), x);
    oz_split<P>(f(line, k + 8), f(line, k + 9), e(k + 8), e(k + 9), y);
    uint2* o = frag + (size_t)(ks * nt + tile) * kOzDigits * 32 + lane;
#pragma unroll
    for (int d = 0; d < kOzDigits; ++d) o[d * 32] = make_uint2(x[d], y[d]);
  }
}

// ----------------------------------------------------------------- general product
// out(r, c, v0, v1) receives entries (r, c), (r + 1, c) of the M x N product sum_k A(r, k) B(k, c):
// fa(r, k), fb(k, c) values (asked only inside the ranges), ea(r), eb(c) bounds.  Row blocks of RB
// rows of A are split once into shared-memory fragments (all K terms); a warp then takes 16
// columns x 8 NT rows, splitting its columns of B in registers, so no other barrier is needed.
// kTri: A(r, k) = 0 for k < r (the sum starts at the row block's first row).  sk(k), k < K: exponent that moves from B's
// terms to A's (the bounds are those of A(r, k) 2^sk(k) and B(k, c) 2^-sk(k)).
template <int NT, bool kWide, bool kTri, class FA, class EA, class FB, class EB, class OUT, class SK = OzNoShift>
__device__ __forceinline__ void oz_gemm(int M, int N, int K, int RB, uint2* frag, FA fa, EA ea, FB fb, EB eb,
                                        OUT out, SK sk = SK()) {
  constexpr int P = kOzP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int nk = (K + 15) >> 4, ncg = (N + 15) >> 4, nt = RB >> 3;
  for (int r0 = 0; r0 < M; r0 += RB) {
    const int k0 = kTri ? r0 >> 4 : 0;
    __syncthreads();
    oz_stage<P>(frag, k0, nk, nt,
                [&](int line, int k) { return (r0 + line < M && k < K) ? fa(r0 + line, k) : 0.0; },
                [&](int line) { return r0 + line < M ? ea(r0 + line) : 128; }, sk, K);
    __syncthreads();
    const int nh = (min(RB, M - r0) + 8 * NT - 1) / (8 * NT);
    for (int unit = warp; unit < ncg * nh; unit += HQ_WARPS) {
      const int c0 = (unit % ncg) * 16, part = unit / ncg;
      const int ca = c0 + g, cb = c0 + g + 8;
      const int Ea = ca < N ? eb(ca) : 128, Eb = cb < N ? eb(cb) : 128;
      long long T[NT][4], H[NT][4];
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) T[j][e] = H[j][e] = 0;
#pragma unroll 1
      for (int ks = k0; ks < nk; ++ks) {
        const int k = 16 * ks + 2 * t;
        auto get = [&](int kk, int c) { return (kk < K && c < N) ? fb(kk, c) : 0.0; };
        const int s0 = oz_shift_at(sk, k, K), s1 = oz_shift_at(sk, k + 1, K), s8 = oz_shift_at(sk, k + 8, K),
                  s9 = oz_shift_at(sk, k + 9, K);
        uint32_t a[4][kOzDigits];
        oz_split<P>(get(k, ca), get(k + 1, ca), oz_shifted<SK>(Ea, s0), oz_shifted<SK>(Ea, s1), a[0]);
        oz_split<P>(get(k, cb), get(k + 1, cb), oz_shifted<SK>(Eb, s0), oz_shifted<SK>(Eb, s1), a[1]);
        oz_split<P>(get(k + 8, ca), get(k + 9, ca), oz_shifted<SK>(Ea, s8), oz_shifted<SK>(Ea, s9), a[2]);
        oz_split<P>(get(k + 8, cb), get(k + 9, cb), oz_shifted<SK>(Eb, s8), oz_shifted<SK>(Eb, s9), a[3]);
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          const uint2* fr = frag + (size_t)(ks * nt + part * NT + j) * kOzDigits * 32 + lane;
          if (kWide) oz_mma_wide(a, [&](int d) { return fr[d * 32]; }, H[j], T[j]);
          else oz_mma(a, [&](int d) { return fr[d * 32]; }, T[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int r = r0 + part * 8 * NT + 8 * j + 2 * t;
        if (r >= M) continue;
        double v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = kWide ? oz_wide_value(H[j][e], T[j][e]) : (double)T[j][e];
        const int E0 = ea(r), E1 = ea(r + 1);
        if (ca < N) out(r, ca, oz_scale(v[0], oz_expo<P>(E0, Ea)), oz_scale(v[1], oz_expo<P>(E1, Ea)));
        if (cb < N) out(r, cb, oz_scale(v[2], oz_expo<P>(E0, Eb)), oz_scale(v[3], oz_expo<P>(E1, Eb)));
      }
    }
  }
  __syncthreads();
}

// ------------------------------------------------------- updates of up to 16 terms
// Right-operand fragments of the nr x kb coefficient matrix f(r, k) (kb <= 16, zero beyond) with a
// bound per row in er[]; all threads, no barrier.
template <class F>
__device__ __forceinline__ void oz_stage_rows(uint2* frag, int* er, int nr, int kb, F f) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int nt = ((nr + 15) >> 4) * 2;
  for (int tile = threadIdx.x >> 5; tile < nt; tile += HQ_WARPS) {
    const int r = 8 * tile + g, k = 2 * t;
    auto get = [&](int kk) { return (r < nr && kk < kb) ? f(r, kk) : 0.0; };
    const double v0 = get(k), v1 = get(k + 1), v2 = get(k + 8), v3 = get(k + 9);
    uint32_t m = max(max(oz_abs_hi(v0), oz_abs_hi(v1)), max(oz_abs_hi(v2), oz_abs_hi(v3)));
    m = max(m, __shfl_xor_sync(HQ_FULL, m, 1));
    m = max(m, __shfl_xor_sync(HQ_FULL, m, 2));
    const int E = oz_bound(m);
    if (t == 0) er[r] = E;
    uint32_t x[kOzDigits], y[kOzDigits];
    oz_split<kOzP>(v0, v1, E, E, x);
    oz_split<kOzP>(v2, v3, E, E, y);
    uint2* o = frag + (size_t)tile * kOzDigits * 32 + lane;
#pragma unroll
    for (int d = 0; d < kOzDigits; ++d) o[d * 32] = make_uint2(x[d], y[d]);
  }
}

// Left fragment (16 lines x 16 terms) from values in accumulator layout w[tile][4], one bound per
// line: E[0] for line g, E[1] for line g + 8.
__device__ __forceinline__ void oz_left_from_acc(const double (&w)[2][4], uint32_t (&a)[4][kOzDigits], int (&E)[2]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t m = max(max(oz_abs_hi(w[0][2 * h]), oz_abs_hi(w[0][2 * h + 1])),
                     max(oz_abs_hi(w[1][2 * h]), oz_abs_hi(w[1][2 * h + 1])));
    m = max(m, __shfl_xor_sync(HQ_FULL, m, 1));
    m = max(m, __shfl_xor_sync(HQ_FULL, m, 2));
    E[h] = oz_bound(m);
    oz_split<kOzP>(w[0][2 * h], w[0][2 * h + 1], E[h], E[h], a[h]);
    oz_split<kOzP>(w[1][2 * h], w[1][2 * h + 1], E[h], E[h], a[2 + h]);
  }
}

// T as a double by integer instructions (rounded to nearest, halves away from zero).  A conversion and a DFMA hold the
// scheduler's FP64 pipe 64 cycles each; with every second conversion of a rank update done here (about 18 instructions
// of 2 cycles) the two pipes are about equally loaded.  16x16 local sweeps 345 -> 332 ms, 329 with three of four,
// which costs the small class as much.
__device__ __forceinline__ double oz_to_double(long long T) {
  const uint32_t sgn = (uint32_t)((unsigned long long)T >> 32) & 0x80000000u;
  const unsigned long long m = (unsigned long long)(T < 0 ? -T : T);
  uint32_t w1 = (uint32_t)(m >> 32), w0 = (uint32_t)m;
  int e = (1023 + 62) << 20;
  if (w1 == 0) {
    w1 = w0;
    w0 = 0;
    e -= 32 << 20;
  }
  const int c = __clz((int)w1);
  w1 = __funnelshift_l(w0, w1, c);
  w0 <<= c;
  const unsigned long long r = (((unsigned long long)w1 << 32 | w0) >> 11) + ((w0 >> 10) & 1u);
  const uint32_t nh = (uint32_t)(r >> 32) + e - ((uint32_t)c << 20);
  return __hiloint2double((int)(w1 == 0 ? 0u : nh | sgn), (int)r);
}

// 2^x with oz_scale's limits: zero below the normal range, infinity above it and for a marked line.
__device__ __forceinline__ double oz_pow2(int x) {
  return __hiloint2double((int)((unsigned)min(max(x + 1023, 0), 2047) << 20), 0);
}

// For the warp's 16 columns ca = c0 + g, cb = c0 + g + 8 and rows 0 .. nr - 1: io(r, c, v0, v1, p0, p1, old) gets the
// products v0 p0, v1 p1 (p powers of two) of rows r, r + 1 (from the staged coefficients) with the column's left
// fragment, and old = ld(r, c), the entries that they are added to: one DFMA each, where scaling the products first
// would put twelve more instructions on the integer pipe.  NT tiles of 8 rows at a time: with two, one tile's conversions fill the gaps of
// the other's MMA chains.  With kAhead the next tiles' entries are fetched before this one's MMAs: N = 256 reads
// them from L2 or beyond (16x16 block moves 145 -> 139 ms, weights' stacks 66 -> 64 ms); the small class has no registers
// to spare for it and its matrices stay in L1 (8x8 block moves 202 -> 206 ms with it).
template <int NT, bool kAhead, class LD, class IO>
__device__ __forceinline__ void oz_apply_rows(const uint2* frag, const int* er, int nr, const uint32_t (&a)[4][kOzDigits],
                                              const int (&E)[2], int ca, int cb, int cend, LD ld, IO io) {
  const int lane = threadIdx.x & 31, t = lane & 3;
  double2 old[NT][2];
  auto fetch = [&](int tile) {
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int r = 8 * (tile + j) + 2 * t;
      if (r < nr && ca < cend) old[j][0] = ld(r, ca);
      if (r < nr && cb < cend) old[j][1] = ld(r, cb);
    }
  };
  if (kAhead) fetch(0);
#pragma unroll 1
  for (int tile = 0; 8 * tile < nr; tile += NT) {
    double2 now[NT][2];
    if (kAhead) {
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        now[j][0] = old[j][0];
        now[j][1] = old[j][1];
      }
      fetch(tile + NT);
    }
    long long T[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const uint2* fr = frag + (size_t)(tile + j) * kOzDigits * 32 + lane;
#pragma unroll
      for (int e = 0; e < 4; ++e) T[j][e] = 0;
      oz_mma(a, [&](int d) { return fr[d * 32]; }, T[j]);
    }
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int r = 8 * (tile + j) + 2 * t;
      if (r < nr) {
        const int E0 = er[r], E1 = er[r + 1];
        if (ca < cend)
          io(r, ca, (double)T[j][0], oz_to_double(T[j][1]), oz_pow2(oz_expo<kOzP>(E0, E[0])), oz_pow2(oz_expo<kOzP>(E1, E[0])),
             kAhead ? now[j][0] : ld(r, ca));
        if (cb < cend)
          io(r, cb, (double)T[j][2], oz_to_double(T[j][3]), oz_pow2(oz_expo<kOzP>(E0, E[1])), oz_pow2(oz_expo<kOzP>(E1, E[1])),
             kAhead ? now[j][1] : ld(r, cb));
      }
    }
  }
}

// (The callers keep to few instances with runtime strides: a chunk of the chain runs through all of this
// code once per factorisation step, and what is instantiated twice is fetched twice.)
// out(r, c, v0, v1, p0, p1, old): v p = sum_k A(r, k) B(k, c) for r0 <= r < r1, c0 <= c < c1 and kb <= 16 terms; fa, fb
// values, old = ld(r, c).  Reads of fa and fb must not overlap what `out` writes, except that with one_part (a warp
// owns its columns whole) `out` may overwrite the column entries that fb reads.  Ends with a barrier.
template <int NT, class FA, class FB, class LD, class OUT>
__device__ __forceinline__ void oz_rank16(bool one_part, int r0, int r1, int c0, int c1, int kb, uint2* frag, int* er,
                                          FA fa, FB fb, LD ld, OUT out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int nr = r1 - r0;
  oz_stage_rows(frag, er, nr, kb, [&](int r, int k) { return fa(r0 + r, k); });
  __syncthreads();
  // few columns: the row range is shared out too, so that every warp has work
  const int ncg = (c1 - c0 + 15) >> 4;
  const int parts = one_part || ncg >= HQ_WARPS ? 1 : HQ_WARPS / ncg;
  const int rp = (((nr + parts - 1) / parts) + 8 * NT - 1) / (8 * NT) * (8 * NT);
  for (int unit = warp; unit < ncg * parts; unit += HQ_WARPS) {
    const int ca = c0 + (unit % ncg) * 16 + g, cb = ca + 8, rb = (unit / ncg) * rp;
    if (rb >= nr) continue;
    double w[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = 8 * j + 2 * t + (e & 1), c = e < 2 ? ca : cb;
        w[j][e] = (k < kb && c < c1) ? fb(k, c) : 0.0;
      }
    uint32_t a[4][kOzDigits];
    int E[2];
    oz_left_from_acc(w, a, E);
    oz_apply_rows<NT, (NT > 1)>(frag + (size_t)(rb >> 3) * kOzDigits * 32, er + rb, min(rp, nr - rb), a, E, ca, cb, c1,
                                [&](int r, int c) { return ld(r0 + rb + r, c); },
                                [&](int r, int c, double v0, double v1, double p0, double p1, double2 old) {
                                  out(r0 + rb + r, c, v0, v1, p0, p1, old);
                                });
  }
  __syncthreads();
}

// ------------------------------------------------------- separable kinetic propagator
// exp(-+dtau K) = E_y (x) E_x on 16 x 16 tiles held by a warp: a tile is one column of the matrix
// as Z[y][x] (z[w][2h + p]: row g + 8h, column 8w + 2t + p), or with sides up to 8 two or four
// columns side by side (block-diagonal factors).  The factors' digits sit in shared memory: fx
// as right fragments [2][6][32] (contraction over x), fy as left fragments [6][32] (over y).
struct OzKin {
  const uint2* fx;
  const uint4* fy;
  int ex, ey;  // bounds of the factors
};

constexpr int kOzKinBytes = 2 * 6 * 32 * 8 + 6 * 32 * 16;  // one OzKin's fragments

// Fragments of F_x (nx x nx) and F_y (ny x ny), symmetric, row-major; all threads, no barrier.
__device__ inline OzKin oz_kin_build(const double* Fx, const double* Fy, int nx, int ny, char* mem) {
  uint2* fx = reinterpret_cast<uint2*>(mem);
  uint4* fy = reinterpret_cast<uint4*>(mem + 2 * 6 * 32 * 8);
  uint32_t mx = 0, my = 0;
  for (int k = 0; k < nx; ++k) mx = max(mx, oz_abs_hi(Fx[k]));  // circulant: the first row has every value
  for (int k = 0; k < ny; ++k) my = max(my, oz_abs_hi(Fy[k]));
  OzKin K{fx, fy, oz_bound(mx), oz_bound(my)};
  const int px = nx <= 8 ? 8 : 16, py = ny <= 8 ? 8 : 16;
  auto val = [](const double* F, int m, int p, int a, int b) {
    if (a / p != b / p) return 0.0;
    a %= p;
    b %= p;
    return a < m && b < m ? F[a * m + b] : 0.0;
  };
  for (int it = threadIdx.x; it < 64; it += HQ_THREADS) {
    const int lane = it & 31, j = it >> 5, g = lane >> 2, t = lane & 3, c = 8 * j + g;
    uint32_t x[kOzDigits], y[kOzDigits];
    oz_split<kOzP>(val(Fx, nx, px, c, 2 * t), val(Fx, nx, px, c, 2 * t + 1), K.ex, K.ex, x);
    oz_split<kOzP>(val(Fx, nx, px, c, 2 * t + 8), val(Fx, nx, px, c, 2 * t + 9), K.ex, K.ex, y);
    for (int d = 0; d < kOzDigits; ++d) fx[(j * 6 + d) * 32 + lane] = make_uint2(x[d], y[d]);
  }
  for (int lane = threadIdx.x; lane < 32; lane += HQ_THREADS) {
    const int g = lane >> 2, t = lane & 3;
    uint32_t q[4][kOzDigits];
    for (int r = 0; r < 4; ++r) {
      const int a = g + 8 * (r & 1), k = 2 * t + 8 * (r >> 1);
      oz_split<kOzP>(val(Fy, ny, py, a, k), val(Fy, ny, py, a, k + 1), K.ey, K.ey, q[r]);
    }
    for (int d = 0; d < kOzDigits; ++d) fy[d * 32 + lane] = make_uint4(q[0][d], q[1][d], q[2][d], q[3][d]);
  }
  return K;
}

// Digits of a tile: q[2w + h] the 8 x 8 block (row half h, column half w), E[h][w] its bound.  With one
// column per tile (or two) the bounds of the halves it spans are merged.
__device__ __forceinline__ void oz_kin_split(const double (&z)[2][4], bool two_x, bool two_y,
                                             uint32_t (&q)[4][kOzDigits], int (&E)[2][2]) {
  uint32_t m[2][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int w = 0; w < 2; ++w) m[h][w] = max(oz_abs_hi(z[w][2 * h]), oz_abs_hi(z[w][2 * h + 1]));
  if (!two_x) {
    m[0][0] = m[0][1] = max(m[0][0], m[0][1]);
    m[1][0] = m[1][1] = max(m[1][0], m[1][1]);
  }
  if (!two_y) {
    m[0][0] = m[1][0] = max(m[0][0], m[1][0]);
    m[0][1] = m[1][1] = max(m[0][1], m[1][1]);
  }
  if (!two_x && !two_y) {
    const int e = oz_bound(__reduce_max_sync(HQ_FULL, m[0][0]));
    E[0][0] = E[0][1] = E[1][0] = E[1][1] = e;
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int w = 0; w < 2; ++w) E[h][w] = oz_bound(__reduce_max_sync(HQ_FULL, m[h][w]));
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int w = 0; w < 2; ++w)
      oz_split<kOzP>(z[w][2 * h], z[w][2 * h + 1], E[h][w], E[h][w], q[2 * w + h]);
}

// Digits of the tile sums T (units as oz_mma's) straight from the integers: the sums of a block share one
// scale (E, with the factor's bound kex), so all they need is a common shift that brings the largest
// below 2^58.  Without the way through doubles (conversion, exponent, mantissa) this is about half of the
// instructions of a split.  E becomes the bounds of the shifted blocks.
__device__ __forceinline__ void oz_kin_resplit(const long long (&T)[2][4], int kex, bool two_x, bool two_y,
                                               uint32_t (&q)[4][kOzDigits], int (&E)[2][2]) {
  constexpr unsigned long long kBias = 512ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) + (1ull << 40) +
                                                 (1ull << 50));
  auto mag = [](long long v) { return (uint32_t)((v ^ (v >> 63)) >> 32); };
  uint32_t m[2][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int w = 0; w < 2; ++w) m[h][w] = max(mag(T[w][2 * h]), mag(T[w][2 * h + 1]));
  if (!two_x) {
    m[0][0] = m[0][1] = max(m[0][0], m[0][1]);
    m[1][0] = m[1][1] = max(m[1][0], m[1][1]);
  }
  if (!two_y) {
    m[0][0] = m[1][0] = max(m[0][0], m[1][0]);
    m[0][1] = m[1][1] = max(m[0][1], m[1][1]);
  }
  if (!two_x && !two_y) {
    m[0][0] = m[0][1] = m[1][0] = m[1][1] = __reduce_max_sync(HQ_FULL, m[0][0]);
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int w = 0; w < 2; ++w) m[h][w] = __reduce_max_sync(HQ_FULL, m[h][w]);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int up = 58 - (64 - __clz((int)m[h][w]));  // |T| < 2^(64 - clz)
      const unsigned long long u = up >= 0 ? (unsigned long long)T[w][2 * h] << up : (unsigned long long)(T[w][2 * h] >> -up);
      const unsigned long long v =
          up >= 0 ? (unsigned long long)T[w][2 * h + 1] << up : (unsigned long long)(T[w][2 * h + 1] >> -up);
      oz_pack(kBias + u, kBias + v, q[2 * w + h]);
      E[h][w] += kex - 1021 - up;
    }
}

// Z <- F_y Z F_x^T for a tile.
__device__ __forceinline__ void oz_kin_tile(const OzKin& K, double (&z)[2][4], bool two_x, bool two_y) {
  const int lane = threadIdx.x & 31;
  uint32_t q[4][kOzDigits];
  int E[2][2];
  // over x: the tile is the left operand
  oz_kin_split(z, two_x, two_y, q, E);
  long long T[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const uint2* fr = K.fx + w * 6 * 32 + lane;
    oz_mma(q, [&](int d) { return fr[d * 32]; }, T[w]);
  }
  // over y: the tile is the right operand (8 x 8 blocks transposed in registers)
  oz_kin_resplit(T, K.ex, two_x, two_y, q, E);
#pragma unroll
  for (int b = 0; b < 4; ++b)
#pragma unroll
    for (int d = 0; d < kOzDigits; ++d) q[b][d] = oz_trans8x8(q[b][d]);
  uint32_t a[4][kOzDigits];
#pragma unroll
  for (int d = 0; d < kOzDigits; ++d) {
    const uint4 v = K.fy[d * 32 + lane];
    a[0][d] = v.x;
    a[1][d] = v.y;
    a[2][d] = v.z;
    a[3][d] = v.w;
  }
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    long long S[4] = {0, 0, 0, 0};
    oz_mma(a, [&](int d) { return make_uint2(q[2 * w][d], q[2 * w + 1][d]); }, S);
#pragma unroll
    for (int e = 0; e < 4; ++e) z[w][e] = oz_scale((double)S[e], oz_expo<kOzP>(E[e >> 1][w], K.ey));
  }
}

// Visits the tiles of `lines` matrix columns (or rows): load(line, site) gives a pair of values of
// sites site, site + 1 (site = x + nx y, x even), store(line, site, v0, v1) takes them back; step(z,
// visit) transforms the tile in between, with visit(f) calling f(line, site, v0, v1) for every pair.
template <class LOAD, class STEP, class STORE>
__device__ __forceinline__ void oz_kin_lines(int nx, int ny, int lines, LOAD load, STEP step, STORE store) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const bool two_x = nx <= 8, two_y = ny <= 8;
  const int per = (two_x ? 2 : 1) * (two_y ? 2 : 1), tiles = (lines + per - 1) / per;
  for (int tile = warp; tile < tiles; tile += HQ_WARPS) {
    double z[2][4];
    auto visit = [&](auto f) {
#pragma unroll
      for (int w = 0; w < 2; ++w)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int x = two_x ? 2 * t : 8 * w + 2 * t, y = two_y ? g : 8 * h + g;
          const int line = tile * per + (two_y ? h : 0) * (two_x ? 2 : 1) + (two_x ? w : 0);
          const bool on = x < nx && y < ny && line < lines;
          f(on, line, x + nx * y, z[w][2 * h], z[w][2 * h + 1]);
        }
    };
    visit([&](bool on, int line, int site, double& v0, double& v1) {
      v0 = v1 = 0.0;
      if (on) load(line, site, v0, v1);
    });
    step(z, two_x, two_y, visit);
    visit([&](bool on, int line, int site, double& v0, double& v1) {
      if (on) store(line, site, v0, v1);
    });
  }
}

}  // namespace hq
