// Householder panel of up to 16 columns in registers, and the triangular factor of its block reflector.
//
// On GB300 a dependent FP64 instruction takes about 60 cycles, and a warp's FP64 instruction holds its
// scheduler's FP64 pipe for as long whatever the number of active lanes.  A panel is therefore bound
// by the number of FP64 instructions per scheduler and step:
//
//   * Four warps, one per scheduler, hold the panel: column c belongs to warp c % 4 whole, its rows
//     spread over the lanes (RPL = 1, 2, 4, 8 rows per lane for m <= 32, 64, 128, 256).
//   * Per step the pivot column goes to all warps through shared memory (one barrier).  Every warp
//     reduces its own columns' products with it and the norm together, as a reduce-scatter (up to five
//     values over 32 lanes in eight adds, fewer as columns finish), so no partial sums cross warps.
//   * 1 / norm and 2 / v^T v come from single-precision seeds with one third-order step each; factors
//     of two are exponent adds.
//   * Squares and products of columns have to stay normal numbers.  They do for largest entries of 2^-200 .. 2^200 and
//     residuals with squared norms of 2^-512 .. 2^512 (sampling at beta = 16: 2^-100 .. 2^100); the first column
//     outside, a zero or a non-finite one included, and those behind it go through a second form of the loop, in which a
//     column is passed on scaled by its largest entry: norms of 1e-308 to 1e308.  (Scaling in every step costs block
//     moves 2 % at 8x8 and 3 % at 16x16, a second pass over the sums inside the step 3 to 4 %.)
//   * The loop over the columns is rolled; a warp's columns rotate through the registers so that its
//     next one is x[.][0] and the finished ones are at the end, where the loops skip them.
//
// 33 FP64 instructions per step at m = 64.  Measured for 64 x 16 (256 x 16), cycles: column by column with
// two warp reductions per step 82 (145) thousand; rows spread over the warps 67 (146); 64-bit integers with
// 128-bit dot products 62 (130).  Whole QR of n = 64 (256), thousand cycles: rows spread over the warps 375 (3760),
// this form 329 (2890).
#pragma once
#include "hq_device.cuh"
#include "hq_oz.cuh"

namespace hq {

__device__ __forceinline__ void bar_warps(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

__device__ __forceinline__ double float_bits_to_double(float f) {  // normal positive f
  const uint32_t u = __float_as_uint(f);
  return __hiloint2double((int)((((u >> 23) + (1023 - 127)) << 20) | ((u & 0x7fffffu) >> 3)), (int)(u << 29));
}

constexpr int kPanelWarps = 4;  // one per scheduler

// shared scratch of a panel (inside the fragment scratch)
struct PanelShared {
  double col[2][256];
  double a[kPanelWarps][4];
  int e[2];             // scales of the columns: col 2^e is the column
  int out[kPanelWarps];  // a column of the warp is outside the range
};

// Exponents of a column with a non-finite value and of a zero (or subnormal) one, as its largest entry gives them.
constexpr int kPanelBad = 1024, kPanelZero = -1023;

// v 2^k for results below 2^1024: zero below the normal range, infinities and NaN as they are
__device__ __forceinline__ double shift_exponent(double v, int k) {
  const int hi = __double2hiint(v), f = (hi >> 20) & 0x7ff;
  const bool zero = f == 0 || f + k <= 0;
  return f == 0x7ff ? v
                    : __hiloint2double(zero ? hi & (int)0x80000000 : hi + (int)((unsigned)k << 20), zero ? 0 : __double2loint(v));
}

// Exponent of the largest of a warp's values c(r), rows r > 0 and, with r = 0, lanes from `first` on.
template <int RPL, class F>
__device__ __forceinline__ int column_exponent(int first, F c) {
  uint32_t top = 0;
#pragma unroll
  for (int r = 0; r < RPL; ++r)
    if (r > 0 || (int)(threadIdx.x & 31) >= first) top = max(top, oz_abs_hi(c(r)));
  return (int)(__reduce_max_sync(HQ_FULL, top) >> 20) - 1023;
}

// Columns j0 + c0 .. j0 + kb - 1 (kb <= 16) of a panel with rows j0 .. n - 1 of Q.  Writes R (rows j0 .. j0 + c of column
// j0 + c) to Q, the reflector vectors (norms of 1 to 4; H = I - tau v v^T) to the same columns of V with zeros
// above, their bounds to ev[j0 ..], and tau.  Without kScaled it stops before the first column outside the range, with
// all columns behind it updated in Q, and *done counts the columns finished.  From a column with a non-finite
// value on, R, V and tau are NaN (the bound kOzBad).  Ends with a barrier.
template <int LM, int RPL, bool kScaled>
__device__ __noinline__ void panel_columns(double* Q, double* V, int ld, int n, int j0, int c0, int kb, PanelShared* ps,
                                           double* tau, int* ev, int* done_out) {
  constexpr int kThreads = 32 * kPanelWarps;
  const int m = n - j0, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp < kPanelWarps) {
    double x[RPL][4];
#pragma unroll
    for (int r = 0; r < RPL; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = 4 * (i + (c0 >> 2)) + warp, row = lane + 32 * r;
        x[r][i] = (row < m && c < kb) ? Q[(size_t)(j0 + c) * ld + j0 + row] : 0.0;
      }
    // column j (`next`: the warp's second one in its registers) to the other warps
    auto publish = [&](int j, bool next) {
      auto c = [&](int r) { return next ? x[r][1] : x[r][0]; };
      if (kScaled) {
        const int e = column_exponent<RPL>(j, c);
#pragma unroll
        for (int r = 0; r < RPL; ++r) ps->col[j & 1][lane + 32 * r] = shift_exponent(c(r), -e);
        if (lane == 0) ps->e[j & 1] = e;
      } else {
#pragma unroll
        for (int r = 0; r < RPL; ++r) ps->col[j & 1][lane + 32 * r] = c(r);
      }
    };
    if (!kScaled) {
      bool out = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = column_exponent<RPL>(0, [&](int r) { return x[r][i]; });
        out = out || (4 * i + warp < kb && (e < -200 || e > 200));
      }
      if (lane == 0) ps->out[warp] = out;
    }
    if (warp == (c0 & 3)) publish(c0, false);
    bar_warps(kThreads);
    int j = c0;
    if (!kScaled && (ps->out[0] | ps->out[1] | ps->out[2] | ps->out[3])) j = kb;  // (leaves *done at 0)
    int finished = j == kb ? 0 : kb;
#pragma unroll 1
    for (; j < kb; ++j) {
      // x[.][i] is column 4 (i + done) + warp; the warp's columns after j are entries first .. left - 1
      const int jw = j & 3, done = j >> 2, left = 4 - done, first = warp <= jw ? 1 : 0;
      double xj[RPL], p[5];
#pragma unroll
      for (int r = 0; r < RPL; ++r) xj[r] = ps->col[j & 1][lane + 32 * r];
      const double al0 = __shfl_sync(HQ_FULL, xj[0], j);
      if (lane < j) xj[0] = 0.0;  // rows above j hold entries of R
      const int ej = kScaled ? ps->e[j & 1] : 0;
      const bool zero = kScaled && ej == kPanelZero, bad = kScaled && ej == kPanelBad;
      if (lane == j) {
#pragma unroll
        for (int i = 0; i < 4; ++i) ps->a[warp][i] = x[0][i];
      }
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        p[i] = 0.0;
        if (i == 4 || (i < left && i >= first)) {
          p[i] = xj[0] * (i == 4 ? xj[0] : x[0][i]);
#pragma unroll
          for (int r = 1; r < RPL; ++r) p[i] = fma(xj[r], i == 4 ? xj[r] : x[r][i], p[i]);
        }
      }
      // reduce-scatter: value i (4: the norm) ends in lanes with bit 4 = i & 1, bit 3 = (i >> 1) & 1,
      // bit 2 = i >> 2
      {
        const bool u4 = lane & 16, u3 = lane & 8, u2 = lane & 4;
        double q0 = 0.0, q1 = 0.0;
        if (left > 0) q0 = (u4 ? p[1] : p[0]) + __shfl_xor_sync(HQ_FULL, u4 ? p[0] : p[1], 16);
        if (left > 2) q1 = (u4 ? p[3] : p[2]) + __shfl_xor_sync(HQ_FULL, u4 ? p[2] : p[3], 16);
        double q2 = p[4] + __shfl_xor_sync(HQ_FULL, p[4], 16);
        q0 = (u3 ? q1 : q0) + __shfl_xor_sync(HQ_FULL, u3 ? q0 : q1, 8);
        q2 += __shfl_xor_sync(HQ_FULL, q2, 8);
        q0 = (u2 ? q2 : q0) + __shfl_xor_sync(HQ_FULL, u2 ? q0 : q2, 4);
        q0 += __shfl_xor_sync(HQ_FULL, q0, 2);
        p[0] = q0 + __shfl_xor_sync(HQ_FULL, q0, 1);
      }
      const double d = p[0];
      const double Sj = __shfl_sync(HQ_FULL, d, 4);
      __syncwarp();  // lane j's entries (shuffles order no memory)
      const double a = ps->a[warp][((lane >> 4) & 1) | ((lane >> 2) & 2)];
      const int hs = __double2hiint(Sj), es = (hs >> 20) - 1023, h = es >> 1;
      if (!kScaled && (unsigned)(es + 512) >= 1024u) {  // the same in every warp
        finished = j;
        break;
      }
      // s = S / 4^h in [1, 4); the scalars are in units of 2^h of the column as it was passed on
      const double s = zero ? 1.0 : __hiloint2double((hs & 0xfffff) | ((1023 + (es & 1)) << 20), __double2loint(Sj));
      const float sf = __uint_as_float((uint32_t)__double2hiint(s) * 8u - ((1023u - 127u) << 23) +
                                       ((uint32_t)__double2loint(s) >> 29));
      const float yf = rsqrtf(sf);
      const double q = s * float_bits_to_double(yf);
      const double al = shift_exponent(al0, -h);
      const bool neg = __double2hiint(al) < 0;
      const double aa = fabs(al);
      // |al| < 2 as a float, from its bits (0 when it does not matter for the seed)
      const int ah = __double2hiint(aa);
      const float af =
          ah > (900 << 20) ? __uint_as_float(((uint32_t)(ah - (896 << 20)) << 3) | ((uint32_t)__double2loint(aa) >> 29)) : 0.f;
      const double g0 = float_bits_to_double(__fdividef(1.f, fmaf(af, sf * yf, sf)));
      const double e1 = fma(-q, float_bits_to_double(yf), 1.0);
      const double nrm = fma(q * e1, fma(0.375, e1, 0.5), q);  // sqrt(s), third order
      const double td = fma(aa, nrm, s);
      const double wc = fma(neg ? -nrm : nrm, a, shift_exponent(d, -h));  // v^T x_c
      const double e2 = fma(-td, g0, 1.0);
      const double gam = fma(g0, fma(e2, e2, e2), g0);  // 2 / v^T v
      const double nan = __hiloint2double(0x7ff80000, 0);
      // (gam is 1/16 to 1, the norm 1 to 2: normal numbers with these h)
      auto units = [&](double v, int k) { return __hiloint2double(__double2hiint(v) + k * (1 << 20), __double2loint(v)); };
      const double phi = bad ? nan : zero ? 0.0 : units(gam, -h) * wc;
      const double beta = zero ? 0.0 : units(neg ? nrm : -nrm, h);
      if (lane == j) xj[0] = al0 - beta;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < left && i >= first) {
          const double f = -__shfl_sync(HQ_FULL, phi, ((i & 1) << 4) | ((i & 2) << 2));
#pragma unroll
          for (int r = 0; r < RPL; ++r) x[r][i] = fma(f, xj[r], x[r][i]);
        }
      // the next column goes out before this one's records
      if (j + 1 < kb && warp == ((j + 1) & 3)) publish(j + 1, jw == 3);  // (warp 0 takes its next one)
      if (warp == jw) {
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          const int row = lane + 32 * r;
          if (row < m) V[(size_t)(j0 + j) * ld + j0 + row] = zero ? 0.0 : oz_scale(xj[r], bad ? kOzBad : -h);
        }
        // x[0][0] holds the column's entries of R above row j, and entry j before the reflection
        if (lane <= j && lane < m)
          Q[(size_t)(j0 + j) * ld + j0 + lane] =
              lane < j || zero ? x[0][0] : kScaled ? oz_scale(beta, bad ? kOzBad : ej) : beta;
        if (lane == 0) {
          tau[j] = bad ? nan : zero ? 0.0 : gam;
          ev[j0 + j] = bad ? kOzBad : zero ? kOzUnit : oz_bound(oz_abs_hi(aa + nrm));
        }
      }
      if (jw == 3) {
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
#pragma unroll
          for (int i = 0; i < 3; ++i) x[r][i] = x[r][i + 1];
        }
      }
      bar_warps(kThreads);
    }
    if (!kScaled) {
      if (finished < kb) {  // what is left of the columns behind, for the second form
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
          const int c = 4 * ((finished >> 2) + i) + warp;
#pragma unroll
          for (int r = 0; r < RPL; ++r) {
            const int row = lane + 32 * r;
            if (c >= finished && c < kb && row < m) Q[(size_t)(j0 + c) * ld + j0 + row] = x[r][0];
#pragma unroll
            for (int k = 0; k < 3; ++k) x[r][k] = x[r][k + 1];
          }
        }
      }
      if (tid == 0) *done_out = finished;
    }
  }
  __syncthreads();
}

// A panel's columns (as panel_columns).  done: an int of shared memory that the panel's fragments do not cover.
template <int LM, int RPL>
__device__ __forceinline__ void panel_house(double* Q, double* V, int ld, int n, int j0, int kb, PanelShared* ps, double* tau,
                                            int* ev, int* done) {
  panel_columns<LM, RPL, false>(Q, V, ld, n, j0, 0, kb, ps, tau, ev, done);
  const int c0 = *done;
  if (c0 < kb) panel_columns<LM, RPL, true>(Q, V, ld, n, j0, c0, kb, ps, tau, ev, nullptr);
}

// Right-operand fragments of V's panel with the rows as terms (fragment order of oz_stage, 2 tiles of 8
// vectors): all threads, no barrier.
__device__ __forceinline__ void stage_panel(uint2* vk, const double* V, int ld, int n, int j0, int kb, const int* ev) {
  const int nr = n - j0;
  oz_stage<kOzP>(vk, 0, (nr + 15) >> 4, 2,
                 [&](int line, int k) { return (line < kb && k < nr) ? V[(size_t)(j0 + line) * ld + j0 + k] : 0.0; },
                 [&](int line) { return line < kb ? ev[j0 + line] : 128; });
}

// T of H_j0 ... = I - V T V^T (upper triangular, compact WY: Schreiber and Van Loan, SIAM J. Sci. Stat.
// Comput. 10 (1989)).  V^T V comes from the staged fragments (a right fragment holds the same values
// as the left fragment of its transpose), the k-steps shared out over the warps and their integer sums
// added in shared memory.  S, T: [16][16]; ends with a barrier.
__device__ inline void panel_t(const uint2* vk, int nk, int kb, const double* tau, const int* ev, unsigned long long* sum,
                               double* S, double* T) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  for (int idx = tid; idx < 256; idx += HQ_THREADS) {
    sum[idx] = 0;
    T[idx] = 0.0;
  }
  __syncthreads();
  if (warp < nk) {
    long long acc[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
    for (int ks = warp; ks < nk; ks += HQ_WARPS) {
      const uint2* f0 = vk + (size_t)(2 * ks) * kOzDigits * 32 + lane;
      const uint2* f1 = f0 + kOzDigits * 32;
      uint32_t a[4][kOzDigits];
#pragma unroll
      for (int d = 0; d < kOzDigits; ++d) {
        const uint2 u = f0[d * 32], w = f1[d * 32];
        a[0][d] = u.x;
        a[1][d] = w.x;
        a[2][d] = u.y;
        a[3][d] = w.y;
      }
      oz_mma(a, [&](int d) { return f0[d * 32]; }, acc[0]);
      oz_mma(a, [&](int d) { return f1[d * 32]; }, acc[1]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        atomicAdd(&sum[(g + 8 * (e >> 1)) * 16 + 8 * j + 2 * t + (e & 1)], (unsigned long long)acc[j][e]);
  }
  __syncthreads();
  {
    const int a = tid >> 4, b = tid & 15;  // HQ_THREADS = 256 entries
    S[tid] = (a < b && b < kb) ? oz_scale((double)(long long)sum[tid], oz_expo<kOzP>(ev[a], ev[b])) : 0.0;
  }
  __syncthreads();
  // T by doubling: 4 x 4 diagonal blocks (a row per lane), then off-diagonal blocks -T11 S12 T22 of 4 and
  // of 8; S12 T22 is kept in S's place.  34 dependent FP64 instructions instead of 136 of the recurrence.
  if (warp == 0) {
    if (lane < 16) {
      const int i = lane & 3, o = lane & 12;
      double x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double tj = o + j < kb ? tau[o + j] : 0.0;
        double a = 0.0;
#pragma unroll
        for (int k = 0; k < j; ++k) a = fma(x[k], S[(o + k) * 16 + o + j], a);
        x[j] = j < i ? 0.0 : (j == i ? tj : -tj * a);
        T[(o + i) * 16 + o + j] = x[j];
      }
    }
    __syncwarp();
    const int o = lane < 16 ? 0 : 8, r = (lane >> 2) & 3, c = lane & 3;
    double a = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) a = fma(S[(o + r) * 16 + o + 4 + k], T[(o + 4 + k) * 16 + o + 4 + c], a);
    __syncwarp();
    S[(o + r) * 16 + o + 4 + c] = a;
    __syncwarp();
    a = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) a = fma(T[(o + r) * 16 + o + k], S[(o + k) * 16 + o + 4 + c], a);
    T[(o + r) * 16 + o + 4 + c] = -a;
  }
  __syncthreads();
  if (tid < 64) {
    const int r = tid >> 3, c = tid & 7;
    double a = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) a = fma(S[r * 16 + 8 + k], T[(8 + k) * 16 + 8 + c], a);
    bar_warps(64);
    S[r * 16 + 8 + c] = a;
    bar_warps(64);
    a = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) a = fma(T[r * 16 + k], S[k * 16 + 8 + c], a);
    T[r * 16 + 8 + c] = -a;
  }
  __syncthreads();
}

}  // namespace hq
