// Householder panel of up to 16 columns in 64-bit fixed point, and the triangular factor of its block
// reflector.
//
// On GB300 a dependent FP64 instruction takes about 60 cycles, and a warp's FP64 instruction holds its
// scheduler's FP64 pipe for as long whatever the number of active lanes, while integer multiply-adds
// and adds issue every other cycle.  A Householder step in FP64 needs some 55 instructions per scheduler
// (dot products, their reductions, scalars, updates): 3900 cycles in the best arrangement found, and it
// leaves no FP64 time to a second CTA.  Here the panel lives in registers as integers, one scale per
// column:
//
//   * Householder reflections keep column norms, so a column scaled once (largest entry below 2^B,
//     norm below 2^60) never overflows; an entry's unit is 2^-B of the column's largest entry, no
//     coarser than the FP64 rounding of a column-wise backward stable QR.
//   * The dot products of a step with the columns to come are exact 128-bit sums, reduce-scattered by
//     integer shuffles (neighbouring columns first, so that the finished ones drop out).
//   * Only the step's scalars (norm, beta, 2 / v^T v, the coefficients) are FP64, in one warp, with
//     single-precision seeds and one third-order step each.  The vector is shifted so that its norm has
//     all bits (v = 2^k x - beta e_j, norm of x in [2^59, 2^60)), so the reflector is orthogonal to 2^-53
//     however small the rest of the column is.
//   * Updates are four integer multiply-adds per entry.
//
// Thread layout: one matrix row per thread (m <= 256 rows), or G = 2, 4 threads per row for m <= 128,
// 64, each with CPT = 16 / G columns (column c in thread c % G of its row).  The loop over the columns is
// rolled; a thread's columns rotate through its registers so that the current one is always x[0].
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

constexpr int kPanelWarps = 4;  // warps of a panel held in FP64 (hq_lu.cuh): one per scheduler

// shared scratch of a panel (inside the fragment scratch)
struct PanelShared {
  __int128 part[HQ_WARPS][16];
  double arow[16];
  long long m[16];
  long long b;
  uint32_t cmax[16];
  int shift;
};

// a b / 2^59 for |a|, |b| < 2^61, to the nearest unit (within 2^-28 of a unit)
__device__ __forceinline__ long long mul_shift59(int a1, int a0, long long b) {
  const int b1 = (int)(b >> 30), b0 = (int)(b & 0x3fffffff);
  const long long hi = (long long)a1 * b1;
  const long long mid = (long long)a1 * b0 + (long long)a0 * b1 + (((long long)a0 * b0) >> 30);
  return hi * 2 + ((mid + (1ll << 28)) >> 29);
}

// v 2^k for a v that is zero or stays in the normal range
__device__ __forceinline__ double shift_exponent(double v, int k) {
  const int hi = __double2hiint(v);
  return __hiloint2double((hi & 0x7fffffff) == 0 ? hi : hi + (int)((unsigned)k << 20), __double2loint(v));
}

// Columns j0 .. j0 + kb - 1 (kb <= 16), rows j0 .. n - 1 of Q.  Writes R (rows j0 .. j0 + c of column
// j0 + c) to Q, the reflector vectors (norms of 1 to 4; H = I - tau v v^T) to the same columns of V with zeros
// above, their bounds to ev[j0 ..], and tau.  Ends with a barrier.
template <int LM, int CPT>
__device__ __noinline__ void panel_fixed(double* Q, double* V, int ld, int n, int j0, int kb, PanelShared* ps,
                                         double* tau, int* ev) {
  constexpr int G = 16 / CPT, LG = G == 4 ? 2 : G == 2 ? 1 : 0, kRowsPerWarp = 32 / G;
  const int m = n - j0, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nw = (m + kRowsPerWarp - 1) / kRowsPerWarp, nthr = nw * 32;
  if (warp < nw) {
    const int row = tid >> LG, cq = tid & (G - 1);
    const bool in = row < m;
    // norm <= sqrt(m) 2^B <= 2^60
    const int B = m <= 64 ? 57 : 56;
    if (tid < 16) ps->cmax[tid] = 0;
    bar_warps(nthr);
    long long x[CPT];
    {
      double v[CPT];
#pragma unroll
      for (int i = 0; i < CPT; ++i) {
        const int c = i * G + cq;
        v[i] = (in && c < kb) ? Q[(size_t)(j0 + c) * ld + j0 + row] : 0.0;
        uint32_t h = oz_abs_hi(v[i]);
#pragma unroll
        for (int o = 16; o >= G; o >>= 1) h = max(h, __shfl_xor_sync(HQ_FULL, h, o));
        if (lane < G) atomicMax(&ps->cmax[c], h);
      }
      bar_warps(nthr);
#pragma unroll
      for (int i = 0; i < CPT; ++i) {
        const uint32_t hi = (uint32_t)__double2hiint(v[i]);
        const int r = (int)min((unsigned)(oz_bound(ps->cmax[i * G + cq]) - 1 - (int)((hi >> 20) & 0x7ffu)), 63u);
        unsigned long long u = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | (uint32_t)__double2loint(v[i]);
        u = (((u << (B - 52)) >> r) + 1) >> 1;  // to the nearest unit
        x[i] = (int)hi < 0 ? -(long long)u : (long long)u;
      }
    }
    // a non-finite entry anywhere in the panel makes all of its results NaN
    uint32_t top = 0;
#pragma unroll
    for (int c = 0; c < 16; ++c) top = max(top, ps->cmax[c]);
    const bool bad = oz_bound(top) == kOzBad;
    const double nanv = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll 1
    for (int j = 0; j < kb; ++j) {
      // x[i] holds column ((i + jb) % CPT) G + cq; entries i < CPT - jb are the columns not yet done.  In a
      // finished column c, rows up to c hold R and the others v.
      const int jo = j & (G - 1), jb = j >> LG, left = CPT - jb;
      long long xj = G == 1 ? x[0] : __shfl_sync(HQ_FULL, x[0], (lane & ~(G - 1)) | jo);
      if (row < j) xj = 0;
      // exact products with the thread's columns, summed over the warp's rows: a column per lane
      __int128 p[CPT];
      {
        const int a1 = (int)(xj >> 30), a0 = (int)(xj & 0x3fffffff);
#pragma unroll
        for (int i = 0; i < CPT; ++i) {
          p[i] = 0;
          if (i < left) {
            const int b1 = (int)(x[i] >> 30), b0 = (int)(x[i] & 0x3fffffff);
            const long long hi = (long long)a1 * b1, mid = (long long)a1 * b0 + (long long)a0 * b1;
            const long long lo = (long long)a0 * b0;  // in [0, 2^60)
            p[i] = ((__int128)hi << 60) + ((__int128)mid << 30) + lo;
          }
        }
      }
      auto add_from = [&](__int128 mine, __int128 theirs, int o) {
        unsigned long long lo = (unsigned long long)theirs;
        long long hi = (long long)(theirs >> 64);
        lo = __shfl_xor_sync(HQ_FULL, lo, o);
        hi = __shfl_xor_sync(HQ_FULL, hi, o);
        return mine + (__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo);
      };
      int o = 16, idx = 0, cnt = left;
#pragma unroll
      for (int w = CPT / 2; w > 0; w >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < w; ++k)
          if (2 * k < cnt) p[k] = add_from(up ? p[2 * k + 1] : p[2 * k], up ? p[2 * k] : p[2 * k + 1], o);
        if (up) idx += CPT / (2 * w);
        cnt = (cnt + 1) >> 1;
        o >>= 1;
      }
      p[0] = add_from(p[0], p[0], o);
      if (!(lane & o)) ps->part[warp][((idx + jb) & (CPT - 1)) * G + cq] = idx < left ? p[0] : (__int128)0;
      if (row == j) {
#pragma unroll
        for (int i = 0; i < CPT; ++i)
          if (i < left) ps->arow[(i + jb) * G + cq] = (double)x[i];
      }
      bar_warps(nthr);
      // warp 0: the step's scalars.  Every FP64 instruction holds the pipe for 64 cycles, so their number
      // counts, not the depth of the chain: 13 up to the coefficients; records come after the barrier.
      double nrm = 0.0, gam = 0.0, aa = 0.0;
      int h = 0;
      bool zero = false, neg = false;
      if (warp == 0) {
        const int c = lane & 15;
        __int128 t = 0;
        for (int w = lane >> 4; w < nw; w += 2) t += ps->part[w][c];
        if (nw > 1) t = add_from(t, t, 16);
        else t = lane < 16 ? t : (__int128)0;
        // leading 62 bits of the sum: one conversion
        const bool minus = t < 0;
        const unsigned __int128 u = minus ? (unsigned __int128)(-t) : (unsigned __int128)t;
        const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
        const int up = uh ? 66 - __clzll((long long)uh) : 0;  // bits above 62
        const long long lead = uh ? (long long)((uh << (64 - up)) | (ul >> up)) : (long long)(ul >> 2);
        const double d0 = (double)lead;
        const double a = ps->arow[c];
        const int ud = uh ? up : 2;
        double d = shift_exponent(minus ? -d0 : d0, ud);
        const double Sj = __shfl_sync(HQ_FULL, d, j);
        const double al0 = ps->arow[j];
        const int hs = __double2hiint(Sj), es = (hs >> 20) - 1023;
        h = es >> 1;
        zero = (hs & 0x7fffffff) == 0;
        // s = S / 4^h in [1, 4): everything below is in units of 2^h of column j
        const double s = zero ? 1.0 : __hiloint2double((hs & 0xfffff) | ((1023 + (es & 1)) << 20), __double2loint(Sj));
        const float sf = __uint_as_float((uint32_t)__double2hiint(s) * 8u - ((1023u - 127u) << 23) +
                                         ((uint32_t)__double2loint(s) >> 29));
        const float yf = rsqrtf(sf);
        const double y0 = float_bits_to_double(yf);
        const double q = s * y0;
        const double al = shift_exponent(al0, -h);
        neg = __double2hiint(al) < 0;
        aa = fabs(al);
        // |al| <= 2 as a float, from its bits (0 when it does not matter for the seed)
        const int ah = __double2hiint(aa);
        const float af = ah > (900 << 20) ? __uint_as_float(((uint32_t)(ah - (896 << 20)) << 3) | ((uint32_t)__double2loint(aa) >> 29))
                                          : 0.f;
        const double g0 = float_bits_to_double(__fdividef(1.f, fmaf(af, sf * yf, sf)));
        const double e1 = fma(-q, y0, 1.0);
        nrm = fma(q * e1, fma(0.375, e1, 0.5), q);  // sqrt(s): s / sqrt(s), third order
        const double td = fma(aa, nrm, s);
        const double wc = fma(neg ? -nrm : nrm, a, shift_exponent(d, -h));  // v^T x_c
        const double e2 = fma(-td, g0, 1.0);
        gam = fma(g0, fma(e2, e2, e2), g0);  // 2 / v^T v
        const double phi = gam * wc;
        if (lane < 16) ps->m[c] = (c > j && c < kb && !zero) ? __double2ll_rn(phi) : 0ll;
        if (lane == 0) {
          // b 2^59 as an integer, from the bits of |b| in [1, 2]
          const unsigned long long bits = (unsigned long long)__double_as_longlong(nrm);
          const unsigned long long bi = ((bits & 0xfffffffffffffull) | 0x10000000000000ull) << ((int)(bits >> 52) - 1023 + 7);
          ps->b = zero ? 0ll : (neg ? (long long)bi : -(long long)bi);
          ps->shift = zero ? 0 : max(59 - h, 0);
        }
      }
      bar_warps(nthr);
      if (tid == 0) {
        tau[j] = bad ? nanv : (zero ? 0.0 : gam);
        ev[j0 + j] = zero ? kOzUnit : oz_bound(oz_abs_hi(aa + nrm));
        const int k = h + oz_bound(ps->cmax[j]) - 1023 - B;
        Q[(size_t)(j0 + j) * ld + j0 + j] = bad ? nanv : (zero ? 0.0 : oz_scale(neg ? nrm : -nrm, k));
      }
      const long long v = row < j ? 0ll : (long long)((unsigned long long)xj << ps->shift) - (row == j ? ps->b : 0ll);
      const int v1 = (int)(v >> 30), v0 = (int)(v & 0x3fffffff);
#pragma unroll
      for (int i = 0; i < CPT; ++i)
        if (i < left) {
          const int c = (i + jb) * G + cq;
          if (c == j) x[i] = row < j ? x[i] : v;
          else x[i] -= mul_shift59(v1, v0, ps->m[c]);  // m is zero for the columns done
        }
      if (jo == G - 1) {
        const long long first = x[0];
#pragma unroll
        for (int i = 0; i + 1 < CPT; ++i) x[i] = x[i + 1];
        x[CPT - 1] = first;
      }
    }
    if (in) {
      const int jb = kb >> LG;
#pragma unroll
      for (int i = 0; i < CPT; ++i) {
        const int c = ((i + jb) & (CPT - 1)) * G + cq;
        if (c < kb) {
          const size_t at = (size_t)(j0 + c) * ld + j0 + row;
          const double val = (double)x[i];
          V[at] = row < c ? 0.0 : oz_scale(val, -59);
          if (row < c) Q[at] = bad ? nanv : oz_scale(val, oz_bound(ps->cmax[c]) - 1023 - B);
        }
      }
    }
  }
  __syncthreads();
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
