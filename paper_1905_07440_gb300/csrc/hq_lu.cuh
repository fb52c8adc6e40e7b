// LU with partial pivoting and its solves: panels of 16 columns in registers, everything else as 16-term products on the tensor cores (hq_oz.cuh).
//
// A panel is held by four warps as in hq_panel.cuh (column c in warp c % 4, its rows over the lanes).  Per step
// the pivot column goes to all warps through shared memory (one barrier); every warp then finds the pivot
// (largest high word, one REDUX) and updates its own columns, so no row crosses warps.  Rows are not moved;
// every lane tracks the position its rows end at.  The column-by-column form in memory took four barriers
// and about 5800 cycles per column at n = 64.
// Triangles: the 16 x 16 diagonal blocks are inverted once (one warp each, 60 dependent FP64
// instructions), so the triangular solves become products too.
#pragma once
#include "hq_device.cuh"
#include "hq_oz.cuh"
#include "hq_panel.cuh"

namespace hq {

// 1 / u by a float seed and one third-order step in FP64 (no special cases: 0 and non-finite pivots
// show up in log|U_jj|).
__device__ __forceinline__ double recip_fp64(double u) {
  const int hi = __double2hiint(u), lo = __double2loint(u), e = (hi >> 20) & 0x7ff;
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, lo);  // |u| 2^(1023 - e) in [1, 2)
  const float f = __uint_as_float(((uint32_t)(hi & 0xfffff) << 3) | 0x3f800000u | ((uint32_t)lo >> 29));
  const double g = float_bits_to_double(__frcp_rn(f));
  const double r = fma(-m, g, 1.0);
  const double v = oz_scale(fma(g, fma(r, r, r), g), 1023 - e);
  return hi < 0 ? -v : v;
}

struct LuShared {
  double col[2][256];
};

// Columns p0 .. p0 + kb - 1, rows p0 .. n - 1 of A, in place (L below, U on and above the diagonal, rows
// in pivot order); piv[p0 + j] = the row swapped with p0 + j at step j.  Ends with a barrier.
template <int LM, int RPL>
__device__ __noinline__ void lu_panel_rows(double* A, int ld, int n, int p0, int kb, int* piv, LuShared* ls) {
  constexpr int kThreads = 32 * kPanelWarps;
  const int m = n - p0, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp < kPanelWarps) {
    double x[RPL][4];
    int pos[RPL];
    bool active[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
      pos[r] = lane + 32 * r;
      active[r] = pos[r] < m;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = 4 * i + warp;
        x[r][i] = (active[r] && c < kb) ? A[(size_t)(p0 + c) * ld + p0 + pos[r]] : 0.0;
      }
    }
    if (warp == 0) {
#pragma unroll
      for (int r = 0; r < RPL; ++r) ls->col[0][lane + 32 * r] = x[r][0];
    }
    bar_warps(kThreads);
#pragma unroll 1
    for (int j = 0; j < kb; ++j) {
      // x[.][i] is column 4 ((i + done) % 4) + warp; the warp's columns after j are entries first .. left - 1
      const int jw = j & 3, done = j >> 2, left = 4 - done, first = warp <= jw ? 1 : 0;
      double xj[RPL];
      uint32_t key = 0;
      int kr = 0;
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        xj[r] = ls->col[j & 1][lane + 32 * r];
        const uint32_t k = active[r] ? oz_abs_hi(xj[r]) + 1u : 0u;
        if (k > key) {
          key = k;
          kr = r;
        }
      }
      const uint32_t best = __reduce_max_sync(HQ_FULL, key);
      const int win = __ffs(__ballot_sync(HQ_FULL, key == best)) - 1;
      auto pick = [&](const double (&v)[RPL]) {
        double w = v[0];
#pragma unroll
        for (int r = 1; r < RPL; ++r)
          if (kr == r) w = v[r];
        return __shfl_sync(HQ_FULL, w, win);
      };
      int pk = pos[0];
#pragma unroll
      for (int r = 1; r < RPL; ++r)
        if (kr == r) pk = pos[r];
      const int from = __shfl_sync(HQ_FULL, pk, win);
      const double rp = recip_fp64(pick(xj));
      if (tid == 0) piv[p0 + j] = p0 + from;
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        if (lane == win && kr == r) {
          pos[r] = j;
          active[r] = false;
        } else if (pos[r] == j) {
          pos[r] = from;
        }
      }
      double l[RPL];
#pragma unroll
      for (int r = 0; r < RPL; ++r) l[r] = active[r] ? xj[r] * rp : 0.0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < left && i >= first) {
          double col[RPL];
#pragma unroll
          for (int r = 0; r < RPL; ++r) col[r] = x[r][i];
          const double u = pick(col);
#pragma unroll
          for (int r = 0; r < RPL; ++r) x[r][i] = fma(-l[r], u, x[r][i]);
        }
      if (j + 1 < kb && warp == ((j + 1) & 3)) {
        const bool turned = jw == 3;  // warp 0 takes its next column
#pragma unroll
        for (int r = 0; r < RPL; ++r) ls->col[(j + 1) & 1][lane + 32 * r] = turned ? x[r][1] : x[r][0];
      }
      if (warp == jw) {
#pragma unroll
        for (int r = 0; r < RPL; ++r)
          if (active[r]) x[r][0] = l[r];
      }
      if (jw == 3) {
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          const double f = x[r][0];
#pragma unroll
          for (int i = 0; i < 3; ++i) x[r][i] = x[r][i + 1];
          x[r][3] = f;
        }
      }
      bar_warps(kThreads);
    }
    const int done = kb >> 2;
#pragma unroll
    for (int r = 0; r < RPL; ++r)
      if (lane + 32 * r < m) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = 4 * ((i + done) & 3) + warp;
          if (c < kb) A[(size_t)(p0 + c) * ld + p0 + pos[r]] = x[r][i];
        }
      }
  }
  __syncthreads();
}

// Inverse of a triangular 16 x 16 block by one warp: M[16][16] row-major in shared memory, read from the
// kb x kb block at (p0, p0) of A (identity beyond kb).  kUnitLower: unit lower triangle, else upper.
template <bool kUnitLower>
__device__ inline void invert_triangle(const double* A, int ld, int p0, int kb, double* M) {
  const int lane = threadIdx.x & 31;
  auto a = [&](int r, int c) { return (r < kb && c < kb) ? A[(size_t)(p0 + c) * ld + p0 + r] : 0.0; };
  if (lane < 16) {
    const int o = lane & 8, c = lane & 7;
    double x[8];
    if (kUnitLower) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        double v = r == c ? 1.0 : 0.0;
#pragma unroll
        for (int k = 0; k < r; ++k) v = fma(-a(o + r, o + k), x[k], v);
        x[r] = v;
      }
    } else {
#pragma unroll
      for (int r = 7; r >= 0; --r) {
        double v = r == c ? 1.0 : 0.0;
#pragma unroll
        for (int k = r + 1; k < 8; ++k) v = fma(-a(o + r, o + k), x[k], v);
        x[r] = o + r < kb ? v * recip_fp64(a(o + r, o + r)) : v;
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      M[(o + r) * 16 + o + c] = x[r];
      M[(o + r) * 16 + (8 - o) + c] = 0.0;
    }
  }
  __syncwarp();
  // off-diagonal block: -B22 A21 B11 (lower), -B11 A12 B22 (upper)
  const int ro = kUnitLower ? 8 : 0, co = 8 - ro;
  double y[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = (lane >> 3) + 4 * u, c = lane & 7;
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) v = fma(a(ro + r, co + k), M[(co + k) * 16 + co + c], v);
    y[u] = v;
  }
  double* X = M + ro * 16 + co;
#pragma unroll
  for (int u = 0; u < 2; ++u) X[((lane >> 3) + 4 * u) * 16 + (lane & 7)] = y[u];
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = (lane >> 3) + 4 * u, c = lane & 7;
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) v = fma(M[(ro + r) * 16 + ro + k], X[k * 16 + c], v);
    y[u] = -v;
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u) X[((lane >> 3) + 4 * u) * 16 + (lane & 7)] = y[u];
  __syncwarp();
}

// C(r, c) <- base Cin(r, c) + sign sum_k A(r, k) B(k, c) for r0 <= r < r1, c0 <= c < c1, k < kb <= 16, with A(r, k) =
// A[r ar + k ak], B(k, c) = B[k bk + c bc] and C column-major (ldc).  With base = 0 B may be rows of C's
// own columns (each warp reads a column's terms before it writes).  Ends with a barrier.
struct Rank16 {
  const double* A;
  int ar, ak;
  const double* B;
  int bk, bc;
  const double* Cin;
  double* C;
  int ldc;
  double sign, base;
};

template <int LM>
__device__ __noinline__ void oz_rank(const Rank16 q, int r0, int r1, int c0, int c1, int kb, uint2* frag, int* er) {
  oz_rank16<LM <= 8 ? 1 : 2>(q.base == 0.0, r0, r1, c0, c1, kb, frag, er, [&](int r, int k) { return q.A[(size_t)r * q.ar + (size_t)k * q.ak]; },
            [&](int k, int c) { return q.sign * q.B[(size_t)k * q.bk + (size_t)c * q.bc]; },
            [&](int r, int c) {
              return q.base != 0.0 ? *reinterpret_cast<const double2*>(q.Cin + (size_t)c * q.ldc + r) : make_double2(0.0, 0.0);
            },
            [&](int r, int c, double v0, double v1, double p0, double p1, double2 x) {
              *reinterpret_cast<double2*>(q.C + (size_t)c * q.ldc + r) = make_double2(fma(v0, p0, x.x), fma(v1, p1, x.y));
            });
}

// Y(p0 : p0 + kb, c0 : c1) <- M Y(p0 : p0 + kb, c0 : c1) for a 16 x 16 row-major M.
template <int LM>
__device__ inline void oz_left16(const double* M, double* Y, int ld, int p0, int kb, int c0, int c1, uint2* frag, int* er) {
  oz_rank<LM>(Rank16{M, 16, 1, Y + p0, 1, ld, nullptr, Y + p0, ld, 1.0, 0.0}, 0, kb, c0, c1, kb, frag, er);
}

// C(r0:r1, c0:c1) -= A(r0:r1, k0:k0+kb) B(k0:k0+kb, c0:c1), kb <= 16.
template <int LM>
__device__ inline void oz_rank_update(double* C, const double* A, const double* B, int ld, int r0, int r1, int c0, int c1,
                                      int k0, int kb, uint2* frag, int* er) {
  oz_rank<LM>(Rank16{A + (size_t)k0 * ld, 1, ld, B + k0, 1, ld, C, C, ld, -1.0, 1.0}, r0, r1, c0, c1, kb, frag, er);
}

// In place LU of A; tri: oz_pad(n) / 16 blocks of 16 x 16, left holding the inverses of L's diagonal
// blocks.  Returns sum_j log|U_jj| (in every thread).
template <int LM>
__device__ inline double oz_lu(double* A, int n, int* piv, double* red, double* tri, uint2* frag, int* er) {
  const int tid = threadIdx.x;
  LuShared* ls = reinterpret_cast<LuShared*>(frag);
  for (int p0 = 0; p0 < n; p0 += 16) {
    const int kb = min(16, n - p0), p1 = p0 + kb, m = n - p0;
    if (m <= 32) lu_panel_rows<LM, 1>(A, n, n, p0, kb, piv, ls);
    else if (LM <= 8 || m <= 64) lu_panel_rows<LM, 2>(A, n, n, p0, kb, piv, ls);  // LM <= 8: n <= 64
    else if (m <= 128) lu_panel_rows<LM, LM <= 8 ? 2 : 4>(A, n, n, p0, kb, piv, ls);
    else lu_panel_rows<LM, LM <= 8 ? 2 : 8>(A, n, n, p0, kb, piv, ls);
    double* M = tri + (p0 >> 4) * 256;
    if (tid < 32) invert_triangle<true>(A, n, p0, kb, M);
    else
      for (int c = tid - 32; c < n; c += HQ_THREADS - 32) {  // the panel's swaps on the other columns
        if (c >= p0 && c < p1) continue;
        double* ac = A + (size_t)c * n;
        for (int j = p0; j < p1; ++j) {
          const int p = piv[j];
          if (p != j) { const double v = ac[j]; ac[j] = ac[p]; ac[p] = v; }
        }
      }
    __syncthreads();
    if (p1 < n) {
      oz_left16<LM>(M, A, n, p0, kb, p1, n, frag, er);
      oz_rank_update<LM>(A, A, A, n, p1, n, p1, n, p0, kb, frag, er);
    }
  }
  double a = 0.0;
  for (int j = tid; j < n; j += HQ_THREADS) a += log(fabs(A[(size_t)j * n + j]));
  return block_sum(a, red);
}

// Y <- A^-1 Y (n right-hand sides) for the factors of oz_lu; tri as oz_lu left it (overwritten).
template <int LM>
__device__ inline void oz_lu_solve(const double* A, int n, const int* piv, double* Y, double* tri, uint2* frag,
                                   int* er) {
  const int tid = threadIdx.x, warp = tid >> 5;
  // all row swaps at once: thread 0 turns them into a permutation, then a warp moves a column
  int* perm = er;
  if (tid == 0) {
    for (int r = 0; r < n; ++r) perm[r] = r;
    for (int j = 0; j < n; ++j) {
      const int p = piv[j], v = perm[j];
      perm[j] = perm[p];
      perm[p] = v;
    }
  }
  __syncthreads();
  for (int c = warp; c < n; c += HQ_WARPS) {
    double* y = Y + (size_t)c * n;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if ((tid & 31) + 32 * u < n) v[u] = y[perm[(tid & 31) + 32 * u]];
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if ((tid & 31) + 32 * u < n) y[(tid & 31) + 32 * u] = v[u];
  }
  __syncthreads();
  for (int p0 = 0; p0 < n; p0 += 16) {
    const int kb = min(16, n - p0), p1 = p0 + kb;
    oz_left16<LM>(tri + (p0 >> 4) * 256, Y, n, p0, kb, 0, n, frag, er);
    if (p1 < n) oz_rank_update<LM>(Y, A, Y, n, p1, n, 0, n, p0, kb, frag, er);
  }
  for (int b = warp; 16 * b < n; b += HQ_WARPS) invert_triangle<false>(A, n, 16 * b, min(16, n - 16 * b), tri + b * 256);
  __syncthreads();
  for (int p0 = ((n - 1) >> 4) << 4; p0 >= 0; p0 -= 16) {
    const int kb = min(16, n - p0);
    oz_left16<LM>(tri + (p0 >> 4) * 256, Y, n, p0, kb, 0, n, frag, er);
    if (p0 > 0) oz_rank_update<LM>(Y, A, Y, n, 0, p0, 0, n, p0, kb, frag, er);
  }
}

}  // namespace hq
