// Dense linear algebra of a chain with its contractions on the tensor cores (hq_oz.cuh): blocked QR and Q formation, the triangular factor, LU and solves, products.
// Column-major n x n matrices with stride ld = n (a multiple of 4, so that row pairs are 16-byte
// aligned), one CTA per matrix.  What stays on the FP64 pipe is O(n^2) or narrow: panels of 16
// columns, 16 x 16 triangles, scalings.
#pragma once
#include <climits>
#include "hq_device.cuh"
#include "hq_oz.cuh"
#include "hq_lu.cuh"
#include "hq_panel.cuh"

namespace hq {

// Rows of a staged block: 64, or 32 where 64 rows of n terms would not fit beside the rest.
__host__ __device__ constexpr int oz_rows(int n) { return n <= 160 ? 64 : 32; }
__host__ __device__ constexpr int oz_pad(int n) { return (n + 15) & ~15; }
// bytes of the fragment scratch: a staged row block, or a QR panel in both fragment orders plus T
__host__ __device__ constexpr size_t oz_frag_bytes(int n) {
  return (size_t)oz_pad(n) * oz_rows(n) * 12 + 2 * 6 * 32 * 8;
}

struct OzScratch {
  uint2* frag;   // oz_frag_bytes(n)
  int* er;       // [oz_pad(n)] row bounds
  int* ec;       // [oz_pad(n)] column bounds
  double* tall;  // [oz_pad(n) / 16][16][16] triangular factors T of the QR panels
  double* ws;    // [16][16]
  int* ev;       // [oz_pad(n)] bounds of the reflector vectors
  int n;
};

// Scratch of the QR: reflector scalars, 1 / D, pivot order.
struct QrScratch {
  double* tau;   // [16]
  double* rinv;  // [n] 1 / D
  int* perm;     // [n] perm[j] = original column placed at position j
};

struct RowPair {
  double v0, v1;
};
__device__ __forceinline__ RowPair load_pair(const double* p) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  return {v.x, v.y};
}
__device__ __forceinline__ void store_pair(double* p, double a, double b) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
}

// Matrices of up to kTiny rows (lattices of up to 16 sites): one MMA step holds a whole product, and its
// splits and conversions take 12 thousand cycles where the FP64 pipe needs 2 thousand for the 16 DFMAs per
// thread.  So products, the triangular factor and Q stay in FP64 there.
constexpr int kTiny = 16;

// ---------------------------------------------------------------------- blocked QR
// Column-pivoted QR in the form used for DQMC stabilisation by Bauer (SciPost Phys. Core 2,
// 011 (2020)): the columns are ordered once by decreasing Euclidean norm, then factored by
// unpivoted Householder QR.  The product being factored is column-graded (B..B U D), so the
// one-time ordering gives the graded R that the UDV decomposition needs, without per-step
// pivot searches and norm downdates.

// Ordering key of a squared norm a 4^e: the IEEE bit pattern, which orders positive doubles exactly like their values,
// with the exponent counted from 0 and free to leave its eleven bits downwards.
__device__ __forceinline__ long long norm_key(double a, int e) {
  return __double_as_longlong(a) - (1023ll << 52) + (long long)min(2 * e, 2036) * (1ll << 52);
}

// The key of a column whose squares leave the normal range (norms outside 2^-450 .. 2^511), by a group of 4 lanes: the
// column is summed scaled by its largest entry.  Zero columns come last, columns with a non-finite value first.
static __device__ __noinline__ long long scaled_norm_key(const double* col, int n) {
  const int sub = threadIdx.x & 3;
  uint32_t top = 0;
  for (int r = sub; r < n; r += 4) top = max(top, oz_abs_hi(col[r]));
  top = max(top, __shfl_xor_sync(HQ_FULL, top, 1));
  top = max(top, __shfl_xor_sync(HQ_FULL, top, 2));
  const int e = (int)(top >> 20) - 1023;
  double b = 0.0;
  for (int r = sub; r < n; r += 4) {
    const double v = shift_exponent(col[r], -e);
    b = fma(v, v, b);
  }
  b = group_sum<4>(b);
  return e == kPanelBad ? LLONG_MAX : e == kPanelZero ? LLONG_MIN : norm_key(b, e);
}

// Q <- columns of P ordered by decreasing norm (stable: ties keep index order); perm records the order.
// norm2: n doubles of scratch.
__device__ inline void prepivot(const double* P, double* Q, int ld, int n, const QrScratch& s, double* norm2) {
  const int g = threadIdx.x >> 2, sub = threadIdx.x & 3;
  for (int base = 0; base < n; base += HQ_THREADS / 4) {
    const int c = base + g;
    double a = 0.0;
    if (c < n) {
      const double* col = P + (size_t)c * ld;
      for (int r = sub; r < n; r += 4) a = fma(col[r], col[r], a);
    }
    a = group_sum<4>(a);
    const int f = __double2hiint(a) >> 20;
    const bool out = c < n && (f < 1023 - 900 || f >= 0x7ff);
    long long key = norm_key(a, 0);
    if (__any_sync(HQ_FULL, out)) {
      const long long k = scaled_norm_key(P + (size_t)min(c, n - 1) * ld, n);
      if (out) key = k;
    }
    if (c < n && sub == 0) norm2[c] = __longlong_as_double(key);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < n; c += HQ_THREADS) {
    const long long mine = __double_as_longlong(norm2[c]);
    int rank = 0;
    for (int o = 0; o < n; ++o) {
      const long long other = __double_as_longlong(norm2[o]);
      rank += (other > mine) || (other == mine && o < c);
    }
    s.perm[rank] = c;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < n * n; idx += HQ_THREADS) {
    const int r = idx % n, j = idx / n;
    Q[(size_t)j * ld + r] = P[(size_t)s.perm[j] * ld + r];
  }
  __syncthreads();
}

// Panel of kb <= 16 columns from j0 and its T factor; leaves the panel's row-term fragments in z.frag.
template <int LM>
__device__ __noinline__ void oz_panel(double* Q, double* V, int ld, int n, int j0, int kb, double* tau,
                                      const OzScratch& z) {
  PanelShared* ps = reinterpret_cast<PanelShared*>(z.frag);
  const int m = n - j0;
  if (m <= 32) panel_house<LM, 1>(Q, V, ld, n, j0, kb, ps, tau, z.ev, z.er);
  else if (LM <= 8 || m <= 64) panel_house<LM, 2>(Q, V, ld, n, j0, kb, ps, tau, z.ev, z.er);  // LM <= 8: n <= 64
  else if (m <= 128) panel_house<LM, LM <= 8 ? 2 : 4>(Q, V, ld, n, j0, kb, ps, tau, z.ev, z.er);
  else panel_house<LM, LM <= 8 ? 2 : 8>(Q, V, ld, n, j0, kb, ps, tau, z.ev, z.er);
  stage_panel(z.frag, V, ld, n, j0, kb, z.ev);
  // the sums go behind the fragments, where the block application stages T
  const int nk = (m + 15) >> 4;
  panel_t(z.frag, nk, kb, tau, z.ev + j0, reinterpret_cast<unsigned long long*>(z.frag + (size_t)nk * 2 * kOzDigits * 32),
          z.ws, z.tall + (j0 >> 4) * 256);
}

// The reflectors in columns j0 .. j1 - 1 of V (zero above their first row) applied at once to columns c0 .. cend - 1, rows j0 .. n - 1, of A:
//   trans:  A <- (I - V T V^T)^T A     (trailing update of the QR)
//   !trans: A <- (I - V T V^T) A       (Q formation)
// A warp takes 16 columns and runs W^T = A^T V, Z^T = W^T T (or W^T T^T) and A^T -= Z^T V^T back to back:
// each result leaves the accumulators in the layout of the next left operand, so nothing but V's
// and T's fragments is shared and A is read and written in place.  With fewer column groups than
// warps, several warps form W of the same columns and share out the rows of the update.  trans follows
// oz_panel, which has left V's row-term fragments in place.
template <int LM>
__device__ __noinline__ void oz_wy_apply(bool trans, const double* V, int ld, int n, int j0, int j1, const double* T, double* A,
                                         int c0, int cend, const OzScratch& z) {
  const int kb = j1 - j0, nr = n - j0, nk = (nr + 15) >> 4;
  uint2* vk = z.frag;
  uint2* vn = vk + (size_t)nk * 2 * kOzDigits * 32;
  uint2* tf = vn + (size_t)nk * 2 * kOzDigits * 32;
  int* et = z.ec;  // [16]
  auto v = [&](int rr, int k) { return (k < kb && rr < nr) ? V[(size_t)(j0 + k) * ld + j0 + rr] : 0.0; };
  auto evk = [&](int k) { return k < kb ? z.ev[j0 + k] : 128; };
  if (!trans) stage_panel(vk, V, ld, n, j0, kb, z.ev);
  oz_stage_rows(vn, z.er, nr, 16, [&](int r, int k) { return v(r, k); });
  oz_stage_rows(tf, et, 16, 16, [&](int r, int k) { return trans ? T[k * 16 + r] : T[r * 16 + k]; });
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int ncg = (cend - c0 + 15) >> 4;
  const int parts = ncg >= HQ_WARPS ? 1 : HQ_WARPS / ncg;
  constexpr int kTiles = LM <= 8 ? 1 : 2;
  const int rp = ((nr + parts - 1) / parts + 8 * kTiles - 1) / (8 * kTiles) * (8 * kTiles);
  for (int unit = warp; unit < ((ncg * parts + HQ_WARPS - 1) / HQ_WARPS) * HQ_WARPS; unit += HQ_WARPS) {
    const bool work = unit < ncg * parts;
    const int ca = c0 + (unit % ncg) * 16 + g, cb = ca + 8, rb = work ? (unit / ncg) * rp : nr;
    const double* pa = A + (size_t)(ca < cend ? ca : c0) * ld + j0;
    const double* pb = A + (size_t)(cb < cend ? cb : c0) * ld + j0;
    uint32_t a[4][kOzDigits];
    int E[2] = {128, 128};
    if (work && rb < nr) {
      uint32_t ma = 0, mb = 0;
#pragma unroll 2
      for (int r = 2 * t; r < nr; r += 8) {
        const RowPair x = load_pair(pa + r), y = load_pair(pb + r);
        ma = max(ma, max(oz_abs_hi(x.v0), oz_abs_hi(x.v1)));
        mb = max(mb, max(oz_abs_hi(y.v0), oz_abs_hi(y.v1)));
      }
      ma = max(ma, __shfl_xor_sync(HQ_FULL, ma, 1));
      mb = max(mb, __shfl_xor_sync(HQ_FULL, mb, 1));
      ma = max(ma, __shfl_xor_sync(HQ_FULL, ma, 2));
      mb = max(mb, __shfl_xor_sync(HQ_FULL, mb, 2));
      E[0] = oz_bound(ma);
      E[1] = oz_bound(mb);
      // W^T: sums over up to 256 rows fit one accumulator, because |v|^2 < 16 bounds the sum by
      // 4 sqrt(n) times the column's largest entry
      long long Tw[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
      RowPair nx[4];
      auto fetch = [&](int r) {  // a step ahead in the wide class
        const RowPair z0{0.0, 0.0};
        nx[0] = r < nr ? load_pair(pa + r) : z0;
        nx[1] = r < nr ? load_pair(pb + r) : z0;
        nx[2] = r + 8 < nr ? load_pair(pa + r + 8) : z0;
        nx[3] = r + 8 < nr ? load_pair(pb + r + 8) : z0;
      };
      if (LM > 8) fetch(2 * t);
#pragma unroll 1
      for (int ks = 0; ks < nk; ++ks) {
        if (LM <= 8) fetch(16 * ks + 2 * t);
        const RowPair x0 = nx[0], x1 = nx[1], x2 = nx[2], x3 = nx[3];
        if (LM > 8) fetch(16 * (ks + 1) + 2 * t);
        oz_split<kOzP>(x0.v0, x0.v1, E[0], E[0], a[0]);
        oz_split<kOzP>(x1.v0, x1.v1, E[1], E[1], a[1]);
        oz_split<kOzP>(x2.v0, x2.v1, E[0], E[0], a[2]);
        oz_split<kOzP>(x3.v0, x3.v1, E[1], E[1], a[3]);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint2* fr = vk + (size_t)(ks * 2 + j) * kOzDigits * 32 + lane;
          oz_mma(a, [&](int d) { return fr[d * 32]; }, Tw[j]);
        }
      }
      double w[2][4];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) w[j][e] = oz_scale((double)Tw[j][e], oz_expo<kOzP>(evk(8 * j + 2 * t + (e & 1)), E[e >> 1]));
      oz_left_from_acc(w, a, E);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        long long Tz[4] = {0, 0, 0, 0};
        const uint2* fr = tf + (size_t)j * kOzDigits * 32 + lane;
        oz_mma(a, [&](int d) { return fr[d * 32]; }, Tz);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          w[j][e] = oz_scale((double)Tz[e], oz_expo<kOzP>(et[8 * j + 2 * t + (e & 1)], E[e >> 1]));
      }
      oz_left_from_acc(w, a, E);
    }
    if (parts > 1) __syncthreads();  // W of every warp is formed before rows change
    if (work && rb < nr)
      oz_apply_rows<kTiles, (kTiles > 1)>(
          vn + (size_t)(rb >> 3) * kOzDigits * 32, z.er + rb, min(rp, nr - rb), a, E, ca, cb, cend,
          [&](int r, int c) { return *reinterpret_cast<const double2*>(A + (size_t)c * ld + j0 + rb + r); },
          [&](int r, int c, double v0, double v1, double p0, double p1, double2 x) {
            store_pair(A + (size_t)c * ld + j0 + rb + r, fma(-v0, p0, x.x), fma(-v1, p1, x.y));
          });
  }
  __syncthreads();
}

// Householder QR in panels of 16 columns; the trailing columns take each panel's reflectors as one
// block.  R goes to the upper triangle of Q (below it Q is left undefined), the reflector vectors to V,
// and the panels' T factors are kept for the Q formation.
template <int LM>
__device__ inline void oz_qr(double* Q, double* V, int ld, int n, const QrScratch& s, const OzScratch& z) {
  for (int j0 = 0; j0 < n; j0 += 16) {
    const int j1 = min(j0 + 16, n);
    oz_panel<LM>(Q, V, ld, n, j0, j1 - j0, s.tau, z);
    if (j1 < n) oz_wy_apply<LM>(true, V, ld, n, j0, j1, z.tall + (j0 >> 4) * 256, Q, j1, n, z);
  }
}

// U <- H_0 ... H_{n-1}: the panels' blocks applied to the identity, last panel first (columns left
// of a panel are still unit vectors there).
template <int LM>
__device__ inline void oz_form_q(const double* V, int ld, int n, double* U, const OzScratch& z) {
  if (n <= kTiny) {  // one panel: U = I - V (T V^T), an entry per thread
    double* W = z.ws;
    const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
    double a = 0.0;
    if (c < n)
      for (int k = r; k < n; ++k) a = fma(z.tall[r * 16 + k], V[(size_t)k * ld + c], a);
    W[r * 16 + c] = a;
    __syncthreads();
    if (r < n && c < n) {
      a = r == c ? 1.0 : 0.0;
      for (int k = 0; k <= r; ++k) a = fma(-V[(size_t)k * ld + r], W[k * 16 + c], a);
      U[(size_t)c * ld + r] = a;
    }
    __syncthreads();
    return;
  }
  set_identity(U, ld, n);
  __syncthreads();
  for (int j0 = ((n - 1) >> 4) << 4; j0 >= 0; j0 -= 16)
    oz_wy_apply<LM>(false, V, ld, n, j0, min(j0 + 16, n), z.tall + (j0 >> 4) * 256, U, j0, n, z);
}

// Tout = D^-1 R (rows of Tprev in pivot order): T' Tprev with T' = D^-1 R Pi^T.  The rows of Tprev differ in size, and
// R(r, k) makes up for it: with one exponent per line the small rows would keep few bits of the digits, where a
// sum of FP64 products keeps all (G of an 8x8 lattice at beta = 16, charge-ordered: error 2e-14 against 5e-15; with a
// site lowered by 6: 4e-10 against 1e-12).  So the terms of the sum are scaled to rows of Tprev in 1/2 .. 1.
template <int LM, bool kWide>
__device__ __noinline__ void oz_t_product(const double* P, int n, const int* perm, const double* rinv,
                                          const double* Tprev, double* Tout, const OzScratch& z) {
  auto fr = [&](int r, int k) { return k >= r ? P[(size_t)k * n + r] * rinv[r] : 0.0; };
  int* se = z.ev;  // exponents of the rows of Tprev, in the end in pivot order (the reflectors' bounds are done with)
  const int tid = threadIdx.x;  // n <= HQ_THREADS
  oz_line_bounds(false, n, n, se, [&](int k, int c) { return Tprev[(size_t)c * n + k]; });
  if (tid < n) se[tid] = se[tid] == kOzBad ? 0 : se[tid] - 1023;
  __syncthreads();
  oz_line_bounds(true, n, n, z.ec, [&](int c, int k) { return oz_scale_any(Tprev[(size_t)c * n + k], -se[k]); });
  const int mine = tid < n ? se[perm[tid]] : 0;
  __syncthreads();
  if (tid < n) se[tid] = mine;
  __syncthreads();
  oz_line_bounds(false, n, n, z.er, [&](int r, int k) { return oz_scale_any(fr(r, k), se[k]); });
  oz_gemm<LM <= 8 ? 2 : 4, kWide, true>(
      n, n, n, oz_rows(n), z.frag, fr, [&](int r) { return z.er[r]; },
      [&](int k, int c) { return Tprev[(size_t)c * n + perm[k]]; }, [&](int c) { return z.ec[c]; },
      [&](int r, int c, double v0, double v1) { store_pair(Tout + (size_t)c * n + r, v0, v1); },
      [&](int k) { return se[k]; });
}

template <int LM>
__device__ inline void oz_t_update(const double* P, int n, const QrScratch& s, double* D, const double* Tprev,
                                   double* Tout, const OzScratch& z) {
  for (int j = threadIdx.x; j < n; j += HQ_THREADS) {
    const double dj = fabs(P[(size_t)j * n + j]);
    D[j] = dj;
    s.rinv[j] = 1.0 / dj;
  }
  __syncthreads();
  if (Tprev == nullptr) {
    for (int idx = threadIdx.x; idx < n * n; idx += HQ_THREADS) {
      const int j = idx % n, c = idx / n;
      Tout[(size_t)s.perm[c] * n + j] = (c >= j) ? P[(size_t)c * n + j] * s.rinv[j] : 0.0;
    }
    __syncthreads();
  } else if (n <= kTiny) {
    const int r = threadIdx.x & 15, c = threadIdx.x >> 4;
    if (r < n && c < n) {
      double a = 0.0;
      for (int k = r; k < n; ++k) a = fma(P[(size_t)k * n + r], Tprev[(size_t)c * n + s.perm[k]], a);
      Tout[(size_t)c * n + r] = a * s.rinv[r];
    }
    __syncthreads();
  } else if (LM > 8 && n > 64) {
    oz_t_product<LM, true>(P, n, s.perm, s.rinv, Tprev, Tout, z);
  } else {
    oz_t_product<LM, false>(P, n, s.perm, s.rinv, Tprev, Tout, z);
  }
}

// C = A diag(kd) B diag(cd) (kd, cd may be null) with A(r, k) = A[r ar + k ak], B(k, c) = B[k bk + c bc] (each with a
// unit stride), C column-major.
template <int LM, bool kWide>
__device__ __noinline__ void oz_product_mm(int n, const double* A, int ar, int ak, const double* B, int bk, int bc,
                                           const double* kd, const double* cd, double* C, const OzScratch& z) {
  auto fa = [&](int r, int k) { return A[(size_t)r * ar + (size_t)k * ak]; };
  auto fb = [&](int k, int c) {
    const double v = B[(size_t)k * bk + (size_t)c * bc];
    return kd ? v * kd[k] : v;
  };
  oz_line_bounds(ak == 1, n, n, z.er, fa);
  oz_line_bounds(bk == 1, n, n, z.ec, [&](int c, int k) { return fb(k, c); });
  oz_gemm<LM <= 8 ? 2 : 4, kWide, false>(
      n, n, n, oz_rows(n), z.frag, fa, [&](int r) { return z.er[r]; }, fb, [&](int c) { return z.ec[c]; },
      [&](int r, int c, double v0, double v1) {
        if (cd) {
          v0 *= cd[c];
          v1 *= cd[c];
        }
        store_pair(C + (size_t)c * n + r, v0, v1);
      });
}

template <int LM, bool TA, bool TB>
__device__ inline void oz_mm(int n, const double* A, const double* B, const double* kd, const double* cd, double* C,
                             const OzScratch& z) {
  if (n <= kTiny) {
    const int r = threadIdx.x & 15, c = threadIdx.x >> 4;
    __syncthreads();
    if (r < n && c < n) {
      double a = 0.0;
      for (int k = 0; k < n; ++k) {
        const double b = TB ? B[k * n + c] : B[c * n + k];
        a = fma(TA ? A[r * n + k] : A[k * n + r], kd ? b * kd[k] : b, a);
      }
      C[c * n + r] = cd ? a * cd[c] : a;
    }
    __syncthreads();
    return;
  }
  const int ar = TA ? n : 1, ak = TA ? 1 : n, bk = TB ? n : 1, bc = TB ? 1 : n;
  if (LM > 8 && n > 64) oz_product_mm<LM, true>(n, A, ar, ak, B, bk, bc, kd, cd, C, z);
  else oz_product_mm<LM, false>(n, A, ar, ak, B, bk, bc, kd, cd, C, z);
}

// Flush of delayed updates: G(r, c) += sum_m A[m][r] B[m][c], m < kk (A, B [kk][n]).  The wide class has an
// instance of its own (its 65 thousand entries outweigh the code; 16x16 local sweeps 430 -> 390 ms).
template <int LM>
__device__ __noinline__ void oz_flush(double* G, const double* A, const double* B, int n, int kk, const OzScratch& z) {
  for (int m0 = 0; m0 < kk; m0 += 16) {
    const int kb = min(16, kk - m0);
    if (LM <= 8)
      oz_rank<LM>(Rank16{A + (size_t)m0 * n, 1, n, B + (size_t)m0 * n, n, 1, G, G, n, 1.0, 1.0}, 0, n, 0, n, kb, z.frag, z.er);
    else
      oz_rank16<2>(false, 0, n, 0, n, kb, z.frag, z.er, [&](int r, int k) { return A[(m0 + k) * n + r]; },
                [&](int k, int c) { return B[(m0 + k) * n + c]; },
                [&](int r, int c) { return *reinterpret_cast<const double2*>(G + c * n + r); },
                [&](int r, int c, double v0, double v1, double p0, double p1, double2 x) {
                  store_pair(G + c * n + r, fma(v0, p0, x.x), fma(v1, p1, x.y));
                });
  }
}

// ------------------------------------------------------------ separable propagator
// P <- the product of `count` slice matrices times the start: identity, or with U its columns times D.
//   kAfter:  P <- diag(d_k) E P per slice (B^T = exp(-dtau V) exp(-dtau K), top-down products)
//   !kAfter: P <- E diag(d_k) P           (B = exp(-dtau K) exp(-dtau V))
// dv(k, r): diagonal entry r of the k-th slice applied.  A warp keeps its columns in registers through
// all slices; dbuf holds the diagonals of `cap` slices at a time.
template <bool kAfter, class DV>
__device__ __forceinline__ void oz_slices(int nx, int ny, int n, const OzKin& K, double* P, const double* U,
                                          const double* D, int count, DV dv, double* dbuf, int cap) {
  for (int k0 = 0; k0 < count; k0 += cap) {
    const int m = min(cap, count - k0);
    __syncthreads();
    for (int idx = threadIdx.x; idx < m * n; idx += HQ_THREADS) dbuf[idx] = dv(k0 + idx / n, idx % n);
    __syncthreads();
    oz_kin_lines(
        nx, ny, n,
        [&](int c, int i, double& v0, double& v1) {
          if (k0 > 0) {
            const RowPair p = load_pair(P + (size_t)c * n + i);
            v0 = p.v0;
            v1 = p.v1;
          } else if (U) {
            const RowPair p = load_pair(U + (size_t)c * n + i);
            v0 = p.v0 * D[c];
            v1 = p.v1 * D[c];
          } else {
            v0 = i == c ? 1.0 : 0.0;
            v1 = i + 1 == c ? 1.0 : 0.0;
          }
        },
        [&](double (&z)[2][4], bool two_x, bool two_y, auto visit) {
          for (int k = 0; k < m; ++k) {
            const double* dk = dbuf + k * n;
            auto scale = [&](bool on, int, int i, double& v0, double& v1) {
              if (on) {
                v0 *= dk[i];
                v1 *= dk[i + 1];
              }
            };
            if (!kAfter) visit(scale);
            oz_kin_tile(K, z, two_x, two_y);
            if (kAfter) visit(scale);
          }
        },
        [&](int c, int i, double v0, double v1) { store_pair(P + (size_t)c * n + i, v0, v1); });
  }
  __syncthreads();
}

// The same for n <= kTiny in FP64: a matrix entry per thread, the columns in shared memory (buf: 512
// doubles and `cap` slices' diagonals) between the two passes of a slice.
template <bool kAfter, class DV>
__device__ __forceinline__ void tiny_slices(int nx, int ny, int n, const double* ex, const double* ey, double* P,
                                            const double* U, const double* D, int count, DV dv, double* buf, int cap) {
  double* dbuf = buf + 512;  // [cap][n] diagonals of a run of slices
  const int i = threadIdx.x & 15, c = threadIdx.x >> 4, x = i % nx, y = i / nx;
  const bool on = i < n && c < n;
  double *A = buf + 16 * c, *T = buf + 256 + 16 * c;
  double v = 0.0;
  if (on) v = U ? U[(size_t)c * n + i] * D[c] : (i == c ? 1.0 : 0.0);
  for (int k = 0; k < count; ++k) {
    if (k % cap == 0) {
      __syncthreads();
      for (int w = threadIdx.x; w < min(cap, count - k) * n; w += HQ_THREADS) dbuf[w] = dv(k + w / n, w % n);
      __syncthreads();
    }
    const double d = on ? dbuf[(k % cap) * n + i] : 0.0;
    A[i] = kAfter ? v : v * d;
    __syncthreads();
    double a = 0.0;
    if (on)
      for (int b = 0; b < nx; ++b) a = fma(ex[x * nx + b], A[b + nx * y], a);
    T[i] = a;
    __syncthreads();
    v = 0.0;
    if (on)
      for (int b = 0; b < ny; ++b) v = fma(ey[y * ny + b], T[x + nx * b], v);
    if (kAfter) v *= d;
  }
  if (on) P[(size_t)c * n + i] = v;
  __syncthreads();
}

// Correction vectors of a block move at `site` (chunk q: slices lo .. lo + m - 1, lo = q nw, D_t = exp(-dtau V_t)
// from ev [L][n], D'_t the same with the shifted entry xs[t] at the site):
//   V column lo + s: D'_lo E ... D'_(lo+s-1) E e_site             (s = 0 .. m - 1 slices)
//   R column lo + m - s: E D_(lo+m-1) ... E D_(lo+m-s) e_site     (s = 1 .. m)
// A vector is a matrix column to the kinetic tiles; columns of different chunks with the same s share a
// tile, and a warp runs a tile's s slices in registers.  Longest first over the warps.  (As FP64 line
// passes over all vectors, one slice per barrier pair, this took 1.1 million cycles per move at 8x8, L = 80.)
template <int LM>
__device__ __noinline__ void oz_corr(int nx, int ny, int n, int L, int nw, int nq, const OzKin& K, int site,
                                     const double* ev, const double* xs, double* V, double* R) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const bool two_x = nx <= 8, two_y = ny <= 8;
  const int per = (two_x ? 2 : 1) * (two_y ? 2 : 1), tg = (nq + per - 1) / per;
  for (int idx = threadIdx.x; idx < nq * n; idx += HQ_THREADS)
    V[(size_t)(idx / n) * nw * n + idx % n] = idx % n == site ? 1.0 : 0.0;
#pragma unroll 1
  for (int task = warp; task < (2 * nw - 1) * tg; task += HQ_WARPS) {
    const int rest = task - tg;
    const bool right = task < tg || rest % (2 * tg) < tg;
    const int s = task < tg ? nw : nw - 1 - rest / (2 * tg), gq = task < tg ? task : rest % tg;
    double z[2][4];
    auto visit = [&](auto f) {
#pragma unroll
      for (int w = 0; w < 2; ++w)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int x = two_x ? 2 * t : 8 * w + 2 * t, y = two_y ? g : 8 * h + g;
          const int q = gq * per + (two_y ? h : 0) * (two_x ? 2 : 1) + (two_x ? w : 0);
          const int lo = q * nw, m = min(nw, L - lo);
          f(x < nx && y < ny && q < nq && (right ? s <= m : s < m), right ? lo + m - s : lo + s, x + nx * y, z[w][2 * h],
            z[w][2 * h + 1]);
        }
    };
    visit([&](bool on, int, int i, double& v0, double& v1) {
      v0 = on && i == site ? 1.0 : 0.0;
      v1 = on && i + 1 == site ? 1.0 : 0.0;
    });
#pragma unroll 1
    for (int u = 0; u < s; ++u) {
      auto scale = [&](bool on, int col, int i, double& v0, double& v1) {
        if (!on) return;
        const int at = right ? col + u : col - 1 - u;
        const RowPair e = load_pair(ev + (size_t)at * n + i);
        v0 *= !right && i == site ? xs[at] : e.v0;
        v1 *= !right && i + 1 == site ? xs[at] : e.v1;
      };
      if (right) visit(scale);
      oz_kin_tile(K, z, two_x, two_y);
      if (!right) visit(scale);
    }
    double* W = right ? R : V;
    visit([&](bool on, int col, int i, double& v0, double& v1) {
      if (on) store_pair(W + (size_t)col * n + i, v0, v1);
    });
  }
  __syncthreads();
}

// G <- E diag(d) G diag(rd) E^-1 (the wrap; F the fragments of E, Fi those of E^-1).
template <int LM>
__device__ __noinline__ void oz_wrap(int nx, int ny, int n, const OzKin& F, const OzKin& Fi, double* G, const double* d,
                                     const double* rd) {
  oz_kin_lines(
      nx, ny, n,
      [&](int c, int i, double& v0, double& v1) {
        const RowPair p = load_pair(G + (size_t)c * n + i);
        v0 = (d[i] * p.v0) * rd[c];
        v1 = (d[i + 1] * p.v1) * rd[c];
      },
      [&](double (&z)[2][4], bool two_x, bool two_y, auto) { oz_kin_tile(F, z, two_x, two_y); },
      [&](int c, int i, double v0, double v1) { store_pair(G + (size_t)c * n + i, v0, v1); });
  __syncthreads();
  oz_kin_lines(
      nx, ny, n,
      [&](int r, int i, double& v0, double& v1) {
        v0 = G[(size_t)i * n + r];
        v1 = G[(size_t)(i + 1) * n + r];
      },
      [&](double (&z)[2][4], bool two_x, bool two_y, auto) { oz_kin_tile(Fi, z, two_x, two_y); },
      [&](int r, int i, double v0, double v1) {
        G[(size_t)i * n + r] = v0;
        G[(size_t)(i + 1) * n + r] = v1;
      });
  __syncthreads();
}

}  // namespace hq
