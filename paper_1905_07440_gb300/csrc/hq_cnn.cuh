// Periodic 3D convolutional action (device functions shared by the inner-move and the CNN
// kernels).
//
// Paper: "Global Updates" -- a convolutional network on the whole phonon field stands for
// the weight, so a move of a whole imaginary-time column is cheap to estimate.  Here the
// network is three 3x3x3 cross-correlations with periodic padding on the (x, y, tau) torus,
// 1 -> 16 -> 16 -> 1 channels, ReLU after the first two, and F_cnn(X) = sum of the last
// layer over every point; the input is z = X - x0 with x0 = -g/(M Omega^2).  Tap
// t = 9 (dl + 1) + 3 (dy + 1) + (dx + 1) reads (l + dl, y + dy, x + dx).  Weights are
// bfloat16, arithmetic FP32.
#pragma once
#include "hq_device.cuh"
#include "hq_internal.h"
#include "hq_nn_tc.cuh"

namespace hq {

constexpr int CN_T = 27, CN_C = kCnnC;
constexpr int CN_W1 = 0, CN_B1 = CN_T * CN_C, CN_W2 = CN_B1 + CN_C, CN_B2 = CN_W2 + CN_T * CN_C * CN_C,
              CN_W3 = CN_B2 + CN_C, CN_B3 = CN_W3 + CN_T * CN_C, CN_NP = CN_B3 + 1;
constexpr int CN_WPAD = (CN_NP + 3) & ~3;

// Evaluation and block-move windows on the tensor cores (training: hq_cnn.cu).  Two facts keep the work small:
//
//   * F_cnn sums the last layer over the whole torus, so F_cnn = L N b3 + sum_q wbar . h2(q) with
//     wbar = sum_t W3[t]: the third convolution is a dot product per point.  wbar is kept as two floats.
//     A point's cache is that one number, and a block move recomputes layer 1 within lattice distance 1
//     and layer 2 within 2 of its site (every slice), no outputs beyond.
//   * Layer 2 (27 taps x 16 x 16) runs as m16n8k16 MMAs, 16 points per warp.  Weights are bfloat16
//     already; a layer-1 value is split into three bfloat16 terms (24 bits: exact), once when it is
//     written, and stored as fragments' register pairs: uint4 (hi, mid, lo, 0) per two channels.  The tensor
//     core truncates its sums, which would bias F: a tap's leading products, nearly exact within 24 bits, are
//     added to the FP32 sums with FADDs, and only the other terms, 2^-8 of them, stay in its accumulators.
//
// Every path computes a point through cn_tile in the same order, so a value recomputed in a window
// equals the cached one bit for bit.  (The scalar form took 600 thousand cycles per block move at 8x8,
// L = 40: FP64 input conversions, a window list built by one thread, weights re-read per point.)
struct CnSm {
  const uint2* w2;                       // [27][2][32] fragments of W2
  const float *w1, *b1, *b2, *wh, *wl;   // W1 [27][16], biases, wbar = wh + wl
  float b3;
};

constexpr int CN_FRAGS = CN_T * 2 * 32, CN_FLOATS = CN_T * CN_C + 4 * CN_C + 4;
__host__ __device__ inline size_t cn_smem_bytes() { return sizeof(uint2) * CN_FRAGS + sizeof(float) * CN_FLOATS; }

// all threads; ends with a barrier (kL2: with the fragments of W2)
template <bool kL2 = true>
__device__ inline CnSm cn_setup(const uint16_t* wb, char* mem) {
  uint2* fr = reinterpret_cast<uint2*>(mem);
  float* f = reinterpret_cast<float*>(fr + CN_FRAGS);
  for (int e = threadIdx.x; kL2 && e < CN_FRAGS; e += blockDim.x) {
    const int lane = e & 31, nt = (e >> 5) & 1, tap = e >> 6, g = lane >> 2, t = lane & 3;
    const uint16_t* W = wb + CN_W2 + tap * CN_C * CN_C + 8 * nt + g;
    auto w = [&](int ci) { return (uint32_t)W[ci * CN_C]; };
    fr[e] = make_uint2(w(2 * t) | (w(2 * t + 1) << 16), w(2 * t + 8) | (w(2 * t + 9) << 16));
  }
  float *w1 = f, *b1 = w1 + CN_T * CN_C, *b2 = b1 + CN_C, *wh = b2 + CN_C, *wl = wh + CN_C;
  for (int e = threadIdx.x; e < CN_T * CN_C; e += blockDim.x) w1[e] = bf16_to_float(wb[CN_W1 + e]);
  for (int c = threadIdx.x; c < CN_C; c += blockDim.x) {
    b1[c] = bf16_to_float(wb[CN_B1 + c]);
    b2[c] = bf16_to_float(wb[CN_B2 + c]);
    double s = 0.0;
    for (int t = 0; t < CN_T; ++t) s += (double)bf16_to_float(wb[CN_W3 + t * CN_C + c]);
    wh[c] = (float)s;
    wl[c] = (float)(s - (double)(float)s);
  }
  __syncthreads();
  return CnSm{fr, w1, b1, b2, wh, wl, bf16_to_float(wb[CN_B3])};
}

// Two values as packed bfloat16 pairs hi + mid + lo (24 bits: exact).
__device__ __forceinline__ uint4 cn_split(float a, float b) {
  const uint32_t h = cvt_bf16x2(a, b);
  const float ra = a - __uint_as_float(h << 16), rb = b - __uint_as_float(h & 0xffff0000u);
  const uint32_t m = cvt_bf16x2(ra, rb);
  return make_uint4(h, m, cvt_bf16x2(ra - __uint_as_float(m << 16), rb - __uint_as_float(m & 0xffff0000u)), 0u);
}

__device__ __forceinline__ uint32_t cn_trans8x8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(v));
  return r;
}

__device__ __forceinline__ int cn_wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Channels 8 half .. 8 half + 7 of layer 1 (after ReLU) at (l, x, y) to out[4 half ..]; z(ll, j): input.
template <class Z>
__device__ __forceinline__ void cn_point1(const Dev& d, const CnSm& w, int l, int x, int y, int half, Z z, uint4* out) {
  float a[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) a[c] = w.b1[8 * half + c];
#pragma unroll 1
  for (int dl = -1; dl <= 1; ++dl) {
    const int ll = cn_wrap(l + dl, d.L);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const float v = z(ll, cn_wrap(x + q % 3 - 1, d.nx) + d.nx * cn_wrap(y + q / 3 - 1, d.ny));
      const float* W = w.w1 + (9 * (dl + 1) + q) * CN_C + 8 * half;
#pragma unroll
      for (int c = 0; c < 8; ++c) a[c] = fmaf(v, W[c], a[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) out[4 * half + c] = cn_split(fmaxf(a[2 * c], 0.f), fmaxf(a[2 * c + 1], 0.f));
}

// Lattice window around a site: columns x0 .. x0 + wx - 1 (periodic), rows likewise; all of the lattice in a
// direction shorter than the window.
struct CnBox {
  int x0, y0, wx, wy;
  __device__ __forceinline__ int count() const { return wx * wy; }
  __device__ __forceinline__ int x(const Dev& d, int k) const { return cn_wrap(x0 + k % wx, d.nx); }
  __device__ __forceinline__ int y(const Dev& d, int k) const { return cn_wrap(y0 + k / wx, d.ny); }
};
__device__ __forceinline__ CnBox cn_box(const Dev& d, int i, int radius) {
  const int w = 2 * radius + 1, x = i % d.nx, y = i / d.nx;
  return CnBox{w < d.nx ? cn_wrap(x - radius, d.nx) : 0, w < d.ny ? cn_wrap(y - radius, d.ny) : 0, min(w, d.nx), min(w, d.ny)};
}

// Layer 2 before bias and ReLU for 16 points by one warp: rows g, g + 8 are the points (l, x, y)[2], acc[nt][2h + e]
// channel 8 nt + 2t + e of row g + 8h.  Layer-1 values of sites in `box` come from `win` ([L][box][8]), of the
// others from `cur` ([L][n][8]).
__device__ __forceinline__ void cn_tile_acc(const Dev& d, const CnSm& w, const int (&l)[2], const int (&x)[2],
                                            const int (&y)[2], const uint4* cur, const uint4* win, const CnBox& box,
                                            float (&acc)[2][4]) {
  const int lane = threadIdx.x & 31, t = lane & 3;
  float rest[2][4];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[nt][k] = rest[nt][k] = 0.f;
  // per row: site columns and rows of the three offsets, and their places in the window (-1 outside)
  int xs[2][3], ys[2][3], px[2][3], py[2][3];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      xs[h][o] = cn_wrap(x[h] + o - 1, d.nx);
      ys[h][o] = cn_wrap(y[h] + o - 1, d.ny);
      const int a = cn_wrap(xs[h][o] - box.x0, d.nx), b = cn_wrap(ys[h][o] - box.y0, d.ny);
      px[h][o] = a < box.wx ? a : -1;
      py[h][o] = b < box.wy ? b : -1;
      ys[h][o] *= d.nx;
    }
  const int n1 = box.count();
#pragma unroll 1
  for (int dl = 0; dl < 3; ++dl) {
    const uint4 *c[2], *v[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int ll = cn_wrap(l[h] + dl - 1, d.L);
      c[h] = cur + (size_t)ll * d.n * 8;
      v[h] = win + (size_t)ll * n1 * 8;
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const uint4* p[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int a = px[h][q % 3], b = py[h][q / 3];
        p[h] = (a >= 0 && b >= 0) ? v[h] + (b * box.wx + a) * 8 : c[h] + (ys[h][q / 3] + xs[h][q % 3]) * 8;
      }
      const uint4 a0 = p[0][t], a1 = p[1][t], a2 = p[0][t + 4], a3 = p[1][t + 4];
      const uint32_t hi[4] = {a0.x, a1.x, a2.x, a3.x}, mid[4] = {a0.y, a1.y, a2.y, a3.y}, lo[4] = {a0.z, a1.z, a2.z, a3.z};
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const uint2 b = w.w2[((9 * dl + q) * 2 + nt) * 32 + lane];
        float e[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(e, hi, b);
        mma_bf16(rest[nt], lo, b);
        mma_bf16(rest[nt], mid, b);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[nt][k] += e[k];
      }
    }
  }
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[nt][k] += rest[nt][k];
}

// wbar . h2 of the 16 points; every lane of a quad gets both rows' values.
__device__ __forceinline__ void cn_tile(const Dev& d, const CnSm& w, const int (&l)[2], const int (&x)[2], const int (&y)[2],
                                        const uint4* cur, const uint4* win, const CnBox& box, float (&s)[2]) {
  const int t = threadIdx.x & 3;
  float acc[2][4];
  cn_tile_acc(d, w, l, x, y, cur, win, box, acc);
  s[0] = s[1] = 0.f;
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int ch = 8 * nt + 2 * t + (k & 1);
      const float h2 = fmaxf(acc[nt][k] + w.b2[ch], 0.f);
      s[k >> 1] = fmaf(h2, w.wh[ch], fmaf(h2, w.wl[ch], s[k >> 1]));
    }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    s[h] += __shfl_xor_sync(HQ_FULL, s[h], 1);
    s[h] += __shfl_xor_sync(HQ_FULL, s[h], 2);
  }
}

// F_cnn of one configuration by the whole CTA from the network inputs xf [L][n]; layer 1 goes to h1
// [L][n][8] and every point's wbar . h2 to s2 [L][n].  Returns F in every thread.
__device__ inline double cn_refresh(const Dev& d, const CnSm& w, const float* xf, uint4* h1, float* s2, double* red) {
  const int n = d.n, NL = d.n * d.L, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2;
  for (int e = threadIdx.x; e < 2 * NL; e += HQ_THREADS) {
    const int p = e >> 1, l = p / n, i = p % n;
    cn_point1(d, w, l, i % d.nx, i / d.nx, e & 1, [&](int ll, int j) { return xf[ll * n + j]; }, h1 + (size_t)p * 8);
  }
  __syncthreads();
  const CnBox none{0, 0, 0, 0};
  double part = 0.0;
  for (int base = warp * 16; base < NL; base += HQ_WARPS * 16) {
    int l[2], x[2], y[2];
    float s[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int p = min(base + g + 8 * h, NL - 1), i = p % n;
      l[h] = p / n;
      x[h] = i % d.nx;
      y[h] = i / d.nx;
    }
    cn_tile(d, w, l, x, y, h1, h1, none, s);
    if ((lane & 3) == 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int p = base + g + 8 * h;
        if (p < NL) {
          s2[p] = s[h];
          part += (double)s[h];
        }
      }
    }
  }
  return block_sum(part, red) + (double)NL * (double)w.b3;
}

// F_cnn(X') - F_cnn(X) for X'(i, .) = X(i, .) + dx: z'(l, i) = xsh[l], the other inputs from xf; h1, s2 the caches
// of X; the proposal's layer 1 (radius 1) goes to h1p, its points (radius 2) to s2p.  Called by the
// whole CTA; returns the difference in every thread.
__device__ inline double cn_block_delta(const Dev& d, const CnSm& w, const float* xf, const float* xsh, int i,
                                        const uint4* h1, const float* s2, uint4* h1p, float* s2p, double* red) {
  const int n = d.n, L = d.L, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2;
  const CnBox b1 = cn_box(d, i, 1), b2 = cn_box(d, i, 2);
  const int n1 = b1.count(), n2 = b2.count();
  for (int e = threadIdx.x; e < 2 * n1 * L; e += HQ_THREADS) {
    const int q = e >> 1, l = q / n1, k = q % n1;
    cn_point1(d, w, l, b1.x(d, k), b1.y(d, k), e & 1, [&](int ll, int j) { return j == i ? xsh[ll] : xf[ll * n + j]; },
              h1p + (size_t)q * 8);
  }
  __syncthreads();
  double part = 0.0;
  for (int base = warp * 16; base < n2 * L; base += HQ_WARPS * 16) {
    int l[2], x[2], y[2];
    float s[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = min(base + g + 8 * h, n2 * L - 1), k = q % n2;
      l[h] = q / n2;
      x[h] = b2.x(d, k);
      y[h] = b2.y(d, k);
    }
    cn_tile(d, w, l, x, y, h1, h1p, b1, s);
    if ((lane & 3) == 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = base + g + 8 * h;
        if (q < n2 * L) {
          s2p[q] = s[h];
          part += (double)s[h] - (double)s2[l[h] * n + x[h] + d.nx * y[h]];
        }
      }
    }
  }
  return block_sum(part, red);
}

// Accepted block move: the window values become the caches.  Ends with a barrier.
__device__ inline void cn_block_commit(const Dev& d, int i, uint4* h1, float* s2, const uint4* h1p, const float* s2p) {
  const CnBox b1 = cn_box(d, i, 1), b2 = cn_box(d, i, 2);
  const int n = d.n, L = d.L, n1 = b1.count(), n2 = b2.count();
  for (int e = threadIdx.x; e < n1 * L * 8; e += HQ_THREADS) {
    const int q = e >> 3, l = q / n1, k = q % n1;
    h1[((size_t)l * n + b1.x(d, k) + d.nx * b1.y(d, k)) * 8 + (e & 7)] = h1p[e];
  }
  for (int q = threadIdx.x; q < n2 * L; q += HQ_THREADS) {
    const int l = q / n2, k = q % n2;
    s2[l * n + b2.x(d, k) + d.nx * b2.y(d, k)] = s2p[q];
  }
  __syncthreads();
}

}  // namespace hq
