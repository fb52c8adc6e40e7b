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
#include <type_traits>
#include "hq_device.cuh"
#include "hq_internal.h"
#include "hq_nn_tc.cuh"

namespace hq {

constexpr int CN_T = 27, CN_C = kCnnC;
constexpr int CN_W1 = 0, CN_B1 = CN_T * CN_C, CN_W2 = CN_B1 + CN_C, CN_B2 = CN_W2 + CN_T * CN_C * CN_C,
              CN_W3 = CN_B2 + CN_C, CN_B3 = CN_W3 + CN_T * CN_C, CN_NP = CN_B3 + 1;
constexpr int CN_WPAD = (CN_NP + 3) & ~3;

// F_cnn sums the last layer over the whole torus, so F_cnn = L N b3 + sum_q wbar . h2(q) with wbar = sum_t W3[t]: the
// third convolution is a dot product per point (wbar is kept as two floats).  A point's cache is that one number, and a
// block move recomputes layer 1 within lattice distance 1 and layer 2 within 2 of its site (every slice).
//
// Layer 2 (27 taps x 16 x 16) runs in FP32 FMAs, which round to nearest.  On the tensor cores, with activations in three
// bfloat16 terms, the truncation of the leading products' sums gives every point an error that depends on the weights,
// and F, a sum over all points, keeps it: 16x16, L = 160, error of F 3e-9 of the sum of its terms' sizes, 6e-10 with FMAs.
// (With MMAs a learned step of 8x8, L = 40, 64 chains takes 8.6 ms, with this 9.2.)  FMAs come two at a time
// (fma.rn.f32x2); eight channels of up to four points belong to a thread, the other eight to its neighbour, because
// operands reach the registers at 128 bytes a clock: with two points per thread the moves take half as long again.
// Every path computes a point through cn_points in the same order, so a value recomputed in a window equals the cached
// one bit for bit.
struct CnSm {
  const float4* w2;                      // [27][16][4] W2, rows of 16 channels
  const float *w1, *b1, *b2, *wh, *wl;   // W1 [27][16], biases, wbar = wh + wl
  float b3;
};

constexpr int CN_W2F = CN_T * CN_C * CN_C, CN_FLOATS = CN_T * CN_C + 4 * CN_C + 4;
__host__ __device__ inline size_t cn_smem_bytes(bool layer2) { return sizeof(float) * (CN_FLOATS + (layer2 ? CN_W2F : 0)); }

// all threads; ends with a barrier (kL2: with W2)
template <bool kL2 = true>
__device__ inline CnSm cn_setup(const uint16_t* wb, char* mem) {
  float *w1 = reinterpret_cast<float*>(mem), *w2 = w1 + CN_FLOATS, *b1 = w1 + CN_T * CN_C, *b2 = b1 + CN_C, *wh = b2 + CN_C, *wl = wh + CN_C;
  for (int e = threadIdx.x; kL2 && e < CN_W2F; e += blockDim.x) w2[e] = bf16_to_float(wb[CN_W2 + e]);
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
  return CnSm{reinterpret_cast<const float4*>(w2), w1, b1, b2, wh, wl, bf16_to_float(wb[CN_B3])};
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

// Channels 8 half .. 8 half + 7 of layer 1 (after ReLU) at (l, x, y) in a; z(ll, j): input.
template <class Z>
__device__ __forceinline__ void cn_point1(const Dev& d, const CnSm& w, int l, int x, int y, int half, Z z, float (&a)[8]) {
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
  for (int c = 0; c < 8; ++c) a[c] = fmaxf(a[c], 0.f);
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

// Layer 1 is kept by channel quads: channels 4q .. 4q + 3 of point p = l n + i at h1[q NL + p].
__device__ __forceinline__ void cn_store1(float4* h1, int NL, int p, int half, const float (&a)[8]) {
  h1[(2 * half) * NL + p] = make_float4(a[0], a[1], a[2], a[3]);
  h1[(2 * half + 1) * NL + p] = make_float4(a[4], a[5], a[6], a[7]);
}

// (z, z), and c += a b for pairs of floats
__device__ __forceinline__ unsigned long long cn_both(float z) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(z));
  return r;
}
__device__ __forceinline__ void cn_fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// wbar . h2 at the points (l, x, y)[.] by a pair of threads (channels 0 .. 7 in the even one), both of which get them.
template <int P>
__device__ __forceinline__ void cn_points(const Dev& d, const CnSm& w, const int (&l)[P], const int (&x)[P], const int (&y)[P],
                                          const float4* h1, float (&s)[P]) {
  const int half = threadIdx.x & 1, NL = d.n * d.L;
  unsigned long long acc[P][4];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[p][c] = 0ull;
  const float4* W = w.w2 + 2 * half;
#pragma unroll 1
  for (int dl = -1; dl <= 1; ++dl)
#pragma unroll 1
    for (int dy = -1; dy <= 1; ++dy) {
      int row[P];
#pragma unroll
      for (int p = 0; p < P; ++p) row[p] = cn_wrap(l[p] + dl, d.L) * d.n + cn_wrap(y[p] + dy, d.ny) * d.nx;
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx, W += 4 * CN_C) {
        const float4* h[P];
#pragma unroll
        for (int p = 0; p < P; ++p) h[p] = h1 + row[p] + cn_wrap(x[p] + dx, d.nx);
#pragma unroll
        for (int q = 0; q < CN_C / 4; ++q) {
          float4 v[P];
#pragma unroll
          for (int p = 0; p < P; ++p) v[p] = h[p][q * NL];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(W + 4 * (4 * q + e)), g = *reinterpret_cast<const ulonglong2*>(W + 4 * (4 * q + e) + 1);
#pragma unroll
            for (int p = 0; p < P; ++p) {
              const float z = e == 0 ? v[p].x : e == 1 ? v[p].y : e == 2 ? v[p].z : v[p].w;
              const unsigned long long zz = cn_both(z);
              cn_fma2(acc[p][0], zz, f.x);
              cn_fma2(acc[p][1], zz, f.y);
              cn_fma2(acc[p][2], zz, g.x);
              cn_fma2(acc[p][3], zz, g.y);
            }
          }
        }
      }
    }
#pragma unroll
  for (int p = 0; p < P; ++p) {
    float sum = 0.f, low = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int ch = 8 * half + c;
      const float h2 = fmaxf(__uint_as_float((uint32_t)(acc[p][c >> 1] >> (32 * (c & 1)))) + w.b2[ch], 0.f);
      sum = fmaf(h2, w.wh[ch], sum);
      low = fmaf(h2, w.wl[ch], low);
    }
    s[p] = sum + low;
    s[p] += __shfl_xor_sync(HQ_FULL, s[p], 1);
  }
}

// The points at(q, l, x, y), q < count, by the whole CTA: put(q, l, x, y, wbar . h2) is called once for each.  Four points per
// pair of threads, fewer in a last round that they would leave half empty.
template <class AT, class PUT>
__device__ __forceinline__ void cn_layer2(const Dev& d, const CnSm& w, const float4* h1, int count, AT at, PUT put) {
  constexpr int kPairs = HQ_THREADS / 2;
  auto round = [&](int q0, auto points) {
    constexpr int P = decltype(points)::value;
    int l[P], x[P], y[P];
    float s[P];
#pragma unroll
    for (int p = 0; p < P; ++p) at(min(q0 + p * kPairs + (int)(threadIdx.x >> 1), count - 1), l[p], x[p], y[p]);
    cn_points<P>(d, w, l, x, y, h1, s);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const int q = q0 + p * kPairs + (int)(threadIdx.x >> 1);
      if (q < count && !(threadIdx.x & 1)) put(q, l[p], x[p], y[p], s[p]);
    }
  };
  int q0 = 0;
#pragma unroll 1
  for (; count - q0 > 2 * kPairs; q0 += 4 * kPairs) round(q0, std::integral_constant<int, 4>());
  if (q0 < count) round(q0, std::integral_constant<int, 2>());
}

// F_cnn of one configuration by the whole CTA from the network inputs xf [L][n]; layer 1 goes to h1
// [4][L n] and every point's wbar . h2 to s2 [L][n].  Returns F in every thread.
static __device__ __noinline__ double cn_refresh(const Dev& d, const CnSm& w, const float* xf, float4* h1, float* s2, double* red) {
  const int n = d.n, NL = d.n * d.L;
  for (int e = threadIdx.x; e < 2 * NL; e += HQ_THREADS) {
    const int p = e >> 1, l = p / n, i = p % n;
    float a[8];
    cn_point1(d, w, l, i % d.nx, i / d.nx, e & 1, [&](int ll, int j) { return xf[ll * n + j]; }, a);
    cn_store1(h1, NL, p, e & 1, a);
  }
  __syncthreads();
  double part = 0.0;
  cn_layer2(
      d, w, h1, NL,
      [&](int q, int& l, int& x, int& y) {
        const int i = q % n;
        l = q / n;
        x = i % d.nx;
        y = i / d.nx;
      },
      [&](int q, int, int, int, float s) {
        s2[q] = s;
        part += (double)s;
      });
  return block_sum(part, red) + (double)NL * (double)w.b3;
}

// F_cnn(X') - F_cnn(X) for X'(i, .) = X(i, .) + dx: z'(l, i) = xsh[l], the other inputs from xf; h1, s2 the caches
// of X.  Layer 1 of the proposal (radius 1) takes the place of the cached values, which go to h1p [L][box][4]; its points
// (radius 2) go to s2p.  cn_block_end accepts or takes back.  Called by the whole CTA; returns the difference in
// every thread.
static __device__ __noinline__ double cn_block_delta(const Dev& d, const CnSm& w, const float* xf, const float* xsh, int i,
                                        float4* h1, const float* s2, float4* h1p, float* s2p, double* red) {
  const int n = d.n, L = d.L, NL = n * L;
  const CnBox b1 = cn_box(d, i, 1), b2 = cn_box(d, i, 2);
  const int n1 = b1.count(), n2 = b2.count();
  for (int e = threadIdx.x; e < 2 * n1 * L; e += HQ_THREADS) {
    const int q = e >> 1, half = e & 1, l = q / n1, k = q % n1, x = b1.x(d, k), y = b1.y(d, k), p = l * n + x + d.nx * y;
    float a[8];
    cn_point1(d, w, l, x, y, half, [&](int ll, int j) { return j == i ? xsh[ll] : xf[ll * n + j]; }, a);
    h1p[4 * q + 2 * half] = h1[(2 * half) * NL + p];
    h1p[4 * q + 2 * half + 1] = h1[(2 * half + 1) * NL + p];
    cn_store1(h1, NL, p, half, a);
  }
  __syncthreads();
  double part = 0.0;
  cn_layer2(
      d, w, h1, n2 * L,
      [&](int q, int& l, int& x, int& y) {
        const int k = q % n2;
        l = q / n2;
        x = b2.x(d, k);
        y = b2.y(d, k);
      },
      [&](int q, int l, int x, int y, float s) {
        s2p[q] = s;
        part += (double)s - (double)s2[l * n + x + d.nx * y];
      });
  return block_sum(part, red);
}

// After cn_block_delta (all reads of h1 done): the proposal's points become the cache, or its layer 1 is taken back.  Ends
// with a barrier.
static __device__ __noinline__ void cn_block_end(const Dev& d, int i, bool accept, float4* h1, float* s2, const float4* h1p, const float* s2p) {
  const int n = d.n, L = d.L;
  const CnBox b = cn_box(d, i, accept ? 2 : 1);
  const int nb = b.count();
  if (accept) {
    for (int q = threadIdx.x; q < nb * L; q += HQ_THREADS) {
      const int l = q / nb, k = q % nb;
      s2[l * n + b.x(d, k) + d.nx * b.y(d, k)] = s2p[q];
    }
  } else {
    for (int e = threadIdx.x; e < 4 * nb * L; e += HQ_THREADS) {
      const int q = e >> 2, l = q / nb, k = q % nb;
      h1[(e & 3) * n * L + l * n + b.x(d, k) + d.nx * b.y(d, k)] = h1p[e];
    }
  }
  __syncthreads();
}

}  // namespace hq
