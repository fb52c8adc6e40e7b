// Convolutional action for block moves: evaluation and training kernels.
//
// F_cnn(X) = sum over the (x, y, tau) torus of a three-layer periodic 3x3x3 network (see
// hq_cnn.cuh).  Training fits F_cnn(X_a) to log|det M(X_a)| minus the sample mean by mean
// squared error, as for the patch network.  Because F_cnn is a plain sum of the last layer,
// dF/d(layer-2 output at any point) is the same vector sum_t W3[t][.], so the error behind layer 2
// is a mask times a constant: both contractions with it (the gradient of W2 over points, the error of
// layer 1 over channels) are MMAs with an exact 0/1 operand; layer 2 itself runs in FP32 FMAs.  Every sample is shared out over
// several CTAs; sums run in a fixed order and the per-CTA partials are added in a fixed order by the
// Adam kernel, so training is deterministic.
#include <algorithm>

#include "hq_cnn.cuh"
#include "../../include/holstein_dqmc.h"

namespace hq {

static_assert(CN_NP == HQ_CNN_PARAMS, "parameter count");

// ------------------------------------------------------------------------ evaluation
// F_cnn of every chain (grid = chains).  The chain's caches and its input table (the patch network's too) become those of
// Xall, so this is called on the current fields only.
__global__ void __launch_bounds__(HQ_THREADS, 2) cnn_eval_kernel(const __grid_constant__ Dev d, CnnState cn, const double* Xall, double* Fout,
                                                                 double x0) {
  extern __shared__ __align__(16) char craw[];
  __shared__ double red[HQ_WARPS];
  const int c = blockIdx.x, NL = d.n * d.L;
  const double* X = Xall + (size_t)c * NL;
  float* xf = cn.xf + (size_t)c * NL;
  for (int k = threadIdx.x; k < NL; k += HQ_THREADS) xf[k] = (float)(X[k] - x0);
  const CnSm w = cn_setup(cn.wbf, craw);  // (ends with a barrier)
  const double F = cn_refresh(d, w, xf, cn.h1c + (size_t)c * NL * 4, cn.s2c + (size_t)c * NL, red);
  if (threadIdx.x == 0) Fout[c] = F;
}

// ------------------------------------------------------------------------ training
// Scratch of one sample of a round (samples trained at a time), in cn.tr: layer-1 activations (split), network
// inputs, layer-2 masks (a bit per channel), per-part channel sums of layer 2 and shares of F.
struct CnSample {
  uint4* h1;       // [L N][8]
  float* z;        // [L N]
  uint16_t* mask;  // [L N]
  float* hs;       // [kCnnParts][16]
  double* f;       // [kCnnParts]
};
__host__ __device__ inline size_t cn_sample_bytes(size_t NL) {
  return NL * 128 + ((NL * 4 + 15) & ~(size_t)15) + ((NL * 2 + 15) & ~(size_t)15) + kCnnParts * (16 * 4 + 8);
}
size_t cnn_sample_bytes(size_t NL) { return (cn_sample_bytes(NL) + 255) & ~(size_t)255; }

__device__ __forceinline__ CnSample cn_sample(const CnnState& cn, size_t NL, int a) {
  char* p = cn.tr + (size_t)a * ((cn_sample_bytes(NL) + 255) & ~(size_t)255);
  CnSample s;
  s.h1 = (uint4*)p; p += NL * 128;
  s.z = (float*)p; p += (NL * 4 + 15) & ~(size_t)15;
  s.mask = (uint16_t*)p; p += (NL * 2 + 15) & ~(size_t)15;
  s.f = (double*)p; p += kCnnParts * 8;
  s.hs = (float*)p;
  return s;
}

// Network inputs of the round's samples.
__global__ void cnn_inputs_kernel(Dev d, CnnState cn, const double* Xs, const int* idx, double x0) {
  const int NL = d.n * d.L, a = blockIdx.y;
  const CnSample s = cn_sample(cn, NL, a);
  const double* X = Xs + (size_t)idx[a] * NL;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < NL; k += gridDim.x * blockDim.x) s.z[k] = (float)(X[k] - x0);
}

__global__ void __launch_bounds__(HQ_THREADS) cnn_layer1_kernel(Dev d, CnnState cn) {
  extern __shared__ __align__(16) char craw[];
  const CnSm w = cn_setup<false>(cn.wbf, craw);
  const int n = d.n, NL = d.n * d.L;
  const CnSample s = cn_sample(cn, NL, blockIdx.y);
  for (int e = blockIdx.x * HQ_THREADS + threadIdx.x; e < 2 * NL; e += gridDim.x * HQ_THREADS) {
    const int p = e >> 1, l = p / n, i = p % n;
    float a[8];
    cn_point1(d, w, l, i % d.nx, i / d.nx, e & 1, [&](int ll, int j) { return s.z[ll * n + j]; }, a);
#pragma unroll
    for (int c = 0; c < 4; ++c) s.h1[(size_t)p * 8 + 4 * (e & 1) + c] = cn_split(a[2 * c], a[2 * c + 1]);
  }
}

// the points of part `part` of `parts`: whole tiles of 16
__device__ __forceinline__ void cn_part(int NL, int part, int parts, int& p0, int& p1) {
  const int tiles = (NL + 15) >> 4;
  p0 = (int)((long long)tiles * part / parts) * 16;
  p1 = min((int)((long long)tiles * (part + 1) / parts) * 16, NL);
}

// Layer 2 of the round's samples: masks, channel sums and shares of F (grid: parts x samples), a point per thread in
// FP32.  F enters the gradient as F - y, and the tensor core's truncation biases F by about 2e-8 of itself (three
// terms, leading products apart), which the residuals' cancellation made 5e-7 of a gradient; FMAs round to nearest.
// (With MMAs the gradient of 32 samples of 8x8, L = 40 took 196 us, with this 303, at the start 1713.)
__global__ void __launch_bounds__(HQ_THREADS, 2) cnn_layer2_kernel(Dev d, CnnState cn) {
  extern __shared__ __align__(16) char craw[];
  __shared__ double red[HQ_WARPS];
  __shared__ float ch[HQ_WARPS][CN_C];
  const CnSm w = cn_setup(cn.wbf, craw);  // (ends with a barrier)
  const int n = d.n, NL = d.n * d.L, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CnSample s = cn_sample(cn, NL, blockIdx.y);
  int p0, p1;
  cn_part(NL, blockIdx.x, gridDim.x, p0, p1);
  float hs[CN_C];
#pragma unroll
  for (int c = 0; c < CN_C; ++c) hs[c] = 0.f;
  double part = 0.0;
  for (int p = p0 + threadIdx.x; p < p1; p += HQ_THREADS) {
    const int l = p / n, i = p % n, x = i % d.nx, y = i / d.nx;
    float acc[CN_C];
#pragma unroll
    for (int c = 0; c < CN_C; ++c) acc[c] = 0.f;
#pragma unroll 1
    for (int tap = 0; tap < CN_T; ++tap) {
      const int j = cn_wrap(l + tap / 9 - 1, d.L) * n + cn_wrap(x + tap % 3 - 1, d.nx) + d.nx * cn_wrap(y + (tap / 3) % 3 - 1, d.ny);
      const uint4* h = s.h1 + (size_t)j * 8;
      const float4* W = w.w2 + tap * CN_C * (CN_C / 4);
#pragma unroll
      for (int k = 0; k < CN_C / 2; ++k) {
        const uint4 u = h[k];
        const float v[2] = {__uint_as_float(u.x << 16) + (__uint_as_float(u.y << 16) + __uint_as_float(u.z << 16)),
                            __uint_as_float(u.x & 0xffff0000u) +
                                (__uint_as_float(u.y & 0xffff0000u) + __uint_as_float(u.z & 0xffff0000u))};
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int q = 0; q < CN_C / 4; ++q) {
            const float4 f = W[(2 * k + e) * (CN_C / 4) + q];
            acc[4 * q] = fmaf(v[e], f.x, acc[4 * q]);
            acc[4 * q + 1] = fmaf(v[e], f.y, acc[4 * q + 1]);
            acc[4 * q + 2] = fmaf(v[e], f.z, acc[4 * q + 2]);
            acc[4 * q + 3] = fmaf(v[e], f.w, acc[4 * q + 3]);
          }
      }
    }
    uint32_t bits = 0;
    float sum = 0.f, low = 0.f;
#pragma unroll
    for (int c = 0; c < CN_C; ++c) {
      const float a = acc[c] + w.b2[c], h2 = fmaxf(a, 0.f);
      if (a > 0.f) bits |= 1u << c;
      hs[c] += h2;
      sum = fmaf(h2, w.wh[c], sum);
      low = fmaf(h2, w.wl[c], low);
    }
    s.mask[p] = (uint16_t)bits;
    part += (double)(sum + low);
  }
#pragma unroll
  for (int c = 0; c < CN_C; ++c) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) hs[c] += __shfl_xor_sync(HQ_FULL, hs[c], o);
    if (lane == 0) ch[warp][c] = hs[c];
  }
  part = block_sum(part, red);  // (its barriers cover ch)
  if (threadIdx.x < CN_C) {
    float a = 0.f;
    for (int k = 0; k < HQ_WARPS; ++k) a += ch[k][threadIdx.x];
    s.hs[blockIdx.x * CN_C + threadIdx.x] = a;
  }
  if (threadIdx.x == 0) s.f[blockIdx.x] = part + (double)(p1 - p0) * (double)w.b3;
}

// Backward pass of the round's samples (grid: parts x samples).  With m(p)[co] the masks, s = dL/dF and
// w = sum_t W3[t]:  gW2[t][ci][co] = s w[co] sum_p h1(p + t)[ci] m(p)[co];
// d1(q)[ci] = [h1(q)[ci] > 0] s sum_t sum_co (W2[t][ci][co] w[co]) m(q - t)[co];  gW1[t][co] = sum_p d1(p)[co] z(p + t).
// Blocks of 128 points share a table of their 27 neighbours (without it, integer divisions and the latency of
// the loads behind them were most of 169 us for 32 samples of 8x8, L = 40).  A warp owns taps warp, warp + 8, ... of
// gW2: per 16 points the masks are the left operand of all of them and the layer-1 fragments, transposed in registers,
// the right ones.  d1 goes through shared memory to gW1, whose (tap, channel) entries are owned by threads.
// Partials are written in the first round and added to later.
constexpr int kCnBlk = 128, kCnLd = kCnBlk + 4;
constexpr int CN_WT = CN_T * 3 * 2 * 32;  // fragments of W2 w, three terms
constexpr int kCnOwn = (CN_T + HQ_WARPS - 1) / HQ_WARPS;

__host__ __device__ inline size_t cn_back_smem_bytes() {
  return cn_smem_bytes(false) + sizeof(uint2) * CN_WT + sizeof(float) * kCnLd * (CN_T + CN_C) + sizeof(int) * kCnBlk * CN_T;
}

__global__ void __launch_bounds__(HQ_THREADS) cnn_backward_kernel(Dev d, CnnState cn, const double* ys, const int* idx,
                                                                  int B, int parts2, int first, double* Fb,
                                                                  float* partials) {
  extern __shared__ __align__(16) char craw[];
  __shared__ float sw[2][CN_C];
  __shared__ int cnt[CN_C];
  const CnSm w = cn_setup<false>(cn.wbf, craw);
  uint2* wt = reinterpret_cast<uint2*>(craw + cn_smem_bytes(false));
  float* zn = reinterpret_cast<float*>(wt + CN_WT);  // [27][kCnLd] inputs at p + t
  float* ds = zn + kCnLd * CN_T;                     // [16][kCnLd] d1 / s
  int* nb = reinterpret_cast<int*>(ds + kCnLd * CN_C);  // [27][kCnBlk] places of p + t
  const int n = d.n, L = d.L, NL = n * L, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int a = blockIdx.y, parts = gridDim.x;
  const CnSample s = cn_sample(cn, NL, a);
  int p0, p1;
  cn_part(NL, blockIdx.x, parts, p0, p1);
  double F = 0.0;
  for (int k = 0; k < parts2; ++k) F += s.f[k];
  if (tid == 0 && blockIdx.x == 0) Fb[a] = F;
  // s and s w[co] as two floats, so that a gradient entry is rounded once
  const double sd = 2.0 * (F - ys[idx[a]]) / B;
  const float sg = (float)sd, sl = (float)(sd - (double)sg);
  auto scaled = [&](float v) { return fmaf(sg, v, sl * v); };
  if (tid < CN_C) {
    const double v = sd * ((double)w.wh[tid] + (double)w.wl[tid]);
    sw[0][tid] = (float)v;
    sw[1][tid] = (float)(v - (double)(float)v);
    cnt[tid] = 0;
  }
  // right fragments of (W2[t] w)^T: k = co, column ci
  for (int e = tid; e < CN_T * 2 * 32; e += HQ_THREADS) {
    const int ln = e & 31, nt = (e >> 5) & 1, tap = e >> 6, gg = ln >> 2, tt = ln & 3, ci = 8 * nt + gg;
    auto v = [&](int co) { return bf16_to_float(cn.wbf[CN_W2 + tap * CN_C * CN_C + ci * CN_C + co]) * (w.wh[co] + w.wl[co]); };
    const uint4 x = cn_split(v(2 * tt), v(2 * tt + 1)), y = cn_split(v(2 * tt + 8), v(2 * tt + 9));
    wt[((tap * 3 + 0) * 2 + nt) * 32 + ln] = make_uint2(x.x, y.x);
    wt[((tap * 3 + 1) * 2 + nt) * 32 + ln] = make_uint2(x.y, y.y);
    wt[((tap * 3 + 2) * 2 + nt) * 32 + ln] = make_uint2(x.z, y.z);
  }
  // channels c, c + 1 of a mask, and channel c of two masks, as bfloat16 pairs of 0 and 1
  auto cols = [](uint32_t m, int c) { return ((m >> c) & 1u) * 0x3f80u | ((m >> (c + 1)) & 1u) * 0x3f800000u; };
  auto pair = [](uint32_t m0, uint32_t m1, int c) { return ((m0 >> c) & 1u) * 0x3f80u | ((m1 >> c) & 1u) * 0x3f800000u; };
  float acc2[kCnOwn][2][4], low2[kCnOwn][2][4], rest2[kCnOwn][2][4];
#pragma unroll
  for (int o = 0; o < kCnOwn; ++o)
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc2[o][nt][k] = low2[o][nt][k] = rest2[o][nt][k] = 0.f;
  float g1[2] = {0.f, 0.f}, gb1 = 0.f;
  int cnt2 = 0;
#pragma unroll 1
  for (int b0 = p0; b0 < p1; b0 += kCnBlk) {
    __syncthreads();
    {
      const int p = min(b0 + (tid & (kCnBlk - 1)), NL - 1), l = p / n, i = p % n, x = i % d.nx, y = i / d.nx;
      const int t0 = tid < kCnBlk ? 0 : 14, t1 = tid < kCnBlk ? 14 : CN_T;
      for (int tap = t0; tap < t1; ++tap)
        nb[tap * kCnBlk + (tid & (kCnBlk - 1))] = cn_wrap(l + tap / 9 - 1, L) * n + cn_wrap(x + tap % 3 - 1, d.nx) +
                                                  d.nx * cn_wrap(y + (tap / 3) % 3 - 1, d.ny);
    }
    __syncthreads();
#pragma unroll 4
    for (int e = tid; e < CN_T * kCnBlk; e += HQ_THREADS) zn[(e / kCnBlk) * kCnLd + e % kCnBlk] = s.z[nb[e]];
    {  // d1 / s of the warp's 16 points
      const int pt = warp * 16 + g, base = b0 + warp * 16;
      float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, rest[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
      if (base < p1) {
#pragma unroll 9
        for (int tap = 0; tap < CN_T; ++tap) {
          const int* q = nb + (CN_T - 1 - tap) * kCnBlk + pt;  // p - t
          const uint32_t m0 = s.mask[q[0]], m1 = s.mask[q[8]];
          const uint32_t A[4] = {cols(m0, 2 * t), cols(m1, 2 * t), cols(m0, 2 * t + 8), cols(m1, 2 * t + 8)};
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            float e[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(e, A, wt[((tap * 3 + 0) * 2 + nt) * 32 + lane]);
            mma_bf16(rest[nt], A, wt[((tap * 3 + 2) * 2 + nt) * 32 + lane]);
            mma_bf16(rest[nt], A, wt[((tap * 3 + 1) * 2 + nt) * 32 + lane]);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[nt][k] += e[k];
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool on = base + g + 8 * h < p1;
        const uint4* h1 = s.h1 + (size_t)min(base + g + 8 * h, NL - 1) * 8;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const uint32_t hi = h1[4 * nt + t].x;  // h1 > 0 where its leading term is not zero
          float* o = ds + (8 * nt + 2 * t) * kCnLd + pt + 8 * h;
          o[0] = on && (hi & 0x7fffu) ? acc[nt][2 * h] + rest[nt][2 * h] : 0.f;
          o[kCnLd] = on && (hi & 0x7fff0000u) ? acc[nt][2 * h + 1] + rest[nt][2 * h + 1] : 0.f;
        }
      }
    }
    if (tid < kCnBlk) {
      const uint32_t m = b0 + tid < p1 ? s.mask[b0 + tid] : 0u;
#pragma unroll
      for (int c = 0; c < CN_C; ++c) {
        const int k = __popc(__ballot_sync(HQ_FULL, (m >> c) & 1u));
        if (lane == c) cnt2 += k;
      }
    }
    // gW2
    const int np = min(kCnBlk, p1 - b0);
#pragma unroll 1
    for (int q = 0; q < np; q += 16) {
      uint32_t m[4];  // masks of points 2t, 2t + 1, 2t + 8, 2t + 9 (none beyond the part)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int p = b0 + q + 2 * t + (k & 1) + 8 * (k >> 1);
        m[k] = p < p1 ? s.mask[p] : 0u;
      }
      const uint32_t A[4] = {pair(m[0], m[1], g), pair(m[0], m[1], g + 8), pair(m[2], m[3], g), pair(m[2], m[3], g + 8)};
#pragma unroll
      for (int o = 0; o < kCnOwn; ++o) {
        const int tap = warp + HQ_WARPS * o;
        if (tap < CN_T) {
          const uint4* h0 = s.h1 + (size_t)nb[tap * kCnBlk + q + g] * 8;
          const uint4* h1 = s.h1 + (size_t)nb[tap * kCnBlk + q + g + 8] * 8;
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            const uint4 u = h0[4 * nt + t], v = h1[4 * nt + t];
            // the leading terms' sum is nearly exact and is added with its rounding error kept; the other terms,
            // 2^-8 of it, stay in the tensor core's accumulators
            float e[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(e, A, make_uint2(cn_trans8x8(u.x), cn_trans8x8(v.x)));
            mma_bf16(rest2[o][nt], A, make_uint2(cn_trans8x8(u.z), cn_trans8x8(v.z)));
            mma_bf16(rest2[o][nt], A, make_uint2(cn_trans8x8(u.y), cn_trans8x8(v.y)));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float x = acc2[o][nt][k], sum = x + e[k];  // neither is negative
              low2[o][nt][k] += fminf(x, e[k]) - (sum - fmaxf(x, e[k]));
              acc2[o][nt][k] = sum;
            }
          }
        }
      }
    }
    __syncthreads();
    // gW1, gb1
    const int n4 = (np + 3) >> 2;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q = tid + u * HQ_THREADS;
      if (q < CN_T * CN_C) {
        const float4* zt = reinterpret_cast<const float4*>(zn + (q / CN_C) * kCnLd);
        const float4* dd = reinterpret_cast<const float4*>(ds + (q % CN_C) * kCnLd);
        float acc = 0.f;
#pragma unroll 4
        for (int k = 0; k < n4; ++k) {
          const float4 x = zt[k], y = dd[k];
          acc = fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, fmaf(x.x, y.x, acc))));
        }
        g1[u] += acc;
      }
    }
    if (tid >= 176 && tid < 192) {
      const float4* dd = reinterpret_cast<const float4*>(ds + (tid - 176) * kCnLd);
      float acc = 0.f;
#pragma unroll 4
      for (int k = 0; k < n4; ++k) {
        const float4 y = dd[k];
        acc += (y.x + y.y) + (y.z + y.w);
      }
      gb1 += acc;
    }
  }
  if (tid < kCnBlk && lane < CN_C) atomicAdd(&cnt[lane], cnt2);  // integers: any order
  __syncthreads();
  float* out = partials + ((size_t)a * parts + blockIdx.x) * CN_WPAD;
  auto put = [&](int k, float v) { out[k] = first ? v : out[k] + v; };
  // rows co = g, g + 8; columns ci = 8 nt + 2t, + 1
#pragma unroll
  for (int o = 0; o < kCnOwn; ++o) {
    const int tap = warp + HQ_WARPS * o;
    if (tap < CN_T)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int co = g + 8 * (k >> 1), ci = 8 * nt + 2 * t + (k & 1);
          const float v = acc2[o][nt][k], r = low2[o][nt][k] + rest2[o][nt][k];
          put(CN_W2 + (tap * CN_C + ci) * CN_C + co, fmaf(sw[0][co], v, fmaf(sw[0][co], r, sw[1][co] * v)));
        }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (tid + u * HQ_THREADS < CN_T * CN_C) put(CN_W1 + tid + u * HQ_THREADS, scaled(g1[u]));
  if (tid >= 176 && tid < 192) put(CN_B1 + tid - 176, scaled(gb1));
  if (tid >= 192 && tid < 208) put(CN_B2 + tid - 192, fmaf(sw[0][tid - 192], (float)cnt[tid - 192], sw[1][tid - 192] * (float)cnt[tid - 192]));
  if (tid < CN_C) {
    float hs = 0.f;
    for (int k = blockIdx.x; k < parts2; k += parts) hs += s.hs[k * CN_C + tid];
    const float v = scaled(hs);
    for (int k = 0; k < CN_T; ++k) put(CN_W3 + k * CN_C + tid, v);
  } else if (tid == CN_C) {
    put(CN_B3, scaled((float)(p1 - p0)));
  }
}

// Sum of the per-CTA partials (fixed order) into grad; with lr > 0 an Adam step on the FP32
// master weights and a fresh bfloat16 copy.
__global__ void cnn_adam_kernel(CnnState cn, const float* partials, int nparts, float lr, int t_step) {
  const int k = blockIdx.x * kSumParams + threadIdx.x % kSumParams;
  const float g = sum_partials(partials, nparts, CN_WPAD, k < CN_NP ? k : CN_NP - 1);
  if (k >= CN_NP || threadIdx.x >= kSumParams) return;
  cn.grad[k] = g;
  if (lr > 0.f) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float m = b1 * cn.adam_m[k] + (1.f - b1) * g;
    const float v = b2 * cn.adam_v[k] + (1.f - b2) * g * g;
    cn.adam_m[k] = m;
    cn.adam_v[k] = v;
    const float mh = m / (1.f - powf(b1, (float)t_step)), vh = v / (1.f - powf(b2, (float)t_step));
    const float w = cn.master[k] - lr * mh / (sqrtf(vh) + eps);
    cn.master[k] = w;
    cn.wbf[k] = float_to_bf16(w);
  }
}

__global__ void cnn_set_kernel(CnnState cn, const float* src) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < CN_NP) {
    cn.master[k] = src[k];
    cn.wbf[k] = float_to_bf16(src[k]);
    cn.adam_m[k] = 0.f;
    cn.adam_v[k] = 0.f;
  }
}

__global__ void cnn_loss_kernel(CnnState cn, const double* ys, const int* idx, int B, double scale, double* loss) {
  squared_error(cn.Fb, ys, idx, B, scale, loss);
}

// ------------------------------------------------------------------------ launchers
static double mean_field_shift(const Dev& d) { return -d.g / (d.mass * d.omega * d.omega); }

cudaError_t cnn_launch_eval(const Dev& d, const CnnState& cn, const double* X, double* F, cudaStream_t s) {
  const size_t sb = cn_smem_bytes(true);
  opt_in_smem((const void*)cnn_eval_kernel, sb);
  cnn_eval_kernel<<<d.n_chains, HQ_THREADS, sb, s>>>(d, cn, X, F, mean_field_shift(d));
  return cudaGetLastError();
}

cudaError_t cnn_launch_set(const CnnState& cn, const float* src_device, cudaStream_t s) {
  cnn_set_kernel<<<(CN_NP + 255) / 256, 256, 0, s>>>(cn, src_device);
  return cudaGetLastError();
}

cudaError_t cnn_launch_batch(const Dev& d, const CnnState& cn, const double* Xs, const double* ys, const int* idx,
                             int B, float lr, int t_step, cudaStream_t s) {
  // rounds of up to train_ctas samples, each sample on as many CTAs as fill the chip (in layer 2 a CTA per 256 points); a
  // part of the backward pass keeps its partial through the rounds
  const int NL = d.n * d.L, round = B < cn.train_ctas ? B : cn.train_ctas, tiles = (NL + 15) / 16;
  auto parts_of = [&](int ctas, int most) { return std::min(std::max(ctas / round, 1), std::min(most, tiles)); };
  const int parts = parts_of(kCnnTrainCtas, 8), parts2 = std::min((NL + HQ_THREADS - 1) / HQ_THREADS, kCnnParts);
  const size_t s1 = cn_smem_bytes(false), s2 = cn_smem_bytes(true), s3 = cn_back_smem_bytes();
  cudaError_t st = opt_in_smem((const void*)cnn_backward_kernel, s3);
  if (st != cudaSuccess) return st;
  const double x0 = mean_field_shift(d);
  for (int a0 = 0; a0 < B; a0 += round) {
    const int r = B - a0 < round ? B - a0 : round;
    cnn_inputs_kernel<<<dim3((NL + 1023) / 1024, r), 256, 0, s>>>(d, cn, Xs, idx + a0, x0);
    cnn_layer1_kernel<<<dim3((2 * NL + 511) / 512, r), HQ_THREADS, s1, s>>>(d, cn);
    cnn_layer2_kernel<<<dim3(parts2, r), HQ_THREADS, s2, s>>>(d, cn);
    cnn_backward_kernel<<<dim3(parts, r), HQ_THREADS, s3, s>>>(d, cn, ys, idx + a0, B, parts2, a0 == 0, cn.Fb + a0,
                                                              cn.partials);
  }
  cnn_adam_kernel<<<(CN_NP + kSumParams - 1) / kSumParams, HQ_THREADS, 0, s>>>(cn, cn.partials, round * parts, lr, t_step);
  return cudaGetLastError();
}

cudaError_t cnn_launch_loss(const CnnState& cn, const double* ys, const int* idx, int B, double scale, double* loss,
                            cudaStream_t s) {
  cnn_loss_kernel<<<1, 32, 0, s>>>(cn, ys, idx, B, scale, loss);
  return cudaGetLastError();
}

}  // namespace hq
