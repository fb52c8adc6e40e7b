// Learned effective action and the cumulative (network-driven) sampler.
//
// Paper: "Local Updates" -- a fully connected network on the fields around a spacetime point
// predicts the weight change of a move -- and the cumulative update of the benchmark section:
// after network-driven sweeps the whole proposal X -> X' is accepted with min(1, p_c),
// p_c = [W(X')/W(X)] [exp(-beta E_NN[X]) / exp(-beta E_NN[X'])], so the chain stays exact.
//
// Here E_NN is one scalar function: F(X) = sum_{i,l} f(patch_{i,l}(X)), patch = X on the
// 5-site cross x 5 slices around (i, l) minus the mean field -g/(M Omega^2), f a 25-64-64-1
// ReLU network with bfloat16 weights and FP32 arithmetic.  Local moves are Metropolis moves on
// exp(-dtau S_ph + 2F) (exact phonon action); block moves on the same weight, or with the
// periodic convolutional action F_cnn in place of F (hq_cnn.cuh).  Each move is reversible for
// its own weight, so p_c = exp(2 dlog|det M| - 2 sum of the accepted moves' network changes)
// (the phonon action cancels; for one network the sum telescopes to F(X') - F(X)).
// Every evaluation of f runs nn_layer1, nn_layer2 and nn_layer3 (hq_nn_tc.cuh: 16 patches per tile on the
// tensor cores, bfloat16 operands, FP32 accumulation) with the sums of an entry in the same order, in one warp
// (nn_tile_f) or shared by two (local moves), so the inner chain and the acceptance see bit-identical values of f.
#include <cooperative_groups.h>
#include <cstdio>
#include "hq_cnn.cuh"
#include "hq_device.cuh"
#include "hq_nn_tc.cuh"
#include "hq_internal.h"
#include "../../include/holstein_dqmc.h"

namespace hq {
namespace cg = cooperative_groups;

// parameter layout: W1[25][64], b1[64], W2[64][64], b2[64], W3[64], b3
constexpr int NN_IN = 25, NN_H = 64;
constexpr int NN_W1 = 0, NN_B1 = NN_IN * NN_H, NN_W2 = NN_B1 + NN_H, NN_B2 = NN_W2 + NN_H * NN_H,
              NN_W3 = NN_B2 + NN_H, NN_B3 = NN_W3 + NN_H, NN_NP = NN_B3 + 1;
static_assert(NN_NP == HQ_NN_PARAMS, "parameter count");
constexpr int NN_WPAD = (NN_NP + 3) & ~3;
constexpr int NN_GROUPS = HQ_THREADS / 8;


struct NNSmem {
  uint2* frag;   // [TC_FRAGS] weight fragments of the tensor-core layers
  float* tcf;    // [TC_FLOATS] b1, b2, W3, b3
  float* f25;    // [32] f of the patches of a local move
  float* pxf;    // [n] network inputs of the proposed values (local moves)
  int* nbr;      // [n][5] cross neighbours of every site: self, +x, -x, +y, -y
  float* part;   // [128] layer-3 chains handed between warps (local moves)
  volatile int* flag;  // [4] decision of a local move
  double* red;   // [HQ_WARPS]
  double* pu2;   // [n] proposal uniforms (local)
  double* pxn;   // [n] proposed values
  double* pds;   // [n] dtau dS_ph
  double* gacc;  // [NN_GROUPS] per-group sums
  double* scal;  // [8]
  char* cw;      // convolutional weights (with_cnn)
};

__host__ __device__ inline size_t nn_smem_bytes(int n, bool with_cnn = false) {
  size_t b = sizeof(uint2) * TC_FRAGS + sizeof(double) * (HQ_WARPS + 3 * (size_t)n + NN_GROUPS + 8) +
             sizeof(float) * (TC_FLOATS + 32 + 128 + (size_t)n) + sizeof(int) * (4 + 5 * (size_t)n);
  b = (b + 15) & ~(size_t)15;
  if (with_cnn) b += cn_smem_bytes(true);
  return b;
}

__device__ inline NNSmem nn_carve(int n, char* base, bool with_cnn = false) {
  NNSmem s;
  s.frag = (uint2*)base;
  double* p = (double*)(s.frag + TC_FRAGS);
  s.red = p; p += HQ_WARPS;
  s.pu2 = p; p += n;
  s.pxn = p; p += n;
  s.pds = p; p += n;
  s.gacc = p; p += NN_GROUPS;
  s.scal = p; p += 8;
  float* f = (float*)p;
  s.tcf = f; f += TC_FLOATS;
  s.f25 = f; f += 32;
  s.part = f; f += 128;
  s.flag = (volatile int*)f; f += 4;
  s.pxf = f; f += n;
  s.nbr = (int*)f; f += 5 * n;
  s.cw = with_cnn ? base + nn_smem_bytes(n) : nullptr;
  return s;
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// sum over the warp of (double)a - (double)b: a 64-bit integer sum in units of 2^-57 of the largest term
// (a dependent FP64 instruction takes 64 cycles here, an integer shuffle-and-add about 35).  Infinite terms are summed
// in FP64: a patch value of minus infinity has to reject its move.
__device__ __forceinline__ double warp_sum_diff(float a, float b) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  const uint32_t top = __reduce_max_sync(HQ_FULL, max(ua & 0x7fffffffu, ub & 0x7fffffffu));
  const int E = (int)(top >> 23);
  if (E == 255) return warp_sum((double)a - (double)b);
  auto fix = [&](uint32_t u) {
    const int e = (int)((u >> 23) & 0xffu);
    const long long m = e ? (long long)((((unsigned long long)((u & 0x7fffffu) | 0x800000u)) << 33) >> min(E - e, 63)) : 0ll;
    return (int)u < 0 ? -m : m;
  };
  long long v = fix(ua) - fix(ub);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(HQ_FULL, v, o);
  if (v == 0) return 0.0;
  const double d = (double)v;
  return __hiloint2double(__double2hiint(d) + (E - 183) * (1 << 20), __double2loint(d));
}

// u < exp(arg): by a single-precision exponential unless the two are within 1e-4 of each other, whose
// error (|arg| <= 709 rounded to float, and the function's) is below 5e-5.
__device__ __forceinline__ int metropolis(double u, double arg) {
  const float pf = expf((float)arg), uf = (float)u;
  if (uf > pf * 1.0001f) return 0;
  if (uf < pf * 0.9999f) return 1;
  return u < exp(arg);
}

// Cross neighbours of every site: nbr[5 i + c], c = 0 the site itself, then +x, -x, +y, -y.  No barrier.
__device__ inline void build_cross(const Dev& d, int* nbr) {
  for (int r = threadIdx.x; r < d.n; r += HQ_THREADS) {
    const int x = r % d.nx, y = r / d.nx;
    nbr[5 * r + 0] = r;
    nbr[5 * r + 1] = (x + 1) % d.nx + d.nx * y;
    nbr[5 * r + 2] = (x - 1 + d.nx) % d.nx + d.nx * y;
    nbr[5 * r + 3] = x + d.nx * ((y + 1) % d.ny);
    nbr[5 * r + 4] = x + d.nx * ((y - 1 + d.ny) % d.ny);
  }
}

__device__ __forceinline__ int wrap_slice(int l, int L) { return l < 0 ? l + L : (l >= L ? l - L : l); }

// Inputs of the patch centred at (l, i), in the lane's order, from the input table xf [L][n].
__device__ __forceinline__ void patch_inputs(const Dev& d, const NNLane& k, const int* nbr, const float* xf, int l,
                                             int i, float (&z)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
    z[q] = k.c[q] < 0 ? 0.f : xf[wrap_slice(l + k.dl[q], d.L) * d.n + nbr[5 * i + k.c[q]]];
}

// Network input of a field value: the value minus the mean field x0, rounded to float.  Every
// kernel forms inputs through this one expression, so a value gives the same input bits
// wherever it is formed.
__device__ __forceinline__ float net_input(double v, double x0) { return (float)(v - x0); }

// xf[k] = net_input(X[k]) for the L N values of a configuration (all threads; ends with a
// barrier).  Each value enters 25 patches: converting it once keeps the FP64 pipe (which does
// the subtraction and the rounding) out of the patch loops.
__device__ inline void to_inputs(const double* X, double x0, float* xf, int NL) {
  for (int k = threadIdx.x; k < NL; k += HQ_THREADS) xf[k] = net_input(X[k], x0);
  __syncthreads();
}

// Warp sum in a fixed order (every lane gets the same bits).
__device__ __forceinline__ double warp_sum_fixed(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(HQ_FULL, v, o);
  return v;
}

// F of one configuration by the whole CTA: warp w takes the tiles of 16 patch rows w, w + 8, ...
// (fixed order); the patch values go to fc when fc != nullptr.  Returns F in every thread.
__device__ inline double fc_eval_all(const Dev& d, const NNSmem& s, const NNFrags& w, const float* xf, float* fc,
                                     int part_of = 0, int parts = 1) {
  const int n = d.n, NL = d.n * d.L;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, g = lane >> 2, t = lane & 3;
  double part = 0.0;
  const NNLane kin = nn_lane_inputs();
  for (int base = (part_of * HQ_WARPS + warp) * 16; base < NL; base += parts * HQ_WARPS * 16) {
    float f0, f1, z[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = base + g + 8 * h < NL ? base + g + 8 * h : NL - 1;
      patch_inputs(d, kin, s.nbr, xf, r / n, r % n, z[h]);
    }
    nn_tile_f(w, z, f0, f1);
    if (t == 0) {
      if (base + g < NL) {
        part += (double)f0;
        if (fc) fc[base + g] = f0;
      }
      if (base + g + 8 < NL) {
        part += (double)f1;
        if (fc) fc[base + g + 8] = f1;
      }
    }
  }
  part = warp_sum_fixed(part);
  if (lane == 0) s.gacc[warp] = part;
  __syncthreads();
  double F = 0.0;
  for (int k = 0; k < HQ_WARPS; ++k) F += s.gacc[k];
  __syncthreads();
  return F;
}

// F(X) of every chain (grid = chains); also refreshes the patch cache fc.
__global__ void __launch_bounds__(HQ_THREADS) nn_eval_kernel(Dev d, NNState nn, const double* Xall, double* Fout,
                                                             int write_cache) {
  extern __shared__ __align__(16) char nraw[];
  const int c = blockIdx.x, n = d.n, NL = d.n * d.L;
  const NNSmem s = nn_carve(n, nraw);
  build_cross(d, s.nbr);
  const NNFrags w = nn_build_frags(nn.wbf, s.frag, s.tcf);  // (ends with a barrier)
  float* xf = nn.xf + (size_t)c * NL;
  to_inputs(Xall + (size_t)c * NL, nn.x0, xf, NL);
  const double F = fc_eval_all(d, s, w, xf, write_cache ? nn.fcache + (size_t)c * NL : nullptr);
  if (threadIdx.x == 0) Fout[c] = F;
}

// n_inner network-driven sweeps of every chain: local moves at every (l, i), then block
// moves at every site, each accepted on exp(2 dF - dtau dS_ph) with the exact phonon action
// (dF from the patch network, or for block moves with use_cnn from the convolutional action).
// A fixed visiting order of reversible moves is not reversible as a whole, and the
// cumulative accept needs a reversible proposal; so each step draws a direction (second
// uniform of the step's Philox block, tag 4): forward (l, i ascending, then block moves i
// ascending) or the exact reverse of that sequence, with probability 1/2 each.  The accepted
// moves' dF are summed in their order (local moves by warp 1, block moves by thread 0) into nn.dFpath for the
// cumulative accept.
// The caches of the current fields (fc; with use_cnn also the convolutional activations) are
// valid on entry; with use_cnn each network's cache is rebuilt before its part when the other
// part has changed the fields.
__global__ void __launch_bounds__(HQ_THREADS, 2) nn_inner_kernel(const __grid_constant__ Dev d, NNState nn, CnnState cn, int n_inner,
                                                              int do_local, int do_block, int use_cnn, int window,
                                                              int site_window) {
  extern __shared__ __align__(16) char nraw[];
  const int c = blockIdx.x, n = d.n, L = d.L, NL = n * L;
  if (!d.active[c]) return;
  const NNSmem s = nn_carve(n, nraw, use_cnn != 0);
  build_cross(d, s.nbr);
  const NNFrags w = nn_build_frags(nn.wbf, s.frag, s.tcf);  // (ends with a barrier)
  CnSm cw{};
  if (use_cnn) cw = cn_setup(cn.wbf, s.cw);
  double* X = d.X + (size_t)c * NL;
  float* xf = nn.xf + (size_t)c * NL;  // inputs of the current fields, kept with X below
  to_inputs(X, nn.x0, xf, NL);
  float* fc = nn.fcache + (size_t)c * NL;
  float* fnew = nn.fnew + (size_t)c * 6 * L;
  float* xsh = fnew + 5 * L;  // inputs of the moved site's proposed values (block moves)
  float4* h1c = cn.h1c + (size_t)c * NL * 4;
  float* s2c = cn.s2c + (size_t)c * NL;
  float4* h1p = cn.h1p + (size_t)c * 9 * L * 4;
  float* s2p = cn.s2p + (size_t)c * 25 * L;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, g = lane >> 2, t = lane & 3;
  const uint32_t* id = d.cid + 4 * (size_t)c;
  const uint32_t key0 = id[0], key1 = id[1], chain = id[2], step = id[3];
  long long nl_acc = 0, nb_acc = 0;
  double path = 0.0;                   // thread 0
  const NNLane kin = nn_lane_inputs();
  auto opposite = [](int c5) { return c5 == 0 ? 0 : (c5 & 1) ? c5 + 1 : c5 - 1; };
  int pdl[2], opp[2];  // local moves: patch row g + 8h of the warp's tile
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int q = min(16 * ((warp >> 1) & 1) + g + 8 * h, 24);
    pdl[h] = q / 5 - 2;
    opp[h] = opposite(q % 5);
  }
  bool fc_stale = false, cn_stale = false;  // uniform over the CTA
  const double kfac = d.mass / (2.0 * d.dtau), pfac = 0.5 * d.dtau * d.mass * (d.omega * d.omega);
  double du1, du2;
  proposal_uniforms(key0, key1, 0u, step, chain, 4u, du1, du2);
  const bool fwd = du2 < 0.5;
  // local moves on W consecutive slices from a random start l0, block moves on Wb consecutive
  // sites (in index order, periodic) from a random start j0: the two uniforms of event 1 of
  // the step's tag-4 stream, independent of the fields, so each window's move sequence stays
  // reversible
  const int W = (window > 0 && window < L) ? window : L;
  const int Wb = (site_window > 0 && site_window < n) ? site_window : n;
  int l0 = 0, j0 = 0;
  if (W < L || Wb < n) {
    double wu1, wu2;
    proposal_uniforms(key0, key1, 1u, step, chain, 4u, wu1, wu2);
    l0 = (int)(wu1 * (double)L);
    if (l0 > L - 1) l0 = L - 1;
    j0 = (int)(wu2 * (double)n);
    if (j0 > n - 1) j0 = n - 1;
    if (W == L) l0 = 0;
    if (Wb == n) j0 = 0;
  }
  for (int u = 0; u < n_inner; ++u) {
    const uint32_t isw = step * (uint32_t)n_inner + (uint32_t)u;
    for (int part = 0; part < 2; ++part) {
    const bool local_part = (part == 0) == fwd;
    if (local_part && do_local) {
      double lpath = 0.0;  // warp 1
      int lacc = 0;
      if (fc_stale) {
        fc_eval_all(d, s, w, xf, fc);
        fc_stale = false;
      }
      for (int sl0 = 0; sl0 < W; ++sl0) {
        const int sl = (l0 + (fwd ? sl0 : W - 1 - sl0)) % L;
        for (int i = threadIdx.x; i < n; i += HQ_THREADS) {
          double u1, u2;
          proposal_uniforms(key0, key1, (uint32_t)(sl * n + i), isw, chain, 2u, u1, u2);
          const double dx = d.dx_local * (2.0 * u1 - 1.0);
          const double xo = X[(size_t)sl * n + i], xn = xo + dx;
          const double xp = X[(size_t)((sl + 1) % L) * n + i], xm = X[(size_t)((sl - 1 + L) % L) * n + i];
          const double kin = (xp - xn) * (xp - xn) + (xn - xm) * (xn - xm) - (xp - xo) * (xp - xo) - (xo - xm) * (xo - xm);
          s.pu2[i] = u2;
          s.pxn[i] = xn;
          s.pxf[i] = net_input(xn, nn.x0);
          s.pds[i] = kfac * kin + pfac * (xn * xn - xo * xo);
        }
        __syncthreads();
        // The moves of the slice run in warps 0 .. 3 (the others wait for the slice): a move's 25
        // patches are two tiles of 16, warps 2 tau and 2 tau + 1 take tile tau, both forming layer 1 and
        // half of layer 2 each; the first hands its part of layer 3's chain to the second.  Warp 1
        // sums dF and decides.  While it does, the inputs of the next move are already loaded; the one
        // value that an acceptance changes is replaced after the decision.
        if (warp < 4) {
          const int tau = warp >> 1;
          float z[2][8];
          int pos[2][8];  // table position of every input of the move in hand
          auto gather = [&](int i) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              // patch q = 5 (dl + 2) + c contains (sl, i): centre slice sl - dl, centre site the
              // neighbour of i opposite to c (q >= 25: padding rows)
              const int centre = s.nbr[5 * i + opp[h]];
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                pos[h][q] = kin.c[q] < 0 ? -1 : wrap_slice(sl - pdl[h] + kin.dl[q], L) * n + s.nbr[5 * centre + kin.c[q]];
                z[h][q] = pos[h][q] < 0 ? 0.f : xf[pos[h][q]];
              }
            }
          };
          const int ifirst = fwd ? 0 : n - 1, istep = fwd ? 1 : -1;
          gather(ifirst);
          for (int i0 = 0; i0 < n; ++i0) {
            const int i = ifirst + istep * i0, here = sl * n + i;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int q = 0; q < 8; ++q)
                if (pos[h][q] == here) z[h][q] = s.pxf[i];
            float acc1[8][4], acc2[4][4], o0 = 0.f, o1 = 0.f;
            nn_layer1(w, z, acc1);
            if (i0 + 1 < n) gather(i + istep);
            if (!(warp & 1)) {
              nn_layer2<0, 4>(w, acc1, acc2);
              nn_layer3<0, 4>(w, acc2, o0, o1);
              s.part[64 * tau + lane] = o0;
              s.part[64 * tau + 32 + lane] = o1;
              bar_arrive(2 + tau, 64);
            } else {
              nn_layer2<4, 4>(w, acc1, acc2);
              bar_sync(2 + tau, 64);
              o0 = s.part[64 * tau + lane];
              o1 = s.part[64 * tau + 32 + lane];
              nn_layer3<4, 4>(w, acc2, o0, o1);
              o0 = nn_output(w, o0);
              o1 = nn_output(w, o1);
              if (t == 0) {
                s.f25[16 * tau + g] = o0;
                s.f25[16 * tau + g + 8] = o1;
              }
              if (warp == 3) {
                bar_arrive(4, 64);
              } else {
                // lane q < 25: patch q
                const bool on = lane < 25;
                const int ql = lane / 5 - 2, qc = lane % 5;
                const int at = on ? wrap_slice(sl - ql, L) * n + s.nbr[5 * i + (qc == 0 ? 0 : (qc & 1) ? qc + 1 : qc - 1)] : 0;
                const float fold = on ? fc[at] : 0.f;
                bar_sync(4, 64);
                const float fnow = on ? s.f25[lane] : 0.f;
                const double dF = warp_sum_diff(fnow, fold);
                const int acc = metropolis(s.pu2[i], fmin(2.0 * dF - s.pds[i], 709.0));
                if (acc && on) fc[at] = fnow;
                if (lane == 0) {
                  s.flag[0] = acc;
                  if (acc) {
                    X[(size_t)here] = s.pxn[i];
                    xf[here] = s.pxf[i];
                  }
                }
                if (acc) {
                  lpath += dF;
                  ++lacc;
                }
              }
            }
            bar_sync(1, 128);
            if (s.flag[0] && i0 + 1 < n) {
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 8; ++q)
                  if (pos[h][q] == here) z[h][q] = s.pxf[i];
            }
          }
        }
        __syncthreads();
      }
      if (threadIdx.x == 32) {
        s.scal[3] = (double)lacc;
        s.scal[4] = lpath;
      }
      __syncthreads();
      if (s.scal[3] != 0.0) cn_stale = true;
      if (threadIdx.x == 0) {
        nl_acc += (long long)s.scal[3];
        path += s.scal[4];
      }
      __syncthreads();
    }
    if (!local_part && do_block) {
      if (use_cnn && cn_stale) {
        cn_refresh(d, cw, xf, h1c, s2c, s.red);
        cn_stale = false;
      }
      for (int i0 = 0; i0 < Wb; ++i0) {
        const int i = (j0 + (fwd ? i0 : Wb - 1 - i0)) % n;
        if (threadIdx.x == 0) {
          double u1, u2;
          proposal_uniforms(key0, key1, (uint32_t)i, isw, chain, 3u, u1, u2);
          s.scal[1] = d.dx_global * (2.0 * u1 - 1.0);
          s.scal[2] = u2;
        }
        __syncthreads();
        const double dx = s.scal[1];
        double a = 0.0;
        for (int sl = threadIdx.x; sl < L; sl += HQ_THREADS) {
          const double x = X[(size_t)sl * n + i];
          a += (x + dx) * (x + dx) - x * x;
          xsh[sl] = net_input(x + dx, nn.x0);
        }
        a = block_sum(a, s.red);
        const double dS = pfac * a;
        double dF;
        if (use_cnn) {
          dF = cn_block_delta(d, cw, xf, xsh, i, h1c, s2c, h1p, s2p, s.red);
        } else {
          // the 5 L patches containing site i: patch q has centre (q / 5, i - c), c = q % 5; warp
          // w takes the tiles w, w + 8, ... of 16 patches
          double pt = 0.0;
          for (int base = warp * 16; base < 5 * L; base += HQ_WARPS * 16) {
            float f0, f1, z[2][8];
            int at[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int q = min(base + g + 8 * h, 5 * L - 1), l = q / 5, site = s.nbr[5 * i + opposite(q % 5)];
              at[h] = l * n + site;
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                z[h][k] = 0.f;
                if (kin.c[k] >= 0) {
                  const int ll = wrap_slice(l + kin.dl[k], L), j = s.nbr[5 * site + kin.c[k]];
                  z[h][k] = j == i ? xsh[ll] : xf[ll * n + j];
                }
              }
            }
            nn_tile_f(w, z, f0, f1);
            if (t == 0) {
              const int q0 = base + g, q1 = q0 + 8;
              if (q0 < 5 * L) {
                fnew[q0] = f0;
                pt += (double)f0 - (double)fc[at[0]];
              }
              if (q1 < 5 * L) {
                fnew[q1] = f1;
                pt += (double)f1 - (double)fc[at[1]];
              }
            }
          }
          pt = warp_sum_fixed(pt);
          if (lane == 0) s.gacc[warp] = pt;
          __syncthreads();
          dF = 0.0;
          for (int k = 0; k < HQ_WARPS; ++k) dF += s.gacc[k];
        }
        if (threadIdx.x == 0) {
          const double prob = exp(fmin(2.0 * dF - dS, 709.0));
          const int acc = s.scal[2] < prob;
          s.scal[0] = acc;
          if (acc) path += dF;
          nb_acc += acc;
        }
        __syncthreads();
        if (s.scal[0] != 0.0) {
          for (int sl = threadIdx.x; sl < L; sl += HQ_THREADS) {
            const double v = X[(size_t)sl * n + i] + dx;
            X[(size_t)sl * n + i] = v;
            xf[(size_t)sl * n + i] = net_input(v, nn.x0);
          }
          if (use_cnn) {
            fc_stale = true;
          } else {
            for (int q = threadIdx.x; q < 5 * L; q += HQ_THREADS)
              fc[(q / 5) * n + s.nbr[5 * i + opposite(q % 5)]] = fnew[q];
          }
        }
        if (use_cnn) cn_block_end(d, i, s.scal[0] != 0.0, h1c, s2c, h1p, s2p);
        __syncthreads();
      }
    }
    }
  }
  if (threadIdx.x == 0) {
    long long* cnt = nn.counters + (size_t)c * kNNCounters;
    cnt[0] += (long long)n_inner * (do_local ? W * n : 0);
    cnt[1] += nl_acc;
    cnt[2] += (long long)n_inner * (do_block ? Wb : 0);
    cnt[3] += nb_acc;
    nn.dFpath[c] = path;
  }
}

// Cumulative accept of X' (fields now in d.X, log|det M(X')| in d.logdet after the stack
// build) against X (saved in nn.X0 with nn.ld0): p_c = exp(2 dlog|det M| - 2 nn.dFpath).
// With restore_g, a rejected chain also gets back G_0 of X (saved in nn.G0 before the inner
// sweep), so every chain's G holds G_0 of its final fields without another stack build.
__global__ void __launch_bounds__(HQ_THREADS) nn_decide_kernel(Dev d, NNState nn, int restore_g) {
  const int c = blockIdx.x, NL = d.n * d.L;
  if (!d.active[c]) return;
  __shared__ int acc;
  if (threadIdx.x == 0) {
    double u1, u2;
    const uint32_t* id = d.cid + 4 * (size_t)c;
    proposal_uniforms(id[0], id[1], 0u, id[3], id[2], 4u, u1, u2);
    const double ld1 = d.logdet[c], ld0 = nn.ld0[c];
    const double arg = 2.0 * (ld1 - ld0) - 2.0 * nn.dFpath[c];
    const double pc = exp(fmin(arg, 709.0));
    acc = u1 < pc;
    nn.last_pc[c] = pc;
    long long* cnt = nn.counters + (size_t)c * kNNCounters;
    cnt[4] += 1;
    cnt[5] += acc;
    if (!acc) d.logdet[c] = ld0;
    if (!isfinite(arg)) d.status[c] = HQ_ENAN;
  }
  __syncthreads();
  if (!acc) {
    double* X = d.X + (size_t)c * NL;
    const double* X0 = nn.X0 + (size_t)c * NL;
    for (int k = threadIdx.x; k < NL; k += HQ_THREADS) X[k] = X0[k];
    if (restore_g) {
      const size_t nn2 = (size_t)d.n * d.n;
      double* G = d.G + (size_t)c * nn2;
      const double* G0 = nn.G0 + (size_t)c * nn2;
      for (size_t k = threadIdx.x; k < nn2; k += HQ_THREADS) G[k] = G0[k];
    }
  }
}

// ------------------------------------------------------------------------ training
// Mean squared error (1/B) sum_a (F(X_a) - y_a)^2 over a minibatch.  Forward: F_a per sample
// (nn_batch_forward_kernel, the same tensor-core tiles as every other evaluation).  Backward:
// nn_batch_backward_tc_kernel, per-CTA partial gradients summed in a fixed order by the Adam
// kernel.

// A sample's rows are shared out over a cluster (88 us with one CTA per sample at 64 samples of 8x8, L = 80: 64 of
// 152 SMs at work).  Also writes dL/dF of the sample as a float, once, where the backward kernel's FP64 division per
// row held its warps up for a sixth of their time.
__global__ void __launch_bounds__(HQ_THREADS) nn_batch_forward_kernel(Dev d, NNState nn, const double* Xs,
                                                                      const double* ys, const int* idx, int B,
                                                                      double* Fb) {
  extern __shared__ __align__(16) char nraw[];
  __shared__ double Fpart;
  const cg::cluster_group cl = cg::this_cluster();
  const int parts = cl.num_blocks(), rank = cl.block_rank(), a = blockIdx.x / parts, n = d.n, NL = d.n * d.L;
  const NNSmem s = nn_carve(n, nraw);
  build_cross(d, s.nbr);
  const NNFrags w = nn_build_frags(nn.wbf, s.frag, s.tcf);  // (ends with a barrier)
  float* xa = nn.xb + (size_t)a * NL;  // read again by the backward pass
  const int k0 = (int)((long long)NL * rank / parts), k1 = (int)((long long)NL * (rank + 1) / parts);
  to_inputs(Xs + (size_t)idx[a] * NL + k0, nn.x0, xa + k0, k1 - k0);
  cl.sync();
  const double F = fc_eval_all(d, s, w, xa, nullptr, rank, parts);
  if (threadIdx.x == 0) Fpart = F;
  cl.sync();
  if (rank == 0 && threadIdx.x == 0) {
    double sum = 0.0;
    for (int r = 0; r < parts; ++r) sum += *cl.map_shared_rank(&Fpart, r);
    Fb[a] = sum;
    nn.dout[a] = (float)(2.0 * (sum - ys[idx[a]]) / B);
  }
  cl.sync();  // (a peer's shared memory is read up to here)
}

// Backward pass on the tensor cores (see hq_nn_tc.cuh): CTA k takes the 128-row chunks k, k +
// grid, ... of the minibatch's rows (row R = sample a * L N + patch), warp w rows 16 w .. 16 w + 15
// of a chunk.  Inputs come from nn.xb, written by the forward kernel.  partials[k] receives the
// CTA's gradient (every entry written once).
__global__ void __launch_bounds__(HQ_THREADS) nn_batch_backward_tc_kernel(Dev d, NNState nn, int B,
                                                                          float* partials) {
  extern __shared__ __align__(16) char nraw[];
  const int n = d.n, NL = d.n * d.L, rows = B * NL;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, g = lane >> 2, t = lane & 3;
  uint2* frag = (uint2*)nraw;
  float* tcf = (float*)(frag + TR_FRAGS);
  float* colp = tcf + TC_FLOATS;              // [3][8 warps][64] column partials, then gb3 [8]
  uint16_t* h1h = (uint16_t*)(colp + 3 * 8 * TC_H + 8);
  uint16_t* h1l = h1h + TC_H * TR_LD;
  uint16_t* d2h = h1l + TC_H * TR_LD;
  uint16_t* d2l = d2h + TC_H * TR_LD;
  uint16_t* zh = d2l + TC_H * TR_LD;
  uint16_t* zl = zh + TC_K1 * TR_LD;
  uint16_t* d1h = zl + TC_K1 * TR_LD;
  uint16_t* d1l = d1h + TC_H * TR_LD;
  int* nbr = (int*)(d1l + TC_H * TR_LD);
  build_cross(d, nbr);
  const NNLane kin = nn_lane_inputs();
  const NNFrags w = nn_build_frags(nn.wbf, frag, tcf);
  // W2^T fragments for d1 = d2 W2^T: B[k = u][n = v] = W2[v][u]
  uint2* w2t = frag + TC_FRAGS;
  for (int e = threadIdx.x; e < 4 * 8 * 32; e += HQ_THREADS) {
    const int ln = e % 32, j = (e / 32) % 8, st = e / 256;
    const int gg = ln >> 2, tt = ln & 3, v = 8 * j + gg, u = 16 * st + 2 * tt;
    const uint16_t* row = nn.wbf + NN_W2 + v * NN_H;
    w2t[e] = make_uint2(pack_bf16(row[u], row[u + 1]), pack_bf16(row[u + 8], row[u + 9]));
  }
  __syncthreads();
  // owned accumulators: gW2 block (m-tile warp/2, n-tiles 4 (warp%2) ..), gW1 block (m-tile
  // warp/4, n-tiles 2 (warp%4) ..), column partials of this lane's 16 columns
  float gw2[4][4], gw1[2][4], cw3[16], cb2[16], cb1[16], cb3 = 0.f;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int e = 0; e < 4; ++e) gw2[a][e] = 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int e = 0; e < 4; ++e) gw1[a][e] = 0.f;
#pragma unroll
  for (int c = 0; c < 16; ++c) cw3[c] = cb2[c] = cb1[c] = 0.f;
  const int nchunk = (rows + TR_ROWS - 1) / TR_ROWS;
  for (int chunk = blockIdx.x; chunk < nchunk; chunk += gridDim.x) {
    const int r0 = chunk * TR_ROWS + 16 * warp;
    auto rowpos = [&](int row, int& a, int& pr) {
      const int R = r0 + row < rows ? r0 + row : rows - 1;
      a = R / NL;
      pr = R % NL;
    };
    // forward of the warp's 16 rows, keeping what the backward pass needs
    float acc1[8][4], acc2[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc1[j][e] = acc2[j][e] = 0.f;
    float z[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int a, pr;
      rowpos(g + 8 * h, a, pr);  // the minibatch inputs of the forward kernel
      patch_inputs(d, kin, nbr, nn.xb + (size_t)a * NL, pr / n, pr % n, z[h]);
    }
#pragma unroll
    for (int st = 0; st < 2; ++st) {
      uint32_t ahi[4], alo[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        split2(z[q & 1][4 * st + 2 * (q >> 1)], z[q & 1][4 * st + 2 * (q >> 1) + 1], ahi[q], alo[q]);
      }
      store_transposed(zh + 16 * st * TR_LD + 16 * warp, ahi);  // (rows k >= 25 are zero)
      store_transposed(zl + 16 * st * TR_LD + 16 * warp, alo);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint2 b = w.w1[(st * 8 + j) * 32 + lane];
        mma_bf16(acc1[j], ahi, b);
        mma_bf16(acc1[j], alo, b);
      }
    }
    // a1 -> h1 (kept as hi/lo A fragments and staged transposed), masks in acc1's sign
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int v = 8 * j + 2 * t;
      acc1[j][0] += w.b1[v];
      acc1[j][1] += w.b1[v + 1];
      acc1[j][2] += w.b1[v];
      acc1[j][3] += w.b1[v + 1];
    }
#pragma unroll
    for (int st = 0; st < 4; ++st) {
      uint32_t ahi[4], alo[4];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int j = 2 * st + half;
        split2(fmaxf(acc1[j][0], 0.f), fmaxf(acc1[j][1], 0.f), ahi[2 * half], alo[2 * half]);
        split2(fmaxf(acc1[j][2], 0.f), fmaxf(acc1[j][3], 0.f), ahi[2 * half + 1], alo[2 * half + 1]);
      }
      store_transposed(h1h + 16 * st * TR_LD + 16 * warp, ahi);
      store_transposed(h1l + 16 * st * TR_LD + 16 * warp, alo);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint2 b = w.w2[(st * 8 + j) * 32 + lane];
        mma_bf16(acc2[j], ahi, b);
        mma_bf16(acc2[j], alo, b);
      }
    }
    // output gradients of the two rows of this lane
    float dout[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int a, pr;
      rowpos(g + 8 * h, a, pr);
      dout[h] = (r0 + g + 8 * h < rows) ? nn.dout[a] : 0.f;
    }
    if (t == 0) cb3 += dout[0] + dout[1];
    // d2 = relu'(a2) dout W3 (in acc2), gW3 and gb2 column sums, d2 staged transposed
#pragma unroll
    for (int j = 0; j < 8; ++j) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int u = 8 * j + 2 * t + (e & 1);
        const float a2 = acc2[j][e] + w.b2[u];
        const float dv = a2 > 0.f ? dout[e >> 1] * w.w3[u] : 0.f;
        cw3[2 * j + (e & 1)] = fmaf(fmaxf(a2, 0.f), dout[e >> 1], cw3[2 * j + (e & 1)]);
        cb2[2 * j + (e & 1)] += dv;
        acc2[j][e] = dv;
      }
    }
    // d1 = relu'(a1) (d2 W2^T)
    float acc3[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc3[j][e] = 0.f;
#pragma unroll
    for (int st = 0; st < 4; ++st) {
      uint32_t ahi[4], alo[4];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int j = 2 * st + half;
        split2(acc2[j][0], acc2[j][1], ahi[2 * half], alo[2 * half]);
        split2(acc2[j][2], acc2[j][3], ahi[2 * half + 1], alo[2 * half + 1]);
      }
      store_transposed(d2h + 16 * st * TR_LD + 16 * warp, ahi);
      store_transposed(d2l + 16 * st * TR_LD + 16 * warp, alo);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint2 b = w2t[(st * 8 + j) * 32 + lane];
        mma_bf16(acc3[j], ahi, b);
        mma_bf16(acc3[j], alo, b);
      }
    }
#pragma unroll
    for (int st = 0; st < 4; ++st) {
      uint32_t dhi[4], dlo[4];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int j = 2 * st + half;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc3[j][e] = acc1[j][e] > 0.f ? acc3[j][e] : 0.f;
          cb1[2 * j + (e & 1)] += acc3[j][e];
        }
        split2(acc3[j][0], acc3[j][1], dhi[2 * half], dlo[2 * half]);
        split2(acc3[j][2], acc3[j][3], dhi[2 * half + 1], dlo[2 * half + 1]);
      }
      store_transposed(d1h + 16 * st * TR_LD + 16 * warp, dhi);
      store_transposed(d1l + 16 * st * TR_LD + 16 * warp, dlo);
    }
    __syncthreads();
    // gW2 = h1^T d2 and gW1 = z^T d1 over the chunk's 128 rows
#pragma unroll
    for (int ks = 0; ks < TR_ROWS / 16; ++ks) {
      const int m2 = 16 * (warp / 2) * TR_LD + 16 * ks, n2 = 32 * (warp % 2) * TR_LD + 16 * ks;
      mma_tiles3<2>(gw2, h1h + m2, h1l + m2, d2h + n2, d2l + n2);
      const int m1 = 16 * (warp / 4) * TR_LD + 16 * ks, n1 = 16 * (warp % 4) * TR_LD + 16 * ks;
      mma_tiles3<1>(gw1, zh + m1, zl + m1, d1h + n1, d1l + n1);
    }
    __syncthreads();
  }
  // column sums: over the 8 row groups of the warp, then over the warps (fixed order)
#pragma unroll
  for (int c = 0; c < 16; ++c) {
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      cw3[c] += __shfl_xor_sync(HQ_FULL, cw3[c], o);
      cb2[c] += __shfl_xor_sync(HQ_FULL, cb2[c], o);
      cb1[c] += __shfl_xor_sync(HQ_FULL, cb1[c], o);
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) cb3 += __shfl_xor_sync(HQ_FULL, cb3, o);
  if (g == 0) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int u = 8 * j + 2 * t + e;
        colp[(0 * 8 + warp) * TC_H + u] = cw3[2 * j + e];
        colp[(1 * 8 + warp) * TC_H + u] = cb2[2 * j + e];
        colp[(2 * 8 + warp) * TC_H + u] = cb1[2 * j + e];
      }
    if (t == 0) colp[3 * 8 * TC_H + warp] = cb3;
  }
  __syncthreads();
  float* out = partials + (size_t)blockIdx.x * NN_WPAD;
  // gW2 [v][u] at NN_W2 + v * 64 + u: C rows = v (m-tile warp / 2), cols = u
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int v0 = 16 * (warp / 2) + g, u0 = 8 * (4 * (warp % 2) + a) + 2 * t;
    out[NN_W2 + v0 * NN_H + u0] = gw2[a][0];
    out[NN_W2 + v0 * NN_H + u0 + 1] = gw2[a][1];
    out[NN_W2 + (v0 + 8) * NN_H + u0] = gw2[a][2];
    out[NN_W2 + (v0 + 8) * NN_H + u0 + 1] = gw2[a][3];
  }
  // gW1 [k][v] at NN_W1 + k * 64 + v for k < 25
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int k0 = 16 * (warp / 4) + g, v0 = 8 * (2 * (warp % 4) + a) + 2 * t;
    if (k0 < NN_IN) {
      out[NN_W1 + k0 * NN_H + v0] = gw1[a][0];
      out[NN_W1 + k0 * NN_H + v0 + 1] = gw1[a][1];
    }
    if (k0 + 8 < NN_IN) {
      out[NN_W1 + (k0 + 8) * NN_H + v0] = gw1[a][2];
      out[NN_W1 + (k0 + 8) * NN_H + v0 + 1] = gw1[a][3];
    }
  }
  for (int e = threadIdx.x; e < 3 * TC_H + 1; e += HQ_THREADS) {
    float acc = 0.f;
    if (e < 3 * TC_H) {
      const int which = e / TC_H, u = e % TC_H;
      for (int ww = 0; ww < 8; ++ww) acc += colp[(which * 8 + ww) * TC_H + u];
      out[(which == 0 ? NN_W3 : which == 1 ? NN_B2 : NN_B1) + u] = acc;
    } else {
      for (int ww = 0; ww < 8; ++ww) acc += colp[3 * 8 * TC_H + ww];
      out[NN_B3] = acc;
    }
  }
}

// Sum of the per-CTA partials (fixed order) into grad; with lr > 0 an Adam step on the FP32
// master weights and a fresh bfloat16 copy.
__global__ void nn_adam_kernel(NNState nn, const float* partials, int nparts, float lr, int t_step) {
  const int k = blockIdx.x * kSumParams + threadIdx.x % kSumParams;
  const float g = sum_partials(partials, nparts, NN_WPAD, k < NN_NP ? k : NN_NP - 1);
  if (k >= NN_NP || threadIdx.x >= kSumParams) return;
  nn.grad[k] = g;
  if (lr > 0.f) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float m = b1 * nn.adam_m[k] + (1.f - b1) * g;
    const float v = b2 * nn.adam_v[k] + (1.f - b2) * g * g;
    nn.adam_m[k] = m;
    nn.adam_v[k] = v;
    const float mh = m / (1.f - powf(b1, (float)t_step)), vh = v / (1.f - powf(b2, (float)t_step));
    const float w = nn.master[k] - lr * mh / (sqrtf(vh) + eps);
    nn.master[k] = w;
    nn.wbf[k] = float_to_bf16(w);
  }
}

__global__ void nn_loss_kernel(NNState nn, const double* ys, const int* idx, int B, double scale) {
  squared_error(nn.Fb, ys, idx, B, scale, nn.loss);
}

__global__ void nn_set_kernel(NNState nn, const float* src) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < NN_NP) {
    nn.master[k] = src[k];
    nn.wbf[k] = float_to_bf16(src[k]);
    nn.adam_m[k] = 0.f;
    nn.adam_v[k] = 0.f;
  }
}

// ------------------------------------------------------------------------ launchers
static inline cudaError_t smem_opt_in(const void* k, size_t bytes) { return opt_in_smem(k, bytes); }

cudaError_t nn_launch_eval(const Dev& d, const NNState& nn, const double* X, double* F, int write_cache,
                           cudaStream_t s) {
  const size_t sb = nn_smem_bytes(d.n);
  smem_opt_in((const void*)nn_eval_kernel, sb);
  nn_eval_kernel<<<d.n_chains, HQ_THREADS, sb, s>>>(d, nn, X, F, write_cache);
  return cudaGetLastError();
}

cudaError_t nn_launch_inner(const Dev& d, const NNState& nn, const CnnState& cn, int n_inner, int do_local,
                            int do_block, int use_cnn, int window, int site_window, cudaStream_t s) {
  const size_t sb = nn_smem_bytes(d.n, use_cnn != 0);
  smem_opt_in((const void*)nn_inner_kernel, sb);
  nn_inner_kernel<<<d.n_chains, HQ_THREADS, sb, s>>>(d, nn, cn, n_inner, do_local, do_block, use_cnn, window,
                                                      site_window);
  return cudaGetLastError();
}

cudaError_t nn_launch_decide(const Dev& d, const NNState& nn, int restore_g, cudaStream_t s) {
  nn_decide_kernel<<<d.n_chains, HQ_THREADS, 0, s>>>(d, nn, restore_g);
  return cudaGetLastError();
}

cudaError_t nn_launch_loss(const NNState& nn, const double* ys, const int* idx, int B, double scale, cudaStream_t s) {
  nn_loss_kernel<<<1, 32, 0, s>>>(nn, ys, idx, B, scale);
  return cudaGetLastError();
}

cudaError_t nn_launch_set(const NNState& nn, const float* src_device, cudaStream_t s) {
  nn_set_kernel<<<(NN_NP + 255) / 256, 256, 0, s>>>(nn, src_device);
  return cudaGetLastError();
}

// One minibatch: forward, backward partials, reduction (+ Adam step when lr > 0).
cudaError_t nn_launch_batch(const Dev& d, const NNState& nn, const double* Xs, const double* ys, const int* idx,
                            int B, float lr, int t_step, cudaStream_t s) {
  const size_t sf = nn_smem_bytes(d.n);
  smem_opt_in((const void*)nn_batch_forward_kernel, sf);
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      sms = kNNTrainCtas;
  }
  // as many CTAs per sample as still make one wave
  int parts = 8;
  while (parts > 1 && (B * parts > sms || parts * HQ_WARPS * 16 > d.n * d.L)) parts /= 2;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = parts;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(B * parts);
  cfg.blockDim = dim3(HQ_THREADS);
  cfg.dynamicSmemBytes = sf;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaError_t st = cudaLaunchKernelEx(&cfg, nn_batch_forward_kernel, d, nn, Xs, ys, idx, B, nn.Fb);
  if (st != cudaSuccess) return st;
  const size_t sbk = nn_train_tc_smem_bytes();
  smem_opt_in((const void*)nn_batch_backward_tc_kernel, sbk);
  // one wave: one CTA per SM (the kernel takes a whole SM's registers), at most kNNTrainCtas
  const int grid = sms < kNNTrainCtas ? sms : kNNTrainCtas;
  nn_batch_backward_tc_kernel<<<grid, HQ_THREADS, sbk, s>>>(d, nn, B, nn.partials);
  nn_adam_kernel<<<(NN_NP + kSumParams - 1) / kSumParams, HQ_THREADS, 0, s>>>(nn, nn.partials, grid, lr, t_step);
  return cudaGetLastError();
}

}  // namespace hq
