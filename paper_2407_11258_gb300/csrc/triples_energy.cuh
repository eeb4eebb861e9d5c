// FP32 block energies of the mixed (T) path (included by triples_energy_*.cu).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "triples_energy.h"

namespace lnocc {
namespace {

// ---- FP32 block energies of the mixed path.
//
// With w(y0,y1,y2), v(y0,y1,y2) the scaled block of the sorted virtual triple a <= b <= c and i, j, k
// running over all occupied triples, the sum over the six orderings of (a, b, c) needs two things:
//  * canonical: sum_ijk w_ijk X_ijk, X = 18 v_ijk + 6 (v_ijk + v_jki + v_kij) - 12 (v_ikj + v_jik + v_kji).
//    (Summing (4w + w' + w'')(v - v_rev) over the orderings and all ijk, the three reversals of one
//    unordered {i,j,k} run over the whole other class of placements.) One visit per unordered {i,j,k}
//    loads each element once and serves six elements.
//  * projected: sum_jk sum_alpha Z Y with Z, Y the combinations of w and v of each ordering contracted over i
//    with U. The contraction only depends on which slot i sits in, so each slot is contracted once:
//    A0[y1][y2] = sum_y0 U w, A1[y0][y2] = sum_y1 U w, A2[y0][y1] = sum_y2 U w (and v), and the orderings are
//    combined from these o x o matrices.
// Against a walk over i for every (j, k) with the six placements loaded and combined per element, shared-memory
// reads fall from six per element to four (each element is written once and read by two contractions and one
// triple) and the products to a third; shared-memory bandwidth is what bounds the kernels now (78% of its peak
// at nocc 16; HBM 16%). (16, 240, 960) with 2 LOs 36.2 -> 27.4 ms per call, (8, 120, 480) with one LO 3.1 ->
// 1.5 ms, (19, 125, 500) 14.6 -> 8.0 ms, (32, 200, 800) 268 -> 165 ms.
// Blocks with equal labels (a = b or b = c): the orderings repeat in pairs (W^{aac}_ijk = W^{aac}_jik), so the
// sum over all six is halved (a sixth for a = b = c).

// Compensated FP32 summation of the block partials: a running sum s and the sum c of the
// rounding errors of its additions, each error obtained exactly by Knuth's TwoSum (TAOCP vol. 2,
// 4.2.2), cascaded as in the Sum2 algorithm of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26, 1955
// (2005)). s + c is as accurate as a sum formed in twice the FP32 precision (error about
// u|S| + (n u)^2 sum|x_i|, u = 2^-24), which keeps the block partials as accurate as the FP64 sums
// they replace without FP64-pipe work (the part's FP64 rate is a small fraction of its FP32 rate).
// The _rn intrinsics keep the compiler from fusing or reordering the error terms.
struct CSum {
  float s, c;
};
__device__ __forceinline__ void csum_add(CSum& a, float x) {
  const float t = __fadd_rn(a.s, x);
  const float bp = __fsub_rn(t, a.s);
  const float err = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
  a.s = t;
  a.c = __fadd_rn(a.c, err);
}
__device__ __forceinline__ void csum_merge(CSum& a, const CSum& b) {
  csum_add(a, b.s);
  a.c = __fadd_rn(a.c, b.c);
}
// Block result {canonical, projected} of two compensated sums: warp trees, then warp 0 over the warps'
// sums, in a fixed order; thread 0 writes -(s + c) / (3 rep) in FP64 (the 1/3 of Eq. 16; rep: how often each
// distinct ordering of the block's labels was counted).
__device__ __forceinline__ void csum_block_out(CSum e0, CSum e1, double* out, long long blk_id, double rep) {
  __shared__ float4 sh[32];
  for (int off = 16; off > 0; off >>= 1) {
    CSum o0, o1;
    o0.s = __shfl_xor_sync(0xffffffffu, e0.s, off);
    o0.c = __shfl_xor_sync(0xffffffffu, e0.c, off);
    o1.s = __shfl_xor_sync(0xffffffffu, e1.s, off);
    o1.c = __shfl_xor_sync(0xffffffffu, e1.c, off);
    csum_merge(e0, o0);
    csum_merge(e1, o1);
  }
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) sh[w] = make_float4(e0.s, e0.c, e1.s, e1.c);
  __syncthreads();
  if (threadIdx.x == 0) {
    CSum a0{0.f, 0.f}, a1{0.f, 0.f};
    for (int q = 0; q < static_cast<int>(blockDim.x / 32); ++q) {
      const float4 t = sh[q];
      csum_merge(a0, CSum{t.x, t.y});
      csum_merge(a1, CSum{t.z, t.w});
    }
    out[2 * blk_id] = -(static_cast<double>(a0.s) + static_cast<double>(a0.c)) / (3.0 * rep);
    out[2 * blk_id + 1] = -(static_cast<double>(a1.s) + static_cast<double>(a1.c)) / (3.0 * rep);
  }
}

// X of the six placements of {i,j,k} (cyclic class p[0..2], the other q[0..2]). X does not change when one
// value is taken from all six, so q[0] is subtracted first: the common part of the six v, which cancels, is
// removed before it can round (a block with one occupied orbital gives exactly zero).
__device__ __forceinline__ void tri_x(const float (&p)[3], const float (&q)[3], float (&xp)[3], float (&xq)[3]) {
  const float p0 = p[0] - q[0], p1 = p[1] - q[0], p2 = p[2] - q[0], q1 = q[1] - q[0], q2 = q[2] - q[0];
  const float c = p0 + p1 + p2, n = q1 + q2;
  const float tc = 6.f * fmaf(-2.f, n, c), tn = 6.f * fmaf(-2.f, c, n);
  xp[0] = fmaf(18.f, p0, tc);
  xp[1] = fmaf(18.f, p1, tc);
  xp[2] = fmaf(18.f, p2, tc);
  xq[0] = tn;
  xq[1] = fmaf(18.f, q1, tn);
  xq[2] = fmaf(18.f, q2, tn);
}

// Projected sum at (j, k) from the six contracted placements (w, v): pairs of orderings (z_q - z_r) y_q.
__device__ __forceinline__ float proj_jk(const float2 p0, const float2 p1, const float2 p2, const float2 p3,
                                         const float2 p4, const float2 p5) {
  const float dS = (p0.x + p3.x + p4.x) - (p1.x + p2.x + p5.x);
  float f = fmaf(3.f, p0.x - p5.x, dS) * (p0.y - p5.y);
  f = fmaf(fmaf(3.f, p3.x - p1.x, dS), p3.y - p1.y, f);
  return fmaf(fmaf(3.f, p4.x - p2.x, dS), p4.y - p2.y, f);
}

// Slices and vectors of one block in shared memory.
struct EnergySmem {
  float *Sab, *Sac, *Sbc, *tb, *tc;  // (y0 a|y1 b), (y0 a|y2 c), (y1 b|y2 c) with row stride o | 1; t1 columns
  float4* ad;  // (t1[y][a], d_y, U[y][al], U[y][al + 1]), d_y = (e_a + e_b + e_c)/3 - e_y > 0 formed in FP64
};
__device__ __forceinline__ EnergySmem energy_stage(float* base, const EnergyArgs& g, int a, int c, int o) {
  const int P1 = o | 1, o2 = o * o, v = g.v, b = g.b, nlo = g.nlo;
  EnergySmem m;
  m.ad = reinterpret_cast<float4*>(base);
  m.Sab = reinterpret_cast<float*>(m.ad + o);
  m.Sac = m.Sab + o * P1;
  m.Sbc = m.Sac + o * P1;
  m.tb = m.Sbc + o * P1;
  m.tc = m.tb + o;
  const float* oab = g.ovT + (1LL * a * v + b) * o2;  // o^2 consecutive floats per slice
  const float* oac = g.ovT + (1LL * a * v + c) * o2;
  const float* obc = g.ovT + (1LL * b * v + c) * o2;
  for (int idx = threadIdx.x; idx < o2; idx += blockDim.x) {
    const int p = idx / o, d = p * P1 + idx - p * o;
    m.Sab[d] = oab[idx];
    m.Sac[d] = oac[idx];
    m.Sbc[d] = obc[idx];
  }
  for (int y = threadIdx.x; y < o; y += blockDim.x) {
    const double ex3 = (g.eps[o + a] + g.eps[o + b] + g.eps[o + c]) * (1.0 / 3.0);  // FP64 in these o threads only
    m.ad[y] = make_float4(static_cast<float>(g.t1[y * v + a]), static_cast<float>(ex3 - g.eps[y]),
                          nlo > 0 ? static_cast<float>(g.U[y * nlo]) : 0.f,
                          nlo > 1 ? static_cast<float>(g.U[y * nlo + 1]) : 0.f);
    m.tb[y] = static_cast<float>(g.t1[y * v + b]);
    m.tc[y] = static_cast<float>(g.t1[y * v + c]);
  }
  return m;
}

// Thread t of a block owns the pairs (h, l) with l = t mod o, h = t / o + p H, p < P, H = ceil(o / P). One pair
// a thread while that makes at most 1024 threads an SM's worth of warps can come from (at nocc 16 two pairs
// need fewer shared-memory reads but leave half the warps: 90 against 80 us for a slab of 6480 blocks).
__host__ __device__ constexpr int energy_pairs(int o) { return o <= 22 || (o > kMaxPairOcc && o <= 32) ? 1 : 2; }
__host__ __device__ constexpr int energy_rows(int o) { return (o + energy_pairs(o) - 1) / energy_pairs(o); }
__host__ __device__ constexpr int energy_threads(int o) { return (o * energy_rows(o) + 31) / 32 * 32; }
// resident blocks per SM the registers are limited for: what shared memory allows, at 48 registers or more
__host__ __device__ constexpr int energy_min_blocks(int o) {
  const int smem = (o * blk_s0(o) + 3) * 8 + (energy_small_floats(o) + 1) * 4 + 1024;
  const int by_smem = 232448 / smem, by_regs = 65536 / (48 * energy_threads(o));
  const int n = by_smem < by_regs ? by_smem : by_regs;
  return n < 1 ? 1 : n > 32 ? 32 : n;
}
// 1 / sqrt(x) for normal x > 0 without the scaling of subnormal arguments
__device__ __forceinline__ float rsqrt_pos(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The walk over y0 of a thread's P pairs: W in batches of eight per pair, one batch ahead. begin() issues
// the first batch and may be called long before run(): a block's loads come from DRAM or L2 and their latency
// was the kernels' largest stall (6.5 of 12.8 cycles per instruction without the lead).
template <int P, int O>
struct WalkW {
  static constexpr int kLoads = 8;
  const float* wp[P];
  float nxt[P][kLoads];
  __device__ __forceinline__ void load(int i0, int o) {
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int u = 0; u < kLoads; ++u)
        if (O > 0 ? i0 + u < O : i0 + u < o) nxt[p][u] = wp[p][(i0 + u) * (O > 0 ? O * w_row(O) : o * w_row(o))];
  }
  __device__ __forceinline__ void begin(int o) { load(0, o); }
  // f(p, y0, W of pair p, ad[y0]) for every y0
  template <typename F>
  __device__ __forceinline__ void run(const float4* ad, int o, F&& f) {
#pragma unroll
    for (int i0 = 0; i0 < (O > 0 ? O : o); i0 += kLoads) {
      float cur[P][kLoads];
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int u = 0; u < kLoads; ++u) cur[p][u] = nxt[p][u];
      load(i0 + kLoads, o);
#pragma unroll
      for (int u = 0; u < kLoads; ++u)
        if (O > 0 ? i0 + u < O : i0 + u < o) {
          const float4 x = ad[i0 + u];
#pragma unroll
          for (int p = 0; p < P; ++p) f(p, i0 + u, cur[p][u], x);
        }
    }
  }
};

// The table entries of one thread (t, t + T, ...), all loaded at once when their number is known.
template <int O, int T>
struct TriList {
  static constexpr int N = O > 0 ? (tri_count(O) + T - 1) / T : 1;
  unsigned e[N];
  __device__ __forceinline__ void load(const unsigned* __restrict__ tri) {
    if constexpr (O > 0) {
#pragma unroll
      for (int n = 0; n < N; ++n) e[n] = threadIdx.x + n * T < tri_count(O) ? tri[threadIdx.x + n * T] : ~0u;
    }
  }
  template <typename F>
  __device__ __forceinline__ void each(const unsigned* __restrict__ tri, int o, F&& f) {
    if constexpr (O > 0) {
#pragma unroll
      for (int n = 0; n < N; ++n)
        if (e[n] != ~0u) f(e[n], threadIdx.x + n * T);
    } else {
      for (int t = threadIdx.x; t < tri_count(o); t += blockDim.x) f(tri[t], t);
    }
  }
};

// Shared offsets of the six placements of {i,j,k}: cyclic class p, the other q.
__device__ __forceinline__ void tri_offsets(unsigned e, int S0, int S1, int (&p)[3], int (&q)[3]) {
  const int i = e & 255, j = (e >> 8) & 255, k = e >> 16;
  const int i0 = i * S0, j0 = j * S0, k0 = k * S0, i1 = i * S1, j1 = j * S1, k1 = k * S1;
  p[0] = i0 + j1 + k;
  p[1] = j0 + k1 + i;
  p[2] = k0 + i1 + j;
  q[0] = i0 + k1 + j;
  q[1] = j0 + i1 + k;
  q[2] = k0 + j1 + i;
}

// w and v side by side in shared memory (up to nocc 28). NLG LOs are contracted per sweep (0: canonical
// energy only); with more of them the sweep is repeated (NLG = 1) and the contracted matrices get memory of
// their own behind the small arrays, else they reuse the block's. O > 0: compiled for nocc = O (constant
// offsets, loops unrolled: about half the instructions of O = 0).
template <int NLG, int O>
__global__ void __launch_bounds__(O > 0 ? energy_threads(O) : 64, O > 0 ? energy_min_blocks(O) : 1) k_t_energy_pair(const EnergyArgs g, int ngrp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int slot = blockIdx.y, a = blockIdx.x, c = g.c0 + slot;
  const long long blk_id = static_cast<long long>(blockIdx.y) * gridDim.x + blockIdx.x;
  constexpr int P = O > 0 ? energy_pairs(O) : 1;
  const int o = O > 0 ? O : g.o;
  const int o2 = o * o, S1 = blk_s1(o), S0 = blk_s0(o), P1 = o | 1, T = blockDim.x, H = (o + P - 1) / P;
  float2* swv = reinterpret_cast<float2*>(smraw);
  float* small = reinterpret_cast<float*>(swv + ((o * S0 + 1) & ~1));
  const float* Wb = g.W + slot * g.slot_stride + static_cast<long long>(a) * o2 * w_row(o);
  constexpr int NA = NLG > 0 ? NLG : 1;
  const int hb = threadIdx.x / o, l = threadIdx.x - hb * o;
  const bool own = hb < H;
  // W is stored [i][k][j] (j fastest). A thread owns pairs (j, k) = (y1, y2) = (l, h), consecutive threads
  // consecutive j, and walks i = y0; what depends on (j, k) only stays in registers, and the contraction
  // over y0 comes along. A missing pair repeats the first one (the same
  // values to the same place); its contractions are dropped.
  WalkW<P, O> walk;
  TriList<O, (O > 0 ? energy_threads(O) : 32)> tris;
  int hp[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    hp[p] = own && hb + p * H < o ? hb + p * H : (own ? hb : 0);
    walk.wp[p] = Wb + hp[p] * w_row(o) + l;
  }
  if (own) walk.begin(o);
  const EnergySmem m = energy_stage(small, g, a, c, o);
  float2* Am = ngrp > 1 ? reinterpret_cast<float2*>(small + ((energy_small_floats(o) + 1) & ~1)) : swv;
  tris.load(g.tri);
  __syncthreads();
  float2 A0[P][NA], A1[P][NA], A2[P][NA];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int al = 0; al < NA; ++al) A0[p][al] = A1[p][al] = A2[p][al] = make_float2(0.f, 0.f);
  if (own) {
    float tcv[P], sbc[P], d12[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
      tcv[p] = m.tc[hp[p]];
      sbc[p] = m.Sbc[l * P1 + hp[p]];
      d12[p] = m.ad[l].y + m.ad[hp[p]].y;
    }
    const float tbv = m.tb[l];
    const float* sab = m.Sab + l;
    walk.run(m.ad, o, [&](int p, int y0, float W, const float4& ad) {
      const float disc = fmaf(sab[y0 * P1], tcv[p], fmaf(m.Sac[y0 * P1 + hp[p]], tbv, sbc[p] * ad.x));
      const float sc = rsqrt_pos(ad.y + d12[p]);
      const float w = W * sc;
      const float2 x = make_float2(w, fmaf(disc, sc, w));
      swv[l * S1 + hp[p] + y0 * S0] = x;  // (a repeated pair writes the same value)
      if constexpr (NLG > 0) A0[p][0] = __ffma2_rn(make_float2(ad.z, ad.z), x, A0[p][0]);
      if constexpr (NLG > 1) A0[p][1] = __ffma2_rn(make_float2(ad.w, ad.w), x, A0[p][1]);
    });
  }
  __syncthreads();
  // canonical: one visit per unordered triple. The first o^2 entries of the table have equal members and count
  // half (three of the six placements are distinct; with all three equal X = 0).
  CSum r_can{0.f, 0.f}, r_frag{0.f, 0.f};
  float acc = 0.f;
  tris.each(g.tri, o, [&](unsigned e, int t) {
    int ip[3], iq[3];
    tri_offsets(e, S0, S1, ip, iq);
    float2 p[3], q[3];
    float pv[3], qv[3], xp[3], xq[3];
#pragma unroll
    for (int h = 0; h < 3; ++h) {
      p[h] = swv[ip[h]];
      q[h] = swv[iq[h]];
      pv[h] = p[h].y;
      qv[h] = q[h].y;
    }
    tri_x(pv, qv, xp, xq);
    float f = p[0].x * xp[0];
    f = fmaf(p[1].x, xp[1], f);
    f = fmaf(p[2].x, xp[2], f);
    f = fmaf(q[0].x, xq[0], f);
    f = fmaf(q[1].x, xq[1], f);
    f = fmaf(q[2].x, xq[2], f);
    acc = fmaf(t < o2 ? 0.5f : 1.f, f, acc);
  });
  csum_add(r_can, acc);
  if constexpr (NLG > 0) {
    for (int gr = 0; gr < ngrp; ++gr) {
      if (gr > 0) {  // the next LO takes the place of the last one's coefficients
        __syncthreads();
        for (int y = threadIdx.x; y < o; y += T) m.ad[y].z = static_cast<float>(g.U[y * g.nlo + gr]);
        __syncthreads();
      }
      if (own) {
        if (gr > 0) {  // the first sweep's A0 came with the staging, A0[y1 = l][y2 = h]
#pragma unroll
          for (int p = 0; p < P; ++p)
#pragma unroll
            for (int al = 0; al < NLG; ++al) A0[p][al] = A1[p][al] = A2[p][al] = make_float2(0.f, 0.f);
          for (int y = 0; y < o; ++y) {
            const float u = m.ad[y].z;
#pragma unroll
            for (int p = 0; p < P; ++p)
              A0[p][0] = __ffma2_rn(make_float2(u, u), swv[y * S0 + l * S1 + hp[p]], A0[p][0]);
          }
        }
#pragma unroll (O > 0 ? O : 4)
        for (int y = 0; y < o; ++y) {
          const float4 ad = m.ad[y];
          const float2 u0 = make_float2(ad.z, ad.z), u1 = make_float2(ad.w, ad.w);
#pragma unroll
          for (int p = 0; p < P; ++p) {
            const float2 x1 = swv[hp[p] * S0 + l + y * S1], x2 = swv[hp[p] * S0 + l * S1 + y];
            A1[p][0] = __ffma2_rn(u0, x1, A1[p][0]);
            A2[p][0] = __ffma2_rn(u0, x2, A2[p][0]);
            if constexpr (NLG > 1) {
              A1[p][1] = __ffma2_rn(u1, x1, A1[p][1]);
              A2[p][1] = __ffma2_rn(u1, x2, A2[p][1]);
            }
          }
        }
      }
      __syncthreads();  // everybody is done with the block (or with the previous sweep's matrices)
      if (own) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const int h = hb + p * H;
          if (h >= o) continue;
#pragma unroll
          for (int al = 0; al < NLG; ++al) {
            float2* M = Am + al * 3 * o * P1;
            M[l * P1 + h] = A0[p][al];                   // A0[y1 = l][y2 = h]
            M[o * P1 + h * P1 + l] = A1[p][al];          // A1[y0 = h][y2 = l]
            M[2 * o * P1 + h * P1 + l] = A2[p][al];      // A2[y0 = h][y1 = l]
          }
        }
      }
      __syncthreads();
      if (own) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const int h = hb + p * H;
          if (h >= o) continue;
          const int jk = h * P1 + l, kj = l * P1 + h;
#pragma unroll
          for (int al = 0; al < NLG; ++al) {
            const float2 *M0 = Am + al * 3 * o * P1, *M1 = M0 + o * P1, *M2 = M1 + o * P1;
            csum_add(r_frag, proj_jk(M0[jk], M0[kj], M1[jk], M1[kj], M2[jk], M2[kj]));
          }
        }
      }
    }
  }
  csum_block_out(r_can, r_frag, g.out, blk_id, a == g.b || g.b == c ? (a == c ? 6.0 : 2.0) : 1.0);
}

// One FP32 value per element in shared memory (nocc 29 to 37, where w and v do not fit together): w is staged
// and contracted, then v takes its place, then X; the block of W is read three times (the later ones from
// L2) instead of being kept.
template <int NLG, int O>
__global__ void __launch_bounds__(energy_threads(O), 1) k_t_energy_single(const EnergyArgs g, int ngrp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int o = O, o2 = O * O, P = energy_pairs(O), H = energy_rows(O), S1 = blk_s1(O), S0 = blk_s0(O), P1 = O | 1,
                T = energy_threads(O);
  const int slot = blockIdx.y, a = blockIdx.x, c = g.c0 + slot;
  const long long blk_id = static_cast<long long>(blockIdx.y) * gridDim.x + blockIdx.x;
  float* sx = reinterpret_cast<float*>(smraw);
  const float* Wb = g.W + slot * g.slot_stride + static_cast<long long>(a) * o2 * w_row(o);
  constexpr int NA = NLG > 0 ? NLG : 1;
  CSum r_can{0.f, 0.f}, r_frag{0.f, 0.f};
  const int hb = threadIdx.x / o, l = threadIdx.x - hb * o;
  const bool own = hb < H;
  WalkW<P, O> walk;
  int hp[P];
  bool ok[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    ok[p] = own && hb + p * H < o;
    hp[p] = ok[p] ? hb + p * H : (own ? hb : 0);
    walk.wp[p] = Wb + hp[p] * w_row(o) + l;
  }
  if (own) walk.begin(o);
  const EnergySmem m = energy_stage(sx + ((o * S0 + 3) & ~3), g, a, c, o);
  __syncthreads();
  float d12[P];
#pragma unroll
  for (int p = 0; p < P; ++p) d12[p] = m.ad[l].y + m.ad[hp[p]].y;
  // one sweep per group of NLG LOs (one when there are none); the canonical part comes with the first
  for (int gr = 0; gr < (NLG > 0 ? ngrp : 1); ++gr) {
    if (gr > 0) {
      for (int y = threadIdx.x; y < o; y += T) m.ad[y].z = static_cast<float>(g.U[y * g.nlo + gr]);
      __syncthreads();
    }
    float2 A0[P][NA], A1[P][NA], A2[P][NA];  // (w, v)
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int al = 0; al < NA; ++al) A0[p][al] = A1[p][al] = A2[p][al] = make_float2(0.f, 0.f);
    auto contract12 = [&](bool isv) {
      float c1[P][NA], c2[P][NA];
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int al = 0; al < NA; ++al) c1[p][al] = c2[p][al] = 0.f;
#pragma unroll
      for (int y = 0; y < o; ++y) {
        const float4 ad = m.ad[y];
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const float x1 = sx[hp[p] * S0 + l + y * S1], x2 = sx[hp[p] * S0 + l * S1 + y];
          c1[p][0] = fmaf(ad.z, x1, c1[p][0]);
          c2[p][0] = fmaf(ad.z, x2, c2[p][0]);
          if constexpr (NLG > 1) {
            c1[p][1] = fmaf(ad.w, x1, c1[p][1]);
            c2[p][1] = fmaf(ad.w, x2, c2[p][1]);
          }
        }
      }
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int al = 0; al < NLG; ++al) {
          if (isv) {
            A1[p][al].y = c1[p][al];
            A2[p][al].y = c2[p][al];
          } else {
            A1[p][al].x = c1[p][al];
            A2[p][al].x = c2[p][al];
          }
        }
    };
    if constexpr (NLG > 0) {
      if (own)
        walk.run(m.ad, o, [&](int p, int y0, float W, const float4& ad) {
          const float w = W * rsqrt_pos(ad.y + d12[p]);
          sx[l * S1 + hp[p] + y0 * S0] = w;
          A0[p][0].x = fmaf(ad.z, w, A0[p][0].x);
          if constexpr (NLG > 1) A0[p][1].x = fmaf(ad.w, w, A0[p][1].x);
        });
      __syncthreads();
      if (own) walk.begin(o);  // the next walk's loads come in during the contraction
      if (own) contract12(false);
      __syncthreads();
    }
    if (own) {
      const float tbv = m.tb[l];
      const float* sab = m.Sab + l;
      float tcv[P], sbc[P];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        tcv[p] = m.tc[hp[p]];
        sbc[p] = m.Sbc[l * P1 + hp[p]];
      }
      walk.run(m.ad, o, [&](int p, int y0, float W, const float4& ad) {
        const float disc = fmaf(sab[y0 * P1], tcv[p], fmaf(m.Sac[y0 * P1 + hp[p]], tbv, sbc[p] * ad.x));
        const float sc = rsqrt_pos(ad.y + d12[p]);
        const float vv = fmaf(disc, sc, W * sc);
        sx[l * S1 + hp[p] + y0 * S0] = vv;
        if constexpr (NLG > 0) A0[p][0].y = fmaf(ad.z, vv, A0[p][0].y);
        if constexpr (NLG > 1) A0[p][1].y = fmaf(ad.w, vv, A0[p][1].y);
      });
    }
    __syncthreads();
    if (own && (gr == 0 || gr + 1 < ngrp)) walk.begin(o);
    if constexpr (NLG > 0) {
      if (own) contract12(true);
      __syncthreads();
    }
    if (gr == 0) {
      // X in place of v; the placements of a triple with equal members coincide in pairs with equal X
      constexpr int NT = (tri_count(O) + T - 1) / T;
#pragma unroll 4
      for (int n = 0; n < NT; ++n) {
        const int t = threadIdx.x + n * T;
        if (t >= tri_count(O)) break;
        int ip[3], iq[3];
        tri_offsets(g.tri[t], S0, S1, ip, iq);
        float pv[3], qv[3], xp[3], xq[3];
#pragma unroll
        for (int h = 0; h < 3; ++h) {
          pv[h] = sx[ip[h]];
          qv[h] = sx[iq[h]];
        }
        tri_x(pv, qv, xp, xq);
#pragma unroll
        for (int h = 0; h < 3; ++h) {
          sx[ip[h]] = xp[h];
          sx[iq[h]] = xq[h];
        }
      }
      __syncthreads();
      if (own) {
        float f[P];
#pragma unroll
        for (int p = 0; p < P; ++p) f[p] = 0.f;
        walk.run(m.ad, o, [&](int p, int y0, float W, const float4& ad) {
          f[p] = fmaf(W * rsqrt_pos(ad.y + d12[p]), sx[l * S1 + hp[p] + y0 * S0], f[p]);
        });
        if (ngrp > 1) walk.begin(o);
#pragma unroll
        for (int p = 0; p < P; ++p)
          if (ok[p]) csum_add(r_can, f[p]);
      }
      __syncthreads();
    }
    if constexpr (NLG > 0) {
      float2* Am = reinterpret_cast<float2*>(sx);  // the block is no longer needed in this sweep
#pragma unroll
      for (int p = 0; p < P; ++p) {
        if (!ok[p]) continue;
        const int h = hp[p];
#pragma unroll
        for (int al = 0; al < NLG; ++al) {
          float2* M = Am + al * 3 * o * P1;
          M[l * P1 + h] = A0[p][al];
          M[o * P1 + h * P1 + l] = A1[p][al];
          M[2 * o * P1 + h * P1 + l] = A2[p][al];
        }
      }
      __syncthreads();
#pragma unroll
      for (int p = 0; p < P; ++p) {
        if (!ok[p]) continue;
        const int jk = hp[p] * P1 + l, kj = l * P1 + hp[p];
#pragma unroll
        for (int al = 0; al < NLG; ++al) {
          const float2 *M0 = Am + al * 3 * o * P1, *M1 = M0 + o * P1, *M2 = M1 + o * P1;
          csum_add(r_frag, proj_jk(M0[jk], M0[kj], M1[jk], M1[kj], M2[jk], M2[kj]));
        }
      }
      __syncthreads();
    }
  }
  csum_block_out(r_can, r_frag, g.out, blk_id, a == g.b || g.b == c ? (a == c ? 6.0 : 2.0) : 1.0);
}

constexpr int kEnergySmemMax = 226 * 1024;
constexpr int kRuntimeMaxOcc = 7;  // O = 0: nocc below 8, where a block is too small for the unrolling to matter

// The attribute is per kernel and process-wide: set once, to the largest size, so that concurrent calls on
// fragments of other sizes never lower it under one another's launches.
template <typename K>
void energy_attr(std::once_flag& once, K fn) {
  std::call_once(once, [&] { cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kEnergySmemMax); });
}

// One or two LOs are contracted in one sweep, more in sweeps of one.
template <int NLG, int O>
void launch_energy_one(const EnergyArgs& p, cudaStream_t s) {
  const int o = p.o, ngrp = NLG > 0 ? p.nlo / NLG : 1;
  const size_t small = static_cast<size_t>(energy_small_floats(o) + 1) * 4;
  const size_t blk = static_cast<size_t>(o) * blk_s0(o) + 3, mats = static_cast<size_t>(3) * o * (o | 1) * 8;
  const dim3 grid(p.na, p.nc);
  static std::once_flag once;
  count_launch();
  if constexpr (O > kMaxPairOcc) {
    energy_attr(once, k_t_energy_single<NLG, O>);
    k_t_energy_single<NLG, O><<<grid, energy_threads(O), std::max(blk * 4 + small, mats * NLG), s>>>(p, ngrp);
  } else {
    // matrices in place of the block when there is one sweep (for tiny nocc they can be the larger)
    const size_t smem = ngrp > 1 ? blk * 8 + small + 8 + mats : std::max(blk * 8 + small, mats * NLG);
    energy_attr(once, k_t_energy_pair<NLG, O>);
    k_t_energy_pair<NLG, O><<<grid, energy_threads(o), smem, s>>>(p, ngrp);
  }
}
template <int O>
void launch_energy_o(const EnergyArgs& p, cudaStream_t s) {
  if (p.nlo == 0)
    launch_energy_one<0, O>(p, s);
  else if (p.nlo == 2)
    launch_energy_one<2, O>(p, s);
  else
    launch_energy_one<1, O>(p, s);
}
template <int LO, int HI>
bool launch_energy_range(const EnergyArgs& p, cudaStream_t s) {
  if (p.o < LO || p.o > HI) return false;
  if (p.o == LO) {
    launch_energy_o<LO>(p, s);
    return true;
  }
  if constexpr (LO < HI) return launch_energy_range<LO + 1, HI>(p, s);
  return false;
}

}  // namespace
}  // namespace lnocc
