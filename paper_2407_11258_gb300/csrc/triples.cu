// LNO-(T): W and V intermediates of the supplementary Sec. S1 and the projected (T) pair energy of
// Eq. 16, summed as E^(F) = sum_alpha sum_ii' U_i,alpha E_ii',(T) U_i',alpha (Eq. 15).
//
// Loop structure ("virtual-outer"): for each pair b <= c and every a <= b the block
// W^{abc}_{ijk} over all occupied (i,j,k) is formed. Because W and V are invariant under a
// simultaneous permutation of (i,a), (j,b), (k,c), the block of the sorted triple a<=b<=c yields
// W^{pi(abc)} for every ordering pi by permuting (i,j,k), so each distinct virtual triple is formed
// once (2 o^3 v^4 + 2 o^4 v^3 flops in the contractions), and the projection over (i, i') stays
// local to the block.
//
// Within a slab of fixed b (virtual c >= b in chunks of up to 768 MB of W, a <= b) each of the six
// permutation terms is one GEMM over K = v + o: the d-part (K = v) and the l-part (K = o) operands are
// packed side by side along K (listed per fixed (b, c); rows run over a and one or two occupied indices):
//   G_i  rows (a,i), cols (k,j): (ai|bd) t_kj^cd + (ai|cd) t_jk^bd - t_il^ab (ck|jl) - t_il^ac (bj|kl)
//   G_j  rows (a,j), cols (k,i): (bj|ad) t_ki^cd - t_jl^ba (ck|il)
//   G_k  rows (a,k), cols (j,i): (ck|ad) t_ji^bd - t_kl^ca (bj|il)
//   G_4  rows (a,i,k), cols j  : t_ik^ad (bj|cd) - (ai|kl) t_jl^bc
//   G_6  rows (a,i,j), cols k  : t_ij^ad (ck|bd) - (ai|jl) t_kl^cb
// all accumulated into W[a][i][j][k]; a block energy kernel then applies V = W + (ai|bj) t_k^c +
// (ai|ck) t_j^b + (bj|ck) t_i^a, w = W / sqrt(-Delta), v = V / sqrt(-Delta) and the contraction
// -1/3 sum (4 w^abc + w^bca + w^cab)(v^abc - v^cba) for every distinct ordering of (a, b, c).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "ccsd_kernels.h"
#include "fragment.h"
#include "gemm_slices.h"
#include "internal.h"
#include "triples_energy.h"

namespace lnocc {

static inline Ax A_(int n, long long s) { return Ax{n, s}; }

namespace {

// Position permutations of three slots, listed as (p1, p2, p3) in 0-based slots.
__constant__ int kPerm[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};

// Block energy, generic form: one CTA per (pair, a) with a <= b; threads over (j, k). Any nocc and any
// number of LOs: the projected i-sums are kept for up to kLoChunk LOs at a time, and for more LOs the
// i loop is repeated per chunk (the canonical part is accumulated in the first pass only). W is FP64
// (plain path) or FP32 (mixed path); the arithmetic here is FP64 on both.
// W: [slot][a][i][k][j]; out: per block {canonical, projected} partials (FP64).
constexpr int kLoChunk = 8;

template <typename TW>
__global__ void k_t_energy(const TW* __restrict__ W, long long slot_stride, int b, int c0, int o, int v,
                           const double* __restrict__ eps, const double* __restrict__ t1,
                           const double* __restrict__ ovov, const double* __restrict__ U, int nlo,
                           double* __restrict__ out, int jp) {
  const int slot = blockIdx.y;
  const int a = blockIdx.x;
  const int c = c0 + slot;
  const long long oblk = 1LL * o * o * jp;
  const long long blk_id = static_cast<long long>(blockIdx.y) * gridDim.x + blockIdx.x;
  const TW* Wb = W + slot * slot_stride + a * oblk;
  const int x[3] = {a, b, c};
  const double ex = eps[o + a] + eps[o + b] + eps[o + c];
  const long long ov = 1LL * o * v;
  auto widx = [&](int y0, int y1, int y2) { return (1LL * y0 * o + y2) * jp + y1; };  // W stored [a][i][k][j], rows of jp
  // w and v of the block at occupied (y0, y1, y2)
  auto wv = [&](int y0, int y1, int y2, double& w, double& vv) {
    const double Wv = static_cast<double>(Wb[widx(y0, y1, y2)]);
    const double Vv = Wv + ovov[(1LL * y0 * v + a) * ov + 1LL * y1 * v + b] * t1[y2 * v + c] +
                      ovov[(1LL * y0 * v + a) * ov + 1LL * y2 * v + c] * t1[y1 * v + b] +
                      ovov[(1LL * y1 * v + b) * ov + 1LL * y2 * v + c] * t1[y0 * v + a];
    const double s = 1.0 / sqrt(ex - eps[y0] - eps[y1] - eps[y2]);
    w = Wv * s;
    vv = Vv * s;
  };
  double e_can = 0.0, e_frag = 0.0;
  const int nchunk = nlo > 0 ? (nlo + kLoChunk - 1) / kLoChunk : 1;
  for (int jk = threadIdx.x; jk < o * o; jk += blockDim.x) {
    const int j = jk / o, k = jk % o;
    for (int pi = 0; pi < 6; ++pi) {
      const int p0 = kPerm[pi][0], p1 = kPerm[pi][1], p2 = kPerm[pi][2];
      // skip orderings already counted (equal labels)
      bool dup = false;
      for (int q = 0; q < pi && !dup; ++q)
        dup = x[kPerm[q][0]] == x[p0] && x[kPerm[q][1]] == x[p1] && x[kPerm[q][2]] == x[p2];
      if (dup) continue;
      // ordering T = (x[p0], x[p1], x[p2]); W^T_{ijk} = W^{abc}_y with y[p0]=i, y[p1]=j, y[p2]=k
      for (int ch = 0; ch < nchunk; ++ch) {
        const int al0 = ch * kLoChunk;
        const int nal = nlo > 0 ? min(kLoChunk, nlo - al0) : 0;
        double zu[kLoChunk], yu[kLoChunk];
#pragma unroll
        for (int q = 0; q < kLoChunk; ++q) zu[q] = yu[q] = 0.0;
        for (int i = 0; i < o; ++i) {
          int y[3];
          double w0, w1, w2, v0, v3, dummy;
          y[p0] = i; y[p1] = j; y[p2] = k;        // T
          wv(y[0], y[1], y[2], w0, v0);
          y[p1] = i; y[p2] = j; y[p0] = k;        // T o c   = (t2, t3, t1): slots (p1, p2, p0)
          wv(y[0], y[1], y[2], w1, dummy);
          y[p2] = i; y[p0] = j; y[p1] = k;        // T o c^2 = (t3, t1, t2): slots (p2, p0, p1)
          wv(y[0], y[1], y[2], w2, dummy);
          y[p2] = i; y[p1] = j; y[p0] = k;        // (t3, t2, t1): slots (p2, p1, p0)
          wv(y[0], y[1], y[2], dummy, v3);
          const double z = 4.0 * w0 + w1 + w2;
          const double yy = v0 - v3;
          if (ch == 0) e_can += z * yy;
#pragma unroll
          for (int q = 0; q < kLoChunk; ++q) {
            if (q < nal) {
              const double u = U[i * nlo + al0 + q];
              zu[q] += u * z;
              yu[q] += u * yy;
            }
          }
        }
#pragma unroll
        for (int q = 0; q < kLoChunk; ++q)
          if (q < nal) e_frag += zu[q] * yu[q];
      }
    }
  }
  // block reduction (fixed order)
  __shared__ double sh[2][32];
  for (int off = 16; off > 0; off >>= 1) {
    e_can += __shfl_xor_sync(0xffffffffu, e_can, off);
    e_frag += __shfl_xor_sync(0xffffffffu, e_frag, off);
  }
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) {
    sh[0][w] = e_can;
    sh[1][w] = e_frag;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int q = 0; q < static_cast<int>(blockDim.x / 32); ++q) {
      s0 += sh[0][q];
      s1 += sh[1][q];
    }
    out[2 * blk_id] = -s0 / 3.0;
    out[2 * blk_id + 1] = -s1 / 3.0;
  }
}

// Staged block energy: one CTA per (pair, a), a <= b. w = W s and v = (W + disconnected) s are formed once
// per block in shared memory (Real = float on the mixed path, double on the FP64 path), with
// s = 1/sqrt(-Delta) and -Delta = d_i + d_j + d_k, d_m = (e_a + e_b + e_c)/3 - e_m > 0 evaluated in FP64
// (a sum of positive terms: no cancellation when it is rounded to Real). Threads then run over (j, k)
// and every distinct ordering of (a, b, c); the i-sums are accumulated in Real and the block sum in FP64.
// VFLY: only w is staged and v = w + disc s is recomputed where it is read (the slices, t1 columns and
// d_m are in shared memory already); half the shared memory, for blocks too large to stage both.
// Launched for the FP64 path; the mixed path runs k_t_energy_pair or k_t_energy_single below.
template <typename TW, typename Real, int NLO, bool VFLY>
__global__ void k_t_energy_staged(const TW* __restrict__ W, long long slot_stride, int b, int c0, int o, int v,
                                  const double* __restrict__ eps, const double* __restrict__ t1,
                                  const double* __restrict__ ovov, const double* __restrict__ U, int nlo_rt,
                                  double* __restrict__ out) {
  // NLO: number of fragment LO columns of U, fixed at compile time (0 = canonical energy only);
  // U is zero-padded to NLO columns by the host, so nlo_rt (the caller's count) is not needed here
  (void)nlo_rt;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int slot = blockIdx.y, a = blockIdx.x;
  const int c = c0 + slot;
  const long long blk_id = static_cast<long long>(blockIdx.y) * gridDim.x + blockIdx.x;
  const int o2 = o * o, o3 = o2 * o;
  // shared-memory blocks w and v use padded strides (S0 = o(o+1)+1, S1 = o+1, S2 = 1, all odd for
  // even o) so that the permuted reads of the orderings below spread over the banks
  const int S1 = o + 1, S0 = o * S1 + 1;
  const int blk = o * S0;
  Real* sw = reinterpret_cast<Real*>(smraw);
  Real* sv = sw + blk;
  const int P1 = o + 1, o2p = o * P1;  // o x o slices padded to odd row stride
  Real* Sab = VFLY ? sv : sv + blk;  // (y0 a|y1 b)
  Real* Sac = Sab + o2p;    // (y0 a|y2 c)
  Real* Sbc = Sac + o2p;    // (y1 b|y2 c)
  Real* ta = Sbc + o2p;     // t1[y][a], t1[y][b], t1[y][c]
  Real* tb = ta + o;
  Real* tc = tb + o;
  Real* dm = tc + o;        // d_m
  Real* Us = dm + o;        // U[i][alpha]
  const long long ov = 1LL * o * v;
  const double ex3 = (eps[o + a] + eps[o + b] + eps[o + c]) / 3.0;
  for (int idx = threadIdx.x; idx < o2; idx += blockDim.x) {
    const int p = idx / o, q = idx % o;
    Sab[p * P1 + q] = static_cast<Real>(ovov[(1LL * p * v + a) * ov + 1LL * q * v + b]);
    Sac[p * P1 + q] = static_cast<Real>(ovov[(1LL * p * v + a) * ov + 1LL * q * v + c]);
    Sbc[p * P1 + q] = static_cast<Real>(ovov[(1LL * p * v + b) * ov + 1LL * q * v + c]);
  }
  for (int y = threadIdx.x; y < o; y += blockDim.x) {
    ta[y] = static_cast<Real>(t1[y * v + a]);
    tb[y] = static_cast<Real>(t1[y * v + b]);
    tc[y] = static_cast<Real>(t1[y * v + c]);
    dm[y] = static_cast<Real>(ex3 - eps[y]);
  }
  for (int idx = threadIdx.x; idx < o * NLO; idx += blockDim.x) Us[idx] = static_cast<Real>(U[idx]);
  __syncthreads();
  const TW* Wb = W + slot * slot_stride + static_cast<long long>(a) * o3;
  // W is stored [i][k][j] (j fastest): read it in that order (coalesced)
  // (y0, y2, y1) of idx advance by the fixed stride blockDim.x with carries: no division in the loop
  const int st = blockDim.x, d1 = st % o, d2 = (st / o) % o, d0 = st / o2;
  int y1 = threadIdx.x % o, y2 = (threadIdx.x / o) % o, y0 = threadIdx.x / o2;
  for (int idx = threadIdx.x; idx < o3; idx += st) {
    const Real Wv = static_cast<Real>(Wb[idx]);
    const Real disc = Sab[y0 * P1 + y1] * tc[y2] + Sac[y0 * P1 + y2] * tb[y1] + Sbc[y1 * P1 + y2] * ta[y0];
    const Real d = dm[y0] + dm[y1] + dm[y2];
    Real sc;
    if (sizeof(Real) == 4)
      sc = static_cast<Real>(rsqrtf(static_cast<float>(d)));
    else
      sc = static_cast<Real>(1.0 / sqrt(static_cast<double>(d)));
    const int sidx = y0 * S0 + y1 * S1 + y2;
    sw[sidx] = Wv * sc;
    if (!VFLY) sv[sidx] = (Wv + disc) * sc;
    y1 += d1;
    int cy = y1 >= o;
    y1 -= cy ? o : 0;
    y2 += d2 + cy;
    cy = y2 >= o;
    y2 -= cy ? o : 0;
    y0 += d0 + cy;
  }
  __syncthreads();
  // The six placements of (i, j, k) into the slots of W^{abc}_y: placement q puts i in slot PM[q][0],
  // j in PM[q][1], k in PM[q][2]. For ordering (p0, p1, p2) of the virtual labels, the four W values it
  // needs -- T, T o c, T o c^2 and the reversal -- are the placements (p0,p1,p2), (p1,p2,p0), (p2,p0,p1)
  // and (p2,p1,p0). Each thread loads the six w (and v) placements once per i and evaluates every
  // distinct ordering from registers. With the loops fully unrolled every index is a compile-time choice.
  constexpr int PM[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
  const int x0 = a, x1 = b, x2 = c;
  auto X = [&](int p) { return p == 0 ? x0 : (p == 1 ? x1 : x2); };
  auto SS = [&](int p) { return p == 0 ? S0 : (p == 1 ? S1 : 1); };
  bool act[6];  // orderings with distinct label sequences (equal labels repeat an ordering)
#pragma unroll
  for (int pi = 0; pi < 6; ++pi) {
    bool dup = false;
#pragma unroll
    for (int q = 0; q < pi; ++q)
      dup = dup || (X(PM[q][0]) == X(PM[pi][0]) && X(PM[q][1]) == X(PM[pi][1]) && X(PM[q][2]) == X(PM[pi][2]));
    act[pi] = !dup;
  }
  // per-thread partials in FP64: FP32 (Real = float) sums run over one (j, k) only (6 nocc terms)
  double r_can = 0, r_frag = 0;
  for (int jk = threadIdx.x; jk < o2; jk += blockDim.x) {
    const int j = jk / o, k = jk % o;
    int off[6], si[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      off[q] = j * SS(PM[q][1]) + k * SS(PM[q][2]);
      si[q] = SS(PM[q][0]);
    }
    Real acc = 0, zu[6][NLO > 0 ? NLO : 1], yu[6][NLO > 0 ? NLO : 1];
#pragma unroll
    for (int pi = 0; pi < 6; ++pi)
#pragma unroll
      for (int al = 0; al < NLO; ++al) zu[pi][al] = yu[pi][al] = 0;
    for (int i = 0; i < o; ++i) {
      Real wq[6], vq[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        wq[q] = sw[off[q]];
        if (!VFLY) {
          vq[q] = sv[off[q]];
        } else {
          // v = w + disc s at this placement (slices, t1 columns and d_m are staged)
          const int y0 = PM[q][0] == 0 ? i : (PM[q][1] == 0 ? j : k);
          const int y1 = PM[q][0] == 1 ? i : (PM[q][1] == 1 ? j : k);
          const int y2 = PM[q][0] == 2 ? i : (PM[q][1] == 2 ? j : k);
          const Real dd = Sab[y0 * P1 + y1] * tc[y2] + Sac[y0 * P1 + y2] * tb[y1] + Sbc[y1 * P1 + y2] * ta[y0];
          const Real d = dm[y0] + dm[y1] + dm[y2];
          Real sc;
          if (sizeof(Real) == 4)
            sc = static_cast<Real>(rsqrtf(static_cast<float>(d)));
          else
            sc = static_cast<Real>(1.0 / sqrt(static_cast<double>(d)));
          vq[q] = wq[q] + dd * sc;
        }
        off[q] += si[q];
      }
#pragma unroll
      for (int pi = 0; pi < 6; ++pi) {
        if (!act[pi]) continue;
        const int p0 = PM[pi][0], p1 = PM[pi][1], p2 = PM[pi][2];
        auto idx = [&](int s0, int s1) {  // placement index of the tuple (s0, s1, 3 - s0 - s1)
          return s0 == 0 ? (s1 == 1 ? 0 : 1) : (s0 == 1 ? (s1 == 0 ? 2 : 3) : (s1 == 0 ? 4 : 5));
        };
        const Real z = 4 * wq[idx(p0, p1)] + wq[idx(p1, p2)] + wq[idx(p2, p0)];
        const Real y = vq[idx(p0, p1)] - vq[idx(p2, p1)];
        acc += z * y;
#pragma unroll
        for (int al = 0; al < NLO; ++al) {
          zu[pi][al] += Us[i * NLO + al] * z;
          yu[pi][al] += Us[i * NLO + al] * y;
        }
      }
    }
    r_can += acc;
#pragma unroll
    for (int pi = 0; pi < 6; ++pi)
#pragma unroll
      for (int al = 0; al < NLO; ++al) r_frag += zu[pi][al] * yu[pi][al];
  }
  double e_can = static_cast<double>(r_can), e_frag = static_cast<double>(r_frag);
  __shared__ double sh[2][32];
  for (int off = 16; off > 0; off >>= 1) {
    e_can += __shfl_xor_sync(0xffffffffu, e_can, off);
    e_frag += __shfl_xor_sync(0xffffffffu, e_frag, off);
  }
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) {
    sh[0][w] = e_can;
    sh[1][w] = e_frag;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int q = 0; q < static_cast<int>(blockDim.x / 32); ++q) {
      s0 += sh[0][q];
      s1 += sh[1][q];
    }
    out[2 * blk_id] = -s0 / 3.0;
    out[2 * blk_id + 1] = -s1 / 3.0;
  }
}

// Unordered occupied triples, i | j << 8 | k << 16 (nocc <= 255), grouped by the gaps between their members
// around the circle 0 .. o-1: consecutive entries are one triple shifted by one orbital, so that consecutive
// threads read the staged block at a constant odd stride whatever the placement (lexicographic order cost four
// bank conflicts per load). Gap sequences (g1, g2, o - g1 - g2), one per class of cyclic rotations; one warp.
__global__ void k_tri_table(int o, unsigned* __restrict__ tri) {
  int pos = 0;
  for (int g1 = 0; g1 <= o / 3; ++g1) {
    for (int g2 = g1; g2 <= o - 2 * g1; ++g2) {
      const int g3 = o - g1 - g2;
      // the smallest rotation stands for the class: g1 <= g2, g1 <= g3, and with g3 = g1 only g2 = g1
      if (g3 == g1 && g2 != g1) continue;
      const int n = g1 == g2 && g2 == g3 ? g1 : o;  // equal gaps: the triple repeats after a third of the circle
      for (int i = threadIdx.x; i < n; i += 32) {
        const int j = (i + g1) % o, k = (i + g1 + g2) % o;
        tri[pos + i] = static_cast<unsigned>(i) | static_cast<unsigned>(j) << 8 | static_cast<unsigned>(k) << 16;
      }
      pos += n;
    }
  }
}

// Per-c tables of the batched (T) terms, one entry per (b, c >= b) in b-major order (the order of the
// chunk plan: entry (b, c) at b v - b (b - 1) / 2 + c - b). For W chunks of ncmax(b) = max(1, welems /
// ((b + 1) o^2 jp)) values of c, c sits at position q = (c - b) mod ncmax(b) of its chunk. bat: sigma5
// (rows (c, a, k) of XT2 against rows (b, i, j) of TOT); bat12: sigma1 (rows (b, a, i) of XT1 against rows
// (c, k, j) of TO) then sigma2 (rows (c, a, i) of XT1 against rows (b, k, j) of TOT) into one accumulator.
__global__ void k_batch_tables(int o, int v, int jp, long long welems, BatchEntry* __restrict__ bat,
                               BatchEntry* __restrict__ bat12) {
  const long long oo = 1LL * o * o, ooj = oo * jp;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < v; b += gridDim.x * blockDim.x) {
    const long long slab = (b + 1) * ooj;
    const long long ncmax = welems / slab > 1 ? welems / slab : 1;
    const long long base = 1LL * b * v - 1LL * b * (b - 1) / 2;
    const int Ma = (b + 1) * o;
    const int brow = b * static_cast<int>(oo);
    for (int c = b; c < v; ++c) {
      const long long q = (c - b) % ncmax;
      const int arow = c * v * o;
      bat[base + c - b] = BatchEntry{arow, brow, Ma, arow, brow, 0, q * slab};
      bat12[base + c - b] = BatchEntry{b * v * o, c * static_cast<int>(oo), Ma, arow, brow, 0, q * slab};
    }
  }
}

// FP32 copy of (ia|jb) in the order the block energy reads it: ovT[a][b][i][j] = (ia|jb).
__global__ void k_ovov_t(const double* __restrict__ ovov, float* __restrict__ ovT, int o, int v) {
  const long long ov = 1LL * o * v, n = ov * ov, oo = 1LL * o * o;
  for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < n;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int b = static_cast<int>(idx % v), j = static_cast<int>((idx / v) % o);
    const int a = static_cast<int>((idx / ov) % v), i = static_cast<int>(idx / (ov * v));
    ovT[(1LL * a * v + b) * oo + 1LL * i * o + j] = static_cast<float>(ovov[idx]);
  }
}

// Sum of the per-block partials in a fixed order: out[0] canonical, out[1] projected.
// Block g sums partials [g * chunk, min((g + 1) * chunk, nblk)) into out[2g], out[2g + 1] (the first of
// two fixed-order passes; one 1024-thread block alone took about 1.3 ms for the 2.3e6 block partials
// of a diamond-like call).
__global__ void k_t_finish_part(const double* part, long long nblk, long long chunk, double* out) {
  __shared__ double sh[2][32];
  double s0 = 0.0, s1 = 0.0;
  const long long i0 = blockIdx.x * chunk, i1 = min(nblk, i0 + chunk);
  for (long long i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    s0 += part[2 * i];
    s1 += part[2 * i + 1];
  }
  for (int off = 16; off > 0; off >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, off);
    s1 += __shfl_xor_sync(0xffffffffu, s1, off);
  }
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) {
    sh[0][w] = s0;
    sh[1][w] = s1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a0 = 0.0, a1 = 0.0;
    for (int q = 0; q < static_cast<int>(blockDim.x / 32); ++q) {
      a0 += sh[0][q];
      a1 += sh[1][q];
    }
    out[2 * blockIdx.x] = a0;
    out[2 * blockIdx.x + 1] = a1;
  }
}

__global__ void k_t_finish(const double* part, long long nblk, double* out) {
  __shared__ double sh[2][32];
  double s0 = 0.0, s1 = 0.0;
  for (long long i = threadIdx.x; i < nblk; i += blockDim.x) {
    s0 += part[2 * i];
    s1 += part[2 * i + 1];
  }
  for (int off = 16; off > 0; off >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, off);
    s1 += __shfl_xor_sync(0xffffffffu, s1, off);
  }
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) {
    sh[0][w] = s0;
    sh[1][w] = s1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a0 = 0.0, a1 = 0.0;
    for (int q = 0; q < static_cast<int>(blockDim.x / 32); ++q) {
      a0 += sh[0][q];
      a1 += sh[1][q];
    }
    out[0] = a0;
    out[1] = a1;
  }
}

// dst row (y, a, i) <- src row (a, y, i) of a packed [planes][rows][Kp] operand (rows = v*v*o): one
// warp per row, 16-byte copies (a packed row is a multiple of 128 bytes)
__global__ void k_swap_outer_rows(const uint4* __restrict__ src, uint4* __restrict__ dst, int v, int o, int nvec,
                                  int planes) {
  const long long rows = 1LL * v * v * o;
  const int lane = threadIdx.x % 32;
  const long long nw = static_cast<long long>(gridDim.x) * blockDim.x / 32;
  for (long long w = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) / 32; w < rows * planes;
       w += nw) {
    const long long r = w % rows, pl = w / rows;
    const int i = static_cast<int>(r % o);
    const long long q = r / o;
    const int a = static_cast<int>(q % v);
    const long long y = q / v;
    const long long sr = (1LL * a * v + y) * o + i;
    const uint4* s = src + (pl * rows + sr) * nvec;
    uint4* d = dst + (pl * rows + r) * nvec;
    for (int e = lane; e < nvec; e += 32) d[e] = s[e];
  }
}

}  // namespace

// Device temporaries of one lnocc_triples call, in allocation order. Every size here is what the call
// asks for; with a caller workspace attached the call carves them from it in this order (256-byte
// aligned), so lnocc_workspace_bytes and the call agree by construction.
//
// What makes the call faster but can be done without never decides whether a workspace is large enough:
//   * mixed: rows of W padded to 16 bytes, and the table of occupied triples. In an attached workspace W starts
//     early by what the padding adds, inside the temporaries of the operands' assembly, which are no longer
//     read when the first W is written, and the table lies at their start. Where those are too small for that
//     (nvir below about nocc) and the workspace has no room, W is unpadded, the contractions run one per
//     term and the energies in the generic kernel.
//   * FP64: the digit planes of the four operands, cut once per call instead of in every product that reads them.
//     An attached workspace without room for them, or a call whose allocations fail, runs without: sigma3, 4
//     and 6 then cut their operands for every chunk into the handle's slice workspace, and the batched
//     sigma1, 2 and 5 run on the SIMT kernel. The planes are left out beyond 32 GB (nocc 24 with nvir above 250).
TriplesPlan triples_plan(int o, int v, int N, bool bf, int chunk_mb, size_t avail) {
  TriplesPlan p{};
  const long long oo = 1LL * o * o, vv = 1LL * v * v, ooo = oo * o;
  const size_t esz = bf ? 4 : 8;
  auto packed = [&](long long rows, int K) { return static_cast<size_t>(rows) * round_up(std::max(K, 1), 64) * esz; };
  auto al = [](size_t x) { return (std::max<size_t>(x, 256) + 255) / 256 * 256; };
  const int Kt = v + o;
  p.xt = packed(vv * o, Kt);
  p.to = packed(v * oo, Kt);
  p.ovoo = static_cast<size_t>(ooo * v * 8);
  p.pbvv = packed(vv, N);
  p.bc = static_cast<int>(std::max(1LL, std::min<long long>(v, (1LL << 26) / (o * vv))));
  p.ovvv_chunk = static_cast<size_t>(p.bc) * o * vv * 8;
  p.nblk = 0;
  for (int b = 0; b < v; ++b) p.nblk += 1LL * (b + 1) * (v - b);
  p.tpart = static_cast<size_t>(p.nblk + 256) * 2 * 8;  // block partials, then 256 first-pass sums
  p.batch = sizeof(BatchEntry) * static_cast<size_t>(std::max(1LL, vv / 2 + v));  // one entry per (b, c >= b)
  p.u = static_cast<size_t>(o) * 8 * 8;  // U padded to at most 8 LOs
  p.ovt = bf ? static_cast<size_t>(vv * oo) * 4 : 0;  // FP32 (ia|jb) in block-energy order (mixed)
  // W chunk: up to chunk_mb (fewer, larger contraction launches measured faster than chunks that fit
  // L2), but never more than the largest slab (b + 1)(v - b) o^2 jp needs, and at least one c of a slab
  long long max_slab = 0;
  for (int bb = 0; bb < v; ++bb) max_slab = std::max(max_slab, 1LL * (bb + 1) * (v - bb));
  const long long cmb = chunk_mb > 0 ? chunk_mb : 768;
  auto set_rows = [&](int jp) {  // rows of W of jp elements
    p.jp = jp;
    const long long most = std::min<long long>((cmb << 20) / static_cast<long long>(esz), max_slab * oo * jp);
    p.welems = std::max<long long>(most, v * oo * jp);
    p.w = static_cast<size_t>(p.welems) * esz;
  };
  set_rows(o);
  const size_t fixed = 2 * al(p.xt) + 2 * al(p.to) + al(p.ovoo) + al(p.pbvv) + al(p.ovvv_chunk) + al(p.tpart) +
                       2 * al(p.batch) + al(p.u) + (bf ? al(p.ovt) : 0);
  const size_t w_plain = al(p.w);
  p.need = fixed + w_plain;
  if (bf) {
    p.tri = static_cast<size_t>(tri_count(std::min(o, kMaxStagedOcc))) * 4;
    set_rows(round_up(o, 4));  // 16-byte rows for the copies
    p.alloc = fixed + al(p.w) + al(p.tri);
    const size_t over = al(p.w) - w_plain;
    const bool fits = al(p.tri) + over <= al(p.pbvv) + al(p.ovvv_chunk);
    p.total = fits ? p.need : p.alloc;
    if (avail > 0 && fits) {
      p.w_over = over;
      p.tri_over = true;
    } else if (avail > 0 && avail < p.total) {
      set_rows(o);
      p.tri = 0;
    }
  } else {
    const int Ktp = round_up(Kt, 64);
    const size_t slxt = slice_bytes(vv * o, Ktp, kFarDigits), slto = slice_bytes(v * oo, Ktp, kFarDigits);
    const size_t planes = 2 * al(slxt) + 2 * al(slto);
    p.total = p.need + (planes <= (size_t(32) << 30) ? planes : 0);
    p.alloc = p.total;
    if (p.total > p.need && (avail == 0 || avail >= p.total)) {
      p.slxt = slxt;
      p.slto = slto;
    }
  }
  return p;
}

int Frag::triples(int nlo, const double* U, double* e_full, double* e_frag, double* e_dev, int* st_dev) {
  const long long oo = 1LL * o * o, vv = 1LL * v * v, ov = 1LL * o * v, ooo = oo * o;
  const bool bf = mixed;
  // device-output mode: enqueue only (no host synchronisation, no event timing, no allocation, no
  // tile timing), so that the call can be captured into a CUDA graph; the energies and the device
  // status word are copied to the caller's device memory at the end of the stream's work
  const bool dev_out = e_dev != nullptr;
  const TriplesPlan tp = triples_plan(o, v, N, bf, opts.triples_chunk_mb, ws_ext ? ws_ext_bytes : 0);
  if (ws_ext && ws_ext_bytes < tp.need) {
    set_error("lnocc_triples: attached workspace smaller than lnocc_workspace_bytes (at least " + std::to_string(tp.need) +
              " bytes)");
    return LNOCC_EINVAL;
  }
  if (dev_out && !ws_ext) {
    set_error("lnocc_triples_device: attach a workspace first (lnocc_frag_set_workspace)");
    return LNOCC_EINVAL;
  }
  struct TimingGuard {  // no tile timing (it synchronises and allocates) in device-output mode
    bool saved, active;
    explicit TimingGuard(bool on) : saved(autotune_timing_allowed()), active(on) {
      if (active) autotune_timing_allowed() = false;
    }
    ~TimingGuard() {
      if (active) autotune_timing_allowed() = saved;
    }
  } timing_guard(dev_out);
  cudaMemsetAsync(dstatus, 0, 16 * 4, s);
  const double* t1 = xcur;
  const double* t2 = xcur + ov;
  cudaEvent_t ev_call0 = nullptr, ev_call1 = nullptr;
  if (!dev_out) {
    cudaEventCreate(&ev_call0);
    cudaEventCreate(&ev_call1);
    cudaEventRecord(ev_call0, s);
  }
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> gev;  // around each chunk's contraction launches

  // ---- operands (packed once per call)
  std::vector<void*> mine;
  size_t ws_used = 0;
  // temporaries: carved in plan order from the caller's workspace when one is attached (no device
  // allocation), else allocated in the fragment's memory mode and freed before returning
  auto tmp_alloc = [&](size_t bytes) -> void* {
    bytes = (std::max<size_t>(bytes, 256) + 255) / 256 * 256;
    if (ws_ext) {
      if (ws_used + bytes > ws_ext_bytes) return nullptr;
      void* p = static_cast<unsigned char*>(ws_ext) + ws_used;
      ws_used += bytes;
      return p;
    }
    void* p = dev_alloc(bytes);
    if (p) mine.push_back(p);
    return p;
  };
  auto cleanup = [&]() {
    if (!dev_out) cudaStreamSynchronize(s);
    for (void* p : mine) dev_free(p);
    if (ev_call0) cudaEventDestroy(ev_call0);
    if (ev_call1) cudaEventDestroy(ev_call1);
    ev_call0 = ev_call1 = nullptr;
  };
  auto mk = [&](int rows, int K) -> Packed {
    Packed P;
    P.rows = rows;
    P.Kp = round_up(std::max(K, 1), 64);
    P.bf16 = bf;
    P.p = tmp_alloc(static_cast<size_t>(rows) * P.Kp * (bf ? 4 : 8));
    if (P.p) cudaMemsetAsync(P.p, 0, static_cast<size_t>(rows) * P.Kp * (bf ? 4 : 8), s);
    return P;
  };
  // Each (T) term is d-part (K = v) + l-part (K = o): the two operands of a side share one packed row
  // space, so they are packed side by side along K (columns [0, v) and [v, v + o)) and every term is a
  // single contraction of length v + o (no second, mostly padded, K segment).
  //   XT1[x][a][i] = [ (ai|xd) | -t_il^ax ],   XT2[c][a][k] = [ (kc|ad) | -t_kl^ca ]
  //   TO[z][r][q]  = [ t_rq^zd | (zr|ql) ],     TOT[z][k][j] = [ t_jk^zd | (zj|kl) ]
  const int Kt = v + o;
  Packed XT1 = mk(static_cast<int>(vv * o), Kt), XT2 = mk(static_cast<int>(vv * o), Kt);
  Packed TO = mk(static_cast<int>(v * oo), Kt), TOT = mk(static_cast<int>(v * oo), Kt);
  double* ovoo = static_cast<double*>(tmp_alloc(ooo * v * 8));
  const double* dU = nlo > 0 ? U : nullptr;
  if (!XT1.p || !XT2.p || !TO.p || !TOT.p || !ovoo) {
    cleanup();
    set_error("lnocc_triples: device allocation failed (operands)");
    return LNOCC_ENOMEM;
  }
  const int wl = XT1.Kp - v;  // width of the l-part columns, zero padding included
  // amplitudes: TO[z][r][q][d] = t_rq^zd, TOT[z][k][j][d] = t_jk^zd (columns [0, v))
  pack_cols(view(t2, A_(v, v), A_(o, o * vv), A_(o, vv), kOne, kOne, A_(v, 1)), TO, 0, 0, v, s);
  pack_cols(view(t2, A_(v, v), A_(o, vv), A_(o, o * vv), kOne, kOne, A_(v, 1)), TOT, 0, 0, v, s);
  // (kz|jl) -> TO[z][k][j][v + l] = (zk|jl), TOT[z][k][j][v + l] = (zj|kl)
  contract(view(Bov, kOne, kOne, A_(static_cast<int>(ov), 1), kOne, kOne, A_(N, ov)),
           view(Boo, kOne, kOne, A_(static_cast<int>(oo), 1), kOne, kOne, A_(N, oo)), out_rowmajor(ovoo, oo), true);
  pack_cols(view(ovoo, A_(v, oo), A_(o, v * oo), A_(o, o), kOne, kOne, A_(o, 1)), TO, 0, v, wl, s);
  pack_cols(view(ovoo, A_(v, oo), A_(o, o), A_(o, v * oo), kOne, kOne, A_(o, 1)), TOT, 0, v, wl, s);
  // (jb|ad) -> XT2[b][a][j][d], in chunks of b; XT1[y][a][i][d] = (ai|yd) = XT2[a][y][i][d]
  void* dead = nullptr;  // start of the B_vv and (jb|ad) temporaries: free for others after this block
  {
    Packed PBvv = mk(static_cast<int>(vv), N);
    dead = PBvv.p;
    if (!PBvv.p) {
      cleanup();
      set_error("lnocc_triples: device allocation failed (B_vv)");
      return LNOCC_ENOMEM;
    }
    pack(view(Bvv, kOne, kOne, A_(static_cast<int>(vv), 1), kOne, kOne, A_(N, vv)), PBvv, s);
    const int bc = tp.bc;
    double* tmp = static_cast<double*>(tmp_alloc(tp.ovvv_chunk));
    if (!tmp) {
      cleanup();
      set_error("lnocc_triples: device allocation failed (ovvv chunk)");
      return LNOCC_ENOMEM;
    }
    const bool keep = mixed;
    mixed = bf;
    for (int b0 = 0; b0 < v; b0 += bc) {
      const int nb = std::min(bc, v - b0);
      contract_packed_b(view(Bov + b0, kOne, A_(o, v), A_(nb, 1), kOne, kOne, A_(N, ov)), PBvv, static_cast<int>(vv),
                        out_rowmajor(tmp, vv));
      pack_cols(view(tmp, A_(nb, vv), A_(v, v), A_(o, nb * vv), kOne, kOne, A_(v, 1)), XT2, b0 * v * o, 0, v, s);
    }
    mixed = keep;
    const int planes = bf ? 2 : 1;
    const int nvec = XT2.Kp * (bf ? 2 : 8) / 16;
    const long long nrows = static_cast<long long>(XT2.rows) * planes;
    const int blocks = static_cast<int>(std::min<long long>((nrows + 7) / 8, 152LL * 16));
    count_launch();
    k_swap_outer_rows<<<blocks, 256, 0, s>>>(static_cast<const uint4*>(XT2.p), static_cast<uint4*>(XT1.p), v, o,
                                             nvec, planes);
  }
  // l-parts (after the row swap, which copies whole rows): XT1[x][a][i][v + l] = -t_il^ax,
  // XT2[c][a][k][v + l] = -t_kl^ca (the l-terms enter W with a minus sign)
  pack_cols(view(t2, A_(v, 1), A_(v, v), A_(o, o * vv), kOne, kOne, A_(o, vv), -1.0), XT1, 0, v, wl, s);
  pack_cols(view(t2, A_(v, v), A_(v, 1), A_(o, o * vv), kOne, kOne, A_(o, vv), -1.0), XT2, 0, v, wl, s);

  // ---- slabs of fixed b: virtual c in [b, v) in chunks, a in [0, b]; W_chunk[c - c0][a][i][j][k]
  const size_t wsz = bf ? 4 : 8;
  const int jp = tp.jp;
  const long long ooj = oo * jp;  // W elements of one (c, a)
  const long long welems = tp.welems;
  void* W = nullptr;
  if (ws_ext && tp.w_over > 0) {
    W = static_cast<unsigned char*>(ws_ext) + ws_used - tp.w_over;
    ws_used += (std::max<size_t>(tp.w, 256) + 255) / 256 * 256 - tp.w_over;
  } else {
    W = tmp_alloc(tp.w);
  }
  const long long nblk_total = tp.nblk;
  double* tpart = static_cast<double*>(tmp_alloc(tp.tpart));
  // chunk plan and the per-c batch tables of the sigma2 / sigma5 terms (uploaded once)
  struct Chunk {
    int b, c0, nc;
    long long tab, part;
  };
  std::vector<Chunk> plan;
  long long ntab = 0;  // entries of the per-c tables: one per (b, c >= b), b-major
  {
    long long part = 0;
    for (int b = 0; b < v; ++b) {
      const long long slab = (b + 1) * ooj;  // W elements per c
      const int ncmax = static_cast<int>(std::max(1LL, welems / slab));
      for (int c0 = b; c0 < v; c0 += ncmax) {
        const int nc = std::min(ncmax, v - c0);
        plan.push_back(Chunk{b, c0, nc, ntab, part});
        ntab += nc;
        part += 1LL * (b + 1) * nc;
      }
    }
  }
  BatchEntry* dbat = static_cast<BatchEntry*>(tmp_alloc(tp.batch));
  BatchEntry* dbat12 = static_cast<BatchEntry*>(tmp_alloc(tp.batch));
  if (sizeof(BatchEntry) * static_cast<size_t>(ntab) > tp.batch) {
    cleanup();
    set_error("lnocc_triples: internal error (launch tables larger than planned)");
    return LNOCC_EINVAL;
  }
  if (!W || !tpart || !dbat || !dbat12) {
    cleanup();
    set_error("lnocc_triples: device allocation failed (W chunk)");
    return LNOCC_ENOMEM;
  }
  // grouped launches (two per chunk instead of five): nocc 16 and 32, where 128-row tiles hold whole a values
  // and a (y, z) plane is one or four 256-column tiles, in gemm.cu; any other nocc from 4 to 32 in triples_gemm.cu
  const bool grouped = bf && o >= 4 && o <= 32 && jp % 4 == 0 && opts.triples_kernel != LNOCC_TK_PER_TERM;
  if (!grouped) {  // the tables serve the batched per-term launches
    count_launch();
    k_batch_tables<<<(v + 127) / 128, 128, 0, s>>>(o, v, jp, welems, dbat, dbat12);
  }

  // Block energy kernel. Mixed: w and v staged side by side while they fit (nocc <= 28: 182 KB at 28), one
  // value per element up to nocc 37 (203 KB), at most 8 LOs; FP64: w and v or w alone within 200 KB.
  // Otherwise the generic kernel (any nocc and nlo, nothing staged).
  const long long sblk = 1LL * o * (1LL * o * (o + 1) + 1);  // padded w / v block of the FP64 kernel
  const long long small_smem = (3LL * o * (o + 1) + 4LL * o + 16LL * o + 4) * wsz;
  const bool staged_full = 2LL * sblk * wsz + small_smem <= 200LL * 1024;
  const bool staged =
      (bf ? o <= kMaxStagedOcc && tp.tri > 0 : staged_full || sblk * wsz + small_smem <= 200LL * 1024) && nlo <= 8;
  // the FP64 kernel is compiled for 0, 1, 2, 4 or 8 LOs: U zero-padded to the next size
  const int nlo_t = bf || nlo == 0 ? nlo : nlo <= 1 ? 1 : nlo <= 2 ? 2 : nlo <= 4 ? 4 : 8;
  const size_t esmem = (staged_full ? 2 : 1) * sblk * wsz + static_cast<size_t>(small_smem);  // FP64 kernel
  double* dUp = nullptr;
  if (staged && nlo_t > 0) {
    dUp = static_cast<double*>(tmp_alloc(tp.u));
    if (!dUp) {
      cleanup();
      set_error("lnocc_triples: device allocation failed (U)");
      return LNOCC_ENOMEM;
    }
    cudaMemsetAsync(dUp, 0, static_cast<size_t>(o) * nlo_t * 8, s);
    cudaMemcpy2DAsync(dUp, nlo_t * 8, U, nlo * 8, nlo * 8, o, cudaMemcpyDeviceToDevice, s);
  }
  float* ovT = nullptr;  // the FP32 kernels read (ia|jb) from this copy
  unsigned* tri = nullptr;
  if (bf && staged) {
    ovT = static_cast<float*>(tmp_alloc(tp.ovt));
    tri = static_cast<unsigned*>(ws_ext && tp.tri_over ? dead : tmp_alloc(tp.tri));
    if (!ovT || !tri) {
      cleanup();
      set_error("lnocc_triples: device allocation failed (ovT)");
      return LNOCC_ENOMEM;
    }
    count_launch(2);
    k_ovov_t<<<1216, 256, 0, s>>>(ovov, ovT, o, v);
    k_tri_table<<<1, 32, 0, s>>>(o, tri);
  }
  Sliced sls[4];
  if (tp.slxt > 0) {
    // allocated last: the call runs without them if they do not fit (triples_plan)
    Packed* ops[4] = {&XT1, &XT2, &TO, &TOT};
    void* mem[4];
    const size_t n_mine = mine.size();
    bool room = !(opts.fault_inject & LNOCC_FAULT_NO_PLANES);
    for (int k = 0; k < 4 && room; ++k) {
      mem[k] = tmp_alloc(k < 2 ? tp.slxt : tp.slto);
      room = mem[k] != nullptr;
    }
    if (room) {
      for (int k = 0; k < 4; ++k) {
        sls[k] = slice_at(mem[k], ops[k]->rows, ops[k]->Kp, static_cast<const double*>(ops[k]->p), ops[k]->Kp,
                          kFarDigits);
        slice(sls[k], s);
        ops[k]->sl = &sls[k];
      }
    } else {
      for (size_t k = n_mine; k < mine.size(); ++k) dev_free(mine[k]);
      mine.resize(n_mine);
    }
  }

  auto energy_launch = [&](const void* Wp, long long Sc, int b, int c0, int na, int nc, double* part) {
    if (bf) {
      launch_block_energy(EnergyArgs{static_cast<const float*>(Wp), Sc, b, c0, o, v, eps, t1, ovT, dUp, nlo, tri, part, na, nc},
                          s);
      return;
    }
    dim3 grid(na, nc);
    count_launch();
#define LN_D(K)                                                                                          \
  do {                                                                                                   \
    if (staged_full)                                                                                     \
      k_t_energy_staged<double, double, K, false><<<grid, 256, esmem, s>>>(static_cast<const double*>(Wp), Sc, \
                                                                           b, c0, o, v, eps, t1, ovov,   \
                                                                           dUp, nlo_t, part);            \
    else                                                                                                 \
      k_t_energy_staged<double, double, K, true><<<grid, 256, esmem, s>>>(static_cast<const double*>(Wp), Sc, \
                                                                          b, c0, o, v, eps, t1, ovov, dUp, \
                                                                          nlo_t, part);                  \
  } while (0)
    switch (nlo_t) {
      case 0: LN_D(0); break;
      case 1: LN_D(1); break;
      case 2: LN_D(2); break;
      case 4: LN_D(4); break;
      default: LN_D(8); break;
    }
#undef LN_D
  };
  if (staged && !bf) {
    // The attribute is per kernel and process-wide: set it once to the largest size a staged kernel can be
    // launched with, so that concurrent calls on fragments of other sizes never lower it under one
    // another's launches.
    static std::once_flag once;
    std::call_once(once, [] {
      auto attr = [](const void* fn, int bytes) {
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      };
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 0, false>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 1, false>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 2, false>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 4, false>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 8, false>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 0, true>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 1, true>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 2, true>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 4, true>), 200 * 1024);
      attr(reinterpret_cast<const void*>(k_t_energy_staged<double, double, 8, true>), 200 * 1024);
    });
  }
  auto omap = [&](double beta) {
    OutMap m{bf ? nullptr : static_cast<double*>(W), 0, 0, 0, 0, 1 << 30, 1 << 30, 1.0, beta};
    if (bf) m.dst32 = static_cast<float*>(W);
    return m;
  };
  const int o2 = static_cast<int>(oo);
  const long long oj = 1LL * o * jp;  // W strides: a ooj, i oj, k jp, j 1
  const Packed* ops_k2[4] = {&TO, &XT2, &XT2, &XT1};
  const Packed* ops_a[4] = {&XT1, &TO, &XT2, &TOT};
  const Packed* ops_b[4] = {&TO, &XT2, &TO, &XT1};
  const int box_ab[4] = {128, 256, 128, 256};
  // FP64 without planes: products that cut their operands per chunk take twelve digits like the planes
  const FarRows far_rows(bf ? FarRows::kNone : FarRows::kAll);
  // tuning passes (t_max_chunks > 0) visit about t_max_chunks chunks spread over the plan
  const size_t chunk_stride = t_max_chunks > 0 ? std::max<size_t>(1, plan.size() / t_max_chunks) : 1;
  size_t chunk_idx = 0;
  for (const Chunk& ch : plan) {
    if (chunk_idx++ % chunk_stride != 0) continue;
    const int b = ch.b, c0 = ch.c0, nc = ch.nc;
    const int na = b + 1, Ma = na * o, Ma2 = na * o2;
    const long long Sc = na * ooj;  // W stride of c
    const int xb = b * v * o;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (!dev_out) {
      cudaEventCreate(&e0);
      cudaEventCreate(&e1);
      cudaEventRecord(e0, s);
    }
    // W layout [c - c0][a][i][k][j]; each term is one contraction over K = v + o (d-part, then l-part).
    if (grouped && o != 16 && o != 32) {
      TgSpec g{};
      g.b = b;
      g.c0 = c0;
      g.nc = nc;
      g.o = o;
      g.bvo = xb;
      g.vo = v * o;
      g.Sc = Sc;
      g.kind = 1;
      gemm_grouped_any(ops_a, g, static_cast<float*>(W), Kt, s, dstatus);
      g.kind = 2;
      gemm_grouped_any(ops_k2, g, static_cast<float*>(W), Kt, s, dstatus);
    } else if (grouped) {
      // launch 1, per (c, 128-row tile of (a, x)): sigma1 + sigma2 stored, then sigma3 and sigma5 added
      // (the output maps of the per-term launches below, restricted to one c)
      GrpSpec g{};
      g.kind = 1;
      g.Ma = Ma;
      g.mt = (Ma + 127) / 128;
      g.nkb = XT1.Kp / 64;
      g.c0 = c0;
      g.nc = nc;
      g.cblk = 256 / o;
      g.ncol = o2 / 256;
      g.b = b;
      g.bvo = xb;
      g.vo = v * o;
      g.oo = o2;
      g.o = o;
      g.Sc = Sc;
      g.nreg = nc * g.mt;
      OutMap ca[3] = {omap(0.0), omap(1.0), omap(1.0)};
      ca[0].sm1 = ooo; ca[0].sm0 = oo; ca[0].mdiv = o; ca[0].sn1 = o; ca[0].sn0 = 1; ca[0].ndiv = o;   // (a,i) x (k,j)
      ca[1].sm1 = ooo; ca[1].sm0 = 1; ca[1].mdiv = o; ca[1].sn1 = o; ca[1].sn0 = oo; ca[1].ndiv = o;   // (a,j) x (k,i)
      ca[2].sm1 = ooo; ca[2].sm0 = o; ca[2].mdiv = o; ca[2].sn1 = oo; ca[2].sn0 = 1; ca[2].ndiv = o;   // (a,k) x (i,j)
      gemm_grouped(ops_a, box_ab, g, ca, 3, s, dstatus);
      // launch 2, per (128-row tile of (a, x, y), block of 256 / o values of c): sigma4 and sigma6 added
      GrpSpec h = g;
      h.kind = 2;
      h.Ma = Ma2;
      h.mt = (Ma2 + 127) / 128;
      h.nreg = h.mt * ((nc + g.cblk - 1) / g.cblk);
      OutMap cb[2] = {omap(1.0), omap(1.0)};
      cb[0].sm2 = ooo; cb[0].sm1 = oo; cb[0].sm0 = o; cb[0].mdiv = o; cb[0].mdiv1 = o;   // (a,i,k) x (c,j)
      cb[0].sn1 = Sc; cb[0].sn0 = 1; cb[0].ndiv = o;
      cb[1].sm2 = ooo; cb[1].sm1 = oo; cb[1].sm0 = 1; cb[1].mdiv = o; cb[1].mdiv1 = o;   // (a,i,j) x (c,k)
      cb[1].sn1 = Sc; cb[1].sn0 = o; cb[1].ndiv = o;
      gemm_grouped(ops_b, box_ab, h, cb, 2, s, dstatus);
    } else {
    // sigma1 + sigma2 (batched over c, two K segments into one accumulator; first writer of W):
    // rows (a,i), cols (k,j): (ai|bd) t_kj^cd - t_il^ab (ck|jl) + (ai|cd) t_jk^bd - t_il^ac (bj|kl)
    {
      OutMap m = omap(0.0);
      m.sm1 = ooj; m.sm0 = oj; m.mdiv = o;
      m.sn1 = jp; m.sn0 = 1; m.ndiv = o;
      gemm2_batched(XT1, TO, &XT1, &TOT, dbat12 + ch.tab, nc, Ma, o2, Kt, Kt, m, s, dstatus);
    }
    // sigma3: rows (a,j), cols (c,k,i): (bj|ad) t_ki^cd - t_jl^ba (ck|il)
    {
      OutMap m = omap(1.0);
      m.sm1 = ooj; m.sm0 = 1; m.mdiv = o;
      m.sn2 = Sc; m.sn1 = jp; m.sn0 = oj; m.ndiv = o; m.ndiv1 = o;
      gemm_off(XT2, xb, TO, c0 * o2, Ma, nc * o2, Kt, m, s, dstatus);
    }
    // sigma4: rows (a,i,k), cols (c,j): t_ik^ad (bj|cd) - (ai|kl) t_jl^bc
    {
      OutMap m = omap(1.0);
      m.sm2 = ooj; m.sm1 = oj; m.sm0 = jp; m.mdiv = o; m.mdiv1 = o;
      m.sn1 = Sc; m.sn0 = 1; m.ndiv = o;
      gemm_off(TO, 0, XT2, xb + c0 * o, Ma2, nc * o, Kt, m, s, dstatus);
    }
    // sigma6: rows (a,i,j), cols (c,k): t_ij^ad (ck|bd) - (ai|jl) t_kl^cb
    {
      OutMap m = omap(1.0);
      m.sm2 = ooj; m.sm1 = oj; m.sm0 = 1; m.mdiv = o; m.mdiv1 = o;
      m.sn1 = Sc; m.sn0 = jp; m.ndiv = o;
      gemm_off(TO, 0, XT1, xb + c0 * o, Ma2, nc * o, Kt, m, s, dstatus);
    }
    // sigma5 (batched over c): rows (a,k), cols (i,j): (ck|ad) t_ji^bd - t_kl^ca (bj|il)
    // (TOT[b][i][j] = [t_ji^bd | (bj|il)]: j runs fastest in the columns)
    {
      OutMap m = omap(1.0);
      m.sm1 = ooj; m.sm0 = jp; m.mdiv = o;
      m.sn1 = oj; m.sn0 = 1; m.ndiv = o;
      gemm_batched(XT2, TOT, dbat + ch.tab, nc, Ma, o2, Kt, m, s, dstatus);
    }
    }
    if (!dev_out) {
      cudaEventRecord(e1, s);
      gev.emplace_back(e0, e1);
    }
    if (staged) {
      energy_launch(W, Sc, b, c0, na, nc, tpart + 2 * ch.part);
    } else {
      count_launch();
      if (bf)
        k_t_energy<float><<<dim3(na, nc), 128, 0, s>>>(static_cast<const float*>(W), Sc, b, c0, o, v, eps, t1, ovov,
                                                       dU, nlo, tpart + 2 * ch.part, jp);
      else
        k_t_energy<double><<<dim3(na, nc), 128, 0, s>>>(static_cast<const double*>(W), Sc, b, c0, o, v, eps, t1,
                                                        ovov, dU, nlo, tpart + 2 * ch.part, jp);
    }
  }
  {
    constexpr int kParts = 256;  // first-pass blocks; their sums sit after the nblk block partials
    const long long chunk = (nblk_total + kParts - 1) / kParts;
    count_launch(2);
    k_t_finish_part<<<kParts, 1024, 0, s>>>(tpart, nblk_total, chunk, tpart + 2 * nblk_total);
    k_t_finish<<<1, 1024, 0, s>>>(tpart + 2 * nblk_total, kParts, scal + 4);
  }
  if (dev_out) {
    // E_T and E_T^(F) (zero without LOs: the kernels sum no projected terms then) and the status word
    cudaMemcpyAsync(e_dev, scal + 4, 16, cudaMemcpyDeviceToDevice, s);
    if (st_dev) cudaMemcpyAsync(st_dev, dstatus, 4, cudaMemcpyDeviceToDevice, s);
    cleanup();
    const cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) {
      set_error(std::string("lnocc_triples_device: ") + cudaGetErrorString(ce));
      return LNOCC_ECUDA;
    }
    return LNOCC_OK;
  }
  cudaMemcpyAsync(h_scal + 4, scal + 4, 16, cudaMemcpyDeviceToHost, s);
  cudaEventRecord(ev_call1, s);
  cudaStreamSynchronize(s);
  {
    float ms = 0.f;
    t_gemm_ms = 0.0;
    for (auto& pr : gev) {
      cudaEventElapsedTime(&ms, pr.first, pr.second);
      t_gemm_ms += ms;
      cudaEventDestroy(pr.first);
      cudaEventDestroy(pr.second);
    }
    cudaEventElapsedTime(&ms, ev_call0, ev_call1);
    t_triples_ms = ms;
  }
  const int st = check_device();
  if (e_full) *e_full = h_scal[4];
  if (e_frag) *e_frag = nlo > 0 ? h_scal[5] : 0.0;
  cleanup();
  if (st == LNOCC_OK && !std::isfinite(h_scal[4])) {
    set_error("non-finite (T) energy");
    return LNOCC_ENUMERIC;
  }
  return st;
}

}  // namespace lnocc
