// FP64 contractions on the BF16 tensor pipe.
//
// GB300 runs FP64 at two FMA lanes per clock and SM, a thousandth of its BF16 tensor rate, so an FP64
// product is formed from exact BF16 products instead, after Ozaki, Ogita, Oishi and Rump (Numer.
// Algorithms 59, 95 (2012)) and its tensor-core form (Mukunoki et al., ISC 2020):
//   * Each operand row is cut into chunks of kChunk = 512 columns. A chunk shares one exponent E (all
//     |x| < 2^E) and every x 2^-E becomes P balanced radix-128 digits (nine, or twelve where the caller says that
//     rows decay away from centres far apart), x = 2^(E-6) sum_i d_i 2^(-7(i-1)), integers in [-64, 64]; plane i
//     holds d_i 2^(-7(i-1)), exact in BF16.
//   * A(m, :) . B(n, :) = 2^(Ea+Eb-12) sum_g S_g with S_g the digit products of i + j = g + 1, one FP32 TMEM
//     accumulator per g = 1..P. Every term of S_g is an integer times 2^(-7(g-1)) and |S_g| <= g 512 64 64 <= 2^24
//     units for g <= 8, so the accumulation is exact; beyond, it can round at 2^-68 of 2^(Ea+Eb), and only if nearly all
//     digits of both rows are large.
//   * The epilogue adds the accumulators as one integer and rounds it once to FP64.
// What is dropped is absolute in 2^(Ea+Eb): the pairs i + j > P + 1, in root mean square sqrt(K (P - 1)) 2^(-1.6 - 7 P)
// (digits uniform; 2^-63.1 sqrt(K) with nine, 2^-83.9 with twelve), and what of the operands lies below the last
// digit. An FP64 FMA chain instead errs relative to T = sum |a||b| of the element: at least about 0.6 2^-53 T. So
// that no element is less exact than by the chain, one more plane holds |x| 2^-E, one more accumulator sums T, and an
// element with T below a line of 2^-9 sqrt(K) 2^(Ea+Eb) (twelve digits: 2^-29), where the digits would give less, is
// summed in FP64 from the packed operands. (At that line the digits' error is 0.5 2^-53 T.) T = 0 means that no nonzero
// meets another: zero exactly.
// On the library's operands 0 to 0.3% of the elements fall below the first line up to about 100 virtuals (half in
// three products whose rows decay away from a centre: amplitudes times F_vv and the two rotations of B into an
// active space), 14 to 48% at 240 virtuals in the ladder, the rings, Z and (T); those take twelve digits.
// Eight planes and no such check (128 x 64 tiles) were somewhat faster, 3 CCSD iterations at (12, 96, 320) 11.8 instead of
// 13.4 ms, (T) at (8, 64, 256) 15.1 instead of 15.6, the LNO space of (16, 160, 640) 14.0 instead of 14.9 ms, an FP64 solve
// of (16, 240, 960) 3.5 instead of 5.6 s, but an element 1e-16 of its row's largest was kept to 6e-3. The SIMT kernel:
// 131.6, 67.1, 30.4 ms and 45 s.
// Rows whose chunk holds an infinity, a NaN, or only subnormal values are marked and summed in FP64 too.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>

#include "gemm_slices.h"
#include "internal.h"
#include "out_map.cuh"
#include "ptx.cuh"

namespace lnocc {
namespace {

constexpr int kChunk = kSliceChunk;     // columns that share an exponent and an exact accumulation
constexpr int kBadExp = 0x40000000;     // chunk that cannot be sliced

// Tile, pipeline and epilogue of products with P digits. P + 1 accumulators of BN columns fit the 512 TMEM columns;
// a stage holds the P + 1 planes of both operands, BK columns wide (12 digits: 65 KB of 16 columns).
template <int P>
struct Sl {
  static constexpr int BM = 128, BN = P == 9 ? 48 : 32, BK = P == 9 ? 32 : 16, STAGES = P == 9 ? 2 : 3;
  static constexpr int A_BYTES = (P + 1) * BM * BK * 2, B_BYTES = (P + 1) * BN * BK * 2, STAGE = A_BYTES + B_BYTES;
  static constexpr int PER_MMA = 256 / BN;  // planes of B one MMA multiplies (48: N = 240, 32: N = 256)
  static constexpr int EPI_WARPS = P == 9 ? 16 : 8, THREADS = 128 + 32 * EPI_WARPS;
  static constexpr int UNITS = 2 * (BN / 8) / (EPI_WARPS / 4);  // units of 16 rows x 8 columns of one epilogue warp
  static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
  static constexpr int LO_BITS = 7 * (P - 6);  // bits of the digit sum below its 64-bit part
  // T below this, times sqrt(K), is summed in FP64: 2^54.1 sqrt(P - 1) 2^(-1.6 - 7 P), rounded up
  static constexpr float LINE = P == 9 ? 0x1p-9f : 0x1p-29f;
  static_assert(P == 9 || P == 12, "digits");
  static_assert(SMEM <= 232448 && (P + 1) * BN <= 512 && STAGE % 1024 == 0 && A_BYTES % 1024 == 0, "tile");
};

// ---------------------------------------------------------------------------------------------
// Slicing: one warp per (row, chunk), 16 columns per lane, one read of the source. One launch cuts both
// operands of a product (the items of the second follow those of the first).
struct SliceJob {
  const double* src;
  long long ld;
  int rows, Kp;
  __nv_bfloat16* out;
  int* ex;
};
template <int P>
__global__ void __launch_bounds__(256) k_slice(const SliceJob j0, const SliceJob j1) {
  const int lane = threadIdx.x % 32;
  const long long n0 = static_cast<long long>(j0.rows) * ((j0.Kp + kChunk - 1) / kChunk);
  const long long items = n0 + static_cast<long long>(j1.rows) * ((j1.Kp + kChunk - 1) / kChunk);
  const long long nw = static_cast<long long>(gridDim.x) * blockDim.x / 32;
  for (long long i = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) / 32; i < items; i += nw) {
    const SliceJob& j = i < n0 ? j0 : j1;
    const long long it = i < n0 ? i : i - n0, ld = j.ld, plane = static_cast<long long>(j.rows) * j.Kp;
    const int Kp = j.Kp, ex_rows = j.rows, nch = (Kp + kChunk - 1) / kChunk;
    int* ex = j.ex;
    __nv_bfloat16* out = j.out;
    const int r = static_cast<int>(it / nch), ch = static_cast<int>(it % nch);
    const int k0 = ch * kChunk, kw = min(kChunk, Kp - k0);  // kw is a multiple of 64
    const double* s = j.src + r * ld + k0;
    double2 x[8];
    unsigned emax = 0, any = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int k = 2 * (lane + 32 * t);
      x[t] = k < kw ? *reinterpret_cast<const double2*>(s + k) : make_double2(0.0, 0.0);
      const unsigned h0 = static_cast<unsigned>(__double2hiint(x[t].x)) & 0x7fffffffu;
      const unsigned h1 = static_cast<unsigned>(__double2hiint(x[t].y)) & 0x7fffffffu;
      emax = max(emax, max(h0, h1));
      any |= h0 | h1 | static_cast<unsigned>(__double2loint(x[t].x)) | static_cast<unsigned>(__double2loint(x[t].y));
    }
    emax = __reduce_max_sync(0xffffffffu, emax) >> 20;
    any = __reduce_or_sync(0xffffffffu, any);
    const bool bad = emax == 0x7ffu || (emax == 0u && any != 0u);
    if (lane == 0) ex[static_cast<long long>(ch) * ex_rows + r] = bad ? kBadExp : static_cast<int>(emax) - 1022;
    __nv_bfloat16* o = out + static_cast<long long>(r) * Kp + k0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = 2 * (lane + 32 * q);
      if (k >= kw) break;
      // x 2^-E as nine digits of 62 fraction bits in all, rounded. With twelve, the nine start at the first plane that
      // the element reaches (first), so that it keeps its 53 bits down to the last one.
      long long F[2];
      int first[2];
      float t[2];  // |x| 2^-E; a nonzero keeps at least 2^-60, so that no product of two of them is lost
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long u = __double_as_longlong(h ? x[q].y : x[q].x);
        const int e = static_cast<int>(u >> 52) & 0x7ff;
        long long m = (u & 0xfffffffffffffLL) | (e > 0 ? 0x10000000000000LL : 0);
        int sh = static_cast<int>(emax) + 1 - max(e, 1);  // >= 1: x 2^-E = m 2^(-52 - sh)
        const float a = m == 0 ? 0.f : fmaxf(static_cast<float>(m >> 24) * __int_as_float((127 - 28 - min(sh, 60)) << 23), 0x1p-60f);
        first[h] = P > 9 ? min(P, (sh - 1) / 7) : 0;
        sh -= 7 * first[h];
        m = sh <= 10 ? m << (10 - sh) : (sh < 65 ? (m + (1LL << (sh - 11))) >> (sh - 10) : 0);
        F[h] = bad ? 0 : (u < 0 ? -m : m);
        t[h] = bad ? 0.f : a;
      }
      float w = 1.f;
#pragma unroll
      for (int i = 1; i <= P; ++i) {
        float f[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          long long d = 0;
          const int sft = 63 - 7 * (i - first[h]);
          if (P == 9 || (sft >= 0 && sft < 63)) {
            d = sft > 0 ? (F[h] + (1LL << (sft > 0 ? sft - 1 : 0))) >> sft : F[h];
            F[h] -= d << sft;
          }
          // d in [-64, 64] to FP32 through the exponent of 1.5 2^23, scaled by the plane's weight (exact)
          const float g = __int_as_float(0x4B400000 + static_cast<int>(d));
          f[h] = fmaf(g, w, -12582912.f * w);
        }
        *reinterpret_cast<__nv_bfloat162*>(o + (i - 1) * plane + k) = __floats2bfloat162_rn(f[0], f[1]);
        w *= 0.0078125f;
      }
      *reinterpret_cast<__nv_bfloat162*>(o + P * plane + k) = __floats2bfloat162_rn(t[0], t[1]);
    }
  }
}

// ---------------------------------------------------------------------------------------------
struct SlArgs {
  int M, N;
  int a_row0, b_row0;       // first rows in the sliced operands
  int mbase, nbase;         // output row / column of local row / column 0
  int nkb, kper;            // K blocks of this launch and per work item (kper divides those of a chunk)
  int kblk0;                // first K block in the operands
  int tiles_m, tiles_n, tiles_z;
  int sym;                  // C = A A^T: tiles on or above the diagonal, mirrored
  int tri, tri_row0;        // tri > 0: only columns n with n / tri <= (tri_row0 + m) / tri are needed
  const int *ea, *eb;       // chunk exponents [chunk][rows]
  int ea_rows, eb_rows;
  const double *A64, *B64;  // the packed FP64 operands (rows as a_row0 / b_row0), for elements summed in FP64
  long long lda, ldb;
  int asign, ashift;        // alpha = asign 2^ashift when asign != 0, else C.alpha multiplies
  OutMap C;
  double* ws;               // split-K partials [z][M][N], or null
  const BatchEntry* batch;  // one problem per z
  int seg;
  int* status;
};

struct SlTile {
  int m0, n0, z, M, a0, b0, kb0, nkb;
  long long cbase;
};

// Work item t; false for an empty one (outside the problem, below the diagonal).
template <int P>
__device__ __forceinline__ bool sl_tile(const SlArgs& p, int t, SlTile& ti) {
  constexpr int kBM = Sl<P>::BM, kBN = Sl<P>::BN;
  const int tm = t % p.tiles_m, tn = (t / p.tiles_m) % p.tiles_n;
  ti.z = t / (p.tiles_m * p.tiles_n);
  ti.m0 = tm * kBM;
  ti.n0 = tn * kBN;
  ti.M = p.M;
  ti.a0 = p.a_row0;
  ti.b0 = p.b_row0;
  ti.cbase = 0;
  ti.kb0 = ti.z * p.kper;
  if (p.batch) {
    const BatchEntry be = p.batch[ti.z];
    ti.M = be.M;
    ti.a0 = p.seg ? be.a_row1 : be.a_row0;
    ti.b0 = p.seg ? be.b_row1 : be.b_row0;
    ti.cbase = be.cbase;
    ti.kb0 = 0;
  }
  ti.nkb = min(p.kper, p.nkb - ti.kb0);
  ti.kb0 += p.kblk0;
  if (p.sym && p.nbase + ti.n0 + kBN <= p.mbase + ti.m0) return false;
  if (p.tri > 0 && (p.nbase + ti.n0) / p.tri > (p.tri_row0 + p.mbase + min(ti.m0 + kBM, p.M) - 1) / p.tri) return false;
  return ti.m0 < ti.M && ti.nkb > 0;
}

// 16 lanes x 8 columns: lane l of the warp gets (row l / 4, columns 2 (l % 4), + 1), then the same of row l / 4 + 8.
__device__ __forceinline__ void tmem_ld_16x8(uint32_t taddr, float (&v)[4]) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
template <int G>
__device__ __forceinline__ void tmem_wait_ld(float (&v)[G][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  // the loaded values are only defined after the wait: tie them to it
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int i = 0; i < 4; ++i) asm volatile("" : "+f"(v[g][i]));
}

// X = hi 2^L + lo (0 <= lo < 2^L, L = LO_BITS) in units of 2^(-47 - L): the sum of the accumulators.
template <int P>
__device__ __forceinline__ void sl_combine(const float* a, long long& hi, unsigned long long& lo) {
  const int s1 = __float2int_rn(a[0]), s2 = __float2int_rn(a[1] * 0x1p7f), s3 = __float2int_rn(a[2] * 0x1p14f);
  const int s4 = __float2int_rn(a[3] * 0x1p21f), s5 = __float2int_rn(a[4] * 0x1p28f), s6 = __float2int_rn(a[5] * 0x1p35f);
  // |s1| <= 2^21, |s2| <= 2^22, ..., |s8| <= 2^24: each of these pairs fits 32 bits
  const int p1 = s1 * 128 + s2, p2 = s3 * 128 + s4, p3 = s5 * 128 + s6;
  const int s7 = __float2int_rn(a[6] * 0x1p42f), s8 = __float2int_rn(a[7] * 0x1p49f), s9 = __float2int_rn(a[8] * 0x1p56f);
  long long t = static_cast<long long>(s7) * (1 << 14) + (static_cast<long long>(s8) * 128 + s9);
  if constexpr (P == 12) {
    const int s10 = __float2int_rn(a[9] * 0x1p63f), s11 = __float2int_rn(a[10] * 0x1p70f), s12 = __float2int_rn(a[11] * 0x1p77f);
    const long long z = static_cast<long long>(s10) * (1 << 14) + (static_cast<long long>(s11) * 128 + s12);
    t += z >> 21;
    lo = static_cast<unsigned long long>(t & 0x1fffff) << 21 | static_cast<unsigned long long>(z & 0x1fffff);
  } else {
    lo = static_cast<unsigned long long>(t & 0x1fffff);
  }
  hi = static_cast<long long>(p1) * (1 << 28) + (static_cast<long long>(p2) * (1 << 14) + p3) + (t >> 21);
}

// (hi 2^L + lo) 2^(e - 47 - L) rounded once to FP64; flip changes the sign.
template <int L>
__device__ __forceinline__ double sl_round(long long hi, unsigned long long lo, int e, bool flip) {
  bool neg = hi < 0;
  if (neg) {
    hi = lo ? ~hi : -hi;
    lo = ((1ull << L) - lo) & ((1ull << L) - 1);
  }
  unsigned long long m;
  int lz;
  if (hi != 0) {
    lz = __clzll(hi);
    m = (static_cast<unsigned long long>(hi) << lz) | (lz >= L ? lo << (lz - L) : lo >> (L - lz));
  } else if (lo != 0) {
    lz = __clzll(static_cast<long long>(lo)) + L;
    m = lo << (lz - L);
  } else {
    return 0.0;
  }
  neg ^= flip;
  // value = m 2^(-lz) 2^(e - 47), the top bit of m set
  const int be = 63 - lz + e - 47 + 1023;
  const unsigned long long f = (m >> 11) + ((m >> 10) & 1ull);
  if (be >= 1 && be < 2046)
    return __longlong_as_double(static_cast<long long>((static_cast<unsigned long long>(be - 1) << 52) + f) |
                                (neg ? static_cast<long long>(0x8000000000000000ull) : 0ll));
  const double r = ldexp(static_cast<double>(f), be - 1023 - 52);
  return neg ? -r : r;
}

// FP64 sums in place of the digits' for the elements of a warp's unit of 16 rows x 8 columns that `need` marks
// (bit 2 r + c: row r_lane + 8 r, column c_lane + c of this lane's four), from the packed operands' rows
// (a0, b0: the lane's first ones; 8 lda and ldb further on the others), k columns. Four elements at a
// time, eight lanes each: FP64-pipe work is k / 8 + 3 instructions per four elements, half of what a walk of every
// lane over its own four would take when half of the unit is marked, and no more when all is.
__device__ __noinline__ void sl_dot64(const double* a0, long long lda8, const double* b0, long long ldb, int k, unsigned need,
                                      double (&r)[4]) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, sub = lane & 7;
  unsigned any = __ballot_sync(0xffffffffu, need != 0u);
  while (any) {
    // group g takes the first marked element of the g-th marked lane
    unsigned t = any;
    for (int q = 0; q < grp; ++q) t &= t - 1;
    const int src = t ? __ffs(t) - 1 : lane, e = need ? __ffs(need) - 1 : 0;
    const unsigned long long x = reinterpret_cast<unsigned long long>((e & 2) ? a0 + lda8 : a0);
    const unsigned long long y = reinterpret_cast<unsigned long long>((e & 1) ? b0 + ldb : b0);
    const double* xs = reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, x, src)) + 2 * sub;
    const double* ys = reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, y, src)) + 2 * sub;
    double acc = 0.0;
    if (t) {
#pragma unroll 4
      for (int q = 0; q < k; q += 16) {
        const double2 u = *reinterpret_cast<const double2*>(xs + q), v = *reinterpret_cast<const double2*>(ys + q);
        acc = fma(u.y, v.y, fma(u.x, v.x, acc));
      }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    const int rank = __popc(any & ((1u << lane) - 1u));
    const double got = __shfl_sync(0xffffffffu, acc, 8 * (rank & 3));
    if (need && rank < 4) {
#pragma unroll
      for (int h = 0; h < 4; ++h)
        if (h == e) r[h] = got;
      need &= need - 1;
    }
    any = __ballot_sync(0xffffffffu, need != 0u);
  }
}

// Persistent: warp 0 TMA producer, warp 1 MMA issuer, warp 2 TMEM owner, the others epilogue (16 or 8 warps, over the
// TMEM lane quadrants: the accumulators nearly fill TMEM, so the next tile's products wait until all are read).
// Accumulator g of a tile sits at TMEM column BN (g - 1), T last, and the digit planes of B sit one after the
// other in shared memory, so one MMA of N = 240 or 256 multiplies plane i of A with five or eight planes of B into as
// many neighbouring accumulators: A is read once per five or eight products.
template <int P>
__global__ void __launch_bounds__(Sl<P>::THREADS, 1) k_gemm_sl(const __grid_constant__ CUtensorMap tA,
                                                               const __grid_constant__ CUtensorMap tB, const SlArgs p) {
  using C_ = Sl<P>;
  constexpr int kBM = C_::BM, kBN = C_::BN, kBK = C_::BK, kStages = C_::STAGES, kABytes = C_::A_BYTES,
                kStageBytes = C_::STAGE, kEpiWarps = C_::EPI_WARPS, kEpiUnits = C_::UNITS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* accf = empty + kStages;
  uint64_t* acce = accf + 1;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(acce + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int ntiles = p.tiles_m * p.tiles_n * p.tiles_z;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, 32 * kEpiWarps);
    fence_barrier_init();
    prefetch_tensormap(&tA);
    prefetch_tensormap(&tB);
  }
  if (warp == 2) tmem_alloc(tmem_holder, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == 0 && lane == 0) {
    int g = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < ntiles; t += gridDim.x) {
      SlTile ti;
      if (!sl_tile<P>(p, t, ti)) continue;
      for (int kb = 0; kb < ti.nkb; ++kb, ++g) {
        const int s = g % kStages;
        if (g >= kStages && !mbar_wait(&empty[s], ((g / kStages) - 1) & 1)) {
          atomicExch(p.status, kDevTimeoutProducer);
          ok = false;
          break;
        }
        uint8_t* st = smem + s * kStageBytes;
        mbar_arrive_expect_tx(&full[s], kStageBytes);
        const int kc = (ti.kb0 + kb) * kBK;
        tma_load_3d(st, &tA, &full[s], kc, ti.a0 + ti.m0, 0);
        tma_load_3d(st + kABytes, &tB, &full[s], kc, ti.b0 + ti.n0, 0);
      }
    }
    for (int q = (g > kStages ? g - kStages : 0); q < g; ++q) mbar_wait(&full[q % kStages], (q / kStages) & 1);
  } else if (warp == 1 && lane == 0) {
    int g = 0, it = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < ntiles; t += gridDim.x) {
      SlTile ti;
      if (!sl_tile<P>(p, t, ti)) continue;
      if (it > 0 && !mbar_wait(acce, (it - 1) & 1)) {
        atomicExch(p.status, kDevTimeoutMma);
        break;
      }
      tc_fence_after();
      for (int kb = 0; kb < ti.nkb; ++kb, ++g) {
        const int s = g % kStages;
        if (!mbar_wait(&full[s], (g / kStages) & 1)) {
          atomicExch(p.status, kDevTimeoutMma);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t a0 = smem_u32(smem + s * kStageBytes), b0 = a0 + kABytes;
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          const uint32_t off = kk * 32;
          const uint32_t first = (kb | kk) != 0 ? 1u : 0u;
#pragma unroll
          for (int i = 0; i < P; ++i) {
            // plane i of A against planes 0 .. P - 1 - i of B: accumulators i .. P - 1
            const uint64_t da = sdesc_k<kBK>(a0 + i * (kBM * kBK * 2) + off);
#pragma unroll
            for (int j = 0; j < P - i; j += C_::PER_MMA) {
              const int nj = P - i - j < C_::PER_MMA ? P - i - j : C_::PER_MMA;
              mma_bf16(tmem + (i + j) * kBN, da, sdesc_k<kBK>(b0 + j * (kBN * kBK * 2) + off),
                       idesc_bf16_f32(kBM, nj * kBN), i == 0 ? first : 1u);
            }
          }
          // T
          mma_bf16(tmem + P * kBN, sdesc_k<kBK>(a0 + P * (kBM * kBK * 2) + off),
                   sdesc_k<kBK>(b0 + P * (kBN * kBK * 2) + off), idesc_bf16_f32(kBM, kBN), first);
        }
        mma_commit(&empty[s]);
      }
      mma_commit(accf);
      ++it;
    }
  } else if (warp >= 4) {
    const int ew = warp - 4, quad = ew & 3, part = ew >> 2;
    const OutMap C = p.ws ? OutMap{p.ws, 0, p.N, 0, 1, 1 << 30, 1 << 30, 1.0, 0.0} : p.C;
    const int mb = p.ws ? 0 : p.mbase, nb = p.ws ? 0 : p.nbase;  // split-K partials are local
    const bool flip = !p.ws && p.asign < 0;
    const int ash = p.ws ? 0 : p.ashift;
    const bool mul = !p.ws && p.asign == 0;
    int it = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      SlTile ti;
      if (!sl_tile<P>(p, t, ti)) continue;
      if (!mbar_wait(accf, it & 1)) {
        if (lane == 0) atomicExch(p.status, kDevTimeoutEpilogue);
        break;
      }
      ++it;
      tc_fence_after();
      const int ch = ti.kb0 / (kChunk / kBK), kcol = ti.nkb * kBK;
      const long long cb = ti.cbase + (p.ws ? static_cast<long long>(ti.z) * p.M * p.N : 0);
      const float thr = C_::LINE * sqrtf(static_cast<float>(kcol));
      const uint32_t acc = tmem + (static_cast<uint32_t>(quad * 32) << 16);
      auto put = [&](long long off, double x) {
        if (C.dst32) {
          float y = static_cast<float>(x);
          if (C.beta != 0.0) y += static_cast<float>(C.beta) * C.dst32[off];
          C.dst32[off] = y;
        } else if (C.beta == 0.0) {
          C.dst[off] = x;
        } else if (C.beta == 1.0) {
          asm volatile("red.global.add.f64 [%0], %1;" ::"l"(C.dst + off), "d"(x) : "memory");
        } else {
          C.dst[off] = x + C.beta * C.dst[off];
        }
      };
      // unit: rows [16 half, + 16) of the quadrant, columns [8 grp, + 8) of the tile; a lane has rows m, m + 8 and
      // columns n, n + 1 of it, na and nb2 of them inside
      int m, n, na, nb2;
      auto unit_at = [&](int x) {
        const int unit = part + x * (kEpiWarps / 4);
        m = ti.m0 + quad * 32 + 16 * (unit & 1) + lane / 4;
        n = ti.n0 + 8 * (unit >> 1) + 2 * (lane & 3);
        na = m + 8 < ti.M ? 2 : m < ti.M ? 1 : 0;
        nb2 = n + 1 < p.N ? 2 : n < p.N ? 1 : 0;
      };
      auto store = [&](const double (&r)[4], unsigned which) {
        long long moff[2], noff[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          moff[h] = h < na ? cb + out_moff(C, mb + m + 8 * h) : 0;
          noff[h] = h < nb2 ? out_noff(C, nb + n + h) : 0;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int mm = mb + m + 8 * (e >> 1), nn = nb + n + (e & 1);
          if (!(which >> e & 1u) || (e >> 1) >= na || (e & 1) >= nb2 || (p.sym && nn < mm)) continue;
          put(moff[e >> 1] + noff[e & 1], r[e]);
          if (p.sym && nn > mm) put(cb + out_moff(C, nn) + out_noff(C, mm), r[e]);
        }
      };
      unsigned todo = 0;  // four bits per unit: elements to be summed in FP64
#pragma unroll 1
      for (int x = 0; x < kEpiUnits; ++x) {
        const int unit = part + x * (kEpiWarps / 4);
        float v[P + 1][4];
#pragma unroll
        for (int g = 0; g <= P; ++g)
          tmem_ld_16x8(acc + (static_cast<uint32_t>(16 * (unit & 1)) << 16) + g * kBN + 8 * (unit >> 1), v[g]);
        tmem_wait_ld(v);
        if (x == kEpiUnits - 1) {  // everything read: the next tile's products may start
          tc_fence_before();
          mbar_arrive(acce);
        }
        if (ti.m0 + quad * 32 + 16 * (unit & 1) >= ti.M || ti.n0 + 8 * (unit >> 1) >= p.N) continue;  // nothing inside
        unit_at(x);
        int ea[2], eb[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ea[h] = h < na ? p.ea[static_cast<long long>(ch) * p.ea_rows + ti.a0 + m + 8 * h] : 0;
          eb[h] = h < nb2 ? p.eb[static_cast<long long>(ch) * p.eb_rows + ti.b0 + n + h] : 0;
        }
        double r[4];
        unsigned bad = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {  // row e / 2, column e % 2
          float a[P];
#pragma unroll
          for (int g = 0; g < P; ++g) a[g] = v[g][e];
          long long hi;
          unsigned long long lo;
          sl_combine<P>(a, hi, lo);
          const int xa = ea[e >> 1], xb = eb[e & 1];
          const float T = v[P][e];
          const bool f = xa == kBadExp || xb == kBadExp || (T > 0.f && T < thr);
          bad |= f ? 1u << e : 0u;
          r[e] = sl_round<C_::LO_BITS>(hi, lo, f ? 0 : xa + xb + ash, flip);
          if (mul) r[e] *= C.alpha;
        }
        store(r, ~bad);
        if (na < 2) bad &= na == 0 ? 0u : 3u;
        if (nb2 < 2) bad &= nb2 == 0 ? 0u : 5u;
        todo |= bad << (4 * x);
      }
      if (__any_sync(0xffffffffu, todo != 0u)) {
#pragma unroll 1
        for (int x = 0; x < kEpiUnits; ++x) {
          const unsigned need = todo >> (4 * x) & 15u;
          if (!__any_sync(0xffffffffu, need != 0u)) continue;
          unit_at(x);
          double d[4] = {0.0, 0.0, 0.0, 0.0};
          sl_dot64(p.A64 + (ti.a0 + m) * p.lda + ti.kb0 * kBK, 8 * p.lda, p.B64 + (ti.b0 + n) * p.ldb + ti.kb0 * kBK, p.ldb, kcol,
                   need, d);
          if (!p.ws) {
#pragma unroll
            for (int e = 0; e < 4; ++e) d[e] *= C.alpha;
          }
          store(d, need);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem, 512);
}

template <int P>
bool make_slice_map(CUtensorMap* map, const Sliced& X, int box_rows) {
  const cuuint64_t rows = static_cast<cuuint64_t>(X.rows), row = static_cast<cuuint64_t>(X.Kp) * 2;
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(X.Kp), rows, P + 1}, strides[2] = {row, row * rows};
  const cuuint32_t box[3] = {Sl<P>::BK, static_cast<cuuint32_t>(box_rows), P + 1};
  return encode_tensor_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, X.p, dims, strides, box,
                           Sl<P>::BK == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

template <int P>
void launch_sl(const Sliced& A, const Sliced& B, SlArgs a, cudaStream_t s) {
  static std::once_flag once;
  std::call_once(once, [] { cudaFuncSetAttribute(k_gemm_sl<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sl<P>::SMEM); });
  CUtensorMap ta, tb;
  if (!make_slice_map<P>(&ta, A, Sl<P>::BM) || !make_slice_map<P>(&tb, B, Sl<P>::BN)) {
    set_error("cuTensorMapEncodeTiled failed (slices)");
    return;
  }
  a.ea = A.ex;
  a.eb = B.ex;
  a.ea_rows = A.rows;
  a.eb_rows = B.rows;
  a.A64 = A.src;
  a.B64 = B.src;
  a.lda = A.ld;
  a.ldb = B.ld;
  int e = 0;
  const double f = std::frexp(a.C.alpha, &e);
  a.asign = f == 0.5 ? 1 : f == -0.5 ? -1 : 0;
  a.ashift = a.asign ? e - 1 : 0;
  const long long n = static_cast<long long>(a.tiles_m) * a.tiles_n * a.tiles_z;
  const int grid = static_cast<int>(std::min<long long>(n, num_sms()));
  count_launch();
  k_gemm_sl<P><<<grid, Sl<P>::THREADS, Sl<P>::SMEM, s>>>(ta, tb, a);
}

}  // namespace

Sliced slice_at(void* mem, long long rows, int Kp, const double* src, long long ld, int digits) {
  Sliced s;
  s.digits = digits;
  s.rows = static_cast<int>(rows);
  s.Kp = Kp;
  s.p = mem;
  s.ex = reinterpret_cast<int*>(static_cast<unsigned char*>(mem) +
                                (static_cast<size_t>(rows) * Kp * 2 * (digits + 1) + 255) / 256 * 256);
  s.src = src;
  s.ld = ld;
  return s;
}

static SliceJob slice_job(const Sliced& d) {
  return SliceJob{d.src, d.ld, d.rows, d.Kp, static_cast<__nv_bfloat16*>(d.p), d.ex};
}
static void launch_slice(const Sliced& d, const Sliced* e, cudaStream_t s) {
  auto items = [](const Sliced& x) { return static_cast<long long>(x.rows) * ((x.Kp + kChunk - 1) / kChunk); };
  const long long n = items(d) + (e ? items(*e) : 0);
  if (n <= 0) return;
  SliceJob j1 = slice_job(d);
  j1.rows = 0;
  if (e) j1 = slice_job(*e);
  count_launch();
  const int blocks = static_cast<int>(std::min<long long>((n + 7) / 8, 152LL * 16));
  if (d.digits == kFarDigits)
    k_slice<kFarDigits><<<blocks, 256, 0, s>>>(slice_job(d), j1);
  else
    k_slice<kDigits><<<blocks, 256, 0, s>>>(slice_job(d), j1);
}
void slice(const Sliced& d, cudaStream_t s) { launch_slice(d, nullptr, s); }

// One product of sliced operands (rows from a_row0 / b_row0), K in launches of one chunk unless the
// partials of several fit the split-K workspace.
template <int P>
static void gemm_sliced_p(const Sliced& A, int a_row0, const Sliced& B, int b_row0, int M, int N, int K, const OutMap& C,
                          int mbase, int nbase, const BatchEntry* batch, int nbatch, int seg, int sym, int tri,
                          int tri_row0, cudaStream_t s, int* dstatus) {
  constexpr int kBM = Sl<P>::BM, kBN = Sl<P>::BN, kBK = Sl<P>::BK;
  SlArgs a{};
  a.M = M;
  a.N = N;
  a.a_row0 = a_row0;
  a.b_row0 = b_row0;
  a.mbase = mbase;
  a.nbase = nbase;
  a.tiles_m = (M + kBM - 1) / kBM;
  a.tiles_n = (N + kBN - 1) / kBN;
  a.sym = sym;
  a.tri = tri;
  a.tri_row0 = tri_row0;
  a.C = C;
  a.batch = batch;
  a.seg = seg;
  a.status = dstatus;
  const int nkb = (K + kBK - 1) / kBK;  // columns from K on are zero
  const long long tiles = static_cast<long long>(a.tiles_m) * a.tiles_n, MN = static_cast<long long>(M) * N;
  constexpr int kcb = kChunk / kBK;
  if (!batch && !sym && K > 160) {
    // Split K over work items while they do not fill the SMs, the FP64 partials summed by the fixed-order
    // reduction. 32 columns of a tile are about 1.2 us of MMAs; up to 160 cost less in one item than the
    // reduction's launch (about 5 us) and half the MMAs.
    const SplitWs& w = split_ws();
    int kper = kcb;
    while (kper > 1 && tiles * ((nkb + kper - 1) / kper) < num_sms()) kper /= 2;
    auto fits = [&](int k) { return w.p && static_cast<size_t>((nkb + k - 1) / k) * static_cast<size_t>(MN) <= w.cap; };
    while (kper < kcb && !fits(kper)) kper *= 2;
    const int z = (nkb + kper - 1) / kper;
    if (z > 1 && fits(kper)) {
      a.nkb = nkb;
      a.kper = kper;
      a.tiles_z = z;
      a.ws = w.p;
      launch_sl<P>(A, B, a, s);
      splitk_reduce(z, M, N, C, s, mbase, nbase);
      return;
    }
  }
  for (int k0 = 0; k0 < nkb; k0 += kcb) {
    a.kblk0 = k0;
    a.nkb = std::min(kcb, nkb - k0);
    a.kper = kcb;
    a.tiles_z = batch ? nbatch : 1;
    launch_sl<P>(A, B, a, s);
    a.C.beta = 1.0;
  }
}
static void gemm_sliced_rows(const Sliced& A, int a_row0, const Sliced& B, int b_row0, int M, int N, int K, const OutMap& C,
                             int mbase, int nbase, const BatchEntry* batch, int nbatch, int seg, int sym, int tri,
                             int tri_row0, cudaStream_t s, int* dstatus) {
  auto run = A.digits == kFarDigits ? gemm_sliced_p<kFarDigits> : gemm_sliced_p<kDigits>;  // the same of both operands
  run(A, a_row0, B, b_row0, M, N, K, C, mbase, nbase, batch, nbatch, seg, sym, tri, tri_row0, s, dstatus);
}

void gemm_sliced(const Sliced& A, int a_row0, const Sliced& B, int b_row0, int M, int N, int K, const OutMap& C,
                 cudaStream_t s, int* dstatus) {
  gemm_sliced_rows(A, a_row0, B, b_row0, M, N, K, C, 0, 0, nullptr, 1, 0, 0, 0, 0, s, dstatus);
}

void gemm_sliced_batched(const Sliced& A, const Sliced& B, const BatchEntry* dbatch, int nbatch, int maxM, int N, int K,
                         int seg, const OutMap& C, cudaStream_t s, int* dstatus) {
  gemm_sliced_rows(A, 0, B, 0, maxM, N, K, C, 0, 0, dbatch, nbatch, seg, 0, 0, 0, s, dstatus);
}

void gemm_sliced_lower(const Sliced& A, int a_row0, int M, int N, int K, int block, const OutMap& C, cudaStream_t s,
                       int* dstatus) {
  GemmStats& st = gemm_stats();
  st.launches++;
  st.flops += 2.0 * M * N * K;
  gemm_sliced_rows(A, a_row0, A, 0, M, N, K, C, 0, 0, nullptr, 1, 0, 0, block, a_row0, s, dstatus);
}

// A (M rows) and B (N rows) packed FP64, K = Kp: slices panels of both into the slice workspace.
bool gemm_f64_slices(const double* A, const double* B, int M, int N, int K, int Kp, const OutMap& C, bool sym,
                     cudaStream_t s, int* dstatus) {
  const SplitWs& w = split_ws();
  if (!w.sl || !dstatus) return false;
  unsigned char* base = static_cast<unsigned char*>(w.sl);
  // does K have to be split below a chunk to fill the SMs (the rule of gemm_sliced_p)?
  const bool split = K > 160 && 1LL * ((M + 127) / 128) * ((N + 47) / 48) * ((K + kChunk - 1) / kChunk) < num_sms();
  const int dg = w.far == FarRows::kAll || (w.far == FarRows::kSmall && split) ? kFarDigits : kDigits;
  const bool same = A == B && M == N;
  if (same && slice_bytes(M, Kp, dg) <= w.sl_bytes) {
    const Sliced SA = slice_at(base, M, Kp, A, Kp, dg);
    slice(SA, s);
    gemm_sliced_rows(SA, 0, SA, 0, M, N, K, C, 0, 0, nullptr, 1, 0, sym ? 1 : 0, 0, 0, s, dstatus);
    return true;
  }
  const SlicePanels pl = plan_slice_panels(M, N, Kp, w.sl_bytes, dg);
  if (pl.kw == 0) return false;
  OutMap Ck = C;
  for_each_slice_panel(pl, M, N, Kp, sym, [&](int k0, int kw, int n0, int nn, int m0, int mm, bool first) {
    const int ku = std::min(kw, K - k0);
    if (ku <= 0) return;
    const Sliced SB = slice_at(base, nn, kw, B + static_cast<size_t>(n0) * Kp + k0, Kp, dg);
    const Sliced SA = slice_at(base + slice_bytes(nn, kw, dg), mm, kw, A + static_cast<size_t>(m0) * Kp + k0, Kp, dg);
    launch_slice(SA, first ? &SB : nullptr, s);
    Ck.beta = k0 == 0 ? C.beta : 1.0;
    gemm_sliced_rows(SA, 0, SB, 0, mm, nn, ku, Ck, m0, n0, nullptr, 1, 0, sym ? 1 : 0, 0, 0, s, dstatus);
  });
  return true;
}

}  // namespace lnocc
