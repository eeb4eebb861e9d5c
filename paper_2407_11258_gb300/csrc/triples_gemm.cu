// Grouped (T) contractions for any nocc from 4 to 32 (nocc 16 and 32 have forms of their own in gemm.cu).
//
// One W chunk takes two launches. Kind 1 runs, per region (c, ta whole a values), sigma1 + sigma2 (two K
// segments into one accumulator, stored), sigma3 and sigma5 (added); kind 2 runs, per region (ta whole (a, i)
// pairs, a block of c), sigma4 and sigma6 (added). A region belongs to one CTA, whose one copying thread waits
// until the copies of a term are performed before it sends those of the next term: bulk copies of one thread are
// not ordered by themselves, and FP32 additions in another order give other bits.
//   * Rows: a 128-row tile holds ta = 128 / nocc whole a values (kind 1) or (a, i) pairs (kind 2) and starts at
//     a multiple of ta nocc rows; the rows left over (at most nocc - 1) are computed and dropped.
//   * Columns: whole values of the column's outer index (k, i or c), as many as fit 256 and evenly spread over
//     the column tiles of a plane, so the MMA's N is that width rounded up to 16 instead of a padded 256.
//   * Epilogue: for one value of the outer index the tile's 128 x nocc results are exactly the box
//     [ta][nocc][j] of W. The four epilogue warps write it to shared memory in W order (a thread's row as
//     16-byte pieces, or as one column of the box for sigma3 and sigma6) and one thread sends it with a TMA
//     store or a TMA reduce-add, performed in L2. W rows are padded to jp = nocc rounded up to 4 for that.
// The per-term launches (gemm.cu) reduce W element by element from the epilogue threads (scalar for odd nocc):
// their epilogue took nine tenths of the time. (19, 125, 500): 72.0 -> 25.5 ms of contractions per call,
// (8, 120, 480): 10.2 -> 5.2 ms.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "ptx.cuh"

namespace lnocc {
namespace {

constexpr int kBM = 128, kBK = 32, kStages = 4;
constexpr int kABytes = 2 * kBM * kBK * 2;  // hi and lo planes
constexpr int kSmem = 232448;               // all a CTA may hold: four operand stages, the rest boxes of W
constexpr int kSmemBoxes = kSmem - 1024 - 256;
constexpr int kMaxBoxes = 4;  // more gain nothing: (19, 125, 500) 36.5, 33.8, 32.7, 32.7 ms per (T) call with 2, 3, 4, 8
// B planes of N rows after the A planes; at N = 256 and the largest box (128 rows of 32 floats) two boxes fit
constexpr int stage_bytes(int N) { return kABytes + 2 * N * kBK * 2; }
static_assert(kSmemBoxes - kStages * stage_bytes(256) >= 2 * kBM * 32 * 4, "grouped (T) pipeline does not fit");

struct TgArgs {
  TgSpec g;
  int rows;     // valid rows of a tile, ta * o
  int N;        // MMA width
  int stage;    // bytes of an operand stage
  int box, nbox;  // bytes of a box (a multiple of 128) and how many there are, 2 to kMaxBoxes
  int* status;
};

struct TgTile {
  int term, r;          // region
  int a0, m0;           // first unit (a, or (a, i) pair) and first row of the tile
  int n0;               // first column in the (y, z) plane (kind 1)
  int nout, out0;       // outer column values of the tile, and the first one
  int cl;               // chunk-local c (kind 1) or first c of the block (kind 2)
  int ma0, mb0, arow0, brow0, ma1, mb1, arow1, brow1, nseg;
};

// Tile w of this CTA (maps as in gemm.cu's grouped launches: kind 1 XT1, TO, XT2, TOT; kind 2 TO, XT2, -, XT1).
__device__ __forceinline__ bool tg_tile(const TgSpec& g, int w, TgTile& t) {
  const int per = g.kind == 1 ? 3 * g.ncol : 2;
  t.r = blockIdx.x + (w / per) * gridDim.x;
  if (t.r >= g.nreg) return false;
  const int q = w % per, tile = t.r % g.mt, outer = t.r / g.mt;
  t.a0 = tile * g.ta;
  t.m0 = t.a0 * g.o;
  t.nseg = 1;
  t.ma1 = t.mb1 = t.arow1 = t.brow1 = 0;
  if (g.kind == 1) {
    const int ct = q % g.ncol, c = g.c0 + outer, bc = c * g.oo, bb = g.b * g.oo;
    t.term = q / g.ncol;
    t.out0 = ct * g.nk;
    t.nout = min(g.nk, g.o - t.out0);
    t.n0 = t.out0 * g.o;
    t.cl = outer;
    if (t.term == 0) {
      t.nseg = 2;
      t.ma0 = 0; t.arow0 = g.bvo;    t.mb0 = 1; t.brow0 = bc;
      t.ma1 = 0; t.arow1 = c * g.vo; t.mb1 = 3; t.brow1 = bb;
    } else if (t.term == 1) {
      t.ma0 = 2; t.arow0 = g.bvo;    t.mb0 = 1; t.brow0 = bc;
    } else {
      t.ma0 = 2; t.arow0 = c * g.vo; t.mb0 = 3; t.brow0 = bb;
    }
  } else {
    t.term = q;
    t.cl = outer * g.nk;
    t.out0 = 0;
    t.nout = min(g.nk, g.nc - t.cl);
    t.n0 = 0;
    t.ma0 = 0; t.arow0 = 0;
    t.mb0 = q == 0 ? 1 : 3;
    t.brow0 = g.bvo + (g.c0 + t.cl) * g.o;
  }
  return true;
}

__device__ __forceinline__ const CUtensorMap* pick(int id, const CUtensorMap* m0, const CUtensorMap* m1,
                                                   const CUtensorMap* m2, const CUtensorMap* m3) {
  return id == 0 ? m0 : id == 1 ? m1 : id == 2 ? m2 : m3;
}
__device__ __forceinline__ uint32_t idesc_n(int N) {  // idesc_bf16_f32 for a width known at run time
  return (idesc_bf16_f32(kBM, 0)) | (static_cast<uint32_t>(N >> 3) << 17);
}
// At most n copies of this thread still reading their boxes.
__device__ __forceinline__ void bulk_wait_read(int n) {
  if (n >= 2)
    asm volatile("cp.async.bulk.wait_group.read 2;" ::: "memory");
  else if (n == 1)
    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
  else
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
// The same barrier with a vote: true when every epilogue thread passes true.
__device__ __forceinline__ bool epi_all(bool x) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(x ? 1u : 0u)
      : "memory");
  return r != 0;
}

// Warp 0 TMA producer, warp 1 MMA issuer, warp 2 TMEM owner, warps 4..7 epilogue.
__global__ void __launch_bounds__(256, 1)
    k_gemm_tg(const __grid_constant__ CUtensorMap t0, const __grid_constant__ CUtensorMap t1,
              const __grid_constant__ CUtensorMap t2, const __grid_constant__ CUtensorMap t3,
              const __grid_constant__ CUtensorMap tW0, const __grid_constant__ CUtensorMap tW1, const TgArgs p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* boxes = smem + kStages * p.stage;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kSmemBoxes);
  uint64_t* empty = full + kStages;
  uint64_t* accf = empty + kStages;
  uint64_t* acce = accf + 2;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(acce + 2);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const TgSpec& g = p.g;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 128);
    }
    fence_barrier_init();
    prefetch_tensormap(&t0);
    prefetch_tensormap(&t1);
    prefetch_tensormap(&t2);
    prefetch_tensormap(&t3);
  }
  if (warp == 2) tmem_alloc(tmem_holder, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == 0 && lane == 0) {
    const uint32_t bytes = kABytes + 2 * p.N * kBK * 2;
    int q = 0;
    bool ok = true;
    TgTile t;
    for (int w = 0; ok && tg_tile(g, w, t); ++w) {
      for (int kb = 0; kb < t.nseg * g.nkb; ++kb, ++q) {
        const int s = q % kStages;
        if (q >= kStages && !mbar_wait(&empty[s], ((q / kStages) - 1) & 1)) {
          atomicExch(p.status, kDevTimeoutProducer);
          ok = false;
          break;
        }
        uint8_t* st = smem + s * p.stage;
        mbar_arrive_expect_tx(&full[s], bytes);
        const bool s0 = kb < g.nkb;
        const int kc = (s0 ? kb : kb - g.nkb) * kBK;
        tma_load_3d(st, pick(s0 ? t.ma0 : t.ma1, &t0, &t1, &t2, &t3), &full[s], kc, (s0 ? t.arow0 : t.arow1) + t.m0, 0);
        tma_load_3d(st + kABytes, pick(s0 ? t.mb0 : t.mb1, &t0, &t1, &t2, &t3), &full[s], kc,
                    (s0 ? t.brow0 : t.brow1) + t.n0, 0);
      }
    }
    for (int k = (q > kStages ? q - kStages : 0); k < q; ++k) mbar_wait(&full[k % kStages], (k / kStages) & 1);
  } else if (warp == 1 && lane == 0) {
    const uint32_t idesc = idesc_n(p.N), blo = p.N * kBK * 2;
    int q = 0, it = 0;
    bool ok = true;
    TgTile t;
    for (int w = 0; ok && tg_tile(g, w, t); ++w) {
      const int buf = it & 1;
      if (it >= 2 && !mbar_wait(&acce[buf], ((it / 2) - 1) & 1)) {
        atomicExch(p.status, kDevTimeoutMma);
        break;
      }
      tc_fence_after();
      const uint32_t acc = tmem + buf * 256;
      for (int kb = 0; kb < t.nseg * g.nkb; ++kb, ++q) {
        const int s = q % kStages;
        if (!mbar_wait(&full[s], (q / kStages) & 1)) {
          atomicExch(p.status, kDevTimeoutMma);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t a = smem_u32(smem + s * p.stage), b = a + kABytes;
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          const uint32_t off = kk * 32;
          const uint64_t dah = sdesc_sw64(a + off), dal = sdesc_sw64(a + kABytes / 2 + off);
          const uint64_t dbh = sdesc_sw64(b + off), dbl = sdesc_sw64(b + blo + off);
          mma_bf16(acc, dah, dbh, idesc, (kb | kk) != 0 ? 1u : 0u);
          mma_bf16(acc, dah, dbl, idesc, 1u);
          mma_bf16(acc, dal, dbh, idesc, 1u);
        }
        mma_commit(&empty[s]);
      }
      mma_commit(&accf[buf]);
      ++it;
    }
  } else if (warp >= 4) {
    const int ew = warp - 4, r = ew * 32 + lane;  // accumulator row
    const bool lead = threadIdx.x == 128;         // issues the copies
    const bool rok = r < p.rows;
    const uint32_t box0 = smem_u32(boxes);
    const int npc = g.jp / 4;
    // row of the box, or column r % o of unit r / o
    const uint32_t vrow = static_cast<uint32_t>(r * g.jp * 4);
    const uint32_t srow = static_cast<uint32_t>(((r / g.o) * g.o * g.jp + r % g.o) * 4);
    const uint32_t sstep = static_cast<uint32_t>(g.jp * 4);
    int it = 0, nbox = 0;
    TgTile t;
    for (int w = 0; tg_tile(g, w, t); ++w) {
      const int buf = it & 1;
      // the wait is bounded; whether it ran out anywhere is agreed on, since the boxes below are shared
      if (!epi_all(mbar_wait(&accf[buf], (it / 2) & 1))) {
        if (lane == 0) atomicExch(p.status, kDevTimeoutEpilogue);
        break;
      }
      tc_fence_after();
      const uint32_t acc = tmem + buf * 256 + (static_cast<uint32_t>(ew * 32) << 16);
      if (lead && t.term > 0 && t.out0 == 0) bulk_wait_all();  // the last term's copies are performed first
#pragma unroll 1
      for (int x = 0; x < t.nout; ++x, nbox = nbox + 1 == p.nbox ? 0 : nbox + 1) {
        float v[32];
        tmem_ld32(acc + x * g.o, v);
        const uint32_t box = box0 + nbox * p.box;
        if (rok) {
          if (t.term != 1) {
#pragma unroll
            for (int h = 0; h < 8; ++h)
              if (h < npc) st_shared_v4(box + vrow + 16 * h, v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
          } else {
#pragma unroll
            for (int h = 0; h < 32; ++h)
              if (h < g.o) st_shared_f32(box + srow + h * sstep, v[h]);
          }
        }
        fence_proxy_async();
        // the copy sent from the next box has been read before anybody writes there again
        if (lead) bulk_wait_read(p.nbox - 2);
        epi_barrier();
        if (lead) {
          const int out = t.out0 + x;
          if (g.kind == 2)
            tma_reduce_add_5d(&tW0, box, 0, 0, t.a0, t.cl + x, 0);
          else if (t.term == 0)
            tma_store_5d(&tW0, box, 0, out, 0, t.a0, t.cl);
          else if (t.term == 1)
            tma_reduce_add_5d(&tW0, box, 0, out, 0, t.a0, t.cl);
          else
            tma_reduce_add_5d(&tW1, box, 0, 0, out, t.a0, t.cl);
          bulk_commit();
        }
      }
      tc_fence_before();
      mbar_arrive(&acce[buf]);
      ++it;
    }
    if (lead) bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem, 512);
}

bool operand_map(CUtensorMap* m, const Packed& P, int box_rows) {
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(P.Kp), static_cast<cuuint64_t>(P.rows), 2};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(P.Kp) * 2, static_cast<cuuint64_t>(P.Kp) * 2 * P.rows};
  const cuuint32_t box[3] = {kBK, static_cast<cuuint32_t>(box_rows), 2};
  return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, P.p, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

}  // namespace

void gemm_grouped_any(const Packed* const ops[4], TgSpec g, float* W, int K, cudaStream_t s, int* dstatus) {
  if (g.o < 4 || g.o > 32 || (g.kind != 1 && g.kind != 2)) {
    set_error("gemm_grouped_any: nocc 4 to 32 only");
    return;
  }
  g.oo = g.o * g.o;
  g.jp = round_up(g.o, 4);
  g.ta = kBM / g.o;
  // outer column values of a tile: their columns and the 32 that a TMEM load reads from the last one fit 256
  const int nkmax = 224 / g.o + 1;
  if (g.kind == 1) {
    g.ncol = (g.o + nkmax - 1) / nkmax;
    g.nk = (g.o + g.ncol - 1) / g.ncol;
    g.ncol = (g.o + g.nk - 1) / g.nk;
    g.mt = (g.b + 1 + g.ta - 1) / g.ta;
    g.nreg = g.nc * g.mt;
  } else {
    const int blocks = (g.nc + nkmax - 1) / nkmax;
    g.ncol = 1;
    g.nk = (g.nc + blocks - 1) / blocks;
    g.mt = ((g.b + 1) * g.o + g.ta - 1) / g.ta;
    g.nreg = g.mt * ((g.nc + g.nk - 1) / g.nk);
  }
  g.nkb = (K + kBK - 1) / kBK;
  TgArgs a{};
  a.g = g;
  a.rows = g.ta * g.o;
  a.N = round_up(g.nk * g.o, 16);
  a.stage = stage_bytes(a.N);
  a.box = round_up(a.rows * g.jp * 4, 128);
  a.nbox = std::min(kMaxBoxes, (kSmemBoxes - kStages * a.stage) / a.box);
  a.status = dstatus;
  CUtensorMap m[4], w0, w1;
  for (int k = 0; k < 4; ++k) {
    // A operands: kind 1 XT1 and XT2 (0, 2), kind 2 TO (0)
    const bool isA = k == 0 || (g.kind == 1 && k == 2);
    if (!operand_map(&m[k], *ops[k], isA ? kBM : a.N)) {
      set_error("cuTensorMapEncodeTiled failed (grouped (T))");
      return;
    }
  }
  const cuuint64_t o = g.o, jp = g.jp, na = g.b + 1, nc = g.nc, row = jp * 4;
  bool ok;
  if (g.kind == 1) {  // {j, k, i, a, c}
    const cuuint64_t dims[5] = {jp, o, o, na, nc};
    const cuuint64_t st[4] = {row, o * row, o * o * row, static_cast<cuuint64_t>(g.Sc) * 4};
    const cuuint32_t bk[5] = {static_cast<cuuint32_t>(jp), 1, static_cast<cuuint32_t>(o), static_cast<cuuint32_t>(g.ta), 1};
    const cuuint32_t bi[5] = {static_cast<cuuint32_t>(jp), static_cast<cuuint32_t>(o), 1, static_cast<cuuint32_t>(g.ta), 1};
    ok = encode_tensor_map(&w0, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, W, dims, st, bk, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE) &&
         encode_tensor_map(&w1, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, W, dims, st, bi, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE);
  } else {  // {j, k, (a, i), c, 1}
    const cuuint64_t dims[5] = {jp, o, na * o, nc, 1};
    const cuuint64_t st[4] = {row, o * row, static_cast<cuuint64_t>(g.Sc) * 4, static_cast<cuuint64_t>(g.Sc) * 4 * nc};
    const cuuint32_t bx[5] = {static_cast<cuuint32_t>(jp), static_cast<cuuint32_t>(o), static_cast<cuuint32_t>(g.ta), 1, 1};
    ok = encode_tensor_map(&w0, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, W, dims, st, bx, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE);
    w1 = w0;
  }
  if (!ok) {
    set_error("cuTensorMapEncodeTiled failed (W chunk)");
    return;
  }
  static std::once_flag once;
  std::call_once(once, [] { cudaFuncSetAttribute(k_gemm_tg, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem); });
  GemmStats& st = gemm_stats();
  st.launches++;
  st.flops += g.kind == 1 ? 2.0 * (g.b + 1) * g.o * g.oo * K * 4 * g.nc : 2.0 * (g.b + 1) * g.oo * (1.0 * g.nc * g.o) * K * 2;
  count_launch();
  k_gemm_tg<<<std::min(g.nreg, num_sms()), 256, kSmem, s>>>(m[0], m[1], m[2], m[3], w0, w1, a);
}

}  // namespace lnocc
