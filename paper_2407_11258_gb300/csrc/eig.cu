// Symmetric eigendecomposition in FP64 on the device: parallel cyclic Jacobi.
//
// A sweep visits every pair (p, q) once in m - 1 rounds of the round-robin ("circle") schedule over
// m = n rounded up to even players: in round r, pair 0 is (m - 1, r) and pair k >= 1 is
// ((r + k) mod (m - 1), (r - k) mod (m - 1)). The m / 2 pairs of one round are disjoint, so their plane
// rotations commute: every A_pq of the round is zeroed at once, A <- J^T A J as independent 2 x 2 blocks (rows of
// pair P, columns of pair Q) and V <- V J. Up to order kSweepMax one cooperative kernel runs a whole sweep with a
// grid barrier between rounds (k_jac_sweep); above, a round is two launches (k_jac_angles, k_jac_rotate). A player
// index >= n (odd n) is a bye. Rotation angles follow the classical form: theta = (A_qq - A_pp) / 2A_pq,
// t = sgn(theta) / (|theta| + sqrt(theta^2 + 1)), c = 1 / sqrt(1 + t^2), s = t c, which gives
// A'_pp = A_pp - t A_pq, A'_qq = A_qq + t A_pq, A'_pq = 0. After each sweep the off-diagonal norm is read
// back; the host stops when it is below 1e-15 of the Frobenius norm (Jacobi converges quadratically) or
// after 60 sweeps. Eigenvalues are then sorted (single-block bitonic sort) with their vectors.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "internal.h"
#include "ptx.cuh"

namespace lnocc {
namespace {

__device__ __forceinline__ void jac_pair(int r, int k, int m, int* p, int* q) {
  const int m1 = m - 1;
  if (k == 0) {
    *p = m1;
    *q = r;
  } else {
    *p = (r + k) % m1;
    *q = (r - k + m1) % m1;
  }
}

// Rotation that zeroes A_pq of pair k in round r (identity for a bye or a negligible element).
__device__ __forceinline__ double2 jac_angle(const double* A, int n, int m, int r, int k) {
  int p, q;
  jac_pair(r, k, m, &p, &q);
  double c = 1.0, s = 0.0;
  if (p < n && q < n) {
    const double apq = __ldcg(A + static_cast<long long>(p) * n + q);
    const double app = __ldcg(A + static_cast<long long>(p) * n + p), aqq = __ldcg(A + static_cast<long long>(q) * n + q);
    // skip a rotation whose off-diagonal element is negligible against its diagonal pair
    if (fabs(apq) > 1e-300 && fabs(apq) > 1e-18 * sqrt(fabs(app * aqq))) {
      const double th = (aqq - app) / (2.0 * apq);
      const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
      c = 1.0 / sqrt(t * t + 1.0);
      s = t * c;
    }
  }
  return make_double2(c, s);
}

// The 2 x 2 block (a b; c d) of A under the rotations of its row pair and its column pair; diag: the pair itself,
// whose off-diagonal element the rotation annihilates.
__device__ __forceinline__ void jac_block(double& a, double& b, double& c, double& d, double2 g1, double2 g2, bool diag) {
  // rows: p <- c row_p - s row_q, q <- s row_p + c row_q
  const double a1 = g1.x * a - g1.y * c, b1 = g1.x * b - g1.y * d;
  const double c1 = g1.y * a + g1.x * c, d1 = g1.y * b + g1.x * d;
  // columns: p <- c col_p - s col_q, q <- s col_p + c col_q
  a = g2.x * a1 - g2.y * b1;
  b = diag ? 0.0 : g2.y * a1 + g2.x * b1;
  c = diag ? 0.0 : g2.x * c1 - g2.y * d1;
  d = g2.y * c1 + g2.x * d1;
}

// A round of a large matrix: all angles, then (m/2)^2 blocks of A and n * (m/2) row-pairs of V in place.
__global__ void k_jac_angles(const double* __restrict__ A, int n, int m, int r, double2* __restrict__ cs) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < m / 2) cs[k] = jac_angle(A, n, m, r, k);
}
__global__ void k_jac_rotate(double* __restrict__ A, double* __restrict__ V, int n, int m, int r,
                             const double2* __restrict__ cs) {
  const long long h = m / 2, nA = h * h, nV = static_cast<long long>(n) * h;
  for (long long w = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; w < nA + nV;
       w += static_cast<long long>(gridDim.x) * blockDim.x) {
    if (w < nA) {
      const int kP = static_cast<int>(w / h), kQ = static_cast<int>(w % h);
      int p1, q1, p2, q2;
      jac_pair(r, kP, m, &p1, &q1);
      jac_pair(r, kQ, m, &p2, &q2);
      const bool r1 = p1 < n, r2 = q1 < n, c1 = p2 < n, c2 = q2 < n;  // byes are absent rows / columns
      double* R1 = A + static_cast<long long>(p1) * n;
      double* R2 = A + static_cast<long long>(q1) * n;
      double a = (r1 && c1) ? R1[p2] : 0.0, b = (r1 && c2) ? R1[q2] : 0.0;
      double c = (r2 && c1) ? R2[p2] : 0.0, d = (r2 && c2) ? R2[q2] : 0.0;
      jac_block(a, b, c, d, cs[kP], cs[kQ], kP == kQ);
      if (r1 && c1) R1[p2] = a;
      if (r1 && c2) R1[q2] = b;
      if (r2 && c1) R2[p2] = c;
      if (r2 && c2) R2[q2] = d;
    } else {
      const long long x = w - nA;
      const int k = static_cast<int>(x % h);
      int p, q;
      jac_pair(r, k, m, &p, &q);
      if (p >= n || q >= n) continue;
      const double2 g = cs[k];
      double* row = V + (x / h) * n;
      const double vp = row[p], vq = row[q];
      row[p] = g.x * vp - g.y * vq;
      row[q] = g.y * vp + g.x * vq;
    }
  }
}

// All blocks of the grid arrive and wait for each other (cooperative launch: all are resident). The wait has a
// wall-clock budget; when it runs out the flag is set and every block returns.
__device__ bool jac_barrier(unsigned* count, unsigned target, int* flag) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    const unsigned long long t0 = globaltimer();
    ok = 1;
    unsigned n = 0;
    while (true) {
      unsigned c;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
      if (c >= target) break;
      if ((++n & 63u) == 0 && globaltimer() - t0 > kWaitBudgetNs) {
        ok = 0;
        atomicExch(flag, 1);
        break;
      }
    }
  }
  __syncthreads();
  return ok != 0;
}

// One sweep of m - 1 rounds, reading A and writing A in turn from one buffer into the other (rounds of even
// index read A0), V in place. Block (x, y) owns the row pairs [x tP, ...) and column pairs [y tQ, ...) of A and
// the rows [x tV, ...) of V for the same column pairs, and computes the tP + tQ angles that takes from the old
// matrix. What others wrote in the round before is read past L1 (__ldcg). Bound by latency: a round is one
// dependent chain (three elements from L2, a square root and two divisions in FP64, the barrier). With two
// launches per round (angles, rotations) a round took 10 us; the 1471 rounds of three matrices of order 160, 100
// and 16 and three small ones fell from 15 to 8.8 ms. lnocc_lno_select, sweep against two launches per round:
// order 333 26.4 and 42.3 ms, 500 54 and 81, 1000 222 and 236, 2000 1485 and 1323 (the rotations bound, and in place
// they keep a third less in L2). (t = 2 a_pq / (|d| + sqrt(d^2 + 4 a_pq^2)) would shorten
// the chain, but the zero eigenvalues of rank-deficient LO sets then come out as rounding noise.)
__global__ void __launch_bounds__(256) k_jac_sweep(double* A0, double* A1, double* V, int n, int m, int tP, int tQ,
                                                   int tV, unsigned* count, int* flag) {
  extern __shared__ double2 ang[];  // tP row pairs, then tQ column pairs
  const int h = m / 2, nblk = gridDim.x * gridDim.y;
  const int p0 = blockIdx.x * tP, np = min(tP, h - p0), q0 = blockIdx.y * tQ, nq = min(tQ, h - q0);
  const int v0 = blockIdx.x * tV, nv = min(tV, n - v0);
  for (int r = 0; r < m - 1; ++r) {
    const double* A = (r & 1) ? A1 : A0;
    double* B = (r & 1) ? A0 : A1;
    for (int x = threadIdx.x; x < np + nq; x += blockDim.x)
      ang[x] = jac_angle(A, n, m, r, x < np ? p0 + x : q0 + x - np);
    __syncthreads();
    const int nA = np > 0 && nq > 0 ? np * nq : 0, nV = nv > 0 && nq > 0 ? nv * nq : 0;
    for (int w = threadIdx.x; w < nA + nV; w += blockDim.x) {
      if (w < nA) {
        const int kP = p0 + w / nq, kQ = q0 + w % nq;
        int p1, q1, p2, q2;
        jac_pair(r, kP, m, &p1, &q1);
        jac_pair(r, kQ, m, &p2, &q2);
        const bool r1 = p1 < n, r2 = q1 < n, c1 = p2 < n, c2 = q2 < n;  // byes are absent rows / columns
        double a = (r1 && c1) ? __ldcg(A + static_cast<long long>(p1) * n + p2) : 0.0;
        double b = (r1 && c2) ? __ldcg(A + static_cast<long long>(p1) * n + q2) : 0.0;
        double c = (r2 && c1) ? __ldcg(A + static_cast<long long>(q1) * n + p2) : 0.0;
        double d = (r2 && c2) ? __ldcg(A + static_cast<long long>(q1) * n + q2) : 0.0;
        jac_block(a, b, c, d, ang[w / nq], ang[np + w % nq], kP == kQ);
        if (r1 && c1) B[static_cast<long long>(p1) * n + p2] = a;
        if (r1 && c2) B[static_cast<long long>(p1) * n + q2] = b;
        if (r2 && c1) B[static_cast<long long>(q1) * n + p2] = c;
        if (r2 && c2) B[static_cast<long long>(q1) * n + q2] = d;
      } else {
        const int x = w - nA;
        int p, q;
        jac_pair(r, q0 + x % nq, m, &p, &q);
        if (p >= n || q >= n) continue;
        const double2 g = ang[np + x % nq];
        double* row = V + static_cast<long long>(v0 + x / nq) * n;
        const double vp = __ldcg(row + p), vq = __ldcg(row + q);
        row[p] = g.x * vp - g.y * vq;
        row[q] = g.y * vp + g.x * vq;
      }
    }
    if (!jac_barrier(count, static_cast<unsigned>(r + 1) * nblk, flag)) return;
  }
}

// out[0] = sum of squares of the off-diagonal elements, out[1] = of all elements (one block, fixed order)
__global__ void k_jac_norms(const double* __restrict__ A, int n, double* __restrict__ out) {
  __shared__ double red[2][32];
  double off = 0.0, all = 0.0;
  const long long nn = static_cast<long long>(n) * n;
  for (long long idx = threadIdx.x; idx < nn; idx += blockDim.x) {
    const double x = A[idx];
    all += x * x;
    if (idx / n != idx % n) off += x * x;
  }
  for (int o = 16; o > 0; o >>= 1) {
    off += __shfl_xor_sync(0xffffffffu, off, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  if (threadIdx.x % 32 == 0) {
    red[0][threadIdx.x / 32] = off;
    red[1][threadIdx.x / 32] = all;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int w = 0; w < static_cast<int>(blockDim.x / 32); ++w) {
      s0 += red[0][w];
      s1 += red[1][w];
    }
    out[0] = s0;
    out[1] = s1;
  }
}

__global__ void k_identity(double* V, int n) {
  const long long nn = static_cast<long long>(n) * n;
  for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < nn;
       idx += static_cast<long long>(gridDim.x) * blockDim.x)
    V[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

// Eigenvalues (diagonal of A) sorted with a bitonic sort in one block of 1024 threads; `order[k]` is
// the column of V holding the k-th value (decreasing when `desc`, else increasing; ties by index).
constexpr int kSortMax = 8192;
__global__ void __launch_bounds__(1024) k_eig_sort(const double* __restrict__ A, int n, int desc,
                                                   double* __restrict__ w, int* __restrict__ order) {
  extern __shared__ unsigned char sm[];
  int P = 1;
  while (P < n) P <<= 1;
  double* key = reinterpret_cast<double*>(sm);
  int* idx = reinterpret_cast<int*>(key + P);
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    const double x = i < n ? A[static_cast<long long>(i) * n + i] : 0.0;
    // pad entries sort last in either direction
    key[i] = i < n ? (desc ? -x : x) : INFINITY;
    idx[i] = i;
  }
  __syncthreads();
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int j = i ^ stride;
        if (j > i) {
          const bool up = (i & size) == 0;
          const bool gt = key[i] > key[j] || (key[i] == key[j] && idx[i] > idx[j]);
          if (gt == up) {
            const double tk = key[i];
            key[i] = key[j];
            key[j] = tk;
            const int ti = idx[i];
            idx[i] = idx[j];
            idx[j] = ti;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    w[i] = desc ? -key[i] : key[i];
    order[i] = idx[i];
  }
}

// out[:, k] = V[:, order[k]] for k < ncols (n x ncols output, row-major, leading dimension ldo)
__global__ void k_gather_cols(const double* __restrict__ V, int n, const int* __restrict__ order, int ncols,
                              double* __restrict__ out, int ldo) {
  const long long tot = static_cast<long long>(n) * ncols;
  for (long long x = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; x < tot;
       x += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(x / ncols), k = static_cast<int>(x % ncols);
    out[static_cast<long long>(i) * ldo + k] = V[static_cast<long long>(i) * n + order[k]];
  }
}

int grid_of(long long work, int threads) {
  return static_cast<int>(std::max(1LL, std::min<long long>((work + threads - 1) / threads, 152LL * 32)));
}

}  // namespace

// Largest order whose sweeps run in one launch (both forms measured at k_jac_sweep).
constexpr int kSweepMax = 1024;

// Doubles of scratch that sym_eig needs: norms, barrier and flag, then the second copy of the matrix or the angles.
size_t eig_scratch(int n) { return 16 + (n <= kSweepMax ? static_cast<size_t>(n) * n : static_cast<size_t>(n) + 1); }

// A [n][n] symmetric (destroyed); on return w [n] holds the eigenvalues (decreasing when desc, else
// increasing), order [n] their columns in V, and V [n][n] the eigenvectors as columns (A V = V diag).
// Device pointers; `scratch` holds eig_scratch(n) doubles. Synchronizes `s` once per sweep.
int sym_eig(double* A, double* V, double* w, int* order, int n, bool desc, double* scratch, cudaStream_t s,
            int* sweeps_out) {
  if (n < 1 || n > kSortMax) {
    set_error("eigendecomposition: size must be in [1, " + std::to_string(kSortMax) + "]");
    return LNOCC_EINVAL;
  }
  const int m = n + (n & 1), h = m / 2;
  double* norms = scratch;
  unsigned* count = reinterpret_cast<unsigned*>(scratch + 4);
  int* flag = reinterpret_cast<int*>(scratch + 5);
  double* A2 = scratch + 16;
  LN_CUDA(cudaMemsetAsync(scratch, 0, 16 * sizeof(double), s));
  count_launch();
  k_identity<<<grid_of(1LL * n * n, 256), 256, 0, s>>>(V, n);
  int sweep = 0;
  double hn[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (n > 1) {
    // about one 2 x 2 block or row pair a thread, in one block per SM or, for larger orders, three (768 threads of
    // at most 40 registers: all resident): order 333 26.4 and 26.6 ms with one and three, 500 61 and 54, 1000 299 and
    // 222 (256 with eight: the barrier). A grid of tiles close to square keeps the angles each block needs few.
    const long long work = 1LL * h * h + 1LL * n * h;
    const int cap = num_sms() * (n > 400 ? 3 : 1);
    const int blocks = static_cast<int>(std::max(1LL, std::min<long long>(cap, (work + 255) / 256)));
    int gx = std::max(1, static_cast<int>(std::sqrt(static_cast<double>(blocks))));
    gx = std::min(gx, h);
    const int tP = (h + gx - 1) / gx;
    gx = (h + tP - 1) / tP;
    const int gy0 = std::max(1, std::min(h, blocks / gx)), tQ = (h + gy0 - 1) / gy0, gy = (h + tQ - 1) / tQ;
    int nn = n, mm = m, tPa = tP, tQa = tQ, tV = (n + gx - 1) / gx;
    for (sweep = 0; sweep < 60; ++sweep) {
      count_launch();
      k_jac_norms<<<1, 1024, 0, s>>>(A, n, norms);
      LN_CUDA(cudaMemcpyAsync(hn, norms, 6 * sizeof(double), cudaMemcpyDeviceToHost, s));
      LN_CUDA(cudaStreamSynchronize(s));
      int timed_out = 0;
      std::memcpy(&timed_out, &hn[5], sizeof(int));
      if (timed_out) {
        set_error("eigendecomposition: device wait timed out");
        return LNOCC_ETIMEOUT;
      }
      if (!std::isfinite(hn[1])) {
        set_error("eigendecomposition: non-finite matrix");
        return LNOCC_ENUMERIC;
      }
      if (hn[0] <= 1e-30 * hn[1] || hn[0] == 0.0) break;
      if (n > kSweepMax) {
        double2* cs = reinterpret_cast<double2*>(A2);
        for (int r = 0; r < m - 1; ++r) {
          count_launch(2);
          k_jac_angles<<<grid_of(h, 128), 128, 0, s>>>(A, n, m, r, cs);
          k_jac_rotate<<<grid_of(work, 256), 256, 0, s>>>(A, V, n, m, r, cs);
        }
        continue;
      }
      LN_CUDA(cudaMemsetAsync(count, 0, sizeof(unsigned), s));
      void* args[] = {&A, &A2, &V, &nn, &mm, &tPa, &tQa, &tV, &count, &flag};
      count_launch();
      LN_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_jac_sweep), dim3(gx, gy), dim3(256), args,
                                          static_cast<size_t>(tP + tQ) * sizeof(double2), s));
      std::swap(A, A2);  // m - 1 rounds, an odd number
    }
    if (sweep == 60) {
      set_error("eigendecomposition: Jacobi sweeps did not converge");
      return LNOCC_ENOCONV;
    }
  }
  int P = 1;
  while (P < n) P <<= 1;
  const size_t smem = static_cast<size_t>(P) * (sizeof(double) + sizeof(int));
  if (smem > 48 * 1024) {
    static bool attr_set = false;
    if (!attr_set) {
      LN_CUDA(cudaFuncSetAttribute(k_eig_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
      attr_set = true;
    }
  }
  count_launch();
  k_eig_sort<<<1, 1024, smem, s>>>(A, n, desc ? 1 : 0, w, order);
  if (sweeps_out) *sweeps_out = sweep;
  LN_CUDA(cudaGetLastError());
  return LNOCC_OK;
}

void gather_cols(const double* V, int n, const int* order, int ncols, double* out, int ldo, cudaStream_t s) {
  if (ncols < 1) return;
  count_launch();
  k_gather_cols<<<grid_of(1LL * n * ncols, 256), 256, 0, s>>>(V, n, order, ncols, out, ldo);
}

}  // namespace lnocc
