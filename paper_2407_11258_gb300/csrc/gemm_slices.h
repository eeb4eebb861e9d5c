// FP64 contractions on the BF16 tensor pipe (gemm_slices.cu): operands cut into BF16 digit planes.
#pragma once
#include <cuda_runtime.h>

#include "internal.h"
#include "slice_panels.h"

namespace lnocc {

// Rows of a packed FP64 operand (row stride ld, Kp columns) as BF16 planes [digits + 1][rows][Kp] (nine or twelve digits
// and the magnitudes) and the exponents [ceil(Kp / 512)][rows] of their chunks.
struct Sliced {
  void* p = nullptr;
  int* ex = nullptr;
  int rows = 0, Kp = 0, digits = kDigits;
  const double* src = nullptr;
  long long ld = 0;
};

// Virtuals above which FP64 products take twelve digits, nine / twelve measured on two CCSD iterations: the rings at
// (10, 120, 480) 4.1 / 1.7 ms and at (12, 160, 640) 24 / 4.8 (at 96 virtuals nine are faster); ladder and Z 7.3 / 7.6 and
// 71 / 28.5. (T) always takes them: (8, 64, 256) 18.1 / 15.5 ms (tiles of 32 columns fit its products better),
// (10, 120, 480) 440 / 136, (16, 240, 960) 23.8 / 3.8 s.
constexpr int kFarRings = 100, kFarLadder = 128;
Sliced slice_at(void* mem, long long rows, int Kp, const double* src, long long ld, int digits = kDigits);
void slice(const Sliced& d, cudaStream_t s);  // fill the planes from src
void gemm_sliced(const Sliced& A, int a_row0, const Sliced& B, int b_row0, int M, int N, int K, const OutMap& C,
                 cudaStream_t s, int* dstatus);
void gemm_sliced_batched(const Sliced& A, const Sliced& B, const BatchEntry* dbatch, int nbatch, int maxM, int N, int K,
                         int seg, const OutMap& C, cudaStream_t s, int* dstatus);
// Rows [a_row0, a_row0 + M) of A against rows [0, N) of A; only elements whose column block n / block does not exceed
// the row block (a_row0 + m) / block are needed (others may be left unset).
void gemm_sliced_lower(const Sliced& A, int a_row0, int M, int N, int K, int block, const OutMap& C, cudaStream_t s,
                       int* dstatus);
// C = A B^T for packed FP64 operands through the thread's slice workspace (split_ws().sl): false when
// there is none (or it is too small): the caller then runs the FP64 SIMT kernel. sym: A == B, the upper
// part computed and mirrored.
bool gemm_f64_slices(const double* A, const double* B, int M, int N, int K, int Kp, const OutMap& C, bool sym,
                     cudaStream_t s, int* dstatus);

}  // namespace lnocc
