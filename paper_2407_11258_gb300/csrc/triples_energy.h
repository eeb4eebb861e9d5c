// FP32 block energies of the mixed (T) path: launch interface and shared-memory plan (kernels in
// triples_energy.cuh, compiled per range of nocc by triples_energy_*.cu).
#pragma once
#include <cuda_runtime.h>

namespace lnocc {

constexpr int kMaxPairOcc = 28;    // w and v staged side by side
constexpr int kMaxStagedOcc = 37;  // one value per element staged

// Shared-memory strides of a staged block, all odd (conflict-free for lanes along any slot).
__host__ __device__ constexpr int blk_s1(int o) { return o | 1; }
__host__ __device__ constexpr int blk_s0(int o) { return (o * blk_s1(o)) | 1; }
__host__ __device__ constexpr int w_row(int o) { return (o + 3) & ~3; }  // row length of W (16-byte rows)
__host__ __device__ constexpr int tri_count(int o) { return o * (o + 1) * (o + 2) / 6; }
// floats of the slices and vectors of one block
__host__ __device__ constexpr int energy_small_floats(int o) { return 4 * o + 3 * o * (o | 1) + 2 * o; }

struct EnergyArgs {
  const float* W;             // chunk [slot][a][i][k][j], rows of w_row(o) elements
  long long slot_stride;
  int b, c0, o, v;
  const double *eps, *t1;
  const float* ovT;           // (ia|jb) as [a][b][i][j]
  const double* U;            // [o][nlo]
  int nlo;
  const unsigned* tri;        // unordered occupied triples
  double* out;                // {canonical, projected} per block
  int na, nc;                 // blocks: a < na, slot < nc
};
// Block energies of one W chunk (1 <= o <= kMaxStagedOcc).
void launch_block_energy(const EnergyArgs& p, cudaStream_t s);
// The kernels of one range of nocc; false when o lies outside it.
bool launch_block_energy_0(const EnergyArgs& p, cudaStream_t s);  // below 8
bool launch_block_energy_1(const EnergyArgs& p, cudaStream_t s);  // 8 to 11
bool launch_block_energy_2(const EnergyArgs& p, cudaStream_t s);  // 12 to 15
bool launch_block_energy_3(const EnergyArgs& p, cudaStream_t s);  // 16 to 19
bool launch_block_energy_4(const EnergyArgs& p, cudaStream_t s);  // 20 to 22
bool launch_block_energy_5(const EnergyArgs& p, cudaStream_t s);  // 23 to 25
bool launch_block_energy_6(const EnergyArgs& p, cudaStream_t s);  // 26 to 28
bool launch_block_energy_7(const EnergyArgs& p, cudaStream_t s);  // 29 to 32
bool launch_block_energy_8(const EnergyArgs& p, cudaStream_t s);  // 33 to 37

}  // namespace lnocc
