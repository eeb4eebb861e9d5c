// FP32 block energies: nocc below 8, and the dispatch over the compiled ranges.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_0(const EnergyArgs& p, cudaStream_t s) {
  if (p.o > kRuntimeMaxOcc) return false;
  launch_energy_o<0>(p, s);
  return true;
}
void launch_block_energy(const EnergyArgs& p, cudaStream_t s) {
  (void)(launch_block_energy_0(p, s) || launch_block_energy_1(p, s) || launch_block_energy_2(p, s) || launch_block_energy_3(p, s) || launch_block_energy_4(p, s) || launch_block_energy_5(p, s) || launch_block_energy_6(p, s) || launch_block_energy_7(p, s) || launch_block_energy_8(p, s));
}
}  // namespace lnocc
