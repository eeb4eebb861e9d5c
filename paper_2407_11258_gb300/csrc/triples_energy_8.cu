// FP32 block energies for nocc 33 to 37.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_8(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<33, 37>(p, s); }
}  // namespace lnocc
