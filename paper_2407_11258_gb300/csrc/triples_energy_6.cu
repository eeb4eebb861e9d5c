// FP32 block energies for nocc 26 to 28.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_6(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<26, 28>(p, s); }
}  // namespace lnocc
