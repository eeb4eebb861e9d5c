// FP32 block energies for nocc 29 to 32.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_7(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<29, 32>(p, s); }
}  // namespace lnocc
