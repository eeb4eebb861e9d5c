// FP32 block energies for nocc 23 to 25.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_5(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<23, 25>(p, s); }
}  // namespace lnocc
