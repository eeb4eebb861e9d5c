// FP32 block energies for nocc 12 to 15.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_2(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<12, 15>(p, s); }
}  // namespace lnocc
