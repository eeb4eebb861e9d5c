// FP32 block energies for nocc 16 to 19.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_3(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<16, 19>(p, s); }
}  // namespace lnocc
