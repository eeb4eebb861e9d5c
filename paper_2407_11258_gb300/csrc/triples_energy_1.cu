// FP32 block energies for nocc 8 to 11.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_1(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<8, 11>(p, s); }
}  // namespace lnocc
