// FP32 block energies for nocc 20 to 22.
#include "triples_energy.cuh"

namespace lnocc {
bool launch_block_energy_4(const EnergyArgs& p, cudaStream_t s) { return launch_energy_range<20, 22>(p, s); }
}  // namespace lnocc
