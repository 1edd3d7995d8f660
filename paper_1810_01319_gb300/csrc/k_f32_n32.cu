// Float32 PPM sweep of 32^3-cell blocks.
#include "sweep_f32.cuh"

namespace cello {
template void prepare_sweep_f32<32>();
template void launch_sweep_f32_nb<32>(const DevMesh& m, const SweepParams& p, cudaStream_t s);
}  // namespace cello
