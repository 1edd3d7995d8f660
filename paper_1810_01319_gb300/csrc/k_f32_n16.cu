// Float32 PPM sweep of 16^3-cell blocks.
#include "sweep_f32.cuh"

namespace cello {
template void prepare_sweep_f32<16>();
template void launch_sweep_f32_nb<16>(const DevMesh& m, const SweepParams& p, cudaStream_t s);
}  // namespace cello
