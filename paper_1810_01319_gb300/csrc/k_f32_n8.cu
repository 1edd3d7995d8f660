// Float32 PPM sweep of 8^3-cell blocks.
#include "sweep_f32.cuh"

namespace cello {
template void prepare_sweep_f32<8>();
template void launch_sweep_f32_nb<8>(const DevMesh& m, const SweepParams& p, cudaStream_t s);

int sweep_variant_count_f32() { return kNV; }

int sweep_variant_twin_f32(int v, bool dual) {
  const SweepVariant& a = kVariants[v];
  for (int u = 0; u < v && dual && a.stream; ++u) {
    const SweepVariant& b = kVariants[u];
    if (b.stream && b.pencils == a.pencils && b.vec == a.vec && b.persistent == a.persistent) return u;
  }
  return v;
}
}  // namespace cello
