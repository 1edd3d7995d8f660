// Float32 path: dispatch of the PPM sweep (bulk arithmetic in float32), the
// reduction and the adjoint sweep.
#include "kernels.cuh"
#include "adjoint_kernels.cuh"

namespace cello {

void launch_reduce_partials_f32(const DevMesh& m, const float* U, double* partials, int leaf0, int nleaf, int grid,
                                cudaStream_t s) {
  const int g = (grid > 0 && grid < nleaf) ? grid : nleaf;
  if (m.nf == 6) {
    switch (m.n) {
      case 8: reduce_partials_f32_kernel<8, 6><<<g, kReduceThreads, 0, s>>>(m, U, partials, leaf0, nleaf); break;
      case 16: reduce_partials_f32_kernel<16, 6><<<g, kReduceThreads, 0, s>>>(m, U, partials, leaf0, nleaf); break;
      case 32: reduce_partials_f32_kernel<32, 6><<<g, kReduceThreads, 0, s>>>(m, U, partials, leaf0, nleaf); break;
    }
    return;
  }
  switch (m.n) {
    case 8: reduce_partials_f32_kernel<8><<<g, kReduceThreads, 0, s>>>(m, U, partials, leaf0, nleaf); break;
    case 16: reduce_partials_f32_kernel<16><<<g, kReduceThreads, 0, s>>>(m, U, partials, leaf0, nleaf); break;
    case 32: reduce_partials_f32_kernel<32><<<g, kReduceThreads, 0, s>>>(m, U, partials, leaf0, nleaf); break;
  }
}


void launch_sweep_f32(const DevMesh& m, const SweepParams& p, cudaStream_t s) {
  switch (m.n) {
    case 8: launch_sweep_f32_nb<8>(m, p, s); break;
    case 16: launch_sweep_f32_nb<16>(m, p, s); break;
    case 32: launch_sweep_f32_nb<32>(m, p, s); break;
  }
}

template <int NB>
static void prepare_adj() {
  cudaFuncSetAttribute(adjoint_sweep_kernel<float, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)adjoint_smem<float, NB>());
}

template <int NB>
static void adj_sweep_n(const DevMesh& m, const AdjSweepParams& p, cudaStream_t s) {
  constexpr int threads = (NB + 2 * kGhosts) * adj_pencils(NB, 4);
  adjoint_sweep_kernel<float, NB><<<p.n_items, threads, adjoint_smem<float, NB>(), s>>>(m, p);
}

void launch_adjoint_sweep_f32(const DevMesh& m, const AdjSweepParams& p, cudaStream_t s) {
  if (p.n_items <= 0) return;
  switch (m.n) {
    case 8: adj_sweep_n<8>(m, p, s); break;
    case 16: adj_sweep_n<16>(m, p, s); break;
    case 32: adj_sweep_n<32>(m, p, s); break;
  }
}

void prepare_kernels_f32() {
  prepare_sweep_f32<8>();
  prepare_sweep_f32<16>();
  prepare_sweep_f32<32>();
  prepare_adj<8>();
  prepare_adj<16>();
  prepare_adj<32>();
}


}  // namespace cello
