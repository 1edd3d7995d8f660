// Float64 dual-energy sweeps (the shared-memory form with a sixth field rho
// e; method code RS | 4), built without FMA contraction like the float64
// sweep; k_f64.cu plans the launch and calls launch_sweep_de_f64.
#include "kernels.cuh"

namespace cello {

template <int NB, int RS>
static constexpr size_t de_smem64() {
  return sizeof(double) * sweep_arrays(RS) * (NB + 2 * kGhosts) * 8;
}

template <int NB>
void launch_sweep_de_f64(const DevMesh& m, const SweepParams& p, int grid, cudaStream_t s) {
  constexpr int T = (NB + 2 * kGhosts) * 8;
  switch (method_code(m.riemann, m.steepen)) {
    case 0: sweep_kernel<double, NB, 8, 2, 4><<<grid, T, de_smem64<NB, 4>(), s>>>(m, p); break;
    case 1: sweep_kernel<double, NB, 8, 2, 5><<<grid, T, de_smem64<NB, 5>(), s>>>(m, p); break;
    case 2: sweep_kernel<double, NB, 8, 2, 6><<<grid, T, de_smem64<NB, 6>(), s>>>(m, p); break;
    case 3: sweep_kernel<double, NB, 8, 2, 7><<<grid, T, de_smem64<NB, 7>(), s>>>(m, p); break;
  }
}

template void launch_sweep_de_f64<8>(const DevMesh&, const SweepParams&, int, cudaStream_t);
template void launch_sweep_de_f64<16>(const DevMesh&, const SweepParams&, int, cudaStream_t);
template void launch_sweep_de_f64<32>(const DevMesh&, const SweepParams&, int, cudaStream_t);

template <int NB, int RS>
static void prepare_de64(int (*resident)[8], int nbi, int sms) {
  constexpr int T = (NB + 2 * kGhosts) * 8;
  constexpr size_t sh = de_smem64<NB, RS>();
  int nb = 0;
  cudaFuncSetAttribute(sweep_kernel<double, NB, 8, 2, RS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, sweep_kernel<double, NB, 8, 2, RS>, T, sh);
  resident[nbi][RS] = (nb > 0 ? nb : 1) * sms;
}

template <int NB>
static void prepare_de64_nb(int (*resident)[8], int nbi, int sms) {
  prepare_de64<NB, 4>(resident, nbi, sms);
  prepare_de64<NB, 5>(resident, nbi, sms);
  prepare_de64<NB, 6>(resident, nbi, sms);
  prepare_de64<NB, 7>(resident, nbi, sms);
}

void prepare_kernels_de_f64(int (*resident)[8], int sms) {
  prepare_de64_nb<8>(resident, 0, sms);
  prepare_de64_nb<16>(resident, 1, sms);
  prepare_de64_nb<32>(resident, 2, sms);
}

}  // namespace cello
