// Float32 dual-energy sweeps (both forms with a sixth field rho e; method
// code RS | 4) for blocks of CELLO_DE_NB cells per edge, one translation unit
// per block size.  Compiled with the float32 sweep's flags; the planners in
// sweep_f32.cuh count the items and call launch_sweep_de_f32 (shared-memory
// form) or launch_stream_de_f32 (register streaming).
#pragma once

#include "kernels.cuh"

namespace cello {

template <int NB, int P, int RS>
static constexpr size_t de_smem() {
  return sizeof(float) * sweep_arrays(RS) * (NB + 2 * kGhosts) * P;
}

template <int NB, int P, int MINB>
void launch_sweep_de_f32(const DevMesh& m, const SweepParams& p, cudaStream_t s) {
  constexpr int T = (NB + 2 * kGhosts) * P;
  const int grid = p.n_items;
  switch (method_code(m.riemann, m.steepen)) {
    case 0: sweep_kernel<float, NB, P, MINB, 4><<<grid, T, de_smem<NB, P, 4>(), s>>>(m, p); break;
    case 1: sweep_kernel<float, NB, P, MINB, 5><<<grid, T, de_smem<NB, P, 5>(), s>>>(m, p); break;
    case 2: sweep_kernel<float, NB, P, MINB, 6><<<grid, T, de_smem<NB, P, 6>(), s>>>(m, p); break;
    case 3: sweep_kernel<float, NB, P, MINB, 7><<<grid, T, de_smem<NB, P, 7>(), s>>>(m, p); break;
  }
}

// Register-streaming form: VEC = 3 stages three groups of four cells of the
// six fields per thread in shared memory, and the updated group.  The window of
// six fields does not fit the 128 registers of the five-field kernels (512
// threads per SM): every variant is bounded for 384 threads per SM (168
// registers), where nothing spills.  At 128 registers the spills (100 to 670
// bytes a thread) cost more than the extra warps give: 183 leaves of 32^3 with
// HLLC and steepening, two steps of variants 22, 21, 21, 2.06 -> 1.72 ms.
template <int NB, int CT, int VEC>
void launch_stream_de_f32(const DevMesh& m, const SweepParams& p, cudaStream_t s) {
  constexpr int MINB = 384 / CT;
  constexpr size_t sh = VEC == 3 ? sizeof(float4) * 4 * 6 * CT : 0;
  const int grid = p.n_items;
  switch (method_code(m.riemann, m.steepen)) {
    case 0: sweep_stream_kernel<float, NB, CT, MINB, VEC, 4><<<grid, CT, sh, s>>>(m, p); break;
    case 1: sweep_stream_kernel<float, NB, CT, MINB, VEC, 5><<<grid, CT, sh, s>>>(m, p); break;
    case 2: sweep_stream_kernel<float, NB, CT, MINB, VEC, 6><<<grid, CT, sh, s>>>(m, p); break;
    case 3: sweep_stream_kernel<float, NB, CT, MINB, VEC, 7><<<grid, CT, sh, s>>>(m, p); break;
  }
}

// The streaming variants of the float32 table: {CTA size, vector I/O}.
#define CELLO_DE_STREAM(X, NB) X(NB, 64, 0) X(NB, 128, 0) X(NB, 32, 0) X(NB, 64, 3)
#define CELLO_DE_SINST(NB, CT, VEC) \
  template void launch_stream_de_f32<NB, CT, VEC>(const DevMesh&, const SweepParams&, cudaStream_t);
CELLO_DE_STREAM(CELLO_DE_SINST, CELLO_DE_NB)
#undef CELLO_DE_SINST
#undef CELLO_DE_STREAM

template <int NB, int P, int MINB>
static void prepare_de() {
#define CELLO_DE_ATTR(RS)                                                                                 \
  cudaFuncSetAttribute(sweep_kernel<float, NB, P, MINB, RS>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                       (int)de_smem<NB, P, RS>())
  CELLO_DE_ATTR(4);
  CELLO_DE_ATTR(5);
  CELLO_DE_ATTR(6);
  CELLO_DE_ATTR(7);
#undef CELLO_DE_ATTR
}

// The shared-memory variants of the float32 table: {pencils, min CTAs per SM}.
#define CELLO_DE_VARIANTS(X, NB) X(NB, 8, 3) X(NB, 8, 4) X(NB, 4, 6) X(NB, 16, 1) X(NB, 4, 8) X(NB, 16, 2)
#define CELLO_DE_INST(NB, P, MINB) \
  template void launch_sweep_de_f32<NB, P, MINB>(const DevMesh&, const SweepParams&, cudaStream_t);
CELLO_DE_VARIANTS(CELLO_DE_INST, CELLO_DE_NB)
#undef CELLO_DE_INST

template <>
void prepare_sweep_de_f32<CELLO_DE_NB>() {
#define CELLO_DE_PREP(NB, P, MINB) prepare_de<NB, P, MINB>();
  CELLO_DE_VARIANTS(CELLO_DE_PREP, CELLO_DE_NB)
#undef CELLO_DE_PREP
}
#undef CELLO_DE_VARIANTS

}  // namespace cello
