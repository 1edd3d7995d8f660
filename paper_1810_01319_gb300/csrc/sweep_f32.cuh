// Planners and launchers of the float32 sweep variants for one block size,
// instantiated by k_f32_n8.cu, k_f32_n16.cu and k_f32_n32.cu (one translation
// unit per block size, so that they compile in parallel).
#pragma once

#include "kernels.cuh"

namespace cello {

// Float32 sweep variants.  Shared-memory form: {pencils per CTA, min
// resident CTAs per SM}; register-streaming form: {CTA size = pencils per
// CTA, min resident CTAs per SM}; each without and with the persistent
// schedule (ItemQueue).
static const SweepVariant kVariants[] = {
    {8, 3, false, false},  {8, 4, false, false},  {4, 6, false, false}, {16, 1, false, false},
    {4, 8, false, false},  {16, 2, false, false}, {64, 8, false, true}, {128, 4, false, true},
    {64, 6, false, true},  {32, 16, false, true}, {64, 8, false, true, 3}, {64, 6, false, true, 3},
    {8, 3, true, false},   {8, 4, true, false},   {4, 6, true, false},  {16, 1, true, false},
    {4, 8, true, false},   {16, 2, true, false},  {64, 8, true, true},  {128, 4, true, true},
    {64, 6, true, true},   {32, 16, true, true},  {64, 8, true, true, 3},  {64, 6, true, true, 3},
};
constexpr int kNT = 12;  // distinct kernel instantiations; variant v uses template v % kNT
constexpr int kNV = sizeof(kVariants) / sizeof(kVariants[0]);
static_assert(kNV <= kMaxSweepVariants, "the autotuner keeps a time for each");

// Shared memory of the shared-memory form: sweep_arrays(RS) arrays of N x P
// values (21; 24 with contact steepening).
template <int NB, int P, int RS>
static constexpr size_t sweep_smem() {
  constexpr int N = NB + 2 * kGhosts;
  return sizeof(float) * sweep_arrays(RS) * N * P;
}

template <int NB, int P, int MINB>
static void prepare_variant() {
#define CELLO_ATTR(RS)                                                                                    \
  cudaFuncSetAttribute(sweep_kernel<float, NB, P, MINB, RS>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                       (int)sweep_smem<NB, P, RS>())
  CELLO_ATTR(0);
  CELLO_ATTR(1);
  CELLO_ATTR(2);
  CELLO_ATTR(3);
#undef CELLO_ATTR
}

// Dynamic shared memory of the streaming form: the staged form keeps three
// groups of four cells of five fields per thread, and the updated group.
template <int CT, int VEC>
static constexpr size_t stream_smem() {
  return VEC == 3 ? sizeof(float4) * 4 * 5 * CT : 0;
}

// Work items and schedule of one launch; false if there is no work.
static bool plan_launch(SweepParams& p, int per_cta, int v) {
  p.plan(per_cta);
  p.persistent = kVariants[v].persistent;
  return p.n_items > 0;
}

template <int NB, int P, int MINB>
static void launch_variant(const DevMesh& m, SweepParams p, int v, cudaStream_t s) {
  constexpr int N = NB + 2 * kGhosts;
  if (!plan_launch(p, P, v)) return;
  const int grid = p.n_items;
  switch (method_code(m.riemann, m.steepen, m.nf == 6)) {
    case 0: sweep_kernel<float, NB, P, MINB, 0><<<grid, N * P, sweep_smem<NB, P, 0>(), s>>>(m, p); break;
    case 1: sweep_kernel<float, NB, P, MINB, 1><<<grid, N * P, sweep_smem<NB, P, 1>(), s>>>(m, p); break;
    case 2: sweep_kernel<float, NB, P, MINB, 2><<<grid, N * P, sweep_smem<NB, P, 2>(), s>>>(m, p); break;
    case 3: sweep_kernel<float, NB, P, MINB, 3><<<grid, N * P, sweep_smem<NB, P, 3>(), s>>>(m, p); break;
    default: launch_sweep_de_f32<NB, P, MINB>(m, p, s); break;   // dual energy (sweep_de_f32.cuh)
  }
}

template <int NB, int CT, int MINB, int VEC>
static void launch_stream_variant(const DevMesh& m, SweepParams p, int v, cudaStream_t s) {
  if (!plan_launch(p, CT, v)) return;
  const int grid = p.n_items;
  constexpr size_t sh = stream_smem<CT, VEC>();
  if (m.nf == 6) {   // dual energy (sweep_de_f32.cuh)
    launch_stream_de_f32<NB, CT, VEC>(m, p, s);
    return;
  }
  switch (method_code(m.riemann, m.steepen)) {
    case 0: sweep_stream_kernel<float, NB, CT, MINB, VEC, 0><<<grid, CT, sh, s>>>(m, p); break;
    case 1: sweep_stream_kernel<float, NB, CT, MINB, VEC, 1><<<grid, CT, sh, s>>>(m, p); break;
    case 2: sweep_stream_kernel<float, NB, CT, MINB, VEC, 2><<<grid, CT, sh, s>>>(m, p); break;
    case 3: sweep_stream_kernel<float, NB, CT, MINB, VEC, 3><<<grid, CT, sh, s>>>(m, p); break;
  }
}

template <int NB>
void prepare_sweep_f32() {
  prepare_variant<NB, 8, 3>();
  prepare_variant<NB, 8, 4>();
  prepare_variant<NB, 4, 6>();
  prepare_variant<NB, 16, 1>();
  prepare_variant<NB, 4, 8>();
  prepare_variant<NB, 16, 2>();
  prepare_sweep_de_f32<NB>();
}

// The variant of a sweep that the caller has not chosen one for.  The streaming
// form takes the time of one pencil's walk however few there are (18, 24 and 37
// us for n = 8, 16 and 32), the shared-memory form, a thread per cell, less while
// its CTAs fill one wave: 16.7, 22.8 and 36 us at 14, 16 and 18 thousand pencils,
// 27, 39 and 75 against 22, 31 and 59 us at 33, 37 and 49 thousand.  The
// persistent schedule is never slower than one CTA per item (64 leaves of 16^3:
// 23 against 39 us).  On x the staged form bounded for 6 CTAs per SM is ahead up
// to some hundred thousand pencils (512 leaves of 16^3: 73 against 80 us), for 8
// beyond (4,096 leaves of 32^3: 3.7 against 4.0 ms).
static int default_variant(const SweepParams& p) {
  long pencils = (long)p.nleaf * p.reg3[0].count;
  for (int r = 1; r < 3; ++r) pencils += (long)p.reg3[r].nfaces * p.reg3[r].count;
  if (pencils < 20000) return 12;
  return p.axis != 0 ? 18 : (pencils < 400000 ? 23 : 22);
}

template <int NB>
void launch_sweep_f32_nb(const DevMesh& m, const SweepParams& p, cudaStream_t s) {
  const int v = (p.variant >= 0 && p.variant < kNV) ? p.variant : default_variant(p);
  switch (v % kNT) {
    case 0: launch_variant<NB, 8, 3>(m, p, v, s); break;
    case 1: launch_variant<NB, 8, 4>(m, p, v, s); break;
    case 2: launch_variant<NB, 4, 6>(m, p, v, s); break;
    case 3: launch_variant<NB, 16, 1>(m, p, v, s); break;
    case 4: launch_variant<NB, 4, 8>(m, p, v, s); break;
    case 5: launch_variant<NB, 16, 2>(m, p, v, s); break;
    case 6: launch_stream_variant<NB, 64, 8, 0>(m, p, v, s); break;
    case 7: launch_stream_variant<NB, 128, 4, 0>(m, p, v, s); break;
    case 8: launch_stream_variant<NB, 64, 6, 0>(m, p, v, s); break;
    case 9: launch_stream_variant<NB, 32, 16, 0>(m, p, v, s); break;
    case 10: launch_stream_variant<NB, 64, 8, 3>(m, p, v, s); break;
    case 11: launch_stream_variant<NB, 64, 6, 3>(m, p, v, s); break;
  }
}

}  // namespace cello
