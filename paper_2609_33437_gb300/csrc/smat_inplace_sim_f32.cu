// Row a3 (grid-stride launch, SMAT_FLAG_UNFUSED_STATS) for f32 parameters in
// lists with in-place tensors: the launch of smat_sim_f32.cu instantiated with
// the in-place path (see smat_inplace_f32.cu).
// Compiled once per draw family (the packed layout, and with SMAT_DRAW16
// the 16-bit draw option: the _d16 launchers; smat_internal.h).
#include "smat_simulate.cuh"

namespace smat {

cudaError_t SMAT_FAMILY(launch_simulate_inplace_f32)(const KArgs& a, int grid, int noise, bool per_elem_alpha,
                                                     int rounds, cudaStream_t s) {
  if (a.chunk_end <= a.chunk_begin) return cudaSuccess;
  return (rounds & 0xFF) == 7 ? sim_run<7 | kFamily, DT_F32, true>(a, grid, noise, per_elem_alpha, s)
                              : sim_run<10 | kFamily, DT_F32, true>(a, grid, noise, per_elem_alpha, s);
}

cudaError_t SMAT_FAMILY(launch_direct_inplace_f32)(const KArgs& a, int noise, bool per_elem_alpha, int rounds, cudaStream_t s) {
  if (a.chunk_end <= a.chunk_begin) return cudaSuccess;
  return (rounds & 0xFF) == 7 ? direct_run<7 | kFamily, DT_F32, true>(a, noise, per_elem_alpha, s)
                              : direct_run<10 | kFamily, DT_F32, true>(a, noise, per_elem_alpha, s);
}

}  // namespace smat
