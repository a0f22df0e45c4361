// Rows a2 + a3 (the work-list forward, with the delta statistics of
// sigma_rel tensors) for bf16 parameters. A translation unit of its own so the
// forward kernels compile in parallel.
// Compiled once per draw family (the packed layout, and with SMAT_DRAW16
// the 16-bit draw option: the _d16 launchers; smat_internal.h).
#include "smat_simulate.cuh"

namespace smat {

cudaError_t SMAT_FAMILY(launch_stats_simulate_bf16)(const KArgs& a, int sms, int noise, bool per_elem_alpha,
                                                    int rounds, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  return (rounds & 0xFF) == 7 ? fused_run<7 | kFamily, DT_BF16, false>(a, sms, noise, per_elem_alpha, s)
                              : fused_run<10 | kFamily, DT_BF16, false>(a, sms, noise, per_elem_alpha, s);
}

int SMAT_FAMILY(fused_wide_ctas_per_sm)(int noise, bool per_elem_alpha, int rounds) {
#define SMAT_WIDE_OCC(R, PE) \
  (noise == NOISE_GAUSSIAN ? FusedVariant<R, DT_BF16, NOISE_GAUSSIAN, PE, false>::occ() \
                           : FusedVariant<R, DT_BF16, NOISE_UNIFORM, PE, false>::occ())
  if (per_elem_alpha) return (rounds & 0xFF) == 7 ? SMAT_WIDE_OCC(7 | kFamily, true) : SMAT_WIDE_OCC(10 | kFamily, true);
  return (rounds & 0xFF) == 7 ? SMAT_WIDE_OCC(7 | kFamily, false) : SMAT_WIDE_OCC(10 | kFamily, false);
#undef SMAT_WIDE_OCC
}

}  // namespace smat
