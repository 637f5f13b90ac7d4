// etics_scf_bins_f32.cu -- the per-warp-bin SCF coefficient pass (see
// etics_scf_bins.cuh) at (n_max, l_max) = (14, 8), the expansion the
// surrogate experiment uses for its bar-perturbed Hernquist sphere (the
// coefficients of Sec. 2.4 eq. 18 in the basis of Sec. 2.5).  12 bins of at most 7
// columns: 384 threads, 105 FP32 accumulators per lane, so one block per SM;
// tiles of 576 particles.  Its own translation unit so that it compiles in
// parallel with the other SCF kernels.
#include "etics_internal.h"
#include "etics_scf_bins.cuh"

namespace etics {
size_t scf_bins148_workspace_f32(int num_sms) {
    return scf_bins_workspace<15, 8>(num_sms);
}
int scf_coeffs_bins148_f32(const void* posm, int64_t N, double* coeffs, void* ws, DriftStep drift,
                           const LaunchCtx& ctx) {
    return scf_coeffs_bins_launch<15, 8>(posm, N, coeffs, ws, drift, ctx);
}
}  // namespace etics
