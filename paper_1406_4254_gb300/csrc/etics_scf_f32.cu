// etics_scf_f32.cu -- mixed-precision SCF instantiation (FP32 basis and field
// sums, FP64 coefficient accumulation).
#include <algorithm>

#include "etics_internal.h"
#include "etics_scf_coeffs.cuh"
#include "etics_scf_impl.cuh"

namespace etics {
size_t scf_workspace_f32(int64_t N, int n_max, int l_max, int num_sms) {
    const int rows = coeff_rows(n_max);
    const auto need = rows <= 7 ? scf_coeffs_f32_a_workspace : rows <= 11 ? scf_coeffs_f32_b_workspace
                      : rows <= 15 ? scf_coeffs_f32_c_workspace : scf_coeffs_f32_d_workspace;
    // at least what the register-tile kernel takes (the FP64 path's, and this
    // path's before it ran on particle pairs)
    size_t most = scf_workspace<float>(N, n_max, l_max, num_sms);
    most = std::max(most, need(rows, l_max, num_sms));
    if (n_max == 10 && l_max == 6) most = std::max(most, scf_pairs106_workspace_f32(num_sms));
    if (n_max == 14 && l_max == 8) most = std::max(most, scf_bins148_workspace_f32(num_sms));
    return most;
}
int scf_coeffs_f32(const void* posm, int64_t N, int n_max, int l_max, int basis, double* coeffs,
                   void* ws, DriftStep drift, const LaunchCtx& ctx) {
    // the paper's (10, 6) and the forecast experiment's (14, 8) expansion have
    // kernels with their bins known at compile time: the pass takes 46.5 us at
    // (10, 6) and 2^20 particles, 359 at (14, 8) and 2^22; the general kernel 66
    // and 705 (timed on the other basis)
    if (basis == ETICS_BASIS_HO && n_max == 10 && l_max == 6)
        return scf_coeffs_pairs106_f32(posm, N, coeffs, ws, drift, ctx);
    if (basis == ETICS_BASIS_HO && n_max == 14 && l_max == 8)
        return scf_coeffs_bins148_f32(posm, N, coeffs, ws, drift, ctx);
    // (here several blocks may read the same particle: the drift comes first)
    if (drift.posm)
        if (const int rc = kick_drift_f32(drift.posm, drift.vel, drift.acc, N, drift.dt, ctx)) return rc;
    const int rows = coeff_rows(n_max);
    const auto run = rows <= 7 ? scf_coeffs_f32_a : rows <= 11 ? scf_coeffs_f32_b
                     : rows <= 15 ? scf_coeffs_f32_c : scf_coeffs_f32_d;
    return run(rows, posm, N, n_max, l_max, basis, coeffs, ws, ctx);
}
int scf_field_f32(const void* posm, int64_t N, int n_max, int l_max, int basis,
                  const double* coeffs, void* out, int out_mask, FieldKick kick,
                  const LaunchCtx& ctx) {
    if (N == 0) return ETICS_OK;
    const auto run = basis == ETICS_BASIS_HO
                         ? (l_max <= 6 ? scf_field_f32_ho_low : scf_field_f32_ho_high)
                         : (l_max <= 6 ? scf_field_f32_cb_low : scf_field_f32_cb_high);
    return run(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
}
}  // namespace etics
