// etics_coeffs_f32_a.cu -- the mixed-precision SCF coefficient pass
// (etics_scf_coeffs.cuh) for 3, 5, 7 rows (n_max + 1 rounded up to an odd
// number): its own translation unit so that the instantiations compile in
// parallel.
#include "etics_scf_coeffs.cuh"

namespace etics {
size_t scf_coeffs_f32_a_workspace(int rows, int l_max, int num_sms) {
    if (rows == 3) return scf_coeff_plan_workspace<3>(l_max, num_sms);
    if (rows == 5) return scf_coeff_plan_workspace<5>(l_max, num_sms);
    if (rows == 7) return scf_coeff_plan_workspace<7>(l_max, num_sms);
    return 0;
}
int scf_coeffs_f32_a(int rows, const void* posm, int64_t N, int n_max, int l_max, int basis,
                     double* coeffs, void* ws, const LaunchCtx& ctx) {
    if (rows == 3)
        return l_max <= 8 ? scf_coeff_plan_launch<3, 8>(posm, N, n_max, l_max, basis, coeffs, ws, ctx)
                          : scf_coeff_plan_launch<3, kLmaxLimit>(posm, N, n_max, l_max, basis, coeffs, ws, ctx);
    if (rows == 5)
        return l_max <= 8 ? scf_coeff_plan_launch<5, 8>(posm, N, n_max, l_max, basis, coeffs, ws, ctx)
                          : scf_coeff_plan_launch<5, kLmaxLimit>(posm, N, n_max, l_max, basis, coeffs, ws, ctx);
    if (rows == 7)
        return l_max <= 8 ? scf_coeff_plan_launch<7, 8>(posm, N, n_max, l_max, basis, coeffs, ws, ctx)
                          : scf_coeff_plan_launch<7, kLmaxLimit>(posm, N, n_max, l_max, basis, coeffs, ws, ctx);
    return ETICS_ERR_UNSUPPORTED;
}
}  // namespace etics
