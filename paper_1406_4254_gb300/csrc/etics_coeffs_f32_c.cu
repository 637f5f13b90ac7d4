// etics_coeffs_f32_c.cu -- the mixed-precision SCF coefficient pass
// (etics_scf_coeffs.cuh) for 13, 15 rows (n_max + 1 rounded up to an odd
// number): its own translation unit so that the instantiations compile in
// parallel.
#include "etics_scf_coeffs.cuh"

namespace etics {
size_t scf_coeffs_f32_c_workspace(int rows, int l_max, int num_sms) {
    if (rows == 13) return scf_coeff_plan_workspace<13>(l_max, num_sms);
    if (rows == 15) return scf_coeff_plan_workspace<15>(l_max, num_sms);
    return 0;
}
int scf_coeffs_f32_c(int rows, const void* posm, int64_t N, int n_max, int l_max, int basis,
                     double* coeffs, void* ws, const LaunchCtx& ctx) {
    if (rows == 13)
        return l_max <= 8 ? scf_coeff_plan_launch<13, 8>(posm, N, n_max, l_max, basis, coeffs, ws, ctx)
                          : scf_coeff_plan_launch<13, kLmaxLimit>(posm, N, n_max, l_max, basis, coeffs, ws, ctx);
    if (rows == 15)
        return l_max <= 8 ? scf_coeff_plan_launch<15, 8>(posm, N, n_max, l_max, basis, coeffs, ws, ctx)
                          : scf_coeff_plan_launch<15, kLmaxLimit>(posm, N, n_max, l_max, basis, coeffs, ws, ctx);
    return ETICS_ERR_UNSUPPORTED;
}
}  // namespace etics
