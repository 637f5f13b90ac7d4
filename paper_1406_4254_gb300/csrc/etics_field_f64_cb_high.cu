// etics_field_f64_cb_high.cu -- the SCF field pass (etics_scf_field.cuh),
// FP64, Clutton-Brock basis (paper Sec. 2.5), l_max > 6: its own translation unit so that
// the instantiations compile in parallel.
#include "etics_scf_field.cuh"

namespace etics {
int scf_field_f64_cb_high(const void* posm, int64_t N, int n_max, int l_max,
                          const double* coeffs, void* out, int out_mask, FieldKick kick,
                          const LaunchCtx& ctx) {
    return scf_field_high<double, 1>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
}
}  // namespace etics
