// etics_scf_cb_f64.cu -- SCF with the Clutton-Brock radial basis (the
// Plummer model as zeroth term; the alternative basis of paper Sec. 2.5):
// the generic coefficient kernel instantiated for basis 1 in
// FP64.
#include "etics_internal.h"
#include "etics_scf_impl.cuh"

namespace etics {
int scf_coeffs_cb_f64(const void* posm, int64_t N, int n_max, int l_max, double* coeffs,
                       void* ws, const LaunchCtx& ctx) {
    return scf_coeffs_launch<double, 1>(posm, N, n_max, l_max, coeffs, ws, ctx);
}
}  // namespace etics
