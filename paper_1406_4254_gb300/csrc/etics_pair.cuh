// etics_pair.cuh -- arithmetic on one FP64 value, or on two particles of one
// thread as the halves of a pair: paired FP32 instructions (one issue slot for
// two FMAs; the FMA rate itself is the same, so they pay where issue is what
// limits), or two FP64 ones.  A constant or scalar in both halves (splat) is
// an immediate or broadcast operand and the negation of an operand is free
// (instruction counts measured), so the kernels write both without care.
#pragma once

#include <type_traits>

#include "etics_common.cuh"

namespace etics {

template <typename R> struct PairT;
template <> struct PairT<float> { using type = float2; };
template <> struct PairT<double> { using type = double2; };
template <typename R> using Pair = typename PairT<R>::type;

__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }
// (templates, so that a host program that includes this for the plans compiles
// for any architecture: the intrinsics exist from sm_100 on)
template <typename F> using IfFloat2 = std::enable_if_t<std::is_same<F, float2>::value, F>;
template <typename F> __device__ __forceinline__ IfFloat2<F> mul2(F a, F b) { return __fmul2_rn(a, b); }
template <typename F> __device__ __forceinline__ IfFloat2<F> fma2(F a, F b, F c) {
    return __ffma2_rn(a, b, c);
}
template <typename F> __device__ __forceinline__ IfFloat2<F> add2(F a, F b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ double2 mul2(double2 a, double2 b) {
    return make_double2(a.x * b.x, a.y * b.y);
}
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 add2(double2 a, double2 b) {
    return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double2 neg2(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ double mul2(double a, double b) { return a * b; }
__device__ __forceinline__ double fma2(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double add2(double a, double b) { return a + b; }
__device__ __forceinline__ double neg2(double a) { return -a; }
template <typename P> __device__ __forceinline__ P sub2(P a, P b) { return add2(a, neg2(b)); }
template <typename P, typename R> __device__ __forceinline__ P splat(R a) {
    if constexpr (sizeof(P) == sizeof(R)) return a;
    else return mk2(a, a);
}

// The compiler may not carry a value across this: two walks over the levels
// that evaluate the same harmonics would otherwise keep the first one's for the
// second, far more than the registers hold.
__device__ __forceinline__ void opaque(float& v) { asm volatile("" : "+f"(v)); }
__device__ __forceinline__ void opaque(double& v) { asm volatile("" : "+d"(v)); }

// Solid harmonics R_l^m(kappa u) = kappa^l Z_l^m(u) / (l+m)! at the unit
// vector u, v = kappa u, with Z the unnormalised solid harmonics of
// etics_common.cuh and kappa = 8 (a power of two: the values stay near 1 for
// the orders used, where Z or Z / (l+m)! would spread over 2^60).  In this
// scaling the gradient ladder has no constants:
//   d/dz R_l^m = R_{l-1}^m,  (d/dx -+ i d/dy) R_l^m = +-R_{l-1}^{m-+1}.
// Level L from levels L-1 and L-2, cos parts C[m], sin parts S[m]; with
// |v|^2 = kappa^2 taken out of the recursion:
//   (L^2 - m^2) R_L = kappa^2 [ (2L-1)/kappa^2 v_z R_{L-1} - R_{L-2} ]
constexpr int kKappa = 8;
template <typename R, int L, typename P>
__device__ __forceinline__ void harm_scaled(const P* C1, const P* S1, const P* C2, const P* S2,
                                            P vx, P vy, P vz, P* C, P* S) {
    if constexpr (L == 0) {
        C[0] = splat<P>(R(1));
        S[0] = splat<P>(R(0));
    } else if constexpr (L == 1) {
        C[0] = vz;
        S[0] = splat<P>(R(0));
        C[1] = mul2(vx, splat<P>(R(0.5)));
        S[1] = mul2(vy, splat<P>(R(0.5)));
    } else {
        constexpr R d = R(1.0 / (2 * L)), k2 = R(kKappa * kKappa);
        const P xd = mul2(vx, splat<P>(d)), yd = mul2(vy, splat<P>(d));
        C[L] = fma2(xd, C1[L - 1], neg2(mul2(yd, S1[L - 1])));
        S[L] = fma2(xd, S1[L - 1], mul2(yd, C1[L - 1]));
        C[L - 1] = mul2(vz, C1[L - 1]);
        S[L - 1] = mul2(vz, S1[L - 1]);
        S[0] = splat<P>(R(0));
        const P zl = mul2(vz, splat<P>(R(2 * L - 1) / k2));
#pragma unroll
        for (int m = 0; m + 2 <= L; ++m) {
            const P f = splat<P>(k2 / R(L * L - m * m));
            C[m] = mul2(fma2(zl, C1[m], neg2(C2[m])), f);
            if (m > 0) S[m] = mul2(fma2(zl, S1[m], neg2(S2[m])), f);
        }
    }
}

// warp totals of v[0..K), K a multiple of 32, by a reduce-scatter (each step
// halves the values a lane still holds): lane j ends with the totals of values
// j K/32 .. in v[0..K/32)
template <int K, int O>
__device__ __forceinline__ void warp_scatter(float* v, int lane) {
    if constexpr (O >= 1) {
        const bool up = lane & O;
#pragma unroll
        for (int i = 0; i < K / 2; ++i) {
            const float give = up ? v[i] : v[i + K / 2];
            const float keep = up ? v[i + K / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, O);
        }
        warp_scatter<K / 2, O / 2>(v, lane);
    }
}

// 16-byte asynchronous global -> shared copies
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// kick-drift of one particle: v += h a, x += dt v (h = dt / 2)
template <typename V4, typename R>
__device__ __forceinline__ void kick_drift(V4& x, V4& v, const V4& a, R h, R dt) {
    v.x = fma(h, a.x, v.x);
    v.y = fma(h, a.y, v.y);
    v.z = fma(h, a.z, v.z);
    x.x = fma(dt, v.x, x.x);
    x.y = fma(dt, v.y, x.y);
    x.z = fma(dt, v.z, x.z);
}

}  // namespace etics
