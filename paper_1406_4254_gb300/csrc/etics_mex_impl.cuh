// etics_mex_impl.cuh -- MEX kernels after the radial sort (templated on the
// arithmetic type; instantiated in etics_mex_f32.cu / etics_mex_f64.cu).
//
// Method (paper Sec. 2.4 eqs. 15-17, the sorted cumulative sums of Sec. 2.2):
//   q_lm(i) = sum_{j before i} m_j r_j^l Y_lm(j),  p_lm(i) = sum_{j after i} m_j r_j^-(l+1) Y_lm(j)
//   Phi_i   = -sum_l 4pi/(2l+1) sum_m [q_lm(i) r_i^-(l+1) + p_lm(i) r_i^l] Y_lm(i)
// and a_i = -grad Phi_i at fixed q, p.
//
// GB300 design (the paper ran one library scan per (l, m) and direction):
//   pass 1  reduces each tile of the sorted particles' moments m rho^l Y and
//           m rho^-(l+1) Y (rho = r / s_t, s_t a power of two per tile, so
//           FP32 never overflows) to one FP64 sum per component.
//   carry   scans the per-tile FP64 sums in a fixed order: exclusive forward
//           for the inner moments, exclusive reverse (a true suffix sum) for
//           the outer ones -- deterministic.
//   pass 2  forms the moments of the tile again, scans them in shared memory
//           from the tile carry (forward and reverse) and evaluates the field
//           at every particle from its exclusive q and p together; (a, Phi)
//           is scattered back to the caller's order.
//
// A thread owns two neighbouring particles of the sorted list and runs them
// as the two halves of paired FP32 instructions; it walks the levels one
// after the other, so that only two levels of harmonics and one level of
// sums are live, whatever l_max is.  The per-thread moment sums go through
// shared memory (one row of kMexThreads values per component, padded so that
// both access patterns, thread = particle pair and thread = component, are
// free of bank conflicts); one thread per component then runs down its row.
// Nothing per particle but the sorted copy reaches memory between the passes.
// What bounds them: instruction issue (pass 2), latency and shared memory (pass
// 1, which reads the copy in radial order that the sort leaves).  Measured
// against the form it replaced (seven particles per thread, all 98 sums of
// l_max = 6 in registers, every thread's prefix sums through memory, the
// particles gathered in pass 1): N = 2^20, l_max = 6: pass 1 51 -> 25 us, pass 2
// 61 -> 51 us.  Whole calls with the sort by buckets: N = 500009, l_max = 10:
// 291 -> 145 us; N = 100003, l_max = 6, FP64: 450 -> 323 us (256-particle tiles
// also fill the SMs more evenly).
//
// Harmonics: the scaled ones of etics_pair.cuh, at kappa u.  The product of an
// evaluated and a summed harmonic needs the weight (l-m)!(l+m)! kappa^-2l
// (twice that for m > 0: the twos are applied to the sums over m > 0 as a
// whole).
#pragma once

#include <atomic>

#include "etics_internal.h"
#include "etics_pair.cuh"

namespace etics {

constexpr int kMexThreads = 128;
constexpr int kMexTile = 2 * kMexThreads;         // particles per tile, two per thread
constexpr int kMexLB = kMexLmaxLimit;             // compiled level bound (10)
constexpr int kMexNC = 49;                        // components of one level group, at most
constexpr int kMexRow = kMexThreads + 4;          // row stride of the shared rows (conflict-free
                                                  // for 16-byte reads down a row)

// Level groups: the shared rows hold the components of one group of levels,
// so that l_max up to kMexLB leaves room for several blocks per SM.  A group's
// harmonics are recurred from level 0 (cheap next to the sums).
constexpr int kMexGroups = 3;
__host__ __device__ constexpr int mex_group_l0(int g) { return g == 0 ? 0 : (g == 1 ? 7 : 9); }
__host__ __device__ constexpr int mex_group_l1(int g) { return g == 0 ? 6 : (g == 1 ? 8 : 10); }
__host__ __device__ constexpr int mex_ncomp(int l_max) { return (l_max + 1) * (l_max + 1); }
// components per side that the workspace has room for (one size for all
// l_max <= 6); the passes use mex_ncomp of them
__host__ __device__ constexpr int mex_layout_ncomp(int l_max) {
    return l_max <= 6 ? kMexNC : mex_ncomp(l_max);
}
static_assert(mex_group_l1(kMexGroups - 1) == kMexLB, "groups cover the compiled levels");
static_assert(mex_ncomp(6) <= kMexNC && mex_ncomp(8) - mex_ncomp(6) <= kMexNC &&
              mex_ncomp(10) - mex_ncomp(8) <= kMexNC, "group size");
static_assert(2 * kMexNC <= kMexThreads, "one thread per component and side");
inline int mex_ngroups(int l_max) {
    int g = 1;
    while (g < kMexGroups && mex_group_l0(g) <= l_max) ++g;
    return g;
}
// components per side of the largest group present
inline int mex_row_comps(int l_max) {
    int most = 0;
    for (int g = 0; g < mex_ngroups(l_max); ++g) {
        const int l1 = mex_group_l1(g) < l_max ? mex_group_l1(g) : l_max;
        const int n = mex_ncomp(l1) - mex_group_l0(g) * mex_group_l0(g);
        if (n > most) most = n;
    }
    return most;
}

inline int mex_tiles(int64_t N) { return (int)((N + kMexTile - 1) / kMexTile); }

// (l-m)!(l+m)! kappa^-2l, the weight of component (l, m)
struct MexWeights {
    double w[(kMexLB + 1) * (kMexLB + 2) / 2];
    float wf[(kMexLB + 1) * (kMexLB + 2) / 2];
};
constexpr MexWeights make_mex_weights() {
    MexWeights t{};
    for (int l = 0; l <= kMexLB; ++l)
        for (int m = 0; m <= l; ++m) {
            double v = 1.0;
            for (int k = 2; k <= l - m; ++k) v *= (double)k;
            for (int k = 2; k <= l + m; ++k) v *= (double)k;
            for (int k = 0; k < l; ++k) v /= (double)(kKappa * kKappa);
            t.w[l * (l + 1) / 2 + m] = v;
            t.wf[l * (l + 1) / 2 + m] = (float)v;
        }
    return t;
}
static __constant__ MexWeights c_mex_w = make_mex_weights();
template <typename R> __device__ __forceinline__ R mex_w(int idx);
template <> __device__ __forceinline__ float mex_w<float>(int idx) { return c_mex_w.wf[idx]; }
template <> __device__ __forceinline__ double mex_w<double>(int idx) { return c_mex_w.w[idx]; }

// tile scale exponent: s_t = 2^e with e halfway (in log2) between the first
// and last radius of the tile (first radius 0 -> use the last)
template <typename R>
__device__ __forceinline__ int tile_exponent(R r_first, R r_last) {
    if (!(r_last > R(0))) return 0;
    const int el = ilogb(r_last);
    const int ef = r_first > R(0) ? ilogb(r_first) : el;
    const int s = ef + el;
    return s >= 0 ? s / 2 : -((-s + 1) / 2);
}

template <typename R>
__device__ __forceinline__ R radius(R x, R y, R z) {
    return sqrt(x * x + y * y + z * z);
}

// x 2^k, exact unless the result leaves the normal range: the exponent field
// is edited in place (FP64 instructions are slow on this GPU)
__device__ __forceinline__ double scale_pow2(double x, int k) {
    const int hi = __double2hiint(x);
    const int ef = (hi >> 20) & 0x7ff;
    if (ef != 0 && ef + k > 0 && ef + k < 0x7ff)
        return __hiloint2double(hi + (k << 20), __double2loint(x));
    return ldexp(x, k);
}

// the tile's two particles of a thread, in tile units: v = kappa u, rho = r / s
template <typename R>
struct MexPair {
    Pair<R> x, y, z, rho, irho, m;
    __device__ __forceinline__ void init(const Vec4<R>& a, const Vec4<R>& b, R scale, R iscale) {
        const R ra = radius<R>(a.x, a.y, a.z), rb = radius<R>(b.x, b.y, b.z);
        // a particle at the origin: no direction, no outer moment, rho = 0
        const R ia = ra > R(0) ? R(1) / ra : R(0), ib = rb > R(0) ? R(1) / rb : R(0);
        const R ka = R(kKappa) * ia, kb = R(kKappa) * ib;
        x = mk2(a.x * ka, b.x * kb);
        y = mk2(a.y * ka, b.y * kb);
        z = mk2(a.z * ka, b.z * kb);
        rho = mk2(ra * scale, rb * scale);
        irho = mk2(ia * iscale, ib * iscale);
        m = mk2(a.w, b.w);
    }
};

// The two walks over the levels (moments, field) and the walks of later level
// groups must not keep one another's harmonics (l_max > 6: 2 KB of spills per
// thread without this).
template <typename R> __device__ __forceinline__ void opaque_pair(MexPair<R>& p) {
    opaque(p.x.x); opaque(p.x.y);
    opaque(p.y.x); opaque(p.y.y);
    opaque(p.z.x); opaque(p.z.y);
    opaque(p.rho.x); opaque(p.rho.y);
    opaque(p.irho.x); opaque(p.irho.y);
}

// moments of the pair summed, component c = l*l + 2m-1 (cos) / 2m (sin) of
// levels L0..L1 into this thread's column of the rows (inner components first,
// outer ones nc rows further)
template <typename R, int L0, int L1, int L>
__device__ __forceinline__ void mex_moments(Pair<R> (&C)[3][L1 + 1], Pair<R> (&S)[3][L1 + 1],
                                            const MexPair<R>& p, int l_max, Pair<R> win,
                                            Pair<R> wout, R* col, int nc) {
    if constexpr (L <= L1) {
        if (L > l_max) return;
        constexpr int s0 = L % 3, s1 = (L + 2) % 3, s2 = (L + 1) % 3;
        harm_scaled<R, L>(C[s1], S[s1], C[s2], S[s2], p.x, p.y, p.z, C[s0], S[s0]);
        if constexpr (L >= L0) {
            constexpr int o = L * L - L0 * L0;
#pragma unroll
            for (int c = 0; c <= 2 * L; ++c) {
                const Pair<R> h = c == 0 ? C[s0][0] : ((c & 1) ? C[s0][(c + 1) / 2] : S[s0][c / 2]);
                col[(o + c) * kMexRow] = fma(win.y, h.y, win.x * h.x);
                col[(nc + o + c) * kMexRow] = fma(wout.y, h.y, wout.x * h.x);
            }
        }
        mex_moments<R, L0, L1, L + 1>(C, S, p, l_max, mul2(win, p.rho), mul2(wout, p.irho), col,
                                      nc);
    }
}

template <typename R, int G>
__device__ __forceinline__ void mex_group_moments(const MexPair<R>& p, int l_max, R* col, int nc) {
    constexpr int L0 = mex_group_l0(G), L1 = mex_group_l1(G);
    Pair<R> C[3][L1 + 1], S[3][L1 + 1];
    mex_moments<R, L0, L1, 0>(C, S, p, l_max, p.m, mul2(p.m, p.irho), col, nc);
}

// field of the pair, in tile units (rho = r / s), of levels L0..L1 from the
// weighted exclusive sums in this thread's column.  With s_lm = q rho^-(l+2)
// + p rho^(l-1) (both already weighted), l >= 1:
//   Phi = -(1/s) [ rho sum s R + q_00 / rho + p_00 ]
//   a   = (1/s^2) [ kappa sum s grad R - u (sum (2l+1) q rho^-(l+2) R + q_00 / rho^2) ]
// so one gradient contraction serves both parts.  The potential alone takes
// s_lm = q rho^-(l+1) + p rho^l, which stays in range for wider tiles.  The column holds the sums
// over the particles before (after) the pair; the second particle's q also
// holds the first, the first one's p the second (own: the first particle's
// m rho^l and the second one's m rho^-(l+1); ownf: their factors per level).
template <typename R>
struct MexField {
    using P = Pair<R>;
    P s0, s1;             // sum s R: m = 0, m > 0 (the latter counts twice)
    P rad;                // sum (2l+1) q rho^-(l+2) R
    P vx, vy, vz0, vz1;   // sum s grad R (vz1: k > 0, counts twice)
    P pot0;               // level 0
};

template <typename R, int L0, int L1, int L, bool ACC>
__device__ __forceinline__ void mex_eval(Pair<R> (&C)[3][L1 + 1], Pair<R> (&S)[3][L1 + 1],
                                         const MexPair<R>& p, int l_max, Pair<R> a, Pair<R> b,
                                         Pair<R> own, Pair<R> ownf, const R* col, int nc,
                                         MexField<R>& f) {
    using P = Pair<R>;
    if constexpr (L <= L1) {
        if (L > l_max) return;
        constexpr int s0 = L % 3, s1 = (L + 2) % 3, s2 = (L + 1) % 3;
        harm_scaled<R, L>(C[s1], S[s1], C[s2], S[s2], p.x, p.y, p.z, C[s0], S[s0]);
        if constexpr (L >= L0) {
            constexpr int o = L * L - L0 * L0;
            if constexpr (L == 0) {
                const R q = col[0], pp = col[nc * kMexRow];
                const P q2 = mk2(q, q + own.x), p2 = mk2(pp + own.y, pp);
                f.pot0 = fma2(q2, p.irho, p2);
                if (ACC) f.rad = mul2(q2, a);
            } else if constexpr (!ACC) {
                // the level's sums of q R and p R before their powers of the radius
                P q0, p0, q1, p1;
#pragma unroll
                for (int m = 0; m <= L; ++m) {
                    const P wm = mul2(own, splat<P>(mex_w<R>(L * (L + 1) / 2 + m)));
#pragma unroll
                    for (int s = 0; s < (m > 0 ? 2 : 1); ++s) {
                        const int cc = o + (m == 0 ? 0 : 2 * m - 1 + s);
                        const R q = col[cc * kMexRow], pp = col[(nc + cc) * kMexRow];
                        const P h = s == 0 ? C[s0][m] : S[s0][m];
                        const P q2 = mk2(q, fma(wm.x, h.x, q)), p2 = mk2(fma(wm.y, h.y, pp), pp);
                        if (m == 0) {
                            q0 = mul2(q2, h);
                            p0 = mul2(p2, h);
                        } else {
                            q1 = m == 1 && s == 0 ? mul2(q2, h) : fma2(q2, h, q1);
                            p1 = m == 1 && s == 0 ? mul2(p2, h) : fma2(p2, h, p1);
                        }
                    }
                }
                f.s0 = fma2(a, q0, fma2(b, p0, f.s0));
                f.s1 = fma2(a, q1, fma2(b, p1, f.s1));
            } else {
                P ac[L + 1], as[L + 1];
                P r0 = splat<Pair<R>>(R(0)), r1 = splat<Pair<R>>(R(0));
#pragma unroll
                for (int m = 0; m <= L; ++m) {
                    const R w = mex_w<R>(L * (L + 1) / 2 + m);
                    const P wm = mul2(own, splat<P>(w));
                    {
                        const int cc = o + (m == 0 ? 0 : 2 * m - 1);
                        const R q = col[cc * kMexRow], pp = col[(nc + cc) * kMexRow];
                        const P h = C[s0][m];
                        const P qa = mul2(mk2(q, fma(wm.x, h.x, q)), a);
                        ac[m] = fma2(mk2(fma(wm.y, h.y, pp), pp), b, qa);
                        if (m == 0) f.s0 = fma2(ac[m], h, f.s0);
                        else f.s1 = fma2(ac[m], h, f.s1);
                        if (m == 0) r0 = mul2(qa, h);
                        else r1 = fma2(qa, h, r1);
                    }
                    as[m] = splat<Pair<R>>(R(0));
                    if (m > 0) {
                        const int cc = o + 2 * m;
                        const R q = col[cc * kMexRow], pp = col[(nc + cc) * kMexRow];
                        const P h = S[s0][m];
                        const P qa = mul2(mk2(q, fma(wm.x, h.x, q)), a);
                        as[m] = fma2(mk2(fma(wm.y, h.y, pp), pp), b, qa);
                        f.s1 = fma2(as[m], h, f.s1);
                        r1 = fma2(qa, h, r1);
                    }
                }
                f.rad = fma2(splat<Pair<R>>(R(2 * L + 1)), r0, f.rad);
                f.rad = fma2(splat<Pair<R>>(R(2 * (2 * L + 1))), r1, f.rad);
                // gradient from the level below (the ladder regrouped by the
                // harmonic it multiplies)
                const P* C1 = C[s1];
                const P* S1 = S[s1];
#pragma unroll
                for (int k = 0; k <= L - 1; ++k) {
                    const P xc = k >= 1 ? sub2(ac[k + 1], ac[k - 1]) : ac[k + 1];
                    const P yc = k >= 2 ? add2(as[k + 1], as[k - 1]) : as[k + 1];
                    f.vx = fma2(xc, C1[k], f.vx);
                    f.vy = fma2(yc, C1[k], f.vy);
                    if (k == 0) f.vz0 = fma2(ac[k], C1[k], f.vz0);
                    if (k >= 1) {
                        const P xs = k >= 2 ? sub2(as[k + 1], as[k - 1]) : as[k + 1];
                        const P ys = add2(ac[k + 1], ac[k - 1]);
                        f.vz1 = fma2(ac[k], C1[k], f.vz1);
                        f.vx = fma2(xs, S1[k], f.vx);
                        f.vy = fma2(neg2(ys), S1[k], f.vy);
                        f.vz1 = fma2(as[k], S1[k], f.vz1);
                    }
                }
            }
        }
        // a_l = rho^-(l+2); b_l = rho^(l-1), b_1 = 1 (without the force: once more rho)
        const P bn = L == 0 ? b : mul2(b, p.rho);
        mex_eval<R, L0, L1, L + 1, ACC>(C, S, p, l_max, mul2(a, p.irho), bn, mul2(own, ownf), ownf,
                                        col, nc, f);
    }
}

template <typename R, int G, bool ACC>
__device__ __forceinline__ void mex_group_eval(const MexPair<R>& p, int l_max, const R* col, int nc,
                                               MexField<R>& f) {
    constexpr int L0 = mex_group_l0(G), L1 = mex_group_l1(G);
    Pair<R> C[3][L1 + 1], S[3][L1 + 1];
    mex_eval<R, L0, L1, 0, ACC>(C, S, p, l_max, ACC ? mul2(p.irho, p.irho) : p.irho,
                                ACC ? splat<Pair<R>>(R(1)) : p.rho,
                                mk2(p.m.x, p.m.y * p.irho.y), mk2(p.rho.x, p.irho.y), col, nc, f);
}

// level of component c
__device__ __forceinline__ int comp_level(int c) {
    int l = 0;
    while ((l + 1) * (l + 1) <= c) ++l;
    return l;
}

// tile frame shared by both passes: this thread's two particles and the
// tile's scale exponent
template <typename R>
__device__ __forceinline__ int mex_tile_exponent(const Vec4<R>& a, const Vec4<R>& b, int nt, R* s_end) {
    const int tid = threadIdx.x;
    if (tid == 0) s_end[0] = radius<R>(a.x, a.y, a.z);
    if (2 * tid == nt - 1) s_end[1] = radius<R>(a.x, a.y, a.z);
    if (2 * tid + 1 == nt - 1) s_end[1] = radius<R>(b.x, b.y, b.z);
    __syncthreads();
    return tile_exponent<R>(s_end[0], s_end[1]);
}

// resident blocks per SM the registers are sized for
// (FP32 pass 2: 118 registers for l_max <= 6, 158 with the later level groups;
// FP64 218, and 168 for the potential alone, which three blocks fill the FP64 pipe
// with while one scans: l_max = 2 at 2^20 840 -> 724 us)
template <typename R>
constexpr int mex_pass1_blocks() { return sizeof(R) == 4 ? 4 : 2; }
template <typename R, int NG, bool ACC>
constexpr int mex_pass2_blocks() {
    return sizeof(R) == 4 ? (NG == 1 ? 4 : 3) : NG == 1 && !ACC ? 3 : 2;
}

// ---------------------------------------------------------------------------
// pass 1: per-tile FP64 moment sums
// ---------------------------------------------------------------------------
template <typename R, int NG>
__global__ void __launch_bounds__(kMexThreads, mex_pass1_blocks<R>())
mex_pass1_kernel(const Vec4<R>* sorted, int64_t N, int l_max,
                 double* tile_agg, int stride, unsigned* err) {
    extern __shared__ __align__(16) unsigned char mex_smem[];
    R* rows = reinterpret_cast<R*>(mex_smem);
    __shared__ R s_end[2];
    pdl_wait();
    const int tid = threadIdx.x;
    const int64_t base = (int64_t)blockIdx.x * kMexTile;
    const int64_t rem = N - base;
    const int nt = (int)(rem < kMexTile ? rem : kMexTile);
    Vec4<R> v[2];
#pragma unroll
    for (int j = 0; j < 2; ++j)
        v[j] = 2 * tid + j < nt ? ld4(sorted + base + 2 * tid + j) : mk4<R>(R(0), R(0), R(0), R(0));
    const int e = mex_tile_exponent<R>(v[0], v[1], nt, s_end);
    MexPair<R> p;
    p.init(v[0], v[1], ldexp(R(1), -e), ldexp(R(1), e));
    const int ncomp = mex_ncomp(l_max);
    for (int g = 0; g < NG; ++g) {
        const int L0 = mex_group_l0(g), L1 = mex_group_l1(g);
        if (L0 > l_max) break;
        const int c0 = L0 * L0;
        const int nc = mex_ncomp(L1 < l_max ? L1 : l_max) - c0;
        if (g > 0) __syncthreads();   // the previous group's rows have been read
        opaque_pair(p);
        if (NG == 1 || g == 0) mex_group_moments<R, 0>(p, l_max, rows + tid, nc);
        else if (g == 1) mex_group_moments<R, 1>(p, l_max, rows + tid, nc);
        else mex_group_moments<R, 2>(p, l_max, rows + tid, nc);
        __syncthreads();
        if (tid < 2 * nc) {
            // one thread per component: four interleaved sums down the row
            const Vec4<R>* row = reinterpret_cast<const Vec4<R>*>(rows + tid * kMexRow);
            Vec4<R> s = ld4(row);
#pragma unroll 8
            for (int i = 1; i < kMexThreads / 4; ++i) {
                const Vec4<R> t = ld4(row + i);
                s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
            }
            const R sum = (s.x + s.y) + (s.z + s.w);
            if (!isfinite(sum)) report(err, ETICS_ERR_NONFINITE);
            const bool inner = tid < nc;
            const int cc = c0 + (inner ? tid : tid - nc);
            const int l = comp_level(cc);
            // undo the tile scale: inner moments scale as s^l, outer as s^-(l+1)
            const double d = scale_pow2((double)sum, inner ? l * e : -(l + 1) * e);
            if (!isfinite(d)) report(err, ETICS_ERR_NONFINITE);
            tile_agg[(size_t)((inner ? 0 : ncomp) + cc) * stride + blockIdx.x] = d;
        }
    }
}

// ---------------------------------------------------------------------------
// carry: exclusive scans of the tile sums over tiles, one block per
// component; forward for inner moments, reverse for outer (fixed order).
// The sums of a component lie next to each other ([component][tile]), so a
// thread takes kCarryRun neighbouring ones with wide loads, all in flight at
// once, adds them in order, the run totals are scanned by one warp-shuffle
// scan per warp and one over the warp totals, and each thread writes its
// positions' exclusive sums; longer lists go segment by segment.  FP64
// additions are slow on this GPU (about 1/76 of the FP32 rate): two per sum.
// Every addition order depends only on ntiles: deterministic.
// ---------------------------------------------------------------------------
constexpr int kCarryThreads = 256;
constexpr int kCarryWarps = kCarryThreads / 32;
constexpr int kCarryRun = 16;
static __global__ void __launch_bounds__(kCarryThreads)
mex_carry_kernel(const double* tile_agg, int ntiles, int stride, int ncomp,
                 double* carry) {
    __shared__ double s_w[kCarryWarps + 1];
    pdl_wait();   // the tile sums come from pass 1
    const int c = blockIdx.x;
    const bool rev = c >= ncomp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double* src = tile_agg + (size_t)c * stride;
    double* dst = carry + (size_t)c * stride;
    double before = 0.0;   // sum of the earlier segments
    // scan position o of the component is tile o (forward) or ntiles-1-o
    for (int s0 = 0; s0 < ntiles; s0 += kCarryThreads * kCarryRun) {
        const int left = ntiles - s0;
        const int run = left >= kCarryThreads * kCarryRun
                            ? kCarryRun : (left + kCarryThreads - 1) / kCarryThreads;
        const int o0 = s0 + tid * run;
        double v[kCarryRun];   // read coherently after the wait
#pragma unroll
        for (int k = 0; k < kCarryRun; ++k) {
            const int o = o0 + k;
            v[k] = k < run && o < ntiles ? ld_cg(src + (rev ? ntiles - 1 - o : o)) : 0.0;
        }
        double local = v[0];
#pragma unroll
        for (int k = 1; k < kCarryRun; ++k)
            if (k < run) local += v[k];
        // inclusive scan of the run totals over the warp
        double x = local;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += t;
        }
        double ex = __shfl_up_sync(0xffffffffu, x, 1);
        if (lane == 0) ex = 0.0;
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        if (warp == 0) {
            // exclusive scan of the warp totals, in warp order; the last slot
            // gets the segment's total
            double w = lane < kCarryWarps ? s_w[lane] : 0.0;
#pragma unroll
            for (int d = 1; d <= kCarryWarps; d <<= 1) {
                const double t = __shfl_up_sync(0xffffffffu, w, d);
                if (lane >= d) w += t;
            }
            double we = __shfl_up_sync(0xffffffffu, w, 1);
            if (lane == 0) we = 0.0;
            __syncwarp();
            if (lane <= kCarryWarps) s_w[lane] = we;
        }
        __syncthreads();
        double at = (before + s_w[warp]) + ex;
#pragma unroll
        for (int k = 0; k < kCarryRun; ++k) {
            const int o = o0 + k;
            if (k < run && o < ntiles) {
                dst[rev ? ntiles - 1 - o : o] = at;
                at += v[k];
            }
        }
        before += s_w[kCarryWarps];
        __syncthreads();   // s_w is written again
    }
}

// ---------------------------------------------------------------------------
// pass 2: field from the exclusive sums, per level group
// ---------------------------------------------------------------------------
// exclusive sums of one component over four neighbouring pairs: the values
// before (inner) or after (outer) each of them, of the sum `run` over what
// lies on the other side of the four; then times the component's weight w on
// top of the weighted tile carry `base`.  `run` takes in the four.
template <typename R, bool kInner>
__device__ __forceinline__ Vec4<R> mex_scan4(const Vec4<R>& t, R& run, R w, R base) {
    const R b = fma(w, run, base);
    if constexpr (kInner) {
        const R t2 = t.x + t.y, t3 = t2 + t.z;
        run += t2 + (t.z + t.w);
        return mk4<R>(b, fma(w, t.x, b), fma(w, t2, b), fma(w, t3, b));
    } else {
        const R t2 = t.w + t.z, t3 = t2 + t.y;
        run += t2 + (t.y + t.x);
        return mk4<R>(fma(w, t3, b), fma(w, t2, b), fma(w, t.w, b), b);
    }
}

// one thread down the row of its component: forward for inner, reverse for
// outer components (a true suffix sum, never total minus prefix)
template <typename R>
__device__ __forceinline__ void mex_scan_row(Vec4<R>* row, bool inner, R q0, R w) {
    R run = R(0);
    const R base = w * q0;
    if (inner) {
#pragma unroll 4
        for (int i = 0; i < kMexThreads / 4; ++i)
            st4(row + i, mex_scan4<R, true>(ld4(row + i), run, w, base));
    } else {
#pragma unroll 4
        for (int i = kMexThreads / 4 - 1; i >= 0; --i)
            st4(row + i, mex_scan4<R, false>(ld4(row + i), run, w, base));
    }
}

// one warp over the row of one component (four pairs per lane)
template <typename R>
__device__ __forceinline__ void mex_scan_row_warp(Vec4<R>* row, bool inner, R q0, R w, int lane) {
    static_assert(kMexThreads == 128, "four pairs per lane");
    const Vec4<R> t = ld4(row + lane);
    R x = (t.x + t.y) + (t.z + t.w);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const R o = inner ? __shfl_up_sync(0xffffffffu, x, d) : __shfl_down_sync(0xffffffffu, x, d);
        if (inner ? lane >= d : lane + d < 32) x += o;
    }
    R run = inner ? __shfl_up_sync(0xffffffffu, x, 1) : __shfl_down_sync(0xffffffffu, x, 1);
    if (lane == (inner ? 0 : 31)) run = R(0);
    const R base = w * q0;
    st4(row + lane, inner ? mex_scan4<R, true>(t, run, w, base) : mex_scan4<R, false>(t, run, w, base));
}

// Components left over after whole warps of 32: up to this many go to the
// next warp one after the other, all its lanes on one row (l_max = 6: 96 + 2
// components; a fourth warp walking two rows serially would cost as much as
// the other three).
constexpr int kMexLeftover = 8;

template <typename R, int NG, bool ACC>
__global__ void __launch_bounds__(kMexThreads, (mex_pass2_blocks<R, NG, ACC>()))
mex_pass2_kernel(const Vec4<R>* sorted, const uint32_t* perm, int64_t N,
                 int l_max, const double* carry, int stride,
                 Vec4<R>* out, int out_mask, unsigned* err) {
    extern __shared__ __align__(16) unsigned char mex_smem[];
    R* rows = reinterpret_cast<R*>(mex_smem);
    __shared__ R s_end[2];
    pdl_wait();
    const int tid = threadIdx.x;
    const int64_t base = (int64_t)blockIdx.x * kMexTile;
    const int64_t rem = N - base;
    const int nt = (int)(rem < kMexTile ? rem : kMexTile);
    Vec4<R> v[2];
#pragma unroll
    for (int j = 0; j < 2; ++j)
        v[j] = 2 * tid + j < nt ? ld4(sorted + base + 2 * tid + j) : mk4<R>(R(0), R(0), R(0), R(0));
    uint32_t dst[2];   // in flight until the end
#pragma unroll
    for (int j = 0; j < 2; ++j) dst[j] = 2 * tid + j < nt ? perm[base + 2 * tid + j] : 0u;
    const int e = mex_tile_exponent<R>(v[0], v[1], nt, s_end);
    const R scale = ldexp(R(1), -e);
    MexPair<R> p;
    p.init(v[0], v[1], scale, ldexp(R(1), e));
    MexField<R> f;
    const Pair<R> zero = splat<Pair<R>>(R(0));
    f.s0 = f.s1 = f.rad = f.vx = f.vy = f.vz0 = f.vz1 = f.pot0 = zero;
    const int ncomp = mex_ncomp(l_max);
    for (int g = 0; g < NG; ++g) {
        const int L0 = mex_group_l0(g), L1 = mex_group_l1(g);
        if (L0 > l_max) break;
        const int c0 = L0 * L0;
        const int nc = mex_ncomp(L1 < l_max ? L1 : l_max) - c0;
        // this component's carry, in flight during the moments
        const bool scanner = tid < 2 * nc, inner = tid < nc;
        const int cc = c0 + (inner ? tid : tid - nc);
        double cv = 0.0;
        if (scanner) cv = carry[(size_t)((inner ? 0 : ncomp) + cc) * stride + blockIdx.x];
        if (g > 0) __syncthreads();   // the previous group's rows have been read
        opaque_pair(p);
        if (NG == 1 || g == 0) mex_group_moments<R, 0>(p, l_max, rows + tid, nc);
        else if (g == 1) mex_group_moments<R, 1>(p, l_max, rows + tid, nc);
        else mex_group_moments<R, 2>(p, l_max, rows + tid, nc);
        __syncthreads();
        {
            const int left = (2 * nc) & 31, whole = left <= kMexLeftover ? 2 * nc - left : 2 * nc;
            R q0 = R(0), w = R(0);
            if (scanner) {
                const int l = comp_level(cc), am = (cc - l * l + 1) / 2;
                q0 = (R)scale_pow2(cv, inner ? -l * e : (l + 1) * e);
                w = mex_w<R>(l * (l + 1) / 2 + am);
            }
            if (tid < whole) {
                mex_scan_row<R>(reinterpret_cast<Vec4<R>*>(rows + tid * kMexRow), inner, q0, w);
            } else if ((tid & ~31) == whole) {   // whole is a multiple of 32 here
                for (int j = 0; j < 2 * nc - whole; ++j)
                    mex_scan_row_warp<R>(reinterpret_cast<Vec4<R>*>(rows + (whole + j) * kMexRow),
                                         whole + j < nc, __shfl_sync(0xffffffffu, q0, j),
                                         __shfl_sync(0xffffffffu, w, j), tid & 31);
            }
        }
        __syncthreads();
        opaque_pair(p);
        if (NG == 1 || g == 0) mex_group_eval<R, 0, ACC>(p, l_max, rows + tid, nc, f);
        else if (g == 1) mex_group_eval<R, 1, ACC>(p, l_max, rows + tid, nc, f);
        else mex_group_eval<R, 2, ACC>(p, l_max, rows + tid, nc, f);
    }
    const R s1 = scale, s2 = scale * scale;
    const R two = R(2), kap = R(kKappa), ikap = R(1) / R(kKappa);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        auto at = [&](const Pair<R>& q) { return j == 0 ? q.x : q.y; };
        const int i = 2 * tid + j;
        if (i >= nt) continue;
        const R sum = fma(two, at(f.s1), at(f.s0));
        const R pot = ACC ? fma(at(p.rho), sum, at(f.pot0)) : sum + at(f.pot0);
        const R potv = (out_mask & ETICS_OUT_POT) ? -pot * s1 : R(0);
        R fx = R(0), fy = R(0), fz = R(0);
        if (ACC) {
            const R k = at(f.rad) * ikap;
            fx = s2 * fma(-k, at(p.x), kap * at(f.vx));
            fy = s2 * fma(-k, at(p.y), kap * at(f.vy));
            fz = s2 * fma(-k, at(p.z), kap * fma(two, at(f.vz1), at(f.vz0)));
        }
        if (!finite4(fx, fy, fz, potv)) report(err, ETICS_ERR_NONFINITE);
        // an entry >= N only after a timed-out sort (reported): no store
        if ((int64_t)dst[j] < N) st4(out + dst[j], mk4<R>(fx, fy, fz, potv));
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <typename R>
struct MexBuffers {
    SortBuffers sort;
    Vec4<R>* sorted;
    double* tile_agg;    // [2 * ncomp][tile]: inner then outer sums (ncomp: mex_ncomp)
    double* carry;       // [2 * ncomp][tile]
};

// ncomp = mex_layout_ncomp(l_max) components per side
template <typename R>
inline MexBuffers<R> mex_buffers(void* ws, int64_t N, int l_max, size_t* total) {
    MexBuffers<R> b{};
    size_t off = 0;
    b.sort = sort_buffers(ws, N, &off);
    uint8_t* p = reinterpret_cast<uint8_t*>(ws);
    auto take = [&](size_t bytes) {
        uint8_t* q = p ? p + off : nullptr;
        off += (bytes + 255) / 256 * 256;
        return q;
    };
    const size_t n = (size_t)(N > 0 ? N : 1);
    const size_t nt = (size_t)(mex_tiles(N) > 0 ? mex_tiles(N) : 1);
    const size_t nc = (size_t)mex_layout_ncomp(l_max > 0 ? l_max : 0);
    b.sorted = reinterpret_cast<Vec4<R>*>(take(n * sizeof(Vec4<R>)));
    b.tile_agg = reinterpret_cast<double*>(take(nt * 2 * nc * sizeof(double)));
    b.carry = reinterpret_cast<double*>(take(nt * 2 * nc * sizeof(double)));
    if (total) *total = off;
    return b;
}

template <typename R>
inline size_t mex_workspace_impl(int64_t N, int l_max) {
    size_t total = 0;
    mex_buffers<R>(nullptr, N, l_max, &total);
    return total;
}

// the passes' shared memory: rows of one level group (above 48 KB the kernel
// has to be told once per device)
template <typename R, typename K>
inline cudaError_t mex_allow_smem(K kernel, std::atomic<uint64_t>& done, size_t bytes) {
    int dev = 0;
    const cudaError_t ge = cudaGetDevice(&dev);
    if (ge != cudaSuccess) return ge;
    const uint64_t bit = uint64_t(1) << (dev & 63);
    if (done.load() & bit) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.fetch_or(bit);
    return e;
}

template <typename R, int NG>
inline int mex_passes(const MexBuffers<R>& b, int64_t N, int l_max, void* out, int out_mask,
                      const LaunchCtx& ctx) {
    const int nt = mex_tiles(N);
    const int ncomp = mex_ncomp(l_max);
    constexpr size_t smem_max = (size_t)2 * kMexNC * kMexRow * sizeof(R);
    const size_t smem = (size_t)2 * mex_row_comps(l_max) * kMexRow * sizeof(R);
    static std::atomic<uint64_t> done1{0}, done2{0}, done3{0};
    auto k1 = mex_pass1_kernel<R, NG>;
    if (mex_allow_smem<R>(k1, done1, smem_max)) return ETICS_ERR_CUDA;
    if (launch_pdl(k1, dim3(nt), dim3(kMexThreads), smem, ctx.stream, (const Vec4<R>*)b.sorted, N,
                   l_max, b.tile_agg, nt, ctx.err))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    stage_event(ctx, 3);
    if (launch_pdl(mex_carry_kernel, dim3(2 * ncomp), dim3(kCarryThreads), 0, ctx.stream,
                   (const double*)b.tile_agg, nt, nt, ncomp, b.carry))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    stage_event(ctx, 4);
    Vec4<R>* op = reinterpret_cast<Vec4<R>*>(out);
    const bool acc = out_mask & ETICS_OUT_ACC;
    auto k2 = acc ? mex_pass2_kernel<R, NG, true> : mex_pass2_kernel<R, NG, false>;
    if (mex_allow_smem<R>(k2, acc ? done2 : done3, smem_max)) return ETICS_ERR_CUDA;
    if (launch_pdl(k2, dim3(nt), dim3(kMexThreads), smem, ctx.stream, (const Vec4<R>*)b.sorted,
                   (const uint32_t*)b.sort.vals_a, N, l_max, (const double*)b.carry, nt, op, out_mask,
                   ctx.err))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    stage_event(ctx, 5);
    return ETICS_OK;
}

template <typename R>
inline int mex_field_impl(const void* posm, int64_t N, int l_max, void* out, int out_mask,
                          void* ws, const LaunchCtx& ctx) {
    if (N == 0) return ETICS_OK;
    MexBuffers<R> b = mex_buffers<R>(ws, N, l_max, nullptr);
    stage_event(ctx, 0);
    int rc = radial_sort_impl<R>(posm, N, b.sort, b.sorted, ctx);
    if (rc) return rc;
    stage_event(ctx, 2);
    // l_max <= 6: one level group (the kernels specialised for it)
    if (mex_ngroups(l_max) == 1) return mex_passes<R, 1>(b, N, l_max, out, out_mask, ctx);
    return mex_passes<R, kMexGroups>(b, N, l_max, out, out_mask, ctx);
}

template <typename R>
inline int radial_order_impl(const void* posm, int64_t N, uint32_t* order, void* ws,
                             const LaunchCtx& ctx) {
    if (N == 0) return ETICS_OK;
    MexBuffers<R> b = mex_buffers<R>(ws, N, 0, nullptr);
    int rc = radial_sort_impl<R>(posm, N, b.sort, nullptr, ctx);
    if (rc) return rc;
    if (cudaMemcpyAsync(order, b.sort.vals_a, (size_t)N * 4, cudaMemcpyDeviceToDevice, ctx.stream))
        return ETICS_ERR_CUDA;
    return ETICS_OK;
}

}  // namespace etics
