// etics_scf_field.cuh -- the SCF field pass (paper Sec. 3.3, second part):
// Phi = sum c_nlm phi_nl(r) Y_lm and a = -grad Phi at every particle.
//
// GB300 design: one thread evaluates two particles as the halves of paired
// FP32 instructions (one particle in FP64), walking the levels one after the
// other.  Per level l it keeps the 2l+1 column sums A_c = sum_n c_nc Ct_n(xi);
// the radial derivative needs Q = sum_n Dt_n sum_c c_nc R_c, so the inner sum
// over the columns is formed per row n and no second set of column sums is
// held.  The coefficients (with every normalisation folded in) are broadcast
// from shared memory, one 16-byte load for four columns of both particles.
// The gradient comes from the ladder relations of the scaled solid harmonics
// (etics_pair.cuh), whose constants are all one: regular on the z axis and at
// the origin.
//
// Bound: the FMA pipe.  Per particle (10, 6): 2 x 539 column updates, 308
// recursion steps and about 500 for harmonics, gradient and sums; pairing
// halves the issue slots and the shared loads of these, which limited the
// one-particle form before the pipe did.  Measured, one particle per thread
// and separate column and radial sums before: (10, 6) at 2^20 particles 84 us,
// now 69; (14, 8) at 2^24 2610 us, now 2130; FP64 (10, 6) at 16384 138 us,
// now 66 (there one block per SM instead of 512-thread blocks on a fifth of
// the SMs).
#pragma once

#include <algorithm>

#include "etics_internal.h"
#include "etics_pair.cuh"

namespace etics {

__host__ __device__ constexpr int ncol_pad_c(int l) { return ((2 * l + 1 + 3) / 4) * 4; }
__host__ __device__ constexpr int col_offset_c(int l) {
    int o = 0;
    for (int k = 0; k < l; ++k) o += ncol_pad_c(k);
    return o;
}

// what a coefficient c_nlm is multiplied by in the field's table: the
// normalisation of the harmonic in the scaling of harm_scaled,
// knorm_lm (l+m)! kappa^-l, and the scale gam_n of the rescaled radial
// polynomial.  [basis][n][l(l+1)/2 + m]
struct FieldTable {
    double v[2][kNmaxLimit + 1][(kLmaxLimit + 1) * (kLmaxLimit + 2) / 2];
};
constexpr FieldTable make_field_table() {
    FieldTable t{};
    constexpr BasisTables b = make_tables();
    for (int l = 0; l <= kLmaxLimit; ++l)
        for (int m = 0; m <= l; ++m) {
            double k = b.knorm[l * (l + 1) / 2 + m];
            for (int j = 2; j <= l + m; ++j) k *= (double)j;
            for (int j = 0; j < l; ++j) k /= (double)kKappa;
            for (int s = 0; s < 2; ++s)
                for (int n = 0; n <= kNmaxLimit; ++n)
                    t.v[s][n][l * (l + 1) / 2 + m] = k * b.ggam[s][l][n];
        }
    return t;
}
static __device__ const FieldTable g_field_tab = make_field_table();

// The table: row n holds the levels' 2l+1 columns, each level followed by at
// least one place of padding, the last of which holds -bs_n, so that the
// recursion constant arrives with the columns.  `stride` entries per row (a
// constant of the kernel, so that a round's rows are at immediate offsets), at
// least two rows.
// Warps take rows, lanes columns: one look for a column's level for all rows.
__host__ __device__ constexpr int field_rows(int n_max) { return n_max < 1 ? 2 : n_max + 1; }
template <typename R>
__device__ __forceinline__ void field_table(R* cs, int stride, const double* coeffs, int basis,
                                            int n_max, int l_max) {
    const int nj = (l_max + 1) * (l_max + 1), ncols = col_total(l_max);
    for (int c = threadIdx.x & 31; c < ncols; c += 32) {
        int l = 0, k = c;
        while (k >= ncol_pad(l)) { k -= ncol_pad(l); ++l; }
        const int am = (k + 1) / 2, m = (k & 1) ? am : -am;   // k = 0: m = 0
        for (int n = threadIdx.x >> 5; n < field_rows(n_max); n += blockDim.x >> 5)
            cs[n * stride + c] =
                n > n_max ? R(0)   // at least two rows
                : k < 2 * l + 1 ? (R)(ld_cg(coeffs + (size_t)n * nj + l * l + l + m) *
                                    g_field_tab.v[basis][n][l * (l + 1) / 2 + am])
                : k == ncol_pad(l) - 1 ? -geg_bs_of<R>(basis, l, n) : R(0);
    }
}

// NM1 > 0: specialised for n_max + 1 == NM1 and l_max == LM (n loop unrolled,
// row stride and recursion constants known at compile time); NM1 == 0:
// generic, n_max and l_max <= LM at run time.
template <typename P> struct FieldLane;
template <> struct FieldLane<float2> { using R = float; static constexpr int kParticles = 2; };
template <> struct FieldLane<double> { using R = double; static constexpr int kParticles = 1; };

template <typename P, int LM, bool ACC, int NM1, int BASIS>
struct FieldEval {
    using R = typename FieldLane<P>::R;
    using V4 = Vec4<R>;
    P C[3][LM + 1], S[3][LM + 1];
    // v = kappa u; RadialSeed's factors; pre = pre0 st^l, preR its gradient
    // counterpart (times kappa / 2, the ladder's half)
    P vx, vy, vz, tau, xi, dxdr, st, pre, preR;
    P pot, gr, gx, gy, gz;   // gz at half its value
    const R* cs;
    int n_max, l_max;
    unsigned levels;   // bit l: this thread adds level l

    // one row, v its table entries: acc[c] += v_c t, and (ACC) the sum of v_c Y_c
    template <int L>
    __device__ __forceinline__ void load_row(const R* r, V4 (&v)[ncol_pad_c(L) / 4]) {
#pragma unroll
        for (int q = 0; q < ncol_pad_c(L) / 4; ++q) v[q] = ld4(reinterpret_cast<const V4*>(r) + q);
    }
    template <int L>
    __device__ __forceinline__ void add_row(const V4 (&v)[ncol_pad_c(L) / 4], P t, P (&A)[2 * L + 1],
                                            const P* c, const P* s, P& sum) {
        constexpr int NC = 2 * L + 1;
#pragma unroll
        for (int q = 0; q < ncol_pad_c(L) / 4; ++q) {
            const R e[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = 4 * q + j;
                if (k >= NC) continue;
                A[k] = fma2(splat<P>(e[j]), t, A[k]);
                if constexpr (ACC) {
                    const P y = k == 0 ? c[0] : ((k & 1) ? c[(k + 1) / 2] : s[k / 2]);
                    sum = k == 0 ? mul2(splat<P>(e[j]), y) : fma2(splat<P>(e[j]), y, sum);
                }
            }
        }
    }
    // row n of the level: Ct_n and Dt_n in place of Ct_{n-2} (c0) and Dt_{n-2}
    // (d0), then the row's sums
    template <int L>
    __device__ __forceinline__ void step(const R* r, R nbs_ct, P& c0, const P& c1, P& d0, const P& d1,
                                         P (&A)[2 * L + 1], const P* c, const P* s, P& Q) {
        V4 v[ncol_pad_c(L) / 4];
        load_row<L>(r, v);
        const P nbs = splat<P>(NM1 > 0 ? nbs_ct : v[ncol_pad_c(L) / 4 - 1].w);
        c0 = fma2(xi, c1, mul2(nbs, c0));
        if (ACC) d0 = fma2(nbs, d0, fma2(xi, d1, c1));
        P sum;
        add_row<L>(v, c0, A, c, s, sum);
        if (ACC) Q = fma2(d0, sum, Q);
    }

    template <int L>
    __device__ __forceinline__ void level() {
        if constexpr (L <= LM) {
            if (NM1 == 0 && L > l_max) return;
            constexpr int s0 = L % 3, s1 = (L + 2) % 3, s2 = (L + 1) % 3;
            harm_scaled<R, L, P>(C[s1], S[s1], C[s2], S[s2], vx, vy, vz, C[s0], S[s0]);
            if (levels >> L & 1u) {
            constexpr int NC = 2 * L + 1;
            constexpr int stride = col_offset_c(LM + 1);
            const int nlim = NM1 > 0 ? NM1 - 1 : n_max;
            const R* r = cs + col_offset_c(L);
            P A[NC], Q;
            {
                // rows 0 and 1 (always there): Ct_0 = 1, Dt_0 = 0, Ct_1 = xi,
                // Dt_1 = 1; row 0 is the addend of the first FMAs, not a copy
                V4 v[ncol_pad_c(L) / 4];
                load_row<L>(r, v);
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    const V4 q = v[k / 4];
                    A[k] = splat<P>(k % 4 == 0 ? q.x : k % 4 == 1 ? q.y : k % 4 == 2 ? q.z : q.w);
                }
                r += stride;
                load_row<L>(r, v);
                P sum;
                add_row<L>(v, xi, A, C[s0], S[s0], sum);
                if (ACC) Q = sum;
                // rescaled polynomials (the table holds gam_n c_nlm), two rows
                // per round so that none of them has to be moved
                P ca = splat<P>(R(1)), cb = xi, da = splat<P>(R(0)), db = splat<P>(R(1));
                int n = 2;
#pragma unroll (NM1 > 0 ? NM1 : 1)
                for (; n + 1 <= nlim; n += 2) {
                    step<L>(r + stride, NM1 > 0 ? -geg_bs_of<R>(BASIS, L, n) : R(0), ca, cb, da, db, A,
                            C[s0], S[s0], Q);
                    step<L>(r + 2 * stride, NM1 > 0 ? -geg_bs_of<R>(BASIS, L, n + 1) : R(0), cb, ca, db, da,
                            A, C[s0], S[s0], Q);
                    r += 2 * stride;
                }
                if (n <= nlim)
                    step<L>(r + stride, NM1 > 0 ? -geg_bs_of<R>(BASIS, L, n) : R(0), ca, cb, da, db, A,
                            C[s0], S[s0], Q);
            }
            // angular sum with the level's harmonics
            P sum = mul2(A[0], C[s0][0]);
#pragma unroll
            for (int m = 1; m <= L; ++m) {
                sum = fma2(A[2 * m - 1], C[s0][m], sum);
                sum = fma2(A[2 * m], S[s0][m], sum);
            }
            pot = fma2(pre, sum, pot);
            if (ACC) {
                // d/dr: pre (-(2l+1) tau P + dxi/dr Q)
                const P k = mul2(mul2(tau, splat<P>(R(-(2 * L + 1)))), sum);
                gr = fma2(pre, fma2(dxdr, Q, k), gr);
                if constexpr (L >= 1) {
                    // 2 grad sum_m A R regrouped by the harmonic of the level
                    // below that each term multiplies (A_{-1} terms are zero,
                    // m = 0 counts twice against the halves of m > 0)
                    const P* C1 = C[s1];
                    const P* S1 = S[s1];
                    auto ac = [&](int m) -> P { return A[m == 0 ? 0 : 2 * m - 1]; };
                    auto as = [&](int m) -> P { return A[2 * m]; };
                    P x = mul2(ac(1), C1[0]), y = mul2(as(1), C1[0]), z = mul2(ac(0), C1[0]);
#pragma unroll
                    for (int j = 1; j <= L - 1; ++j) {
                        const P xc = j == 1 ? fma2(splat<P>(R(-2)), ac(0), ac(2)) : sub2(ac(j + 1), ac(j - 1));
                        const P yc = j == 1 ? as(2) : add2(as(j + 1), as(j - 1));
                        const P xs = j == 1 ? as(2) : sub2(as(j + 1), as(j - 1));
                        const P ys = j == 1 ? fma2(splat<P>(R(2)), ac(0), ac(2)) : add2(ac(j + 1), ac(j - 1));
                        x = fma2(xc, C1[j], x);
                        y = fma2(yc, C1[j], y);
                        z = fma2(ac(j), C1[j], z);
                        x = fma2(xs, S1[j], x);
                        y = fma2(neg2(ys), S1[j], y);
                        z = fma2(as(j), S1[j], z);
                    }
                    gx = fma2(preR, x, gx);
                    gy = fma2(preR, y, gy);
                    gz = fma2(preR, z, gz);
                }
            }
            }
            if constexpr (ACC && L >= 1) preR = mul2(preR, st);
            pre = mul2(pre, st);
            level<L + 1>();
        }
    }
};

// one particle's seeds written into half J of the evaluator's values
__device__ __forceinline__ void set_half(float2& p, int j, float v) { if (j == 0) p.x = v; else p.y = v; }
__device__ __forceinline__ void set_half(double& p, int, double v) { p = v; }
__device__ __forceinline__ float half_of(const float2& p, int j) { return j == 0 ? p.x : p.y; }
__device__ __forceinline__ double half_of(const double& p, int) { return p; }

// potential and acceleration of particles pv[0 .. kParticles) from the table;
// the levels not in `levels` are left out (a partial sum)
template <typename P, int LM, bool ACC, int NM1, int BASIS>
__device__ __forceinline__ void field_eval(const Vec4<typename FieldLane<P>::R> (&pv)[FieldLane<P>::kParticles],
                                           const typename FieldLane<P>::R* cs, int n_max, int l_max,
                                           unsigned levels,
                                           Vec4<typename FieldLane<P>::R> (&res)[FieldLane<P>::kParticles]) {
    using R = typename FieldLane<P>::R;
    constexpr int NP = FieldLane<P>::kParticles;
    FieldEval<P, LM, ACC, NM1, BASIS> f;
    P ux, uy, uz;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        const R x = pv[j].x, y = pv[j].y, z = pv[j].z;
        const R r = sqrt(x * x + y * y + z * z);
        const R inv = r > R(0) ? R(1) / r : R(0);
        const RadialSeed<R, BASIS> rs(r);
        set_half(ux, j, x * inv);
        set_half(uy, j, y * inv);
        set_half(uz, j, z * inv);
        set_half(f.tau, j, rs.tau);
        set_half(f.st, j, rs.st);
        set_half(f.xi, j, rs.xi);
        set_half(f.dxdr, j, rs.dxdr);
        set_half(f.pre, j, rs.pre0);
        set_half(f.preR, j, rs.pre0 * rs.q);
    }
    const P kap = splat<P>(R(kKappa));
    f.vx = mul2(kap, ux);
    f.vy = mul2(kap, uy);
    f.vz = mul2(kap, uz);
    f.preR = mul2(f.preR, splat<P>(R(0.5 * kKappa)));
    f.pot = f.gr = f.gx = f.gy = f.gz = splat<P>(R(0));
    f.cs = cs;
    f.n_max = n_max;
    f.l_max = l_max;
    f.levels = levels;
    f.template level<0>();
    P ax, ay, az;
    ax = ay = az = splat<P>(R(0));
    if (ACC) {
        ax = neg2(fma2(f.gr, ux, f.gx));
        ay = neg2(fma2(f.gr, uy, f.gy));
        az = neg2(fma2(f.gr, uz, add2(f.gz, f.gz)));
    }
#pragma unroll
    for (int j = 0; j < NP; ++j)
        res[j] = mk4<R>(half_of(ax, j), half_of(ay, j), half_of(az, j), half_of(f.pot, j));
}

// Few particles leave the SMs with a warp or two each, waiting on their own
// results: then two or kFieldParts warps share the levels of the same particles
// and their partial sums are added through shared memory.  level[w]: warp w's.
constexpr int kFieldParts = 4;
struct FieldSplit { int parts; unsigned level[kFieldParts]; };
inline FieldSplit field_split(int l_max, int parts) {
    FieldSplit s{parts, {~0u, ~0u, ~0u, ~0u}};
    if (parts == 1) return s;
    int load[kFieldParts] = {};
    for (int w = 0; w < parts; ++w) s.level[w] = 0u;
    for (int l = l_max; l >= 0; --l) {   // largest level first, to the least loaded
        int best = 0;
        for (int w = 1; w < parts; ++w)
            if (load[w] < load[best]) best = w;
        s.level[best] |= 1u << l;
        load[best] += 2 * (2 * l + 1) + 6;
    }
    return s;
}

// threads per block the registers are sized for, and blocks per SM: two where the
// potential alone of the smallest expansions leaves nothing but memory to wait for
// (2^21 particles: (0, 0) 13.8 us, (2, 2) 17.3; 19.6 and 24.2 with one)
template <int LM> constexpr int field_threads() { return LM <= 6 ? 512 : LM <= 8 ? 384 : 256; }
template <typename P, int LM, bool ACC> constexpr int field_blocks() {
    return FieldLane<P>::kParticles > 1 && LM <= 2 && !ACC ? 2 : 1;
}

// vel (nullable): the second kick of a leapfrog step, v += kick a, with the
// acceleration still in registers
template <typename P, int LM, bool ACC, int NM1, int B>
__global__ void __launch_bounds__(field_threads<LM>(), (field_blocks<P, LM, ACC>()))
scf_field_kernel(const Vec4<typename FieldLane<P>::R>* posm, int64_t N, int n_max,
                 int l_max, const double* coeffs, Vec4<typename FieldLane<P>::R>* out,
                 int out_mask, Vec4<typename FieldLane<P>::R>* vel,
                 typename FieldLane<P>::R kick, FieldSplit split, unsigned* err) {
    using R = typename FieldLane<P>::R;
    constexpr int NP = FieldLane<P>::kParticles;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R* cs = reinterpret_cast<R*>(smem_raw);
    constexpr int stride = col_offset_c(LM + 1);
    pdl_wait();   // the coefficients come from the previous kernel
    field_table(cs, stride, coeffs, B, n_max, l_max);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int part = warp % split.parts;
    const int per = blockDim.x / split.parts;   // lanes of particles per block
    const int slot = (warp / split.parts) * 32 + lane;
    for (int64_t first = (int64_t)blockIdx.x * per * NP; first < N;
         first += (int64_t)gridDim.x * per * NP) {
        // particle j of the thread: a neighbour, or (kApart) as far on as the
        // block has lanes, so that neighbouring lanes take neighbouring particles
        constexpr bool kApart = field_blocks<P, LM, ACC>() > 1;
        auto at = [&](int j) -> int64_t {
            return kApart ? first + (int64_t)j * per + slot : first + (int64_t)slot * NP + j;
        };
        Vec4<R> pv[NP], res[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            pv[j] = at(j) < N ? ld4(posm + at(j)) : mk4<R>(R(0), R(0), R(0), R(0));
            if (!finite4(pv[j].x, pv[j].y, pv[j].z, pv[j].w)) report(err, ETICS_ERR_NONFINITE);
        }
        field_eval<P, LM, ACC, NM1, B>(pv, cs, n_max, l_max, split.level[part], res);
        if (split.parts > 1) {
            // parts 1.. leave their sums behind the table, part 0 adds them
            Vec4<R>* sums = reinterpret_cast<Vec4<R>*>(cs + field_rows(n_max) * stride);
            if (part > 0) {
#pragma unroll
                for (int j = 0; j < NP; ++j) st4(sums + ((part - 1) * NP + j) * per + slot, res[j]);
            }
            __syncthreads();
            if (part == 0) {
                for (int w = 0; w < split.parts - 1; ++w)
#pragma unroll
                    for (int j = 0; j < NP; ++j) {
                        const Vec4<R> t = ld4(sums + (w * NP + j) * per + slot);
                        res[j].x += t.x; res[j].y += t.y; res[j].z += t.z; res[j].w += t.w;
                    }
            }
            __syncthreads();
            if (part > 0) continue;
        }
        Vec4<R> v[NP];
        if (vel) {
#pragma unroll
            for (int j = 0; j < NP; ++j)
                if (at(j) < N) v[j] = ld4(vel + at(j));
        }
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            if (at(j) >= N) continue;
            if (!(out_mask & ETICS_OUT_POT)) res[j].w = R(0);
            if (!finite4(res[j].x, res[j].y, res[j].z, res[j].w)) report(err, ETICS_ERR_NONFINITE);
            st4(out + at(j), res[j]);
            if (vel) {
                v[j].x = fma(kick, res[j].x, v[j].x);
                v[j].y = fma(kick, res[j].y, v[j].y);
                v[j].z = fma(kick, res[j].z, v[j].z);
                st4(vel + at(j), v[j]);
            }
        }
    }
}

template <typename P, int LM, int NM1, int B>
inline int launch_field_lm(const void* posm, int64_t N, int n_max, int l_max,
                           const double* coeffs, void* out, int out_mask, FieldKick kick,
                           const LaunchCtx& ctx) {
    using R = typename FieldLane<P>::R;
    // One block per SM, so that the coefficient table (FP64 multiplies, slow on
    // this GPU) is built once per SM; as many threads as give every block the
    // same number of rounds over the particles, so that neither a few large
    // blocks on part of the SMs (small N) nor a last round that is nearly
    // empty leaves the GPU idle.  Where a quarter or half of the threads would
    // do, the levels are split over four or two warps (mixed precision: the FP64
    // kernel is bound by the FP64 pipe at any size, and repeats the harmonics).
    // 19456 | 19500 | 38912 particles at (16, 12), four | two | two warps: 20.3 |
    // 23.5 | 23.9 us, with one warp 31.9 and 29.7 for the latter two; (14, 8) at
    // 29200 12.8 us with two, 15.6 with one; (10, 6) at 38912 8 us with four.
    constexpr int kMost = field_threads<LM>();
    const int64_t lanes = (N + FieldLane<P>::kParticles - 1) / FieldLane<P>::kParticles;
    const bool acc = out_mask & ETICS_OUT_ACC;
    const int64_t sms = (int64_t)ctx.num_sms *
                        (acc ? field_blocks<P, LM, true>() : field_blocks<P, LM, false>());
    int parts = sizeof(R) == 4 && l_max >= 2 ? kFieldParts : 1;
    while (parts > 1 && lanes * parts > (int64_t)ctx.num_sms * kMost) parts /= 2;
    const int64_t most = kMost / parts;
    const int64_t rounds = (lanes + sms * most - 1) / (sms * most);
    const int64_t per = (lanes + sms * rounds - 1) / (sms * rounds);
    // (the one warp of a small call's block would load the table's rows one after
    // the other: l_max = 0, n_max = 16, 4219 particles 9.3 us, 6.0 with four)
    const int least = sizeof(R) == 4 ? 4 / parts : 1;
    const int warps = std::max((int)((per + 31) / 32), least);
    const int threads = warps * 32 * parts;
    const int64_t want = (lanes + warps * 32 - 1) / (warps * 32);
    const int grid = (int)(want < sms ? want : sms);
    const size_t smem = (size_t)field_rows(n_max) * col_offset_c(LM + 1) * sizeof(R) +
                        (size_t)(parts - 1) * FieldLane<P>::kParticles * warps * 32 * sizeof(Vec4<R>);
    auto k = acc ? scf_field_kernel<P, LM, true, NM1, B> : scf_field_kernel<P, LM, false, NM1, B>;
    if (smem > 48 * 1024 && allow_dynamic_smem(k)) return ETICS_ERR_CUDA;
    // launched as a programmatic dependent of the coefficient finalize (or
    // whatever precedes it): its launch overlaps the predecessor's tail
    if (launch_pdl(k, dim3(grid), dim3(threads), smem, ctx.stream,
                   reinterpret_cast<const Vec4<R>*>(posm), N, n_max, l_max, coeffs,
                   reinterpret_cast<Vec4<R>*>(out), out_mask, reinterpret_cast<Vec4<R>*>(kick.vel),
                   (R)kick.factor, field_split(l_max, parts), ctx.err) != cudaSuccess)
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}

// dispatch by l_max, the low (l_max <= 6) and the high instantiations in
// translation units of their own; the paper's (10, 6) and the (14, 8)
// expansion of the forecast experiment have n unrolled (basis 0 only)
template <typename P, int B>
inline int scf_field_low(const void* posm, int64_t N, int n_max, int l_max, const double* coeffs,
                         void* out, int out_mask, FieldKick kick, const LaunchCtx& ctx) {
    if (l_max <= 2)
        return launch_field_lm<P, 2, 0, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
    if (l_max <= 4)
        return launch_field_lm<P, 4, 0, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
    if constexpr (B == 0)
        if (n_max == 10 && l_max == 6)
            return launch_field_lm<P, 6, 11, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
    return launch_field_lm<P, 6, 0, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
}
template <typename P, int B>
inline int scf_field_high(const void* posm, int64_t N, int n_max, int l_max, const double* coeffs,
                          void* out, int out_mask, FieldKick kick, const LaunchCtx& ctx) {
    if constexpr (B == 0)
        if (n_max == 14 && l_max == 8)
            return launch_field_lm<P, 8, 15, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
    if (l_max <= 8)
        return launch_field_lm<P, 8, 0, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
    if (l_max <= 10)
        return launch_field_lm<P, 10, 0, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
    return launch_field_lm<P, 14, 0, B>(posm, N, n_max, l_max, coeffs, out, out_mask, kick, ctx);
}

}  // namespace etics
