// etics_scf_coeffs.cuh -- the mixed-precision SCF coefficient pass (paper Sec.
// 2.4 eq. 18, bases of Sec. 2.5, first pass of Sec. 3.3) for any (n_max,
// l_max) and either radial basis, with the particle loop run two particles at
// a time on Blackwell's paired FP32 instructions.
//
//   c_nlm = (1/J_nl) sum_k m_k phi_nl(r_k) Y_lm(x_k)
//   phi_nl Y_lm = w_l(r) Ct_n(xi) H_l^m(u) * (gam_n knorm_lm / (l-m)!)
//   w_l = m pre0 st^l (RadialSeed), Ct_n the rescaled Gegenbauer polynomial,
//   H_l^m = (l-m)! Z_l^m (harm_level_exact); the bracket is applied in FP64
//   by the finalize.
//
// Work split (one block per SM, each over one contiguous range of particles,
// in tiles):
//   * phase 1: thread k of the block evaluates particle k of the next tile:
//     xi and the harmonics already scaled by w_l, into a shared-memory buffer
//     (two buffers: phase 1 of tile t+1 runs while tile t is contracted);
//   * phase 2: a warp owns one bin -- at most CAP columns of one level l, so
//     that it needs one Gegenbauer recursion -- and accumulates c[n][col] for
//     n = 0..NR-1; lane j takes the particle pairs j, j+32, ...: one paired
//     load brings both particles' values of a column, and each of the NR x ncol
//     updates is one paired FMA.  Accumulators are FP32 register pairs;
//     the recursion constants of the bin's level are scalar registers.
//   * every 2048 particles (coeff_flush_tiles) each warp adds its accumulators over its
//     lanes (a reduce-scatter: each step halves the values a lane still holds)
//     and the totals to its FP64 block sums in shared memory.  The per-block
//     sums are added in a fixed order by the finalize kernel: deterministic.
// The accumulators decide the shape: NR x CAP pairs per lane leave room for
// PairShape<NR>::kWarps warps per SM.  An expansion with more bins than warps
// is cut into groups of bins (neighbouring levels) that different blocks
// handle, each group getting a share of the SMs by its cost; one with at most
// half as many bins runs several teams of warps over the same bins, each on
// its share of the tile's pairs.
// Bound: the FMA pipe and, below about 2^18 particles, the latency of the first
// tile and of the finalize.  Clutton-Brock (10, 6), 2^18 particles, both passes:
// 63.7 us with the register-tile kernel this replaces, 46.1 now.
#pragma once

#include <atomic>

#include "etics_internal.h"
#include "etics_pair.cuh"

namespace etics {

constexpr int kCoeffMaxBins = 80;      // sum over l <= 14 of ceil((2l+1)/CAP) <= 64
constexpr int kCoeffMaxGroups = 8;

// rows n = 0..NR-1, columns per bin, and warps per SM that the registers allow
// (the register file is shared out in steps of four warps: 128, 168 or 255
// registers for 16, 12 or 8 warps)
template <int NR> struct PairShape {
    static constexpr int kCap = NR >= 17 ? 5 : 4;
    static constexpr int kWarps = NR <= 11 ? 16 : NR <= 15 ? 12 : 8;
};
// particles per tile: one per thread; fewer for l_max > 8, whose columns would
// not fit twice in shared memory.  A constant, so that the addresses of the
// columns are immediate offsets.
template <int NR, int LMU> constexpr int coeff_tile() {
    return LMU <= 8 ? PairShape<NR>::kWarps * 32 : 256;
}

// tiles between FP64 flushes: the FP32 partial sums span at most 2048 particles
template <int NR, int LMU> constexpr int coeff_flush_tiles() { return 2048 / coeff_tile<NR, LMU>(); }

struct CoeffBin { int16_t l, c0, nc, pad; };
struct CoeffGroup { int bin0, nbins, teams, l_lo, l_hi, block0, nblocks, pad; };
struct CoeffPlan {
    int ngroups, nbins, warps, l_max;
    int nblocks;                       // of all groups
    int slots;                         // bins a block has partial sums for, at most
    CoeffGroup group[kCoeffMaxGroups];
    CoeffBin bin[kCoeffMaxBins];
};

struct ScfCoeffPairParams {
    const float4* posm;
    int64_t N;
    int basis;
    double* partial;   // [block][plan.slots][NR][CAP]
    unsigned* err;
    CoeffPlan plan;
};

// Bins of levels 0..l_max of at most cap columns (each level's 2l+1 split as
// evenly as possible), in groups of at most `warps` consecutive bins; returns
// what a particle costs: per group the harmonics up to its last level on all
// warps, then the recursion and one update per column and row on the warps
// that hold a bin.
inline double coeff_bins(CoeffPlan& p, double* cost, int n_rows, int l_max, int cap, int warps) {
    p = CoeffPlan{};
    p.l_max = l_max;
    p.warps = warps;
    for (int l = 0; l <= l_max; ++l) {
        const int nc = 2 * l + 1, nb = (nc + cap - 1) / cap;
        int c = 0;
        for (int b = 0; b < nb; ++b) {
            if (p.nbins == kCoeffMaxBins) return 1e300;
            const int w = nc / nb + (b < nc % nb ? 1 : 0);
            p.bin[p.nbins++] = CoeffBin{(int16_t)l, (int16_t)c, (int16_t)w, 0};
            c += w;
        }
    }
    p.ngroups = (p.nbins + warps - 1) / warps;
    if (p.ngroups > kCoeffMaxGroups) return 1e300;
    double total = 0.0;
    int b0 = 0;
    for (int g = 0; g < p.ngroups; ++g) {
        CoeffGroup& q = p.group[g];
        q.bin0 = b0;
        q.nbins = p.nbins / p.ngroups + (g < p.nbins % p.ngroups ? 1 : 0);
        q.teams = warps / q.nbins;
        b0 += q.nbins;
        q.l_lo = p.bin[q.bin0].l;
        q.l_hi = p.bin[q.bin0 + q.nbins - 1].l;
        double bins = 0.0;
        for (int b = 0; b < q.nbins; ++b) bins += n_rows * (p.bin[q.bin0 + b].nc + 2.0) + 10.0;
        cost[g] = (4.0 * (q.l_hi + 1) * (q.l_hi + 1) + 60.0) / warps + bins / (q.nbins * q.teams);
        total += cost[g];
    }
    return total;
}

// The plan with the cheapest bins of at most `cap` columns: narrower ones repeat
// the recursion more often but can occupy warps that would idle (l_max = 4: 9
// bins of up to 4 columns or 15 of up to 2, for 16 warps).  Blocks per group in
// proportion to its cost.
// A bin has at least two columns where its level does: at most l + 1 bins of
// level l, and in a group at most one per warp.
inline int coeff_slots(int l_max, int warps) {
    const int n = (l_max + 1) * (l_max + 2) / 2;
    return n < warps ? n : warps;
}
inline CoeffPlan make_coeff_plan(int n_rows, int l_max, int cap, int warps, int64_t N, int num_sms) {
    CoeffPlan p, t;
    double cost[kCoeffMaxGroups], c[kCoeffMaxGroups], total = 1e301;
    for (int k = cap; k >= 2; --k) {
        const double v = coeff_bins(t, c, n_rows, l_max, k, warps);
        if (v < total) {
            total = v;
            p = t;
            for (int g = 0; g < p.ngroups; ++g) cost[g] = c[g];
        }
    }
    p.slots = coeff_slots(l_max, warps);
    // at least 64 particles (one pair per lane) per block
    int64_t most = (N + 63) / 64;
    int left = num_sms;
    double left_cost = total;
    for (int g = 0; g < p.ngroups; ++g) {
        CoeffGroup& q = p.group[g];
        int n = g + 1 == p.ngroups ? left : (int)(left * cost[g] / left_cost + 0.5);
        const int keep = p.ngroups - 1 - g;      // the later groups need one each
        if (n > left - keep) n = left - keep;
        if (n < 1) n = 1;
        left -= n;
        left_cost -= cost[g];
        if (n > most) n = (int)most;
        q.nblocks = n;
        q.block0 = p.nblocks;
        p.nblocks += n;
    }
    return p;
}
inline int coeff_cols(const CoeffPlan& p) {
    int cols = 0;
    for (int g = 0; g < p.ngroups; ++g) {
        const CoeffGroup& q = p.group[g];
        const int n = (q.l_hi + 1) * (q.l_hi + 1) - q.l_lo * q.l_lo;
        if (n > cols) cols = n;
    }
    return cols;
}

// phase 1 for one particle: w_l H_l^m of the columns of levels l_lo..l_hi
// (dense layout l*l + c - l_lo^2: c = 0 -> m = 0, 2m-1 -> cos, 2m -> sin)
template <int L, int LMU, int T>
__device__ __forceinline__ void pair_angular(float (&C)[3][LMU + 1], float (&S)[3][LMU + 1],
                                             float ux, float uy, float uz, float w, float st,
                                             float* H, int l_lo, int l_hi) {
    if constexpr (L <= LMU) {
        if (L > l_hi) return;
        constexpr int s0 = L % 3, s1 = (L + 2) % 3, s2 = (L + 1) % 3;
        harm_level_exact<float, L>(C[s1], S[s1], C[s2], S[s2], ux, uy, uz, C[s0], S[s0]);
        if (L >= l_lo) {
            // H: column 0 of the group would be at -l_lo^2 columns
            H[L * L * T] = w * C[s0][0];
#pragma unroll
            for (int m = 1; m <= L; ++m) {
                H[(L * L + 2 * m - 1) * T] = w * C[s0][m];
                H[(L * L + 2 * m) * T] = w * S[s0][m];
            }
        }
        pair_angular<L + 1, LMU, T>(C, S, ux, uy, uz, w * st, st, H, l_lo, l_hi);
    }
}

// phase 2: NC columns (H2: the first one, TP pairs per column) over the pairs
// p0, p0 + step, ... < np: Ct_n = xi Ct_{n-1} - bs_n Ct_{n-2} (Ct_0 = 1,
// Ct_1 = xi), acc[n][c] += Ct_n y_c; nb[n] = -bs_n
template <int NR, int CAP, int TP, int NC>
__device__ __forceinline__ void pair_rows(float2 (&acc)[NR][CAP], const float (&nb)[NR],
                                          const float2* H2, const float2* X2, int p0, int np,
                                          int step) {
#pragma unroll 1
    for (int p = p0; p < np; p += step) {
        const float2 xi = X2[p];
        float2 y[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) y[c] = H2[c * TP + p];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[0][c] = add2(acc[0][c], y[c]);
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[1][c] = fma2(xi, y[c], acc[1][c]);
        float2 cm1 = mk2(1.0f, 1.0f), cn = xi;
#pragma unroll
        for (int n = 2; n < NR; ++n) {
            const float2 cnew = fma2(splat<float2>(nb[n]), cm1, mul2(xi, cn));
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[n][c] = fma2(cnew, y[c], acc[n][c]);
            cm1 = cn;
            cn = cnew;
        }
    }
}
template <int NR, int CAP, int TP, int NC>
__device__ __forceinline__ void pair_rows_nc(int nc, float2 (&acc)[NR][CAP], const float (&nb)[NR],
                                             const float2* H2, const float2* X2, int p0, int np,
                                             int step) {
    if constexpr (NC >= 1) {
        if (nc == NC) pair_rows<NR, CAP, TP, NC>(acc, nb, H2, X2, p0, np, step);
        else pair_rows_nc<NR, CAP, TP, NC - 1>(nc, acc, nb, H2, X2, p0, np, step);
    }
}

template <int NR, int LMU>
__global__ void __launch_bounds__(PairShape<NR>::kWarps * 32, 1)
scf_coeff_plan_kernel(const __grid_constant__ ScfCoeffPairParams p) {
    constexpr int CAP = PairShape<NR>::kCap;
    constexpr int kPerWarp = NR * CAP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int g = 0;
    while (g + 1 < p.plan.ngroups && (int)blockIdx.x >= p.plan.group[g + 1].block0) ++g;
    const CoeffGroup gr = p.plan.group[g];
    constexpr int T = coeff_tile<NR, LMU>(), TP = T / 2;
    const int ncol = (gr.l_hi + 1) * (gr.l_hi + 1) - gr.l_lo * gr.l_lo;
    double* accd = reinterpret_cast<double*>(smem_raw);
    float* buf0 = reinterpret_cast<float*>(smem_raw + ((size_t)PairShape<NR>::kWarps * kPerWarp * 8 + 15) / 16 * 16);
    // buffer b: ncol x T scaled harmonics, then T values of xi
    auto Hb = [&](int b) { return buf0 + (size_t)b * (ncol + 1) * T; };
    auto Xb = [&](int b) { return buf0 + (size_t)b * (ncol + 1) * T + (size_t)ncol * T; };
    for (int e = tid; e < PairShape<NR>::kWarps * kPerWarp; e += blockDim.x) accd[e] = 0.0;
    // this warp's bin and its share of the tile's pairs
    const bool active = warp < gr.nbins * gr.teams;
    const int team = active ? warp / gr.nbins : 0;
    const CoeffBin bin = p.plan.bin[gr.bin0 + (active ? warp % gr.nbins : 0)];
    float nb[NR];
#pragma unroll
    for (int n = 2; n < NR; ++n) nb[n] = -c_tab.gbs_f[p.basis][bin.l][n];
    float2 acc[NR][CAP];
#pragma unroll
    for (int n = 0; n < NR; ++n)
#pragma unroll
        for (int c = 0; c < CAP; ++c) acc[n][c] = mk2(0.0f, 0.0f);

    // FP64 additions are slow on this GPU: spread over the lanes, each total
    // is one lane's
    auto flush = [&]() {
        constexpr int K = (kPerWarp + 31) / 32 * 32;
        float v[K];
#pragma unroll
        for (int i = 0; i < K; ++i)
            v[i] = i < kPerWarp ? acc[i / CAP][i % CAP].x + acc[i / CAP][i % CAP].y : 0.0f;
        warp_scatter<K, 16>(v, lane);
#pragma unroll
        for (int i = 0; i < K / 32; ++i) {
            const int idx = lane * (K / 32) + i;
            if (idx < kPerWarp) accd[warp * kPerWarp + idx] += (double)v[i];
        }
#pragma unroll
        for (int n = 0; n < NR; ++n)
#pragma unroll
            for (int c = 0; c < CAP; ++c) acc[n][c] = mk2(0.0f, 0.0f);
    };
    // contiguous equal ranges (an even number of particles each); the last
    // tile may be partial and its phase 2 runs over the pairs it holds
    const int64_t per = ((p.N + gr.nblocks - 1) / gr.nblocks + 1) / 2 * 2;
    const int64_t lo = (int64_t)((int)blockIdx.x - gr.block0) * per;
    const int64_t hi = lo + per < p.N ? lo + per : p.N;
    const int ntb = hi > lo ? (int)((hi - lo + T - 1) / T) : 0;
    pdl_wait();   // the particles may come from the previous kernel (a drift)
    auto load = [&](int t) -> float4 {
        const int64_t gi = lo + (int64_t)t * T + tid;
        return (tid < T && t < ntb && gi < hi) ? p.posm[gi] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto pairs_in = [&](int t) {
        const int64_t left = hi - lo - (int64_t)t * T;
        return (int)(((left < T ? left : T) + 1) / 2);
    };
    auto phase1 = [&](const float4& v, float* Hs, float* Xs) {
        if (tid >= T) return;
        float x = 0.f, y = 0.f, z = 0.f, m = 0.f;
        if (finite4(v.x, v.y, v.z, v.w)) { x = v.x; y = v.y; z = v.z; m = v.w; }
        else report(p.err, ETICS_ERR_NONFINITE);
        const float r = sqrtf(x * x + y * y + z * z);
        float w, st, xi;
        if (p.basis == ETICS_BASIS_HO) {
            const RadialSeed<float, 0> rs(r);
            w = m * rs.pre0; st = rs.st; xi = rs.xi;
        } else {
            const RadialSeed<float, 1> rs(r);
            w = m * rs.pre0; st = rs.st; xi = rs.xi;
        }
        Xs[tid] = xi;
        const float inv = r > 0.0f ? 1.0f / r : 0.0f;
        float C[3][LMU + 1], S[3][LMU + 1];
        pair_angular<0, LMU, T>(C, S, x * inv, y * inv, z * inv, w, st,
                                Hs + tid - gr.l_lo * gr.l_lo * T, gr.l_lo, gr.l_hi);
    };

    float4 cur = load(0);
    if (ntb > 0) phase1(cur, Hb(0), Xb(0));
    cur = load(1);
    __syncthreads();
    int since = 0, b = 0;
    const int col0 = bin.l * bin.l - gr.l_lo * gr.l_lo + bin.c0;
    for (int t = 0; t < ntb; ++t, b ^= 1) {
        if (t + 1 < ntb) {
            phase1(cur, Hb(b ^ 1), Xb(b ^ 1));
            cur = load(t + 2);
        }
        if (active)
            pair_rows_nc<NR, CAP, TP, CAP>(bin.nc, acc, nb,
                                           reinterpret_cast<const float2*>(Hb(b)) + (size_t)col0 * TP,
                                           reinterpret_cast<const float2*>(Xb(b)),
                                           lane + 32 * team, pairs_in(t), 32 * gr.teams);
        if (++since == coeff_flush_tiles<NR, LMU>()) {
            if (active) flush();
            since = 0;
        }
        __syncthreads();
    }
    if (since && active) flush();
    __syncthreads();
    // the teams' sums of a bin, in team order
    double* out = p.partial + (size_t)blockIdx.x * p.plan.slots * kPerWarp;
    for (int e = tid; e < gr.nbins * kPerWarp; e += blockDim.x) {
        double sum = accd[e];
        for (int k = 1; k < gr.teams; ++k) sum += accd[k * gr.nbins * kPerWarp + e];
        out[e] = sum;
    }
}

// Block sums added in block order; one warp per output c[n][l*l+l+m], four
// warps per block so that the FP64 additions (slow on this GPU) are spread
// over as many SMs as there are blocks.
constexpr int kFinThreads = 128;
template <int NR>
__global__ void __launch_bounds__(kFinThreads)
scf_finalize_plan_kernel(const __grid_constant__ ScfCoeffPairParams p, int n_max,
                          double* coeffs) {
    constexpr int CAP = PairShape<NR>::kCap;
    const int nj = (p.plan.l_max + 1) * (p.plan.l_max + 1);
    pdl_wait();   // the partials come from the coefficient kernel
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= (n_max + 1) * nj) return;
    const int n = warp / nj, jj = warp % nj;
    int l = 0;
    while ((l + 1) * (l + 1) <= jj) ++l;
    const int m = jj - l * l - l;
    const int col = (m == 0) ? 0 : (m > 0 ? 2 * m - 1 : -2 * m);
    // the bin (each level's bins are neighbours) and its group
    int b = 0;
    while (p.plan.bin[b].l != l || p.plan.bin[b].c0 + p.plan.bin[b].nc <= col) ++b;
    int g = 0;
    while (b >= p.plan.group[g].bin0 + p.plan.group[g].nbins) ++g;
    const CoeffGroup gr = p.plan.group[g];
    const int idx = ((b - gr.bin0) * NR + n) * CAP + col - p.plan.bin[b].c0;
    const size_t stride = (size_t)p.plan.slots * NR * CAP;
    const double* src = p.partial + (size_t)gr.block0 * stride + idx;
    double s = 0.0;
#pragma unroll 4
    for (int k = lane; k < gr.nblocks; k += 32) s += ld_cg(src + (size_t)k * stride);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        const int am = m < 0 ? -m : m;
        coeffs[warp] = s * c_tab.knorm_fact[l * (l + 1) / 2 + am] * inv_j_of(p.basis, n, l) *
                       geg_gamma(p.basis, l, n);
    }
}

// host side: NR is n_max + 1 rounded up to the next odd number (at least 3)
constexpr int coeff_rows(int n_max) { return n_max < 2 ? 3 : (n_max + 1) | 1; }

template <int NR, int LMU>
inline size_t coeff_smem(const CoeffPlan& p) {
    return ((size_t)PairShape<NR>::kWarps * NR * PairShape<NR>::kCap * 8 + 15) / 16 * 16 +
           2 * (size_t)(coeff_cols(p) + 1) * coeff_tile<NR, LMU>() * sizeof(float);
}

template <int NR>
inline size_t scf_coeff_plan_workspace(int l_max, int num_sms) {
    return (size_t)num_sms * coeff_slots(l_max, PairShape<NR>::kWarps) * NR * PairShape<NR>::kCap *
           sizeof(double);
}

template <int NR, int LMU>
inline int scf_coeff_plan_launch(const void* posm, int64_t N, int n_max, int l_max, int basis,
                                  double* coeffs, void* ws, const LaunchCtx& ctx) {
    constexpr int CAP = PairShape<NR>::kCap;
    ScfCoeffPairParams p;
    p.posm = reinterpret_cast<const float4*>(posm);
    p.N = N;
    p.basis = basis;
    p.partial = reinterpret_cast<double*>(ws);
    p.err = ctx.err;
    p.plan = make_coeff_plan(NR, l_max, CAP, PairShape<NR>::kWarps, N, ctx.num_sms);
    if (N > 0) {
        const size_t smem = coeff_smem<NR, LMU>(p.plan);
        auto k = scf_coeff_plan_kernel<NR, LMU>;
        // the function attributes are set once per device (a host call per
        // launch would sit between the caller's events and the kernel)
        static std::atomic<uint64_t> attr_done{0};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return ETICS_ERR_CUDA;
        const uint64_t bit = uint64_t(1) << (dev & 63);
        if (!(attr_done.load() & bit)) {
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) ||
                cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100))
                return ETICS_ERR_CUDA;
            attr_done.fetch_or(bit);
        }
        if (launch_pdl(k, dim3(p.plan.nblocks), dim3(PairShape<NR>::kWarps * 32), smem, ctx.stream, p))
            return ETICS_ERR_CUDA;
        ++*ctx.launches;
    } else {
        for (int g = 0; g < p.plan.ngroups; ++g) p.plan.group[g].nblocks = 0;
    }
    stage_event(ctx, 1);
    const int nc = (n_max + 1) * (l_max + 1) * (l_max + 1);
    if (launch_pdl(scf_finalize_plan_kernel<NR>,
                   dim3((nc * 32 + kFinThreads - 1) / kFinThreads), dim3(kFinThreads), 0,
                   ctx.stream, p, n_max, coeffs))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}

}  // namespace etics
