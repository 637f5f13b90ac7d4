// etics_scf_bins.cuh -- SCF coefficient pass specialised for a fixed
// (n_max, l_max): each warp owns a "bin" of at most kBinCap harmonic columns
// (a compile-time plan), each lane accumulates the contributions of its own
// particles to the bin's (n, column) coefficients in registers over all the
// tiles it visits, and only the angular basis of a tile goes through shared
// memory.  The radial basis of the bin's levels is evaluated by the lane
// itself (Gegenbauer recursion with immediate constants), so there is no
// per-tile cross-thread reduction and no padding work.  Method as in
// etics_scf_impl.cuh (paper Sec. 2.4 eq. 18, Sec. 2.5 basis).
#pragma once

#include "etics_internal.h"
#include "etics_pair.cuh"
#include "etics_scf_impl.cuh"

namespace etics {

constexpr int kBinCap = 7;
constexpr int kBinFlushTiles = 5;

struct BinSeg { int l, c0, n; };          // columns c0..c0+n-1 of level l
struct BinDef { int nseg; BinSeg seg[4]; int ncol; };
template <int LM>
struct BinPlan {
    static constexpr int kCols = (LM + 1) * (LM + 1);
    int nbins;
    BinDef bin[kCols];
};

// full bins of one level first (descending l), then the remainders packed
// first-fit decreasing (each remainder stays whole)
template <int LM>
constexpr BinPlan<LM> make_bin_plan() {
    BinPlan<LM> p{};
    p.nbins = 0;
    int rem_l[LM + 1] = {}, rem_c0[LM + 1] = {}, rem_n[LM + 1] = {};
    int nrem = 0;
    for (int l = LM; l >= 0; --l) {
        const int nc = 2 * l + 1;
        int c = 0;
        for (; c + kBinCap <= nc; c += kBinCap) {
            BinDef& b = p.bin[p.nbins++];
            b.nseg = 1;
            b.seg[0] = BinSeg{l, c, kBinCap};
            b.ncol = kBinCap;
        }
        if (c < nc) { rem_l[nrem] = l; rem_c0[nrem] = c; rem_n[nrem] = nc - c; ++nrem; }
    }
    // sort remainders by size (descending), stable
    for (int i = 1; i < nrem; ++i)
        for (int j = i; j > 0 && rem_n[j] > rem_n[j - 1]; --j) {
            int t = rem_n[j]; rem_n[j] = rem_n[j - 1]; rem_n[j - 1] = t;
            t = rem_l[j]; rem_l[j] = rem_l[j - 1]; rem_l[j - 1] = t;
            t = rem_c0[j]; rem_c0[j] = rem_c0[j - 1]; rem_c0[j - 1] = t;
        }
    const int first_rem_bin = p.nbins;
    for (int i = 0; i < nrem; ++i) {
        int target = -1;
        for (int b = first_rem_bin; b < p.nbins; ++b)
            if (p.bin[b].ncol + rem_n[i] <= kBinCap && p.bin[b].nseg < 4) { target = b; break; }
        if (target < 0) { target = p.nbins++; p.bin[target].nseg = 0; p.bin[target].ncol = 0; }
        BinDef& b = p.bin[target];
        b.seg[b.nseg++] = BinSeg{rem_l[i], rem_c0[i], rem_n[i]};
        b.ncol += rem_n[i];
    }
    return p;
}

// column offset of column c of level l inside its bin (for the finalize)
template <int LM>
struct BinIndex {
    int bin[(LM + 1) * (LM + 1)];
    int slot[(LM + 1) * (LM + 1)];
};
template <int LM>
constexpr BinIndex<LM> make_bin_index() {
    BinIndex<LM> ix{};
    constexpr BinPlan<LM> p = make_bin_plan<LM>();
    for (int b = 0; b < p.nbins; ++b) {
        int off = 0;
        for (int s = 0; s < p.bin[b].nseg; ++s) {
            const BinSeg g = p.bin[b].seg[s];
            for (int c = 0; c < g.n; ++c) {
                ix.bin[g.l * g.l + g.c0 + c] = b;
                ix.slot[g.l * g.l + g.c0 + c] = off + c;
            }
            off += g.n;
        }
    }
    return ix;
}

template <int LM>
struct BinConst {
    static constexpr BinPlan<LM> plan = make_bin_plan<LM>();
    static constexpr int nbins = plan.nbins;
};
// device copy of the column -> (bin, slot) map, read with run-time indices
template <int LM>
static __constant__ BinIndex<LM> c_bin_index = make_bin_index<LM>();

struct ScfBinParams {
    const void* posm;
    int64_t N;
    int64_t per;       // particles per block: block b takes [b per, (b+1) per)
    double* partial;   // [gridDim.x][nbins][NR][kBinCap]
    unsigned* err;
    // the first half of a leapfrog step, if the kernel does it
    void* drift_posm;
    void* vel;
    const void* acc;
    double dt;
};

// rows of segment S of bin B and the segments after it for one particle: the
// Gegenbauer values of the segment's level times its columns y (harmonics
// scaled by mass and radial prefactor)
template <typename R, int NR, int LM, int B, int S>
__device__ __forceinline__ void bin_segment(R (&acc)[NR][kBinCap], const R (&y)[kBinCap], R xi) {
    constexpr BinDef bd = BinConst<LM>::plan.bin[B];
    if constexpr (S < bd.nseg) {
        constexpr BinSeg g = bd.seg[S];
        constexpr int off = [] {
            int o = 0;
            for (int s = 0; s < S; ++s) o += BinConst<LM>::plan.bin[B].seg[s].n;
            return o;
        }();
        R cm1 = R(0), cn = R(1);
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            if (n == 1) {
                cm1 = cn;
                cn = xi;
            } else if (n > 1) {
                const R cnew = fma(xi, cn, -geg_bs<R>(g.l, n) * cm1);   // rescaled
                cm1 = cn;
                cn = cnew;
            }
#pragma unroll
            for (int c = 0; c < g.n; ++c)
                acc[n][off + c] = n == 0 ? acc[n][off + c] + y[off + c]
                                         : fma(cn, y[off + c], acc[n][off + c]);
        }
        bin_segment<R, NR, LM, B, S + 1>(acc, y, xi);
    }
}
template <typename R, int LM, int T, int B, int S = 0>
__device__ __forceinline__ void bin_load(R (&y)[kBinCap], const R* Ys, int k) {
    constexpr BinDef bd = BinConst<LM>::plan.bin[B];
    if constexpr (S < bd.nseg) {
        constexpr BinSeg g = bd.seg[S];
        constexpr int off = [] {
            int o = 0;
            for (int s = 0; s < S; ++s) o += BinConst<LM>::plan.bin[B].seg[s].n;
            return o;
        }();
#pragma unroll
        for (int c = 0; c < g.n; ++c) y[off + c] = Ys[(g.l * g.l + g.c0 + c) * T + k];
        bin_load<R, LM, T, B, S + 1>(y, Ys, k);
    }
}

// the lane's particles of one tile of n; the next one's values are loaded
// before this one's rows
template <typename R, int NR, int LM, int T, int B>
__device__ __forceinline__ void bin_tile(R (&acc)[NR][kBinCap], const R* Ys, const R* Xs, int lane,
                                         int n) {
    R y[kBinCap], xi = Xs[lane];
    bin_load<R, LM, T, B>(y, Ys, lane);
#pragma unroll 1
    for (int k = lane; k < n; k += 32) {
        const int kn = k + 32 < T ? k + 32 : lane;
        R yn[kBinCap];
        const R xn = Xs[kn];
        bin_load<R, LM, T, B>(yn, Ys, kn);
        bin_segment<R, NR, LM, B, 0>(acc, y, xi);
        xi = xn;
#pragma unroll
        for (int c = 0; c < BinConst<LM>::plan.bin[B].ncol; ++c) y[c] = yn[c];
    }
}

template <typename R, int NR, int LM, int T, int B>
__device__ __forceinline__ void bin_dispatch(int warp, R (&acc)[NR][kBinCap], const R* Ys,
                                             const R* Xs, int lane, int n) {
    if constexpr (B < BinConst<LM>::nbins) {
        if (warp == B) bin_tile<R, NR, LM, T, B>(acc, Ys, Xs, lane, n);
        else bin_dispatch<R, NR, LM, T, B + 1>(warp, acc, Ys, Xs, lane, n);
    }
}

// phase 1: w_l H_l^m of the columns of orders m in [M0, M1] into Ys, order by
// order (the recursion in l at fixed m of harm_level_exact), so that two
// threads share a particle and no thread holds more than two levels of one
// order.  w[l] = m pre0 st^l; (c, s) the sectoral value of order M.
template <typename R, int LM, int T, int M, int M1>
__device__ __forceinline__ void bin_orders(const R (&w)[LM + 1], R ux, R uy, R uz, R c, R s, R* Ys) {
    R c1 = c, s1 = s, c2 = R(0), s2 = R(0);   // level l - 1, l - 2 below
#pragma unroll
    for (int l = M; l <= LM; ++l) {
        if (l > M) {
            const R d = R(2 * l - 1) * uz, b = R((l + M - 1) * (l - M - 1));
            const R cn = l == M + 1 ? d * c1 : fma(d, c1, -b * c2);
            const R sn = l == M + 1 ? d * s1 : fma(d, s1, -b * s2);
            c2 = c1; s2 = s1;
            c1 = cn; s1 = sn;
        }
        if constexpr (M == 0) {
            Ys[l * l * T] = w[l] * c1;
        } else {
            Ys[(l * l + 2 * M - 1) * T] = w[l] * c1;
            Ys[(l * l + 2 * M) * T] = w[l] * s1;
        }
    }
    if constexpr (M < M1) {
        constexpr R d = R(2 * M + 1);
        bin_orders<R, LM, T, M + 1, M1>(w, ux, uy, uz, d * (ux * c - uy * s), d * (ux * s + uy * c), Ys);
    }
}
// orders 0..half-1 have about half of the columns
template <int LM>
__host__ __device__ constexpr int bin_half_order() {
    int m = 1, cols = LM + 1;
    while (2 * cols + 2 * (LM + 1 - m) <= (LM + 1) * (LM + 1) + 2) cols += 2 * (LM + 1 - m++);
    return m;
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

// Two threads per particle in phase 1, one warp per bin in phase 2, one block
// per SM: 105 accumulators a lane leave room for 12 warps.  Every bin is
// straight-line code of its own, and so is phase 1: with tiles of 192
// particles a third of the warps' time went to waiting for instructions (six
// rounds per lane and bin), so a tile is as large as shared memory holds once
// and the two phases alternate.  Bound: FMA issue, NR x 7 updates and a
// recursion of 2 NR per bin and particle.  (14, 8), 2^24 particles: 2645 us
// with phase 1 on half of the warps and an FP64 addition per column in the
// flush, 2158 without these and with two buffers of 192, 2050 so.
template <int LM>
__host__ __device__ constexpr int bins_threads() { return BinConst<LM>::nbins * 32; }
template <int LM>
__host__ __device__ constexpr int bins_tile() { return bins_threads<LM>() * 3 / 2; }
template <typename R, int NR, int LM, bool DRIFT>
constexpr size_t bins_smem() {
    return ((size_t)BinConst<LM>::nbins * NR * kBinCap * sizeof(double) + 15) / 16 * 16 +
           (size_t)bins_tile<LM>() * ((DRIFT ? 3 : 1) * sizeof(Vec4<R>) + ((LM + 1) * (LM + 1) + 1) * sizeof(R));
}
// DRIFT: kick and drift the particles as they are read (the copies of a tile's
// velocities and accelerations are hidden behind the contraction of the tile
// before; a kick-drift kernel is bound by memory, 188 us at 2^24).
template <typename R, int NR, int LM, bool DRIFT>
__global__ void __launch_bounds__(bins_threads<LM>(), 1)
scf_coeff_bins_kernel(ScfBinParams p) {
    constexpr int NB = BinConst<LM>::nbins;
    constexpr int TH = NB * 32;         // threads: one warp per bin
    constexpr int T = bins_tile<LM>();  // particles per tile
    constexpr int K1 = TH / 2;          // particles per round of phase 1
    static_assert(T % 32 == 0 && T % K1 == 0, "tile");
    constexpr int NCOL = (LM + 1) * (LM + 1);
    constexpr int NOUT = NB * NR * kBinCap;
    using V4 = Vec4<R>;
    // dynamic shared memory: accd [NOUT] doubles, the next tile's particles
    // P [T], (DRIFT) their velocities and accelerations V [T], A [T], then
    // Ys [NCOL][T] and xi [T]
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* accd = reinterpret_cast<double*>(smem_raw);
    V4* P = reinterpret_cast<V4*>(smem_raw + ((NOUT * sizeof(double) + 15) / 16) * 16);
    V4* V = P + T;
    V4* A = V + T;
    R* Ys = reinterpret_cast<R*>(P + (DRIFT ? 3 : 1) * T);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k1 = tid < K1 ? tid : tid - K1;   // phase 1: this thread's particle
    const V4* posm = reinterpret_cast<const V4*>(p.posm);
    for (int e = tid; e < NOUT; e += TH) accd[e] = 0.0;
    R acc[NR][kBinCap];
#pragma unroll
    for (int n = 0; n < NR; ++n)
#pragma unroll
        for (int c = 0; c < kBinCap; ++c) acc[n][c] = R(0);

    // FP64 additions are slow on this GPU: each total is one lane's, so that a
    // few warp-wide instructions add them all
    auto flush = [&]() {
        constexpr int kPerWarp = NR * kBinCap, K = (kPerWarp + 31) / 32 * 32;
        R v[K];
#pragma unroll
        for (int i = 0; i < K; ++i) v[i] = i < kPerWarp ? acc[i / kBinCap][i % kBinCap] : R(0);
        warp_scatter<K, 16>(v, lane);
#pragma unroll
        for (int i = 0; i < K / 32; ++i) {
            const int idx = lane * (K / 32) + i;
            if (idx < kPerWarp) accd[warp * kPerWarp + idx] += (double)v[i];
        }
#pragma unroll
        for (int n = 0; n < NR; ++n)
#pragma unroll
            for (int c = 0; c < kBinCap; ++c) acc[n][c] = R(0);
    };
    const int64_t lo = (int64_t)blockIdx.x * p.per;
    const int64_t hi = lo + p.per < p.N ? lo + p.per : p.N;
    // asynchronous copy of the particles of the tile at `first`; each thread
    // waits for its own before the barrier
    auto fetch = [&](int64_t first) {
        for (int i = tid; i < T; i += TH) {
            if (first + i < hi) {
                cp_async16(P + i, posm + first + i);
                if (DRIFT) {
                    cp_async16(V + i, reinterpret_cast<const V4*>(p.vel) + first + i);
                    cp_async16(A + i, reinterpret_cast<const V4*>(p.acc) + first + i);
                }
            }
        }
        cp_async_commit();
    };
    // the thread's own copies have arrived: kick, drift, and back to memory
    auto step = [&](int64_t first) {
        const R dt = (R)p.dt, h = R(0.5) * dt;
        for (int i = tid; i < T && first + i < hi; i += TH) {
            V4 x = P[i], v = V[i];
            kick_drift(x, v, A[i], h, dt);
            st4(reinterpret_cast<V4*>(p.vel) + first + i, v);
            st4(reinterpret_cast<V4*>(p.drift_posm) + first + i, x);
            P[i] = x;
        }
    };
    auto basis = [&](const V4& cur, int k) {
        R x = R(0), y = R(0), z = R(0), m = R(0);
        if (finite4(cur.x, cur.y, cur.z, cur.w)) { x = cur.x; y = cur.y; z = cur.z; m = cur.w; }
        else report(p.err, ETICS_ERR_NONFINITE);
        const R r = sqrt(x * x + y * y + z * z);
        const R t = R(1) / (R(1) + r), st = r * t * t;
        const R inv = r > R(0) ? R(1) / r : R(0);
        R w[LM + 1];
        w[0] = -m * t;
#pragma unroll
        for (int l = 1; l <= LM; ++l) w[l] = w[l - 1] * st;
        constexpr int H = bin_half_order<LM>();
        const R ux = x * inv, uy = y * inv, uz = z * inv;
        if (tid < K1) {
            Ys[NCOL * T + k] = R(1) - R(2) * t;
            bin_orders<R, LM, T, 0, H - 1>(w, ux, uy, uz, R(1), R(0), Ys + k);
        } else {
            R c = R(1), s = R(0);
#pragma unroll
            for (int m1 = 1; m1 <= H; ++m1) {
                const R cn = R(2 * m1 - 1) * (ux * c - uy * s);
                s = R(2 * m1 - 1) * (ux * s + uy * c);
                c = cn;
            }
            bin_orders<R, LM, T, H, LM>(w, ux, uy, uz, c, s, Ys + k);
        }
    };

    if (lo < hi) fetch(lo);
    int since = 0;
    for (int64_t first = lo; first < hi; first += T) {
        const int n = hi - first < T ? (int)(hi - first) : T;
        cp_async_wait_all();
        if (DRIFT) step(first);
        __syncthreads();   // P is there; the last tile's columns are read
#pragma unroll 1
        for (int k = k1; k < n; k += K1) basis(P[k], k);
        __syncthreads();   // the columns are there; P is free
        if (first + T < hi) fetch(first + T);
        bin_dispatch<R, NR, LM, T, 0>(warp, acc, Ys, Ys + NCOL * T, lane, n);
        if (++since == kBinFlushTiles) { flush(); since = 0; }
    }
    if (since) flush();
    __syncthreads();
    double* out = p.partial + (size_t)blockIdx.x * NOUT;
    for (int e = tid; e < NOUT; e += TH) out[e] = accd[e];
}

// sum block partials in a fixed order; one warp per output c[n][l*l+l+m]
template <int NR, int LM>
__global__ void scf_finalize_bins_kernel(const double* __restrict__ partial, int nblocks,
                                         double* __restrict__ coeffs) {
    constexpr int NJ = (LM + 1) * (LM + 1);
    constexpr int NOUT = BinConst<LM>::nbins * NR * kBinCap;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= NR * NJ) return;
    const int n = warp / NJ, jj = warp % NJ;
    int l = 0;
    while ((l + 1) * (l + 1) <= jj) ++l;
    const int m = jj - l * l - l;
    const int col = (m == 0) ? 0 : (m > 0 ? 2 * m - 1 : -2 * m);
    const int b = c_bin_index<LM>.bin[l * l + col];
    const int slot = c_bin_index<LM>.slot[l * l + col];
    const int idx = (b * NR + n) * kBinCap + slot;
    double s = 0.0;
    for (int k = lane; k < nblocks; k += 32) s += partial[(size_t)k * NOUT + idx];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        const int am = m < 0 ? -m : m;
        coeffs[warp] = s * c_tab.knorm_fact[l * (l + 1) / 2 + am] * c_tab.inv_j[n][l] *
                       geg_gamma(0, l, n);
    }
}

template <typename R, int NR, int LM>
inline size_t scf_bins_workspace(int num_sms) {
    return (size_t)num_sms * BinConst<LM>::nbins * NR * kBinCap * sizeof(double);
}

template <typename R, int NR, int LM>
inline int scf_coeffs_bins_launch(const void* posm, int64_t N, double* coeffs, void* ws,
                                  DriftStep drift, const LaunchCtx& ctx) {
    constexpr int TH = bins_threads<LM>();
    // contiguous equal ranges of at least 64 particles
    int64_t per = (N + ctx.num_sms - 1) / ctx.num_sms;
    if (per < 64) per = 64;
    const int grid = (int)((N + per - 1) / per);
    ScfBinParams p{posm, N, per, reinterpret_cast<double*>(ws), ctx.err,
                   drift.posm, drift.vel, drift.acc, drift.dt};
    static_assert(bins_smem<R, NR, LM, true>() <= 227 * 1024, "bins kernel shared memory");
    const size_t smem = drift.posm ? bins_smem<R, NR, LM, true>() : bins_smem<R, NR, LM, false>();
    int nblocks = 0;
    if (N > 0) {
        auto k = drift.posm ? scf_coeff_bins_kernel<R, NR, LM, true>
                            : scf_coeff_bins_kernel<R, NR, LM, false>;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) ||
            cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100))
            return ETICS_ERR_CUDA;
        k<<<grid, TH, smem, ctx.stream>>>(p);
        if (cudaGetLastError() != cudaSuccess) return ETICS_ERR_CUDA;
        ++*ctx.launches;
        nblocks = grid;
    }
    stage_event(ctx, 1);
    const int nc = NR * (LM + 1) * (LM + 1);
    scf_finalize_bins_kernel<NR, LM><<<(nc * 32 + 255) / 256, 256, 0, ctx.stream>>>(
        p.partial, nblocks, coeffs);
    if (cudaGetLastError() != cudaSuccess) return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}

}  // namespace etics
