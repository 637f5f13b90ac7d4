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
// A bin's columns in its lane's accumulators 0..6: cos and sin of one order are
// neighbouring columns (c odd, c + 1) and form a pair, so that one paired FMA
// updates both; accumulators 0..5 are three register pairs, 6 is single and
// takes what has no partner in the bin, before the halves of free pairs do.
struct BinItem { int l, c, q; };   // column c (of a pair: c, c + 1) of level l in accumulator q (, q + 1)
struct BinRegs {
    int np, ns;
    BinItem pair[kBinCap / 2], single[kBinCap];
};
constexpr BinRegs make_bin_regs(const BinDef& b) {
    BinRegs r{};
    for (int s = 0; s < b.nseg; ++s)
        for (int c = b.seg[s].c0; c < b.seg[s].c0 + b.seg[s].n; ++c) {
            if (c % 2 == 1 && c + 1 < b.seg[s].c0 + b.seg[s].n) {
                r.pair[r.np] = BinItem{b.seg[s].l, c, 2 * r.np};
                ++r.np;
                ++c;
            } else {
                r.single[r.ns++] = BinItem{b.seg[s].l, c, 0};
            }
        }
    for (int i = 0; i < r.ns; ++i) r.single[i].q = i == 0 ? kBinCap - 1 : 2 * r.np + i - 1;
    return r;
}
template <int LM>
constexpr BinIndex<LM> make_bin_acc_index() {   // column -> (bin, accumulator)
    BinIndex<LM> ix = make_bin_index<LM>();
    constexpr BinPlan<LM> p = make_bin_plan<LM>();
    for (int b = 0; b < p.nbins; ++b) {
        const BinRegs r = make_bin_regs(p.bin[b]);
        for (int i = 0; i < r.np; ++i)
            for (int h = 0; h < 2; ++h)
                ix.slot[r.pair[i].l * r.pair[i].l + r.pair[i].c + h] = r.pair[i].q + h;
        for (int i = 0; i < r.ns; ++i)
            ix.slot[r.single[i].l * r.single[i].l + r.single[i].c] = r.single[i].q;
    }
    return ix;
}
// device copy of it, read with run-time indices
template <int LM>
static __constant__ BinIndex<LM> c_bin_index = make_bin_acc_index<LM>();

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

// A lane's accumulators (or its columns' values) in the order of BinRegs
struct BinValues {
    float2 p[kBinCap / 2];
    float s;
};
// The columns of a tile of T particles in shared memory: the (cos, sin) pairs
// of (l, m), m >= 1, at (l (l-1) / 2 + m - 1) T as float2, the m = 0 columns
// behind them at l T, then xi.
template <int LM, int T>
__device__ __forceinline__ const float* bin_zonal(const float2* Y) {
    return reinterpret_cast<const float*>(Y + LM * (LM + 1) / 2 * T);
}
__host__ __device__ constexpr int bin_pair_column(int l, int c) { return l * (l - 1) / 2 + (c + 1) / 2 - 1; }

// rows of segment S of bin B and the segments after it for one particle: the
// Gegenbauer values of the segment's level times its columns y (harmonics
// scaled by mass and radial prefactor)
template <int NR, int LM, int B, int S>
__device__ __forceinline__ void bin_segment(BinValues (&acc)[NR], const BinValues& y, float xi) {
    constexpr BinDef bd = BinConst<LM>::plan.bin[B];
    if constexpr (S < bd.nseg) {
        constexpr int l = bd.seg[S].l;
        constexpr BinRegs r = make_bin_regs(bd);
        float cm1 = 0.0f, cn = 1.0f;
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            if (n == 1) {
                cm1 = cn;
                cn = xi;
            } else if (n > 1) {
                const float cnew = fma(xi, cn, -geg_bs<float>(l, n) * cm1);   // rescaled
                cm1 = cn;
                cn = cnew;
            }
#pragma unroll
            for (int i = 0; i < r.np; ++i)
                if (r.pair[i].l == l)
                    acc[n].p[i] = n == 0 ? add2(acc[n].p[i], y.p[i])
                                         : fma2(splat<float2>(cn), y.p[i], acc[n].p[i]);
#pragma unroll
            for (int i = 0; i < r.ns; ++i)
                if (r.single[i].l == l) {
                    const int q = r.single[i].q;
                    if (q == kBinCap - 1) acc[n].s = fma(cn, y.s, acc[n].s);
                    else if (q % 2 == 0) acc[n].p[q / 2].x = fma(cn, y.p[q / 2].x, acc[n].p[q / 2].x);
                    else acc[n].p[q / 2].y = fma(cn, y.p[q / 2].y, acc[n].p[q / 2].y);
                }
        }
        bin_segment<NR, LM, B, S + 1>(acc, y, xi);
    }
}
template <int LM, int T, int B>
__device__ __forceinline__ void bin_load(BinValues& y, const float2* Y, int k) {
    constexpr BinRegs r = make_bin_regs(BinConst<LM>::plan.bin[B]);
#pragma unroll
    for (int i = 0; i < r.np; ++i) y.p[i] = Y[bin_pair_column(r.pair[i].l, r.pair[i].c) * T + k];
#pragma unroll
    for (int i = 0; i < r.ns; ++i) {
        const int l = r.single[i].l, c = r.single[i].c, q = r.single[i].q;
        const float v = c == 0 ? bin_zonal<LM, T>(Y)[l * T + k]
                               : reinterpret_cast<const float*>(Y)[2 * (bin_pair_column(l, c) * T + k) +
                                                                   (c + 1) % 2];
        if (q == kBinCap - 1) y.s = v;
        else if (q % 2 == 0) y.p[q / 2].x = v;
        else y.p[q / 2].y = v;
    }
}

// the lane's particles of one tile of n; the next one's values are loaded
// before this one's rows
template <int NR, int LM, int T, int B>
__device__ __forceinline__ void bin_tile(BinValues (&acc)[NR], const float2* Y, int lane, int n) {
    const float* Xs = bin_zonal<LM, T>(Y) + (LM + 1) * T;
    BinValues y = {};
    float xi = Xs[lane];
    bin_load<LM, T, B>(y, Y, lane);
#pragma unroll 1
    for (int k = lane; k < n; k += 32) {
        const int kn = k + 32 < T ? k + 32 : lane;
        BinValues yn = {};
        const float xn = Xs[kn];
        bin_load<LM, T, B>(yn, Y, kn);
        bin_segment<NR, LM, B, 0>(acc, y, xi);
        xi = xn;
        y = yn;
    }
}

template <int NR, int LM, int T, int B>
__device__ __forceinline__ void bin_dispatch(int warp, BinValues (&acc)[NR], const float2* Y, int lane,
                                             int n) {
    if constexpr (B < BinConst<LM>::nbins) {
        if (warp == B) bin_tile<NR, LM, T, B>(acc, Y, lane, n);
        else bin_dispatch<NR, LM, T, B + 1>(warp, acc, Y, lane, n);
    }
}

// sectoral value (cos, sin) of order m from that of order m - 1
__device__ __forceinline__ float2 bin_sectoral(int m, float2 cs, float ux, float uy) {
    const float d = 2 * m - 1;
    return mk2(d * (ux * cs.x - uy * cs.y), d * (ux * cs.y + uy * cs.x));
}

// phase 1: w_l H_l^m of the columns of orders m in [M, M1] of particle k into
// Y, order by order (the recursion in l at fixed m of harm_level_exact, cos and
// sin as one pair), so that two threads share a particle and no thread holds
// more than two levels of one order.  w[l] = m pre0 st^l; cs the sectoral value
// of order M.
template <int LM, int T, int M, int M1>
__device__ __forceinline__ void bin_orders(const float (&w)[LM + 1], float ux, float uy, float uz,
                                           float2 cs, float2* Y, int k) {
    if constexpr (M == 0) {
        float* Z = const_cast<float*>(bin_zonal<LM, T>(Y));
        float c1 = 1.0f, c2 = 0.0f;   // levels l - 1 and l - 2
#pragma unroll
        for (int l = 0; l <= LM; ++l) {
            if (l > 0) {
                const float d = (2 * l - 1) * uz;
                const float cn = l == 1 ? d * c1 : fma(d, c1, -(float)((l - 1) * (l - 1)) * c2);
                c2 = c1;
                c1 = cn;
            }
            Z[l * T + k] = w[l] * c1;
        }
    } else {
        float2 v1 = cs, v2 = mk2(0.0f, 0.0f);
#pragma unroll
        for (int l = M; l <= LM; ++l) {
            if (l > M) {
                const float2 d = splat<float2>((2 * l - 1) * uz);
                const float2 vn = l == M + 1 ? mul2(d, v1)
                                             : fma2(d, v1, mul2(splat<float2>(-(float)((l + M - 1) * (l - M - 1))), v2));
                v2 = v1;
                v1 = vn;
            }
            Y[bin_pair_column(l, 2 * M) * T + k] = mul2(splat<float2>(w[l]), v1);
        }
    }
    if constexpr (M < M1)
        bin_orders<LM, T, M + 1, M1>(w, ux, uy, uz, bin_sectoral(M + 1, cs, ux, uy), Y, k);
}
// orders 0..half-1 have about half of the columns
template <int LM>
__host__ __device__ constexpr int bin_half_order() {
    int m = 1, cols = LM + 1;
    while (2 * cols + 2 * (LM + 1 - m) <= (LM + 1) * (LM + 1) + 2) cols += 2 * (LM + 1 - m++);
    return m;
}

// Two threads per particle in phase 1, one warp per bin in phase 2, one block
// per SM: 105 accumulators a lane leave room for 12 warps.  Every bin is
// straight-line code of its own, and so is phase 1: with tiles of 192
// particles a third of the warps' time went to waiting for instructions (six
// rounds per lane and bin), so a tile is as large as shared memory holds once
// and the two phases alternate.  Bound: FMA issue, NR x 7 updates and a
// recursion of 2 NR per bin and particle.  (14, 8), 2^24 particles: 2645 us
// with phase 1 on half of the warps and an FP64 addition per column in the
// flush, 2158 without these and with two buffers of 192, 2050 with this tile,
// 1390 with cos and sin updated by one paired FMA (fewer instructions to fetch
// and to issue: the FMA pipe's share of busy cycles went from 45% to 56%).
template <int LM>
__host__ __device__ constexpr int bins_threads() { return BinConst<LM>::nbins * 32; }
template <int LM>
__host__ __device__ constexpr int bins_tile() { return bins_threads<LM>() * 3 / 2; }
template <int NR, int LM, bool DRIFT>
constexpr size_t bins_smem() {
    return ((size_t)BinConst<LM>::nbins * NR * kBinCap * sizeof(double) + 15) / 16 * 16 +
           (size_t)bins_tile<LM>() * ((DRIFT ? 3 : 1) * sizeof(float4) + ((LM + 1) * (LM + 1) + 1) * sizeof(float));
}
// DRIFT: kick and drift the particles as they are read (the copies of a tile's
// velocities and accelerations are hidden behind the contraction of the tile
// before; a kick-drift kernel is bound by memory, 188 us at 2^24).
template <int NR, int LM, bool DRIFT>
__global__ void __launch_bounds__(bins_threads<LM>(), 1)
scf_coeff_bins_kernel(ScfBinParams p) {
    constexpr int NB = BinConst<LM>::nbins;
    constexpr int TH = NB * 32;         // threads: one warp per bin
    constexpr int T = bins_tile<LM>();  // particles per tile
    constexpr int K1 = TH / 2;          // particles per round of phase 1
    static_assert(T % 32 == 0 && T % K1 == 0, "tile");
    constexpr int NOUT = NB * NR * kBinCap;
    using V4 = float4;
    // dynamic shared memory: accd [NOUT] doubles, the next tile's particles
    // P [T], (DRIFT) their velocities and accelerations V [T], A [T], then the
    // columns and xi
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* accd = reinterpret_cast<double*>(smem_raw);
    V4* P = reinterpret_cast<V4*>(smem_raw + ((NOUT * sizeof(double) + 15) / 16) * 16);
    V4* V = P + T;
    V4* A = V + T;
    float2* Y = reinterpret_cast<float2*>(P + (DRIFT ? 3 : 1) * T);   // see bin_zonal
    float* Xs = const_cast<float*>(bin_zonal<LM, T>(Y)) + (LM + 1) * T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k1 = tid < K1 ? tid : tid - K1;   // phase 1: this thread's particle
    const V4* posm = reinterpret_cast<const V4*>(p.posm);
    for (int e = tid; e < NOUT; e += TH) accd[e] = 0.0;
    BinValues acc[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) acc[n] = BinValues{};

    // FP64 additions are slow on this GPU: each total is one lane's, so that a
    // few warp-wide instructions add them all
    auto flush = [&]() {
        constexpr int kPerWarp = NR * kBinCap, K = (kPerWarp + 31) / 32 * 32;
        float v[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int q = i % kBinCap;
            if (i >= kPerWarp) { v[i] = 0.0f; continue; }
            const BinValues& a = acc[i / kBinCap];
            v[i] = q == kBinCap - 1 ? a.s : q % 2 == 0 ? a.p[q / 2].x : a.p[q / 2].y;
        }
        warp_scatter<K, 16>(v, lane);
#pragma unroll
        for (int i = 0; i < K / 32; ++i) {
            const int idx = lane * (K / 32) + i;
            if (idx < kPerWarp) accd[warp * kPerWarp + idx] += (double)v[i];
        }
#pragma unroll
        for (int n = 0; n < NR; ++n) acc[n] = BinValues{};
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
        const float dt = (float)p.dt, h = 0.5f * dt;
        for (int i = tid; i < T && first + i < hi; i += TH) {
            V4 x = P[i], v = V[i];
            kick_drift(x, v, A[i], h, dt);
            st4(reinterpret_cast<V4*>(p.vel) + first + i, v);
            st4(reinterpret_cast<V4*>(p.drift_posm) + first + i, x);
            P[i] = x;
        }
    };
    auto basis = [&](const V4& cur, int k) {
        float x = 0.0f, y = 0.0f, z = 0.0f, m = 0.0f;
        if (finite4(cur.x, cur.y, cur.z, cur.w)) { x = cur.x; y = cur.y; z = cur.z; m = cur.w; }
        else report(p.err, ETICS_ERR_NONFINITE);
        const float r = sqrtf(x * x + y * y + z * z);
        const float t = 1.0f / (1.0f + r), st = r * t * t;
        const float inv = r > 0.0f ? 1.0f / r : 0.0f;
        float w[LM + 1];
        w[0] = -m * t;
#pragma unroll
        for (int l = 1; l <= LM; ++l) w[l] = w[l - 1] * st;
        constexpr int H = bin_half_order<LM>();
        const float ux = x * inv, uy = y * inv, uz = z * inv;
        float2 cs = mk2(1.0f, 0.0f);
        if (tid < K1) {
            Xs[k] = 1.0f - 2.0f * t;
            bin_orders<LM, T, 0, H - 1>(w, ux, uy, uz, cs, Y, k);
        } else {
#pragma unroll
            for (int m1 = 1; m1 <= H; ++m1) cs = bin_sectoral(m1, cs, ux, uy);
            bin_orders<LM, T, H, LM>(w, ux, uy, uz, cs, Y, k);
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
        bin_dispatch<NR, LM, T, 0>(warp, acc, Y, lane, n);
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

template <int NR, int LM>
inline size_t scf_bins_workspace(int num_sms) {
    return (size_t)num_sms * BinConst<LM>::nbins * NR * kBinCap * sizeof(double);
}

template <int NR, int LM>
inline int scf_coeffs_bins_launch(const void* posm, int64_t N, double* coeffs, void* ws,
                                  DriftStep drift, const LaunchCtx& ctx) {
    constexpr int TH = bins_threads<LM>();
    // contiguous equal ranges of at least 64 particles
    int64_t per = (N + ctx.num_sms - 1) / ctx.num_sms;
    if (per < 64) per = 64;
    const int grid = (int)((N + per - 1) / per);
    ScfBinParams p{posm, N, per, reinterpret_cast<double*>(ws), ctx.err,
                   drift.posm, drift.vel, drift.acc, drift.dt};
    static_assert(bins_smem<NR, LM, true>() <= 227 * 1024, "bins kernel shared memory");
    const size_t smem = drift.posm ? bins_smem<NR, LM, true>() : bins_smem<NR, LM, false>();
    int nblocks = 0;
    if (N > 0) {
        auto k = drift.posm ? scf_coeff_bins_kernel<NR, LM, true>
                            : scf_coeff_bins_kernel<NR, LM, false>;
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
