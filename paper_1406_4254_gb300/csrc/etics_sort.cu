// etics_sort.cu -- the radial sort of MEX (paper Sec. 2.2: the cumulative
// sums need the particles ordered by radius; Sec. 3.2 used a library merge
// sort).
//
// GB300 design, two paths that give the same order, the exact FP64 order
// (r^2 = (x*x + y*y) + z*z rounded as a CPU does, ties by index):
//
// Up to kSampleMaxN particles, a sample sort: one partition of the particles
// into buckets of about 1024 (by a table of the keys' cumulative distribution,
// from a sample), then one block per bucket sorts it in shared memory by the
// 64-bit pattern of r^2 and writes the order and the particles themselves.  Up
// to kSingleMax particles the last kernel alone does it.  Two dependent launches
// instead of the radix path's six, and three passes over the particles instead
// of ten over keys.
//
// Above, a hand-written stable LSD radix sort (4 passes of 8 bits) of
// the high 32 bits of the FP64 r^2 bit pattern, one kernel per pass
// ("one-sweep": per-tile digit ranking with warp ballots, the tile's keys
// placed in digit order in shared memory, a decoupled lookback over tiles for
// the digit offsets, coalesced writes of digit runs).  Runs of equal high
// words are then ordered by the low 32 bits and the particle index, and the
// particles are gathered into that order.
//
// All kernels are launched with programmatic dependent launch, so each launch
// overlaps its predecessor's tail.
#include <algorithm>
#include <array>
#include <atomic>
#include <utility>
#include <cstddef>

#include "etics_internal.h"
#include "etics_r2.h"

namespace etics {

constexpr int kSortThreads = 256;
constexpr int kSortKpt = 16;
constexpr int kSortTile = kSortThreads * kSortKpt;   // 4096 keys per tile
constexpr int kLookbackWindow = 32;
constexpr int kStatusPad = kLookbackWindow;   // zeroed tiles before tile 0
constexpr int kMatchDigits = 8;               // rank with match_any up to this many digits
constexpr uint32_t kCountMask = (1u << 30) - 1;
constexpr uint32_t kFlagAgg = 1u << 30;
constexpr uint32_t kFlagInc = 2u << 30;
constexpr int64_t kSpinLimit = int64_t(1) << 22;   // default bound of a lookback wait

int sort_tiles(int64_t N) { return (int)((N + kSortTile - 1) / kSortTile); }

// r^2 exactly as a CPU evaluates (x*x + y*y) + z*z in FP64, no contraction
__device__ __forceinline__ double r2_fp64(double x, double y, double z) {
    return __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
}

// High 32 bits of the FP64 bit pattern of r^2 (the sort key; positive doubles
// order like their bit patterns).
//
// FP32 particles: every square is exact in FP64, so fl64(fl64(x*x+y*y)+z*z)
// differs from the exact sum S by at most 2 FP64 ulps.  S is evaluated as an
// FP32 pair (hi, lo) with error ~2^-45 |S| (exact products by FMA, TwoSum),
// and the key is read off the pair: the top 20 mantissa bits of hi, minus one
// when lo < 0 borrows across a bucket boundary (the low 3 mantissa bits of hi
// are zero).  Only when S lies within 2^-40 |S| of a bucket boundary is the
// key recomputed in FP64, so the result always equals the FP64 evaluation.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ uint32_t key_from_fp64(double r2) {
    return (uint32_t)((uint64_t)__double_as_longlong(r2) >> 32);
}

__device__ __forceinline__ uint32_t r2_key(float x, float y, float z) {
    const float hx = x * x, lx = fmaf(x, x, -hx);
    const float hy = y * y, ly = fmaf(y, y, -hy);
    const float hz = z * z, lz = fmaf(z, z, -hz);
    float s1, e1, s2, e2;
    two_sum(hx, hy, s1, e1);
    two_sum(s1, hz, s2, e2);
    const float low = ((lx + ly) + lz) + (e1 + e2);
    const float hi = s2 + low;                  // fast two-sum: |s2| >= |low|
    const float lo = low - (hi - s2);
    const uint32_t hb = __float_as_uint(hi);
    const uint32_t exp8 = hb >> 23, frac = hb & 0x7fffffu;
    // tiny (r^2 < 2^-63), non-finite or overflowing sums take the FP64 route
    bool exact_needed = exp8 < 64u || exp8 == 255u;
    uint32_t key = 0;
    if (!exact_needed) {
        key = ((exp8 + 896u) << 20) | (frac >> 3);   // FP64 exponent field = exp8 - 127 + 1023
        if ((frac & 7u) == 0u) {
            if (fabsf(lo) <= hi * 0x1p-40f) exact_needed = true;   // too close to call
            else if (lo < 0.0f) key -= 1u;                        // borrow below the boundary
        }
    }
    if (exact_needed) {
        const double dx = x, dy = y, dz = z;
        key = key_from_fp64(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)),
                                      __dmul_rn(dz, dz)));
    }
    return key;
}
__device__ __forceinline__ uint32_t r2_key(double x, double y, double z) {
    return key_from_fp64(r2_fp64(x, y, z));
}

constexpr int kKeygenIlp = 4;

template <typename R>
__global__ void __launch_bounds__(256)
keygen_kernel(const Vec4<R>* __restrict__ posm, int64_t N, uint32_t* __restrict__ key,
              uint32_t* __restrict__ hist, unsigned* err) {
    // one private copy of the 4 digit histograms per warp (less atomic contention)
    __shared__ uint32_t sh[8][4 * 256];
    const int warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 8 * 4 * 256; i += blockDim.x) (&sh[0][0])[i] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < N;
         i0 += stride * kKeygenIlp) {
        Vec4<R> v[kKeygenIlp];
#pragma unroll
        for (int u = 0; u < kKeygenIlp; ++u) {
            const int64_t i = i0 + u * stride;
            if (i < N) v[u] = ld4(posm + i);
        }
#pragma unroll
        for (int u = 0; u < kKeygenIlp; ++u) {
            const int64_t i = i0 + u * stride;
            if (i >= N) break;
            uint32_t hi;
            if (finite4(v[u].x, v[u].y, v[u].z, v[u].w)) {
                hi = r2_key(v[u].x, v[u].y, v[u].z);
            } else {
                report(err, ETICS_ERR_NONFINITE);
                hi = 0xffffffffu;
            }
            key[i] = hi;
            // the histograms of digits 1 and 2 are counted by the radix
            // passes 0 and 1 (their keys are in registers there anyway)
            atomicAdd(&sh[warp][hi & 255], 1u);
            // the top byte (sign + high exponent bits) takes very few values:
            // aggregate equal digits within the warp before the atomic
            const uint32_t d3 = hi >> 24;
            const unsigned same = __match_any_sync(__activemask(), d3);
            if ((same & ((1u << (threadIdx.x & 31)) - 1u)) == 0u)
                atomicAdd(&sh[warp][768 + d3], (uint32_t)__popc(same));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * 256; i += blockDim.x) {
        if (i >= 256 && i < 768) continue;   // digits 1, 2: counted by the passes
        uint32_t t = 0;
        for (int w = 0; w < 8; ++w) t += sh[w][i];
        if (t) atomicAdd(&hist[i], t);
    }
}

template <typename R>
__global__ void radial_keys_kernel(const Vec4<R>* __restrict__ posm, int64_t N,
                                   uint32_t* __restrict__ keys, unsigned* err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const Vec4<R> v = ld4(posm + i);
        if (finite4(v.x, v.y, v.z, v.w)) {
            keys[i] = r2_key(v.x, v.y, v.z);
        } else {
            report(err, ETICS_ERR_NONFINITE);
            keys[i] = 0xffffffffu;
        }
    }
}

template <typename R>
int radial_keys_impl(const void* posm, int64_t N, uint32_t* keys, const LaunchCtx& ctx) {
    if (N == 0) return ETICS_OK;
    int g = (int)((N + 255) / 256);
    if (g > ctx.num_sms * 8) g = ctx.num_sms * 8;
    radial_keys_kernel<R><<<g, 256, 0, ctx.stream>>>(reinterpret_cast<const Vec4<R>*>(posm), N,
                                                      keys, ctx.err);
    if (cudaGetLastError()) return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}
template int radial_keys_impl<float>(const void*, int64_t, uint32_t*, const LaunchCtx&);
template int radial_keys_impl<double>(const void*, int64_t, uint32_t*, const LaunchCtx&);

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) {
    return *reinterpret_cast<const volatile uint32_t*>(p);
}
__device__ __forceinline__ void st_volatile(uint32_t* p, uint32_t v) {
    *reinterpret_cast<volatile uint32_t*>(p) = v;
}

// Stable rank of every key among the equal digits of its warp, keys taken in
// tile order (slot s, then lane).  The lanes that share a digit are found
// either with __match_any_sync (fast when a warp holds few distinct digits)
// or with one ballot per digit bit plus one for validity (a cost independent
// of how many distinct digits there are).
template <bool kMatch, int K>
__device__ __forceinline__ void rank_in_warp(const uint32_t (&d)[K], uint32_t (&rank)[K],
                                             uint32_t* whist, int lane) {
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int s = 0; s < K; ++s) {
        unsigned mask;
        if (kMatch) {
            mask = __match_any_sync(0xffffffffu, d[s]);
        } else {
            const unsigned vb = __ballot_sync(0xffffffffu, d[s] < 256u);
            mask = d[s] < 256u ? vb : ~vb;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const bool bit = (d[s] >> b) & 1u;
                const unsigned bal = __ballot_sync(0xffffffffu, bit);
                mask &= bit ? bal : ~bal;
            }
        }
        const unsigned lower = mask & below;
        uint32_t before = 0;
        if (d[s] < 256u) before = whist[d[s]];
        rank[s] = before + (uint32_t)__popc(lower);
        __syncwarp();
        if (d[s] < 256u && lower == 0u) whist[d[s]] = before + (uint32_t)__popc(mask);
        __syncwarp();
    }
}

// Decoupled lookback over the earlier tiles of one digit or bucket (st: this
// tile's status word, stride: words per tile): a window of predecessors is
// read at once; flags become bit masks; counts are summed up to the first
// inclusive prefix, or up to the first predecessor that has not published
// (then that one word is polled before the next window).  The status array
// holds kStatusPad zeroed (never published) tiles before tile 0, so a window
// may reach below tile 0 without a bounds test: tile 0 always publishes an
// inclusive prefix, which ends every walk first.  A tile takes its number from
// a counter, so the tiles waited for have started.  The poll gives up after
// spin_limit tries: the error word records ETICS_ERR_TIMEOUT and the partial
// sum (at most the true one) is returned.
__device__ __forceinline__ uint32_t lookback(const uint32_t* st, size_t stride, int64_t spin_limit,
                                             unsigned* err) {
    uint32_t excl = 0;
    const uint32_t* p = st - stride;   // tile - 1
    int64_t spins = 0;
    for (;;) {
        uint32_t w[kLookbackWindow];
#pragma unroll
        for (int j = 0; j < kLookbackWindow; ++j) w[j] = ld_volatile(p - j * stride);
        uint32_t pub = 0, inc = 0;
#pragma unroll
        for (int j = 0; j < kLookbackWindow; ++j) {
            const uint32_t f = w[j] >> 30;
            pub |= (f != 0u ? 1u : 0u) << j;
            inc |= (f == (kFlagInc >> 30) ? 1u : 0u) << j;
        }
        const int first_wait = ~pub ? __ffs(~pub) - 1 : kLookbackWindow;
        const int first_inc = inc ? __ffs(inc) - 1 : kLookbackWindow;
        const bool done = first_inc < first_wait;
        const int used = done ? first_inc + 1 : first_wait;
        const uint32_t take = used >= 32 ? 0xffffffffu : ((1u << used) - 1u);
#pragma unroll
        for (int j = 0; j < kLookbackWindow; ++j)
            if ((take >> j) & 1u) excl += w[j] & kCountMask;
        if (done) break;
        p -= (size_t)used * stride;
        if (used < kLookbackWindow) {
            bool timed_out = false;
            while ((ld_volatile(p) >> 30) == 0u) {
                if (++spins > spin_limit) { timed_out = true; break; }
                __nanosleep(32);
            }
            if (timed_out) { report(err, ETICS_ERR_TIMEOUT); break; }
        }
    }
    return excl;
}

// One pass of the stable LSD radix sort (8-bit digit at `shift`) over tiles
// of kSortTile keys.  Order of work in a tile: load and rank; publish the
// tile's digit counts (status word: flag | count); scan the global histogram
// and the tile counts together; place the keys in digit order in shared
// memory; then find the exclusive prefix of each digit over earlier tiles by
// a decoupled lookback; finally write the keys out in digit runs.  `status`
// holds kStatusPad zeroed (never published) tiles before tile 0, so a
// lookback window may reach below tile 0 without a bounds test: tile 0
// always publishes an inclusive prefix, which ends every walk first.
// Launched with programmatic stream serialisation: nothing global is touched
// before griddepcontrol.wait.
__global__ void __launch_bounds__(kSortThreads, 2)
onesweep_kernel(const uint32_t* keys_in, const uint32_t* vals_in,
                uint32_t* keys_out, uint32_t* vals_out,
                const uint32_t* hist, uint32_t* status, uint32_t* counter, int shift,
                int64_t N, int64_t spin_limit, uint32_t* next_hist, unsigned* err) {
    __shared__ uint32_t s_keys[kSortTile];
    __shared__ uint32_t s_vals[kSortTile];
    __shared__ uint32_t s_whist[kSortThreads / 32][256];
    __shared__ uint32_t s_dexcl[256];
    __shared__ uint32_t s_gbase[256];
    __shared__ uint32_t s_scan[2][kSortThreads / 32];
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_next[256];   // this tile's histogram of the next digit
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < (kSortThreads / 32) * 256; i += kSortThreads) (&s_whist[0][0])[i] = 0;
    s_next[tid] = 0;
    pdl_wait();
    if (tid == 0) s_tile = atomicAdd(counter, 1u);
    const int dig = tid;
    // the histogram may have been completed by the kernel just before this
    // one (a programmatic dependent launch): a coherent load after the wait,
    // never the non-coherent read-only path
    const uint32_t gcount = ld_cg(hist + dig);
    // digits present in this pass over all keys: few -> rank with match_any
    const int ndig = __syncthreads_count(gcount != 0u);
    const uint32_t tile = s_tile;
    const int64_t start = (int64_t)tile * kSortTile;

    uint32_t k[kSortKpt], v[kSortKpt], d[kSortKpt], rank[kSortKpt];
#pragma unroll
    for (int s = 0; s < kSortKpt; ++s) {
        const int64_t idx = start + (int64_t)warp * kSortKpt * 32 + s * 32 + lane;
        if (idx < N) {
            k[s] = keys_in[idx];
            v[s] = vals_in ? vals_in[idx] : (uint32_t)idx;   // first pass: identity
            d[s] = (k[s] >> shift) & 255u;
        } else {
            k[s] = 0xffffffffu;
            v[s] = 0;
            d[s] = 256u;   // not a digit: out of range
        }
    }
    if (ndig <= kMatchDigits) rank_in_warp<true>(d, rank, s_whist[warp], lane);
    else rank_in_warp<false>(d, rank, s_whist[warp], lane);
    if (next_hist) {
        // the next pass's digit of this tile's keys (the order of the keys
        // does not matter for a histogram): added to the global histogram,
        // which the next pass reads after this one has completed
#pragma unroll
        for (int s = 0; s < kSortKpt; ++s)
            if (d[s] < 256u) atomicAdd(&s_next[(k[s] >> (shift + 8)) & 255u], 1u);
    }
    __syncthreads();
    if (next_hist && s_next[tid]) atomicAdd(&next_hist[tid], s_next[tid]);
    // per digit (one thread each): offsets over warps and the tile count
    uint32_t count = 0;
    for (int w = 0; w < kSortThreads / 32; ++w) {
        const uint32_t t = s_whist[w][dig];
        s_whist[w][dig] = count;
        count += t;
    }
    // publish at once: tile 0 (and any digit no key has) as inclusive
    uint32_t* st = status + (size_t)(tile + kStatusPad) * 256 + dig;
    const bool look = tile != 0 && gcount != 0u;
    st_volatile(st, (look ? kFlagAgg : kFlagInc) | count);
    // exclusive scans of the global histogram (start of each digit) and of
    // the tile counts (start of each digit in the tile), together
    uint32_t xa = gcount, xb = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ta = __shfl_up_sync(0xffffffffu, xa, o);
        const uint32_t tb = __shfl_up_sync(0xffffffffu, xb, o);
        if (lane >= o) { xa += ta; xb += tb; }
    }
    if (lane == 31) { s_scan[0][warp] = xa; s_scan[1][warp] = xb; }
    __syncthreads();
    uint32_t ba = 0, bb = 0;
    for (int w = 0; w < warp; ++w) { ba += s_scan[0][w]; bb += s_scan[1][w]; }
    const uint32_t hexcl = ba + xa - gcount;
    s_dexcl[dig] = bb + xb - count;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < kSortKpt; ++s) {
        if (d[s] < 256u) {
            const uint32_t pos = s_dexcl[d[s]] + s_whist[warp][d[s]] + rank[s];
            s_keys[pos] = k[s];
            s_vals[pos] = v[s];
        }
    }
    // the sum over earlier tiles of this digit; after a wait that gave up (a
    // partial sum, at most the true one) the output positions stay below N;
    // keys that no longer match the histogram (a later pass of a timed-out
    // sort) can compute a position >= N, and such a store is skipped below
    uint32_t excl = 0;
    if (look) {
        excl = lookback(st, 256, spin_limit, err);
        st_volatile(st, kFlagInc | (excl + count));
    }
    s_gbase[dig] = hexcl + excl;
    __syncthreads();
    const int64_t rem = N - start;
    const int nvalid = (int)(rem < kSortTile ? rem : kSortTile);
    if (nvalid == kSortTile) {
#pragma unroll
        for (int s = 0; s < kSortKpt; ++s) {
            const int i = tid + s * kSortThreads;
            const uint32_t kk = s_keys[i];
            const uint32_t dd = (kk >> shift) & 255u;
            const uint32_t pos = s_gbase[dd] + (uint32_t)i - s_dexcl[dd];
            if (pos < N) {
                keys_out[pos] = kk;
                vals_out[pos] = s_vals[i];
            } else {
                report(err, ETICS_ERR_TIMEOUT);
            }
        }
    } else {
        for (int i = tid; i < nvalid; i += kSortThreads) {
            const uint32_t kk = s_keys[i];
            const uint32_t dd = (kk >> shift) & 255u;
            const uint32_t pos = s_gbase[dd] + (uint32_t)i - s_dexcl[dd];
            if (pos < N) {
                keys_out[pos] = kk;
                vals_out[pos] = s_vals[i];
            } else {
                report(err, ETICS_ERR_TIMEOUT);
            }
        }
    }
}

// Runs of equal high words: order by (low word of the FP64 r^2, index).  The
// run's first element owns it; the low words are evaluated here, in FP64, for
// the run members only.  The radix passes are stable and began from index
// order, so a run's members arrive in index order: a stable sort by the low
// word alone gives the (low word, index) order.
// An index >= N (only after a timed-out sort) reads nothing and sorts last.
template <typename R>
__device__ __forceinline__ uint32_t r2_low(const Vec4<R>* posm, uint32_t i, int64_t N) {
    if ((int64_t)i >= N) return 0xffffffffu;
    const Vec4<R> v = ld4(posm + i);
    if (!finite4(v.x, v.y, v.z, v.w)) return 0xffffffffu;
    return (uint32_t)(uint64_t)__double_as_longlong(r2_fp64((double)v.x, (double)v.y, (double)v.z));
}

constexpr int kFixThreads = 256;   // one thread per digit in the block sort below
constexpr int kFixTile = 2048;
constexpr int kFixLocal = 16;      // runs up to this length: one thread, in registers
constexpr int kFixLongMax = kFixTile / (kFixLocal + 1) + 1;   // long runs starting in a tile

// a run of at most kFixLocal members, by one thread (insertion sort)
template <typename R>
__device__ __forceinline__ void sort_run_local(const Vec4<R>* posm, int64_t N, uint32_t* val,
                                               int64_t s, int len) {
    uint32_t lows[kFixLocal], ids[kFixLocal];
    for (int a = 0; a < len; ++a) ids[a] = val[s + a];
    for (int a = 0; a < len; ++a) lows[a] = r2_low<R>(posm, ids[a], N);
    for (int a = 1; a < len; ++a) {
        const uint32_t va = ids[a], la = lows[a];
        int b = a - 1;
        while (b >= 0 && (lows[b] > la || (lows[b] == la && ids[b] > va))) {
            ids[b + 1] = ids[b];
            lows[b + 1] = lows[b];
            --b;
        }
        ids[b + 1] = va;
        lows[b + 1] = la;
    }
    for (int a = 0; a < len; ++a) val[s + a] = ids[a];
}

// A long run (any length), by the whole block: a stable LSD radix sort of
// the members by their low word, 4 passes of 8 bits, ping-ponging between
// val (the sorted order) and tmp (the sort's spare value buffer, over the
// same positions); the low word is re-evaluated from the particle whenever it
// is needed, so nothing is written outside val/tmp[s, s + len).  Each pass:
// digit histogram, exclusive scan, then chunks of kFixThreads members in
// order, each member ranked among equal digits of its warp (ballots) and of
// the earlier warps of the chunk.
template <typename R>
__device__ void sort_run_block(const Vec4<R>* posm, int64_t N, uint32_t* val, uint32_t* tmp,
                               int64_t s, int64_t len, uint32_t (*s_cnt)[256], uint32_t* s_off,
                               uint32_t* s_wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = kFixThreads / 32;
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 8 * pass;
        const uint32_t* src = (pass & 1) ? tmp : val;
        uint32_t* dst = (pass & 1) ? val : tmp;
        for (int w = 0; w < NW; ++w) s_cnt[w][tid] = 0u;
        __syncthreads();
        for (int64_t i = tid; i < len; i += kFixThreads)
            atomicAdd(&s_cnt[0][(r2_low<R>(posm, src[s + i], N) >> shift) & 255u], 1u);
        __syncthreads();
        {
            // exclusive scan over the 256 digits (thread = digit)
            const uint32_t c = s_cnt[0][tid];
            uint32_t x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += t;
            }
            if (lane == 31) s_wsum[warp] = x;
            __syncthreads();
            uint32_t b = 0;
            for (int w = 0; w < warp; ++w) b += s_wsum[w];
            s_off[tid] = b + x - c;
            s_cnt[0][tid] = 0u;
        }
        __syncthreads();
        for (int64_t c0 = 0; c0 < len; c0 += kFixThreads) {
            const int64_t i = c0 + tid;
            const bool valid = i < len;
            const uint32_t v = valid ? src[s + i] : 0u;
            const uint32_t d = valid ? (r2_low<R>(posm, v, N) >> shift) & 255u : 256u;
            const unsigned vb = __ballot_sync(0xffffffffu, valid);
            unsigned mask = valid ? vb : ~vb;
#pragma unroll
            for (int bit = 0; bit < 8; ++bit) {
                const bool on = (d >> bit) & 1u;
                const unsigned bal = __ballot_sync(0xffffffffu, on);
                mask &= on ? bal : ~bal;
            }
            const unsigned lower = mask & ((1u << lane) - 1u);
            if (valid && lower == 0u) s_cnt[warp][d] = (uint32_t)__popc(mask);
            __syncthreads();
            uint32_t total = 0;   // thread = digit: exclusive prefix over the warps
            for (int w = 0; w < NW; ++w) {
                const uint32_t t = s_cnt[w][tid];
                s_cnt[w][tid] = total;
                total += t;
            }
            __syncthreads();
            if (valid) dst[s + s_off[d] + s_cnt[warp][d] + (uint32_t)__popc(lower)] = v;
            __syncthreads();
            s_off[tid] += total;
            for (int w = 0; w < NW; ++w) s_cnt[w][tid] = 0u;
            __syncthreads();
        }
    }
    // 4 passes: the result is back in val
}

// One block per tile of kFixTile sorted positions; the keys of the tile and
// one position on either side are staged in shared memory.  A run belongs to
// the tile where it starts.  The block lists the runs that start in its tile;
// each thread finds the end of its runs by a search over the sorted keys and
// sorts those of at most kFixLocal members itself (so the dependent loads of
// all short runs are in flight together); then the block sorts the longer
// runs one after the other.  A long run may extend over later tiles: no
// other run starts inside it, so no other block touches its positions.
template <typename R>
__global__ void __launch_bounds__(kFixThreads)
tie_fixup_kernel(const uint32_t* key, const Vec4<R>* posm,
                 uint32_t* val, uint32_t* tmp, int64_t N,
                 unsigned* err) {
    __shared__ uint32_t s_key[kFixTile + 2];
    __shared__ int s_runs[kFixTile / 2];
    __shared__ int s_nruns, s_nlong;
    __shared__ int64_t s_long_s[kFixLongMax], s_long_n[kFixLongMax];
    // the long-run sort's counters reuse the staged keys and the run list
    // (both dead by then)
    static_assert(sizeof(uint32_t) * (kFixThreads / 32) * 256 <= sizeof(s_key), "counters");
    static_assert(sizeof(uint32_t) * (256 + kFixThreads / 32) <= sizeof(s_runs), "offsets");
    auto s_cnt = reinterpret_cast<uint32_t (*)[256]>(s_key);
    uint32_t* s_off = reinterpret_cast<uint32_t*>(s_runs);
    uint32_t* s_wsum = s_off + 256;
    const int64_t base = (int64_t)blockIdx.x * kFixTile;
    const int64_t rem = N - base;
    const int nt = (int)(rem < kFixTile ? rem : kFixTile);
    if (threadIdx.x == 0) { s_nruns = 0; s_nlong = 0; }
    pdl_wait();
    // s_key[i + 1] = key[base + i] for i in [-1, nt]; sentinels outside [0, N)
    for (int i = threadIdx.x - 1; i <= nt; i += kFixThreads) {
        const int64_t g = base + i;
        uint32_t v;
        if (g < 0) v = key[0] ^ 1u;             // differs from key[0]
        else if (g >= N) v = key[N - 1] ^ 1u;   // differs from key[N-1]
        else v = key[g];
        s_key[i + 1] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nt; i += kFixThreads) {
        const uint32_t k = s_key[i + 1];
        if (s_key[i] != k && s_key[i + 2] == k) s_runs[atomicAdd(&s_nruns, 1)] = i;
    }
    __syncthreads();
    const int nruns = s_nruns;   // at most kFixTile / 2 (each run has >= 2 members)
    for (int r = threadIdx.x; r < nruns; r += kFixThreads) {
        const int64_t s = base + s_runs[r];
        const uint32_t k = s_key[s_runs[r] + 1];
        // last member: the keys are sorted, so it is the last position
        // holding k.  A run that ends inside the tile is found by bisection
        // over the staged keys (s_key[j + 1] is the key of local index j);
        // only a run that reaches the tile's end continues with doubling
        // steps and bisection over the keys in global memory.
        int64_t lo;
        if (s_key[nt] != k) {
            int a = s_runs[r] + 1, b = nt - 1;   // key(a) == k, key(b) != k
            while (b - a > 1) {
                const int mid = a + (b - a) / 2;
                if (s_key[mid + 1] == k) a = mid;
                else b = mid;
            }
            lo = base + a;
        } else if (s_key[nt + 1] != k) {
            lo = base + nt - 1;
        } else {
            lo = base + nt;                       // key[lo] == k
            int64_t hi = N, step = 1;
            for (;;) {
                const int64_t probe = lo + step;
                if (probe >= N || key[probe] != k) { hi = probe < N ? probe : N; break; }
                lo = probe;
                step <<= 1;
            }
            while (hi - lo > 1) {
                const int64_t mid = lo + (hi - lo) / 2;
                if (key[mid] == k) lo = mid;
                else hi = mid;
            }
        }
        const int64_t len = lo - s + 1;
        if (len <= kFixLocal) {
            sort_run_local<R>(posm, N, val, s, (int)len);
        } else {
            // sorted keys: long runs starting here do not overlap, so there
            // are fewer than kFixLongMax; unsorted keys (only after a
            // timed-out radix pass) can claim more, and those runs stay as
            // they are
            const int slot = atomicAdd(&s_nlong, 1);
            if (slot < kFixLongMax) {
                s_long_s[slot] = s;
                s_long_n[slot] = len;
            } else {
                report(err, ETICS_ERR_TIMEOUT);
            }
        }
    }
    __syncthreads();   // s_key and s_runs are dead from here
    const int nlong = s_nlong < kFixLongMax ? s_nlong : kFixLongMax;
    for (int r = 0; r < nlong; ++r)
        sort_run_block<R>(posm, N, val, tmp, s_long_s[r], s_long_n[r], s_cnt, s_off, s_wsum);
}

// the particles in radial order (radix path; an index >= N, only after a
// timed-out sort, gives a massless particle at the origin, as does a
// non-finite one, which is reported)
template <typename R>
__device__ __forceinline__ Vec4<R> gather_particle(const Vec4<R>* posm, uint32_t i, int64_t N,
                                                   unsigned* err) {
    Vec4<R> v = mk4<R>(R(0), R(0), R(0), R(0));
    if ((int64_t)i < N) {
        v = ld4(posm + i);
        if (!finite4(v.x, v.y, v.z, v.w)) {
            report(err, ETICS_ERR_NONFINITE);
            v = mk4<R>(R(0), R(0), R(0), R(0));
        }
    }
    return v;
}

template <typename R>
__global__ void __launch_bounds__(256)
gather_kernel(const Vec4<R>* posm, const uint32_t* perm, int64_t N,
              Vec4<R>* sorted, unsigned* err) {
    pdl_wait();   // the order comes from the kernel before
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) st4(sorted + i, gather_particle<R>(posm, ld_cg(perm + i), N, err));
}

// ---------------------------------------------------------------------------
// sample sort
// ---------------------------------------------------------------------------
// the whole FP64 bit pattern of r^2; a non-finite particle sorts last
__device__ __forceinline__ uint64_t r2_bits(const float4& v) {
    uint64_t b;
    if (!finite4(v.x, v.y, v.z, v.w)) return ~uint64_t(0);
    if (!r2_bits_from_f32(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), b))
        b = (uint64_t)__double_as_longlong(r2_fp64((double)v.x, (double)v.y, (double)v.z));
    return b;
}
__device__ __forceinline__ uint64_t r2_bits(const dvec4& v) {
    if (!finite4(v.x, v.y, v.z, v.w)) return ~uint64_t(0);
    return (uint64_t)__double_as_longlong(r2_fp64(v.x, v.y, v.z));
}

// Bucket sizes: a bucket's mean is a third of what a block sorts in shared
// memory.  With kOversample random samples per bucket a bucket three times the
// mean has a probability below 1e-7 (the sum of sixteen exponential spacings);
// it is sorted all the same, by the slower sort_bucket_global.
constexpr int kOversample = 16;
constexpr int kMaxBuckets = 1024;
constexpr int kPartThreads = 1024;          // one thread per bucket
constexpr int kPartTiles = 151;             // one block per SM on a 152-SM part, less one
constexpr int kBucketKpt = 12;              // members per thread at capacity
constexpr int kSmallThreads = 256, kLargeThreads = 512;
constexpr int kSmallMean = 1024, kLargeMean = 2048;
static_assert(3 * kSmallMean == kSmallThreads * kBucketKpt && 3 * kLargeMean == kLargeThreads * kBucketKpt,
              "a bucket's capacity is three times its mean");
// One block, no partition, up to kSingleMax: MEX (l_max 4) takes 31.9 us at 6000
// particles and 36.8 at 8192 so, 35.0 and 33.9 with a partition.
constexpr int kSingleMax = 7168, kSingleKpt = kSingleMax / kLargeThreads;

// How many buckets, of which mean, and how many particles per thread of the
// partition.  Above kSampleMaxN: the radix path.  The line lies where the large
// buckets, two blocks per SM, start a fourth round on 152 SMs: MEX (l_max 4)
// takes 195 us at 1.8 million particles and 256 at 2.0 million with buckets, 228
// and 244 with the radix passes (2^20: 118 and 138).
constexpr int64_t kSampleMaxN = int64_t(912) * kLargeMean;
static_assert(kSampleMaxN <= int64_t(kMaxBuckets) * kLargeMean, "buckets");
constexpr int kMaxTiles = (int)((kSampleMaxN + 8 * kPartThreads - 1) / (8 * kPartThreads));
static_assert(kMaxTiles >= kPartTiles, "tiles");
struct SamplePlan { int nbuckets, mean, kpt, ntiles; };
SamplePlan sample_plan(int64_t N) {
    SamplePlan p{};
    if (N > kSampleMaxN) return p;
    p.mean = N <= int64_t(kMaxBuckets) * kSmallMean ? kSmallMean : kLargeMean;
    p.nbuckets = N <= kSingleMax ? 1 : (int)((N + p.mean - 1) / p.mean);
    // as few particles per thread as let the tiles and the block with the table
    // run at once, one block per SM (at 2^20 147 tiles of 7168 instead of 128
    // of 8192)
    p.kpt = (int)std::min<int64_t>(8, (N + int64_t(kPartTiles) * kPartThreads - 1) /
                                          (int64_t(kPartTiles) * kPartThreads));
    if (p.kpt < 1) p.kpt = 1;
    p.ntiles = (int)((N + (int64_t)kPartThreads * p.kpt - 1) / ((int64_t)kPartThreads * p.kpt));
    return p;
}

// Sorts n <= TH KPT pairs (32-bit key, id) of a block, thread t holding the
// pairs t, t + TH, ... in k[], id[]: each key is mapped linearly from the
// block's key range to one of 8 TH bins, the bins are counted and scanned, and
// the pairs placed in bin order in s_key / s_id; within a bin (half a pair on
// average at a bucket's mean size) the caller counts the smaller keys.
// Equal keys are told apart by the caller.
constexpr int kBinLimit = 48;
template <int TH, int KPT>
struct BlockSort {
    static constexpr int CAP = TH * KPT, NB = 8 * TH;
    // keys, ids, bins, and a 16-bit list; s_low (bitonic() only) lies over the
    // last two
    static constexpr size_t kSmem = (size_t)CAP * 10 + (size_t)NB * 4;
    static_assert((size_t)CAP * 4 <= (size_t)CAP * 2 + (size_t)NB * 4, "room for the low words");
    uint32_t *s_key, *s_id, *s_low, *s_bin;
    uint16_t* s_list;
    uint32_t kmin, mult;
    int n;
    bool crowded;   // a bin holds more than kBinLimit pairs

    __device__ __forceinline__ explicit BlockSort(unsigned char* smem)
        : s_key(reinterpret_cast<uint32_t*>(smem)), s_id(s_key + CAP), s_low(s_id + CAP),
          s_bin(s_id + CAP), s_list(reinterpret_cast<uint16_t*>(s_bin + NB)) {}

    __device__ __forceinline__ int bin_of(uint32_t key) const {
        return (int)(mult ? __umulhi(key - kmin, mult) : key - kmin);
    }

    __device__ __forceinline__ void place(const uint32_t (&k)[KPT], const uint32_t (&id)[KPT],
                                          int count) {
        __shared__ uint32_t s_lo, s_hi, s_sum[32];
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        n = count;
        if (tid == 0) { s_lo = 0xffffffffu; s_hi = 0u; }
        uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
        for (int s = 0; s < KPT; ++s)
            if (tid + s * TH < n) {
                lo = k[s] < lo ? k[s] : lo;
                hi = k[s] > hi ? k[s] : hi;
            }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        uint4* bins4 = reinterpret_cast<uint4*>(s_bin);
        bins4[tid] = make_uint4(0, 0, 0, 0);
        bins4[tid + TH] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        if (lane == 0) {
            atomicMin(&s_lo, lo);
            atomicMax(&s_hi, hi);
        }
        __syncthreads();
        // (key - lo) NB / (range + 1); a range below NB is its own bin number
        kmin = s_lo;
        const uint32_t range = s_hi - kmin;
        mult = range < (uint32_t)NB ? 0u : (uint32_t)(((uint64_t)NB << 32) / ((uint64_t)range + 1));
        uint32_t at[KPT];   // bin, then rank within it (16 bits each)
#pragma unroll
        for (int s = 0; s < KPT; ++s)
            if (tid + s * TH < n) {
                const int b = bin_of(k[s]);
                at[s] = (uint32_t)b | (atomicAdd(&s_bin[b], 1u) << 16);
            }
        __syncthreads();
        // exclusive scan of the bins, eight neighbouring ones per thread
        uint4 c0 = bins4[2 * tid], c1 = bins4[2 * tid + 1];
        const uint32_t most = max(max(max(c0.x, c0.y), max(c0.z, c0.w)),
                                  max(max(c1.x, c1.y), max(c1.z, c1.w)));
        const uint32_t h0 = c0.x + c0.y + c0.z + c0.w, sum = h0 + c1.x + c1.y + c1.z + c1.w;
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += t;
        }
        if (lane == 31) s_sum[warp] = x;
        crowded = __syncthreads_or(most > (uint32_t)kBinLimit);
        uint32_t at0 = x - sum + __reduce_add_sync(0xffffffffu, lane < warp ? s_sum[lane] : 0u);
        bins4[2 * tid] = make_uint4(at0, at0 + c0.x, at0 + c0.x + c0.y, at0 + c0.x + c0.y + c0.z);
        at0 += h0;
        bins4[2 * tid + 1] = make_uint4(at0, at0 + c1.x, at0 + c1.x + c1.y, at0 + c1.x + c1.y + c1.z);
        __syncthreads();
#pragma unroll
        for (int s = 0; s < KPT; ++s)
            if (tid + s * TH < n) {
                const uint32_t pos = s_bin[at[s] & 0xffffu] + (at[s] >> 16);
                s_key[pos] = k[s];
                s_id[pos] = id[s];
            }
        __syncthreads();
    }

    // the pairs [0, n) sorted by (key, s_low, id): where keys crowd, a network
    // (of a power of two of places, those from n on taken as infinite: a pair
    // with one of them is never exchanged, as the larger value always belongs
    // to the upper place in the form used, first step mirrored)
    __device__ __noinline__ void bitonic() {
        int p2 = 2;
        while (p2 < n) p2 <<= 1;
        __syncthreads();
        for (int k = 2; k <= p2; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = threadIdx.x; t < p2 / 2; t += TH) {
                    const int i = 2 * t - (t & (j - 1));
                    const int l = j == (k >> 1) ? (i ^ (k - 1)) : i + j;
                    if (l >= n) continue;
                    const uint32_t a = s_key[i], b = s_key[l], la = s_low[i], lb = s_low[l],
                                   ia = s_id[i], ib = s_id[l];
                    const bool after = a > b || (a == b && (la > lb || (la == lb && ia > ib)));
                    if (after) {
                        s_key[i] = b; s_key[l] = a;
                        s_low[i] = lb; s_low[l] = la;
                        s_id[i] = ib; s_id[l] = ia;
                    }
                }
                __syncthreads();
            }
    }

    // bounds of the bin of the pair at p
    __device__ __forceinline__ void bin_range(uint32_t key, int& s, int& e) const {
        const int b = bin_of(key);
        s = (int)s_bin[b];
        e = b + 1 < NB ? (int)s_bin[b + 1] : n;
    }
};

__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x = (x ^ (x >> 16)) * 0x45d9f3bu;
    x = (x ^ (x >> 16)) * 0x45d9f3bu;
    return x ^ (x >> 16);
}

// the 32-bit key of a particle (r2_key); non-finite ones come last
template <typename R>
__device__ __forceinline__ uint32_t sort_key(const Vec4<R>& v) {
    return finite4(v.x, v.y, v.z, v.w) ? r2_key(v.x, v.y, v.z) : 0xffffffffu;
}

// The cumulative distribution of the keys, from a sample of kOversample
// nbuckets particles: one at a random place of each of as many equal stretches
// of the array (a regular stride could fall in step with an order of the
// particles).  kCdfBins bins of equal width over the sample's key range hold
// the number of samples below them; a bin with more than kCdfCrowd samples is
// divided once more into 256 (kCdfFine of them at most).  Within a bin the
// distribution is taken as linear, so that a key's bucket comes from two table
// entries instead of a search among splitters (the binary search cost 12 us at
// 2^20, sorting the sample for splitters another 8).  How good the table is
// only decides how even the buckets are.
constexpr int kCdfBins = 8192, kCdfCrowd = 32, kCdfFine = 64, kCdfFineRow = 264;
struct KeyCdf {                      // 16-byte pieces, copied to shared memory as a whole
    uint32_t kmin, range, mult, nfine;
    uint16_t below[kCdfBins + 8];    // samples below bin b; [kCdfBins]: all of them
    uint8_t fine[kCdfBins];          // row of a divided bin, 255: none
    uint16_t row[kCdfFine][kCdfFineRow];   // samples of the bin below its part
};
static_assert(sizeof(KeyCdf) % 16 == 0 && kOversample * kMaxBuckets < 65536, "table layout");

__device__ __forceinline__ int bucket_of(const KeyCdf& t, uint32_t key, int nbuckets) {
    if (key < t.kmin) return 0;
    if (key - t.kmin > t.range) return nbuckets - 1;
    // bin and place in it (32-bit fraction); mult 0: a bin per key
    const uint64_t p = t.mult ? (uint64_t)(key - t.kmin) * t.mult : (uint64_t)(key - t.kmin) << 32;
    const int b = (int)(p >> 32);
    uint32_t frac = (uint32_t)p, lo = t.below[b], hi = t.below[b + 1];
    if (hi - lo > (uint32_t)kCdfCrowd && t.fine[b] != 255) {
        const uint16_t* r = t.row[t.fine[b]] + (frac >> 24);
        frac <<= 8;
        hi = lo + r[1];
        lo += r[0];
    }
    // in sixteenths of a sample
    const uint32_t c = lo * 16u + (((hi - lo) * (frac >> 16)) >> 12);
    const int k = (int)(c / (16u * kOversample));
    return k < nbuckets ? k : nbuckets - 1;
}

// one block; scratch: (kCdfBins + kCdfFine 256) words of shared memory.
// stride: N / (number of samples), 32.32 fixed point.
constexpr size_t kCdfSmem = ((size_t)kCdfBins + (size_t)kCdfFine * 256) * 4;
static_assert(kCdfSmem >= sizeof(KeyCdf), "the tiles copy the table there");
template <typename R>
__device__ __forceinline__ void make_cdf(const Vec4<R>* posm, int64_t N, int nbuckets,
                                         uint64_t stride, KeyCdf* out, uint32_t* scratch) {
    constexpr int TH = kPartThreads, KPT = kOversample * kMaxBuckets / TH;
    static_assert(kCdfBins == 8 * TH, "eight bins per thread");
    __shared__ uint32_t s_lo, s_hi, s_nfine, s_sum[32];
    uint32_t *s_bin = scratch, *s_part = scratch + kCdfBins;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ns = kOversample * nbuckets;
    uint4* bins4 = reinterpret_cast<uint4*>(s_bin);
    bins4[tid] = bins4[tid + TH] = make_uint4(0, 0, 0, 0);
    if (tid == 0) { s_lo = 0xffffffffu; s_hi = 0u; s_nfine = 0u; }
    uint32_t k[KPT], lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
        const uint32_t i = (uint32_t)(tid + s * TH);
        if ((int)i < ns) {
            const int64_t a = (int64_t)((i * stride) >> 32);
            int64_t b = (int64_t)(((i + 1) * stride) >> 32);
            if (b <= a) b = a + 1;
            const int64_t g = a + (int64_t)__umulhi(mix32(i + 1), (uint32_t)(b - a));
            k[s] = sort_key<R>(ld4(posm + (g < N ? g : N - 1)));
            lo = k[s] < lo ? k[s] : lo;
            hi = k[s] > hi ? k[s] : hi;
        }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    __syncthreads();
    if (lane == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
    }
    __syncthreads();
    const uint32_t kmin = s_lo, range = s_hi - kmin;
    const uint32_t mult = range < (uint32_t)kCdfBins
                              ? 0u : (uint32_t)(((uint64_t)kCdfBins << 32) / ((uint64_t)range + 1));
    auto place = [&](uint32_t key) {
        return mult ? (uint64_t)(key - kmin) * mult : (uint64_t)(key - kmin) << 32;
    };
#pragma unroll
    for (int s = 0; s < KPT; ++s)
        if (tid + s * TH < ns) atomicAdd(&s_bin[(uint32_t)(place(k[s]) >> 32)], 1u);
    __syncthreads();
    // this thread's eight bins: rows for the crowded ones, counts to sums
    uint32_t c[8];
    *reinterpret_cast<uint4*>(c) = bins4[2 * tid];
    *reinterpret_cast<uint4*>(c + 4) = bins4[2 * tid + 1];
    uint32_t rows[2] = {0u, 0u}, sum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        uint32_t r = 255u;
        if (c[j] > (uint32_t)kCdfCrowd) {
            r = atomicAdd(&s_nfine, 1u);
            if (r >= (uint32_t)kCdfFine) r = 255u;
        }
        rows[j / 4] |= r << (8 * (j % 4));
        const uint32_t v = c[j];
        c[j] = sum;
        sum += v;
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) s_sum[warp] = x;
    for (int i = tid; i < kCdfFine * 256; i += TH) s_part[i] = 0u;
    __syncthreads();
    const uint32_t before = x - sum + __reduce_add_sync(0xffffffffu, lane < warp ? s_sum[lane] : 0u);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        out->below[8 * tid + j] = (uint16_t)(before + c[j]);
        // the bin's row for the second count, in place of its count
        s_bin[8 * tid + j] = (rows[j / 4] >> (8 * (j % 4))) & 255u;
    }
    *reinterpret_cast<uint2*>(out->fine + 8 * tid) = make_uint2(rows[0], rows[1]);
    const int nfine = min((int)s_nfine, kCdfFine);
    if (tid == 0) {
        out->below[kCdfBins] = (uint16_t)ns;
        out->kmin = kmin;
        out->range = range;
        out->mult = mult;
        out->nfine = (uint32_t)nfine;
    }
    __syncthreads();
    if (nfine == 0) return;
#pragma unroll
    for (int s = 0; s < KPT; ++s)
        if (tid + s * TH < ns) {
            const uint64_t p = place(k[s]);
            const uint32_t r = s_bin[(uint32_t)(p >> 32)];
            if (r != 255u) atomicAdd(&s_part[r * 256u + ((uint32_t)p >> 24)], 1u);
        }
    __syncthreads();
    for (int r = warp; r < nfine; r += TH / 32) {
        uint32_t v[8], t = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            v[j] = t;
            t += s_part[r * 256 + 8 * lane + j];
        }
        uint32_t y = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += u;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) out->row[r][8 * lane + j] = (uint16_t)(y - t + v[j]);
        if (lane == 31) out->row[r][256] = (uint16_t)y;
    }
}

// Partition.  Blocks take tickets; the block with the first one makes the
// table and raises the flag, the others load their tile's particles and
// evaluate the keys meanwhile and wait for it (bounded; the tickets' order
// makes sure that the block waited for has started).  A tile then counts its
// particles per bucket in shared memory, takes its places in the buckets with
// one addition per bucket to the bucket sizes, and writes the particles' keys
// and indices to region[b * cap + place].  The order inside a bucket's region is
// whatever the additions give: the bucket sort orders by (r^2, index).  A tile's
// particles beyond a bucket's capacity go to a run of places of their own in
// `spill`, runs[tile][bucket] = (first place, count), so that a crowded bucket is
// collected in time proportional to its size.  A tile whose wait runs out
// (ETICS_ERR_TIMEOUT) counts its particles in bucket 0: the sizes still add up
// to N, so that everything after stays inside the buffers.
// part (zero at launch): [0] ticket counter, [1] flag, [2] places of `spill`
// taken, from word kPartHeader on the bucket sizes.
constexpr int kPartHeader = 64;
template <typename R, int KPT>
__global__ void __launch_bounds__(kPartThreads, 1)
partition_kernel(const Vec4<R>* posm, int64_t N, int nbuckets, int cap,
                 uint64_t stride, KeyCdf* cdf, uint32_t* part, uint2* region, uint32_t* spill,
                 uint2* runs, int64_t spin_limit, unsigned* err) {
    extern __shared__ __align__(16) unsigned char sort_smem[];
    __shared__ uint32_t s_hist[kMaxBuckets], s_spill[kMaxBuckets];
    __shared__ uint32_t s_ticket;
    __shared__ int s_ok;
    const int tid = threadIdx.x;
    s_hist[tid] = 0u;
    pdl_wait();
    if (tid == 0) s_ticket = atomicAdd(part, 1u);
    __syncthreads();
    if (s_ticket == 0u) {
        make_cdf<R>(posm, N, nbuckets, stride, cdf, reinterpret_cast<uint32_t*>(sort_smem));
        __threadfence();
        __syncthreads();
        if (tid == 0) st_volatile(part + 1, 1u);
        return;
    }
    const int64_t start = (int64_t)(s_ticket - 1u) * kPartThreads * KPT;
    Vec4<R> v[KPT];
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
        const int64_t i = start + s * kPartThreads + tid;
        if (i < N) v[s] = ld4(posm + i);
    }
    uint32_t key[KPT];
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
        key[s] = 0u;
        if (start + s * kPartThreads + tid < N) {
            key[s] = sort_key<R>(v[s]);
            if (key[s] == 0xffffffffu) report(err, ETICS_ERR_NONFINITE);
        }
    }
    if (tid == 0) {
        int64_t spins = 0;
        int ok = 1;
        while (ld_volatile(part + 1) == 0u) {
            if (++spins > spin_limit) { ok = 0; break; }
            __nanosleep(32);
        }
        if (!ok) report(err, ETICS_ERR_TIMEOUT);
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    const bool ok = s_ok;
    KeyCdf& t = *reinterpret_cast<KeyCdf*>(sort_smem);
    if (ok) {
        // without the rows of divided bins that are not there
        const uint32_t nfine = ld_cg(&cdf->nfine);
        const int pieces = (int)((offsetof(KeyCdf, row) + nfine * sizeof(t.row[0])) / 16);
        for (int i = tid; i < pieces; i += kPartThreads)
            reinterpret_cast<uint4*>(&t)[i] = ld_cg(reinterpret_cast<const uint4*>(cdf) + i);
    }
    __syncthreads();
    uint32_t at[KPT];   // bucket, then place within the tile's share (16 bits each)
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
        at[s] = 0u;
        if (start + s * kPartThreads + tid < N) {
            const int b = ok ? bucket_of(t, key[s], nbuckets) : 0;
            at[s] = (uint32_t)b | (atomicAdd(&s_hist[b], 1u) << 16);
        }
    }
    __syncthreads();
    if (tid < nbuckets) {
        const uint32_t count = s_hist[tid], room = (uint32_t)cap;
        const uint32_t first = count ? atomicAdd(part + kPartHeader + tid, count) : 0u;
        const uint32_t from = first > room ? first : room;   // first place beyond the capacity
        const uint32_t over = first + count > from ? first + count - from : 0u;
        const uint32_t place = over ? atomicAdd(part + 2, over) : 0u;
        s_hist[tid] = first;
        s_spill[tid] = place - from;
        runs[(size_t)(s_ticket - 1u) * nbuckets + tid] = make_uint2(place, over);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
        const int64_t i = start + s * kPartThreads + tid;
        if (i < N) {
            const uint32_t b = at[s] & 0xffffu, slot = s_hist[b] + (at[s] >> 16);
            if (slot < (uint32_t)cap) region[(size_t)b * cap + slot] = make_uint2(key[s], (uint32_t)i);
            else spill[s_spill[b] + slot] = (uint32_t)i;
        }
    }
}

// A bucket larger than a block's shared memory (keys that crowd on one high
// word, or, rarely, an unlucky sample): the block collects its members, `mem`
// holding the first `cap` and `spill` the rest in one run per tile (runs: this
// bucket's of tile 0, `stride` further that of the next), and sorts them by
// (64-bit pattern of r^2, index) with stable 8-bit passes between val and tmp,
// kCrowdKpt members per thread at a time; passes over a digit that is the same
// for all are left out.  The order of 2^20 particles on 300 thin shells takes
// 430 us (5.5 ms when each such bucket's block read all particles again, 86
// for a Hernquist sphere); 1.87 million on 1 / 100 / 300 / 1000 shells 31.7 ms
// / 660 / 530 / 450 us, by the radix path 60.6 ms / 1260 / 870 / 490.
constexpr int kCrowdKpt = 8;
template <typename R, int TH>
__device__ __noinline__ void sort_bucket_global(const Vec4<R>* posm, int64_t N, const uint2* mem,
                                                int cap, const uint32_t* spill, const uint2* runs,
                                                int ntiles, int stride, uint32_t* val, uint32_t* tmp,
                                                int64_t len, uint32_t* scratch) {
    constexpr int NW = TH / 32;
    uint32_t (*s_cnt)[256] = reinterpret_cast<uint32_t (*)[256]>(scratch);   // [NW][256]
    __shared__ uint32_t s_wsum[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // exclusive sum of x over the threads
    auto scan = [&](uint32_t x) -> uint32_t {
        uint32_t y = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += t;
        }
        __syncthreads();
        if (lane == 31) s_wsum[warp] = y;
        __syncthreads();
        return y - x + __reduce_add_sync(0xffffffffu, lane < warp ? s_wsum[lane] : 0u);
    };
    for (int i = tid; i < cap; i += TH) val[i] = ld_cg(mem + i).y;
    // the runs, a warp each (their places in s_cnt, dead here)
    uint32_t *s_at = scratch, *s_first = scratch + TH, *s_n = scratch + 2 * TH;
    static_assert(3 * TH <= NW * 256, "room for the runs");
    int64_t have = cap;
    for (int t0 = 0; t0 < ntiles; t0 += TH) {
        const uint2 r = t0 + tid < ntiles ? ld_cg(runs + (size_t)(t0 + tid) * stride) : make_uint2(0u, 0u);
        const uint32_t first = scan(r.y);
        s_at[tid] = r.x;
        s_first[tid] = first;
        s_n[tid] = r.y;
        __syncthreads();
        for (int q = warp; q < TH; q += NW)
            for (uint32_t j = lane; j < s_n[q]; j += 32) {
                const int64_t pos = have + s_first[q] + j;
                if (pos < len) val[pos] = ld_cg(spill + s_at[q] + j);
            }
        have += s_first[TH - 1] + s_n[TH - 1];
    }
    // the digits of (index, pattern) counted for all passes in one look
    constexpr int kDigits = 12;   // 0..3 of the index, 4..11 of the pattern
    uint32_t (*s_off)[256] = reinterpret_cast<uint32_t (*)[256]>(scratch + NW * 256);
    auto bits = [&](uint32_t i) -> uint64_t {
        return (int64_t)i < N ? r2_bits(ld4(posm + i)) : ~uint64_t(0);
    };
    for (int i = tid; i < kDigits * 256; i += TH) (&s_off[0][0])[i] = 0u;
    __syncthreads();
#pragma unroll 2
    for (int64_t i = tid; i < len; i += TH) {
        const uint32_t v = val[i];
        const uint64_t w = bits(v);
#pragma unroll
        for (int p = 0; p < kDigits; ++p)
            atomicAdd(&s_off[p][(p < 4 ? v >> 8 * p : (uint32_t)(w >> 8 * (p - 4 & 7))) & 255u], 1u);
    }
    __syncthreads();
    uint32_t *src = val, *dst = tmp;
    for (int pass = 0; pass < kDigits; ++pass) {
        const uint32_t count = tid < 256 ? s_off[pass][tid] : 0u;
        if (__syncthreads_or((int64_t)count == len)) continue;   // one digit only
        const uint32_t start = scan(count);
        if (tid < 256) s_off[pass][tid] = start;
        for (int64_t c0 = 0; c0 < len; c0 += TH * kCrowdKpt) {
            for (int i = tid; i < NW * 256; i += TH) (&s_cnt[0][0])[i] = 0u;
            __syncthreads();
            uint32_t v[kCrowdKpt], d[kCrowdKpt], rank[kCrowdKpt];
#pragma unroll
            for (int s = 0; s < kCrowdKpt; ++s) {
                const int64_t i = c0 + (int64_t)warp * kCrowdKpt * 32 + s * 32 + lane;
                v[s] = i < len ? src[i] : 0u;
            }
#pragma unroll
            for (int s = 0; s < kCrowdKpt; ++s) {
                const int64_t i = c0 + (int64_t)warp * kCrowdKpt * 32 + s * 32 + lane;
                d[s] = 256u;
                if (i < len)
                    d[s] = (pass < 4 ? v[s] >> 8 * pass : (uint32_t)(bits(v[s]) >> 8 * (pass - 4))) & 255u;
            }
            rank_in_warp<false>(d, rank, s_cnt[warp], lane);
            __syncthreads();
            if (tid < 256) {   // thread = digit: where each warp's members go
                uint32_t at = s_off[pass][tid];
                for (int w = 0; w < NW; ++w) {
                    const uint32_t t = s_cnt[w][tid];
                    s_cnt[w][tid] = at;
                    at += t;
                }
                s_off[pass][tid] = at;
            }
            __syncthreads();
#pragma unroll
            for (int s = 0; s < kCrowdKpt; ++s)
                if (d[s] < 256u) dst[s_cnt[warp][d[s]] + rank[s]] = v[s];
            __syncthreads();
        }
        uint32_t* t = src;
        src = dst;
        dst = t;
    }
    if (src != val) {
        for (int64_t i = tid; i < len; i += TH) val[i] = src[i];
    }
    __syncthreads();
}

// One block per bucket: its place in the order from the bucket sizes, the sort
// of its members by (64-bit pattern of r^2, index), the order and (sorted not
// null) the particles.  nbuckets == 1: the particles 0..N-1 themselves (at
// most TH KPT), no partition before.
// The members are sorted by the high word of the pattern (the cheap 32-bit
// key); the low word is evaluated only for members that share their high word
// with another one (a few in a hundred), listed first so that whole warps do
// it.  Latency-bound: a chain of loads and block-wide steps, about 12 us per
// block whatever its size, hidden only by other blocks.
template <typename R, int TH, int KPT>
__global__ void __launch_bounds__(TH, 1024 / TH)   // 64 registers
bucket_sort_kernel(const Vec4<R>* posm, int64_t N, int nbuckets, int ntiles, const uint32_t* sizes,
                   const uint2* region, const uint32_t* spill, const uint2* runs, uint32_t* perm,
                   uint32_t* tmp, Vec4<R>* sorted, unsigned* err) {
    extern __shared__ __align__(16) unsigned char sort_smem[];
    using Sort = BlockSort<TH, KPT>;
    constexpr int CAP = Sort::CAP;
    constexpr int kAhead = 5;   // members per thread loaded before the size is known
    __shared__ uint32_t s_base[TH / 32];
    __shared__ int s_ntie;
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
    int64_t base = 0, len = N;
    if (tid == 0) s_ntie = 0;
    uint32_t k[KPT], id[KPT];
    if (nbuckets > 1) {
        const uint2* mem = region + (size_t)b * CAP + tid;
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
            const uint2 m = ld_cg(mem + s * TH);
            k[s] = m.x;
            id[s] = m.y;
        }
        uint32_t before = 0;
        for (int i = tid; i < b; i += TH) before += ld_cg(sizes + i);
        len = ld_cg(sizes + b);
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0) s_base[warp] = before;
        __syncthreads();
        base = __reduce_add_sync(0xffffffffu, lane < TH / 32 ? s_base[lane] : 0u);
        if (base > N) base = N;   // (the sizes add up to N)
        if (base + len > N) len = N - base;
        if (len == 0) return;
        if (len > CAP) {
            sort_bucket_global<R, TH>(posm, N, region + (size_t)b * CAP, CAP, spill, runs + b, ntiles,
                                      nbuckets, perm + base, tmp + base, len,
                                      reinterpret_cast<uint32_t*>(sort_smem));
            if (sorted)
                for (int64_t i = tid; i < len; i += TH)
                    st4(sorted + base + i, gather_particle<R>(posm, perm[base + i], N, err));
            return;
        }
#pragma unroll
        for (int s = kAhead; s < KPT; ++s)
            if (tid + s * TH < (int)len) {
                const uint2 m = ld_cg(mem + s * TH);
                k[s] = m.x;
                id[s] = m.y;
            }
    } else {
#pragma unroll
        for (int s = 0; s < KPT; ++s) {
            const int i = tid + s * TH;
            if (i < (int)len) {
                k[s] = sort_key<R>(ld4(posm + i));
                if (k[s] == 0xffffffffu) report(err, ETICS_ERR_NONFINITE);
                id[s] = (uint32_t)i;
            }
        }
    }
    const int n = (int)len;
    Sort sort(sort_smem);
    sort.place(k, id, n);
    auto low_word = [&](uint32_t i) -> uint32_t {
        return (int64_t)i < N ? (uint32_t)r2_bits(ld4(posm + i)) : 0xffffffffu;
    };
    auto put = [&](int r, uint32_t i) {
        perm[base + r] = i;
        if (sorted) st4(sorted + base + r, gather_particle<R>(posm, i, N, err));
    };
    // a pair's place is the start of its bin plus the smaller ones in it; those
    // with an equal key in the bin go to the list and are placed by (key, low
    // word, index).  Where keys crowd in one bin, or a quarter of the members
    // share their key (comparing those in pairs would be quadratic), the
    // network sorts them all.
    bool net = sort.crowded;
    if (!net) {
        for (int p = tid; p < n; p += TH) {
            const uint32_t key = sort.s_key[p];
            int s, e;
            sort.bin_range(key, s, e);
            int r = s, same = 0;
            for (int j = s; j < e; ++j) {
                r += sort.s_key[j] < key;
                same += sort.s_key[j] == key;
            }
            if (same > 1) sort.s_list[atomicAdd(&s_ntie, 1)] = (uint16_t)p;
            else put(r, sort.s_id[p]);
        }
        __syncthreads();
        net = 4 * s_ntie > n;
    }
    if (net) {
        // (s_low lies over the bins and the list, neither needed any more)
        for (int p = tid; p < n; p += TH) sort.s_low[p] = low_word(sort.s_id[p]);
        sort.bitonic();
        for (int p = tid; p < n; p += TH) put(p, sort.s_id[p]);
        return;
    }
    const int ntie = s_ntie;
    for (int q = tid; q < ntie; q += TH) {
        const int p = sort.s_list[q];
        const uint32_t key = sort.s_key[p], own = sort.s_id[p], low = low_word(own);
        int s, e;
        sort.bin_range(key, s, e);
        int r = s;
        for (int j = s; j < e; ++j) {
            const uint32_t kj = sort.s_key[j];
            if (kj < key) {
                ++r;
            } else if (kj == key && j != p) {
                const uint32_t lj = low_word(sort.s_id[j]);
                r += lj < low || (lj == low && sort.s_id[j] < own);
            }
        }
        put(r, own);
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
SortBuffers sort_buffers(void* ws, int64_t N, size_t* total) {
    SortBuffers b{};
    uint8_t* p = reinterpret_cast<uint8_t*>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        uint8_t* q = p ? p + off : nullptr;
        off += (bytes + 255) / 256 * 256;
        return q;
    };
    const size_t n4 = (size_t)(N > 0 ? N : 1) * 4;
    b.vals_a = reinterpret_cast<uint32_t*>(take(n4));
    b.vals_b = reinterpret_cast<uint32_t*>(take(n4));
    // the two paths' own buffers lie over each other
    const size_t shared = off;
    b.keys_a = reinterpret_cast<uint32_t*>(take(n4));
    b.keys_b = reinterpret_cast<uint32_t*>(take(n4));
    const size_t nst = (size_t)sort_tiles(N);
    b.zero_bytes = (4 * 256 + 4 * (nst + kStatusPad) * 256 + 64) * 4;
    b.zero_bytes = (b.zero_bytes + 255) / 256 * 256;
    uint8_t* z = take(b.zero_bytes);
    b.hist = reinterpret_cast<uint32_t*>(z);
    b.status = b.hist ? b.hist + 4 * 256 : nullptr;
    b.counters = b.status ? b.status + 4 * (nst + kStatusPad) * 256 : nullptr;
    b.zero_base = z;
    const size_t radix_end = off;
    off = shared;
    const SamplePlan sp = sample_plan(N);
    if (sp.nbuckets > 1) {
        b.region = take((size_t)sp.nbuckets * 3 * sp.mean * sizeof(uint2));
        b.cdf = take(sizeof(KeyCdf));
        b.part = reinterpret_cast<uint32_t*>(take((kPartHeader + kMaxBuckets) * 4));
        b.spill = reinterpret_cast<uint32_t*>(take(n4));
        // (bounds of the tiles and buckets that grow with N, as the sizes asked for should)
        const size_t tiles = (size_t)std::min<int64_t>((N + kPartThreads - 1) / kPartThreads, kMaxTiles);
        const size_t buckets = (size_t)std::min<int64_t>((N + kSmallMean - 1) / kSmallMean, kMaxBuckets);
        b.runs = take(tiles * buckets * sizeof(uint2));
    }
    if (radix_end > off) off = radix_end;
    // at least what the largest bucket sort takes: a workspace sized for the
    // largest call serves every smaller one
    size_t least = 0;
    if (total && N > kSampleMaxN) sort_buffers(nullptr, kSampleMaxN, &least);
    if (total) *total = std::max(off, least);
    return b;
}

// dynamic shared memory above 48 KB: allowed once per kernel and device.  The
// carve-out is left alone: a larger one for a third resident block of the
// bucket sort costs its second gather the L1 cache (MEX at 2^20: 158 -> 170 us)
template <typename K>
static int allow_smem(K kernel, std::atomic<uint64_t>& done, size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev)) return ETICS_ERR_CUDA;
    const uint64_t bit = uint64_t(1) << (dev & 63);
    if (done.load() & bit) return ETICS_OK;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes))
        return ETICS_ERR_CUDA;
    done.fetch_or(bit);
    return ETICS_OK;
}

template <typename R, int KPT>
static int launch_partition(const Vec4<R>* pp, int64_t N, const SamplePlan& sp,
                            const SortBuffers& b, const LaunchCtx& ctx) {
    static std::atomic<uint64_t> done{0};
    auto k = partition_kernel<R, KPT>;
    constexpr size_t smem = kCdfSmem;
    if (allow_smem(k, done, smem)) return ETICS_ERR_CUDA;
    if (cudaMemsetAsync(b.part, 0, (kPartHeader + sp.nbuckets) * 4, ctx.stream)) return ETICS_ERR_CUDA;
    const uint64_t stride = ((uint64_t)N << 32) / (uint64_t)(kOversample * sp.nbuckets);
    if (launch_pdl(k, dim3(sp.ntiles + 1), dim3(kPartThreads), smem, ctx.stream, pp, N, sp.nbuckets,
                   3 * sp.mean, stride, reinterpret_cast<KeyCdf*>(b.cdf), b.part,
                   reinterpret_cast<uint2*>(b.region), b.spill, reinterpret_cast<uint2*>(b.runs),
                   ctx.wait_limit > 0 ? ctx.wait_limit : kSpinLimit, ctx.err))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}

// for 1..8 particles per thread
template <typename R, int... I>
static constexpr auto partition_launchers(std::integer_sequence<int, I...>) {
    return std::array<int (*)(const Vec4<R>*, int64_t, const SamplePlan&, const SortBuffers&,
                              const LaunchCtx&), sizeof...(I)>{&launch_partition<R, I + 1>...};
}

template <typename R, int TH, int KPT>
static int launch_buckets(const Vec4<R>* pp, int64_t N, const SamplePlan& sp, const SortBuffers& b,
                          Vec4<R>* sorted, const LaunchCtx& ctx) {
    static std::atomic<uint64_t> done{0};
    constexpr size_t smem = BlockSort<TH, KPT>::kSmem;
    auto k = bucket_sort_kernel<R, TH, KPT>;
    if (allow_smem(k, done, smem)) return ETICS_ERR_CUDA;
    if (launch_pdl(k, dim3(sp.nbuckets), dim3(TH), smem, ctx.stream, pp, N, sp.nbuckets, sp.ntiles,
                   (const uint32_t*)(b.part ? b.part + kPartHeader : nullptr),
                   reinterpret_cast<const uint2*>(b.region), (const uint32_t*)b.spill,
                   reinterpret_cast<const uint2*>(b.runs), b.vals_a, b.vals_b, sorted, ctx.err))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}

template <typename R>
static int sample_sort(const Vec4<R>* pp, int64_t N, const SamplePlan& sp, const SortBuffers& b,
                       Vec4<R>* sorted, const LaunchCtx& ctx) {
    if (sp.nbuckets > 1) {
        static constexpr auto kRun = partition_launchers<R>(std::make_integer_sequence<int, 8>());
        const int rc = kRun[sp.kpt - 1](pp, N, sp, b, ctx);
        if (rc) return rc;
    }
    stage_event(ctx, 1);
    if (sp.nbuckets == 1)
        return launch_buckets<R, kLargeThreads, kSingleKpt>(pp, N, sp, b, sorted, ctx);
    return sp.mean == kSmallMean
               ? launch_buckets<R, kSmallThreads, kBucketKpt>(pp, N, sp, b, sorted, ctx)
               : launch_buckets<R, kLargeThreads, kBucketKpt>(pp, N, sp, b, sorted, ctx);
}

template <typename R>
int radial_sort_impl(const void* posm, int64_t N, const SortBuffers& b, void* sorted,
                     const LaunchCtx& ctx) {
    const Vec4<R>* pp = reinterpret_cast<const Vec4<R>*>(posm);
    Vec4<R>* sp_out = reinterpret_cast<Vec4<R>*>(sorted);
    const SamplePlan sp = sample_plan(N);
    if (sp.nbuckets > 0) return sample_sort<R>(pp, N, sp, b, sp_out, ctx);
    if (cudaMemsetAsync(b.zero_base, 0, b.zero_bytes, ctx.stream)) return ETICS_ERR_CUDA;
    // few, long-lived blocks: each zeroes and merges 8 private histograms
    int kg = (int)((N + 256 * kKeygenIlp - 1) / (256 * kKeygenIlp));
    if (kg > ctx.num_sms * 2) kg = ctx.num_sms * 2;
    keygen_kernel<R><<<kg, 256, 0, ctx.stream>>>(pp, N, b.keys_a, b.hist, ctx.err);
    if (cudaGetLastError()) return ETICS_ERR_CUDA;
    ++*ctx.launches;
    stage_event(ctx, 1);
    const int nst = sort_tiles(N);
    uint32_t *kin = b.keys_a, *vin = b.vals_a, *kout = b.keys_b, *vout = b.vals_b;
    for (int pass = 0; pass < 4; ++pass) {
        const uint32_t* vals_in = pass == 0 ? nullptr : vin;
        // passes 0 and 1 count the histograms of digits 1 and 2
        uint32_t* next_hist = pass < 2 ? b.hist + (pass + 1) * 256 : nullptr;
        if (launch_pdl(onesweep_kernel, dim3(nst), dim3(kSortThreads), 0, ctx.stream, (const uint32_t*)kin,
                       vals_in, kout, vout, (const uint32_t*)(b.hist + pass * 256),
                       b.status + (size_t)pass * (nst + kStatusPad) * 256, b.counters + pass, 8 * pass,
                       N, ctx.wait_limit > 0 ? ctx.wait_limit : kSpinLimit, next_hist, ctx.err))
            return ETICS_ERR_CUDA;
        ++*ctx.launches;
        uint32_t* t = kin; kin = kout; kout = t;
        t = vin; vin = vout; vout = t;
    }
    // after 4 passes the sorted keys/values are back in keys_a / vals_a
    const int fg = (int)((N + kFixTile - 1) / kFixTile);
    if (launch_pdl(tie_fixup_kernel<R>, dim3(fg), dim3(kFixThreads), 0, ctx.stream,
                   (const uint32_t*)b.keys_a, pp, b.vals_a, b.vals_b, N, ctx.err))
        return ETICS_ERR_CUDA;
    ++*ctx.launches;
    if (sp_out) {
        if (launch_pdl(gather_kernel<R>, dim3((unsigned)((N + 255) / 256)), dim3(256), 0, ctx.stream,
                       pp, (const uint32_t*)b.vals_a, N, sp_out, ctx.err))
            return ETICS_ERR_CUDA;
        ++*ctx.launches;
    }
    return ETICS_OK;
}

// One radix pass made to time out: kTimeoutProbeN keys, all 0, so the pass
// histogram has one digit; the tile counter starts at 1, so the single block
// takes tile 1 and looks back at tile 0, which never runs and never
// publishes.  The lookback gives up after `spins` polls, records
// ETICS_ERR_TIMEOUT and writes its tile at positions [0, kSortTile), inside
// the output buffers.
static __global__ void timeout_probe_setup_kernel(uint32_t* hist, uint32_t* counters, uint32_t n) {
    if (threadIdx.x == 0) {
        hist[0] = n;
        counters[0] = 1u;
    }
}

int lookback_timeout_probe(void* ws, int64_t spins, const LaunchCtx& ctx) {
    static_assert(kTimeoutProbeN == 2 * kSortTile, "the probe sorts two tiles");
    const SortBuffers b = sort_buffers(ws, kTimeoutProbeN, nullptr);
    if (cudaMemsetAsync(b.zero_base, 0, b.zero_bytes, ctx.stream) ||
        cudaMemsetAsync(b.keys_a, 0, kTimeoutProbeN * sizeof(uint32_t), ctx.stream))
        return ETICS_ERR_CUDA;
    timeout_probe_setup_kernel<<<1, 32, 0, ctx.stream>>>(b.hist, b.counters,
                                                         (uint32_t)kTimeoutProbeN);
    if (cudaGetLastError()) return ETICS_ERR_CUDA;
    ++*ctx.launches;
    onesweep_kernel<<<1, kSortThreads, 0, ctx.stream>>>(b.keys_a, nullptr, b.keys_b, b.vals_b,
                                                         b.hist, b.status, b.counters, 0,
                                                         kTimeoutProbeN, spins, nullptr, ctx.err);
    if (cudaGetLastError()) return ETICS_ERR_CUDA;
    ++*ctx.launches;
    return ETICS_OK;
}

template int radial_sort_impl<float>(const void*, int64_t, const SortBuffers&, void*,
                                     const LaunchCtx&);
template int radial_sort_impl<double>(const void*, int64_t, const SortBuffers&, void*,
                                      const LaunchCtx&);

}  // namespace etics
