// etics_r2.h -- the FP64 bit pattern of r^2 = (x*x + y*y) + z*z for FP32
// coordinates, in integer arithmetic (plain C++, shared by the radial sort's
// kernels and its host test).
//
// The radial order of MEX (paper Sec. 2.2) is that of r^2 evaluated in FP64 as
// a CPU rounds it.  GB300 runs FP64 at about 1/76 of its FP32 rate: the three
// multiplications and two additions of 2^20 particles alone would take about
// 10 us.  The squares of FP32 numbers are exact (48 bits), so the two
// additions are done on 64-bit integers with the discarded bits kept as a
// sticky bit and rounded to nearest even at 53 bits: the same result in about
// 80 integer instructions per particle (2 us).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define ETICS_HD __host__ __device__ __forceinline__
#else
#define ETICS_HD inline
#endif

namespace etics {

ETICS_HD int r2_clz(uint64_t v) {   // v != 0
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

// v >> d with every discarded bit ORed into bit 0
ETICS_HD uint64_t r2_shift_sticky(uint64_t v, int d) {
    if (d == 0) return v;
    if (d >= 64) return v != 0 ? 1u : 0u;
    return (v >> d) | ((v << (64 - d)) != 0 ? 1u : 0u);
}

// v (top bit at least 60) rounded to nearest even at 53 bits, as q 2^drop
ETICS_HD uint64_t r2_round53(uint64_t v, int& drop) {
    drop = 11 - r2_clz(v);
    const uint64_t half = uint64_t(1) << (drop - 1), rem = v & ((half << 1) - 1);
    uint64_t q = v >> drop;
    q += (rem > half || (rem == half && (q & 1))) ? 1u : 0u;
    return q;
}

// bx, by, bz: the FP32 bit patterns of the coordinates.  False for a
// subnormal, infinite or NaN coordinate (the caller evaluates those in FP64).
ETICS_HD bool r2_bits_from_f32(uint32_t bx, uint32_t by, uint32_t bz, uint64_t& bits) {
    bx &= 0x7fffffffu;
    by &= 0x7fffffffu;
    bz &= 0x7fffffffu;
    auto usual = [](uint32_t b) { return b == 0 || (b >= 0x00800000u && b < 0x7f800000u); };
    if (!usual(bx) || !usual(by) || !usual(bz)) return false;
    const uint32_t ba = bx > by ? bx : by, bb = bx > by ? by : bx;   // larger of x, y first
    auto square = [](uint32_t b) -> uint64_t {
        const uint32_t m = b ? (b & 0x7fffffu) | 0x800000u : 0u;
        return (uint64_t)m * m << 14;          // 0, or top bit 60 or 61
    };
    int ea = (int)(ba >> 23);
    const int eb = (int)(bb >> 23), ez = (int)(bz >> 23);
    // fl64(x^2 + y^2), in units of 2^(2 ea - 314)
    uint64_t s = square(ba);
    if (s != 0) {
        s += r2_shift_sticky(square(bb), 2 * (ea - eb));
        int drop;
        const uint64_t q = r2_round53(s, drop);
        s = q << drop;
    }
    // + z^2, in units of the larger of the two
    uint64_t t = square(bz);
    if (s == 0 && t == 0) {
        bits = 0;
        return true;
    }
    if (s == 0) ea = ez;
    int e = ea;
    if (t == 0 || ez <= ea) {
        t = t == 0 ? 0 : r2_shift_sticky(t, 2 * (ea - ez));
    } else {
        s = r2_shift_sticky(s, 2 * (ez - ea));
        e = ez;
    }
    int drop;
    const uint64_t q = r2_round53(s + t, drop);
    // q in [2^52, 2^53]: value q 2^(drop + 2 e - 314)
    bits = ((uint64_t)(52 + drop + 2 * e - 314 + 1023) << 52) + (q - (uint64_t(1) << 52));
    return true;
}

}  // namespace etics
