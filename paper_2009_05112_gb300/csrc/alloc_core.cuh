// alloc_core.cuh -- n_h of one hypercube (§3 Eq. nh, step a7), shared by the
// contexts' reallocation (adapt.cu) and vp_alloc_static (noalloc.cu).
#pragma once

#include "vp_internal.cuh"

namespace vp {

// ---------------------------------------------------------------------------
// Floor of a double 0 <= q < 2^52 from its bits (no FP64 instructions: they
// are scarce on this part), with two tests on the distance to the integers:
// near -- q is within 2^-40 q of an integer (the reciprocal product below is
// within a few ulp of the IEEE quotient, so only such q need the division);
// tie  -- q lies within 2^-50 q below an integer, i.e. exactly
//         (floor(q) + 1) - q <= q 2^-50, the test of the allocation reading.
// With q = M 2^(e - 52), M in [2^52, 2^53): distances are counted in units
// of 2^(e - 52) and q itself is M units, so "within c q" is "<= floor(c M)".
// ---------------------------------------------------------------------------
struct FloorBits {
    uint64_t iq;
    bool near, tie;
};

__device__ __forceinline__ FloorBits floor_bits(double q) {
    FloorBits r = {0ull, false, false};
    const uint64_t b = (uint64_t)__double_as_longlong(q);
    if (b == 0ull) return r;
    const int e = (int)((b >> 52) & 0x7ffu) - 1023;
    const uint64_t M = (b & ((1ull << 52) - 1ull)) | (1ull << 52);
    if (e >= 52) {  // an integer (not reached: q < 2^32 here)
        r.iq = M << (e - 52);
        return r;
    }
    uint64_t up;  // distance to the next integer, in units
    if (e >= 0) {
        const int sh = 52 - e;
        r.iq = M >> sh;
        const uint64_t frac = M & ((1ull << sh) - 1ull);
        up = (1ull << sh) - frac;
        r.near = frac <= (M >> 40);
    } else if (e == -1) {  // q in [1/2, 1): the next integer is 1 = 2^53 units
        up = (1ull << 53) - M;
    } else {
        return r;  // q < 1/2: floor 0, far from both integers
    }
    r.near = r.near || up <= (M >> 40);
    r.tie = up <= (M >> 50);
    return r;
}

__device__ __forceinline__ bool finite_bits(double x) {
    return ((uint64_t)__double_as_longlong(x) & 0x7ff0000000000000ull) != 0x7ff0000000000000ull;
}

// n_h of one hypercube (§3 Eq. nh with the library's reading): max(2,
// floor(N_ev d_h / sum d)), or floor(.) + 2; the equal split when sum d = 0 or
// on the first allocation.  The quotient is the IEEE one, (N_ev d_h) then
// / sum d.  One FP64 product decides almost every hypercube: q ~ d_h c with
// c = N_ev / sum d (within a few ulp of the IEEE quotient), and only a q within
// 2^-40 q of an integer takes the exact quotient; where N_ev d_h would not be
// a normal number, or c is unavailable (c = 0), the exact quotient
// is taken directly.
struct AllocK {
    double n_ev_d, sum_d, c, dmin;
    uint64_t n_hc;
    bool plus2;
};

__device__ __forceinline__ uint32_t alloc_one(double dh, const AllocK &K, int initial) {
    uint64_t iq;
    if (__double_as_longlong(K.sum_d) > 0ll) {  // sum d > 0 (sum_d is finite here)
        if ((uint64_t)__double_as_longlong(dh) == 0ull) {
            iq = 0ull;  // (a zero numerator is exact)
        } else if ((uint64_t)__double_as_longlong(dh) >= (uint64_t)__double_as_longlong(K.dmin) &&
                   (uint64_t)__double_as_longlong(K.c) != 0ull) {  // (integer compares: d_h, c >= 0)
            const double q = dh * K.c;
            FloorBits f = floor_bits(q);
            iq = f.iq;
            // (below 2 - tol the max(2, .) decides)
            const bool above = (uint64_t)__double_as_longlong(q) > 0x3FF8000000000000ull;  // q > 1.5
            if ((K.plus2 || above) && f.near) {
                f = floor_bits(__ddiv_rn(__dmul_rn(K.n_ev_d, dh), K.sum_d));
                iq = f.iq + (f.tie ? 1ull : 0ull);
            }
        } else {
            const FloorBits f = floor_bits(__ddiv_rn(__dmul_rn(K.n_ev_d, dh), K.sum_d));
            iq = f.iq + (f.tie ? 1ull : 0ull);
        }
    } else {
        const FloorBits f = floor_bits(__ddiv_rn(K.n_ev_d, (double)K.n_hc));
        iq = f.iq + (f.tie ? 1ull : 0ull);
    }
    if (K.plus2 && !initial) return (uint32_t)iq + 2u;
    return iq > 2ull ? (uint32_t)iq : 2u;
}

}  // namespace vp
