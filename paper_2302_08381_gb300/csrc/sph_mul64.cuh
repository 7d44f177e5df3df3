// FP64 products (and conversions to FP32) on the integer pipe, bit for bit the hardware's (IEEE 754
// binary64, round to nearest even): the 53-bit significands as integers,
// their product from four 32 x 32 -> 64-bit multiplies, normalized, rounded
// and put together with the summed exponents.
//
// Why: GB300's FP64 pipe takes one warp instruction per SM every 20 clocks
// (measured, any mix of fma, mul and add; a lone warp 68), while the issue
// slots beside it are idle. A product done here costs 16 clocks per warp and
// SM of those idle slots, and a stream of one fma and one such product runs
// at the rate of the fma alone (measured at 16 warps per SM: 20.05 clocks
// for the two, 40 for two FP64 instructions). So in a kernel bound by the
// FP64 pipe every product that is not part of an fma is moved here.
//
// Range: a factor of exponent within 2^+-300 (Mul64) and operands within
// 2^+-700, so every product is a normal number; subnormals, infinities, NaN and
// the rest of the range are reported, and the caller repeats the work on the
// FP64 pipe. It does so for a whole step of its loop in one branch: with a
// branch around every pair of products the kernel was no faster than on the FP64
// pipe alone (DEGREE, l_max 30, 200k points: 5.6 ms, and 4.4 with one branch per
// step). A zero operand is reported too, unless ZERO: a test and two selects per
// product, taken for tiles with a point that has a zero coordinate.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sph {

// The common factor of several products, taken apart once.
struct Mul64 {
    double v;
    uint32_t hi;      // its high word (sign, exponent)
    uint32_t m1, m0;  // significand, shifted left to fill 64 bits
    uint32_t ex;      // exponent field minus that of 2^1
    bool ok;    // in range
    bool zero;  // +-0

    __device__ __forceinline__ explicit Mul64(double b) : v(b) {
        hi = uint32_t(__double2hiint(b));
        const uint32_t lo = uint32_t(__double2loint(b));
        m1 = __funnelshift_l(lo, (hi & 0x000fffffu) | 0x00100000u, 11);
        m0 = lo << 11;
        const uint32_t e = hi & 0x7ff00000u;
        ok = e - ((1023u - 300u) << 20) <= (600u << 20);
        zero = ((hi & 0x7fffffffu) | lo) == 0u;
        ex = e - (1024u << 20);
    }

    // a * v; `in` (the caller's `ok`) is cleared when a is out of the fast range:
    // the result is then meaningless. ZERO: both ranges checked here, 0 in them.
    template <bool ZERO>
    __device__ __forceinline__ double fast(double a, bool& in) const {
        const uint32_t ah = uint32_t(__double2hiint(a)), al = uint32_t(__double2loint(a));
        const uint32_t ea = ah & 0x7ff00000u;
        const bool az = ZERO && ((ah & 0x7fffffffu) | al) == 0u;
        if constexpr (ZERO)
            in = (ok || zero) && (az || ea - ((1023u - 700u) << 20) <= (1400u << 20));
        else
            in = in && ea - ((1023u - 700u) << 20) <= (1400u << 20);
        const uint32_t am = (ah & 0x000fffffu) | 0x00100000u;
        // the product of the 53-bit and the 64-bit significand, 117 bits: hi:l1:l0
        const uint64_t t0 = uint64_t(al) * m0;
        const uint64_t t1 = uint64_t(am) * m0 + uint32_t(t0 >> 32);
        const uint64_t t2 = uint64_t(al) * m1 + uint32_t(t1);
        const uint64_t h = uint64_t(am) * m1 + uint32_t(t1 >> 32) + uint32_t(t2 >> 32);
        const uint32_t h1 = uint32_t(h >> 32), h0 = uint32_t(h), l1 = uint32_t(t2), l0 = uint32_t(t0);
        // 2^51 <= h < 2^53: shift so that H is the 53-bit significand and one
        // bit to round by, in [2^53, 2^54)
        const uint32_t n = h1 >> 20, s = 2u - n;
        const uint32_t H1 = __funnelshift_l(h0, h1, s), H0 = __funnelshift_l(l1, h0, s);
        // nearest, ties to even: half a unit up, except from an exact tie at an even significand
        const uint32_t up = ((H0 >> 1) & 1u) | (((l1 << s) | l0) != 0u ? 1u : 0u);
        const uint64_t R = ((uint64_t(H1) << 32) | H0) + up;
        const uint32_t rh = uint32_t(R >> 33) + ea + ex + (n << 20);  // a carry out of the significand moves the exponent
        const bool nz = !(ZERO && (az || zero));
        return __hiloint2double(int((nz ? rh : 0u) | ((ah ^ hi) & 0x80000000u)), int(nz ? uint32_t(R >> 1) : 0u));
    }
};

// float(v), rounded to nearest even as the hardware's conversion (which runs
// on the FP64 pipe too): the top 32 of the significand's bits, rebiased, plus
// the carry of the 29 dropped bits; magnitudes that round to zero are done
// here. `in` is cleared where the result is subnormal, infinite or NaN.
__device__ __forceinline__ float f32_of_f64(double v, bool& in) {
    const uint32_t hi = uint32_t(__double2hiint(v)), lo = uint32_t(__double2loint(v));
    const uint32_t e = hi & 0x7ff00000u;
    const bool zero = e < ((1023u - 150u) << 20);
    uint32_t u = __funnelshift_l(lo, hi & 0x7fffffffu, 3) - (896u << 23);
    const uint32_t rem = lo << 3;
    u += (rem + (0x7fffffffu + (u & 1u)) < rem) ? 1u : 0u;
    in = in && (zero || e - (897u << 20) <= (252u << 20));
    return __uint_as_float((zero ? 0u : u) | (hi & 0x80000000u));
}

}  // namespace sph
