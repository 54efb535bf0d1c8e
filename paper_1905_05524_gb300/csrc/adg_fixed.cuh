// Block-scaled 58-bit fixed-point contractions: the FP64 path's small dense
// products on the integer multiply-add pipe.
//
// sm_103a issues one warp-wide FP64 add, multiply or fused multiply-add per 16
// cycles on an SM (19 measured with four busy sub-partitions), a 32 x 32 + 64
// bit integer multiply-add (IMAD.WIDE) per 1.2 cycles.  A dot product of
// doubles sum_p a_p b_p is therefore formed from integers: all b of a group
// (one component of one cell) share a power-of-two scale taken from the group's
// largest magnitude, likewise the a of one matrix row, and both are held as
// m 2^s with |m| < 2^58 in two limbs m = h 2^29 + l.
// The products are exact; h h' and h l' + l h' are summed in two 64-bit
// integers (exact up to 16 terms), l l' is dropped: three IMAD.WIDE per term,
// and the sum does not depend on its order.  Error of a sum of n terms, from
// the truncations to 58 bits, the dropped products and one rounding: below
// (3 n + 1) 2^-57 max|a| max|b| (tests/test_fixed_point.py), against up to
// n 2^-53 sum|a||b| for a chain of FP64 fused multiply-adds.
//
// NaN or infinity anywhere in a group makes every result of the group NaN (an
// FP64 contraction spreads it to the node's row and column, the following
// sweeps to the cell).  Groups below 2^-958 count as zero.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace adg {

struct Limbs {
    int h, l;  // m = h 2^29 + l
};

// smallest group exponent (biased as in a double); at least 58, so that zeros and subnormals, whose
// leading bit fx_from takes for set, shift out
constexpr int kFxMinExp = 64;
constexpr int kFxBadExp = 0x4000;   // group exponent of a group with NaN or infinity

// Order of magnitude as an unsigned integer: exponent and 20 bits of mantissa.
__device__ __forceinline__ uint32_t fx_mag(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// Group exponent E from the largest fx_mag of the group: |x| < 2^(E - 1022),
// m = x 2^(1080 - E).
__device__ __forceinline__ int fx_exp(uint32_t mag) {
    return mag >= 0x7ff00000u ? kFxBadExp : max((int)(mag >> 20), kFxMinExp);
}

// m of x for group exponent E (truncated towards zero)
__device__ __forceinline__ long long fx_from(double x, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int sh = min(E - (int)((hi >> 20) & 0x7ffu), 63);
    const unsigned long long t = (((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 5) >> sh;  // < 2^58
    const long long s = (int)hi >> 31;
    return ((long long)t ^ s) - s;
}

// Limbs of an operand of the data side: 0 <= l < 2^29 (one shift, one mask).
__device__ __forceinline__ Limbs fx_split(long long m) { return Limbs{(int)(m >> 29), (int)m & 0x1fffffff}; }
// Limbs of a matrix entry: |l| <= 2^28, so that h l' + l h' of 16 terms stays below 1.5 2^62.
__device__ __forceinline__ Limbs fx_split_centred(long long m) {
    Limbs r;
    r.h = (int)((m + (1ll << 28)) >> 29);
    r.l = (int)m - (int)((unsigned)r.h << 29);
    return r;
}

__device__ __forceinline__ Limbs fx_limbs(double x, int E) { return fx_split(fx_from(x, E)); }

// The two partial sums of a dot product (a: matrix entry, b: data).
struct FxSum {
    long long hh = 0, mid = 0;
    __device__ __forceinline__ void add(const Limbs& a, const Limbs& b) {
        hh += (long long)a.h * b.h;
        mid += (long long)a.h * b.l;
        mid += (long long)a.l * b.h;
    }
    // in units of 2^(Ea + Eb - 2102)
    __device__ __forceinline__ long long value() const { return hh + ((mid + (1ll << 28)) >> 29); }
};

// a 2^e as a double, |a| < 2^62, rounded to nearest (ties away from zero); NaN
// beyond the double range or for a group exponent of kFxBadExp in e.  The
// magnitude is normalised to bit 62 so that the rounding carry stays in the word.
__device__ __forceinline__ double fx_to(long long a, int e) {
    const uint32_t s = (uint32_t)((int)(a >> 32) >> 31);
    const unsigned long long m = (unsigned long long)((a ^ (long long)(int)s) - (long long)(int)s);
    uint32_t hi = (uint32_t)(m >> 32), lo = (uint32_t)m;
    e += 1022 + 62;
    if (hi == 0) {
        hi = lo;
        lo = 0;
        e -= 32;
    }
    const int lz = __clz((int)hi);  // >= 1 for the high word as it came; 0 possible after the move
    unsigned long long f = ((unsigned long long)hi << 32 | lo) << lz >> 1;  // leading bit at 62
    f += 0x200;
    const int ex = e - lz + 1;  // one below the biased exponent: the leading bit adds it
    uint32_t rh = (uint32_t)(f >> 42) + ((uint32_t)ex << 20), rl = (uint32_t)(f >> 10);
    if ((unsigned)ex >= 2046u || hi == 0) {
        rh = ex >= 2046 ? 0x7ff80000u : 0u;
        rl = 0;
    }
    return __hiloint2double((int)(rh | (s & 0x80000000u)), (int)rl);
}

// Residuals are sums of derivatives, each with the exponents of its own matrix
// row and data.  fx_row_shift: bits by which a row of exponent ed, absolute sum
// `row`, lifts a product above 2^57 in units of the product; the derivative then
// has exponent X = E + ed - 1022 + shift, and its value, moved down by
// fx_down(shift, ER, X) bits, that of the sum, ER >= X.  Three derivatives and a
// source (ER above its own) stay below 2^59.
__device__ __forceinline__ int fx_row_shift(double row, int ed) { return max((int)(fx_mag(row) >> 20) - ed + 1, 0); }
__device__ __forceinline__ int fx_down(int shift, int ER, int X) { return min(shift + ER - X, 63); }

// 1/x: the hardware FP32 reciprocal of the mantissa, then one third-order
// step r (1 + e + e^2), e = 1 - x r (Chebyshev's iteration), whose error e^3 is
// below 2^-60: three FP64 operations where the division takes four to five.
// Zero, subnormal, huge, infinite and NaN x take the division.
__device__ __forceinline__ double fx_rcp(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t ex = (hi >> 20) & 0x7ffu;
    if (ex - 1u >= 2040u) return 1.0 / x;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29))));
    const uint32_t rb = __float_as_uint(r);
    const double r0 = __hiloint2double((int)(((rb >> 3) + ((1023u - 127u + 1023u - ex) << 20)) | (hi & 0x80000000u)),
                                       (int)(rb << 29));
    const double e = fma(-x, r0, 1.0);
    return fma(r0, fma(e, e, e), r0);
}

// SMs of the current device.
inline int sm_count() {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// Blocks of a launch that strides over `tiles` tiles: as many rounds as the
// resident blocks need, the tiles spread evenly over them.
inline int fx_grid(int tiles, int resident) {
    const int sms = sm_count();
    const int rounds = (tiles + sms * resident - 1) / (sms * resident);
    return (tiles + rounds - 1) / rounds;
}

}  // namespace adg
