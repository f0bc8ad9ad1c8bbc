// Complex sums of products in two-limb fixed point, to FP64 accuracy, for sums
// whose operands share a scale. The FP64 unit issues 1.8 FMAs per clock and SM,
// mad.wide.s32 44 (measured), so three mad.wide per real product are eight times
// as fast.
//
// Operands are rounded to 54 fractional bits of 2^e > their block's largest
// magnitude and held as two signed limbs, q = h 2^26 + l, |h| <= 2^28, |l| <= 2^25.
// A real product is h h' (weight 2^52) plus h l' + l h' (2^26); l l' (2^-58 of the
// scales' product) is dropped. Sums of up to 36 complex products stay below 2^63
// (|h h'| <= 2^56, two per part), so nothing overflows. The result is rounded to
// FP64 once. The error is about 2^-56 of the scales' product per sum, against 2^-54
// of the running sum for every FP64 FMA.
#pragma once

#include "common.cuh"

struct Limbs { int rh, rl, ih, il; };   // one complex value

__device__ __forceinline__ Limbs to_limbs(double2 v, int e)
{
    Limbs o;
    const long long r = fixed_point<54>(v.x, e), i = fixed_point<54>(v.y, e);
    o.rl = ((int)r << 6) >> 6;                       // the low 26 bits, signed
    o.rh = (int)((r - o.rl) >> 26);
    o.il = ((int)i << 6) >> 6;
    o.ih = (int)((i - o.il) >> 26);
    return o;
}

// The value of limbs with exponent e, as FP64.
__device__ __forceinline__ double2 limbs_fp64(const Limbs& x, int e)
{
    return make_double2(int_to_fp64((long long)x.rh * (1 << 26) + x.rl, e - 54),
                        int_to_fp64((long long)x.ih * (1 << 26) + x.il, e - 54));
}

struct LimbSum {
    long long rr = 0, ii = 0, im = 0, crr = 0, cii = 0, cim = 0;
    __device__ __forceinline__ void add(const Limbs& a, const Limbs& b)
    {
        rr += (long long)a.rh * b.rh;
        crr += (long long)a.rh * b.rl;
        crr += (long long)a.rl * b.rh;
        ii += (long long)a.ih * b.ih;
        cii += (long long)a.ih * b.il;
        cii += (long long)a.il * b.ih;
        im += (long long)a.rh * b.ih;
        im += (long long)a.ih * b.rh;
        cim += (long long)a.rh * b.il;
        cim += (long long)a.rl * b.ih;
        cim += (long long)a.ih * b.rl;
        cim += (long long)a.il * b.rh;
    }
    // the same with l l' (2^0), for sums of squares, where it does not average out
    __device__ __forceinline__ void add_all(const Limbs& a, const Limbs& b, long long& llr, long long& lli)
    {
        add(a, b);
        llr += (long long)a.rl * b.rl - (long long)a.il * b.il;
        lli += (long long)a.rl * b.il + (long long)a.il * b.rl;
    }
    // minus a b
    __device__ __forceinline__ void sub(const Limbs& a, const Limbs& b) { add(a, Limbs{-b.rh, -b.rl, -b.ih, -b.il}); }
    // both parts in units of 2^-56 of the scales' product
    __device__ __forceinline__ long long re() const { return (rr - ii) + ((crr - cii + (1 << 25)) >> 26); }
    __device__ __forceinline__ long long imag() const { return im + ((cim + (1 << 25)) >> 26); }
};

__device__ __forceinline__ unsigned mag_bits(double2 v)
{
    return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}

// Exponent e of a largest magnitude in mag_bits form: every |x| < 2^e (-1021 for
// subnormal ones; 1025 marks an infinity or a NaN).
__device__ __forceinline__ int mag_exponent(unsigned m) { return max((int)(m >> 20), 1) - 1022; }
#define FIXED_EXP_INF 1025

// The sum of `s` with operand exponents adding up to e, as FP64.
__device__ __forceinline__ double2 limb_value(const LimbSum& s, int e)
{
    return make_double2(int_to_fp64(s.re(), e - 56), int_to_fp64(s.imag(), e - 56));
}

// Largest magnitude of a block's values m (all threads return it; red: one word
// per warp). The block must reach this together.
__device__ __forceinline__ unsigned block_mag(unsigned m, unsigned* red)
{
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) m = max(m, red[k]);
    return m;
}
