// FP64 sums of products on the integer multiply pipe.
//
// GB300 has two FP64 lanes per SM (1.98 DFMA per clock measured, 1/64 of
// FP32), and an FP64 stencil or block-CSR row at that rate takes four to five
// times as long as its bytes. The 32 x 32 -> 64-bit integer multiply-add
// (mad.wide.s32) runs at 63 per clock and SM, so a sum of products
// sum_k u_k v_k is formed in fixed point instead:
//
//   - every factor is a signed 56-bit integer in units of 2^-56 of a power of
//     two that bounds its group (links: 1; block-CSR: the block's largest part;
//     the vector entries that one output needs: the largest of them), kept as
//     two 28-bit limbs of the value's sign, x = h 2^28 + l;
//   - u v = uh vh 2^56 + (uh vl + ul vh) 2^28 + ul vl, with the last term
//     dropped: three multiply-adds into two 64-bit sums that lose nothing more;
//   - the sums go back to FP64 once per output, rounded once.
//
// Error of an output against the exact sum. With B the power of two above the
// largest part of the vector entries that the site gathers (twice that where the
// stencil spares a bit), each product adds at most 2^-57 B (the link part,
// rounded), 2^-56 B |u| (the entry, truncated) and 2^-56 B (the dropped term);
// independent, about 2^-56 B sqrt(terms) together. 48 chained DFMAs round to
// about 2^-54 of their partial sums each. Block-CSR: the same per group of
// blocks, B the largest product of a block's and its entries' powers of two.
// These bounds are relative to the largest entry or product that meets in a sum,
// not to each term, as FP64 roundings are: a term far below the largest keeps
// fewer bits. So the form is taken only where the matrix itself leaves no output
// to such terms alone: links that couple every pair of colours (within 2^-24,
// msc_op_staggered), block rows of like sizes (bsr_even_row). The 2-norm errors
// are at or below FP64's (tests/test_gpu_fixed_fp64.py).
//
// Range of the 64-bit sums: |uh vh| <= 2^56 and |uh vl| + |ul vh| <= 2^57 per
// product, so up to 48 products (48 2^57 < 2^62.6) cannot overflow.
//
// Entries that are Inf or NaN, or so large or small that the scale leaves the
// exponent range (fx_in_range), take the FP64 arithmetic instead.
#pragma once
#include "common.cuh"

namespace msc {

struct FxSum {
    long long h, m;
};

// s += u v
__device__ __forceinline__ void fx_mac(FxSum& s, int uh, int ul, int vh, int vl) {
    s.h += (long long)uh * vh;
    s.m += (long long)uh * vl;
    s.m += (long long)ul * vh;
}

// Running bound of exponents: the high words without their signs.
__device__ __forceinline__ void fx_bound(unsigned& e, double2 v) {
    e = max(e, max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu));
}
// The bound as an exponent field (in place, bits 20..30).
__device__ __forceinline__ unsigned fx_field(unsigned e) { return e & 0x7ff00000u; }

// Whether a group with this exponent field is summed in fixed point: finite,
// its smallest unit a normal number and its largest sum finite.
__device__ __forceinline__ bool fx_in_range(unsigned field) {
    return field >= (160u << 20) && field <= (2000u << 20);
}

// v in units of 2^(e - 1078), e the exponent in `field`, truncated; negated
// where flip = -1 (flip: 0 or -1). Entries below the unit give 0 (the shift is
// then at least 56), and so do zeros, whose implicit bit is not masked, when
// `field` is kFxFloor at least.
constexpr unsigned kFxFloor = 64u << 20;
__device__ __forceinline__ void fx_split(double v, unsigned field, int flip, int& h, int& l) {
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v);
    const unsigned s = (field - ((unsigned)hi & 0x7ff00000u)) >> 20;
    unsigned long long q = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | lo) << 3;
    asm("shr.u64 %0, %0, %1;" : "+l"(q) : "r"(s));
    const int sg = (hi >> 31) ^ flip;
    h = ((int)(q >> 28) ^ sg) - sg;
    l = ((int)((unsigned)q & 0xfffffffu) ^ sg) - sg;
}

// The sums in a unit 2^d times larger (truncated towards minus infinity).
__device__ __forceinline__ void fx_shift(FxSum& s, unsigned d) {
    asm("shr.s64 %0, %0, %1;" : "+l"(s.h) : "r"(d));
    asm("shr.s64 %0, %0, %1;" : "+l"(s.m) : "r"(d));
}

// A factor bounded by 1 (|u| <= 1 + 1e-9) in units of 2^-56, rounded.
__device__ __forceinline__ int2 fx_unit(double u) {
    const long long q = __double2ll_rn(u * 0x1p56);
    const long long a = q < 0 ? -q : q;
    const int h = (int)(a >> 28), l = (int)(a & 0xfffffff);
    return q < 0 ? make_int2(-h, -l) : make_int2(h, l);
}

// The high word of a double (high word hi) times 2^(field - 1078 - half), field
// an exponent in place. Unsigned: an ordinary result's exponent and field add
// up to more than 2^31.
__host__ __device__ __forceinline__ int fx_high(int hi, unsigned field, int half) {
    return (int)((unsigned)hi + field - ((unsigned)(1078 + half) << 20));
}

// t units of the sum of products of unit factors and entries of exponent field
// `field`, times 2^-half.
__device__ __forceinline__ double fx_double(long long t, unsigned field, int half) {
    const double d = (double)t;
    return t == 0 ? 0.0 : __hiloint2double(fx_high(__double2hiint(d), field, half), __double2loint(d));
}
// The sum in units, rounded.
__device__ __forceinline__ long long fx_units(const FxSum& s) { return s.h + ((s.m + (1 << 27)) >> 28); }
__device__ __forceinline__ double fx_value(const FxSum& s, unsigned field, int half) {
    return fx_double(fx_units(s), field, half);
}

}  // namespace msc
