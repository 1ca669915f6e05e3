// Block-CSR row routine shared by the kernels that apply a generic
// block-CSR operator (the generic matrix the paper's solver takes, Sec. 3):
// the matrix is held in sliced ELL, 32 block rows per slice, block k of every
// row of a slice stored lane-interleaved ([slot][component][lane]).
#pragma once
#include "engine.h"
#include "fixed.cuh"

namespace msc {

template <class T> using T2 = typename C2<T>::t;

// y = A src for one row (thread = row, lanes of a warp = rows of a slice).
// Slice bases are 64-bit; offsets inside a slice (k * 32 * BD * BD) stay
// 32-bit; the source gathers go through the read-only path.
template <class T, int BD>
__device__ __forceinline__ void bsr_row(const OpDev& A, const T2<T>* __restrict__ vals,
                                        const T2<T>* __restrict__ src, int row, T2<T> (&y)[BD]) {
    const int slice = row >> 5;
    const int lane = row & 31;
    const int len = __ldg(&A.slice_len[slice]);
    const int64_t st = __ldg(&A.slice_start[slice]);
#pragma unroll
    for (int a = 0; a < BD; ++a) y[a] = {T(0), T(0)};
    const int32_t* __restrict__ cp = A.cols + st * 32 + lane;
    const T2<T>* __restrict__ vp = vals + st * BD * BD * 32 + lane;
#pragma unroll 3
    for (int k = 0; k < len; ++k) {
        const int c = __ldg(cp + k * 32);
        T2<T> xv[BD];
#pragma unroll
        for (int b = 0; b < BD; ++b) xv[b] = __ldg(src + (size_t)c * BD + b);
        const T2<T>* vk = vp + k * (BD * BD * 32);
#pragma unroll
        for (int a = 0; a < BD; ++a)
#pragma unroll
            for (int b = 0; b < BD; ++b) cfma(y[a], __ldg(vk + (a * BD + b) * 32), xv[b]);
    }
}

// y = A src for one row of a matrix of real 1 x 1 blocks in FP64 (valsr,
// [slot][lane]): half the FMAs and half the value bytes. An Inf or NaN among
// the row's entries would meet the zero imaginary parts, so such a row takes
// the complex form.
__device__ __forceinline__ void bsr_row_real(const OpDev& A, const double2* __restrict__ vals,
                                             const double2* __restrict__ src, int row, double2 (&y)[1]) {
    const int slice = row >> 5, lane = row & 31;
    const int len = __ldg(&A.slice_len[slice]);
    const int64_t st = __ldg(&A.slice_start[slice]);
    const int32_t* __restrict__ cp = A.cols + st * 32 + lane;
    const double* __restrict__ vp = A.valsr + st * 32 + lane;
    unsigned e = 0;
    y[0] = {0.0, 0.0};
#pragma unroll 5
    for (int k = 0; k < len; ++k) {
        const double2 x = __ldg(src + __ldg(cp + k * 32));
        const double v = __ldg(vp + k * 32);
        fx_bound(e, x);
        y[0].x = fma(v, x.x, y[0].x);
        y[0].y = fma(v, x.y, y[0].y);
    }
    if (e >= 0x7ff00000u) bsr_row<double, 1>(A, vals, src, row, y);
}

// ---------------------------------------------------------------------------
// FP64 rows by fixed-point sums (fixed.cuh), bd = 2 and 3, for matrices whose
// block rows hold entries of like sizes (bsr_even_row, bsr.cu). A block is stored as
// the 28-bit limbs of its entries in units of 2^-56 of the power of two above
// its largest part (valsfx, [slot][component][lane]) and that exponent (blkfx,
// [slot][lane], biased; 0: a zero block). G blocks of a row share one
// unit, the largest (block exponent + exponent of its column's entries) among
// them, and their 6 or 4 products a block and part go through the same sums,
// which then join the row's FP64 sums: 12 (8) FP64 instructions per group
// instead of 36 (16) per block on the two FP64 lanes of an SM.
// ---------------------------------------------------------------------------
// Product exponents (block + entry, both biased) that a group is summed at:
// its unit and its largest sum are normal numbers.
constexpr int kFxLo = 1100, kFxHi = 3000;

// The group's products in FP64 (entries that are Inf, NaN or out of range):
// the block's entries from their limbs.
template <int BD> struct RowVec {
    double2 y[BD];
};
template <int BD>
__device__ __noinline__ RowVec<BD> bsr_group_f64(RowVec<BD> r, const int4* vp, const uint16_t* ep, const int32_t* cp,
                                                 const double2* src, int count) {
    for (int k = 0; k < count; ++k) {
        const double2* x = src + (size_t)cp[k * 32] * BD;
        const int e = ep[k * 32];
        for (int a = 0; a < BD; ++a)
            for (int b = 0; b < BD; ++b) {
                const int4 u = vp[(k * BD * BD + a * BD + b) * 32];
                const double2 v = {ldexp((double)(((long long)u.x << 28) + u.y), e - 1078),
                                   ldexp((double)(((long long)u.z << 28) + u.w), e - 1078)};
                cfma(r.y[a], v, x[b]);
            }
    }
    return r;
}

// y = A src for one row from the limbs (y as bsr_row), G blocks at a time; the
// columns and exponents of the next group are loaded a group ahead.
template <int BD, int G>
__device__ __forceinline__ void bsr_row_fx(const OpDev& A, const double2* __restrict__ src, int row, double2 (&y)[BD]) {
    constexpr int E2 = BD * BD;
    static_assert(2 * BD * G <= 48, "products of one part in the 64-bit sums (fixed.cuh)");
    const int slice = row >> 5;
    const int lane = row & 31;
    const int len = __ldg(&A.slice_len[slice]);
    const int64_t st = __ldg(&A.slice_start[slice]);
#pragma unroll
    for (int a = 0; a < BD; ++a) y[a] = {0.0, 0.0};
    const int32_t* __restrict__ cp = A.cols + st * 32 + lane;
    const uint16_t* __restrict__ ep = A.blkfx + st * 32 + lane;
    const int4* __restrict__ vp = A.valsfx + st * E2 * 32 + lane;
    int cn[G], en[G];  // columns and exponents of the next group
#pragma unroll
    for (int j = 0; j < G; ++j) {
        cn[j] = j < len ? __ldg(cp + j * 32) : 0;
        en[j] = j < len ? __ldg(ep + j * 32) : 0;
    }
#pragma unroll 1
    for (int k = 0; k < len; k += G) {
        const int count = min(G, len - k);  // the same for the whole slice
        double2 x[G][BD];
        int eb[G], top = 0;
        bool finite = true;
#pragma unroll
        for (int j = 0; j < G; ++j) {
            eb[j] = en[j];
            if (j < count) {
                const double2* xp = src + (size_t)cn[j] * BD;
#pragma unroll
                for (int b = 0; b < BD; ++b) x[j][b] = __ldg(xp + b);
            }
        }
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const int q = k + G + j;
            cn[j] = q < len ? __ldg(cp + q * 32) : 0;
            en[j] = q < len ? __ldg(ep + q * 32) : 0;
        }
#pragma unroll
        for (int j = 0; j < G; ++j)
            if (j < count) {
                unsigned e = 0;
#pragma unroll
                for (int b = 0; b < BD; ++b) fx_bound(e, x[j][b]);
                finite = finite && e < 0x7ff00000u;
                // a block that meets zeros only is like a zero block: taken at the
                // row's own exponent, far above any entry's, so that fx_split gives 0
                if (e == 0) eb[j] = 0;
                if (e < (64u << 20))  // zeros, or next to the subnormals
#pragma unroll
                    for (int b = 0; b < BD; ++b) finite = finite && x[j][b].x == 0.0 && x[j][b].y == 0.0;
                if (eb[j] != 0) top = max(top, (int)(e >> 20) + eb[j]);
            }
        FxSum re[BD], im[BD];
#pragma unroll
        for (int a = 0; a < BD; ++a) re[a] = im[a] = {0, 0};
#pragma unroll
        for (int j = 0; j < G; ++j)
            if (j < count) {
                const unsigned field = (unsigned)(top - eb[j]) << 20;
                const int4* __restrict__ vk = vp + (size_t)(k + j) * (E2 * 32);
#pragma unroll
                for (int b = 0; b < BD; ++b) {
                    int rh, rl, ih, il;
                    fx_split(x[j][b].x, field, 0, rh, rl);
                    fx_split(x[j][b].y, field, 0, ih, il);
#pragma unroll
                    for (int a = 0; a < BD; ++a) {
                        const int4 u = __ldg(vk + (a * BD + b) * 32);
                        fx_mac(re[a], u.x, u.y, rh, rl);
                        fx_mac(im[a], u.x, u.y, ih, il);
                        fx_mac(re[a], u.z, u.w, -ih, -il);
                        fx_mac(im[a], u.z, u.w, rh, rl);
                    }
                }
            }
        if (finite && top >= kFxLo && top <= kFxHi) {
            const double scale = __hiloint2double((top - 1077) << 20, 0);
#pragma unroll
            for (int a = 0; a < BD; ++a) {
                y[a].x = fma((double)fx_units(re[a]), scale, y[a].x);
                y[a].y = fma((double)fx_units(im[a]), scale, y[a].y);
            }
        } else if (!finite || top != 0) {
            RowVec<BD> r;
#pragma unroll
            for (int a = 0; a < BD; ++a) r.y[a] = y[a];
            r = bsr_group_f64<BD>(r, vp + (size_t)k * (E2 * 32), ep + (size_t)k * 32, cp + (size_t)k * 32, src, count);
#pragma unroll
            for (int a = 0; a < BD; ++a) y[a] = r.y[a];
        }
    }
}

}  // namespace msc
