// Device functions of the staggered operator shared by the single-operator
// and the batched kernels:
//   D_xy = 1/2 sum_mu eta_mu(x) [U_mu(x) d_{y,x+mu} - U_mu(x-mu)^dagger d_{y,x-mu}],
//   eta_mu(x) = (-1)^(x_0 + ... + x_{mu-1}), periodic boundaries.
#pragma once
#include <type_traits>

#include "engine.h"
#include "fixed.cuh"

namespace msc {

template <class T> using T2 = typename C2<T>::t;

struct SiteNbrs {
    int fwd[4], bwd[4];
    int par[4];  // parity of x_0 + ... + x_{mu-1}
};

__device__ __forceinline__ SiteNbrs neighbours(int x, const StagGeom& g) {
    SiteNbrs nb;
    int c[4];
    const int q0 = gdiv(x, g, 0), q1 = gdiv(q0, g, 1), q2 = gdiv(q1, g, 2);
    c[0] = x - q0 * g.L[0];
    c[1] = q0 - q1 * g.L[1];
    c[2] = q1 - q2 * g.L[2];
    c[3] = q2;
    int stride = 1, psum = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const int L = g.L[mu];
        nb.fwd[mu] = (c[mu] == L - 1) ? x - (L - 1) * stride : x + stride;
        nb.bwd[mu] = (c[mu] == 0) ? x + (L - 1) * stride : x - stride;
        nb.par[mu] = psum & 1;
        psum += c[mu];
        stride *= L;
    }
    return nb;
}

// Parity-reduced operator (g.eo = 1 + p): site x sits at compressed index
// x / 2 of a parity vector (each pair of sites (2k, 2k+1) along x0 holds one
// site of each parity), and the h-th site of parity par is eo_site(h, par).
__device__ __forceinline__ int vsite(int x, const StagGeom& g) { return g.eo ? (x >> 1) : x; }

__device__ __forceinline__ int eo_site(int h, int par, const StagGeom& g) {
    const int hl = g.L[0] >> 1;
    const int row = gdiv(h, g, 3);
    const int k = h - row * hl;
    const int r1 = gdiv(row, g, 1), r2 = gdiv(r1, g, 2);
    const int c1 = row - r1 * g.L[1];
    const int c2 = r1 - r2 * g.L[2];
    const int c3 = r2;
    return 2 * k + ((par + c1 + c2 + c3) & 1) + g.L[0] * row;
}

// The site a thread of a pass handles at loop index h: on the
// parity-reduced operator, t = D p (PASS_A, OTHER) lives on the other parity
// and every other pass's output on the source's.
template <bool OTHER>
__device__ __forceinline__ int pass_site(int h, const StagGeom& g) {
    if (!g.eo) return h;
    const int src_par = g.eo - 1;
    return eo_site(h, OTHER ? 1 - src_par : src_par, g);
}

// ---------------------------------------------------------------------------
// link loads
// ---------------------------------------------------------------------------
template <class T, int NC, int RECON> struct Links;

// full storage: T2 [4][NC*NC][V]
template <class T, int NC> struct Links<T, NC, 0> {
    __device__ static __forceinline__ void load(const void* base, int mu, int x, int V,
                                                T2<T> (&u)[NC][NC]) {
        const T2<T>* U = (const T2<T>*)base + (size_t)mu * NC * NC * V + x;
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) u[a][b] = U[(size_t)(a * NC + b) * V];
    }
};

// SU(3), two rows in three float4: (u00,u01) (u02,u10) (u11,u12)
template <> struct Links<float, 3, 1> {
    __device__ static __forceinline__ void load(const void* base, int mu, int x, int V,
                                                float2 (&u)[3][3]) {
        const float4* U = (const float4*)base + (size_t)mu * 3 * V + x;
        const float4 q0 = U[0], q1 = U[(size_t)V], q2 = U[(size_t)2 * V];
        u[0][0] = {q0.x, q0.y}; u[0][1] = {q0.z, q0.w};
        u[0][2] = {q1.x, q1.y}; u[1][0] = {q1.z, q1.w};
        u[1][1] = {q2.x, q2.y}; u[1][2] = {q2.z, q2.w};
        // row 2 = conj(row0 x row1)
        u[2][0] = cconj(csub(cmul(u[0][1], u[1][2]), cmul(u[0][2], u[1][1])));
        u[2][1] = cconj(csub(cmul(u[0][2], u[1][0]), cmul(u[0][0], u[1][2])));
        u[2][2] = cconj(csub(cmul(u[0][0], u[1][1]), cmul(u[0][1], u[1][0])));
    }
};

// SU(2), one row in one float4: (u00,u01); row 1 = (-conj u01, conj u00)
template <> struct Links<float, 2, 1> {
    __device__ static __forceinline__ void load(const void* base, int mu, int x, int V,
                                                float2 (&u)[2][2]) {
        const float4 q = ((const float4*)base)[(size_t)mu * V + x];
        u[0][0] = {q.x, q.y};
        u[0][1] = {q.z, q.w};
        u[1][0] = {-q.z, q.w};
        u[1][1] = {q.x, -q.y};
    }
};

// Index of the complex entry (site x, colour a) of a vector of element type
// T. Vectors are site-major (x * NC + a), except FP32 vectors of the
// single-operator stencil path (PL), which are colour-planar (a * V + x): the
// loads of one colour of a warp's 32 consecutive sites are then one
// contiguous 256-byte run instead of three 8-byte loads at a 24-byte stride.
template <class T, bool PL, int NC>
__device__ __forceinline__ size_t vix(int x, int a, int V) {
    return (PL && sizeof(T) == 4) ? (size_t)a * V + x : (size_t)x * NC + a;
}

// y = D src at site x. src may have been written by other blocks of the same
// kernel: it is neither restrict nor read through the read-only path.
template <class T, int NC, int RECON, bool PL = false>
__device__ __forceinline__ void dslash_site_fresh(const void* links, const T2<T>* src, int x, const StagGeom& g,
                                                  T2<T> (&y)[NC]) {
    const SiteNbrs nb = neighbours(x, g);
#pragma unroll
    for (int a = 0; a < NC; ++a) y[a] = {T(0), T(0)};
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        T2<T> u[NC][NC], v[NC];
        Links<T, NC, RECON>::load(links, mu, x, g.V, u);
#pragma unroll
        for (int b = 0; b < NC; ++b) v[b] = src[vix<T, PL, NC>(vsite(nb.fwd[mu], g), b, vlen(g))];
        T2<T> w[NC][NC], z[NC];
        Links<T, NC, RECON>::load(links, mu, nb.bwd[mu], g.V, w);
#pragma unroll
        for (int b = 0; b < NC; ++b) z[b] = src[vix<T, PL, NC>(vsite(nb.bwd[mu], g), b, vlen(g))];
        const T eta = nb.par[mu] ? T(-0.5) : T(0.5);
#pragma unroll
        for (int a = 0; a < NC; ++a) {
            T2<T> f = {T(0), T(0)};
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                cfma(f, u[a][b], v[b]);        // + U_mu(x) src(x+mu)
                cfms_conj(f, w[b][a], z[b]);   // - U_mu(x-mu)^dag src(x-mu)
            }
            y[a].x = fma(eta, f.x, y[a].x);
            y[a].y = fma(eta, f.y, y[a].y);
        }
    }
}

// The same of a vector that nothing writes while the kernel runs.
template <class T, int NC, int RECON, bool PL = false>
__device__ __forceinline__ void dslash_site(const void* links, const T2<T>* __restrict__ src, int x, const StagGeom& g,
                                            T2<T> (&y)[NC]) {
    dslash_site_fresh<T, NC, RECON, PL>(links, src, x, g, y);
}

// y = D src at site x in FP64 on the FP64 pipe, for the sites whose entries
// leave the range of the fixed-point sums (rare: out of line).
template <int NC> struct SiteVec {
    double2 y[NC];
};
template <int NC>
__device__ __noinline__ SiteVec<NC> dslash_site_f64(const void* links64, const double2* src, int x, const StagGeom& g) {
    SiteVec<NC> r;
    dslash_site_fresh<double, NC, 0>(links64, src, x, g, r.y);
    return r;
}

// Whether every entry that site x gathers is zero: y = 0 then without the sums,
// as the links are finite. A source on one site or one parity stays on
// alternating parities under D, and half the lanes of every warp of an FP64 pass
// then ask.
template <int NC>
__device__ __noinline__ bool site_among_zeros(const double2* src, int x, const StagGeom& g) {
    const SiteNbrs nb = neighbours(x, g);
    unsigned long long bits = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const double2* vf = src + (size_t)vsite(nb.fwd[mu], g) * NC;
        const double2* vb = src + (size_t)vsite(nb.bwd[mu], g) * NC;
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            const double2 f = vf[b], w = vb[b];
            bits |= (unsigned long long)(__double_as_longlong(f.x) | __double_as_longlong(f.y) |
                                         __double_as_longlong(w.x) | __double_as_longlong(w.y)) << 1;
        }
    }
    return bits == 0;
}

// Index of entry 0 of link (mu, x) in the limb array: sites in groups of 32,
// the entries of a group 32 apart, so that one address serves a link's NC^2
// loads (constant offsets) and a warp's loads stay contiguous.
template <int NC>
__host__ __device__ __forceinline__ size_t fx_link(int mu, int x, int V) {
    return ((size_t)mu * ((V + 31) >> 5) + (x >> 5)) * (NC * NC * 32) + (x & 31);
}

// y = D src at site x in FP64 by fixed-point sums (see fixed.cuh). lfx: the
// limbs (re.h, re.l, im.h, im.l) of each link entry in units of 2^-56, at
// fx_link().
// The sign of eta_mu and of the backward hop goes into the entries' limbs.
// The entries of one direction (both hops) are loaded and bounded together;
// the first direction sets the sums' unit with one bit to spare (and not below
// kFxFloor, where zeros would not be split into zeros: a direction that holds
// nothing else), and a later one with larger entries shifts the sums (about two
// of three warps do so once on Gaussian entries). Holding all 8 hops' entries for one exact bound
// instead needs 255 registers (32^4, two passes: 506 us).
// FRESH: src may have been written by other blocks of the same kernel, so its
// loads do not take the read-only path.
template <int NC, bool FRESH>
__device__ __forceinline__ void dslash_site_fx(const void* lfx, const void* links64, const double2* src, int x, const StagGeom& g, double2 (&y)[NC]) {
    if (!lfx) {  // links without limbs (batches mix operators)
        const SiteVec<NC> r = dslash_site_f64<NC>(links64, src, x, g);
#pragma unroll
        for (int a = 0; a < NC; ++a) y[a] = r.y[a];
        return;
    }
    const SiteNbrs nb = neighbours(x, g);
    FxSum re[NC], im[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) re[a] = im[a] = {0, 0};
    unsigned field = 0;  // of the sums; Inf and NaN give 2^31, above every entry's
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        double2 v[2][NC];
        const double2* vf = src + (size_t)vsite(nb.fwd[mu], g) * NC;
        const double2* vb = src + (size_t)vsite(nb.bwd[mu], g) * NC;
        unsigned e = 0;
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            v[0][b] = FRESH ? vf[b] : __ldg(vf + b);
            v[1][b] = FRESH ? vb[b] : __ldg(vb + b);
        }
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            fx_bound(e, v[0][b]);
            fx_bound(e, v[1][b]);
        }
        const unsigned f = fx_field(e);
        if (mu == 0) {
            field = max(f + (1u << 20), kFxFloor);
        } else if (f > field) {
            const unsigned d = (f + (1u << 20) - field) >> 20;
            field = f + (1u << 20);
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                fx_shift(re[a], d);
                fx_shift(im[a], d);
            }
        }
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
            const bool fwd = dir == 0;
            const int4* __restrict__ U = (const int4*)lfx + fx_link<NC>(mu, fwd ? x : nb.bwd[mu], g.V);
            const int flip = fwd ? -nb.par[mu] : nb.par[mu] - 1;
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                int rh, rl, ih, il;
                fx_split(v[dir][b].x, field, flip, rh, rl);
                fx_split(v[dir][b].y, field, flip, ih, il);
                // forward: U_ab v_b; backward: conj(U_ba) v_b
                const int zh = fwd ? -ih : ih, zl = fwd ? -il : il;
                const int wh = fwd ? rh : -rh, wl = fwd ? rl : -rl;
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    const int4 u = __ldg(U + (fwd ? a * NC + b : b * NC + a) * 32);
                    fx_mac(re[a], u.x, u.y, rh, rl);
                    fx_mac(im[a], u.x, u.y, ih, il);
                    fx_mac(re[a], u.z, u.w, zh, zl);
                    fx_mac(im[a], u.z, u.w, wh, wl);
                }
            }
        }
    }
    if (!fx_in_range(field)) {
        if (site_among_zeros<NC>(src, x, g)) {
#pragma unroll
            for (int a = 0; a < NC; ++a) y[a] = {0.0, 0.0};
            return;
        }
        const SiteVec<NC> r = dslash_site_f64<NC>(links64, src, x, g);
#pragma unroll
        for (int a = 0; a < NC; ++a) y[a] = r.y[a];
        return;
    }
#pragma unroll
    for (int a = 0; a < NC; ++a) y[a] = {fx_value(re[a], field, 1), fx_value(im[a], field, 1)};
}

// One site of a D pass: y = D src at x, then the epilogue KIND; returns this
// site's contribution to the pass's reduction (0 when d.row < 0).
//   PASS_A: out = y;                       P terms d|aux|^2 + |y|^2
//   PASS_B: r -= alpha (d aux - y);        |r|^2
//   PASS_C: out = b - (d aux - y) (FP64);  |out|^2
//   PASS_D: out = d aux - y
// PL: FP32 vectors (of type T or TO) are colour-planar (see vix).
// A site's share of a pass's reduction: FP32 for the FP32 passes (summed
// over a thread's sites in FP32, then reduced in FP64 across threads), FP64
// for the residual pass and FP64 operators.
template <class T, int KIND>
using SiteAcc = typename std::conditional<(sizeof(T) == 4 && KIND != PASS_C), float, double>::type;

// The epilogue KIND of a D pass at colour a of vector site x, y = (D src)_a
// there; adds to the site's share of the reduction (nothing when d.row < 0).
template <class T, int NC, int KIND, class TO, bool PL>
__device__ __forceinline__ void stag_colour_of(const PassDesc& d, const T2<T>* aux, int x, int a, int V, T2<T> y,
                                               T alpha, SiteAcc<T, KIND>& loc) {
    const T dd = (T)d.d;
    const size_t i = vix<T, PL, NC>(x, a, V);
    if (KIND == PASS_A) {
        ((T2<T>*)d.out)[i] = y;
        if (d.row >= 0) {
            const T2<T> pa = aux[i];
            loc += dd * (pa.x * pa.x + pa.y * pa.y) + y.x * y.x + y.y * y.y;
        }
    } else if (KIND == PASS_B || KIND == PASS_BC) {
        T2<T>* r = (T2<T>*)d.out;
        const T2<T> pa = aux[i];
        const T2<T> ap = {dd * pa.x - y.x, dd * pa.y - y.y};
        T2<T> ra = r[i];
        ra.x -= alpha * ap.x;
        ra.y -= alpha * ap.y;
        r[i] = ra;
        loc += ra.x * ra.x + ra.y * ra.y;
    } else if (KIND == PASS_C) {
        TO* out = (TO*)d.out;
        const T2<T> xa = aux[i];
        const double2 ba = d.b[(size_t)x * NC + a];
        const double vx = ba.x - ((double)dd * xa.x - y.x);
        const double vy = ba.y - ((double)dd * xa.y - y.y);
        if (out) {
            const size_t o = vix<TO, PL, NC>(x, a, V);
            out[2 * o] = (TO)vx;
            out[2 * o + 1] = (TO)vy;
        }
        loc += vx * vx + vy * vy;
    } else {
        const T2<T> xa = aux[i];
        ((T2<T>*)d.out)[i] = {dd * xa.x - y.x, dd * xa.y - y.y};
    }
}

// (FRESH: d.aux, like the source, may be another block's of the same kernel.)
template <class T, int NC, int KIND, class TO, bool PL, bool FRESH>
__device__ __forceinline__ void stag_colour(const PassDesc& d, int x, int a, int V, T2<T> y, T alpha,
                                            SiteAcc<T, KIND>& loc) {
    if constexpr (FRESH) {
        stag_colour_of<T, NC, KIND, TO, PL>(d, (const T2<T>*)d.aux, x, a, V, y, alpha, loc);
    } else {
        const T2<T>* __restrict__ aux = (const T2<T>*)d.aux;
        stag_colour_of<T, NC, KIND, TO, PL>(d, aux, x, a, V, y, alpha, loc);
    }
}

// RECON = kLinksFx (FP64 only): `links` holds fixed-point limbs and links64
// the FP64 links. FRESH: see dslash_site_fresh.
constexpr int kLinksFx = 2;
template <class T, int NC, int RECON, int KIND, class TO, bool PL = false, bool FRESH = false>
__device__ __forceinline__ SiteAcc<T, KIND> stag_site(const PassDesc& d, const StagGeom& g, const void* links,
                                            T alpha, int x, const void* links64 = nullptr) {
    const int V = vlen(g);
    T2<T> y[NC];
    if constexpr (RECON == kLinksFx) dslash_site_fx<NC, FRESH>(links, links64, (const T2<T>*)d.src, x, g, y);
    else if constexpr (FRESH) dslash_site_fresh<T, NC, RECON, PL>(links, (const T2<T>*)d.src, x, g, y);
    else dslash_site<T, NC, RECON, PL>(links, (const T2<T>*)d.src, x, g, y);
    x = vsite(x, g);  // the site's index in the vectors
    SiteAcc<T, KIND> loc = 0;
#pragma unroll
    for (int a = 0; a < NC; ++a) stag_colour<T, NC, KIND, TO, PL, FRESH>(d, x, a, V, y[a], alpha, loc);
    return loc;
}

// The FP64 pass at one site by four lanes (consecutive lanes of a warp, lane & 3
// = the direction): each takes its direction's two hops, the entries' exponent
// is the largest of the four lanes', and the integer sums add across them.
// Lane a < NC then runs the epilogue of colour a. All lanes of the warp call it;
// on = false for those without a site.
template <int NC, int KIND, class TO, bool FRESH>
__device__ __forceinline__ double stag_site_fx4(const PassDesc& d, const StagGeom& g, const void* lfx,
                                                const void* links64, double alpha, int x, bool on) {
    const double2* src = (const double2*)d.src;
    const int mu = threadIdx.x & 3;
    const int q0 = gdiv(x, g, 0), q1 = gdiv(q0, g, 1), q2 = gdiv(q1, g, 2);
    const int c0 = x - q0 * g.L[0], c1 = q0 - q1 * g.L[1], c2 = q1 - q2 * g.L[2];
    const int L = g.L[mu];
    const int c = mu == 0 ? c0 : mu == 1 ? c1 : mu == 2 ? c2 : q2;
    const int stride = (mu > 0 ? g.L[0] : 1) * (mu > 1 ? g.L[1] : 1) * (mu > 2 ? g.L[2] : 1);
    const int par = ((mu > 0 ? c0 : 0) + (mu > 1 ? c1 : 0) + (mu > 2 ? c2 : 0)) & 1;
    const int xf = c == L - 1 ? x - (L - 1) * stride : x + stride;
    const int xb = c == 0 ? x + (L - 1) * stride : x - stride;
    double2 v[2][NC];
    unsigned e = 0, lows = 0;
#pragma unroll
    for (int b = 0; b < NC; ++b) {
        v[0][b] = v[1][b] = {0.0, 0.0};
        if (on) {
            const double2* vf = src + (size_t)vsite(xf, g) * NC + b;
            const double2* vb = src + (size_t)vsite(xb, g) * NC + b;
            v[0][b] = FRESH ? *vf : __ldg(vf);
            v[1][b] = FRESH ? *vb : __ldg(vb);
        }
        fx_bound(e, v[0][b]);
        fx_bound(e, v[1][b]);
        lows |= (unsigned)__double2loint(v[0][b].x) | (unsigned)__double2loint(v[0][b].y) |
                (unsigned)__double2loint(v[1][b].x) | (unsigned)__double2loint(v[1][b].y);
    }
    e = max(e, min(lows, 1u));  // 0 only where every entry is zero
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
    const unsigned field = fx_field(e);
    FxSum re[NC], im[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) re[a] = im[a] = {0, 0};
    if (on) {
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
            const bool fwd = dir == 0;
            const int4* __restrict__ U = (const int4*)lfx + fx_link<NC>(mu, fwd ? x : xb, g.V);
            const int flip = fwd ? -par : par - 1;
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                int rh, rl, ih, il;
                fx_split(v[dir][b].x, field, flip, rh, rl);
                fx_split(v[dir][b].y, field, flip, ih, il);
                const int zh = fwd ? -ih : ih, zl = fwd ? -il : il;
                const int wh = fwd ? rh : -rh, wl = fwd ? rl : -rl;
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    const int4 u = __ldg(U + (fwd ? a * NC + b : b * NC + a) * 32);
                    fx_mac(re[a], u.x, u.y, rh, rl);
                    fx_mac(im[a], u.x, u.y, ih, il);
                    fx_mac(re[a], u.z, u.w, zh, zl);
                    fx_mac(im[a], u.z, u.w, wh, wl);
                }
            }
        }
    }
    // this lane's colour of the sum over the four directions
    long long sr = 0, si = 0;
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        long long r = fx_units(re[a]), i = fx_units(im[a]);
        r += __shfl_xor_sync(0xffffffffu, r, 1);
        i += __shfl_xor_sync(0xffffffffu, i, 1);
        r += __shfl_xor_sync(0xffffffffu, r, 2);
        i += __shfl_xor_sync(0xffffffffu, i, 2);
        if (a == mu) { sr = r; si = i; }
    }
    if (!on || mu >= NC) return 0.0;
    double2 y = {fx_double(sr, field, 1), fx_double(si, field, 1)};
    if (e == 0) {
        y = {0.0, 0.0};
    } else if (!fx_in_range(field)) {
        const SiteVec<NC> r = dslash_site_f64<NC>(links64, src, x, g);
#pragma unroll
        for (int a = 0; a < NC; ++a)
            if (a == mu) y = r.y[a];
    }
    double loc = 0.0;
    stag_colour<double, NC, KIND, TO, true, FRESH>(d, vsite(x, g), mu, vlen(g), y, alpha, loc);
    return loc;
}

}  // namespace msc
