// Shared device-side definitions of the multi-shift CG engine.
//
// The engine runs CG-M (Algorithm 1, Sec. 2) for `nsys` independent systems
// that share one operator. A system has S shifts; its base shift (the
// smallest) is the one the Krylov sequence is built on, so its direction
// vector p_s is p itself and its zeta is exactly 1. Per-shift vectors live in
// global "slots" g = slot0 + s.
//
// Recurrences, textbook convention (alpha = step, beta = direction weight;
// the paper writes beta0 = -alpha and alpha for our beta):
//   alpha = R / P,          P = p^dag (A + sigma0) p
//   zeta_s' = zeta_s zeta_s^- alpha^- /
//             (alpha beta^- (zeta_s^- - zeta_s) + zeta_s^- alpha^- (1 + (sigma_s - sigma0) alpha))
//   alpha_s = alpha zeta_s' / zeta_s,     x_s += alpha_s p_s
//   r -= alpha (A + sigma0) p,  R' = r^dag r,  beta = R'/R
//   beta_s = beta (zeta_s'/zeta_s)^2,     p_s = zeta_s' r + beta_s p_s
//   p = r + beta p
// Shift s has met the tolerance when |zeta_s'| sqrt(R') <= tol |b|.
//
// The per-iteration scalar work (a few flops per shift) is done on the
// device by the last block of the kernel that completes the reduction it
// needs, so the host never waits inside an iteration (Sec. 3: the shift
// constants are computed on the GPU to avoid host round trips).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace msc {

constexpr int kThreads = 256;        // threads per block of every engine kernel
constexpr int kMaxBlocks = 2048;     // partial-sum slots per reduction row
constexpr int kMaxShifts = 128;      // shifts per system

enum : int {
    ST_RUNNING = 0,    // iterate
    ST_FINISHING = 1,  // the current iteration is the last one
    ST_DONE = 2,       // converged or capped
    ST_ERR_NOT_HPD = 4,
    ST_ERR_NONFINITE = 5,
};

// finalize actions of the last block of a reducing kernel
enum : int {
    FIN_NONE = 0,
    FIN_P = 1,        // P known: alpha, zeta', alpha_s
    FIN_R = 2,        // R' known: beta, beta_s, convergence, iteration++
    FIN_SETR = 3,     // R := reduction (reliable update)
    FIN_SETR_INIT = 4,// R := reduction at the start of a solve from a residual
    FIN_INIT = 5,     // R = |b|^2 at the start of a solve from x = 0
    FIN_STORE = 6,    // store the reduction in out_red[row]
};

struct SysScalars {
    double R, P, alpha, alpha_prev, beta, beta_prev;
    double bnorm2;    // |b|^2
    double tol2;      // tol^2
    double d;         // diagonal shift of the operator pass (m^2+sigma0 or sigma0)
    double tol2_acc;  // start-of-solve acceptance: done at once if R <= tol2_acc |b|^2
    double Rmax;      // largest iterated R since the last reliable update
    double delta2;    // reliable update once R <= delta2 * Rmax
    int status, it, max_iter, capped;
    int S, base, slot0, rhs;
    int freeze;
    int ru_every;     // reliable update at the latest after this many iterations (0: never)
    int since_ru;     // iterations since the last reliable update
    int ru;           // 1: the reliable-update kernels of this iteration run
    int nru;          // reliable updates done
    int last_fold;    // iteration count at the last reliable update's fold
};

struct SlotScalars {
    double sigma_rel;                   // sigma_s - sigma0
    double zeta, zeta_prev, zeta_new;
    double alpha_s, beta_s;
    double ratio;                       // zeta_new / zeta of this iteration
    int active;                         // still iterating
    int flag;                           // this iteration: 0 skip, 1 x only, 2 x and p_s
    int conv_iter;                      // iteration at which tol was met (-1)
    int pad;
    double tol2;                        // > 0: this shift's own tol^2 (relative to |b|^2)
                                        //      in place of the system's
};

// One pass of an operator kernel: which vectors, which scalars, which
// reduction. An array of these is indexed by blockIdx.y.
struct PassDesc {
    const void* src;    // vector the operator acts on
    const void* aux;    // vector multiplied by d (p or x); may equal src
    const double2* b;   // right-hand side (residual passes)
    void* out;          // output vector (may be null for residual norms)
    double d;           // diagonal shift
    int sys;            // gating system (-1: always run)
    int row;            // reduction row (-1: no reduction)
    int fin;            // FIN_*
    int gate;           // 0: run while the system iterates; 1: also only when its
                        //    reliable update is due
};

struct Engine {
    SysScalars* sys;
    SlotScalars* slot;
    double* partial;     // [rows][kMaxBlocks]
    unsigned* counter;   // [rows]
    double* out_red;     // [rows]
    // CUDA-graph conditional of this iteration's reliable-update body (0: none)
    // and the flag that lets exactly one system set it
    unsigned long long cond;
    int* cond_flag;
    // error word (bit 0: a bounded wait of a kernel ran out), read by the host
    // after each launch chunk; may be null
    unsigned* err;
};

// ---------------------------------------------------------------------------
// complex helpers (T2 = float2 or double2)
// ---------------------------------------------------------------------------
template <class T> struct C2;
template <> struct C2<float> { using t = float2; };
template <> struct C2<double> { using t = double2; };

template <class T2> __device__ __forceinline__ T2 cmul(T2 a, T2 b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// conj(a) * b
template <class T2> __device__ __forceinline__ T2 cmulc(T2 a, T2 b) {
    return {a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x};
}
template <class T2> __device__ __forceinline__ T2 cadd(T2 a, T2 b) { return {a.x + b.x, a.y + b.y}; }
template <class T2> __device__ __forceinline__ T2 csub(T2 a, T2 b) { return {a.x - b.x, a.y - b.y}; }
template <class T2, class T> __device__ __forceinline__ T2 cscale(T s, T2 a) { return {s * a.x, s * a.y}; }
template <class T2> __device__ __forceinline__ T2 cconj(T2 a) { return {a.x, -a.y}; }

// acc += a b, as four fused multiply-adds
template <class T2> __device__ __forceinline__ void cfma(T2& acc, T2 a, T2 b) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}
// acc -= conj(a) b, as four fused multiply-adds
template <class T2> __device__ __forceinline__ void cfms_conj(T2& acc, T2 a, T2 b) {
    acc.x = fma(-a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(-a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}

__device__ __forceinline__ int load_status(const SysScalars* s) {
    return __ldcg(&s->status);
}

// ---------------------------------------------------------------------------
// block reduction + "last block finalizes" (deterministic)
//
// An FP64 addition holds an SM's two FP64 lanes for 16 clocks a warp and takes
// about 100-150 clocks with its shuffle: in a 256-thread block the sum by
// shuffles in every warp (8 x 5 + 5 additions) and the scalar steps with
// their divisions in every warp took 5,200-5,500 clocks a step (k_persist,
// measured). So one warp sums the block's values from shared memory and runs
// the scalar steps alone, and it adds in fixed point: every value as a 63-bit
// integer in units of 2^-63 of the power of two above the largest, in two
// 32-bit limbs whose sums are exact, rounded to FP64 once. (2,000 clocks
// with FP64 additions by one warp.) The result does not depend on the order,
// and its error is below n 2^-63 of the largest value, under FP64's own.
// ---------------------------------------------------------------------------
constexpr int kRedThreads = 288;  // largest block that reduces

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// The parts of a float or double as a 63-bit integer of a common exponent.
template <class T> struct SumBits;
template <> struct SumBits<float> {
    static constexpr int kBias = 127 + 23 + 39, kInf = 255;
    __device__ static __forceinline__ int exponent(float v) { return max((__float_as_int(v) >> 23) & 255, 1); }
    __device__ static __forceinline__ long long aligned(float v, int top) {
        const int b = __float_as_int(v), e = (b >> 23) & 255;
        unsigned long long q = (unsigned long long)((b & 0x7fffff) | (e ? 0x800000 : 0)) << 39;
        asm("shr.u64 %0, %0, %1;" : "+l"(q) : "r"(top - max(e, 1)));
        return b < 0 ? -(long long)q : (long long)q;
    }
};
template <> struct SumBits<double> {
    static constexpr int kBias = 1023 + 52 + 10, kInf = 2047;
    __device__ static __forceinline__ int exponent(double v) { return max((__double2hiint(v) >> 20) & 2047, 1); }
    __device__ static __forceinline__ long long aligned(double v, int top) {
        const long long b = __double_as_longlong(v);
        const int e = (int)(b >> 52) & 2047;
        unsigned long long q = ((unsigned long long)b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
        q <<= 10;
        asm("shr.u64 %0, %0, %1;" : "+l"(q) : "r"(top - max(e, 1)));
        return b < 0 ? -(long long)q : (long long)q;
    }
};

// Sum over a warp of 64-bit integers below 2^47 in magnitude, in every lane.
__device__ __forceinline__ long long warp_add(long long x) {
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0xffffffu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(x >> 24));
    return ((long long)hi << 24) + lo;
}

// The sum over the warp's lanes of each lane's get(0) .. get(n - 1), in FP64
// in every lane; top: the largest exponent of this lane's values. K > 0: n = K,
// unrolled. At most kMaxBlocks values in all. Inf and NaN come out as in FP64
// additions.
template <class T, int K, class F>
__device__ __forceinline__ double warp_total_at(int top, int n, F get) {
    top = __reduce_max_sync(0xffffffffu, top);
    if (top == SumBits<T>::kInf) {
        double acc = 0.0;
        if constexpr (K > 0) {
#pragma unroll
            for (int i = 0; i < K; ++i) acc += (double)get(i);
        } else {
            for (int i = 0; i < n; ++i) acc += (double)get(i);
        }
        return __shfl_sync(0xffffffffu, warp_sum(acc), 0);
    }
    long long hi = 0, lo = 0;
    auto add = [&](int i) {
        const long long q = SumBits<T>::aligned(get(i), top);
        hi += q >> 32;
        lo += q & 0xffffffffll;
    };
    if constexpr (K > 0) {
#pragma unroll
        for (int i = 0; i < K; ++i) add(i);
    } else {
        for (int i = 0; i < n; ++i) add(i);
    }
    hi = warp_add(hi);
    lo = warp_add(lo);
    const double r = fma((double)hi, 0x1p32, (double)lo);
    const int k = top - SumBits<T>::kBias;  // the unit's exponent
    if (sizeof(T) == 8 && (k < -900 || k > 900)) return scalbn(r, k);
    return r * __hiloint2double((k + 1023) << 20, 0);
}

// The sum of get(0) .. get(n - 1), lane by lane.
template <class T, class F>
__device__ __forceinline__ double warp_total(int n, F get) {
    const int lane = threadIdx.x & 31, mine = (n - lane + 31) / 32;
    int top = 1;
    for (int i = lane; i < n; i += 32) top = max(top, SumBits<T>::exponent(get(i)));
    return warp_total_at<T, 0>(top, mine, [&](int i) { return get(lane + 32 * i); });
}

static __device__ __noinline__ double warp_total_f64(const double* sv, int n) {
    return warp_total<double>(n, [&](int i) { return sv[i]; });
}

// Sum of v over the block in FP64, valid in every lane of warp 0. sv:
// kRedThreads entries of shared memory, free again after the next
// __syncthreads.
template <class T>
__device__ __forceinline__ double block_sum(T v, T* sv) {
    __syncthreads();
    sv[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return 0.0;
    if constexpr (sizeof(T) == 8) return warp_total_f64(sv, (int)blockDim.x);
    else return warp_total<T>((int)blockDim.x, [&](int i) { return sv[i]; });
}

// Sum of n partials, valid in every lane of the calling warp: up to 32 K of
// them in registers, so that they are read once, all in flight.
template <int K>
__device__ __forceinline__ double sum_partials_k(const double* p, int n) {
    double v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int i = (threadIdx.x & 31) + 32 * k;
        v[k] = i < n ? __ldcg(p + i) : 0.0;
    }
    int top = 1;
#pragma unroll
    for (int k = 0; k < K; ++k) top = max(top, SumBits<double>::exponent(v[k]));
    return warp_total_at<double, K>(top, K, [&](int k) { return v[k]; });
}
// (Out of line, as the FP64 sum below: inlined, their registers make the FP64
// kernels spill.)
static __device__ __noinline__ double sum_partials(const double* p, int n) {
    if (n <= 128) return sum_partials_k<4>(p, n);
    if (n <= 640) return sum_partials_k<20>(p, n);
    return warp_total<double>(n, [&](int i) { return __ldcg(p + i); });
}

// Counts an arrival (one thread): earlier writes of this thread, and of those
// it has synchronised with, are visible to whoever sees the count.
__device__ __forceinline__ unsigned arrive(unsigned* counter) {
    unsigned t;
    asm volatile("atom.acq_rel.gpu.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
    return t;
}

// Whether the condition holds in every / any lane, with every lane's earlier
// memory accesses done before any lane's later ones (a vote alone orders none:
// lane 0 goes on to overwrite scalars that the others have read).
__device__ __forceinline__ int warp_all(int v) {
    const int all = __all_sync(0xffffffffu, v);
    __syncwarp();
    return all;
}
__device__ __forceinline__ int warp_any(int v) {
    const int any = __any_sync(0xffffffffu, v);
    __syncwarp();
    return any;
}

// Counts the calling block's arrival (warp 0, all its lanes); true in every
// lane in the last of `nblocks` blocks. A shuffle hands the count on but orders
// no memory, so the barrier after it is what lets the other lanes read what the
// other blocks published before they arrived.
__device__ __forceinline__ bool warp_arrive_last(unsigned* counter, int nblocks) {
    int last = 0;
    if ((threadIdx.x & 31) == 0) last = arrive(counter) == (unsigned)nblocks - 1;
    last = __shfl_sync(0xffffffffu, last, 0);
    __syncwarp();
    return last != 0;
}

// Publishes this block's sum of v to row `row`; returns true in every lane of
// warp 0 of the last of the `nblocks` blocks that reduce into that row to
// arrive (`bidx` = this block's index among them), with the fixed-order total.
template <class T>
__device__ __forceinline__ bool reduce_last_n(const Engine& e, int row, T v, double& total, int nblocks, int bidx) {
    __shared__ T sv[kRedThreads];
    const double s = block_sum(v, sv);
    if (threadIdx.x >= 32) return false;
    double* part = e.partial + (size_t)row * kMaxBlocks;
    if (threadIdx.x == 0) part[bidx] = s;
    if (!warp_arrive_last(&e.counter[row], nblocks)) return false;
    total = sum_partials(part, nblocks);
    if (threadIdx.x == 0) e.counter[row] = 0u;
    return true;
}

template <class T>
__device__ __forceinline__ bool reduce_last(const Engine& e, int row, T v, double& total) {
    return reduce_last_n(e, row, v, total, (int)gridDim.x, (int)blockIdx.x);
}

// True in thread 0 of the last block of a non-reducing kernel to be done.
__device__ __forceinline__ bool arrive_last_n(const Engine& e, int row, int nblocks) {
    __syncthreads();
    if (threadIdx.x != 0 || arrive(&e.counter[row]) != (unsigned)nblocks - 1) return false;
    e.counter[row] = 0u;
    return true;
}

// ---------------------------------------------------------------------------
// real-scalar vector helpers on 16-byte units
// ---------------------------------------------------------------------------
template <class T> struct U16;
template <> struct U16<float> { using t = float4; static constexpr int cpu = 2; };
template <> struct U16<double> { using t = double2; static constexpr int cpu = 1; };

__device__ __forceinline__ float4 axpy(float a, float4 x, float4 y) {
    return {fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w)};
}
__device__ __forceinline__ double2 axpy(double a, double2 x, double2 y) {
    return {fma(a, x.x, y.x), fma(a, x.y, y.y)};
}
// a*x + b*y
__device__ __forceinline__ float4 axpby(float a, float4 x, float b, float4 y) {
    return {fmaf(a, x.x, b * y.x), fmaf(a, x.y, b * y.y), fmaf(a, x.z, b * y.z), fmaf(a, x.w, b * y.w)};
}
__device__ __forceinline__ double2 axpby(double a, double2 x, double b, double2 y) {
    return {fma(a, x.x, b * y.x), fma(a, x.y, b * y.y)};
}
__device__ __forceinline__ float sq(float4 v) { return v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w; }
__device__ __forceinline__ double sq(double2 v) { return v.x * v.x + v.y * v.y; }
__device__ __forceinline__ float4 to_unit(double2 a, double2 b) {
    return {(float)a.x, (float)a.y, (float)b.x, (float)b.y};
}

// ---------------------------------------------------------------------------
// scalar recurrences, run by one warp (all its lanes)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void fin_P(const Engine& e, int j, double P) {
    const int lane = threadIdx.x & 31;
    SysScalars* s = &e.sys[j];
    const double R = s->R, ap = s->alpha_prev, bp = s->beta_prev;
    const int S = s->S, slot0 = s->slot0;
    const bool ok = (P > 0.0) && isfinite(P) && isfinite(R);
    const double alpha = R / P;
    __syncwarp();
    if (!ok) {
        if (lane == 0) s->status = isfinite(P) && isfinite(R) ? ST_ERR_NOT_HPD : ST_ERR_NONFINITE;
        return;
    }
    for (int k = lane; k < S; k += 32) {
        SlotScalars* q = &e.slot[slot0 + k];
        if (!q->active) { q->flag = 0; continue; }
        const double z = q->zeta, zp = q->zeta_prev;
        const double den = alpha * bp * (zp - z) + zp * ap * (1.0 + q->sigma_rel * alpha);
        // zeta'/zeta; exactly 1 for the base shift, whose division would be the
        // longest chain of a one-shift system
        const double w = q->sigma_rel == 0.0 && z == zp ? 1.0 : zp * ap / den;
        q->ratio = w;
        q->zeta_new = z * w;
        q->alpha_s = alpha * w;
    }
    if (lane == 0) { s->P = P; s->alpha = alpha; }
}

// COND: this kernel runs inside a chunk graph with conditional update nodes
// and sets the iteration's condition (a separate instance, so that kernels
// launched elsewhere contain no graph call and stay profilable).
template <bool COND>
__device__ __forceinline__ void fin_R(const Engine& e, int j, double Rn) {
    const int lane = threadIdx.x & 31;
    SysScalars* s = &e.sys[j];
    const double R = s->R, alpha = s->alpha;
    const double thr = s->tol2 * s->bnorm2;
    const int S = s->S, slot0 = s->slot0, it = s->it, freeze = s->freeze, maxit = s->max_iter;
    const double beta = Rn / R;
    const bool finite = isfinite(Rn);
    int all = 1;
    for (int k = lane; k < S; k += 32) {
        SlotScalars* q = &e.slot[slot0 + k];
        if (!q->active) continue;
        const double z = q->zeta, zn = q->zeta_new;
        const double ratio = q->ratio;
        q->beta_s = beta * ratio * ratio;
        const double tk = q->tol2 > 0.0 ? q->tol2 * s->bnorm2 : thr;
        const bool conv = (zn * zn * Rn <= tk) || !(fabs(zn) > 1e-290);
        if (conv && q->conv_iter < 0) q->conv_iter = it + 1;
        if (conv && freeze) { q->active = 0; q->flag = 1; }
        else q->flag = 2;
        q->zeta_prev = z;
        q->zeta = zn;
        if (q->conv_iter < 0) all = 0;
    }
    all = warp_all(all);
    if (lane == 0) {
        s->alpha_prev = alpha;
        s->beta_prev = beta;
        s->beta = beta;
        s->R = Rn;
        s->it = it + 1;
        if (!finite) s->status = ST_ERR_NONFINITE;
        else if (all) s->status = ST_FINISHING;
        else if (it + 1 >= maxit) { s->status = ST_FINISHING; s->capped = 1; }
        // reliable update (mixed precision): once the iterated residual has
        // fallen by delta below its largest value since the last update, or
        // after ru_every iterations, so the FP32 drift stays small relative
        // to the residual being iterated
        const double Rmax = fmax(s->Rmax, Rn);
        s->Rmax = Rmax;
        const int since = s->since_ru + 1;
        s->since_ru = since;
        const int ru = (s->ru_every > 0 && s->status == ST_RUNNING &&
                        (Rn <= s->delta2 * Rmax || since >= s->ru_every)) ? 1 : 0;
        s->ru = ru;
        if constexpr (COND) {
            if (ru && e.cond_flag && atomicExch(e.cond_flag, 1) == 0)
                cudaGraphSetConditional((cudaGraphConditionalHandle)e.cond, 1u);
        }
    }
}

// R := reduction. At the start of a solve from a residual, a system that
// already meets the tolerance is done with nothing to iterate.
__device__ __forceinline__ void fin_setR(const Engine& e, int j, double Rv, bool init) {
    const int lane = threadIdx.x & 31;
    SysScalars* s = &e.sys[j];
    const double thr = s->tol2_acc * s->bnorm2;
    const int S = s->S, slot0 = s->slot0;
    __syncwarp();
    if (!isfinite(Rv)) {
        if (lane == 0) s->status = ST_ERR_NONFINITE;
        return;
    }
    if (init && Rv <= thr) {
        for (int k = lane; k < S; k += 32) {
            e.slot[slot0 + k].active = 0;
            e.slot[slot0 + k].flag = 0;
            e.slot[slot0 + k].conv_iter = 0;
        }
        if (lane == 0) { s->R = Rv; s->status = ST_DONE; }
        return;
    }
    if (lane == 0) {
        s->R = Rv;
        s->Rmax = Rv;
        s->since_ru = 0;
        s->ru = 0;
        if (!init) {
            s->nru += 1;
            s->last_fold = s->it;  // the update's fold ran before this residual
        }
    }
}

// A fold of the system's FP32 x accumulators skips slot k when nothing has
// been added to it since the last fold: it stopped iterating (frozen at
// conv_iter, its last x update) no later than that fold.
__device__ __forceinline__ bool fold_skips(const SlotScalars* q, int last_fold) {
    return !q->active && q->conv_iter >= 0 && q->conv_iter <= last_fold;
}

__device__ __forceinline__ void fin_init(const Engine& e, int j, double b2) {
    const int lane = threadIdx.x & 31;
    SysScalars* s = &e.sys[j];
    const int S = s->S, slot0 = s->slot0;
    __syncwarp();
    if (lane == 0) {
        s->R = b2;
        s->Rmax = b2;
        s->since_ru = 0;
        s->ru = 0;
        s->bnorm2 = b2;
        if (!isfinite(b2)) s->status = ST_ERR_NONFINITE;
        else if (b2 == 0.0) s->status = ST_DONE;
    }
    if (b2 == 0.0) {
        for (int k = lane; k < S; k += 32) {
            e.slot[slot0 + k].active = 0;
            e.slot[slot0 + k].conv_iter = 0;
        }
    }
}

template <bool COND = false>
__device__ __forceinline__ void finalize(const Engine& e, const PassDesc& d, double total) {
    switch (d.fin) {
        case FIN_P: fin_P(e, d.sys, total); break;
        case FIN_R: fin_R<COND>(e, d.sys, total); break;
        case FIN_SETR: fin_setR(e, d.sys, total, false); break;
        case FIN_SETR_INIT: fin_setR(e, d.sys, total, true); break;
        case FIN_INIT: fin_init(e, d.sys, total); break;
        case FIN_STORE: if ((threadIdx.x & 31) == 0) e.out_red[d.row] = total; break;
        default: break;
    }
}

// Which system a block serves. Kernels over several systems use a 1-D grid
// whose blocks are dealt round-robin to the systems of the list `act`
// ({count, indices}, in device memory, rewritten by the host between graph
// launches) or to all `nsys` systems when act is null: block b serves system
// act[1 + b % count] as its block b / count of gridDim.x / count. Systems of
// one operator thus run side by side (shared matrix and link tiles are read
// from DRAM once), and as systems finish the same grid spreads over fewer.
struct SysBlock {
    int j;     // system
    int bx;    // block within the system
    int gx;    // blocks of the system
    bool ok;   // false: this block has no work
};

//
// A 2-D grid instead gives every system gridDim.y blocks of its own
// (blockIdx.x = system, so that the same block of every system runs at about
// the same time and matrix or link tiles come from L2 for all but one): used by passes that only some listed systems need (reliable updates, FP64
// checks), where the others' blocks exit at once and the busy ones keep the
// full device.
__device__ __forceinline__ SysBlock sys_block(int nsys, const int* act) {
    SysBlock s;
    if (gridDim.y > 1 || !act) {
        if (gridDim.y > 1) {
            s.j = blockIdx.x;
            s.bx = blockIdx.y;
            s.gx = gridDim.y;
            s.ok = s.j < nsys;
            return s;
        }
    }
    if (nsys == 1) {  // the list can hold no other (its two loads would come before every other)
        s.j = 0;
        s.bx = blockIdx.x;
        s.gx = gridDim.x;
        s.ok = true;
        return s;
    }
    const int na = act ? __ldg(act) : nsys;
    s.ok = na > 0;
    if (!s.ok) { s.j = s.bx = s.gx = 0; return s; }
    const int k = blockIdx.x % na;
    s.bx = blockIdx.x / na;
    s.gx = gridDim.x / na;
    s.ok = s.bx < s.gx;
    s.j = act ? __ldg(act + 1 + k) : k;
    return s;
}

// Gate at kernel entry: true if this pass has nothing to do.
__device__ __forceinline__ bool gated_off(const Engine& e, const PassDesc& d) {
    if (d.sys < 0) return false;
    if (load_status(&e.sys[d.sys]) != ST_RUNNING) return true;
    return d.gate == 1 && __ldcg(&e.sys[d.sys].ru) == 0;
}

}  // namespace msc
