// CG-M iterations of small staggered systems in one cooperative kernel.
//
// On a small lattice an iteration's three kernels take 25-37 us (4^4 to 16^4)
// for a few microseconds of work: each ends in a serial tail (fence, atomic,
// the last block's sums, divisions and scalar stores) and the next begins with
// a chain of dependent loads. Here the blocks stay resident: every block
// holds the scalars of all systems in shared memory and updates its own copy
// (the same sums in the same order, so all copies are equal), and the passes
// are separated by grid barriers:
//
//   t = D p, P terms           -> barrier -> alpha, zeta' (every block)
//   r -= alpha A p, |r|^2      -> barrier -> beta, beta_s, convergence
//   x_base, p                  -> arrive; x_s, p_s of the other shifts; wait
//
// A launch ends when every system has stopped, when one is due a reliable
// update, or after a number of iterations; block 0 then stores the scalars.
// The sums are those of the per-pass kernels up to their order and to where
// they are rounded (here one site per thread and a partial per 256 sites, or 64
// with four lanes a site), so that a solve by either agrees to rounding, not in
// its bits.
//
// Measured, one system, mixed, per iteration: 4^4 with 8 shifts 37 -> 12 us,
// 16^4 with one shift 29 -> 18 us (of which three barriers 3.8, the scalar
// steps 3.7, the passes with their sums 7); the 4^4 8-shift solve 15.0 ->
// 5.4 ms. FP64 (fixed-point passes): 4^4 16 us, 8^4 17 us.
//
// Barrier waits are bounded by the global timer (wait_ns): a wait that runs
// out sets the context's error word and the block returns; launches queued
// behind it find the word set and return at once.
#include <algorithm>

#include "async.cuh"
#include "stencil.cuh"

namespace msc {

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

struct GridBar {
    unsigned* word;
    unsigned target;
    uint64_t wait_ns;
    unsigned* err;
};

// Every thread's writes before are visible to the grid once it has arrived.
__device__ __forceinline__ void bar_arrive(GridBar& b) {
    __syncthreads();
    if (gridDim.x > 1 && threadIdx.x == 0) arrive(b.word);
    b.target += gridDim.x;
}

// False (in every thread) if the wait ran out.
__device__ __forceinline__ bool bar_wait(GridBar& b) {
    __shared__ int s_ok;
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    if (threadIdx.x == 0) {
        int ok = 1;
        if (ld_acquire(b.word) < b.target) {
            const uint64_t t0 = global_ns();
            while (ld_acquire(b.word) < b.target)
                if (global_ns() - t0 > b.wait_ns) {
                    ok = 0;
                    if (b.err) atomicOr(b.err, 1u);
                    break;
                }
        }
        s_ok = ok;
    }
    __syncthreads();
    const bool ok = s_ok != 0;
    __syncthreads();
    return ok;
}

// The sums of every running system's partials and the scalar step FIN on
// them, one warp per system (in the order of reduce_last_n). The partials of
// the two passes lie in halves of a row: a block may write those of the second
// pass while another still sums those of the first.
constexpr int kHalfRow = kMaxBlocks / 2;
//
// The scalars that the vector loops use are stored in their type: a
// conversion from FP64 costs a warp 16 clocks of the FP64 lanes, and three of
// them per shift in every thread were most of the update (13,000 of 15,000
// clocks an iteration at 11 shifts).
template <class T> struct ShiftCoefs {
    T alpha, zeta, beta;
    int flag;
};
template <class T> struct SysCoefs {
    T alpha, beta;
};
template <int FIN, class T>
__device__ __forceinline__ void persist_finalize(const Engine& e, int nsys, int chunks, ShiftCoefs<T>* cs, SysCoefs<T>* cy) {
    const double* part = e.partial + (FIN == FIN_P ? 0 : kHalfRow);
    for (int j = threadIdx.x >> 5; j < nsys; j += (int)(blockDim.x >> 5)) {
        if (e.sys[j].status != ST_RUNNING) continue;
        const double tot = sum_partials(part + (size_t)j * kMaxBlocks, chunks);
        if (FIN == FIN_P) fin_P(e, j, tot);
        else fin_R<false>(e, j, tot);
        __syncwarp();
        const SysScalars& y = e.sys[j];
        const int lane = threadIdx.x & 31;
        if (FIN == FIN_P) {
            if (lane == 0) cy[j].alpha = (T)y.alpha;
        } else {
            if (lane == 0) cy[j].beta = (T)y.beta;
            for (int k = lane; k < y.S; k += 32) {
                const SlotScalars& q = e.slot[y.slot0 + k];
                cs[y.slot0 + k] = {(T)q.alpha_s, (T)q.zeta_new, (T)q.beta_s, q.flag};
            }
        }
    }
    __syncthreads();
}

template <class D>
__device__ __forceinline__ void copy_words(D* to, const D* from, int count) {
    static_assert(sizeof(D) % 8 == 0, "copied as 8-byte words");
    const int n = count * (int)(sizeof(D) / 8);
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        ((unsigned long long*)to)[i] = __ldcg((const unsigned long long*)from + i);
}

constexpr int kShiftBatch = 4;  // shifts whose loads are in flight together in the update

// FX4 (FP64): four lanes share a site (stag_site_fx4), 64 sites to a task
// instead of 256. Chosen up to kFx4PersistSites sites of all systems, where a
// pass is the latency of one site's instructions: 8^4 16.9 us an iteration
// against 27.6, 4 x 8^4 24.0 against 27.8, but 12^4 31.9 against 27.6.
// BPS blocks per SM: FP64 with a thread per site at one (255 registers) when no
// more blocks are wanted than SMs (8^4: 27.6 us against 32.7 at two, which
// spill), at two otherwise (16^4: 44.9 against 47.0).
constexpr int64_t kFx4PersistSites = 16384;

template <class T, int NC, int RECON, int BPS, bool FX4>
__global__ void __launch_bounds__(kThreads, BPS) k_persist(PersistArgs a) {
    using V = typename U16<T>::t;
    extern __shared__ unsigned long long dyn[];
    __shared__ SiteAcc<T, PASS_A> sv[kRedThreads];
    const int nsys = a.nsys;
    SysScalars* ss = (SysScalars*)dyn;
    SlotScalars* sl = (SlotScalars*)(ss + nsys);
    PassDesc* k1 = (PassDesc*)(sl + a.nslots);
    PassDesc* k2 = k1 + nsys;
    SysCoefs<T>* cy = (SysCoefs<T>*)(k2 + nsys);
    ShiftCoefs<T>* cs = (ShiftCoefs<T>*)(((uintptr_t)(cy + nsys) + 15) / 16 * 16);
    __shared__ unsigned s_err;
    if (threadIdx.x == 0) s_err = a.e.err ? ld_acquire(a.e.err) : 0u;
    copy_words(ss, a.e.sys, nsys);
    copy_words(sl, a.e.slot, a.nslots);
    copy_words(k1, a.k1, nsys);
    copy_words(k2, a.k2, nsys);
    __syncthreads();
    if (s_err) return;  // an earlier launch's wait ran out: its results are void
    Engine e = a.e;
    e.sys = ss;
    e.slot = sl;
    const StagGeom& g = a.g;
    const int nh = vlen(g);
    constexpr int kSites = FX4 ? kThreads / 4 : kThreads;
    const int chunks = (nh + kSites - 1) / kSites;
    const int ntask = nsys * chunks;
    const int64_t upv = a.v.npad / U16<T>::cpu;
    const int vchunks = (int)((upv + kThreads - 1) / kThreads);
    const int nvtask = nsys * vchunks;
    GridBar bar{a.bar, a.absent, a.wait_ns, a.e.err};
    bool fine = true;
    for (int it = 0; it < a.iters; ++it) {
        bool go = false, ru = false;
        for (int j = 0; j < nsys; ++j) {
            go = go || ss[j].status == ST_RUNNING;
            ru = ru || (ss[j].status == ST_RUNNING && ss[j].ru);
        }
        if (!go || ru) break;
        // t = D p and the P terms
        for (int q = blockIdx.x; q < ntask; q += gridDim.x) {
            const int j = q / chunks, ch = q - j * chunks;
            if (ss[j].status != ST_RUNNING) continue;
            SiteAcc<T, PASS_A> local = 0;
            if constexpr (FX4) {
                const int h = ch * kSites + (threadIdx.x >> 2);
                local = stag_site_fx4<NC, PASS_A, double, true>(k1[j], g, a.links, a.links64, T(0),
                                                                 pass_site<true>(h < nh ? h : 0, g), h < nh);
            } else {
                const int h = ch * kSites + threadIdx.x;
                if (h < nh)
                    local = stag_site<T, NC, RECON, PASS_A, T, true, true>(k1[j], g, a.links, T(0),
                                                                           pass_site<true>(h, g), a.links64);
            }
            const double s = block_sum(local, sv);
            if (threadIdx.x == 0) e.partial[(size_t)j * kMaxBlocks + ch] = s;
        }
        bar_arrive(bar);
        fine = bar_wait(bar);
        if (!fine) break;
        persist_finalize<FIN_P>(e, nsys, chunks, cs, cy);
        // r -= alpha A p and |r|^2
        for (int q = blockIdx.x; q < ntask; q += gridDim.x) {
            const int j = q / chunks, ch = q - j * chunks;
            if (ss[j].status != ST_RUNNING) continue;
            SiteAcc<T, PASS_B> local = 0;
            if constexpr (FX4) {
                const int h = ch * kSites + (threadIdx.x >> 2);
                local = stag_site_fx4<NC, PASS_B, double, true>(k2[j], g, a.links, a.links64, cy[j].alpha,
                                                                 pass_site<false>(h < nh ? h : 0, g), h < nh);
            } else {
                const int h = ch * kSites + threadIdx.x;
                if (h < nh)
                    local = stag_site<T, NC, RECON, PASS_B, T, true, true>(k2[j], g, a.links, cy[j].alpha,
                                                                           pass_site<false>(h, g), a.links64);
            }
            const double s = block_sum(local, sv);
            if (threadIdx.x == 0) e.partial[(size_t)j * kMaxBlocks + kHalfRow + ch] = s;
        }
        bar_arrive(bar);
        fine = bar_wait(bar);
        if (!fine) break;
        persist_finalize<FIN_R>(e, nsys, chunks, cs, cy);
        // the base shift's x and p
        for (int q = blockIdx.x; q < nvtask; q += gridDim.x) {
            const int j = q / vchunks;
            const int64_t i = (int64_t)(q - j * vchunks) * kThreads + threadIdx.x;
            const int st = ss[j].status;
            if ((st != ST_RUNNING && st != ST_FINISHING) || i >= upv) continue;
            const V rv = ((const V*)a.v.r)[(size_t)j * upv + i];
            V* p = (V*)a.v.p + (size_t)j * upv + i;
            const V pv = *p;
            const int b = ss[j].slot0 + ss[j].base;
            if (cs[b].flag) {
                V* x = (V*)a.v.xit + (size_t)b * upv + i;
                *x = axpy(cs[b].alpha, pv, *x);
            }
            *p = axpy(cy[j].beta, pv, rv);
        }
        bar_arrive(bar);
        // the other shifts
        for (int q = blockIdx.x; q < nvtask; q += gridDim.x) {
            const int j = q / vchunks;
            const int64_t i = (int64_t)(q - j * vchunks) * kThreads + threadIdx.x;
            const int st = ss[j].status, S = ss[j].S, base = ss[j].base, slot0 = ss[j].slot0;
            if ((st != ST_RUNNING && st != ST_FINISHING) || S == 1 || i >= upv) continue;
            const V rv = ((const V*)a.v.r)[(size_t)j * upv + i];
            V* ps = (V*)a.v.ps + (size_t)slot0 * upv + i;
            V* xs = (V*)a.v.xit + (size_t)slot0 * upv + i;
            for (int k0 = 0; k0 < S; k0 += kShiftBatch) {
                V xv[kShiftBatch], pk[kShiftBatch];
                int f[kShiftBatch];
#pragma unroll
                for (int u = 0; u < kShiftBatch; ++u) {
                    const int k = k0 + u;
                    f[u] = k < S && k != base ? cs[slot0 + k].flag : 0;
                    if (f[u]) {
                        pk[u] = ps[(size_t)k * upv];
                        xv[u] = xs[(size_t)k * upv];
                    }
                }
#pragma unroll
                for (int u = 0; u < kShiftBatch; ++u) {
                    if (!f[u]) continue;
                    const ShiftCoefs<T> c = cs[slot0 + k0 + u];
                    xs[(size_t)(k0 + u) * upv] = axpy(c.alpha, pk[u], xv[u]);
                    if (f[u] == 2) ps[(size_t)(k0 + u) * upv] = axpby(c.zeta, rv, c.beta, pk[u]);
                }
            }
        }
        fine = bar_wait(bar);
        if (!fine) break;
        for (int j = threadIdx.x; j < nsys; j += blockDim.x)
            if (ss[j].status == ST_FINISHING) ss[j].status = ST_DONE;
        __syncthreads();
    }
    if (blockIdx.x != 0) return;
    __syncthreads();
    const int nw = nsys * (int)(sizeof(SysScalars) / 8), mw = a.nslots * (int)(sizeof(SlotScalars) / 8);
    for (int i = threadIdx.x; i < nw; i += blockDim.x) ((unsigned long long*)a.e.sys)[i] = ((unsigned long long*)ss)[i];
    for (int i = threadIdx.x; i < mw; i += blockDim.x) ((unsigned long long*)a.e.slot)[i] = ((unsigned long long*)sl)[i];
}

static size_t persist_smem(int nsys, int nslots) {
    return (size_t)nsys * (sizeof(SysScalars) + 2 * sizeof(PassDesc) + sizeof(SysCoefs<double>)) +
           (size_t)nslots * (sizeof(SlotScalars) + sizeof(ShiftCoefs<double>)) + 32;
}

// The line: 256-site blocks of all systems, against three kernels an
// iteration. One system at 16^4 (256 blocks): 18 us an iteration against 29;
// 12 systems at 16^4 (3,072): the 12-shift quadratic form and its gradients
// 35.7 ms against 40.7 with the refinement's passes left to k_stag_group;
// 8,192: the same as 4,096. Beyond, the grouped passes share their links.
constexpr int kPersistTasks = 4096;

bool persist_applies(const OpDev& op, int prec, int nsys, int nslots) {
    if (op.kind != OP_STAGGERED || (prec == PREC_F64 && !op.linksfx)) return false;
    const int64_t chunks = (vlen(op.g) + kThreads - 1) / kThreads;
    return nsys * chunks <= kPersistTasks && chunks <= kHalfRow && persist_smem(nsys, nslots) <= 40 * 1024;
}

template <class T, int NC, int RECON, int BPS, bool FX4 = false>
static cudaError_t launch_persist_t(PersistArgs a, int sms, cudaStream_t st) {
    auto k = k_persist<T, NC, RECON, BPS, FX4>;
    const size_t sm = persist_smem(a.nsys, a.nslots);
    int per_sm = 0;
    cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)k, kThreads, sm);
    if (err != cudaSuccess) return err;
    const int sites = FX4 ? kThreads / 4 : kThreads;
    const int64_t tasks = a.nsys * (int64_t)((vlen(a.g) + sites - 1) / sites);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(tasks, (int64_t)per_sm * sms));
    void* ptrs[] = {&a};
    return cudaLaunchCooperativeKernel((const void*)k, dim3(grid), dim3(kThreads), ptrs, sm, st);
}

template <int NC>
static cudaError_t launch_persist_nc(const OpDev& op, int prec, const PersistArgs& a, int sms, cudaStream_t st) {
    if (prec == PREC_F64) {
        const int64_t V = vlen(a.g);
        if (a.nsys * V <= kFx4PersistSites) return launch_persist_t<double, NC, kLinksFx, 2, true>(a, sms, st);
        if (a.nsys * ((V + kThreads - 1) / kThreads) <= sms) return launch_persist_t<double, NC, kLinksFx, 1>(a, sms, st);
        return launch_persist_t<double, NC, kLinksFx, 2>(a, sms, st);
    }
    if (op.recon) return launch_persist_t<float, NC, 1, 2>(a, sms, st);
    return launch_persist_t<float, NC, 0, 2>(a, sms, st);
}

cudaError_t launch_persist(const OpDev& op, int prec, const PersistArgs& a, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    return op.nc == 3 ? launch_persist_nc<3>(op, prec, a, sms, st) : launch_persist_nc<2>(op, prec, a, sms, st);
}

}  // namespace msc
