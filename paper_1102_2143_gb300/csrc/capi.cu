// C ABI of libmsc and the host driver of the multi-shift solves.
//
// CG-M (Algorithm 1, Sec. 2) runs entirely on the device: the host only
// launches CUDA graphs, each holding a chunk of iterations (operator pass,
// residual update, fused multi-shift update per iteration), and reads a few
// bytes of status after each chunk. In mixed precision each iteration ends
// with a conditional graph node that runs an FP64 reliable update of a
// system's base residual when the device decided one is due (its residual
// fell by reliable_delta, or reliable_every iterations passed). After the
// multi-shift stage the FP64 true residual of every shift is measured and
// each shift above the tolerance is refined by a single-shift solve
// warm-started from its x_s. The same driver serves batches of uneven
// systems (msc_solve_batched) and, with its own kernels, BiCGStab-M for
// non-Hermitian families (msc_solve_nonherm).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/msc.h"
#include "bicgstab.cuh"
#include "engine.h"

using namespace msc;

namespace {

struct Buf {
    void* p = nullptr;
    size_t bytes = 0;
};

// desc sections, each `rows` entries long
enum { D_INIT = 0, D_K1, D_K2, D_RUA, D_RUC, D_RIA, D_RIC, D_AP1, D_AP2, D_NSECT };

struct GraphEntry {
    cudaGraphExec_t exec = nullptr;
    int gen = -1;
    int kernels = 0;       // kernels launched unconditionally per launch
    int cond_chunk = 0;    // iterations with a conditional update body (0: none)
    int cond_kernels = 0;  // kernels in one such body
};

long g_op_uid = 0;

// A named range on the profiler timeline for the lifetime of the object (a
// no-op unless a profiling tool is attached).
struct Range {
    explicit Range(const char* name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
    Range(const Range&) = delete;
    Range& operator=(const Range&) = delete;
};

}  // namespace

// small results of the set-up kernels, behind the context's error word
constexpr size_t kSetupWord = 4, kSetupDev = 8, kErrBytes = kSetupDev + kLinkDevs * sizeof(double);

struct msc_ctx {
    int device = 0;
    int num_sms = 0;
    cudaStream_t user = nullptr;
    cudaStream_t work = nullptr;
    cudaEvent_t ev_sync = nullptr;
    cudaEvent_t prof[4] = {nullptr, nullptr, nullptr, nullptr};
    // device workspace (grow only; `gen` changes whenever a buffer moves)
    Buf sys, slot, partial, counter, out_red, descs;
    Buf b64, x64, t64, r, p, t, ps, xit;
    Buf coef, force;  // adjoint: weights c_s and a link-shaped output
    Buf bvb;          // batched solves: virtual-block tables
    Buf btab;         // batched solves: system table, operator table, block maps
    Buf actb;         // {count, indices} of the systems still iterating (refinement)
    Buf bcg;          // BiCGStab-M scalars: one BcgSys, then S BcgSlot
    Buf condf;        // one flag per iteration of a chunk graph (conditional update bodies)
    Buf pb, px0, ptmp;// polynomial right-hand sides: b_s, x_s0, two scratch vectors per shift
    Buf gbar;         // barrier word of the cooperative iterations
    Buf errf;         // device error word (bit 0: a bounded wait in a kernel ran out), then
                      // scratch words of the operators' set-up (offsets kSetupWord, kSetupDev)
    unsigned* h_err = nullptr;  // pinned copy of it
    uint64_t wait_ns = 2000000000ull;  // limit of a kernel's wait on its own copies or grid barrier
    int use_tile = 0;  // one-system FP32 stencil passes stage their links (when the lattice tiles)
    int test_no_copy = 0;  // tests only: the staged passes issue no copies, so their waits run out
    int test_absent = 0;   // tests only: grid barriers wait for an arrival that never comes
    int use_persist = 1;  // small staggered stages iterate in one cooperative kernel
    int use_cond = 1; // build reliable updates as conditional graph nodes
    int* h_flags = nullptr;  // pinned copy of the conditional flags of a chunk
    int* h_act = nullptr;
    int64_t h_act_cap = 0;
    int64_t rows_cap = 0;  // rows the desc sections were laid out for
    int gen = 0;
    // pinned host mirrors
    SysScalars* h_sys = nullptr;
    SlotScalars* h_slot = nullptr;
    double* h_red = nullptr;
    PassDesc* h_desc = nullptr;
    int64_t h_rows = 0, h_slots = 0;
    std::map<std::string, GraphEntry> graphs;
    long launches = 0;
};

struct msc_op {
    msc_ctx* ctx = nullptr;
    long uid = 0;
    OpDev dev{};
    int64_t nnzb = 0;
    // staggered: the parity-reduced operators of sources on even (0) or odd
    // (1) sites, made on first use; they share this operator's device data
    msc_op* view[2] = {nullptr, nullptr};
    bool is_view = false;
};

#define CK(call)                                      \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess) return cuda_status(e_);\
    } while (0)

static int cuda_status(cudaError_t e) {
    return e == cudaErrorMemoryAllocation ? MSC_ERR_OOM : MSC_ERR_CUDA;
}

static bool is_device_ptr(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Grows a workspace buffer (never while the work stream is capturing). The
// new memory is zeroed on the context's work stream: the work stream is
// non-blocking, so a cudaMemset on the legacy default stream would not be
// ordered before the kernels that read the buffer (recycled memory then held
// the previous owner's reduction counters and accumulators).
static cudaError_t grow(msc_ctx* c, Buf& b, size_t bytes, bool& moved) {
    if (bytes <= b.bytes) return cudaSuccess;
    if (b.p) {
        cudaError_t e = cudaStreamSynchronize(c->work);
        if (e != cudaSuccess) return e;
        cudaFree(b.p);
    }
    b.p = nullptr;
    b.bytes = 0;
    size_t want = bytes + bytes / 8;
    cudaError_t e = cudaMalloc(&b.p, want);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(b.p, 0, want, c->work);
    if (e != cudaSuccess) return e;
    b.bytes = want;
    moved = true;
    return cudaSuccess;
}

static int ensure_ws(msc_ctx* c, int64_t npad, int64_t rows, int64_t slots, int64_t rhs, size_t elem) {
    bool moved = false;
    rows = std::max<int64_t>(rows, 3);
    slots = std::max<int64_t>(slots, 1);
    rhs = std::max<int64_t>(rhs, 1);
    if (rows > c->rows_cap) {
        c->rows_cap = rows;
        moved = true;
    }
    const int64_t R = c->rows_cap;
    CK(grow(c, c->sys, sizeof(SysScalars) * R, moved));
    CK(grow(c, c->slot, sizeof(SlotScalars) * std::max(slots, R), moved));
    CK(grow(c, c->partial, sizeof(double) * kMaxBlocks * std::max(slots, R), moved));
    CK(grow(c, c->counter, sizeof(unsigned) * std::max(slots, R), moved));
    CK(grow(c, c->out_red, sizeof(double) * std::max(slots, R), moved));
    CK(grow(c, c->descs, sizeof(PassDesc) * D_NSECT * R, moved));
    CK(grow(c, c->b64, (size_t)rhs * npad * 16, moved));
    CK(grow(c, c->x64, (size_t)slots * npad * 16, moved));
    CK(grow(c, c->t64, (size_t)std::max(rows, slots) * npad * 16, moved));
    // per-system vectors: this call's rows (rows_cap only lays out the
    // descriptor sections; a large batch before must not scale them)
    CK(grow(c, c->r, (size_t)rows * npad * elem, moved));
    CK(grow(c, c->p, (size_t)rows * npad * elem, moved));
    CK(grow(c, c->t, (size_t)rows * npad * elem, moved));
    CK(grow(c, c->ps, (size_t)slots * npad * elem, moved));
    CK(grow(c, c->xit, (size_t)slots * npad * 8, moved));
    if (moved) c->gen++;
    const int64_t hs = std::max(slots, R);
    if (R > c->h_rows || hs > c->h_slots) {
        if (c->h_sys) cudaFreeHost(c->h_sys);
        if (c->h_slot) cudaFreeHost(c->h_slot);
        if (c->h_red) cudaFreeHost(c->h_red);
        if (c->h_desc) cudaFreeHost(c->h_desc);
        CK(cudaMallocHost((void**)&c->h_sys, sizeof(SysScalars) * R));
        CK(cudaMallocHost((void**)&c->h_slot, sizeof(SlotScalars) * hs));
        CK(cudaMallocHost((void**)&c->h_red, sizeof(double) * hs));
        CK(cudaMallocHost((void**)&c->h_desc, sizeof(PassDesc) * D_NSECT * R));
        c->h_rows = R;
        c->h_slots = hs;
    }
    return MSC_OK;
}

static PassDesc* dsec(msc_ctx* c, int s) { return (PassDesc*)c->descs.p + (size_t)s * c->rows_cap; }
static PassDesc* hsec(msc_ctx* c, int s) { return c->h_desc + (size_t)s * c->rows_cap; }

static cudaError_t upload_sec(msc_ctx* c, int s, int count) {
    return cudaMemcpyAsync(dsec(c, s), hsec(c, s), sizeof(PassDesc) * count, cudaMemcpyHostToDevice,
                           c->work);
}

static Engine engine_of(msc_ctx* c) {
    Engine e{};
    e.sys = (SysScalars*)c->sys.p;
    e.slot = (SlotScalars*)c->slot.p;
    e.partial = (double*)c->partial.p;
    e.counter = (unsigned*)c->counter.p;
    e.out_red = (double*)c->out_red.p;
    e.err = (unsigned*)c->errf.p;
    return e;
}

// FP32 vectors of a staggered operator are colour-planar (see VecSet).
static VecSet vecs_of(msc_ctx* c, int prec, int64_t npad, const OpDev& A) {
    VecSet v;
    if (A.kind == OP_STAGGERED && prec == PREC_F32) {
        v.pl_nc = A.nc;
        v.pl_V = vlen(A.g);
    }
    v.r = c->r.p;
    v.p = c->p.p;
    v.t = c->t.p;
    v.ps = c->ps.p;
    v.x64 = (double2*)c->x64.p;
    v.xit = prec == PREC_F32 ? c->xit.p : c->x64.p;
    v.b64 = (const double2*)c->b64.p;
    v.npad = npad;
    return v;
}

static PassDesc mkdesc(const void* src, const void* aux, const double2* b, void* out, double d,
                       int sys, int row, int fin) {
    PassDesc p;
    p.src = src;
    p.aux = aux;
    p.b = b;
    p.out = out;
    p.d = d;
    p.sys = sys;
    p.row = row;
    p.fin = fin;
    p.gate = 0;
    return p;
}

// the same pass, run only in iterations where the system's reliable update is due
static PassDesc ru_pass(PassDesc d) {
    d.gate = 1;
    return d;
}

// per_system: a whole grid per pass (passes only some systems need:
// reliable updates, FP64 residual checks); otherwise the passes share one
// grid over the active list `act` (see sys_block).
static cudaError_t op_pass(msc_ctx* c, const OpDev& A, int prec, int kind, int out_f32, int sec,
                           int npass, const Engine* eng = nullptr, const int* act = nullptr,
                           bool per_system = false) {
    Engine e = eng ? *eng : engine_of(c);
    c->launches++;
    if (A.kind == OP_STAGGERED) {
        if (!per_system && npass == 1 && prec == PREC_F32 && (kind == PASS_A || kind == PASS_B) && A.recon &&
            c->use_tile && stag_tile_fits(A.g, A.nc))
            return launch_stag_tile(A, kind, e, dsec(c, sec), c->wait_ns, c->test_no_copy, c->work);
        if (!per_system && stag_group_applies(A, prec, kind, npass))
            return launch_stag_group(A, kind, e, dsec(c, sec), npass, c->work, act);
        return launch_stag_pass(A, prec, kind, out_f32, e, dsec(c, sec), npass, c->work, act, per_system);
    }
    return launch_bsr_pass(A, prec, kind, out_f32, e, dsec(c, sec), npass, c->work, act, per_system,
                           npass == 1 ? hsec(c, sec) : nullptr);
}


// One chunk of `chunk` iterations for `nsys` systems. In mixed precision each
// iteration ends with the reliable-update kernels, which only do work for the
// systems whose update is due (flag set by the iteration's finalize).
static cudaError_t enqueue_chunk(msc_ctx* c, const OpDev& A, int prec, int nsys, int chunk,
                                 bool reliable, bool profile, int64_t npad, int group, int groups,
                                 int& kernels) {
    Engine e = engine_of(c);
    VecSet v = vecs_of(c, prec, npad, A);
    const int* act = (const int*)c->actb.p;
    kernels = 0;
    for (int it = 0; it < chunk; ++it) {
        const bool prof = profile && it == 0;
        if (prof) cudaEventRecordWithFlags(c->prof[0], c->work, cudaEventRecordExternal);
        cudaError_t err;
        if (group > 0) {
            c->launches++;
            err = launch_bsr_multi(A, e, dsec(c, D_K1), nsys, act, group, groups, c->work);
        } else {
            err = op_pass(c, A, prec, PASS_A, 0, D_K1, nsys, &e, act);
        }
        if (err != cudaSuccess) return err;
        if (prof) cudaEventRecordWithFlags(c->prof[1], c->work, cudaEventRecordExternal);
        if (A.kind == OP_STAGGERED) err = op_pass(c, A, prec, PASS_B, 0, D_K2, nsys, &e, act);
        else err = launch_axpy_norm(prec, e, v, dsec(c, D_K2), nsys, c->work, act);
        if (err != cudaSuccess) return err;
        if (prof) cudaEventRecordWithFlags(c->prof[2], c->work, cudaEventRecordExternal);
        err = launch_update(prec, e, v, nsys, c->work, act);
        if (err != cudaSuccess) return err;
        if (prof) cudaEventRecordWithFlags(c->prof[3], c->work, cudaEventRecordExternal);
        kernels += 3;
        if (reliable) {
            err = launch_fold(e, v, nsys, 1, c->work, act, true);
            if (err != cudaSuccess) return err;
            kernels++;
            if (A.kind == OP_STAGGERED) {
                err = op_pass(c, A, PREC_F64, PASS_A, 0, D_RUA, nsys, &e, act, true);
                if (err != cudaSuccess) return err;
                kernels++;
            }
            err = op_pass(c, A, PREC_F64, PASS_C, 1, D_RUC, nsys, &e, act, true);
            if (err != cudaSuccess) return err;
            kernels++;
        }
    }
    return cudaSuccess;
}

static cudaError_t begin_capture_into(cudaStream_t st, cudaGraph_t g, const std::vector<cudaGraphNode_t>& deps) {
    return cudaStreamBeginCaptureToGraph(st, g, deps.empty() ? nullptr : deps.data(), nullptr, deps.size(),
                                         cudaStreamCaptureModeThreadLocal);
}

// The nodes the next captured operation would depend on (copied).
static cudaError_t capture_tail(cudaStream_t st, std::vector<cudaGraphNode_t>& tail) {
    cudaStreamCaptureStatus cs;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(st, &cs, nullptr, nullptr, &deps, nullptr, &nd);
    if (e != cudaSuccess) return e;
    tail.assign(deps, deps + nd);
    return cudaSuccess;
}

// A chunk graph whose reliable-update kernels sit in one conditional IF node
// per iteration: the iteration's residual kernel sets the condition on the
// device when some system's update is due, so iterations without an update
// launch nothing for it.
static cudaError_t build_chunk_graph_cond(msc_ctx* c, const OpDev& A, int prec, int nsys, int chunk,
                                          bool profile, int64_t npad, int group, int groups,
                                          cudaGraph_t* out, int& kernels) {
    bool moved = false;
    cudaError_t err = grow(c, c->condf, sizeof(int) * chunk, moved);
    if (err != cudaSuccess) return err;
    if (moved) c->gen++;
    int* flags = (int*)c->condf.p;
    cudaGraph_t g = nullptr;
    err = cudaGraphCreate(&g, 0);
    if (err != cudaSuccess) return err;
    VecSet v = vecs_of(c, prec, npad, A);
    std::vector<cudaGraphNode_t> tail;
    kernels = 0;
    for (int it = 0; it < chunk && err == cudaSuccess; ++it) {
        cudaGraphConditionalHandle h = 0;
        err = cudaGraphConditionalHandleCreate(&h, g, 0, cudaGraphCondAssignDefault);
        if (err != cudaSuccess) break;
        Engine e = engine_of(c);
        Engine e2 = e;
        e2.cond = (unsigned long long)h;
        e2.cond_flag = flags + it;
        err = begin_capture_into(c->work, g, tail);
        if (err != cudaSuccess) break;
        const bool prof = profile && it == 0;
        if (it == 0) err = cudaMemsetAsync(flags, 0, sizeof(int) * chunk, c->work);
        if (prof) cudaEventRecordWithFlags(c->prof[0], c->work, cudaEventRecordExternal);
        const int* act = (const int*)c->actb.p;
        if (err == cudaSuccess) {
            if (group > 0) err = launch_bsr_multi(A, e, dsec(c, D_K1), nsys, act, group, groups, c->work);
            else err = op_pass(c, A, prec, PASS_A, 0, D_K1, nsys, &e, act);
        }
        if (prof) cudaEventRecordWithFlags(c->prof[1], c->work, cudaEventRecordExternal);
        if (err == cudaSuccess) {
            if (A.kind == OP_STAGGERED) err = op_pass(c, A, prec, PASS_B, 0, D_K2, nsys, &e2, act);
            else err = launch_axpy_norm(prec, e2, v, dsec(c, D_K2), nsys, c->work, act);
        }
        if (prof) cudaEventRecordWithFlags(c->prof[2], c->work, cudaEventRecordExternal);
        if (err == cudaSuccess) err = launch_update(prec, e, v, nsys, c->work, act);
        if (prof) cudaEventRecordWithFlags(c->prof[3], c->work, cudaEventRecordExternal);
        kernels += 3;
        cudaError_t et = capture_tail(c->work, tail);
        cudaGraph_t gg = nullptr;
        cudaError_t ee = cudaStreamEndCapture(c->work, &gg);
        if (err == cudaSuccess) err = et != cudaSuccess ? et : ee;
        if (err != cudaSuccess) break;
        cudaGraphNodeParams cp = {};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeIf;
        cp.conditional.size = 1;
        cudaGraphNode_t ifn = nullptr;
        err = cudaGraphAddNode(&ifn, g, tail.empty() ? nullptr : tail.data(), nullptr, tail.size(), &cp);
        if (err != cudaSuccess) break;
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        err = begin_capture_into(c->work, body, {});
        if (err != cudaSuccess) break;
        err = launch_fold(e, v, nsys, 1, c->work, act, true);
        if (err == cudaSuccess && A.kind == OP_STAGGERED) err = op_pass(c, A, PREC_F64, PASS_A, 0, D_RUA, nsys, &e, act, true);
        if (err == cudaSuccess) err = op_pass(c, A, PREC_F64, PASS_C, 1, D_RUC, nsys, &e, act, true);
        ee = cudaStreamEndCapture(c->work, &gg);
        if (err == cudaSuccess) err = ee;
        tail.assign(1, ifn);
    }
    if (err != cudaSuccess) {
        cudaStreamCaptureStatus cs;
        if (cudaStreamIsCapturing(c->work, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
            cudaGraph_t junk = nullptr;
            cudaStreamEndCapture(c->work, &junk);
            if (junk && junk != g) cudaGraphDestroy(junk);
        }
        cudaGetLastError();
        cudaGraphDestroy(g);
        return err;
    }
    *out = g;
    return cudaSuccess;
}

static int get_graph(msc_ctx* c, const msc_op* op, int prec, int nsys, int chunk, bool reliable,
                     bool profile, int64_t npad, int group, int groups, GraphEntry** out) {
    // a one-system block-CSR SpMV takes its vector pointers as kernel
    // parameters (see launch_bsr_pass): they are part of the graph's identity
    const PassDesc& k1 = hsec(c, D_K1)[0];
    char key[224];
    snprintf(key, sizeof key, "%ld|%d|%d|%d|%d|%d|%lld|%d|%d|%p|%p", op->uid, prec, nsys, chunk, (int)reliable,
             (int)profile, (long long)npad, group, groups, nsys == 1 ? k1.src : nullptr,
             nsys == 1 ? k1.out : nullptr);
    GraphEntry& ge = c->graphs[key];
    if (ge.exec && ge.gen == c->gen) {
        *out = &ge;
        return MSC_OK;
    }
    if (ge.exec) {
        cudaGraphExecDestroy(ge.exec);
        ge.exec = nullptr;
    }
    long saved = c->launches;
    int kernels = 0;
    cudaGraph_t g = nullptr;
    cudaError_t err = cudaErrorNotSupported;
    if (reliable && c->use_cond) {
        err = build_chunk_graph_cond(c, op->dev, prec, nsys, chunk, profile, npad, group, groups, &g, kernels);
        if (err != cudaSuccess) {
            c->use_cond = 0;  // conditional nodes unavailable: gate the update kernels instead
            cudaGetLastError();
        }
    }
    if (err != cudaSuccess) {
        CK(cudaStreamBeginCapture(c->work, cudaStreamCaptureModeThreadLocal));
        err = enqueue_chunk(c, op->dev, prec, nsys, chunk, reliable, profile, npad, group, groups, kernels);
        cudaError_t err2 = cudaStreamEndCapture(c->work, &g);
        if (err != cudaSuccess) { if (g) cudaGraphDestroy(g); c->launches = saved; return cuda_status(err); }
        if (err2 != cudaSuccess) { c->launches = saved; return cuda_status(err2); }
    }
    c->launches = saved;
    const bool cond = reliable && c->use_cond;
    err = cudaGraphInstantiate(&ge.exec, g, 0);
    cudaGraphDestroy(g);
    if (err != cudaSuccess) return cuda_status(err);
    ge.gen = c->gen;
    ge.kernels = kernels;
    ge.cond_chunk = cond ? chunk : 0;
    ge.cond_kernels = op->dev.kind == OP_STAGGERED ? 3 : 2;
    if (cond && !c->h_flags) CK(cudaMallocHost((void**)&c->h_flags, sizeof(int) * 1024));
    *out = &ge;
    return MSC_OK;
}

struct ProfAcc {
    double k1 = 0, k2 = 0, k3 = 0;
    double act = 0;  // non-base shifts still iterating at the sampled iterations (summed)
    int n = 0;
};

// A stage of small staggered systems: cooperative launches that each run
// iterations until the systems stop or one is due a reliable update
// (persist.cu), every one followed by the gated kernels of that update. No
// graph: a handful of launches per update, and nothing to instantiate for a
// new operator. c->h_sys holds the systems' scalars.
static int run_stage_persist(msc_ctx* c, const msc_op* op, int prec, int nsys, int nslots, bool reliable, int64_t npad,
                             int max_iter, int* rel_updates) {
    const OpDev& A = op->dev;
    bool moved = false;
    CK(grow(c, c->gbar, 256, moved));
    PersistArgs a;
    a.e = engine_of(c);
    a.v = vecs_of(c, prec, npad, A);
    a.k1 = dsec(c, D_K1);
    a.k2 = dsec(c, D_K2);
    a.g = A.g;
    a.links = prec == PREC_F64 ? (const void*)A.linksfx : A.links32;
    a.links64 = A.links64;
    a.bar = (unsigned*)c->gbar.p;
    a.wait_ns = c->wait_ns;
    a.absent = (unsigned)c->test_absent;
    a.nsys = nsys;
    a.nslots = nslots;
    a.iters = reliable ? 50 : 100;
    const int reps = reliable ? 4 : 1;  // launches between two looks at the status
    // every launch but the last of a stage ends in an iteration or an update
    const long most = max_iter > 0 ? 2L * max_iter + 8 : 0;
    for (long k = 0; k < most; ++k) {
        bool any = false;
        for (int j = 0; j < nsys; ++j) any = any || c->h_sys[j].status < ST_DONE;
        if (!any) break;
        for (int q = 0; q < reps; ++q) {
            CK(cudaMemsetAsync(c->gbar.p, 0, sizeof(unsigned), c->work));
            CK(launch_persist(A, prec, a, c->work));
            c->launches++;
            if (!reliable) continue;
            CK(launch_fold(a.e, a.v, nsys, 1, c->work, nullptr, true));
            CK(op_pass(c, A, PREC_F64, PASS_A, 0, D_RUA, nsys, &a.e, nullptr, true));
            CK(op_pass(c, A, PREC_F64, PASS_C, 1, D_RUC, nsys, &a.e, nullptr, true));
            c->launches++;
        }
        CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * nsys, cudaMemcpyDeviceToHost, c->work));
        CK(cudaMemcpyAsync(c->h_err, c->errf.p, sizeof(unsigned), cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
        if (*c->h_err) {
            // a barrier's bounded wait ran out: the launch's results are void
            CK(cudaMemsetAsync(c->errf.p, 0, sizeof(unsigned), c->work));
            CK(cudaStreamSynchronize(c->work));
            return MSC_ERR_TIMEOUT;
        }
    }
    if (rel_updates)
        for (int j = 0; j < nsys; ++j) *rel_updates += c->h_sys[j].nru;
    return MSC_OK;
}

// Launch chunks until every system has stopped. With `compact` (several
// systems sharing a block-CSR matrix in FP32), the SpMV of each chunk runs
// only the systems still iterating, in groups sized for their number.
static int run_stage(msc_ctx* c, const msc_op* op, int prec, int nsys, int chunk, bool reliable,
                     bool profile, int64_t npad, int max_iter, ProfAcc* pa, int* rel_updates,
                     bool compact = false) {
    // group sizes of the shared-matrix SpMV follow the number still iterating
    compact = compact && op->dev.kind == OP_BSR && prec == PREC_F32 && nsys > 1;
    {
        bool moved = false;
        CK(grow(c, c->actb, sizeof(int) * (nsys + 1), moved));
        if (moved) c->gen++;
        if (c->h_act_cap < nsys + 1) {
            if (c->h_act) cudaFreeHost(c->h_act);
            CK(cudaMallocHost((void**)&c->h_act, sizeof(int) * (nsys + 1)));
            c->h_act_cap = nsys + 1;
        }
    }
    CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * nsys, cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    int nslot_all = 0;
    for (int j = 0; j < nsys; ++j) nslot_all = std::max(nslot_all, c->h_sys[j].slot0 + c->h_sys[j].S);
    const bool tiled = c->use_tile && nsys == 1 && prec == PREC_F32 && op->dev.kind == OP_STAGGERED && op->dev.recon &&
                       stag_tile_fits(op->dev.g, op->dev.nc);
    if (c->use_persist && !tiled && persist_applies(op->dev, prec, nsys, nslot_all))
        return run_stage_persist(c, op, prec, nsys, nslot_all, reliable, npad, max_iter, rel_updates);
    GraphEntry* ge = nullptr;
    int st = MSC_OK;
    if (!compact) {
        // nsys > 1 block-CSR stages without regrouping keep all groups
        const bool multi = op->dev.kind == OP_BSR && prec == PREC_F32 && nsys > 1;
        st = get_graph(c, op, prec, nsys, chunk, reliable, profile, npad, multi ? kMultiGroup : 0,
                       multi ? (nsys + kMultiGroup - 1) / kMultiGroup : 0, &ge);
        if (st != MSC_OK) return st;
    }
    // profiled stages: the non-base shifts still iterating when a chunk
    // starts (the shifts its first, sampled, update kernel moves)
    const bool track = profile && pa;
    auto count_active = [&]() {
        int a = 0;
        for (int j = 0; j < nsys; ++j)
            for (int k = 0; k < c->h_sys[j].S; ++k)
                if (k != c->h_sys[j].base && c->h_slot[c->h_sys[j].slot0 + k].active) ++a;
        return a;
    };
    if (track) {
        CK(cudaMemcpyAsync(c->h_slot, c->slot.p, sizeof(SlotScalars) * nslot_all, cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
    }
    int act_now = track ? count_active() : 0;
    // max_iter = 0 runs no iteration (the device sees the cap only after one)
    const long max_chunks = max_iter > 0 ? (long)max_iter / chunk + 2 : 0;
    for (long k = 0; k < max_chunks; ++k) {
        bool any = false, all_running = true;
        int active = 0;
        for (int j = 0; j < nsys; ++j) {
            if (c->h_sys[j].status < ST_DONE) any = true;
            if (c->h_sys[j].status != ST_RUNNING) all_running = false;
            else c->h_act[1 + active++] = j;
        }
        if (!any) break;
        c->h_act[0] = active;
        CK(cudaMemcpyAsync(c->actb.p, c->h_act, sizeof(int) * (active + 1), cudaMemcpyHostToDevice, c->work));
        if (compact) {
            const int group = active <= 1 ? 1 : kMultiGroup;
            const int groups = (active + group - 1) / group;
            st = get_graph(c, op, prec, nsys, chunk, reliable, profile, npad, group, groups, &ge);
            if (st != MSC_OK) return st;
        }
        CK(cudaGraphLaunch(ge->exec, c->work));
        c->launches += ge->kernels;
        CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * nsys, cudaMemcpyDeviceToHost,
                           c->work));
        const int ncf = std::min(ge->cond_chunk, 1024);
        if (ncf) CK(cudaMemcpyAsync(c->h_flags, c->condf.p, sizeof(int) * ncf, cudaMemcpyDeviceToHost, c->work));
        if (track)
            CK(cudaMemcpyAsync(c->h_slot, c->slot.p, sizeof(SlotScalars) * nslot_all, cudaMemcpyDeviceToHost,
                               c->work));
        CK(cudaMemcpyAsync(c->h_err, c->errf.p, sizeof(unsigned), cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
        if (*c->h_err) {
            // a kernel's bounded wait ran out: the chunk's results are void
            CK(cudaMemsetAsync(c->errf.p, 0, sizeof(unsigned), c->work));
            CK(cudaStreamSynchronize(c->work));
            return MSC_ERR_TIMEOUT;
        }
        for (int i = 0; i < ncf; ++i) c->launches += c->h_flags[i] ? ge->cond_kernels : 0;
        if (track && all_running) {
            float a = 0, b = 0, d = 0;
            if (cudaEventElapsedTime(&a, c->prof[0], c->prof[1]) == cudaSuccess &&
                cudaEventElapsedTime(&b, c->prof[1], c->prof[2]) == cudaSuccess &&
                cudaEventElapsedTime(&d, c->prof[2], c->prof[3]) == cudaSuccess) {
                pa->k1 += a;
                pa->k2 += b;
                pa->k3 += d;
                pa->act += act_now;
                pa->n++;
            }
        }
        if (track) act_now = count_active();
    }
    if (rel_updates)
        for (int j = 0; j < nsys; ++j) *rel_updates += c->h_sys[j].nru;
    return MSC_OK;
}

static void init_sys(SysScalars& s, int S, int base, int slot0, int rhs, double d, double tol,
                     int max_iter, int freeze, const msc_params& prm) {
    memset(&s, 0, sizeof s);
    if (prm.precision == MSC_MIXED) {
        s.ru_every = prm.reliable_every;
        s.delta2 = prm.reliable_delta * prm.reliable_delta;
    }
    s.alpha_prev = 1.0;
    s.beta_prev = 0.0;
    s.tol2 = tol * tol;
    s.tol2_acc = tol * tol;
    s.d = d;
    s.status = ST_RUNNING;
    s.max_iter = max_iter;
    s.S = S;
    s.base = base;
    s.slot0 = slot0;
    s.rhs = rhs;
    s.freeze = freeze;
}

static void init_slot(SlotScalars& q, double sigma_rel) {
    memset(&q, 0, sizeof q);
    q.sigma_rel = sigma_rel;
    q.zeta = 1.0;
    q.zeta_prev = 1.0;
    q.zeta_new = 1.0;
    q.active = 1;
    q.flag = 0;
    q.conv_iter = -1;
}

extern "C" {

const char* msc_strerror(int code) {
    switch (code) {
        case MSC_OK: return "ok";
        case MSC_ERR_ARG: return "invalid argument";
        case MSC_ERR_CUDA: return "CUDA runtime error";
        case MSC_ERR_OOM: return "out of device memory";
        case MSC_ERR_NOT_HPD: return "operator is not Hermitian positive definite";
        case MSC_ERR_NONFINITE: return "non-finite value in source or iteration";
        case MSC_ERR_NOT_CONVERGED: return "iteration cap reached before tolerance";
        case MSC_ERR_TIMEOUT: return "bounded device wait gave up";
        case MSC_ERR_UNSUPPORTED: return "unsupported request";
        case MSC_ERR_BREAKDOWN: return "BiCGStab-M breakdown (a recurrence denominator vanished)";
        default: return "unknown status";
    }
}

void msc_params_default(msc_params* p) {
    if (!p) return;
    p->tol = 1e-10;
    p->max_iter = 100000;
    p->precision = MSC_MIXED;
    p->reliable_every = 50;
    p->freeze_converged = 1;
    p->refine = 4;
    p->reliable_delta = 0.01;
}

int msc_create(msc_ctx** out, int device, void* stream) {
    if (!out) return MSC_ERR_ARG;
    *out = nullptr;
    int ndev = 0;
    CK(cudaGetDeviceCount(&ndev));
    if (device < 0 || device >= ndev) return MSC_ERR_ARG;
    CK(cudaSetDevice(device));
    msc_ctx* c = new msc_ctx();
    c->device = device;
    cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device);
    c->user = (cudaStream_t)stream;
    // MSC_GRAPH_COND=0 builds reliable updates as always-launched kernels that
    // exit when no update is due, instead of conditional graph nodes (for
    // profilers that replay kernels one by one)
    if (const char* ev = getenv("MSC_GRAPH_COND")) c->use_cond = atoi(ev) != 0;
    // MSC_STAG_TILE=1: one-system FP32 stencil passes stage their links in
    // shared memory by bulk asynchronous copies (lattices that tile; off by
    // default, the direct passes are faster). MSC_WAIT_NS: the limit of a
    // kernel's wait on its own asynchronous copies or, in a cooperative launch,
    // on the other blocks. For tests of the timeout paths only:
    // MSC_TEST_NO_COPY=1, the staged passes issue no copies; MSC_TEST_ABSENT=1,
    // the grid barriers wait for one arrival more than there are.
    // MSC_PERSIST=0: small staggered stages run the per-pass kernels, whose times
    // msc_info samples, instead of the cooperative one.
    if (const char* ev = getenv("MSC_PERSIST")) c->use_persist = atoi(ev) != 0;
    if (const char* ev = getenv("MSC_STAG_TILE")) c->use_tile = atoi(ev) != 0;
    if (const char* ev = getenv("MSC_WAIT_NS")) {
        const long long w = atoll(ev);
        if (w > 0) c->wait_ns = (uint64_t)w;
    }
    if (const char* ev = getenv("MSC_TEST_NO_COPY")) c->test_no_copy = atoi(ev) != 0;
    if (const char* ev = getenv("MSC_TEST_ABSENT")) c->test_absent = atoi(ev) != 0;
    cudaError_t e = cudaStreamCreateWithFlags(&c->work, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_sync, cudaEventDisableTiming);
    for (int i = 0; i < 4 && e == cudaSuccess; ++i) e = cudaEventCreate(&c->prof[i]);
    if (e == cudaSuccess) e = cudaMalloc(&c->errf.p, kErrBytes);
    if (e == cudaSuccess) {
        c->errf.bytes = kErrBytes;
        e = cudaMemsetAsync(c->errf.p, 0, kErrBytes, c->work);
    }
    if (e == cudaSuccess) e = cudaMallocHost((void**)&c->h_err, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
    if (e != cudaSuccess) {
        msc_destroy(c);
        return cuda_status(e);
    }
    *out = c;
    return MSC_OK;
}

int msc_set_stream(msc_ctx* c, void* stream) {
    if (!c) return MSC_ERR_ARG;
    c->user = (cudaStream_t)stream;
    return MSC_OK;
}

int msc_destroy(msc_ctx* c) {
    if (!c) return MSC_ERR_ARG;
    cudaSetDevice(c->device);
    if (c->work) cudaStreamSynchronize(c->work);
    for (auto& kv : c->graphs)
        if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
    Buf* bufs[] = {&c->sys, &c->slot, &c->partial, &c->counter, &c->out_red, &c->descs,
                   &c->b64, &c->x64, &c->t64, &c->r, &c->p, &c->t, &c->ps, &c->xit,
                   &c->coef, &c->force, &c->btab, &c->bvb, &c->actb, &c->condf, &c->bcg,
                   &c->pb, &c->px0, &c->ptmp, &c->gbar, &c->errf};
    for (Buf* b : bufs)
        if (b->p) cudaFree(b->p);
    if (c->h_sys) cudaFreeHost(c->h_sys);
    if (c->h_slot) cudaFreeHost(c->h_slot);
    if (c->h_red) cudaFreeHost(c->h_red);
    if (c->h_desc) cudaFreeHost(c->h_desc);
    if (c->h_act) cudaFreeHost(c->h_act);
    if (c->h_flags) cudaFreeHost(c->h_flags);
    if (c->h_err) cudaFreeHost(c->h_err);
    if (c->ev_sync) cudaEventDestroy(c->ev_sync);
    for (int i = 0; i < 4; ++i)
        if (c->prof[i]) cudaEventDestroy(c->prof[i]);
    if (c->work) cudaStreamDestroy(c->work);
    delete c;
    return MSC_OK;
}

static void free_op_dev(OpDev& d) {
    // links64 holds the staggered operator's one allocation
    void* ps[] = {d.links64, d.slice_len, d.slice_start, d.cols, d.vals64, d.valsr, d.valsfx, d.blkfx, d.vals32};
    for (void* p : ps)
        if (p) cudaFree(p);
    memset(&d, 0, sizeof d);
}

// Drops the context's graphs of operator uid ("<uid>|..." and "bcg|<uid>|...").
static void drop_graphs(msc_ctx* c, long uid) {
    const std::string a = std::to_string(uid) + "|", b = "bcg|" + a;
    for (auto it = c->graphs.begin(); it != c->graphs.end();) {
        if (it->first.compare(0, a.size(), a) == 0 || it->first.compare(0, b.size(), b) == 0) {
            if (it->second.exec) cudaGraphExecDestroy(it->second.exec);
            it = c->graphs.erase(it);
        } else {
            ++it;
        }
    }
}

int msc_op_destroy(msc_op* op) {
    if (!op || op->is_view) return MSC_ERR_ARG;
    if (msc_ctx* c = op->ctx) {
        cudaSetDevice(c->device);
        // the context's graphs of this operator and of its parity views go
        // with it, after the work stream has drained
        if (c->work) cudaStreamSynchronize(c->work);
        drop_graphs(c, op->uid);
        for (msc_op* v : op->view)
            if (v) drop_graphs(c, v->uid);
    }
    for (msc_op* v : op->view) delete v;
    free_op_dev(op->dev);
    delete op;
    return MSC_OK;
}

static int begin(msc_ctx* c) {
    CK(cudaSetDevice(c->device));
    CK(cudaEventRecord(c->ev_sync, c->user));
    CK(cudaStreamWaitEvent(c->work, c->ev_sync, 0));
    return MSC_OK;
}

// Whether the device has room for an optional second copy of `bytes` of an
// operator's data beside the `needed` bytes that it cannot do without. A copy
// serves speed alone: it may not make an operator or a solve fail that fits
// without it, so eight times its size has to stay free for the solves. (The
// query is left out for copies that no card is short of.)
static bool room_for_copy(size_t bytes, size_t needed) {
    if (bytes <= (size_t)64 << 20) return true;
    size_t free_b = 0, total = 0;
    if (cudaMemGetInfo(&free_b, &total) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return free_b >= needed + 9 * bytes;
}

int msc_op_staggered(msc_ctx* c, msc_op** out, int nc, const int dims[4], const double* links,
                     double mass, unsigned flags) {
    if (!c || !out || !dims || !links) return MSC_ERR_ARG;
    *out = nullptr;
    if (nc != 2 && nc != 3) return MSC_ERR_ARG;
    if (!std::isfinite(mass)) return MSC_ERR_ARG;
    int64_t V = 1;
    for (int mu = 0; mu < 4; ++mu) {
        if (dims[mu] < 2 || (dims[mu] & 1)) return MSC_ERR_ARG;
        V *= dims[mu];
    }
    if (V * nc > (int64_t)1 << 30) return MSC_ERR_UNSUPPORTED;
    int st = begin(c);
    if (st) return st;
    msc_op* op = new msc_op();
    op->ctx = c;
    op->uid = ++g_op_uid;
    OpDev& d = op->dev;
    d.kind = OP_STAGGERED;
    d.nc = nc;
    d.g = stag_geom(dims);
    d.n = V * nc;
    d.mass = mass;
    const size_t nlink_bytes = (size_t)4 * V * nc * nc * 16;
    const double2* src = (const double2*)links;
    void* tmp = nullptr;
    double* ddev = (double*)((char*)c->errf.p + kSetupDev);
    cudaError_t e = cudaSuccess;
    auto fail = [&](cudaError_t err) {
        if (tmp) cudaFree(tmp);
        free_op_dev(d);
        delete op;
        return cuda_status(err);
    };
    if (!is_device_ptr(links)) {
        e = cudaMalloc(&tmp, nlink_bytes);
        if (e == cudaSuccess) e = cudaMemcpyAsync(tmp, links, nlink_bytes, cudaMemcpyHostToDevice, c->work);
        if (e != cudaSuccess) return fail(e);
        src = (const double2*)tmp;
    }
    double dev[kLinkDevs];
    e = cudaMemsetAsync(ddev, 0, sizeof dev, c->work);
    if (e == cudaSuccess) e = stag_unitarity(d, src, ddev, c->work);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dev, ddev, sizeof dev, cudaMemcpyDeviceToHost, c->work);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
    if (e != cudaSuccess) return fail(e);
    // Rebuilding a row needs determinant 1 too. Limbs need entries of at most 1,
    // and links that couple every pair of colours: they hold an entry to 2^-57
    // and sum a site's colours in one unit, so that an entry, or a colour that
    // meets no other, far below 1 would keep fewer bits than in FP64 (unit links:
    // a colour of 1e-20 beside one of 1 came out as 0). With the smallest entry
    // of all at 2^-24 or more no colour's sum is that far below the unit alone; the
    // smallest of the 4e7 entries of a random 32^4 field is about 1e-4.
    const bool unitary = dev[0] < 1e-9, coupled = dev[2] <= 0x1p24;
    d.recon = (!(flags & MSC_LINKS_FULL) && unitary && dev[1] < 1e-9) ? 1 : 0;
    const size_t l32 = d.recon ? (size_t)4 * V * (nc == 3 ? 3 : 1) * 16 : (size_t)4 * V * nc * nc * 8;
    size_t lfx = unitary && coupled ? (size_t)4 * ((V + 31) / 32 * 32) * nc * nc * 16 : 0;
    if (lfx && !room_for_copy(lfx, nlink_bytes + l32)) lfx = 0;
    // one allocation for the three forms (each cudaMalloc and cudaFree costs
    // tens of microseconds of a small operator's set-up): FP64, limbs, FP32
    const size_t at_fx = (nlink_bytes + 255) / 256 * 256;
    size_t at_32 = at_fx + (lfx + 255) / 256 * 256;
    char* block = nullptr;
    e = cudaMalloc((void**)&block, at_32 + l32);
    if (e == cudaErrorMemoryAllocation && lfx) {  // without the limbs, then
        cudaGetLastError();
        lfx = 0;
        at_32 = at_fx;
        e = cudaMalloc((void**)&block, at_32 + l32);
    }
    if (e != cudaSuccess) return fail(e);
    d.links64 = (double2*)block;
    d.linksfx = lfx ? (int4*)(block + at_fx) : nullptr;
    d.links32 = block + at_32;
    e = stag_pack_links(d, src, c->work);
    if (e == cudaSuccess) e = stag_pack_links32(d, src, c->work);
    if (e == cudaSuccess && lfx) e = stag_pack_linksfx(d, src, c->work);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
    if (e != cudaSuccess) return fail(e);
    if (tmp) cudaFree(tmp);
    *out = op;
    return MSC_OK;
}

// MSC_CHECK_HERMITIAN: entries may differ from the conjugate of their
// transposed partner by this much relative to the largest entry (rounding of
// a matrix assembled in FP64 by different paths for (i, j) and (j, i)).
constexpr double kHermitianTol = 1e-12;

int msc_op_bsr(msc_ctx* c, msc_op** out, int64_t nbr, int bd, const int64_t* row_ptr,
               const int32_t* col_idx, const double* vals, unsigned flags) {
    if (!c || !out || !row_ptr || !col_idx || !vals) return MSC_ERR_ARG;
    if (flags & ~MSC_CHECK_HERMITIAN) return MSC_ERR_ARG;
    *out = nullptr;
    if (bd < 1 || bd > 3 || nbr <= 0 || nbr > ((int64_t)1 << 31) - 1) return MSC_ERR_ARG;
    int st = begin(c);
    if (st) return st;
    std::vector<int64_t> rp(nbr + 1);
    if (is_device_ptr(row_ptr)) {
        CK(cudaMemcpyAsync(rp.data(), row_ptr, sizeof(int64_t) * (nbr + 1), cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
    } else {
        memcpy(rp.data(), row_ptr, sizeof(int64_t) * (nbr + 1));
    }
    if (rp[0] != 0) return MSC_ERR_ARG;
    for (int64_t i = 0; i < nbr; ++i)
        if (rp[i + 1] < rp[i]) return MSC_ERR_ARG;
    const int64_t nnzb = rp[nbr];
    const int64_t nslices = (nbr + 31) / 32;
    std::vector<int32_t> slen(nslices);
    std::vector<int64_t> sstart(nslices);
    int64_t acc = 0;
    for (int64_t s = 0; s < nslices; ++s) {
        int64_t m = 0;
        for (int64_t i = s * 32; i < std::min(nbr, s * 32 + 32); ++i) m = std::max(m, rp[i + 1] - rp[i]);
        // the kernels index inside a slice with 32-bit offsets (k * 32 * bd * bd)
        if (m * 32 * bd * bd >= ((int64_t)1 << 31)) return MSC_ERR_ARG;
        slen[s] = (int32_t)m;
        sstart[s] = acc;
        acc += m;
    }
    msc_op* op = new msc_op();
    op->ctx = c;
    op->uid = ++g_op_uid;
    op->nnzb = nnzb;
    OpDev& d = op->dev;
    d.kind = OP_BSR;
    d.bd = bd;
    d.nbr = nbr;
    d.n = nbr * bd;
    d.nslices = nslices;
    d.nslots_blk = acc;
    void *trp = nullptr, *tcol = nullptr, *tval = nullptr;
    int* dbad = (int*)((char*)c->errf.p + kSetupWord);
    unsigned long long* dherm = nullptr;
    auto fail = [&](int code) {
        if (trp) cudaFree(trp);
        if (tcol) cudaFree(tcol);
        if (tval) cudaFree(tval);
        if (dherm) cudaFree(dherm);
        free_op_dev(d);
        delete op;
        return code;
    };
    const size_t e2 = (size_t)bd * bd;
    cudaError_t e = cudaMalloc((void**)&d.slice_len, sizeof(int32_t) * nslices);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d.slice_start, sizeof(int64_t) * nslices);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d.cols, sizeof(int32_t) * 32 * std::max<int64_t>(acc, 1));
    // FP64 entries: limbs and block exponents for bd > 1, doubles for bd = 1
    // (a 1 x 1 block has four FMAs against 36 bytes: nothing to gain)
    if (e == cudaSuccess && bd > 1) e = cudaMalloc((void**)&d.valsfx, 16 * e2 * 32 * std::max<int64_t>(acc, 1));
    if (e == cudaSuccess && bd > 1) e = cudaMalloc((void**)&d.blkfx, 2 * 32 * std::max<int64_t>(acc, 1));
    if (e == cudaSuccess && bd == 1) e = cudaMalloc((void**)&d.vals64, 16 * e2 * 32 * std::max<int64_t>(acc, 1));
    if (e == cudaSuccess) e = cudaMalloc((void**)&d.vals32, 8 * e2 * 32 * std::max<int64_t>(acc, 1));
    if (e == cudaSuccess) e = cudaMalloc((void**)&trp, sizeof(int64_t) * (nbr + 1));
    if (e != cudaSuccess) return fail(cuda_status(e));
    e = cudaMemcpyAsync(d.slice_len, slen.data(), sizeof(int32_t) * nslices, cudaMemcpyHostToDevice, c->work);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d.slice_start, sstart.data(), sizeof(int64_t) * nslices, cudaMemcpyHostToDevice, c->work);
    if (e == cudaSuccess) e = cudaMemcpyAsync(trp, rp.data(), sizeof(int64_t) * (nbr + 1), cudaMemcpyHostToDevice, c->work);
    if (e == cudaSuccess) e = cudaMemsetAsync(dbad, 0, sizeof(int), c->work);
    const int32_t* dcol = col_idx;
    const double2* dval = (const double2*)vals;
    if (e == cudaSuccess && !is_device_ptr(col_idx)) {
        e = cudaMalloc(&tcol, sizeof(int32_t) * std::max<int64_t>(nnzb, 1));
        if (e == cudaSuccess && nnzb) e = cudaMemcpyAsync(tcol, col_idx, sizeof(int32_t) * nnzb, cudaMemcpyHostToDevice, c->work);
        dcol = (const int32_t*)tcol;
    }
    if (e == cudaSuccess && !is_device_ptr(vals)) {
        e = cudaMalloc(&tval, 16 * e2 * std::max<int64_t>(nnzb, 1));
        if (e == cudaSuccess && nnzb) e = cudaMemcpyAsync(tval, vals, 16 * e2 * nnzb, cudaMemcpyHostToDevice, c->work);
        dval = (const double2*)tval;
    }
    if (e == cudaSuccess) e = bsr_pack(d, (const int64_t*)trp, dcol, dval, dbad, c->work);
    int bad = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bad, dbad, sizeof(int), cudaMemcpyDeviceToHost, c->work);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
    if (e != cudaSuccess) return fail(cuda_status(e));
    if (bad & 1) return fail(MSC_ERR_ARG);
    const size_t lre = 8 * 32 * (size_t)std::max<int64_t>(acc, 1);
    if (bd == 1 && !(bad & 4) && room_for_copy(lre, 0)) {
        e = cudaMalloc((void**)&d.valsr, lre);
        if (e == cudaErrorMemoryAllocation) {  // without the copy, then
            cudaGetLastError();
            d.valsr = nullptr;
            e = cudaSuccess;
        }
        if (e == cudaSuccess && d.valsr) e = bsr_pack_real(d, c->work);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
        if (e != cudaSuccess) return fail(cuda_status(e));
    }
    if (bad & 2) {  // some block row does not fit the limbs: the whole matrix in FP64
        cudaFree(d.valsfx);
        cudaFree(d.blkfx);
        d.valsfx = nullptr;
        d.blkfx = nullptr;
        e = cudaMalloc((void**)&d.vals64, 16 * e2 * 32 * std::max<int64_t>(acc, 1));
        if (e == cudaSuccess) e = bsr_pack(d, (const int64_t*)trp, dcol, dval, dbad, c->work);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&bad, dbad, sizeof(int), cudaMemcpyDeviceToHost, c->work);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
        if (e != cudaSuccess) return fail(cuda_status(e));
        if (bad & 1) return fail(MSC_ERR_ARG);  // in rows that the first packing left out
    }
    if (flags & MSC_CHECK_HERMITIAN) {
        // the columns are known to be in range now (the packing checked them)
        double hm[2] = {0.0, 0.0};
        e = cudaMalloc((void**)&dherm, 2 * sizeof(unsigned long long));
        if (e == cudaSuccess) e = cudaMemsetAsync(dherm, 0, 2 * sizeof(unsigned long long), c->work);
        if (e == cudaSuccess) e = bsr_check_hermitian((const int64_t*)trp, dcol, dval, nbr, bd, dherm, c->work);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hm, dherm, sizeof hm, cudaMemcpyDeviceToHost, c->work);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
        if (e != cudaSuccess) return fail(cuda_status(e));
        if (!(hm[0] <= kHermitianTol * hm[1])) return fail(MSC_ERR_NOT_HPD);
        cudaFree(dherm);
        dherm = nullptr;
    }
    cudaFree(trp);
    if (tcol) cudaFree(tcol);
    if (tval) cudaFree(tval);
    *out = op;
    return MSC_OK;
}

int msc_op_size(const msc_op* op, int64_t* n) {
    if (!op || !n) return MSC_ERR_ARG;
    *n = op->dev.n;
    return MSC_OK;
}

int msc_op_recon(const msc_op* op, int* recon) {
    if (!op || !recon) return MSC_ERR_ARG;
    *recon = op->dev.kind == OP_STAGGERED ? op->dev.recon : 0;
    return MSC_OK;
}

int msc_op_bsr_size(const msc_op* op, int64_t* nbr, int64_t* nnzb, int* bd) {
    if (!op || op->dev.kind != OP_STAGGERED) return MSC_ERR_ARG;
    if (nbr) *nbr = op->dev.g.V;
    if (nnzb) *nnzb = (int64_t)33 * op->dev.g.V;
    if (bd) *bd = op->dev.nc;
    return MSC_OK;
}

int msc_staggered_export_bsr(msc_ctx* c, const msc_op* op, int64_t* row_ptr, int32_t* col_idx,
                             double* vals) {
    if (!c || !op || !row_ptr || !col_idx || !vals || op->dev.kind != OP_STAGGERED) return MSC_ERR_ARG;
    int st = begin(c);
    if (st) return st;
    const OpDev& d = op->dev;
    const int64_t V = d.g.V, nnzb = 33 * V;
    const size_t vb = (size_t)nnzb * d.nc * d.nc * 16;
    const bool drp = is_device_ptr(row_ptr), dci = is_device_ptr(col_idx), dva = is_device_ptr(vals);
    void *trp = nullptr, *tci = nullptr, *tva = nullptr;
    cudaError_t e = cudaSuccess;
    if (!drp) e = cudaMalloc(&trp, sizeof(int64_t) * (V + 1));
    if (e == cudaSuccess && !dci) e = cudaMalloc(&tci, sizeof(int32_t) * nnzb);
    if (e == cudaSuccess && !dva) e = cudaMalloc(&tva, vb);
    if (e == cudaSuccess)
        e = stag_export_bsr(d, drp ? row_ptr : (int64_t*)trp, dci ? col_idx : (int32_t*)tci,
                            dva ? (double2*)vals : (double2*)tva, c->work);
    if (e == cudaSuccess && !drp) e = cudaMemcpyAsync(row_ptr, trp, sizeof(int64_t) * (V + 1), cudaMemcpyDeviceToHost, c->work);
    if (e == cudaSuccess && !dci) e = cudaMemcpyAsync(col_idx, tci, sizeof(int32_t) * nnzb, cudaMemcpyDeviceToHost, c->work);
    if (e == cudaSuccess && !dva) e = cudaMemcpyAsync(vals, tva, vb, cudaMemcpyDeviceToHost, c->work);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
    if (trp) cudaFree(trp);
    if (tci) cudaFree(tci);
    if (tva) cudaFree(tva);
    return e == cudaSuccess ? MSC_OK : cuda_status(e);
}

// Whether the FP64 kernels can read or write [n] complex at p themselves:
// memory of this device (not managed, not a peer's) on a 16-byte boundary.
static bool kernel_ready(const void* p, int device) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice && a.device == device && ((uintptr_t)p & 15) == 0;
}

// FP64 applies on the fixed-point kernels: the passes' descriptors are kernel
// parameters and the caller's vectors are used in place where the kernels can
// (a staged copy of a 4^4 to 24^4 vector and the two descriptor uploads took
// as long as the passes: A x at 10 x 6 x 14 x 18 47 us a call against 28).
// Input and output may be the same vector of a staggered A x (its second
// pass reads the input at the output's own site only); other overlaps are
// staged.
static int apply_direct(msc_ctx* c, const OpDev& A, double sigma, const double* in, double* out, bool dslash) {
    const int64_t n = A.n, npad = (n + 63) / 64 * 64;
    const int ws = ensure_ws(c, npad, 3, 1, 1, 16);
    if (ws) return ws;
    double2* t64 = (double2*)c->t64.p;
    const double2* src = (const double2*)in;
    double2* dst = (double2*)out;
    const bool stag = A.kind == OP_STAGGERED;
    const bool apart = in + 2 * n <= out || out + 2 * n <= in;
    const bool same_ok = stag && !dslash && (const double*)out == in;
    if (!kernel_ready(in, c->device) || !(apart || same_ok)) {
        CK(cudaMemcpyAsync(t64, in, n * 16, cudaMemcpyDefault, c->work));
        src = t64;
    }
    const bool direct_out = kernel_ready(out, c->device);
    if (!direct_out) dst = t64 + 2 * npad;
    double2* mid = t64 + npad;
    const Engine none{};
    if (stag) {
        const PassDesc d1 = mkdesc(src, nullptr, nullptr, dslash ? dst : mid, 0.0, -1, -1, FIN_NONE);
        CK(launch_stag_pass(A, PREC_F64, PASS_A, 0, none, nullptr, 1, c->work, nullptr, false, &d1));
        c->launches++;
        if (!dslash) {
            const PassDesc d2 = mkdesc(mid, src, nullptr, dst, A.mass * A.mass + sigma, -1, -1, FIN_NONE);
            CK(launch_stag_pass(A, PREC_F64, PASS_D, 0, none, nullptr, 1, c->work, nullptr, false, &d2));
            c->launches++;
        }
    } else {
        const PassDesc d = mkdesc(src, src, nullptr, dst, sigma, -1, -1, FIN_NONE);
        CK(launch_bsr_pass(A, PREC_F64, PASS_D, 0, none, nullptr, 1, c->work, nullptr, false, &d));
        c->launches++;
    }
    if (!direct_out) CK(cudaMemcpyAsync(out, dst, n * 16, cudaMemcpyDefault, c->work));
    CK(cudaStreamSynchronize(c->work));
    return MSC_OK;
}

// out = (A + sigma) in (or D in when dslash) through the operator kernels.
static int apply_impl(msc_ctx* c, const msc_op* op, double sigma, const double* in, double* out,
                      int precision, bool dslash) {
    if (!c || !op || !in || !out) return MSC_ERR_ARG;
    if (precision != MSC_FP64 && precision != MSC_FP32) return MSC_ERR_ARG;
    if (dslash && (op->dev.kind != OP_STAGGERED || precision != MSC_FP64)) return MSC_ERR_ARG;
    int st = begin(c);
    if (st) return st;
    const OpDev& A = op->dev;
    if (precision == MSC_FP64 && (A.kind == OP_STAGGERED ? (void*)A.linksfx : (void*)A.valsfx))
        return apply_direct(c, A, sigma, in, out, dslash);
    const int64_t n = A.n, npad = (n + 63) / 64 * 64;
    st = ensure_ws(c, npad, 3, 1, 1, 16);
    if (st) return st;
    double2* t64 = (double2*)c->t64.p;
    double2* in64 = t64;
    double2* mid64 = t64 + npad;
    double2* out64 = t64 + 2 * npad;
    CK(cudaMemcpyAsync(in64, in, n * 16, cudaMemcpyDefault, c->work));
    const double dstag = A.kind == OP_STAGGERED ? A.mass * A.mass : 0.0;
    if (precision == MSC_FP64) {
        if (dslash) {
            hsec(c, D_AP1)[0] = mkdesc(in64, nullptr, nullptr, out64, 0.0, -1, -1, FIN_NONE);
            CK(upload_sec(c, D_AP1, 1));
            CK(op_pass(c, A, PREC_F64, PASS_A, 0, D_AP1, 1));
        } else if (A.kind == OP_STAGGERED) {
            hsec(c, D_AP1)[0] = mkdesc(in64, nullptr, nullptr, mid64, 0.0, -1, -1, FIN_NONE);
            hsec(c, D_AP2)[0] = mkdesc(mid64, in64, nullptr, out64, dstag + sigma, -1, -1, FIN_NONE);
            CK(upload_sec(c, D_AP1, 1));
            CK(upload_sec(c, D_AP2, 1));
            CK(op_pass(c, A, PREC_F64, PASS_A, 0, D_AP1, 1));
            CK(op_pass(c, A, PREC_F64, PASS_D, 0, D_AP2, 1));
        } else {
            hsec(c, D_AP2)[0] = mkdesc(in64, in64, nullptr, out64, sigma, -1, -1, FIN_NONE);
            CK(upload_sec(c, D_AP2, 1));
            CK(op_pass(c, A, PREC_F64, PASS_D, 0, D_AP2, 1));
        }
    } else {
        float2* in32 = (float2*)c->r.p;
        float2* mid32 = (float2*)c->t.p;
        float2* out32 = (float2*)c->p.p;
        if (A.kind == OP_STAGGERED) CK(launch_convert_planar(in64, in32, A.nc, A.g.V, true, c->work));
        else CK(launch_convert(in64, 0, in32, 1, n, c->work));
        if (A.kind == OP_STAGGERED) {
            hsec(c, D_AP1)[0] = mkdesc(in32, nullptr, nullptr, mid32, 0.0, -1, -1, FIN_NONE);
            hsec(c, D_AP2)[0] = mkdesc(mid32, in32, nullptr, out32, dstag + sigma, -1, -1, FIN_NONE);
            CK(upload_sec(c, D_AP1, 1));
            CK(upload_sec(c, D_AP2, 1));
            CK(op_pass(c, A, PREC_F32, PASS_A, 0, D_AP1, 1));
            CK(op_pass(c, A, PREC_F32, PASS_D, 0, D_AP2, 1));
        } else {
            hsec(c, D_AP2)[0] = mkdesc(in32, in32, nullptr, out32, sigma, -1, -1, FIN_NONE);
            CK(upload_sec(c, D_AP2, 1));
            CK(op_pass(c, A, PREC_F32, PASS_D, 0, D_AP2, 1));
        }
        if (A.kind == OP_STAGGERED) CK(launch_convert_planar(out32, out64, A.nc, A.g.V, false, c->work));
        else CK(launch_convert(out32, 1, out64, 0, n, c->work));
    }
    CK(cudaMemcpyAsync(out, out64, n * 16, cudaMemcpyDefault, c->work));
    CK(cudaMemcpyAsync(c->h_err, c->errf.p, sizeof(unsigned), cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    if (*c->h_err) {  // a staged pass's bounded wait ran out: out is void
        CK(cudaMemsetAsync(c->errf.p, 0, sizeof(unsigned), c->work));
        CK(cudaStreamSynchronize(c->work));
        return MSC_ERR_TIMEOUT;
    }
    return MSC_OK;
}

int msc_op_apply(msc_ctx* c, const msc_op* op, double sigma, const double* in, double* out,
                 int precision) {
    return apply_impl(c, op, sigma, in, out, precision, false);
}

int msc_op_dslash(msc_ctx* c, const msc_op* op, const double* in, double* out) {
    return apply_impl(c, op, 0.0, in, out, MSC_FP64, true);
}

}  // extern "C"

// Right-hand sides of polynomial form, b_s = q_s(A) b (Sec. 5, eq. linprobgen):
// q_s(t) = sum_k coef[s * (deg + 1) + k] t^k.
struct PolyRhs {
    const double* coef;
    int deg;
};

// b_s = q_s(A) b into c->pb and x_s0 = s_s(A) b into c->px0 for every shift,
// where q_s(t) = q_s(-sigma_s) + (t + sigma_s) s_s(t) (synthetic division by
// t + sigma_s); cs[s] = q_s(-sigma_s), bs2[s] = |b_s|^2, b2 = |b|^2. Horner's
// rule on the device with the FP64 operator, every shift in one launch per
// step.
static int poly_setup(msc_ctx* c, const OpDev& A, const double2* b, int64_t n, int64_t npad,
                      const double* sigma, int S, const PolyRhs& pr, std::vector<double>& cs,
                      std::vector<double>& bs2, double& b2) {
    const int d = pr.deg;
    std::vector<double> sco((size_t)S * std::max(d, 1), 0.0);  // s_s: [S][d], constant term first
    for (int s = 0; s < S; ++s) {
        const double* a = pr.coef + (size_t)s * (d + 1);
        const double r = -sigma[s];
        if (d == 0) {
            cs[s] = a[0];
            continue;
        }
        double* q = sco.data() + (size_t)s * d;
        q[d - 1] = a[d];
        for (int k = d - 1; k >= 1; --k) q[k - 1] = a[k] + r * q[k];
        cs[s] = a[0] + r * q[0];
    }
    bool moved = false;
    const size_t vb = (size_t)S * npad * 16;
    CK(grow(c, c->pb, vb, moved));
    CK(grow(c, c->px0, vb, moved));
    CK(grow(c, c->ptmp, 2 * vb, moved));
    if (moved) c->gen++;
    double2* pb = (double2*)c->pb.p;
    double2* px0 = (double2*)c->px0.p;
    double2* mid = (double2*)c->ptmp.p;
    double2* out = mid + (size_t)S * npad;
    const double dstag = A.kind == OP_STAGGERED ? A.mass * A.mass : 0.0;
    // v_s <- sum_k co[s][k] A^k b, co given constant term first, `deg` + 1 terms
    auto horner = [&](double2* v, int deg, auto coef_of) -> int {
        ShiftCoef a{};
        for (int s = 0; s < S; ++s) a.v[s] = coef_of(s, deg);
        CK(launch_poly_step(v, nullptr, a, b, S, n, npad, c->work));
        c->launches++;
        if (deg == 0) return MSC_OK;
        // descriptors of out_s = A v_s for every shift (FP64)
        CK(cudaStreamSynchronize(c->work));
        for (int s = 0; s < S; ++s) {
            double2* vs = v + (size_t)s * npad;
            if (A.kind == OP_STAGGERED) {
                hsec(c, D_AP1)[s] = mkdesc(vs, nullptr, nullptr, mid + (size_t)s * npad, 0.0, -1, -1, FIN_NONE);
                hsec(c, D_AP2)[s] = mkdesc(mid + (size_t)s * npad, vs, nullptr, out + (size_t)s * npad, dstag, -1, -1,
                                           FIN_NONE);
            } else {
                hsec(c, D_AP2)[s] = mkdesc(vs, vs, nullptr, out + (size_t)s * npad, 0.0, -1, -1, FIN_NONE);
            }
        }
        CK(upload_sec(c, D_AP1, S));
        CK(upload_sec(c, D_AP2, S));
        for (int k = deg - 1; k >= 0; --k) {
            if (A.kind == OP_STAGGERED) CK(op_pass(c, A, PREC_F64, PASS_A, 0, D_AP1, S));
            CK(op_pass(c, A, PREC_F64, PASS_D, 0, D_AP2, S));
            for (int s = 0; s < S; ++s) a.v[s] = coef_of(s, k);
            CK(launch_poly_step(v, out, a, b, S, n, npad, c->work));
            c->launches++;
        }
        CK(cudaStreamSynchronize(c->work));
        return MSC_OK;
    };
    int st = horner(pb, d, [&](int s, int k) { return pr.coef[(size_t)s * (d + 1) + k]; });
    if (st) return st;
    if (d >= 1) st = horner(px0, d - 1, [&](int s, int k) { return sco[(size_t)s * d + k]; });
    else CK(cudaMemsetAsync(px0, 0, vb, c->work));
    if (st) return st;
    // |b_s|^2 (rows 0 .. S-1) and |b|^2 (row S)
    CK(cudaMemcpyAsync(mid, b, n * 16, cudaMemcpyDeviceToDevice, c->work));
    Engine e = engine_of(c);
    CK(launch_norms(e, pb, S, n, npad, c->work));
    CK(cudaMemcpyAsync(c->h_red, c->out_red.p, sizeof(double) * S, cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    for (int s = 0; s < S; ++s) bs2[s] = c->h_red[s];
    CK(launch_norms(e, mid, 1, n, npad, c->work));
    CK(cudaMemcpyAsync(c->h_red, c->out_red.p, sizeof(double), cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    b2 = c->h_red[0];
    c->launches += 2;
    return MSC_OK;
}

static int solve_impl(msc_ctx* c, const msc_op* op, const double* b, int nrhs, const double* sigma, int S,
                      const msc_params* prm_in, double* x, msc_info* info, const PolyRhs* poly) {
    const auto t0 = std::chrono::steady_clock::now();
    const Range whole(poly ? "msc_solve_poly_rhs" : "msc_solve");
    if (!c || !op || !b || !x || !sigma || nrhs <= 0 || S <= 0 || S > kMaxShifts) return MSC_ERR_ARG;
    if (poly && nrhs != 1) return MSC_ERR_ARG;
    msc_params prm;
    msc_params_default(&prm);
    if (prm_in) prm = *prm_in;
    if (!(prm.tol > 0) || prm.max_iter < 0 || prm.refine < 0) return MSC_ERR_ARG;
    if (prm.precision != MSC_FP64 && prm.precision != MSC_MIXED) return MSC_ERR_ARG;
    if (prm.precision == MSC_MIXED && (prm.reliable_every < 1 || !(prm.reliable_delta >= 0.0) ||
                                       !(prm.reliable_delta < 1.0))) return MSC_ERR_ARG;
    for (int s = 0; s < S; ++s)
        if (!(sigma[s] >= 0.0) || !std::isfinite(sigma[s])) return MSC_ERR_ARG;
    const int prec = prm.precision == MSC_MIXED ? PREC_F32 : PREC_F64;
    const bool mixed = prec == PREC_F32;
    int st = begin(c);
    if (st) return st;
    const OpDev& A = op->dev;
    const int64_t n = A.n, npad = (n + 63) / 64 * 64;
    const int nslots = nrhs * S;
    const int rows = std::max(nrhs, nslots) + (poly ? 1 : 0);
    st = ensure_ws(c, npad, rows, nslots, nrhs, mixed ? 8 : 16);
    if (st) return st;
    const long launches0 = c->launches;
    const size_t elem = mixed ? 8 : 16;
    char* r = (char*)c->r.p;
    char* p = (char*)c->p.p;
    char* t = (char*)c->t.p;
    double2* x64 = (double2*)c->x64.p;
    double2* t64 = (double2*)c->t64.p;
    double2* b64 = (double2*)c->b64.p;
    // source in (pads cleared: the layout stride may differ from a previous solve)
    if (npad > n) {
        CK(cudaMemset2DAsync(b64 + n, npad * 16, 0, (npad - n) * 16, nrhs, c->work));
        CK(cudaMemset2DAsync(t + n * elem, npad * elem, 0, (npad - n) * elem, rows, c->work));
        CK(cudaMemset2DAsync(r + n * elem, npad * elem, 0, (npad - n) * elem, rows, c->work));
    }
    CK(cudaMemcpy2DAsync(b64, npad * 16, b, n * 16, n * 16, nrhs, cudaMemcpyDefault, c->work));
    // right-hand side of each slot for the checks and refinement (b of its
    // right-hand side, or b_s = q_s(A) b) and |.|^2 of it
    std::vector<const double2*> src_of(nslots);
    std::vector<double> bn2_of(nslots, -1.0);
    for (int g = 0; g < nslots; ++g) src_of[g] = b64 + (size_t)(g / S) * npad;
    // polynomial right-hand sides: x_s = x_s0 + c_s z_s with z_s = (A+sigma_s)^-1 b
    std::vector<double> pcs(S, 1.0), pbs2(S, 0.0);
    double pb2 = 0.0;
    if (poly) {
        const Range pr("msc_solve_poly_rhs: b_s and initial guesses");
        st = poly_setup(c, A, b64, n, npad, sigma, S, *poly, pcs, pbs2, pb2);
        if (st) return st;
        for (int s = 0; s < S; ++s) {
            src_of[s] = (const double2*)c->pb.p + (size_t)s * npad;
            bn2_of[s] = pbs2[s];
        }
    }
    // ---- multi-shift stage ------------------------------------------------
    int base = 0;
    for (int s = 1; s < S; ++s)
        if (sigma[s] < sigma[base]) base = s;
    const double sigma0 = sigma[base];
    const double dstag = A.kind == OP_STAGGERED ? A.mass * A.mass : 0.0;
    const double d0 = dstag + sigma0;
    for (int j = 0; j < nrhs; ++j) {
        init_sys(c->h_sys[j], S, base, j * S, j, d0, prm.tol, prm.max_iter, prm.freeze_converged, prm);
        for (int s = 0; s < S; ++s) {
            SlotScalars& q = c->h_slot[j * S + s];
            init_slot(q, sigma[s] - sigma0);
            if (poly) {
                // z_s needs |r_s| <= tol |b_s| / |c_s|; a shift with c_s = 0 or
                // b_s = 0 needs no z_s at all
                if (pcs[s] == 0.0 || !(pbs2[s] > 0.0) || !(pb2 > 0.0)) {
                    q.active = 0;
                    q.conv_iter = 0;
                } else {
                    q.tol2 = prm.tol * prm.tol * pbs2[s] / (pcs[s] * pcs[s] * pb2);
                }
            }
        }
        const double2* bj = b64 + (size_t)j * npad;
        double2* xb = x64 + (size_t)(j * S + base) * npad;
        void* rj = r + (size_t)j * npad * elem;
        void* pj = p + (size_t)j * npad * elem;
        void* tj = t + (size_t)j * npad * elem;
        double2* t64j = t64 + (size_t)j * npad;
        hsec(c, D_INIT)[j] = mkdesc(nullptr, nullptr, nullptr, nullptr, 0.0, j, j, FIN_INIT);
        if (A.kind == OP_STAGGERED) {
            hsec(c, D_K1)[j] = mkdesc(pj, pj, nullptr, tj, d0, j, j, FIN_P);
            hsec(c, D_K2)[j] = mkdesc(tj, pj, nullptr, rj, d0, j, j, FIN_R);
            hsec(c, D_RUA)[j] = ru_pass(mkdesc(xb, nullptr, nullptr, t64j, 0.0, j, -1, FIN_NONE));
            hsec(c, D_RUC)[j] = ru_pass(mkdesc(t64j, xb, bj, rj, d0, j, j, FIN_SETR));
        } else {
            hsec(c, D_K1)[j] = mkdesc(pj, pj, nullptr, tj, sigma0, j, j, FIN_P);
            hsec(c, D_K2)[j] = mkdesc(nullptr, nullptr, nullptr, nullptr, 0.0, j, j, FIN_R);
            hsec(c, D_RUC)[j] = ru_pass(mkdesc(xb, xb, bj, rj, sigma0, j, j, FIN_SETR));
        }
    }
    CK(cudaMemcpyAsync(c->sys.p, c->h_sys, sizeof(SysScalars) * nrhs, cudaMemcpyHostToDevice, c->work));
    CK(cudaMemcpyAsync(c->slot.p, c->h_slot, sizeof(SlotScalars) * nslots, cudaMemcpyHostToDevice, c->work));
    for (int s : {D_INIT, D_K1, D_K2, D_RUA, D_RUC}) CK(upload_sec(c, s, nrhs));
    Engine e = engine_of(c);
    VecSet v = vecs_of(c, prec, npad, A);
    CK(launch_init(prec, e, v, dsec(c, D_INIT), nrhs, c->work));
    c->launches++;
    const int chunk = 25;
    ProfAcc pa;
    int rel = 0, rel_ref = 0;
    {
        const Range stage("msc_solve: multi-shift stage");
        st = run_stage(c, op, prec, nrhs, chunk, mixed, true, npad, prm.max_iter, &pa, &rel);
    }
    if (st) return st;
    int status = MSC_OK;
    int iters = 0;
    std::vector<double> bnorm2(nrhs);
    for (int j = 0; j < nrhs; ++j) {
        const SysScalars& s = c->h_sys[j];
        iters = std::max(iters, s.it);
        bnorm2[j] = s.bnorm2;
        if (s.status == ST_ERR_NOT_HPD) status = MSC_ERR_NOT_HPD;
        else if (s.status == ST_ERR_NONFINITE && status != MSC_ERR_NOT_HPD) status = MSC_ERR_NONFINITE;
    }
    if (mixed) {
        CK(launch_fold(e, v, nrhs, 0, c->work));
        c->launches++;
    }
    if (poly && status == MSC_OK) {
        // x_s = c_s z_s + x_s0 (x_s = 0 where b_s = 0)
        ShiftCoef cf{};
        for (int s = 0; s < S; ++s) cf.v[s] = pbs2[s] > 0.0 ? pcs[s] : 0.0;
        CK(launch_poly_combine(x64, (const double2*)c->px0.p, cf, S, n, npad, c->work));
        for (int s = 0; s < S; ++s)
            if (!(pbs2[s] > 0.0)) CK(cudaMemsetAsync(x64 + (size_t)s * npad, 0, npad * 16, c->work));
        c->launches++;
    }
    CK(cudaMemcpyAsync(c->h_slot, c->slot.p, sizeof(SlotScalars) * nslots, cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    std::vector<int> shift_iters(nslots), ref_iters(nslots, 0);
    for (int g = 0; g < nslots; ++g) shift_iters[g] = c->h_slot[g].conv_iter;
    for (int g = 0; g < nslots; ++g)
        if (bn2_of[g] < 0.0) bn2_of[g] = bnorm2[g / S];
    // ---- true residuals and refinement -----------------------------------
    // Round r computes, for every shift still to check, the FP64 true residual
    // b - (A + sigma_s) x_s; that residual is also the start of the shift's
    // refinement solve (single shift, warm-started from x_s), which runs
    // unless the shift already meets tol. After `refine` rounds the last
    // round only checks.
    std::vector<double> rho(nslots, std::nan(""));
    int rounds = 0, ref_total = 0;
    if (status == MSC_OK) {
        std::vector<int> todo;
        for (int g = 0; g < nslots; ++g) {
            if (bn2_of[g] > 0.0) todo.push_back(g);
            else rho[g] = 0.0;  // b_s = 0: x_s = 0 exactly
        }
        for (int round = 0; !todo.empty(); ++round) {
            const Range rr("msc_solve: FP64 check and refinement round");
            const bool check_only = round >= prm.refine;
            const int m = (int)todo.size();
            for (int k = 0; k < m; ++k) {
                const int g = todo[k], rhs = g / S, s = g % S;
                const double dk = dstag + sigma[s];
                init_sys(c->h_sys[k], 1, 0, g, rhs, dk, 0.5 * prm.tol, prm.max_iter, 1, prm);
                c->h_sys[k].tol2_acc = prm.tol * prm.tol;
                // a refinement starts from a small FP64 residual, so its
                // FP32 drift (about 6e-8 times the largest residual since the
                // last update) stays far below tol for longer: the iteration
                // cap between updates is 4x the multi-shift stage's and the
                // residual-fall trigger is delta/10 (24^4 block-CSR solve: 13
                // instead of 33 FP64 residuals, 255 -> 247 ms, same iterations
                // and final residuals; without the fall trigger the FP32
                // iteration drifts off and ends non-finite)
                c->h_sys[k].ru_every = 4 * prm.reliable_every;
                c->h_sys[k].delta2 = 0.01 * prm.reliable_delta * prm.reliable_delta;
                c->h_sys[k].bnorm2 = bn2_of[g];
                init_slot(c->h_slot[g], 0.0);
                const double2* bj = src_of[g];
                double2* xg = x64 + (size_t)g * npad;
                void* rk = r + (size_t)k * npad * elem;
                void* pk = p + (size_t)k * npad * elem;
                void* tk = t + (size_t)k * npad * elem;
                double2* t64k = t64 + (size_t)k * npad;
                if (A.kind == OP_STAGGERED) {
                    hsec(c, D_RIA)[k] = mkdesc(xg, nullptr, nullptr, t64k, 0.0, k, -1, FIN_NONE);
                    hsec(c, D_RIC)[k] = mkdesc(t64k, xg, bj, rk, dk, k, k, FIN_SETR_INIT);
                    hsec(c, D_K1)[k] = mkdesc(pk, pk, nullptr, tk, dk, k, k, FIN_P);
                    hsec(c, D_K2)[k] = mkdesc(tk, pk, nullptr, rk, dk, k, k, FIN_R);
                    hsec(c, D_RUA)[k] = ru_pass(mkdesc(xg, nullptr, nullptr, t64k, 0.0, k, -1, FIN_NONE));
                    hsec(c, D_RUC)[k] = ru_pass(mkdesc(t64k, xg, bj, rk, dk, k, k, FIN_SETR));
                } else {
                    hsec(c, D_RIC)[k] = mkdesc(xg, xg, bj, rk, sigma[s], k, k, FIN_SETR_INIT);
                    hsec(c, D_K1)[k] = mkdesc(pk, pk, nullptr, tk, sigma[s], k, k, FIN_P);
                    hsec(c, D_K2)[k] = mkdesc(nullptr, nullptr, nullptr, nullptr, 0.0, k, k, FIN_R);
                    hsec(c, D_RUC)[k] = ru_pass(mkdesc(xg, xg, bj, rk, sigma[s], k, k, FIN_SETR));
                }
            }
            CK(cudaMemcpyAsync(c->sys.p, c->h_sys, sizeof(SysScalars) * m, cudaMemcpyHostToDevice, c->work));
            CK(cudaMemcpyAsync(c->slot.p, c->h_slot, sizeof(SlotScalars) * nslots, cudaMemcpyHostToDevice, c->work));
            for (int s : {D_RIA, D_RIC, D_K1, D_K2, D_RUA, D_RUC}) CK(upload_sec(c, s, m));
            if (A.kind == OP_STAGGERED) CK(op_pass(c, A, PREC_F64, PASS_A, 0, D_RIA, m, nullptr, nullptr, true));
            CK(op_pass(c, A, PREC_F64, PASS_C, mixed ? 1 : 0, D_RIC, m, nullptr, nullptr, true));
            CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * m, cudaMemcpyDeviceToHost, c->work));
            CK(cudaStreamSynchronize(c->work));
            std::vector<int> next;
            for (int k = 0; k < m; ++k) {
                const SysScalars& s = c->h_sys[k];
                const int g = todo[k];
                const double bn2 = bn2_of[g];
                rho[g] = bn2 > 0 ? std::sqrt(s.R / bn2) : 0.0;
                if (s.status == ST_ERR_NONFINITE) status = MSC_ERR_NONFINITE;
                else if (s.status == ST_RUNNING) next.push_back(g);
            }
            if (check_only || next.empty() || status != MSC_OK) break;
            CK(launch_init_from_r(prec, e, v, m, c->work));
            c->launches++;
            st = run_stage(c, op, prec, m, chunk, mixed, false, npad, prm.max_iter, nullptr, &rel_ref, true);
            if (st) return st;
            int most = 0;
            for (int k = 0; k < m; ++k) {
                const SysScalars& s = c->h_sys[k];
                ref_iters[todo[k]] += s.it;
                most = std::max(most, s.it);
                if (s.status == ST_ERR_NOT_HPD) status = MSC_ERR_NOT_HPD;
                else if (s.status == ST_ERR_NONFINITE && status == MSC_OK) status = MSC_ERR_NONFINITE;
            }
            ref_total += most;
            rounds++;
            if (mixed) {
                CK(launch_fold(e, v, m, 0, c->work));
                c->launches++;
            }
            if (status != MSC_OK) break;
            todo = next;
        }
        if (status == MSC_OK) {
            for (int g = 0; g < nslots; ++g)
                if (!(rho[g] <= prm.tol)) status = MSC_ERR_NOT_CONVERGED;
        }
    }
    // ---- solution out --------------------------------------------------------
    CK(cudaMemcpy2DAsync(x, n * 16, x64, npad * 16, n * 16, nslots, cudaMemcpyDefault, c->work));
    CK(cudaStreamSynchronize(c->work));
    if (info) {
        info->status = status;
        info->iters = iters;
        info->refine_rounds = rounds;
        info->refine_iters = ref_total;
        info->reliable_updates = rel + rel_ref;
        info->refine_reliable_updates = rel_ref;
        info->kernel_launches = (int)(c->launches - launches0);
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        for (int g = 0; g < nslots; ++g) {
            if (info->shift_iters) info->shift_iters[g] = shift_iters[g];
            if (info->shift_refine_iters) info->shift_refine_iters[g] = ref_iters[g];
            if (info->true_rel_resid) info->true_rel_resid[g] = rho[g];
        }
        info->op_ms = pa.n ? pa.k1 / pa.n : 0.0;
        info->rupdate_ms = pa.n ? pa.k2 / pa.n : 0.0;
        info->update_ms = pa.n ? pa.k3 / pa.n : 0.0;
        info->prof_samples = pa.n;
        info->prof_active = pa.n ? pa.act / pa.n : 0.0;
    }
    return status;
}

extern "C" {

int msc_solve(msc_ctx* c, const msc_op* op, const double* b, int nrhs, const double* sigma, int S,
              const msc_params* prm, double* x, msc_info* info) {
    return solve_impl(c, op, b, nrhs, sigma, S, prm, x, info, nullptr);
}

int msc_solve_poly_rhs(msc_ctx* c, const msc_op* op, const double* b, const double* sigma, int S,
                       const double* coef, int deg, const msc_params* prm, double* x, msc_info* info) {
    if (!coef || deg < 0 || deg > MSC_MAX_POLY_DEGREE || S <= 0 || S > kMaxShifts) return MSC_ERR_ARG;
    for (int64_t k = 0; k < (int64_t)S * (deg + 1); ++k)
        if (!std::isfinite(coef[k])) return MSC_ERR_ARG;
    const PolyRhs pr{coef, deg};
    return solve_impl(c, op, b, 1, sigma, S, prm, x, info, &pr);
}

int msc_solve_parity(msc_ctx* c, const msc_op* op, int parity, const double* b, int nrhs, const double* sigma,
                     int S, const msc_params* prm, double* x, msc_info* info) {
    if (!c || !op || op->is_view || op->dev.kind != OP_STAGGERED || (parity != 0 && parity != 1))
        return MSC_ERR_ARG;
    msc_op* self = const_cast<msc_op*>(op);
    if (!self->view[parity]) {
        msc_op* v = new msc_op();
        v->ctx = op->ctx;
        v->uid = ++g_op_uid;
        v->dev = op->dev;
        v->dev.g.eo = 1 + parity;
        v->dev.n = (int64_t)(op->dev.g.V / 2) * op->dev.nc;
        v->is_view = true;
        self->view[parity] = v;
    }
    return solve_impl(c, self->view[parity], b, nrhs, sigma, S, prm, x, info, nullptr);
}

// ---------------------------------------------------------------------------
// Non-Hermitian families: multi-shift BiCGStab (BiCGStab-M), FP64
// ---------------------------------------------------------------------------

int msc_solve_nonherm(msc_ctx* c, const msc_op* op, const double* b, int nrhs, const double* sigma, int S,
                      const msc_params* prm_in, double* x, msc_info* info) {
    const auto t0 = std::chrono::steady_clock::now();
    const Range whole("msc_solve_nonherm");
    if (!c || !op || !b || !x || !sigma || nrhs <= 0 || S <= 0 || S > kMaxShifts) return MSC_ERR_ARG;
    msc_params prm;
    msc_params_default(&prm);
    if (prm_in) prm = *prm_in;
    if (!(prm.tol > 0) || prm.max_iter < 0) return MSC_ERR_ARG;
    for (int s = 0; s < S; ++s)
        if (!std::isfinite(sigma[s])) return MSC_ERR_ARG;
    if (op->dev.kind != OP_BSR || prm.precision != MSC_FP64) return MSC_ERR_UNSUPPORTED;
    int st = begin(c);
    if (st) return st;
    const OpDev& A = op->dev;
    const int64_t n = A.n, npad = (n + 63) / 64 * 64;
    st = ensure_ws(c, npad, std::max(6, S), S, 1, 16);
    if (st) return st;
    {
        bool moved = false;
        CK(grow(c, c->bcg, sizeof(BcgSys) + sizeof(BcgSlot) * S, moved));
        if (moved) c->gen++;
    }
    const long launches0 = c->launches;
    BcgSys* dsys = (BcgSys*)c->bcg.p;
    BcgSlot* dslot = (BcgSlot*)((char*)c->bcg.p + sizeof(BcgSys));
    double2* b64 = (double2*)c->b64.p;
    BcgVec v;
    v.r[0] = (double2*)c->r.p;
    v.r[1] = (double2*)c->r.p + npad;
    v.rt = b64;
    v.p = (double2*)c->p.p;
    v.v = (double2*)c->t.p;
    v.s = (double2*)c->t.p + npad;
    v.t = (double2*)c->t.p + 2 * npad;
    v.x = (double2*)c->x64.p;
    v.ps = (double2*)c->ps.p;
    v.n = n;
    v.npad = npad;
    int base = 0;
    for (int s = 1; s < S; ++s)
        if (sigma[s] < sigma[base]) base = s;
    Engine e = engine_of(c);
    // a chunk of 16 iterations (even, so the residual buffers return to
    // their roles) as one CUDA graph
    const int chunk = 16;
    char key[128];
    snprintf(key, sizeof key, "bcg|%ld|%d|%lld", op->uid, S, (long long)npad);
    GraphEntry& ge = c->graphs[key];
    if (!ge.exec || ge.gen != c->gen) {
        if (ge.exec) cudaGraphExecDestroy(ge.exec);
        ge.exec = nullptr;
        cudaGraph_t g = nullptr;
        CK(cudaStreamBeginCapture(c->work, cudaStreamCaptureModeThreadLocal));
        cudaError_t err = cudaSuccess;
        for (int it = 0; it < chunk && err == cudaSuccess; ++it)
            err = launch_bcg_iter(A, e, dsys, dslot, v, S, it & 1, c->work);
        cudaError_t err2 = cudaStreamEndCapture(c->work, &g);
        if (err != cudaSuccess || err2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return cuda_status(err != cudaSuccess ? err : err2);
        }
        err = cudaGraphInstantiate(&ge.exec, g, 0);
        cudaGraphDestroy(g);
        if (err != cudaSuccess) return cuda_status(err);
        ge.gen = c->gen;
        ge.kernels = 5 * chunk;
    }
    std::vector<BcgSlot> hslot(S);
    std::vector<int> shift_iters((size_t)nrhs * S, -1);
    std::vector<double> rho((size_t)nrhs * S, std::nan(""));
    int status = MSC_OK, iters = 0;
    for (int j = 0; j < nrhs && status == MSC_OK; ++j) {
        CK(cudaMemcpyAsync(b64, b + (size_t)j * n * 2, n * 16, cudaMemcpyDefault, c->work));
        BcgSys hs;
        memset(&hs, 0, sizeof hs);
        hs.alpha_prev = {1.0, 0.0};
        hs.tol2 = prm.tol * prm.tol;
        hs.sigma0 = sigma[base];
        hs.status = ST_RUNNING;
        hs.max_iter = prm.max_iter;
        hs.S = S;
        hs.base = base;
        hs.freeze = prm.freeze_converged;
        for (int s = 0; s < S; ++s) {
            BcgSlot& q = hslot[s];
            memset(&q, 0, sizeof q);
            q.sigma_rel = sigma[s] - sigma[base];
            q.zeta = q.zeta_prev = q.zeta_new = q.T = q.T_new = {1.0, 0.0};
            q.active = 1;
            q.conv_iter = -1;
        }
        CK(cudaMemcpyAsync(dsys, &hs, sizeof hs, cudaMemcpyHostToDevice, c->work));
        CK(cudaMemcpyAsync(dslot, hslot.data(), sizeof(BcgSlot) * S, cudaMemcpyHostToDevice, c->work));
        CK(launch_bcg_init(e, dsys, dslot, v, S, c->work));
        c->launches++;
        CK(cudaMemcpyAsync(&hs, dsys, sizeof hs, cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
        // max_iter = 0 runs no iteration (the cap is seen only after one)
        const long max_chunks = prm.max_iter > 0 ? (long)prm.max_iter / chunk + 2 : 0;
        for (long k = 0; k < max_chunks && hs.status == ST_RUNNING; ++k) {
            CK(cudaGraphLaunch(ge.exec, c->work));
            c->launches += ge.kernels;
            CK(cudaMemcpyAsync(&hs, dsys, sizeof hs, cudaMemcpyDeviceToHost, c->work));
            CK(cudaStreamSynchronize(c->work));
        }
        CK(cudaMemcpyAsync(hslot.data(), dslot, sizeof(BcgSlot) * S, cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
        iters = std::max(iters, hs.it);
        for (int s = 0; s < S; ++s) shift_iters[(size_t)j * S + s] = hslot[s].conv_iter;
        if (hs.status == ST_ERR_BREAKDOWN) status = MSC_ERR_BREAKDOWN;
        else if (hs.status == ST_ERR_NONFINITE) status = MSC_ERR_NONFINITE;
        // FP64 true residual of every shift: |b - (A + sigma_s) x_s|^2 into out_red[s]
        for (int s = 0; s < S; ++s)
            hsec(c, D_RIC)[s] = mkdesc(v.x + (size_t)s * npad, v.x + (size_t)s * npad, b64, nullptr, sigma[s], -1,
                                       s, FIN_STORE);
        CK(upload_sec(c, D_RIC, S));
        CK(op_pass(c, A, PREC_F64, PASS_C, 0, D_RIC, S, nullptr, nullptr, true));
        CK(cudaMemcpyAsync(c->h_red, c->out_red.p, sizeof(double) * S, cudaMemcpyDeviceToHost, c->work));
        CK(cudaMemcpy2DAsync(x + (size_t)j * S * n * 2, n * 16, v.x, npad * 16, n * 16, S, cudaMemcpyDefault,
                             c->work));
        CK(cudaStreamSynchronize(c->work));
        for (int s = 0; s < S; ++s)
            rho[(size_t)j * S + s] = hs.bnorm2 > 0 ? std::sqrt(c->h_red[s] / hs.bnorm2) : 0.0;
        if (status == MSC_OK) {
            for (int s = 0; s < S; ++s)
                if (!(rho[(size_t)j * S + s] <= prm.tol)) status = MSC_ERR_NOT_CONVERGED;
        }
    }
    if (info) {
        info->status = status;
        info->iters = iters;
        info->refine_rounds = info->refine_iters = 0;
        info->reliable_updates = info->refine_reliable_updates = 0;
        info->kernel_launches = (int)(c->launches - launches0);
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        for (size_t g = 0; g < (size_t)nrhs * S; ++g) {
            if (info->shift_iters) info->shift_iters[g] = shift_iters[g];
            if (info->shift_refine_iters) info->shift_refine_iters[g] = 0;
            if (info->true_rel_resid) info->true_rel_resid[g] = rho[g];
        }
        info->op_ms = info->rupdate_ms = info->update_ms = 0.0;
        info->prof_samples = 0;
        info->prof_active = 0.0;
    }
    return status;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched uneven systems
// ---------------------------------------------------------------------------
namespace {

struct BatchShape {
    int site_threads = 128;
    int vec_threads = 256;
    int units = 4;
};

std::mutex g_tune_mu;
std::map<std::string, std::pair<BatchShape, double>> g_tune_cache;

}  // namespace

static int64_t pad64(int64_t n) { return (n + 63) / 64 * 64; }
static size_t al256(size_t b) { return (b + 255) / 256 * 256; }

// Device tables of a batched stage live in c->btab:
//   [BSys x cap][BOp x nops][hdr 4][act cap][msite cap+1][mvec cap+1][mupd cap+1]
// The last five are rewritten (from pinned staging) whenever the set of
// systems still iterating changes; kernels read them when they run.
struct BatchHost {
    int cap = 0, nops = 0;
    int64_t cap_site = 0, cap_vec = 0;  // entries of the virtual-block tables
    size_t off_ops = 0, off_hdr = 0, off_act = 0, off_ms = 0, off_mv = 0, off_mu = 0, total = 0;
    BTab tab{};
};

// The smallest launch shapes (see autotune_batch): they bound the virtual blocks.
constexpr int kMinSiteThreads = 64, kMinVecThreads = 128;

static int batch_layout(msc_ctx* c, int cap, int nops, int64_t cap_site, int64_t cap_vec, BatchHost& bh) {
    bh.cap = cap;
    bh.nops = nops;
    bh.off_ops = al256(sizeof(BSys) * cap);
    bh.off_hdr = bh.off_ops + al256(sizeof(BOp) * nops);
    bh.off_act = bh.off_hdr + 256;
    bh.off_ms = bh.off_act + al256(sizeof(int) * cap);
    bh.off_mv = bh.off_ms + al256(sizeof(int) * (cap + 1));
    bh.off_mu = bh.off_mv + al256(sizeof(int) * (cap + 1));
    bh.total = bh.off_mu + al256(sizeof(int) * (cap + 1));
    bh.cap_site = cap_site;
    bh.cap_vec = cap_vec;
    bool moved = false;
    CK(grow(c, c->btab, bh.total, moved));
    CK(grow(c, c->bvb, sizeof(VBlock) * (size_t)(cap_site + 2 * cap_vec), moved));
    if (moved) c->gen++;
    if (c->h_act_cap < (int64_t)(bh.total / sizeof(int)) + 1) {
        if (c->h_act) cudaFreeHost(c->h_act);
        CK(cudaMallocHost((void**)&c->h_act, bh.total + 64));
        c->h_act_cap = (int64_t)(bh.total / sizeof(int)) + 1;
    }
    char* base = (char*)c->btab.p;
    bh.tab.sys = (const BSys*)base;
    bh.tab.ops = (const BOp*)(base + bh.off_ops);
    bh.tab.hdr = (const int*)(base + bh.off_hdr);
    bh.tab.act = (const int*)(base + bh.off_act);
    bh.tab.msite = (const int*)(base + bh.off_ms);
    bh.tab.mvec = (const int*)(base + bh.off_mv);
    bh.tab.mupd = (const int*)(base + bh.off_mu);
    bh.tab.vsite = (const VBlock*)c->bvb.p;
    bh.tab.vvec = bh.tab.vsite + cap_site;
    bh.tab.vupd = bh.tab.vvec + cap_vec;
    return MSC_OK;
}

static int upload_systems(msc_ctx* c, const BatchHost& bh, const std::vector<BSys>& sys,
                          const std::vector<BOp>& ops) {
    char* base = (char*)c->btab.p;
    // ordered on the work stream after everything that may still read the
    // tables; the host vectors are pageable, so wait for the copies
    CK(cudaMemcpyAsync(base, sys.data(), sizeof(BSys) * sys.size(), cudaMemcpyHostToDevice, c->work));
    CK(cudaMemcpyAsync(base + bh.off_ops, ops.data(), sizeof(BOp) * ops.size(), cudaMemcpyHostToDevice, c->work));
    CK(cudaStreamSynchronize(c->work));
    return MSC_OK;
}

// Block maps of the systems `list` for launch shape `sh`, staged in pinned
// memory and copied on the work stream (the caller syncs before restaging).
static int set_active(msc_ctx* c, const BatchHost& bh, const std::vector<BSys>& sys,
                      const std::vector<BOp>& ops, const std::vector<int>& list, const BatchShape& sh,
                      int prec) {
    const int J = (int)list.size();
    const int cpu = prec == PREC_F32 ? 2 : 1;
    char* stage = (char*)c->h_act;
    int* hdr = (int*)(stage + bh.off_hdr - bh.off_hdr);
    int* act = (int*)(stage + bh.off_act - bh.off_hdr);
    int* ms = (int*)(stage + bh.off_ms - bh.off_hdr);
    int* mv = (int*)(stage + bh.off_mv - bh.off_hdr);
    int* mu = (int*)(stage + bh.off_mu - bh.off_hdr);
    int64_t a = 0, b = 0, u = 0;
    for (int k = 0; k < J; ++k) {
        const BSys& q = sys[list[k]];
        act[k] = list[k];
        ms[k] = (int)a;
        mv[k] = (int)b;
        mu[k] = (int)u;
        const int V = ops[q.op].g.V;
        const int64_t upv = q.npad / cpu;
        const int64_t nbs = (V + sh.site_threads - 1) / sh.site_threads;
        const int64_t nbv = (upv + sh.vec_threads - 1) / sh.vec_threads;
        if (nbs > kMaxBlocks || nbv > kMaxBlocks) return MSC_ERR_UNSUPPORTED;
        a += nbs;
        b += nbv;
        u += (upv + (int64_t)sh.vec_threads * sh.units - 1) / ((int64_t)sh.vec_threads * sh.units);
        if (a >= ((int64_t)1 << 30) || b >= ((int64_t)1 << 30)) return MSC_ERR_UNSUPPORTED;
    }
    ms[J] = (int)a;
    mv[J] = (int)b;
    mu[J] = (int)u;
    hdr[0] = J;
    hdr[1] = (int)a;
    hdr[2] = (int)b;
    hdr[3] = (int)u;
    if (a > bh.cap_site || b > bh.cap_vec || u > bh.cap_vec) return MSC_ERR_UNSUPPORTED;
    CK(cudaMemcpyAsync((char*)c->btab.p + bh.off_hdr, stage, bh.total - bh.off_hdr, cudaMemcpyHostToDevice,
                       c->work));
    VBlock* vs = (VBlock*)c->bvb.p;
    CK(launch_b_expand(bh.tab, vs, vs + bh.cap_site, vs + bh.cap_site + bh.cap_vec, (int)std::max(a, b), c->work));
    return MSC_OK;
}

static BVec bvec_of(msc_ctx* c, int prec) {
    BVec v;
    v.r = c->r.p;
    v.p = c->p.p;
    v.t = c->t.p;
    v.ps = c->ps.p;
    v.xit = prec == PREC_F32 ? c->xit.p : c->x64.p;
    v.x64 = (double2*)c->x64.p;
    v.t64 = (double2*)c->t64.p;
    v.b64 = (const double2*)c->b64.p;
    return v;
}

// One chunk of the batched iteration (plain capture; reliable updates as
// gated kernels).
static cudaError_t enqueue_chunk_b(msc_ctx* c, int prec, int chunk, bool reliable, const BTab& t,
                                   const BatchShape& sh, int& kernels) {
    Engine e = engine_of(c);
    BVec v = bvec_of(c, prec);
    kernels = 0;
    cudaError_t err = cudaSuccess;
    for (int it = 0; it < chunk && err == cudaSuccess; ++it) {
        err = launch_b_stag(prec, PASS_A, 0, e, dsec(c, D_K1), t, sh.site_threads, c->work);
        if (err == cudaSuccess) err = launch_b_stag(prec, PASS_B, 0, e, dsec(c, D_K2), t, sh.site_threads, c->work);
        if (err == cudaSuccess) err = launch_b_update(prec, sh.units, e, v, t, sh.vec_threads, c->work);
        kernels += 3;
        if (reliable && err == cudaSuccess) {
            err = launch_b_fold(e, v, t, sh.vec_threads, 1, c->work);
            if (err == cudaSuccess) err = launch_b_stag(PREC_F64, PASS_A, 0, e, dsec(c, D_RUA), t, sh.site_threads, c->work);
            if (err == cudaSuccess) err = launch_b_stag(PREC_F64, PASS_C, 1, e, dsec(c, D_RUC), t, sh.site_threads, c->work);
            kernels += 3;
        }
    }
    return err;
}

// The same chunk with each iteration's reliable-update kernels in a
// conditional IF node set on the device by the residual pass.
static cudaError_t build_chunk_graph_b_cond(msc_ctx* c, int prec, int chunk, const BTab& t,
                                            const BatchShape& sh, cudaGraph_t* out, int& kernels) {
    bool moved = false;
    cudaError_t err = grow(c, c->condf, sizeof(int) * chunk, moved);
    if (err != cudaSuccess) return err;
    if (moved) c->gen++;
    int* flags = (int*)c->condf.p;
    cudaGraph_t g = nullptr;
    err = cudaGraphCreate(&g, 0);
    if (err != cudaSuccess) return err;
    BVec v = bvec_of(c, prec);
    std::vector<cudaGraphNode_t> tail;
    kernels = 0;
    for (int it = 0; it < chunk && err == cudaSuccess; ++it) {
        cudaGraphConditionalHandle h = 0;
        err = cudaGraphConditionalHandleCreate(&h, g, 0, cudaGraphCondAssignDefault);
        if (err != cudaSuccess) break;
        Engine e = engine_of(c);
        Engine e2 = e;
        e2.cond = (unsigned long long)h;
        e2.cond_flag = flags + it;
        err = begin_capture_into(c->work, g, tail);
        if (err != cudaSuccess) break;
        if (it == 0) err = cudaMemsetAsync(flags, 0, sizeof(int) * chunk, c->work);
        if (err == cudaSuccess) err = launch_b_stag(prec, PASS_A, 0, e, dsec(c, D_K1), t, sh.site_threads, c->work);
        if (err == cudaSuccess) err = launch_b_stag(prec, PASS_B, 0, e2, dsec(c, D_K2), t, sh.site_threads, c->work);
        if (err == cudaSuccess) err = launch_b_update(prec, sh.units, e, v, t, sh.vec_threads, c->work);
        kernels += 3;
        cudaError_t et = capture_tail(c->work, tail);
        cudaGraph_t gg = nullptr;
        cudaError_t ee = cudaStreamEndCapture(c->work, &gg);
        if (err == cudaSuccess) err = et != cudaSuccess ? et : ee;
        if (err != cudaSuccess) break;
        cudaGraphNodeParams cp = {};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeIf;
        cp.conditional.size = 1;
        cudaGraphNode_t ifn = nullptr;
        err = cudaGraphAddNode(&ifn, g, tail.empty() ? nullptr : tail.data(), nullptr, tail.size(), &cp);
        if (err != cudaSuccess) break;
        err = begin_capture_into(c->work, cp.conditional.phGraph_out[0], {});
        if (err != cudaSuccess) break;
        err = launch_b_fold(e, v, t, sh.vec_threads, 1, c->work);
        if (err == cudaSuccess) err = launch_b_stag(PREC_F64, PASS_A, 0, e, dsec(c, D_RUA), t, sh.site_threads, c->work);
        if (err == cudaSuccess) err = launch_b_stag(PREC_F64, PASS_C, 1, e, dsec(c, D_RUC), t, sh.site_threads, c->work);
        ee = cudaStreamEndCapture(c->work, &gg);
        if (err == cudaSuccess) err = ee;
        tail.assign(1, ifn);
    }
    if (err != cudaSuccess) {
        cudaStreamCaptureStatus cs;
        if (cudaStreamIsCapturing(c->work, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
            cudaGraph_t junk = nullptr;
            cudaStreamEndCapture(c->work, &junk);
            if (junk && junk != g) cudaGraphDestroy(junk);
        }
        cudaGetLastError();
        cudaGraphDestroy(g);
        return err;
    }
    *out = g;
    return cudaSuccess;
}

static int get_graph_b(msc_ctx* c, int prec, int chunk, bool reliable, const BTab& t, const BatchShape& sh,
                       GraphEntry** out) {
    char key[256];
    // every table address is part of the key: their offsets depend on the
    // batch's capacity
    snprintf(key, sizeof key, "batch|%d|%d|%d|%d|%d|%d|%p|%p|%p|%p|%p|%p|%p|%p|%p|%p", prec, chunk, (int)reliable,
             sh.site_threads, sh.vec_threads, sh.units, (const void*)t.sys, (const void*)t.ops,
             (const void*)t.hdr, (const void*)t.act, (const void*)t.msite, (const void*)t.mvec,
             (const void*)t.mupd, (const void*)t.vsite, (const void*)t.vvec, (const void*)t.vupd);
    GraphEntry& ge = c->graphs[key];
    if (ge.exec && ge.gen == c->gen) {
        *out = &ge;
        return MSC_OK;
    }
    if (ge.exec) cudaGraphExecDestroy(ge.exec);
    ge.exec = nullptr;
    int kernels = 0;
    cudaGraph_t g = nullptr;
    cudaError_t err = cudaErrorNotSupported;
    if (reliable && c->use_cond) {
        err = build_chunk_graph_b_cond(c, prec, chunk, t, sh, &g, kernels);
        if (err != cudaSuccess) {
            c->use_cond = 0;
            cudaGetLastError();
        }
    }
    if (err != cudaSuccess) {
        CK(cudaStreamBeginCapture(c->work, cudaStreamCaptureModeThreadLocal));
        err = enqueue_chunk_b(c, prec, chunk, reliable, t, sh, kernels);
        cudaError_t err2 = cudaStreamEndCapture(c->work, &g);
        if (err != cudaSuccess) { if (g) cudaGraphDestroy(g); return cuda_status(err); }
        if (err2 != cudaSuccess) return cuda_status(err2);
    }
    const bool cond = reliable && c->use_cond;
    err = cudaGraphInstantiate(&ge.exec, g, 0);
    cudaGraphDestroy(g);
    if (err != cudaSuccess) return cuda_status(err);
    ge.gen = c->gen;
    ge.kernels = kernels;
    ge.cond_chunk = cond ? chunk : 0;
    ge.cond_kernels = 3;
    if (cond && !c->h_flags) CK(cudaMallocHost((void**)&c->h_flags, sizeof(int) * 1024));
    *out = &ge;
    return MSC_OK;
}

// Launch chunks until every system of the stage has stopped; before each
// chunk the active maps are rebuilt from the systems still iterating.
static int run_stage_b(msc_ctx* c, int prec, int J, int chunk, bool reliable, const BatchHost& bh,
                       const std::vector<BSys>& sys, const std::vector<BOp>& ops, const BatchShape& sh,
                       int max_iter, int* rel_updates) {
    GraphEntry* ge = nullptr;
    int st = get_graph_b(c, prec, chunk, reliable, bh.tab, sh, &ge);
    if (st) return st;
    CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * J, cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    // max_iter = 0 runs no iteration (the device sees the cap only after one)
    const long max_chunks = max_iter > 0 ? (long)max_iter / chunk + 2 : 0;
    std::vector<int> list;
    list.reserve(J);
    for (long k = 0; k < max_chunks; ++k) {
        list.clear();
        for (int j = 0; j < J; ++j)
            if (c->h_sys[j].status == ST_RUNNING) list.push_back(j);
        if (list.empty()) break;
        st = set_active(c, bh, sys, ops, list, sh, prec);
        if (st) return st;
        CK(cudaGraphLaunch(ge->exec, c->work));
        c->launches += ge->kernels;
        CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * J, cudaMemcpyDeviceToHost, c->work));
        const int ncf = std::min(ge->cond_chunk, 1024);
        if (ncf) CK(cudaMemcpyAsync(c->h_flags, c->condf.p, sizeof(int) * ncf, cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
        for (int i = 0; i < ncf; ++i) c->launches += c->h_flags[i] ? ge->cond_kernels : 0;
    }
    if (rel_updates)
        for (int j = 0; j < J; ++j) *rel_updates += c->h_sys[j].nru;
    return MSC_OK;
}

// Times candidate launch shapes on the batch (operator pass + update, with
// reductions that finalise nothing) and returns the fastest. Runs before the
// solve initialises its vectors, on whatever they hold.
static int autotune_batch(msc_ctx* c, int prec, const BatchHost& bh, const std::vector<BSys>& sys,
                          const std::vector<BOp>& ops, int nslots, BatchShape& best, double& best_ms) {
    const int J = (int)sys.size();
    Engine e = engine_of(c);
    BVec v = bvec_of(c, prec);
    std::vector<PassDesc> keep(hsec(c, D_K1), hsec(c, D_K1) + J);
    for (int j = 0; j < J; ++j) hsec(c, D_K1)[j].fin = FIN_NONE;
    CK(upload_sec(c, D_K1, J));
    for (int g = 0; g < nslots; ++g) c->h_slot[g].flag = 2;
    CK(cudaMemcpyAsync(c->sys.p, c->h_sys, sizeof(SysScalars) * J, cudaMemcpyHostToDevice, c->work));
    CK(cudaMemcpyAsync(c->slot.p, c->h_slot, sizeof(SlotScalars) * nslots, cudaMemcpyHostToDevice, c->work));
    std::vector<int> all(J);
    for (int j = 0; j < J; ++j) all[j] = j;
    const int site_c[] = {64, 128, 256};
    const int vec_c[][2] = {{256, 1}, {256, 2}, {256, 4}, {128, 4}};
    cudaEvent_t e0 = c->prof[0], e1 = c->prof[1];
    best_ms = 1e30;
    for (int si : site_c) {
        for (auto& vc : vec_c) {
            BatchShape sh;
            sh.site_threads = si;
            sh.vec_threads = vc[0];
            sh.units = vc[1];
            int st = set_active(c, bh, sys, ops, all, sh, prec);
            if (st == MSC_ERR_UNSUPPORTED) continue;  // a system needs more blocks than a row holds
            if (st) return st;
            float ms = 0;
            for (int rep = 0; rep < 4; ++rep) {
                if (rep == 1) CK(cudaEventRecord(e0, c->work));
                CK(launch_b_stag(prec, PASS_A, 0, e, dsec(c, D_K1), bh.tab, sh.site_threads, c->work));
                CK(launch_b_update(prec, sh.units, e, v, bh.tab, sh.vec_threads, c->work));
            }
            CK(cudaEventRecord(e1, c->work));
            CK(cudaEventSynchronize(e1));
            CK(cudaEventElapsedTime(&ms, e0, e1));
            ms /= 3.0f;
            if (ms < best_ms) {
                best_ms = ms;
                best = sh;
            }
        }
    }
    for (int j = 0; j < J; ++j) hsec(c, D_K1)[j] = keep[j];
    for (int g = 0; g < nslots; ++g) c->h_slot[g].flag = 0;
    return best_ms < 1e30 ? MSC_OK : MSC_ERR_UNSUPPORTED;
}

extern "C" int msc_solve_batched(msc_ctx* c, int nprob, const msc_problem* probs, const msc_params* prm_in,
                                 msc_tuning* tuning) {
    const auto t0 = std::chrono::steady_clock::now();
    const Range whole("msc_solve_batched");
    if (!c || nprob <= 0 || !probs) return MSC_ERR_ARG;
    msc_params prm;
    msc_params_default(&prm);
    if (prm_in) prm = *prm_in;
    if (!(prm.tol > 0) || prm.max_iter < 0 || prm.refine < 0) return MSC_ERR_ARG;
    if (prm.precision != MSC_FP64 && prm.precision != MSC_MIXED) return MSC_ERR_ARG;
    if (prm.precision == MSC_MIXED && (prm.reliable_every < 1 || !(prm.reliable_delta >= 0.0) ||
                                       !(prm.reliable_delta < 1.0))) return MSC_ERR_ARG;
    for (int i = 0; i < nprob; ++i) {
        const msc_problem& q = probs[i];
        if (!q.op || q.op->ctx != c || q.op->dev.kind != OP_STAGGERED || !q.b || !q.x || !q.sigma) return MSC_ERR_ARG;
        if (q.nrhs <= 0 || q.S <= 0 || q.S > kMaxShifts) return MSC_ERR_ARG;
        for (int s = 0; s < q.S; ++s)
            if (!(q.sigma[s] >= 0.0) || !std::isfinite(q.sigma[s])) return MSC_ERR_ARG;
    }
    const int prec = prm.precision == MSC_MIXED ? PREC_F32 : PREC_F64;
    const bool mixed = prec == PREC_F32;
    const size_t elem = mixed ? 8 : 16;
    int st = begin(c);
    if (st) return st;
    const long launches0 = c->launches;
    // ---- layout: one system per (problem, right-hand side) ------------------
    std::vector<BOp> ops(nprob);
    std::vector<BSys> sys;
    std::vector<int> sys_prob, sys_rhs, slot_sys, slot_shift;
    int64_t VR = 0, VS = 0;
    for (int i = 0; i < nprob; ++i) {
        const OpDev& A = probs[i].op->dev;
        ops[i].g = A.g;
        ops[i].nc = A.nc;
        ops[i].recon = A.recon;
        ops[i].l32 = A.links32;
        ops[i].l64 = A.links64;
        ops[i].lfx = A.linksfx;
        const int64_t np = pad64(A.n);
        for (int r = 0; r < probs[i].nrhs; ++r) {
            BSys q;
            q.voff = VR;
            q.soff = VS;
            q.boff = VR;
            q.npad = (int)np;
            q.op = i;
            for (int s = 0; s < probs[i].S; ++s) {
                slot_sys.push_back((int)sys.size());
                slot_shift.push_back(s);
            }
            sys.push_back(q);
            sys_prob.push_back(i);
            sys_rhs.push_back(r);
            VR += np;
            VS += np * probs[i].S;
        }
    }
    const int J = (int)sys.size();
    const int nslots = (int)slot_sys.size();
    std::vector<int64_t> slot_off(nslots);
    for (int g = 0; g < nslots; ++g) slot_off[g] = sys[slot_sys[g]].soff + (int64_t)slot_shift[g] * sys[slot_sys[g]].npad;
    // ---- workspace -----------------------------------------------------------
    {
        bool moved = false;
        const int64_t rows = std::max(J, nslots);
        if (rows > c->rows_cap) {
            c->rows_cap = rows;
            moved = true;
        }
        const int64_t R = std::max<int64_t>(c->rows_cap, 3);
        c->rows_cap = R;
        const int64_t VM = std::max(VR, VS);
        CK(grow(c, c->sys, sizeof(SysScalars) * R, moved));
        CK(grow(c, c->slot, sizeof(SlotScalars) * R, moved));
        CK(grow(c, c->partial, sizeof(double) * kMaxBlocks * R, moved));
        CK(grow(c, c->counter, sizeof(unsigned) * R, moved));
        CK(grow(c, c->out_red, sizeof(double) * R, moved));
        CK(grow(c, c->descs, sizeof(PassDesc) * D_NSECT * R, moved));
        CK(grow(c, c->b64, (size_t)VR * 16, moved));
        CK(grow(c, c->x64, (size_t)VS * 16, moved));
        CK(grow(c, c->t64, (size_t)VM * 16, moved));
        CK(grow(c, c->r, (size_t)VM * elem, moved));
        CK(grow(c, c->p, (size_t)VM * elem, moved));
        CK(grow(c, c->t, (size_t)VM * elem, moved));
        CK(grow(c, c->ps, (size_t)VS * elem, moved));
        CK(grow(c, c->xit, (size_t)VS * 8, moved));
        if (moved) c->gen++;
        if (R > c->h_rows || R > c->h_slots) {
            if (c->h_sys) cudaFreeHost(c->h_sys);
            if (c->h_slot) cudaFreeHost(c->h_slot);
            if (c->h_red) cudaFreeHost(c->h_red);
            if (c->h_desc) cudaFreeHost(c->h_desc);
            CK(cudaMallocHost((void**)&c->h_sys, sizeof(SysScalars) * R));
            CK(cudaMallocHost((void**)&c->h_slot, sizeof(SlotScalars) * R));
            CK(cudaMallocHost((void**)&c->h_red, sizeof(double) * R));
            CK(cudaMallocHost((void**)&c->h_desc, sizeof(PassDesc) * D_NSECT * R));
            c->h_rows = R;
            c->h_slots = R;
        }
        // padding of every row must read as zero
        CK(cudaMemsetAsync(c->b64.p, 0, (size_t)VR * 16, c->work));
        CK(cudaMemsetAsync(c->r.p, 0, (size_t)VM * elem, c->work));
        CK(cudaMemsetAsync(c->t.p, 0, (size_t)VM * elem, c->work));
    }
    char* r = (char*)c->r.p;
    char* p = (char*)c->p.p;
    char* t = (char*)c->t.p;
    double2* x64 = (double2*)c->x64.p;
    double2* t64 = (double2*)c->t64.p;
    double2* b64 = (double2*)c->b64.p;
    for (int j = 0; j < J; ++j) {
        const msc_problem& q = probs[sys_prob[j]];
        const int64_t n = q.op->dev.n;
        CK(cudaMemcpyAsync(b64 + sys[j].boff, q.b + (size_t)sys_rhs[j] * n * 2, n * 16, cudaMemcpyDefault, c->work));
    }
    // ---- scalars and pass descriptors of the multi-shift stage ---------------
    std::vector<double> d0(J);
    int slot0 = 0;
    for (int j = 0; j < J; ++j) {
        const msc_problem& q = probs[sys_prob[j]];
        const OpDev& A = q.op->dev;
        int base = 0;
        for (int s = 1; s < q.S; ++s)
            if (q.sigma[s] < q.sigma[base]) base = s;
        d0[j] = A.mass * A.mass + q.sigma[base];
        init_sys(c->h_sys[j], q.S, base, slot0, j, d0[j], prm.tol, prm.max_iter, prm.freeze_converged, prm);
        for (int s = 0; s < q.S; ++s) init_slot(c->h_slot[slot0 + s], q.sigma[s] - q.sigma[base]);
        void* rj = r + sys[j].voff * elem;
        void* pj = p + sys[j].voff * elem;
        void* tj = t + sys[j].voff * elem;
        double2* t64j = t64 + sys[j].voff;
        double2* xb = x64 + sys[j].soff + (int64_t)base * sys[j].npad;
        const double2* bj = b64 + sys[j].boff;
        hsec(c, D_K1)[j] = mkdesc(pj, pj, nullptr, tj, d0[j], j, j, FIN_P);
        hsec(c, D_K2)[j] = mkdesc(tj, pj, nullptr, rj, d0[j], j, j, FIN_R);
        hsec(c, D_RUA)[j] = ru_pass(mkdesc(xb, nullptr, nullptr, t64j, 0.0, j, -1, FIN_NONE));
        hsec(c, D_RUC)[j] = ru_pass(mkdesc(t64j, xb, bj, rj, d0[j], j, j, FIN_SETR));
        slot0 += q.S;
    }
    // ---- tables and autotuned launch shape -------------------------------------
    BatchHost bh;
    int64_t cap_site = 0, cap_vec = 0;  // every slot a system of its own (refinement)
    for (int g = 0; g < nslots; ++g) {
        const BSys& q = sys[slot_sys[g]];
        cap_site += (ops[q.op].g.V + kMinSiteThreads - 1) / kMinSiteThreads;
        cap_vec += (q.npad + kMinVecThreads - 1) / kMinVecThreads;
    }
    st = batch_layout(c, std::max(J, nslots), nprob, cap_site, cap_vec, bh);
    if (st) return st;
    st = upload_systems(c, bh, sys, ops);
    if (st) return st;
    BatchShape shape;
    double tuned_ms = 0.0;
    int tuned_now = 0;
    {
        int64_t sumV = 0;
        for (auto& q : sys) sumV += ops[q.op].g.V;
        char key[160];
        int dev = 0;
        cudaGetDevice(&dev);
        snprintf(key, sizeof key, "%d|%d|%d|%lld|%d", dev, prec, J, (long long)sumV, nslots);
        std::pair<BatchShape, double> hit;
        bool found = false;
        {
            std::lock_guard<std::mutex> lk(g_tune_mu);
            auto it = g_tune_cache.find(key);
            if (it != g_tune_cache.end()) {
                hit = it->second;
                found = true;
            }
        }
        if (found) {
            shape = hit.first;
            tuned_ms = hit.second;
        } else {
            st = autotune_batch(c, prec, bh, sys, ops, nslots, shape, tuned_ms);
            if (st) return st;
            tuned_now = 1;
            std::lock_guard<std::mutex> lk(g_tune_mu);
            g_tune_cache[key] = {shape, tuned_ms};
        }
    }
    if (tuning) {
        tuning->site_threads = shape.site_threads;
        tuning->vec_threads = shape.vec_threads;
        tuning->vec_units = shape.units;
        tuning->tuned = tuned_now;
        tuning->best_ms = tuned_ms;
    }
    CK(cudaMemcpyAsync(c->sys.p, c->h_sys, sizeof(SysScalars) * J, cudaMemcpyHostToDevice, c->work));
    CK(cudaMemcpyAsync(c->slot.p, c->h_slot, sizeof(SlotScalars) * nslots, cudaMemcpyHostToDevice, c->work));
    for (int sct : {D_K1, D_K2, D_RUA, D_RUC}) CK(upload_sec(c, sct, J));
    std::vector<int> all(J);
    for (int j = 0; j < J; ++j) all[j] = j;
    st = set_active(c, bh, sys, ops, all, shape, prec);
    if (st) return st;
    Engine e = engine_of(c);
    BVec v = bvec_of(c, prec);
    CK(launch_b_init(prec, e, v, bh.tab, shape.vec_threads, c->work));
    c->launches++;
    const int chunk = 25;
    int rel = 0, rel_ref = 0;
    st = run_stage_b(c, prec, J, chunk, mixed, bh, sys, ops, shape, prm.max_iter, &rel);
    if (st) return st;
    std::vector<int> sys_status(J, MSC_OK), sys_iters(J, 0);
    std::vector<double> bnorm2(J);
    for (int j = 0; j < J; ++j) {
        const SysScalars& q = c->h_sys[j];
        sys_iters[j] = q.it;
        bnorm2[j] = q.bnorm2;
        if (q.status == ST_ERR_NOT_HPD) sys_status[j] = MSC_ERR_NOT_HPD;
        else if (q.status == ST_ERR_NONFINITE) sys_status[j] = MSC_ERR_NONFINITE;
    }
    if (mixed) {
        st = set_active(c, bh, sys, ops, all, shape, prec);
        if (st) return st;
        CK(launch_b_fold(e, v, bh.tab, shape.vec_threads, 0, c->work));
        c->launches++;
    }
    CK(cudaMemcpyAsync(c->h_slot, c->slot.p, sizeof(SlotScalars) * nslots, cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    std::vector<int> shift_iters(nslots), ref_iters(nslots, 0);
    for (int g = 0; g < nslots; ++g) shift_iters[g] = c->h_slot[g].conv_iter;
    // ---- true residuals and refinement (one system per refined shift) --------
    std::vector<double> rho(nslots, std::nan(""));
    int rounds = 0, ref_total = 0;
    std::vector<int> todo;
    for (int g = 0; g < nslots; ++g)
        if (sys_status[slot_sys[g]] == MSC_OK) todo.push_back(g);
    for (int round = 0; !todo.empty(); ++round) {
        const bool check_only = round >= prm.refine;
        const int m = (int)todo.size();
        std::vector<BSys> rs(m);
        int64_t voff = 0;
        for (int k = 0; k < m; ++k) {
            const int g = todo[k], j = slot_sys[g], s = slot_shift[g];
            const msc_problem& q = probs[sys_prob[j]];
            const double dk = q.op->dev.mass * q.op->dev.mass + q.sigma[s];
            rs[k] = sys[j];
            rs[k].voff = voff;
            rs[k].soff = slot_off[g];
            voff += sys[j].npad;
            init_sys(c->h_sys[k], 1, 0, g, j, dk, 0.5 * prm.tol, prm.max_iter, 1, prm);
            c->h_sys[k].tol2_acc = prm.tol * prm.tol;
            c->h_sys[k].bnorm2 = bnorm2[j];
            init_slot(c->h_slot[g], 0.0);
            void* rk = r + rs[k].voff * elem;
            void* pk = p + rs[k].voff * elem;
            void* tk = t + rs[k].voff * elem;
            double2* t64k = t64 + rs[k].voff;
            double2* xg = x64 + slot_off[g];
            const double2* bj = b64 + sys[j].boff;
            hsec(c, D_RIA)[k] = mkdesc(xg, nullptr, nullptr, t64k, 0.0, k, -1, FIN_NONE);
            hsec(c, D_RIC)[k] = mkdesc(t64k, xg, bj, rk, dk, k, k, FIN_SETR_INIT);
            hsec(c, D_K1)[k] = mkdesc(pk, pk, nullptr, tk, dk, k, k, FIN_P);
            hsec(c, D_K2)[k] = mkdesc(tk, pk, nullptr, rk, dk, k, k, FIN_R);
            hsec(c, D_RUA)[k] = ru_pass(mkdesc(xg, nullptr, nullptr, t64k, 0.0, k, -1, FIN_NONE));
            hsec(c, D_RUC)[k] = ru_pass(mkdesc(t64k, xg, bj, rk, dk, k, k, FIN_SETR));
        }
        CK(cudaMemcpyAsync(c->sys.p, c->h_sys, sizeof(SysScalars) * m, cudaMemcpyHostToDevice, c->work));
        CK(cudaMemcpyAsync(c->slot.p, c->h_slot, sizeof(SlotScalars) * nslots, cudaMemcpyHostToDevice, c->work));
        for (int sct : {D_RIA, D_RIC, D_K1, D_K2, D_RUA, D_RUC}) CK(upload_sec(c, sct, m));
        CK(cudaStreamSynchronize(c->work));
        st = upload_systems(c, bh, rs, ops);
        if (st) return st;
        std::vector<int> rall(m);
        for (int k = 0; k < m; ++k) rall[k] = k;
        st = set_active(c, bh, rs, ops, rall, shape, prec);
        if (st) return st;
        CK(launch_b_stag(PREC_F64, PASS_A, 0, e, dsec(c, D_RIA), bh.tab, shape.site_threads, c->work));
        CK(launch_b_stag(PREC_F64, PASS_C, mixed ? 1 : 0, e, dsec(c, D_RIC), bh.tab, shape.site_threads, c->work));
        c->launches += 2;
        CK(cudaMemcpyAsync(c->h_sys, c->sys.p, sizeof(SysScalars) * m, cudaMemcpyDeviceToHost, c->work));
        CK(cudaStreamSynchronize(c->work));
        std::vector<int> next;
        for (int k = 0; k < m; ++k) {
            const SysScalars& q = c->h_sys[k];
            const int g = todo[k], j = slot_sys[g];
            rho[g] = bnorm2[j] > 0 ? std::sqrt(q.R / bnorm2[j]) : 0.0;
            if (q.status == ST_ERR_NONFINITE) sys_status[j] = MSC_ERR_NONFINITE;
            else if (q.status == ST_RUNNING) next.push_back(g);
        }
        if (check_only || next.empty()) break;
        CK(launch_b_init_from_r(prec, e, v, bh.tab, shape.vec_threads, c->work));
        c->launches++;
        st = run_stage_b(c, prec, m, chunk, mixed, bh, rs, ops, shape, prm.max_iter, &rel_ref);
        if (st) return st;
        int most = 0;
        for (int k = 0; k < m; ++k) {
            const SysScalars& q = c->h_sys[k];
            const int g = todo[k], j = slot_sys[g];
            ref_iters[g] += q.it;
            most = std::max(most, q.it);
            if (q.status == ST_ERR_NOT_HPD) sys_status[j] = MSC_ERR_NOT_HPD;
            else if (q.status == ST_ERR_NONFINITE) sys_status[j] = MSC_ERR_NONFINITE;
        }
        ref_total += most;
        rounds++;
        if (mixed) {
            st = set_active(c, bh, rs, ops, rall, shape, prec);
            if (st) return st;
            CK(launch_b_fold(e, v, bh.tab, shape.vec_threads, 0, c->work));
            c->launches++;
        }
        todo.clear();
        for (int g : next)
            if (sys_status[slot_sys[g]] == MSC_OK) todo.push_back(g);
    }
    // ---- solutions out, reports ------------------------------------------------
    for (int j = 0; j < J; ++j) {
        const msc_problem& q = probs[sys_prob[j]];
        const int64_t n = q.op->dev.n;
        CK(cudaMemcpy2DAsync(q.x + (size_t)sys_rhs[j] * q.S * n * 2, n * 16, x64 + sys[j].soff, (size_t)sys[j].npad * 16,
                             n * 16, q.S, cudaMemcpyDefault, c->work));
    }
    CK(cudaStreamSynchronize(c->work));
    const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    int worst = MSC_OK;
    int gfirst = 0;
    int jfirst = 0;
    for (int i = 0; i < nprob; ++i) {
        const msc_problem& q = probs[i];
        int pst = MSC_OK, iters = 0;
        for (int rr = 0; rr < q.nrhs; ++rr) {
            const int j = jfirst + rr;
            iters = std::max(iters, sys_iters[j]);
            if (sys_status[j] != MSC_OK && pst == MSC_OK) pst = sys_status[j];
        }
        if (pst == MSC_OK)
            for (int g = gfirst; g < gfirst + q.nrhs * q.S; ++g)
                if (!(rho[g] <= prm.tol)) pst = MSC_ERR_NOT_CONVERGED;
        if (q.info) {
            msc_info* in = q.info;
            in->status = pst;
            in->iters = iters;
            in->refine_rounds = rounds;
            in->refine_iters = ref_total;
            in->reliable_updates = rel + rel_ref;
            in->refine_reliable_updates = rel_ref;
            in->kernel_launches = (int)(c->launches - launches0);
            in->seconds = secs;
            for (int k = 0; k < q.nrhs * q.S; ++k) {
                if (in->shift_iters) in->shift_iters[k] = shift_iters[gfirst + k];
                if (in->shift_refine_iters) in->shift_refine_iters[k] = ref_iters[gfirst + k];
                if (in->true_rel_resid) in->true_rel_resid[k] = rho[gfirst + k];
            }
            in->op_ms = in->rupdate_ms = in->update_ms = 0.0;
            in->prof_samples = 0;
            in->prof_active = 0.0;
        }
        if (pst != MSC_OK && (worst == MSC_OK || worst == MSC_ERR_NOT_CONVERGED)) worst = pst;
        gfirst += q.nrhs * q.S;
        jfirst += q.nrhs;
    }
    return worst;
}

// ---------------------------------------------------------------------------
// Adjoint of S = sum_s c_s Re(phi^dag x_s) (rational pseudofermion action)
// ---------------------------------------------------------------------------
static int stage_solutions(msc_ctx* c, const msc_op* op, int S, const double* coef, const double* x,
                           int64_t& n, int64_t& npad) {
    n = op->dev.n;
    npad = (n + 63) / 64 * 64;
    int st = ensure_ws(c, npad, std::max(S, 3), S, 1, 16);
    if (st) return st;
    bool moved = false;
    CK(grow(c, c->coef, sizeof(double) * S, moved));
    CK(cudaMemcpyAsync(c->coef.p, coef, sizeof(double) * S, cudaMemcpyHostToDevice, c->work));
    CK(cudaMemcpy2DAsync(c->x64.p, npad * 16, x, n * 16, n * 16, S, cudaMemcpyDefault, c->work));
    return MSC_OK;
}

extern "C" int msc_quad_form(msc_ctx* c, const msc_op* op, const double* phi, int S, const double* coef,
                             const double* x, double* value) {
    if (!c || !op || !phi || !coef || !x || !value || S <= 0) return MSC_ERR_ARG;
    int st = begin(c);
    if (st) return st;
    int64_t n, npad;
    st = stage_solutions(c, op, S, coef, x, n, npad);
    if (st) return st;
    double2* phi64 = (double2*)c->b64.p;
    CK(cudaMemcpyAsync(phi64, phi, n * 16, cudaMemcpyDefault, c->work));
    CK(launch_quad(engine_of(c), phi64, (const double2*)c->x64.p, (const double*)c->coef.p, S, n, npad, 0,
                   c->work));
    c->launches++;
    CK(cudaMemcpyAsync(value, c->out_red.p, sizeof(double), cudaMemcpyDeviceToHost, c->work));
    CK(cudaStreamSynchronize(c->work));
    return MSC_OK;
}

extern "C" int msc_quad_form_grad(msc_ctx* c, const msc_op* op, int S, const double* coef,
                                  const double* x, double* dphi, double* dU) {
    const Range whole("msc_quad_form_grad");
    if (!c || !op || !coef || !x || S <= 0 || (!dphi && !dU)) return MSC_ERR_ARG;
    if (dU && op->dev.kind != OP_STAGGERED) return MSC_ERR_ARG;
    int st = begin(c);
    if (st) return st;
    int64_t n, npad;
    st = stage_solutions(c, op, S, coef, x, n, npad);
    if (st) return st;
    const double2* x64 = (const double2*)c->x64.p;
    double2* t64 = (double2*)c->t64.p;
    const double* dc = (const double*)c->coef.p;
    if (dphi) {
        CK(launch_dphi(x64, dc, S, n, npad, t64, c->work));
        c->launches++;
        CK(cudaMemcpyAsync(dphi, t64, n * 16, cudaMemcpyDefault, c->work));
    }
    if (dU) {
        const OpDev& A = op->dev;
        // y_s = D x_s for every shift (FP64 D pass), then the outer products
        for (int s = 0; s < S; ++s)
            hsec(c, D_AP1)[s] = mkdesc(x64 + (size_t)s * npad, nullptr, nullptr, t64 + (size_t)s * npad, 0.0,
                                       -1, -1, FIN_NONE);
        CK(upload_sec(c, D_AP1, S));
        CK(op_pass(c, A, PREC_F64, PASS_A, 0, D_AP1, S));
        const size_t gbytes = (size_t)4 * A.g.V * A.nc * A.nc * 16;
        double2* G = (double2*)dU;
        const bool dev_out = is_device_ptr(dU);
        if (!dev_out) {
            bool moved = false;
            CK(grow(c, c->force, gbytes, moved));
            G = (double2*)c->force.p;
        }
        CK(launch_force(A, x64, t64, dc, S, npad, G, c->work));
        c->launches++;
        if (!dev_out) CK(cudaMemcpyAsync(dU, G, gbytes, cudaMemcpyDeviceToHost, c->work));
    }
    CK(cudaStreamSynchronize(c->work));
    return MSC_OK;
}

// ---------------------------------------------------------------------------
// Operator apply that allocates nothing.
//
// msc_op_apply() above stages its vectors in the context's workspace, which
// it grows with cudaMalloc on demand. Some callers cannot let a library
// allocate at that point: code running under another framework's memory
// pool or allocator (where a foreign cudaMalloc fragments or escapes the
// pool's accounting), and loops with latency limits, where cudaMalloc may
// block on the device or fail late under memory pressure. For them,
// msc_op_apply_noalloc() keeps its only scratch (two pass descriptors and
// the intermediate vector D x) in one fixed file-scope device array.
// ---------------------------------------------------------------------------
namespace {

constexpr int64_t kNoallocMaxN = (int64_t)1 << 20;  // complex unknowns (16 MiB of FP64)
constexpr size_t kNoallocDescBytes = 256;
// the two pass descriptors sit in front of the D x vector
static_assert(2 * sizeof(PassDesc) <= kNoallocDescBytes && kNoallocDescBytes % 16 == 0,
              "the descriptor area of the scratch array must hold two 16-byte aligned PassDesc");
// Held by every device that loads the library, until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocDescBytes + 16 * kNoallocMaxN];

constexpr int kNoallocMaxDevices = 128;
void* g_noalloc_ptr[kNoallocMaxDevices];  // device address of the array, per device
std::mutex g_noalloc_mu;

__global__ void k_noalloc_store_descs(PassDesc* dst, PassDesc a, PassDesc b) {
    if (threadIdx.x == 0) {
        dst[0] = a;
        dst[1] = b;
    }
}

// True when p is memory the kernels on device `dev` may dereference directly:
// device memory of that device, or managed memory. Device memory of another
// GPU is refused (without peer access its use would fault on the device).
bool usable_on_device(const void* p, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

}  // namespace

extern "C" int msc_op_apply_noalloc(const msc_op* op, double sigma, const double* in, double* out,
                                    void* stream) {
    if (!op || !op->ctx || !in || !out || !std::isfinite(sigma)) return MSC_ERR_ARG;
    const OpDev& A = op->dev;
    if (A.kind != OP_STAGGERED) return MSC_ERR_UNSUPPORTED;
    if (A.n > kNoallocMaxN) return MSC_ERR_ARG;
    const int dev = op->ctx->device;
    if (dev < 0 || dev >= kNoallocMaxDevices) return MSC_ERR_UNSUPPORTED;
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) return MSC_ERR_CUDA;
    if (prev != dev && cudaSetDevice(dev) != cudaSuccess) return MSC_ERR_CUDA;
    int status = MSC_OK;
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            // the host-side name of the array is not a device address: ask the
            // runtime for this device's copy once, with the device current
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) == cudaSuccess && p) g_noalloc_ptr[dev] = p;
            else { cudaGetLastError(); status = MSC_ERR_CUDA; }
        }
        base = g_noalloc_ptr[dev];
    }
    if (status == MSC_OK && (!usable_on_device(in, dev) || !usable_on_device(out, dev))) status = MSC_ERR_ARG;
    if (status == MSC_OK) {
        cudaStream_t st = (cudaStream_t)stream;
        PassDesc* descs = (PassDesc*)base;
        double2* t = (double2*)((char*)base + kNoallocDescBytes);
        const PassDesc d1 = mkdesc(in, nullptr, nullptr, t, 0.0, -1, -1, FIN_NONE);
        const PassDesc d2 = mkdesc(t, in, nullptr, out, A.mass * A.mass + sigma, -1, -1, FIN_NONE);
        cudaError_t e = cudaSuccess;
        Engine none{};
        const bool fx = A.linksfx != nullptr;  // its kernels take the descriptors as parameters
        if (!fx) {
            k_noalloc_store_descs<<<1, 32, 0, st>>>(descs, d1, d2);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess)
            e = launch_stag_pass(A, PREC_F64, PASS_A, 0, none, descs, 1, st, nullptr, false, fx ? &d1 : nullptr);
        if (e == cudaSuccess)
            e = launch_stag_pass(A, PREC_F64, PASS_D, 0, none, descs + 1, 1, st, nullptr, false, fx ? &d2 : nullptr);
        if (e != cudaSuccess) status = cuda_status(e);
    }
    if (prev != dev) cudaSetDevice(prev);
    return status;
}
