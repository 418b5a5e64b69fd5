// fdph.cu -- device side of the FDP=H time step and the C ABI (include/fdph.h).
//
// Steps run in blocks of up to 16 (step.cuh), a launch per kernel and block: FIR + scatter and transient + Eq. 39
// on two side streams, beside the near field, all joined before the gather.  (Whole rupture blocks, and the
// steps of the delayed-history form, replay a captured graph.)  Causality (min(dm + delay) >= 1, checked at plan
// time) guarantees that the ring slots read at step n were completed by steps < n and that the slots written
// at step n are not read; where min(dm + delay) is less than the block's length, Eq. 39 follows the scatter.
// The near field runs on the CUDA cores (FP64, FP32, and FP16 windows of one right-hand side, step.cuh) or on the
// tensor cores (FP16 windows of several, tensor.cuh).  Several right-hand sides go through one launch.  A rupture
// block (Sec. 6.2) takes what the slip rates before the block do to all its steps at once, then step by step its
// own part, the friction law and the push, then commits the block.  A batch runs its plans on their own
// streams, ordered with one another around each call.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <omp.h>
#include <stdlib.h>

#include <algorithm>
#include <climits>
#include <type_traits>
#include <chrono>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/fdph.h"
#include "internal.h"
#include "kernel2d.cuh"
#include "plan.h"
#include "step.cuh"
#include "tensor.cuh"

namespace fdph {

static thread_local std::string g_last_error;
void set_error(const std::string& msg) { g_last_error = msg; }

}  // namespace fdph

using namespace fdph;

#define FDPH_CUDA(call)                                                                      \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess) {                                                             \
            set_error(std::string(#call) + ": " + cudaGetErrorString(e_));                   \
            return FDPH_E_CUDA;                                                              \
        }                                                                                    \
    } while (0)

static const int kChunk = 64;      // steps of exact kernel per near-field work item at most
static_assert(kRingRoom == kBlk - 1, "the rings leave room for one block of steps");

// FP32 copy of a restored slip-rate ring
__global__ void ring_to_float_kernel(const double* x, float* y, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = (float)x[i];
}

// One ring of a saved state.  It is saved with the slots that one step needs (row of step s at s modulo that
// number), not with the room that a block of steps takes beside them.
struct RingMap {
    long long saved, dev;     // first double of the ring as saved and in device memory
    int rows, room_rows;      // slots as saved and in device memory
    int width, top;           // doubles of a slot, newest step
};

// Doubles x0 ... x1 - 1 of the saved form of an array of rings (in order of `saved`), to or from stage[0 ...]
__global__ void copy_rings_kernel(const RingMap* maps, int n, long long x0, long long x1, double* dev, double* stage,
                                  bool save) {
    for (long long x = x0 + (long long)blockIdx.x * blockDim.x + threadIdx.x; x < x1; x += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (maps[mid].saved <= x) lo = mid; else hi = mid - 1;
        }
        const RingMap g = maps[lo];
        const int slot = (int)((x - g.saved) / g.width), col = (int)((x - g.saved) % g.width);
        const int step = g.top - wrap(g.top - slot, g.rows);   // the step of that slot among the newest g.rows
        double* d = dev + g.dev + (long long)wrap(step, g.room_rows) * g.width + col;
        if (save) stage[x - x0] = *d;
        else *d = stage[x - x0];
    }
}

// Bounded mbarrier wait (PTX)
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_wait_limit(unsigned long long* bar, unsigned phase, long long limit) {
    const unsigned a = smem_u32(bar);
    for (long long it = 0; it < limit; ++it) {
        unsigned ok;
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(a), "r"(phase)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// Self-test of the bounded wait: one CTA waits on an mbarrier that no thread ever completes; the
// wait gives up after `limit` polls and records the timeout in err, and the kernel returns (no
// copy is in flight), so the context stays usable.
__global__ void wait_selftest_kernel(long long limit, int* err) {
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bar)), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait_limit(&bar, 0u, limit)) atomicExch(err, kErrTimeout);
}

// the longest work item (window slices) of a plan
static inline int near_max_chunk(int nrhs, int precision) {
    if (nrhs >= 2 && precision == FDPH_FP16) return kChunk;
    return (nrhs >= 2 && precision != FDPH_FP64 ? 2 * kChunk : kChunk) / nrhs;
}

// the longest aux item: all of a leaf's static tile and tail slices, or half of them where
// there is less than one leaf per scheduler (152 SMs x 4): one item of all 17 slices then takes as
// long as the rest of the step (curved N = 1024, 422 leaves: 0.95 -> 0.80 ms per 64 steps; with 1963 leaves the
// split costs 2.18 -> 2.38 ms)
static inline int near_aux_chunk(int leaves) { return leaves >= 4 * 152 ? 1 + kMaxSoe : 9; }

// ------------------------------------------------------------------------------------------
// plan-time device kernels: near-field windows and exact-kernel tensors

struct GeoDev {
    const double *px, *py, *nx, *ny, *ax, *ay, *tx, *ty, *len;
};

__device__ __forceinline__ Seg dev_seg(const GeoDev& g, int p) {
    Seg s;
    s.ax = g.ax[p];
    s.ay = g.ay[p];
    s.tx = g.tx[p];
    s.ty = g.ty[p];
    s.len = g.len[p];
    return s;
}

// m_S(i, j) = 1 + last k < M with |K_ijk - Kstat_ij dt| >= thr (App. H), 0 if none; M if thr == 0.
// The scan covers only the steps before the tail bound (stress_tail_bound) falls below thr / 2, so it
// costs the pair's wave passage plus its decay to thr rather than M steps.
__global__ void near_ms_kernel(GeoDev g, const int* pr, const int* pnr, const int* ps, const int* pns,
                               const long long* pair0, long long npairs, int nleaf, int M, double dt,
                               double mu, double c, double thr, int* ms) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= npairs) return;
    int lo = 0, hi = nleaf - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pair0[mid] <= q) lo = mid; else hi = mid - 1;
    }
    const long long loc = q - pair0[lo];
    const int il = (int)(loc / pns[lo]), jl = (int)(loc % pns[lo]);
    const int pi = pr[lo] + il, pj = ps[lo] + jl;
    if (thr <= 0.0) {
        ms[q] = M;
        return;
    }
    const Seg s = dev_seg(g, pj);
    // steps from the first k whose tail bound is below thr / 2 on cannot reach thr (the bound falls
    // with k; the factor 2 covers rounding): the backward scan starts below that k
    int k_lo = 0, k_hi = M;
    while (k_lo < k_hi) {
        const int mid = (k_lo + k_hi) >> 1;
        if (stress_tail_bound(g.px[pi], g.py[pi], s, (double)mid * dt, dt, mu, c) < 0.5 * thr)
            k_hi = mid;
        else
            k_lo = mid + 1;
    }
    int res = 0;
    for (int k = k_lo - 1; k >= 0; --k) {
        const Stress2 v = stress_tail(g.px[pi], g.py[pi], s, (double)k * dt, (double)(k + 1) * dt, mu, c);
        const double tval = g.nx[pi] * v.x + g.ny[pi] * v.y;
        if (fabs(tval) >= thr) {
            res = k + 1;
            break;
        }
    }
    ms[q] = res;
}

// coefficients [k][j][i] for k < W: exact kernel below m_S(i, j), static * dt above
template <class H, class A>
__global__ void near_fill_kernel(GeoDev g, NearDev L, const int* ms_leaf, double dt, double mu, double c,
                                 double kscale, H* tensor, A* stat) {
    const long long total = (long long)L.W * L.ns * L.nr;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int il = (int)(q % L.nr);
        const long long r = q / L.nr;
        const int jl = (int)(r % L.ns);
        const int k = (int)(r / L.ns);
        const int pi = L.r0 + il, pj = L.s0 + jl;
        const Seg s = dev_seg(g, pj);
        double v;
        const int mS = ms_leaf[il * L.ns + jl];
        if (k < mS) {
            const Stress2 w = stress_jump(g.px[pi], g.py[pi], s, (double)k * dt, (double)(k + 1) * dt, mu, c);
            v = g.nx[pi] * w.x + g.ny[pi] * w.y;
        } else {
            const Stress2 w = stress_static(g.px[pi], g.py[pi], s, mu);
            v = (g.nx[pi] * w.x + g.ny[pi] * w.y) * dt;
        }
        constexpr int vh = 16 / (int)sizeof(H), va = 16 / (int)sizeof(A);   // source-interleaved slices (plan.h)
        tensor[L.tensor + (long long)k * L.sl + ((jl / vh) * L.nr + il) * vh + jl % vh] = (H)(v * kscale);
        if (k == 0) {
            const Stress2 w = stress_static(g.px[pi], g.py[pi], s, mu);
            stat[L.stat + ((jl / va) * L.nr + il) * va + jl % va] = (A)((g.nx[pi] * w.x + g.ny[pi] * w.y) * dt);
        }
    }
}

// projections g_q = sum_{k' < M - W} rho_q^k' (K_ij,W+k' - Kstat_ij dt) of every pair of the
// inadmissible leaves with a tail, on the exponential basis (least-squares right-hand sides);
// one thread per pair, pairs of leaf l at [pair0[l], pair0[l + 1])
__global__ void near_soe_proj_kernel(GeoDev g, const NearDev* leaves, const long long* pair0, int nleaf,
                                     long long npairs, int M, double dt, double mu, double c, int Q,
                                     const double* rho, double* out) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= npairs) return;
    int lo = 0, hi = nleaf - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pair0[mid] <= q) lo = mid; else hi = mid - 1;
    }
    const NearDev L = leaves[lo];
    const long long loc = q - pair0[lo];
    const int il = (int)(loc / L.ns), jl = (int)(loc % L.ns);
    const int pi = L.r0 + il, pj = L.s0 + jl;
    const Seg s = dev_seg(g, pj);
    double acc[kMaxSoe], pw[kMaxSoe];
#pragma unroll
    for (int r = 0; r < kMaxSoe; ++r) {
        acc[r] = 0.0;
        pw[r] = 1.0;
    }
    for (int k = L.W; k < M; ++k) {
        const Stress2 v = stress_tail(g.px[pi], g.py[pi], s, (double)k * dt, (double)(k + 1) * dt, mu, c);
        const double y = g.nx[pi] * v.x + g.ny[pi] * v.y;
#pragma unroll
        for (int r = 0; r < kMaxSoe; ++r)
            if (r < Q) {
                acc[r] += pw[r] * y;
                pw[r] *= rho[r];
            }
    }
#pragma unroll
    for (int r = 0; r < kMaxSoe; ++r)
        if (r < Q) out[(size_t)q * Q + r] = acc[r];
}

// ------------------------------------------------------------------------------------------
// the plan object

struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
};

struct fdph_plan_s {
    int device = 0;
    int precision = FDPH_FP64;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int N = 0, M = 0, n = 0, WD = 1, WC = 1;
    int nrhs = 1;             // right-hand sides (slip-rate histories) stepped together
    int far_mode = 0;         // 0: Eq. 42 as scatter into delay rings; 1: delayed-history gather
    long long uhist_len = 0;  // far_mode 1: source-value histories (doubles per right-hand side)
    int2 *rec_tasks = nullptr, *gat_tasks = nullptr;
    int n_rec = 0, n_gat = 0;
    double* uhist = nullptr;
    double dt = 0;
    HostPlan hp;
    fdph_stats st;
    // device memory
    std::vector<void*> allocs;
    int* perm = nullptr;
    SbDev* sbs = nullptr;
    void* fac = nullptr;
    int *ints = nullptr, *src_order = nullptr;
    int4 *runs = nullptr, *sc_tasks = nullptr;
    int* last_run = nullptr;
    int n_sct = 0;
    FarEnt* ents = nullptr;
    double* ent_phi = nullptr;
    long long n_ent = 0;
    FirGroup* fir = nullptr;
    void* fir_h = nullptr;
    int* fir_dhat = nullptr;
    int n_fir = 0;
    int *tr_sb = nullptr, *tr_l = nullptr, *g_ptr = nullptr;
    // receiver groups and leaves of a rupture block's own steps, and the steps of such a block (1: the
    // operator acts within kBlk steps elsewhere too)
    RecGroup* rec_groups = nullptr;
    RecLeaf* rec_leaves = nullptr;
    int n_groups = 0, rup_block = 1;
    int margin = 0;           // min(dm + delay) over the far blocks: steps before one of them acts
    NearDev* near = nullptr;
    NearTask* tasks = nullptr;
    int n_win = 0, n_aux = 0; // window and aux items (tensor cores: the window items first)
    void* tensor = nullptr;
    void* stat = nullptr;     // aux slices, storage type
    int *np_ptr = nullptr, *np_idx = nullptr;
    int* err = nullptr;
    double* rho = nullptr;
    // rupture state
    bool rupture = false;
    bool predicted = false;   // fdph_predict issued for step n, fdph_commit pending
    FrictionDev fr;
    double *ustate = nullptr, *vstate = nullptr, *trcoef = nullptr;
    // state
    double *Dring = nullptr, *Cring = nullptr, *C = nullptr, *Ccomp = nullptr;
    float* Dring32 = nullptr;   // FP32 copy of Dring (FP32 / FP16 plans)
    double *tfar = nullptr, *thist = nullptr, *blkD = nullptr, *blkC = nullptr;   // a block's scratch
    std::vector<std::pair<unsigned char*, size_t>> canaries;   // FDPH_CHECK builds: allocation ends
    double *ring = nullptr, *zring = nullptr, *partial = nullptr;
    void* dhat = nullptr;
    size_t state_bytes = 0;
    size_t device_bytes = 0;  // of all allocations
    // host staging for fdph_step_host
    double *dD = nullptr, *dT = nullptr;
    // per-kernel event timing
    bool prof = false;
    struct ProfEvent {
        int id, steps;
        cudaEvent_t b, e;
    };
    std::vector<ProfEvent> prof_ev;
    double prof_ms[FDPH_NUM_KERNELS] = {0};
    int64_t prof_n[FDPH_NUM_KERNELS] = {0};
    // graphs of one rupture block, or of one step of the delayed-history form, replayed with the step
    // index and the call's first step in n_dev[0..1]; kept per (kind, D, T) so that repeated calls on
    // the same buffers reuse them
    struct GraphEntry {
        int kind;
        const void* D;
        const void* T;
        cudaGraphExec_t ex;
    };
    std::vector<GraphEntry> graphs;
    int* n_dev = nullptr;
    // near-field schedule inputs (kept so that the work-item length can be changed later)
    std::vector<int32_t> near_W, near_kz;
    std::vector<char> near_tail;
    int chunk = 0;            // steps of exact kernel per near-field work item
    int aux_chunk = 1;        // aux slices per work item
    double kscale = 1.0;      // FP16 window coefficients are stored as K * kscale (a power of two)
    int sched_version = 0;    // bumped whenever the near-field items are rebuilt
    size_t partial_cap = 0;   // capacity of `partial`, in doubles
    RingMap* maps = nullptr;  // rings of the array being saved or restored
    // branches of a step that run concurrently with the near field: [0] FIR + scatter,
    // [1] transient convolution + Eq. 39 evaluation (fork after push, join before gather)
    cudaStream_t side[2] = {nullptr, nullptr};
    cudaEvent_t ev_fork = nullptr, ev_join[2] = {nullptr, nullptr};
    // fdph_run_host: device staging ring, copy streams and their events
    static const int kIoSlots = 3;   // blocks of rows in the staging ring
    double *io_D = nullptr, *io_T = nullptr;   // [kIoSlots][kBlk] rows
    cudaStream_t h2d = nullptr, d2h = nullptr;
    cudaEvent_t ev_in[kIoSlots] = {}, ev_out[kIoSlots] = {}, ev_free[kIoSlots] = {};
};

#ifdef FDPH_CHECK
// FDPH_CHECK builds: every device allocation of a plan ends in kCanaryBytes of a known pattern,
// compared with the pattern whenever the plan synchronises (check_canaries)
static const size_t kCanaryBytes = 256;
static const unsigned char kCanary = 0xA5;
#endif

template <class T>
static int dalloc(fdph_plan_t P, T** out, size_t count) {
    void* p = nullptr;
    const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
#ifdef FDPH_CHECK
    const size_t extra = kCanaryBytes;
#else
    const size_t extra = 0;
#endif
    cudaError_t e = cudaMalloc(&p, bytes + extra);
    if (e != cudaSuccess) {
        set_error(std::string("cudaMalloc(") + std::to_string(bytes) + "): " + cudaGetErrorString(e));
        return FDPH_E_OOM;
    }
    P->allocs.push_back(p);
    P->device_bytes += bytes + extra;
#ifdef FDPH_CHECK
    P->canaries.push_back({(unsigned char*)p + bytes, extra});
    if (cudaMemsetAsync((unsigned char*)p + bytes, kCanary, extra, P->stream) != cudaSuccess) return FDPH_E_CUDA;
#endif
    *out = (T*)p;
    return FDPH_OK;
}

#ifdef FDPH_CHECK
// FDPH_CHECK builds: FDPH_E_CHECK if a write ran past the end of a device allocation
static int check_canaries(fdph_plan_t P) {
    std::vector<unsigned char> h;
    for (const auto& c : P->canaries) {
        h.assign(c.second, 0);
        FDPH_CUDA(cudaMemcpyAsync(h.data(), c.first, c.second, cudaMemcpyDeviceToHost, P->stream));
        FDPH_CUDA(cudaStreamSynchronize(P->stream));
        for (unsigned char b : h)
            if (b != kCanary) {
                set_error("a device write ran past the end of a plan allocation (canary overwritten)");
                return FDPH_E_CHECK;
            }
    }
    return FDPH_OK;
}
#endif

template <class T>
static int upload(fdph_plan_t P, T** out, const std::vector<T>& v) {
    int rc = dalloc(P, out, v.size());
    if (rc) return rc;
    // ordered on the plan's stream (a pageable source is staged before the call returns)
    if (!v.empty())
        FDPH_CUDA(cudaMemcpyAsync(*out, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, P->stream));
    return FDPH_OK;
}

template <class T>
static StepArgs<T> make_args(fdph_plan_t P, const double* D, double* T_) {
    StepArgs<T> a;
    memset(&a, 0, sizeof(a));
    const HostPlan& hp = P->hp;
    a.n = P->n;
    a.nb = 1;
    a.hist = HIST_ALL;
    a.N = P->N;
    a.WD = P->WD;
    a.WC = P->WC;
    a.io_stride = (long long)P->N * P->nrhs;
    a.dt = P->dt;
    a.D_in = D;
    a.T_out = T_;
    a.perm = P->perm;
    a.Dring = P->Dring;
    a.Dring32 = P->Dring32;
    a.Cring = P->Cring;
    a.C = P->C;
    a.Ccomp = P->Ccomp;
    a.blkD = P->blkD;
    a.blkC = P->blkC;
    a.sbs = P->sbs;
    a.fac = (const T*)P->fac;
    a.ints = P->ints;
    a.runs = P->runs;
    a.src_order = P->src_order;
    a.sc_tasks = P->sc_tasks;
    a.last_run = P->last_run;
    a.n_sct = P->n_sct;
    a.ents = P->ents;
    a.ent_phi = P->ent_phi;
    a.g_ptr = P->g_ptr;
    a.n_ent = P->n_ent;
    a.tfar = P->tfar;
    a.fir = P->fir;
    a.fir_h = (const T*)P->fir_h;
    a.fir_dhat = P->fir_dhat;
    a.n_fir = P->n_fir;
    a.fir_taps = hp.max_taps;
    a.tr_sb = P->tr_sb;
    a.tr_l = P->tr_l;
    a.n_tr = (int)hp.tr_sb.size();
    a.ring = P->ring;
    a.zring = P->zring;
    a.dhat = (T*)P->dhat;
    a.len_ring = std::max<long long>(hp.ring_len, 1);
    a.len_zring = std::max<long long>(hp.zring_len, 1);
    a.len_dhat = std::max<long long>(hp.dhat_len, 1) * kBlk;
    a.len_ustate = std::max<long long>(hp.ustate_len, 1);
    a.len_vstate = std::max<long long>(hp.vstate_len, 1);
    a.tasks = P->tasks;
    a.n_items = P->n_win + P->n_aux;
    a.tensor = P->tensor;
    a.kinv = (float)(1.0 / P->kscale);
    a.stat = P->stat;
    a.len_tensor = hp.near_tensor_len;
    a.len_aux = hp.near_aux_len;
    a.partial = P->partial;
    a.cap_partial = (long long)P->partial_cap;
    a.np_ptr = P->np_ptr;
    a.np_idx = P->np_idx;
    a.err = P->err;
    a.soe = hp.soe;
    a.rho = P->rho;
    a.ustate = P->ustate;
    a.trcoef = P->trcoef;
    a.vstate = P->vstate;
    a.nrhs = P->nrhs;
    a.rs_D = (long long)P->WD * P->N;
    a.rs_C = (long long)P->WC * P->N;
    a.rs_partial = (long long)P->partial_cap * kBlk;
    a.uhist = P->uhist;
    a.len_uhist = std::max<long long>(P->uhist_len, 1);
    a.rec_tasks = P->rec_tasks;
    a.gat_tasks = P->gat_tasks;
    a.n_rec = P->n_rec;
    a.n_gat = P->n_gat;
    a.rec_groups = P->rec_groups;
    a.rec_leaves = P->rec_leaves;
    a.n_groups = P->n_groups;
    return a;
}

static inline int blocks(long long n, int t) { return (int)std::max<long long>(1, (n + t - 1) / t); }

// Event timing of one kernel of a launch sequence (fdph_set_profiling); counts as `steps` launches, so
// that time / launches is the kernel's time per step
struct ProfScope {
    fdph_plan_t P;
    int id, steps;
    cudaEvent_t b = nullptr, e = nullptr;
    ProfScope(fdph_plan_t P_, int id_, int steps_);
    ~ProfScope();
};

// The kernels hold one column per step of a launch in registers: instantiated for one step and for a
// whole block (a shorter block computes unused columns)
// (one step of several right-hand sides: all of them in one lane of the FIR and the scatter)
template <class T, int NR>
static void launch_fir_step(const StepArgs<T>& a, cudaStream_t s) {
    const size_t smem = (size_t)kFirWarps * NR * (a.fir_taps + 2) * sizeof(T);
    const bool staged = smem <= 48 * 1024;   // (no opt-in shared memory)
    fir_step_kernel<T, NR><<<blocks(a.n_fir, kFirWarps * kFirGroups), 32 * kFirWarps, staged ? smem : 0, s>>>(a, staged);
}

template <class T>
static void launch_fir(const StepArgs<T>& a, cudaStream_t s) {
    if (a.nb == 1) {
        switch (a.nrhs) {
            case 2: launch_fir_step<T, 2>(a, s); break;
            case 4: launch_fir_step<T, 4>(a, s); break;
            case 8: launch_fir_step<T, 8>(a, s); break;
            default: launch_fir_step<T, 1>(a, s);
        }
        return;
    }
    const dim3 g(blocks(a.n_fir, kFirWarps), a.nrhs);
    const size_t smem = (size_t)kFirWarps * (a.fir_taps + 2 * kBlk) * sizeof(T);
    const bool staged = smem <= 48 * 1024;
    fir_kernel<T, kBlk><<<g, 32 * kFirWarps, staged ? smem : 0, s>>>(a, staged);
}

// Eq. 42: scatter into the delay rings, or (far_mode 1, one step) record the source values and gather
// the completed slot from the histories
template <class T>
static void launch_eq42(const StepArgs<T>& a, cudaStream_t s) {
    if (a.n_rec) {
        record_kernel<T><<<dim3(blocks(a.n_rec, 128), a.nrhs), 128, 0, s>>>(a);
        if (a.n_gat) hgather_kernel<T><<<dim3(blocks((long long)a.n_gat * 32, 128), a.nrhs), 128, 0, s>>>(a);
    } else if (a.n_sct) {
        const int g = blocks((long long)a.n_sct * 32, 128);
        switch (a.nb == 1 ? a.nrhs : 0) {
            case 1: scatter_kernel<T, 1, true><<<g, 128, 0, s>>>(a); break;
            case 2: scatter_kernel<T, 2, true><<<g, 128, 0, s>>>(a); break;
            case 4: scatter_kernel<T, 4, true><<<g, 128, 0, s>>>(a); break;
            case 8: scatter_kernel<T, 8, true><<<g, 128, 0, s>>>(a); break;
            default: scatter_kernel<T, 1, false><<<dim3(g, a.nrhs), 128, 0, s>>>(a);
        }
    }
}

template <class T>
static void launch_trconv(const StepArgs<T>& a, cudaStream_t s) {
    const dim3 g(blocks(a.n_tr, kTrWarps), a.nrhs);
    if (a.nb == 1) trconv_kernel<T, 1><<<g, 32 * kTrWarps, 0, s>>>(a);
    else trconv_kernel<T, kBlk><<<g, 32 * kTrWarps, 0, s>>>(a);
}

template <class T>
static void launch_far(const StepArgs<T>& a, cudaStream_t s) {
    const dim3 g(blocks((long long)a.N * 32, 128), a.nrhs);
    if (a.nb == 1) far_kernel<T, 1><<<g, 128, 0, s>>>(a);
    else far_kernel<T, kBlk><<<g, 128, 0, s>>>(a);
}

template <class T>
static void launch_gather(const StepArgs<T>& a, cudaStream_t s) {
    gather_kernel<T><<<dim3(blocks((long long)a.N * 8, 256), a.nrhs, a.nb), 256, 0, s>>>(a);
}

template <class T, class H, int B>
static void launch_near_items(const StepArgs<T>& a, int chunk, cudaStream_t s) {
    const size_t wb = NearCfg<H, B>::warp_bytes(chunk);
    near_block_kernel<T, H, B><<<blocks((long long)a.n_items * a.nrhs, kNearWarps), 32 * kNearWarps, wb * kNearWarps, s>>>(
        a, (int)wb);
}

// the tensor-core window items
template <int NR>
static void launch_tc(const StepArgs<float>& a, int n_win, int chunk, cudaStream_t s) {
    if (a.nb == 1) tc_step_kernel<NR><<<blocks(n_win, kTcStepWarps), 32 * kTcStepWarps, 0, s>>>(a, n_win);
    else tc_block_kernel<NR><<<n_win, 32 * TcCfg<NR>::warps, TcCfg<NR>::smem(chunk), s>>>(a, chunk);
}

// The near field of a launch: the window items (FP16 plans), or all items (FP64 and FP32 plans).  FP16 windows of
// one right-hand side meet FP32 slip rates on the CUDA cores: on the tensor cores, as three FP16 parts under a
// common scale, slip rates below 2^-15 of the leaf's largest lost digits (planar N = 1601, 32 steps: 461 us
// there, 545 us here).
template <class T>
static void launch_near(fdph_plan_t P, const StepArgs<T>& a, cudaStream_t s) {
    if (!a.n_items) return;
    if constexpr (sizeof(T) == 8) {
        if (a.nb == 1) launch_near_items<T, double, 1>(a, P->chunk, s);
        else launch_near_items<T, double, kBlk>(a, P->chunk, s);
    } else if (P->precision == FDPH_FP16) {
        const bool all = a.nb == 1 && P->nrhs == 1;   // (see launch_near_aux)
        if (!P->n_win && !all) return;
        StepArgs<T> w = a;   // (a block of one right-hand side)
        w.n_items = P->n_win;
        switch (P->nrhs) {
            case 2: launch_tc<2>(a, P->n_win, P->chunk, s); break;
            case 4: launch_tc<4>(a, P->n_win, P->chunk, s); break;
            case 8: launch_tc<8>(a, P->n_win, P->chunk, s); break;
            default: all ? launch_near_items<T, __half, 1>(a, P->chunk, s) : launch_near_items<T, __half, kBlk>(w, P->chunk, s);
        }
    } else if (a.nb == 1) {
        launch_near_items<T, float, 1>(a, P->chunk, s);
    } else {
        launch_near_items<T, float, kBlk>(a, P->chunk, s);
    }
}

// The static and tail items of FP16 plans: a kernel of their own, far from filling the GPU, so it goes last
// on the far-field branch, beside the windows.  (A single step of one right-hand side takes them along with its
// windows: nothing there is as long as one more kernel on that branch; N = 400, leaves of 13, 43 -> 32 us.)
template <class T>
static void launch_near_aux(fdph_plan_t P, StepArgs<T> a, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (P->precision != FDPH_FP16 || !P->n_aux || (a.nb == 1 && P->nrhs == 1)) return;
        a.tasks += P->n_win;
        a.n_items = P->n_aux;
        if (a.nb == 1) launch_near_items<T, float, 1>(a, P->chunk, s);
        else launch_near_items<T, float, kBlk>(a, P->chunk, s);
    }
}

// The part of a block that only reads slip rates and rings: transient convolution and Eq. 39 beside the
// near field, then the gather
template <class T>
static void enqueue_far(const StepArgs<T>& a, cudaStream_t s) {
    if (a.n_tr) launch_trconv<T>(a, s);
    launch_far<T>(a, s);
}

// Steps a.n ... a.n + a.nb - 1 with given slip rates.  The near field and the far field touch
// disjoint data once push is done.  Within the far field, FIR + scatter write the slots from
// n + delay on and the transient convolution + Eq. 39 read those up to n + nb - 1 - dm: disjoint too when
// no far block acts within the block (nb <= margin = min(dm + delay), always true for one step by
// causality), and then a second branch; otherwise they follow.
template <class T>
static void enqueue_block(fdph_plan_t P, const StepArgs<T>& a, cudaStream_t s) {
    { ProfScope ps(P, 0, a.nb); push_kernel<T><<<dim3(blocks(a.N, 128), a.nrhs), 128, 0, s>>>(a); }
    if (!P->prof) {
        const bool apart = a.nb <= P->margin;
        cudaStream_t f0 = P->side[0], f1 = apart ? P->side[1] : P->side[0];
        cudaEventRecord(P->ev_fork, s);
        cudaStreamWaitEvent(f0, P->ev_fork, 0);
        if (apart) cudaStreamWaitEvent(f1, P->ev_fork, 0);
        launch_near<T>(P, a, s);
        if (a.n_fir) launch_fir<T>(a, f0);
        launch_eq42<T>(a, f0);
        enqueue_far<T>(a, f1);
        launch_near_aux<T>(P, a, f1);
        cudaEventRecord(P->ev_join[0], f0);
        cudaStreamWaitEvent(s, P->ev_join[0], 0);
        if (apart) {
            cudaEventRecord(P->ev_join[1], f1);
            cudaStreamWaitEvent(s, P->ev_join[1], 0);
        }
        launch_gather<T>(a, s);
        return;
    }
    // serial order (per-kernel timing)
    if (a.n_fir) { ProfScope ps(P, 1, a.nb); launch_fir<T>(a, s); }
    { ProfScope ps(P, 2, a.nb); launch_eq42<T>(a, s); }
    if (a.n_tr) { ProfScope ps(P, 3, a.nb); launch_trconv<T>(a, s); }
    { ProfScope ps(P, 4, a.nb); launch_near<T>(P, a, s); launch_near_aux<T>(P, a, s); }
    { ProfScope ps(P, 5, a.nb); launch_far<T>(a, s); launch_gather<T>(a, s); }
}

// The traction of a.nb steps from the slip rates that a.hist admits, into T_out or thist: transient
// convolution and Eq. 39 beside the near field, gather.  Advances the transient and exponential-tail
// states of the steps.
template <class T>
static void enqueue_history(fdph_plan_t P, const StepArgs<T>& a, cudaStream_t s) {
    if (!P->prof) {
        cudaEventRecord(P->ev_fork, s);
        cudaStreamWaitEvent(P->side[1], P->ev_fork, 0);
        launch_near<T>(P, a, s);
        enqueue_far<T>(a, P->side[1]);
        launch_near_aux<T>(P, a, P->side[1]);
        cudaEventRecord(P->ev_join[1], P->side[1]);
        cudaStreamWaitEvent(s, P->ev_join[1], 0);
        launch_gather<T>(a, s);
        return;
    }
    if (a.n_tr) { ProfScope ps(P, 3, a.nb); launch_trconv<T>(a, s); }
    { ProfScope ps(P, 4, a.nb); launch_near<T>(P, a, s); launch_near_aux<T>(P, a, s); }
    { ProfScope ps(P, 5, a.nb); launch_far<T>(a, s); launch_gather<T>(a, s); }
}

// Commit of step n: push D_n into the history, FIR, scatter.
template <class T>
static void enqueue_commit(fdph_plan_t P, const StepArgs<T>& a, cudaStream_t s) {
    { ProfScope ps(P, 0, 1); push_kernel<T><<<dim3(blocks(a.N, 128), a.nrhs), 128, 0, s>>>(a); }
    if (a.n_fir) { ProfScope ps(P, 1, 1); launch_fir<T>(a, s); }
    { ProfScope ps(P, 2, 1); launch_eq42<T>(a, s); }
}

// Rupture steps n ... n + nb - 1 of one aligned block (they do not cross a multiple of kBlk): what the
// slip rates before the block do to all of them, then step by step the block's own part, the friction
// law and the push, then FIR and scatter of the block.
template <class T, class H>
static void enqueue_rupture_h(fdph_plan_t P, StepArgs<T> a, double* D, cudaStream_t s) {
    double* T_out = a.T_out;
    const int recent = P->rup_block > 1;
    a.hist = recent ? HIST_BASE : HIST_STEP;
    a.thist = P->thist;
    enqueue_history<T>(P, a, s);
    a.T_out = T_out;
    for (int b = 0; b < a.nb; ++b) {
        ProfScope ps(P, 0, 1);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(a.n_groups);
        cfg.blockDim = dim3(kRupThreads);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = b > 0 && !P->prof ? 1 : 0;   // (a step's launch overlaps the step before)
        cudaLaunchKernelEx(&cfg, rup_step_kernel<T, H>, a, P->fr, D, b, recent);
    }
    if (a.n_fir) { ProfScope ps(P, 1, a.nb); launch_fir<T>(a, s); }
    { ProfScope ps(P, 2, a.nb); launch_eq42<T>(a, s); }
}

template <class T>
static void enqueue_rupture(fdph_plan_t P, const StepArgs<T>& a, double* D, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (P->precision == FDPH_FP16) {
            enqueue_rupture_h<T, __half>(P, a, D, s);
            return;
        }
    }
    enqueue_rupture_h<T, T>(P, a, D, s);
}

// kinds of cached graphs
enum { GRAPH_RUN = 0, GRAPH_RUPTURE = 1 };

// The cached graph of nb steps of `kind` on buffers (D, T), captured on first use; the step index and
// the first row's step are set on the device before the replays.
template <class T>
static int step_graph(fdph_plan_t P, int kind, int nb, const double* D, double* Tout, cudaGraphExec_t* ex) {
    if (!P->n_dev) {
        int rc = dalloc(P, &P->n_dev, 2);
        if (rc) return rc;
    }
    cudaStream_t s = P->stream;
    for (const auto& ge : P->graphs)
        if (ge.kind == kind && ge.D == (const void*)D && ge.T == (const void*)Tout) {
            *ex = ge.ex;
            return FDPH_OK;
        }
    StepArgs<T> a = make_args<T>(P, kind == GRAPH_RUPTURE ? nullptr : D, Tout);
    a.n_dev = P->n_dev;
    a.nb = nb;
    cudaGraph_t g = nullptr;
    FDPH_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    if (kind == GRAPH_RUPTURE) enqueue_rupture<T>(P, a, (double*)D, s);
    else enqueue_block<T>(P, a, s);
    advance_step_kernel<<<1, 1, 0, s>>>(P->n_dev, nb);
    cudaError_t e = cudaStreamEndCapture(s, &g);
    if (e != cudaSuccess) {
        set_error(std::string("graph capture: ") + cudaGetErrorString(e));
        return FDPH_E_CUDA;
    }
    e = cudaGraphInstantiate(ex, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        set_error(std::string("graph instantiate: ") + cudaGetErrorString(e));
        return FDPH_E_CUDA;
    }
    if (P->graphs.size() >= 8) {   // bounded cache: drop the oldest graph
        cudaStreamSynchronize(s);
        cudaGraphExecDestroy(P->graphs.front().ex);
        P->graphs.erase(P->graphs.begin());
    }
    P->graphs.push_back({kind, (const void*)D, (const void*)Tout, *ex});
    return FDPH_OK;
}

static void drop_graphs(fdph_plan_t P) {
    for (auto& ge : P->graphs) cudaGraphExecDestroy(ge.ex);
    P->graphs.clear();
}

// The longest run of steps that is cheaper step by step than as a block, whose kernels take (nearly) as long for two steps
// as for sixteen.  us, step / block of 2, 3, 5: FP64 N = 1500 193 / 698, 830, 1125, eight right-hand sides of N = 400
// 282 / 978, 1168, 1606; FP16 N = 6000, eight 516 / 2704, 2822, four 375 / 1525, 1576; FP32 N = 1500, eight 347 / 973, four
// 188 / 482; one FP16 with 16 tail terms, N = 1500, 81 / 248, 257; one FP32 without 77 / 163, N = 400 30 / 52.
static int stepwise(fdph_plan_t P) {
    if (P->precision == FDPH_FP64) return 4;
    if (P->precision == FDPH_FP16) return P->nrhs < 4 ? 2 : 3;
    return P->nrhs >= 4 || P->hp.soe > 0 ? 2 : 1;
}

// `steps` steps with given slip rates, in blocks.  A caller may pass D == T (every block reads its rows
// before it writes them) but rows that overlap otherwise are taken one step at a time, as is the
// delayed-history form, whose steps replay a graph.
template <class T>
static int run_steps(fdph_plan_t P, int steps, const double* D, double* Tout) {
    const size_t row = (size_t)P->N * P->nrhs;
    const bool alias = D != Tout && (const char*)D < (const char*)(Tout + steps * row) &&
                       (const char*)Tout < (const char*)(D + steps * row);
    int k = 0;
    if (P->n_rec && steps >= 8 && !P->prof) {
        cudaGraphExec_t ex = nullptr;
        int rc = step_graph<T>(P, GRAPH_RUN, 1, D, Tout, &ex);
        if (rc) return rc;
        place_step_kernel<<<1, 1, 0, P->stream>>>(P->n_dev, P->n, P->n);
        for (; k < steps; ++k) FDPH_CUDA(cudaGraphLaunch(ex, P->stream));
        P->n += steps;
        return FDPH_OK;
    }
    while (k < steps) {
        StepArgs<T> a = make_args<T>(P, D + k * row, Tout + k * row);
        a.nb = alias || P->n_rec || steps - k <= stepwise(P) ? 1 : std::min(kBlk, steps - k);
        enqueue_block<T>(P, a, P->stream);
        FDPH_CUDA(cudaGetLastError());
        P->n += a.nb;
        k += a.nb;
    }
    return FDPH_OK;
}

static int run_any(fdph_plan_t P, int steps, const double* D, double* Tout) {
    return P->precision != FDPH_FP64 ? run_steps<float>(P, steps, D, Tout) : run_steps<double>(P, steps, D, Tout);
}

// Host-buffer steps: the D rows of a block go host -> staging slot on the h2d stream, the block runs on
// the plan stream once that copy is done, and its T rows go back on the d2h stream; a slot is reused
// after its T rows have left it.
static int run_host(fdph_plan_t P, int steps, const double* D_host, double* T_host) {
    const int S = fdph_plan_s::kIoSlots;
    const size_t row = (size_t)P->N * P->nrhs;
    if (!P->io_D) {
        int rc;
        if ((rc = dalloc(P, &P->io_D, S * kBlk * row)) || (rc = dalloc(P, &P->io_T, S * kBlk * row))) return rc;
        FDPH_CUDA(cudaStreamCreateWithFlags(&P->h2d, cudaStreamNonBlocking));
        FDPH_CUDA(cudaStreamCreateWithFlags(&P->d2h, cudaStreamNonBlocking));
        for (int q = 0; q < S; ++q) {
            FDPH_CUDA(cudaEventCreateWithFlags(&P->ev_in[q], cudaEventDisableTiming));
            FDPH_CUDA(cudaEventCreateWithFlags(&P->ev_out[q], cudaEventDisableTiming));
            FDPH_CUDA(cudaEventCreateWithFlags(&P->ev_free[q], cudaEventDisableTiming));
        }
    }
    // the staging slots must not be reused before work still queued from an earlier call is done
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    FDPH_CUDA(cudaStreamSynchronize(P->d2h));
    cudaError_t e = cudaSuccess;
    int rc = FDPH_OK;
    for (int k = 0, i = 0; k < steps && e == cudaSuccess && !rc; ++i) {
        const int q = i % S, nb = std::min(kBlk, steps - k);
        double *dD = P->io_D + q * kBlk * row, *dT = P->io_T + q * kBlk * row;
        if (i >= S) e = cudaStreamWaitEvent(P->h2d, P->ev_free[q], 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(dD, D_host + k * row, nb * row * sizeof(double), cudaMemcpyHostToDevice, P->h2d);
        if (e == cudaSuccess) e = cudaEventRecord(P->ev_in[q], P->h2d);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(P->stream, P->ev_in[q], 0);
        if (e != cudaSuccess || (rc = run_any(P, nb, dD, dT))) break;
        e = cudaEventRecord(P->ev_out[q], P->stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(P->d2h, P->ev_out[q], 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(T_host + k * row, dT, nb * row * sizeof(double), cudaMemcpyDeviceToHost, P->d2h);
        if (e == cudaSuccess) e = cudaEventRecord(P->ev_free[q], P->d2h);
        k += nb;
    }
    // no copy from or to the caller's buffers stays in flight, after an error either
    for (cudaStream_t s : {P->h2d, P->stream, P->d2h}) {
        const cudaError_t w = cudaStreamSynchronize(s);
        if (e == cudaSuccess) e = w;
    }
    if (rc) return rc;
    if (e != cudaSuccess) {
        set_error(std::string("fdph_run_host: ") + cudaGetErrorString(e));
        return FDPH_E_CUDA;
    }
    return FDPH_OK;
}

// `steps` rupture steps: whole aligned blocks replay a captured graph, the rest is launched directly
template <class T>
static int rupture_steps(fdph_plan_t P, int steps, double* D, double* Tout) {
    const size_t row = (size_t)P->N;
    cudaGraphExec_t ex = nullptr;
    const int n0 = P->n, Bk = P->rup_block;
    bool placed = false;   // the device's step index stands at P->n
    for (int k = 0; k < steps;) {
        const int nb = std::min(steps - k, Bk - P->n % Bk);
        if (!P->prof && steps >= 8 && nb == Bk) {
            if (!ex) {
                int rc = step_graph<T>(P, GRAPH_RUPTURE, Bk, D, Tout, &ex);
                if (rc) return rc;
            }
            if (!placed) place_step_kernel<<<1, 1, 0, P->stream>>>(P->n_dev, P->n, n0);
            placed = true;
            FDPH_CUDA(cudaGraphLaunch(ex, P->stream));
        } else {
            StepArgs<T> a = make_args<T>(P, nullptr, Tout + k * row);
            a.nb = nb;
            enqueue_rupture<T>(P, a, D + k * row, P->stream);
            placed = false;
        }
        FDPH_CUDA(cudaGetLastError());
        P->n += nb;
        k += nb;
    }
    return FDPH_OK;
}

ProfScope::ProfScope(fdph_plan_t P_, int id_, int steps_) : P(P_), id(id_), steps(steps_) {
    if (!P->prof) return;
    cudaEventCreate(&b);
    cudaEventCreate(&e);
    cudaEventRecord(b, P->stream);
}

ProfScope::~ProfScope() {
    if (!P->prof || !b) return;
    cudaEventRecord(e, P->stream);
    P->prof_ev.push_back({id, steps, b, e});
}

static void prof_drain(fdph_plan_t P) {
    for (auto& q : P->prof_ev) {
        float ms = 0.f;
        cudaEventSynchronize(q.e);
        cudaEventElapsedTime(&ms, q.b, q.e);
        P->prof_ms[q.id] += ms;
        P->prof_n[q.id] += q.steps;
        cudaEventDestroy(q.b);
        cudaEventDestroy(q.e);
    }
    P->prof_ev.clear();
}

// after a stream synchronisation: report a device error word
static int check_device_error(fdph_plan_t P) {
    int e = 0;
    if (!P->err) return FDPH_OK;
    FDPH_CUDA(cudaMemcpyAsync(&e, P->err, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    if (e) {
        cudaMemsetAsync(P->err, 0, sizeof(int), P->stream);
        if (e == kErrIndex) {
            set_error("a device index check failed (bounded-index debug build); results of the step are invalid");
            return FDPH_E_CHECK;
        }
        set_error("a bounded device wait gave up; results of the step are invalid");
        return FDPH_E_TIMEOUT;
    }
#ifdef FDPH_CHECK
    return check_canaries(P);
#else
    return FDPH_OK;
#endif
}

template <class T>
static int launch_predict(fdph_plan_t P, double* T_pred) {
    StepArgs<T> a = make_args<T>(P, nullptr, T_pred);
    a.hist = HIST_STEP;
    enqueue_history<T>(P, a, P->stream);
    FDPH_CUDA(cudaGetLastError());
    return FDPH_OK;
}

template <class T>
static int launch_commit(fdph_plan_t P, const double* D_n) {
    enqueue_commit<T>(P, make_args<T>(P, D_n, nullptr), P->stream);
    FDPH_CUDA(cudaGetLastError());
    return FDPH_OK;
}

// The plan's near-field work items as the near kernels read them: window items first where they go to
// the tensor cores, else all together, largest first (an item is a warp's or a CTA's work: the last to
// start are the shortest).
template <class T, class H>
static int build_schedule(fdph_plan_t P) {
    using A = typename NearTypes<H>::Aux;
    HostPlan& hp = P->hp;
    const bool tc = std::is_same<H, __half>::value;
    const int ni = (int)hp.items.size();
    std::vector<NearTask> all(ni);
    std::vector<double> cost(ni);
    P->n_win = P->n_aux = 0;
    for (int q = 0; q < ni; ++q) {
        const NearItem& it = hp.items[q];
        const NearLeaf& L = hp.near[it.leaf];
        NearTask& t = all[q];
        memset(&t, 0, sizeof(t));
        t.off = it.kind ? (long long)L.stat + (long long)it.k0 * L.sla : (long long)L.tensor + (long long)it.k0 * L.sl;
        t.item = q;
        t.k0 = it.k0;
        t.k1 = it.k1;
        t.kind = it.kind;
        t.nr = L.nr;
        t.ns = L.ns;
        t.sl = it.kind ? L.sla : L.sl;
        t.s0 = L.s0;
        t.W = L.W;
        t.vstate = (int)L.vstate;
        // bytes, and for aux slices the FP64 work of their rows and sums
        cost[q] = (double)(it.k1 - it.k0) * (t.sl * (double)(it.kind ? sizeof(A) : sizeof(H)) + (it.kind ? 4096.0 : 0.0)) + 4096.0;
        (it.kind ? P->n_aux : P->n_win) += 1;
    }
    std::vector<int> order(ni);
    for (int q = 0; q < ni; ++q) order[q] = q;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        if (tc && all[x].kind != all[y].kind) return all[x].kind < all[y].kind;
        return cost[x] > cost[y];
    });
    std::vector<NearTask> tasks(ni);
    for (int q = 0; q < ni; ++q) tasks[q] = all[order[q]];
    // shared memory of the near kernels for items of this length
    if constexpr (std::is_same<H, __half>::value) {
        FDPH_CUDA(cudaFuncSetAttribute(near_block_kernel<T, H, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)NearCfg<H, 1>::warp_bytes(kChunk) * kNearWarps));
        FDPH_CUDA(cudaFuncSetAttribute(near_block_kernel<T, H, kBlk>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)NearCfg<H, kBlk>::warp_bytes(kChunk) * kNearWarps));
        FDPH_CUDA(cudaFuncSetAttribute(tc_block_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcCfg<2>::smem(kChunk)));
        FDPH_CUDA(cudaFuncSetAttribute(tc_block_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcCfg<4>::smem(kChunk)));
        FDPH_CUDA(cudaFuncSetAttribute(tc_block_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcCfg<8>::smem(kChunk)));
    }
    constexpr int longest = sizeof(H) == 8 ? kChunk : 2 * kChunk;   // (near_max_chunk)
    using I = typename std::conditional<sizeof(H) == 8, double, float>::type;
    FDPH_CUDA(cudaFuncSetAttribute(near_block_kernel<T, I, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)NearCfg<I, 1>::warp_bytes(longest) * kNearWarps));
    FDPH_CUDA(cudaFuncSetAttribute(near_block_kernel<T, I, kBlk>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)NearCfg<I, kBlk>::warp_bytes(longest) * kNearWarps));
    P->sched_version += 1;
    int rc;
    if ((rc = upload(P, &P->tasks, tasks)) || (rc = upload(P, &P->np_ptr, hp.np_ptr)) || (rc = upload(P, &P->np_idx, hp.np_idx)))
        return rc;
    return FDPH_OK;
}

// Near-field build in two phases around the host factorisation of the admissible blocks, which
// it does not need: build_near_begin (windows, exact tensors, tail projections launched on the
// device) and build_near_finish (tail fits on the host, upload, schedule).
struct NearBuild {
    std::vector<NearDev> tl;        // leaves with an exponential tail
    std::vector<long long> tp0;     // their first pair
    double* d_g = nullptr;          // projections on the device
    long long ntp = 0;
    bool tails = false;
};

// T: far-field / step type; H: near-field window storage type (aux slices: NearTypes<H>::Aux)
template <class T, class H>
static int build_near_begin(fdph_plan_t P, const PlanInputs& in, NearBuild& nb) {
    using A = typename NearTypes<H>::Aux;
    HostPlan& hp = P->hp;
    const int nl = (int)hp.near_r0.size();
    const bool verbose = getenv("FDPH_VERBOSE") != nullptr;
    const auto t_start = std::chrono::steady_clock::now();
    auto stamp = [&](const char* what) {   // stage times of the near-field build
        if (!verbose) return;
        fprintf(stderr, "[fdph_plan]   %-26s %8.3f s\n", what,
                std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count());
    };
    GeoDev g;
    double *px, *py, *nx, *ny, *ax, *ay, *tx, *ty, *ln;
    int rc;
    if ((rc = upload(P, &px, hp.px)) || (rc = upload(P, &py, hp.py)) || (rc = upload(P, &nx, hp.pnx)) ||
        (rc = upload(P, &ny, hp.pny)) || (rc = upload(P, &ax, hp.sax)) || (rc = upload(P, &ay, hp.say)) ||
        (rc = upload(P, &tx, hp.stx)) || (rc = upload(P, &ty, hp.sty)) || (rc = upload(P, &ln, hp.slen)))
        return rc;
    g.px = px; g.py = py; g.nx = nx; g.ny = ny; g.ax = ax; g.ay = ay; g.tx = tx; g.ty = ty; g.len = ln;
    std::vector<long long> pair0(nl + 1, 0);
    for (int l = 0; l < nl; ++l) pair0[l + 1] = pair0[l] + (long long)hp.near_nr[l] * hp.near_ns[l];
    const long long npairs = pair0[nl];
    std::vector<int32_t> W(nl, 0);
    std::vector<int> ms;
    int *d_ms = nullptr, *d_r = nullptr, *d_nr = nullptr, *d_s = nullptr, *d_ns = nullptr;
    long long* d_p0 = nullptr;
    if (nl > 0) {
        if ((rc = dalloc(P, &d_ms, npairs)) || (rc = upload(P, &d_r, hp.near_r0)) ||
            (rc = upload(P, &d_nr, hp.near_nr)) || (rc = upload(P, &d_s, hp.near_s0)) ||
            (rc = upload(P, &d_ns, hp.near_ns)))
            return rc;
        std::vector<long long> p0(pair0.begin(), pair0.end() - 1);
        if ((rc = upload(P, &d_p0, p0))) return rc;
        ms.assign(npairs, 0);
        if (in.soe == 0) {   // the paper's cut: exact kernel up to each pair's m_S (App. H)
            const double thr = in.eps_st * in.mu / (2.0 * in.cs);
            near_ms_kernel<<<blocks(npairs, 128), 128, 0, P->stream>>>(g, d_r, d_nr, d_s, d_ns, d_p0, npairs, nl, in.M, in.dt,
                                                          in.mu, in.cs, thr, d_ms);
            FDPH_CUDA(cudaGetLastError());
            FDPH_CUDA(cudaMemcpyAsync(ms.data(), d_ms, npairs * sizeof(int), cudaMemcpyDeviceToHost, P->stream));
            FDPH_CUDA(cudaStreamSynchronize(P->stream));
            for (int l = 0; l < nl; ++l)
                for (long long q = pair0[l]; q < pair0[l + 1]; ++q) W[l] = std::max(W[l], ms[q]);
        }
        stamp("near: windows");
    }
    // kz: leading window slices that vanish, K_ijk = 0 while the wave is on its way (c (k + 1) dt <=
    // the pair's distance; one slice less for rounding), unless a pair's static part starts earlier
    std::vector<int32_t> kz(nl, 0);
    const double cdt = in.cs * in.dt;
#pragma omp parallel for schedule(dynamic, 64) num_threads(in.threads)
    for (int l = 0; l < nl; ++l) {
        int first = in.M;
        for (int il = 0; il < hp.near_nr[l]; ++il) {
            const int pi = hp.near_r0[l] + il;
            for (int jl = 0; jl < hp.near_ns[l]; ++jl) {
                const int pj = hp.near_s0[l] + jl;
                const double dx = hp.px[pi] - hp.sax[pj], dy = hp.py[pi] - hp.say[pj];
                const double along = std::min(std::max(dx * hp.stx[pj] + dy * hp.sty[pj], 0.0), hp.slen[pj]);
                const double ex = dx - along * hp.stx[pj], ey = dy - along * hp.sty[pj];
                const double steps = sqrt(ex * ex + ey * ey) / cdt;
                first = std::min(first, steps < in.M ? (int)steps - 1 : in.M);
                if (in.soe == 0) first = std::min(first, ms[pair0[l] + (long long)il * hp.near_ns[l] + jl]);
            }
        }
        kz[l] = std::max(first, 0);
    }
    std::vector<char> has_tail(nl, 0);
    if (in.soe > 0) {
        // exponential tails: the window covers every pair's wave passage (both end-point fronts +
        // n_c steps), the exact kernel is kept for all pairs up to the leaf's window, and the
        // smooth remainder beyond it is fitted (no m_S cut is needed)
        for (int l = 0; l < nl; ++l) {
            for (int il = 0; il < hp.near_nr[l]; ++il) {
                const int pi = hp.near_r0[l] + il;
                for (int jl = 0; jl < hp.near_ns[l]; ++jl) {
                    const int pj = hp.near_s0[l] + jl;
                    double dx = hp.px[pi] - hp.sax[pj], dy = hp.py[pi] - hp.say[pj];
                    const double da = sqrt(dx * dx + dy * dy);
                    dx = hp.px[pi] - hp.sbx[pj];
                    dy = hp.py[pi] - hp.sby[pj];
                    const double db = sqrt(dx * dx + dy * dy);
                    const int pass = (int)ceil(std::max(da, db) / cdt) + hp.tree.nc;
                    W[l] = std::max(W[l], pass);
                }
            }
            if (in.M - W[l] < soe_min_len(W[l])) W[l] = in.M;
            else has_tail[l] = 1;
            for (long long q = pair0[l]; q < pair0[l + 1]; ++q) ms[q] = W[l];   // exact over the window
        }
        FDPH_CUDA(cudaMemcpyAsync(d_ms, ms.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, P->stream));
    }
    // work-item length: the longest chunk that still yields about four items per resident warp
    // (152 SMs x 16) or CTA (152 x 3), so small problems (the plain N = 256 march) fill the device too
    long long slices = 0;
    for (int l = 0; l < nl; ++l) {
        kz[l] = std::min(kz[l], W[l]);
        slices += std::max(W[l] - kz[l], 1);
    }
    // (an item is a CTA's work on the tensor cores: FP16 with several right-hand sides)
    const bool cta = P->precision == FDPH_FP16 && P->nrhs > 1;
    int chunk = std::min(near_max_chunk(P->nrhs, P->precision), kChunk / 2);
    while (chunk > 8 / std::min(P->nrhs, 2) && slices * P->nrhs / chunk < 4LL * 152 * (cta ? 3 : 16)) chunk /= 2;
    P->aux_chunk = near_aux_chunk(nl);
    finish_near_layout(hp, W, kz, has_tail, chunk, 16 / (int)sizeof(H), 16 / (int)sizeof(A), P->aux_chunk);
    P->near_W = W;
    P->near_kz = kz;
    P->near_tail = has_tail;
    P->chunk = chunk;
    std::vector<NearDev> nd(nl);
    for (int l = 0; l < nl; ++l) {
        const NearLeaf& L = hp.near[l];
        nd[l] = {L.r0, L.nr, L.s0, L.ns, L.W, L.sl, L.sla, 0, (long long)L.tensor, (long long)L.stat, (long long)L.tail,
                 (long long)L.vstate};
    }
    if ((rc = upload(P, &P->near, nd))) return rc;
    // FP16 windows: coefficients are stored times 2^e, e = 13 - ceil(log2(mu / (2 cs))), so that
    // the radiation-damping self term mu / (2 cs), the largest coefficient, sits near 2^13: far
    // from the FP16 overflow (65504) whatever the units, and small coefficients keep the normal
    // FP16 range; the products are scaled back by 2^-e
    P->kscale = std::is_same<H, __half>::value ? std::ldexp(1.0, 13 - (int)std::ceil(std::log2(in.mu / (2.0 * in.cs))))
                                                : 1.0;
    H* tens = nullptr;
    A* aux = nullptr;
    if ((rc = dalloc(P, &tens, hp.near_tensor_len)) || (rc = dalloc(P, &aux, hp.near_aux_len))) return rc;
    P->tensor = tens;
    P->stat = aux;
    if (hp.near_tensor_len) FDPH_CUDA(cudaMemsetAsync(tens, 0, hp.near_tensor_len * sizeof(H), P->stream));  // padding
    if (hp.near_aux_len) FDPH_CUDA(cudaMemsetAsync(aux, 0, hp.near_aux_len * sizeof(A), P->stream));
    for (int l = 0; l < nl; ++l) {
        const long long tot = (long long)nd[l].W * nd[l].ns * nd[l].nr;
        if (tot == 0 && nd[l].ns * nd[l].nr == 0) continue;
        // static tile is written by k == 0 entries; a leaf with W == 0 still needs it
        NearDev L = nd[l];
        if (L.W == 0) {
            // temporarily fill one k-slice into a scratch to get the static tile
            H* tmp = nullptr;
            if ((rc = dalloc(P, &tmp, (size_t)L.sl))) return rc;
            NearDev L1 = L;
            L1.W = 1;
            L1.tensor = 0;
            near_fill_kernel<H, A><<<blocks((long long)L.ns * L.nr, 128), 128, 0, P->stream>>>(g, L1, d_ms + pair0[l], in.dt,
                                                                            in.mu, in.cs, P->kscale, tmp, aux);
        } else {
            near_fill_kernel<H, A><<<std::min<long long>(blocks(tot, 256), 4096), 256, 0, P->stream>>>(
                g, L, d_ms + pair0[l], in.dt, in.mu, in.cs, P->kscale, tens, aux);
        }
        FDPH_CUDA(cudaGetLastError());
    }
    stamp("near: exact windows filled");
    if (in.soe > 0 && hp.near_tail_len > 0) {
        // all tail leaves in one launch (here), then one Cholesky solve per leaf on the host (finish)
        std::vector<NearDev>& tl = nb.tl;
        std::vector<int> tl_id;
        std::vector<long long>& tp0 = nb.tp0;
        tp0.assign(1, 0);
        for (int l = 0; l < nl; ++l)
            if (has_tail[l]) {
                tl.push_back(nd[l]);
                tl_id.push_back(l);
                tp0.push_back(tp0.back() + (long long)nd[l].nr * nd[l].ns);
            }
        const long long ntp = tp0.back();
        NearDev* d_tl = nullptr;
        long long* d_tp0 = nullptr;
        double* d_g = nullptr;
        std::vector<long long> tp0s(tp0.begin(), tp0.end() - 1);
        if ((rc = upload(P, &d_tl, tl)) || (rc = upload(P, &d_tp0, tp0s)) || (rc = dalloc(P, &d_g, (size_t)ntp * in.soe)))
            return rc;
        near_soe_proj_kernel<<<blocks(ntp, 128), 128, 0, P->stream>>>(g, d_tl, d_tp0, (int)tl.size(), ntp, in.M, in.dt, in.mu, in.cs,
                                                        in.soe, P->rho, d_g);
        FDPH_CUDA(cudaGetLastError());
        nb.d_g = d_g;
        nb.ntp = ntp;
        nb.tails = true;
    }
    stamp("near: tail projections launched");
    return FDPH_OK;
}

// near leaves that act within a rupture block
static bool rec_leaf(const NearLeaf& L) { return L.kz < kBlk || (L.W < kBlk && L.tail < 0); }

template <class T, class H>
static int build_near_finish(fdph_plan_t P, const PlanInputs& in, NearBuild& nb) {
    using A = typename NearTypes<H>::Aux;
    HostPlan& hp = P->hp;
    A* aux = (A*)P->stat;
    int rc;
    const bool verbose = getenv("FDPH_VERBOSE") != nullptr;
    const auto t_start = std::chrono::steady_clock::now();
    auto stamp = [&](const char* what) {
        if (!verbose) return;
        fprintf(stderr, "[fdph_plan]   %-26s %8.3f s\n", what,
                std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count());
    };
    if (nb.tails) {
        const std::vector<NearDev>& tl = nb.tl;
        const std::vector<long long>& tp0 = nb.tp0;
        const long long ntp = nb.ntp;
        double* d_g = nb.d_g;
        std::vector<double> gh((size_t)ntp * in.soe), ch((size_t)ntp * in.soe);
        FDPH_CUDA(cudaMemcpyAsync(gh.data(), d_g, gh.size() * sizeof(double), cudaMemcpyDeviceToHost, P->stream));
        FDPH_CUDA(cudaStreamSynchronize(P->stream));
        stamp("near: tail projections done");
        // tail slices q = 1..Q of each leaf's aux block, [q][ns][nr] with slice stride sl
        std::vector<size_t> toff(tl.size() + 1, 0);
        for (size_t t = 0; t < tl.size(); ++t) toff[t + 1] = toff[t] + (size_t)in.soe * tl[t].sla;
        std::vector<A> tail_h(toff.back(), (A)0);
        constexpr int v4 = 16 / (int)sizeof(A);
#pragma omp parallel for schedule(dynamic, 8) num_threads(in.threads)
        for (long t = 0; t < (long)tl.size(); ++t) {
            const NearDev& L = tl[t];
            const size_t b = (size_t)tp0[t] * in.soe;
            soe_solve(hp.rho, in.M - L.W, gh.data() + b, ch.data() + b, L.nr * L.ns);
            for (int il = 0; il < L.nr; ++il)
                for (int jl = 0; jl < L.ns; ++jl)
                    for (int q = 0; q < in.soe; ++q)
                        tail_h[toff[t] + (size_t)q * L.sla + ((size_t)(jl / v4) * L.nr + il) * v4 + jl % v4] =
                            (A)ch[b + ((size_t)il * L.ns + jl) * in.soe + q];
        }
        for (size_t t = 0; t < tl.size(); ++t)
            FDPH_CUDA(cudaMemcpyAsync(aux + tl[t].tail, tail_h.data() + toff[t], (toff[t + 1] - toff[t]) * sizeof(A),
                                      cudaMemcpyHostToDevice, P->stream));
    }
    stamp("near: tail fits");
    if ((rc = build_schedule<T, H>(P))) return rc;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    return FDPH_OK;
}

// Rupture blocks: the near leaves that a wave crosses within kBlk steps, grouped by their maximal
// receiver clusters (clusters of one tree are nested or disjoint, so those are disjoint; every element
// is in one, its own leaf has kz = 0), and whether blocks may be longer than one step: nothing else may
// act within the block, so the far blocks need min(dm + delay) >= kBlk, and tail terms, which start at the
// window's end, W >= kBlk (the static terms of shorter windows are among the block's own).
static int build_recent(fdph_plan_t P) {
    const HostPlan& hp = P->hp;
    const bool far_late = P->margin >= kBlk;
    bool near_late = true;
    std::vector<int> use;
    for (int l = 0; l < (int)hp.near.size(); ++l) {
        near_late = near_late && (hp.near[l].W >= kBlk || hp.near[l].tail < 0);
        if (rec_leaf(hp.near[l])) use.push_back(l);
    }
    P->rup_block = far_late && near_late && P->far_mode == 0 ? kBlk : 1;
    std::vector<int> owner(hp.n, -1);      // first element of the largest receiver range over each element
    std::vector<int> size(hp.n, 1);
    for (int p = 0; p < hp.n; ++p) owner[p] = p;
    for (int l : use) {
        const NearLeaf& L = hp.near[l];
        for (int p = L.r0; p < L.r0 + L.nr; ++p)
            if (L.nr > size[p]) {
                size[p] = L.nr;
                owner[p] = L.r0;
            }
    }
    std::vector<RecGroup> groups;
    std::vector<int> group_of(hp.n, 0);
    for (int p = 0; p < hp.n; p += size[p]) {
        for (int q = p; q < p + size[p]; ++q) group_of[q] = (int)groups.size();
        groups.push_back({p, size[p], 0, 0});
    }
    std::vector<RecLeaf> leaves;
    std::vector<std::vector<int>> per(groups.size());
    for (int l : use) per[group_of[hp.near[l].r0]].push_back(l);
    for (size_t g = 0; g < groups.size(); ++g) {
        groups[g].leaf0 = (int)leaves.size();
        groups[g].nleaf = (int)per[g].size();
        for (int l : per[g]) {
            const NearLeaf& L = hp.near[l];
            const long long stat = L.W < kBlk && L.tail < 0 ? (long long)L.stat : -1;
            leaves.push_back({(long long)L.tensor, stat, L.sl, L.r0, L.nr, L.s0, L.ns, L.kz, L.W, 0});
        }
    }
    P->n_groups = (int)groups.size();
    int rc;
    if ((rc = upload(P, &P->rec_groups, groups)) || (rc = upload(P, &P->rec_leaves, leaves))) return rc;
    return FDPH_OK;
}

static void fill_stats(fdph_plan_t P) {
    HostPlan& hp = P->hp;
    fdph_stats& s = P->st;
    const double ps = P->precision != FDPH_FP64 ? 4.0 : 8.0;   // far factors and near aux slices
    const double pw = P->precision == FDPH_FP16 ? 2.0 : ps;    // near window coefficients
    s.n = hp.n;
    s.M = hp.M;
    s.n_admissible = hp.n_adm;
    s.n_near = hp.n_near;
    s.n_subblocks = (int)hp.sbs.size();
    s.max_rank = hp.max_rank;
    s.mean_rank = hp.mean_rank;
    s.n_exact = hp.n_exact[0] + hp.n_exact[1] + hp.n_exact[2];
    s.n_aca = hp.n_aca;
    s.mean_rank_f = hp.ent_w[SB_F] > 0 ? hp.rank_w[SB_F] / hp.ent_w[SB_F] : 0.0;
    s.mean_rank_s = hp.ent_w[SB_S] > 0 ? hp.rank_w[SB_S] / hp.ent_w[SB_S] : 0.0;
    s.mean_rank_tr = hp.ent_w[SB_TR] > 0 ? hp.rank_w[SB_TR] / hp.ent_w[SB_TR] : 0.0;
    s.extra_steps = hp.tree.nc;
    s.max_window = hp.max_W;
    s.near_entries = hp.near_tensor_len;
    s.far_entries = hp.far_entries;
    // algorithmic bytes of one steady-state step
    double near_b = 0, far_b = 0, flops = 0;
    // slip-rate window rows are read from the FP32 copy of the ring unless the plan is FP64;
    // every right-hand side reads its own rows and keeps its own tail states
    const double prow = P->precision != FDPH_FP64 ? 4.0 : 8.0;
    const double R = P->nrhs;
    for (const NearLeaf& L : hp.near) {
        const double W = L.W - L.kz;                                           // (the first kz slices vanish)
        near_b += W * L.ns * L.nr * pw + (double)L.ns * L.nr * ps;             // tensor + static tile
        near_b += R * (W * L.ns * prow + L.ns * 8.0);                          // window rows + C row
        flops += 2.0 * R * (W + 1) * L.ns * L.nr;
        if (L.tail >= 0) {                                                     // tail coefficients + states
            near_b += (double)hp.soe * L.ns * L.nr * ps + R * hp.soe * L.ns * 16.0;
            flops += 2.0 * R * hp.soe * L.ns * (L.nr + 1.0);
        }
    }
    for (const SubBlock& sb : hp.sbs) {
        const double r = sb.rank;
        far_b += (sb.nr + sb.ns) * 4.0;                                        // delays
        if (sb.ident == 1) {          // F = I: one ring read per receiver
            far_b += sb.nr * 8.0 + sb.ns * r * ps + sb.nruns * r * 16.0;
            flops += 2.0 * sb.ns * r;
        } else if (sb.ident == 2) {   // G = I: one ring store per source
            far_b += sb.nr * r * (ps + 8.0) + sb.ns * 8.0;
            flops += 2.0 * sb.nr * r;
        } else {
            far_b += (sb.nr + sb.ns) * r * ps;                                 // f, g
            far_b += sb.nr * r * 8.0 + sb.nruns * r * 16.0;                    // ring reads / RMW
            flops += 2.0 * (sb.nr + sb.ns) * r;
        }
        if (sb.kind == SB_F) {
            far_b += (double)sb.taps * sb.ns * ps + sb.ns * 8.0;   // h, Dhat (the D history below)
            flops += 2.0 * sb.taps * sb.ns;
        }
        if (sb.kind == SB_TR) {
            if (sb.qn)   // two ring reads, a running-sum update and a value per quantized range
                far_b += r * (sb.qn * (16.0 + 16.0 + ps) + 8.0) + r * sb.soe * 24.0;
            else
                far_b += r * (sb.taps * 8.0 + sb.taps * ps + 8.0) + r * sb.soe * 24.0;
            flops += 2.0 * r * ((sb.qn ? 2.0 * sb.qn : sb.taps) + 2.0 * sb.soe);
        }
    }
    for (int32_t t : hp.sfir_tmax) far_b += t * 8.0;                         // each source's D history, once
    const double push_b = hp.n * (8.0 + 8.0 + 32.0 + 8.0 + 4.0);           // D in, ring, C/comp, Cring, perm
    const double out_b = hp.n * (8.0 + 4.0) + (double)hp.np_idx.size() * 12.0;
    s.bytes_per_step = near_b + far_b + push_b + out_b;
    s.near_bytes_per_step = near_b;
    s.flops_per_step = flops;
    s.state_bytes = (long long)P->state_bytes;
    s.arena_bytes = (long long)(P->device_bytes - P->state_bytes);
}

// Near-field work items of `chunk` kernel steps (1..kChunk): new items, partial slots and
// schedule; the stored coefficients do not move.  Cached step graphs refer to the old
// schedule and are dropped.
template <class T, class H>
static int set_chunk(fdph_plan_t P, int chunk) {
    using A = typename NearTypes<H>::Aux;
    HostPlan& hp = P->hp;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    drop_graphs(P);
    const int64_t tens0 = hp.near_tensor_len, aux0 = hp.near_aux_len, vst0 = hp.vstate_len;
    finish_near_layout(hp, P->near_W, P->near_kz, P->near_tail, chunk, 16 / (int)sizeof(H), 16 / (int)sizeof(A), P->aux_chunk);
    if (hp.near_tensor_len != tens0 || hp.near_aux_len != aux0 || hp.vstate_len != vst0) {
        // the stored coefficients and states must keep their places (only the items change)
        set_error("set_chunk: near-field layout changed; the plan is unusable");
        return FDPH_E_STATE;
    }
    const size_t need = hp.items.size() * 32;
    if (need > P->partial_cap) {
        int rc = dalloc(P, &P->partial, need * P->nrhs * kBlk);
        if (rc) return rc;
        P->partial_cap = need;
    }
    P->chunk = chunk;
    int rc = build_schedule<T, H>(P);
    if (rc) return rc;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    return FDPH_OK;
}

static int set_chunk_any(fdph_plan_t P, int chunk) {
    return P->precision == FDPH_FP16   ? set_chunk<float, __half>(P, chunk)
           : P->precision == FDPH_FP32 ? set_chunk<float, float>(P, chunk)
                                       : set_chunk<double, double>(P, chunk);
}

// a step split by fdph_predict must be completed by fdph_commit before anything else steps or
// copies the state
static int pending_commit(fdph_plan_t P) {
    if (!P->predicted) return FDPH_OK;
    set_error("step predicted by fdph_predict awaits fdph_commit");
    return FDPH_E_STATE;
}

// ------------------------------------------------------------------------------------------
// Batches of plans

// A set of plans (same device, same precision) stepped together: each plan's blocks run on its own
// stream, side by side on the GPU.  (One launch per kernel over the work of all plans was measured
// slower: with a block of steps per launch the launches no longer count.)  A call starts after the work
// queued on the streams of all its plans, and they all wait for its end (batch_join), so that a caller
// may prepare or read the buffers of every plan on the stream of any.
struct fdph_batch_s {
    int device = 0, precision = 0;
    std::vector<fdph_plan_t> plans;
    std::vector<int> version;            // each plan's near-field schedule at creation
    cudaStream_t hub = nullptr;          // where the plans' streams meet
    cudaEvent_t ev_plan = nullptr, ev_hub = nullptr;
};

// What is queued on any of the plans' streams precedes what is queued on any of them from now on
static int batch_join(fdph_batch_t B) {
    if (B->plans.size() < 2) return FDPH_OK;
    for (fdph_plan_t P : B->plans) {   // (a wait holds the event as it was recorded last: one event does)
        FDPH_CUDA(cudaEventRecord(B->ev_plan, P->stream));
        FDPH_CUDA(cudaStreamWaitEvent(B->hub, B->ev_plan, 0));
    }
    FDPH_CUDA(cudaEventRecord(B->ev_hub, B->hub));
    for (fdph_plan_t P : B->plans) FDPH_CUDA(cudaStreamWaitEvent(P->stream, B->ev_hub, 0));
    return FDPH_OK;
}

// batch calls: every plan still has the schedule the batch was built on and no pending predict
static int batch_check(fdph_batch_t B, int steps) {
    for (size_t p = 0; p < B->plans.size(); ++p) {
        fdph_plan_t P = B->plans[p];
        if (P->predicted) return pending_commit(P);
        if (P->sched_version != B->version[p]) {
            set_error("a plan of the batch has rebuilt its near-field items (fdph_autotune): create the batch again");
            return FDPH_E_STATE;
        }
        if (P->prof) {
            set_error("batch run: profiling is on for a plan of the batch");
            return FDPH_E_STATE;
        }
        if (P->n + steps > P->M) {
            set_error("batch run would pass step M of a plan");
            return FDPH_E_STATE;
        }
    }
    return FDPH_OK;
}

// ------------------------------------------------------------------------------------------
// C ABI

extern "C" {

void fdph_default_params(fdph_params* p) {
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->eta = 0.5;
    p->lmin = 0.0;
    p->eps_st = 1e-6;
    p->leaf_size = 32;
    p->extra_steps = -1;
    p->precision = FDPH_FP64;
    p->device = 0;
    p->cuda_stream = nullptr;
    p->nrhs = 1;
}

const char* fdph_strerror(int s) {
    switch (s) {
        case FDPH_OK: return "ok";
        case FDPH_E_ARG: return "invalid argument";
        case FDPH_E_OOM: return "out of memory";
        case FDPH_E_CAUSALITY: return "discretised causality violated (increase l_min/eta or reduce dt)";
        case FDPH_E_CUDA: return "CUDA error";
        case FDPH_E_TIMEOUT: return "device wait timed out";
        case FDPH_E_NAN: return "non-finite value";
        case FDPH_E_STATE: return "invalid plan state";
        case FDPH_E_CHECK: return "device index check failed (bounded-index debug build)";
        default: return "unknown status";
    }
}

const char* fdph_last_error(void) { return g_last_error.c_str(); }

static int check_inputs(const fdph_geometry* g, const fdph_material* m, double dt, const fdph_params* p) {
    if (!g || !m || !g->xy || g->n <= 0 || !(dt > 0.0) || !(m->mu > 0.0) || !(m->cs > 0.0)) {
        set_error("geometry, material and dt must be given, n > 0, dt, mu, cs > 0");
        return FDPH_E_ARG;
    }
    if (p && (p->leaf_size < 1 || p->leaf_size > 32 || p->eta < 0.0 || p->eps_st < 0.0 || p->host_threads < 0 ||
              (p->eta_scheme != 0 && p->eta_scheme != 1) || (p->eta_scheme == 1 && !(p->lmin > 0.0)) ||
              (p->nrhs != 0 && p->nrhs != 1 && p->nrhs != 2 && p->nrhs != 4 && p->nrhs != kMaxRhs) ||
              (p->far_mode != 0 && p->far_mode != 1) || (p->amp_window != 0 && p->amp_window != 1) ||
              !(p->eps_q >= 0.0 && p->eps_q < 1.0) ||
              (p->precision != FDPH_FP64 && p->precision != FDPH_FP32 && p->precision != FDPH_FP16) ||
              (p->soe_terms != 0 && (p->soe_terms < 4 || p->soe_terms > kMaxSoe)))) {
        set_error("params: leaf_size in [1, 32], eta >= 0, eps_st >= 0, host_threads >= 0, eta_scheme 0 or 1 (1 needs "
                  "lmin > 0), nrhs 1, 2, 4 or 8 (0: 1), far_mode 0 or 1, amp_window 0 or 1, eps_q in [0, 1), precision "
                  "FP64, FP32 or "
                  "FP16, "
                  "soe_terms 0 or in [4, 16]");
        return FDPH_E_ARG;
    }
    for (int k = 0; k < 4 * g->n; ++k)
        if (!std::isfinite(g->xy[k])) {
            set_error("geometry holds a non-finite coordinate");
            return FDPH_E_NAN;
        }
    for (int e = 0; e < g->n; ++e) {
        const double dx = g->xy[4 * e + 2] - g->xy[4 * e], dy = g->xy[4 * e + 3] - g->xy[4 * e + 1];
        if (dx * dx + dy * dy == 0.0) {
            set_error("element " + std::to_string(e) + " has zero length");
            return FDPH_E_ARG;
        }
    }
    return FDPH_OK;
}

static PlanInputs make_inputs(const fdph_material* m, double dt, int M, double eps, const fdph_params& p) {
    PlanInputs in;
    in.mu = m->mu;
    in.cs = m->cs;
    in.dt = dt;
    in.M = M;
    in.eps = eps;
    in.eta = p.eta;
    in.lmin = p.lmin;
    in.eps_st = p.eps_st;
    in.leaf = p.leaf_size;
    in.extra_steps = p.extra_steps;
    in.soe = p.soe_terms;
    in.interp = p.art_interp ? 1 : 0;
    in.threads = p.host_threads > 0 ? p.host_threads : omp_get_max_threads();
    in.eta_scheme = p.eta_scheme;
    in.amp_window = p.amp_window;
    in.eps_q = p.eps_q;
    in.aca_min = p.aca_min > 0 ? (long long)p.aca_min : LLONG_MAX;
    return in;
}

int fdph_low_rank(const double* A, int32_t m, int32_t n, double eps, double* F, double* G, int32_t* rank,
                  int32_t* exact) {
    if (!A || !F || !G || !rank || !exact || m < 1 || n < 1) return FDPH_E_ARG;
    for (long long q = 0; q < (long long)m * n; ++q)
        if (!std::isfinite(A[q])) {
            set_error("fdph_low_rank: non-finite entry");
            return FDPH_E_NAN;
        }
    LowRank lr;
    low_rank(A, m, n, eps, lr);
    *rank = lr.rank;
    *exact = lr.exact ? 1 : 0;
    std::copy(lr.F.begin(), lr.F.end(), F);
    std::copy(lr.G.begin(), lr.G.end(), G);
    return FDPH_OK;
}

int fdph_low_rank_aca(const double* A, int32_t m, int32_t n, double eps, double* F, double* G, int32_t* rank,
                      int32_t* converged, int64_t* evaluated) {
    if (!A || !F || !G || !rank || !converged || !evaluated || m < 1 || n < 1 || !(eps > 0.0)) {
        set_error("fdph_low_rank_aca: null pointer, m or n < 1 or eps <= 0");
        return FDPH_E_ARG;
    }
    for (long long q = 0; q < (long long)m * n; ++q)
        if (!std::isfinite(A[q])) {
            set_error("fdph_low_rank_aca: non-finite entry");
            return FDPH_E_NAN;
        }
    long long count = 0;
    auto row = [&](int i, double* out) {
        std::copy(A + (size_t)i * n, A + (size_t)(i + 1) * n, out);
        count += n;
    };
    auto col = [&](int j, double* out) {
        for (int i = 0; i < m; ++i) out[i] = A[(size_t)i * n + j];
        count += m;
    };
    LowRank lr;
    const bool ok = low_rank_aca(row, col, m, n, eps, lr);
    *converged = ok ? 1 : 0;
    *rank = ok ? lr.rank : 0;
    *evaluated = count;
    if (ok) {
        std::copy(lr.F.begin(), lr.F.end(), F);
        std::copy(lr.G.begin(), lr.G.end(), G);
    }
    return FDPH_OK;
}

int fdph_kernel_tail(const double* p, const double* seg, double t1, double dt, double mu, double cs, double* out) {
    if (!p || !seg || !out || !(dt > 0.0) || !(t1 >= 0.0) || !(mu > 0.0) || !(cs > 0.0) || !(seg[4] > 0.0)) {
        set_error("fdph_kernel_tail: null pointer, dt, mu, cs or the length <= 0, or t1 < 0");
        return FDPH_E_ARG;
    }
    const Seg s{seg[0], seg[1], seg[2], seg[3], seg[4]};
    const Stress2 v = stress_tail(p[0], p[1], s, t1, t1 + dt, mu, cs);
    out[0] = v.x;
    out[1] = v.y;
    out[2] = stress_tail_bound(p[0], p[1], s, t1, dt, mu, cs);
    return FDPH_OK;
}

int fdph_quantize(const double* K, int32_t n, double eps_q, int32_t* b, double* khat, int32_t* q) {
    if (!K || !b || !khat || !q || n < 1 || !(eps_q > 0.0)) {
        set_error("fdph_quantize: null pointer, n < 1 or eps_q <= 0");
        return FDPH_E_ARG;
    }
    for (int m = 0; m < n; ++m)
        if (!std::isfinite(K[m])) {
            set_error("fdph_quantize: non-finite value");
            return FDPH_E_NAN;
        }
    std::vector<int32_t> bb;
    std::vector<double> kh;
    quantize_partitions(K, n, eps_q, bb, kh);
    std::copy(bb.begin(), bb.end(), b);
    std::copy(kh.begin(), kh.end(), khat);
    *q = (int32_t)kh.size();
    return FDPH_OK;
}

int fdph_tree_export(const fdph_geometry* geometry, const fdph_material* material, double dt,
                     const fdph_params* params, int32_t* buf, int64_t cap, int64_t* len) {
    int rc = check_inputs(geometry, material, dt, params);
    if (rc) return rc;
    if (!len) return FDPH_E_ARG;
    fdph_params p;
    fdph_default_params(&p);
    if (params) p = *params;
    PlanInputs in = make_inputs(material, dt, 1, 0.0, p);
    Elements el = make_elements(geometry->n, geometry->xy);
    Tree tr;
    build_tree(el, in, tr);
    std::vector<int32_t> out;
    out.push_back(el.n);
    out.insert(out.end(), tr.perm.begin(), tr.perm.end());
    out.push_back((int32_t)tr.leaves.size());
    for (const Leaf& lf : tr.leaves) {
        const ClusterNode& tn = tr.nodes[lf.tau];
        const ClusterNode& sn = tr.nodes[lf.sig];
        out.push_back(lf.kind);
        out.push_back(tn.lo);
        out.push_back(tn.hi - tn.lo);
        out.push_back(sn.lo);
        out.push_back(sn.hi - sn.lo);
        if (lf.kind == 1) {
            ArtInts a = art_integers(el, tr, lf, in);
            if (a.causal < 1) {
                set_error("discretised causality violated");
                return FDPH_E_CAUSALITY;
            }
            out.insert(out.end(), a.dm.begin(), a.dm.end());
            out.insert(out.end(), a.mbar.begin(), a.mbar.end());
            out.insert(out.end(), a.Dm.begin(), a.Dm.end());
        }
    }
    *len = (int64_t)out.size();
    if (buf) {
        if (cap < (int64_t)out.size()) {
            set_error("buffer too small");
            return FDPH_E_ARG;
        }
        memcpy(buf, out.data(), out.size() * sizeof(int32_t));
    }
    return FDPH_OK;
}

int fdph_plan(const fdph_geometry* geometry, const fdph_material* material, double dt, int32_t M, double eps,
              const fdph_params* params, fdph_plan_t* out) {
    if (!out) return FDPH_E_ARG;
    *out = nullptr;
    int rc = check_inputs(geometry, material, dt, params);
    if (rc) return rc;
    if (M <= 0) {
        set_error("M must be positive");
        return FDPH_E_ARG;
    }
    const auto t0 = std::chrono::steady_clock::now();
    fdph_params p;
    fdph_default_params(&p);
    if (params) p = *params;
    fdph_plan_s* P = new (std::nothrow) fdph_plan_s();
    if (!P) return FDPH_E_OOM;
    P->device = p.device;
    P->precision = p.precision;
    P->nrhs = std::max(p.nrhs, 1);
    P->far_mode = p.far_mode;
    P->N = geometry->n;
    P->M = M;
    P->dt = dt;
    auto fail = [&](int code) {
        fdph_destroy(P);
        return code;
    };
    // host trees and the discretised causality of every admissible leaf first: a plan that
    // violates it is refused before any device resource is taken
    PlanInputs in = make_inputs(material, dt, M, eps, p);
    Elements el = make_elements(geometry->n, geometry->xy);
    HostPlan& hp = P->hp;
    build_host_tree(el, in, hp);
    if (check_causality(el, in, hp.tree)) return fail(FDPH_E_CAUSALITY);
    if (cudaSetDevice(p.device) != cudaSuccess) {
        set_error("cudaSetDevice failed");
        return fail(FDPH_E_CUDA);
    }
    if (p.cuda_stream) {
        P->stream = (cudaStream_t)p.cuda_stream;
    } else {
        if (cudaStreamCreateWithFlags(&P->stream, cudaStreamNonBlocking) != cudaSuccess) {
            set_error("cudaStreamCreate failed");
            return fail(FDPH_E_CUDA);
        }
        P->own_stream = true;
    }
    for (int k = 0; k < 2; ++k)
        if (cudaStreamCreateWithFlags(&P->side[k], cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&P->ev_join[k], cudaEventDisableTiming) != cudaSuccess) {
            set_error("cudaStreamCreate / cudaEventCreate failed");
            return fail(FDPH_E_CUDA);
        }
    if (cudaEventCreateWithFlags(&P->ev_fork, cudaEventDisableTiming) != cudaSuccess) {
        set_error("cudaEventCreate failed");
        return fail(FDPH_E_CUDA);
    }
    const bool verbose = getenv("FDPH_VERBOSE") != nullptr;
    auto stamp = [&](const char* what) {
        if (verbose)
            fprintf(stderr, "[fdph_plan] %-28s %8.3f s\n", what,
                    std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count());
    };
    stamp("cluster and block trees");
    // near field on the device (exact windows, tail projections) while the host factorises the
    // admissible blocks
    NearBuild nb;
    if (hp.soe > 0 && (rc = upload(P, &P->rho, hp.rho))) return fail(rc);
    rc = P->precision == FDPH_FP16   ? build_near_begin<float, __half>(P, in, nb)
         : P->precision == FDPH_FP32 ? build_near_begin<float, float>(P, in, nb)
                                     : build_near_begin<double, double>(P, in, nb);
    if (rc) return fail(rc);
    rc = build_host_far(el, in, hp);
    if (verbose) fprintf(stderr, "[fdph_plan] host threads %d\n", in.threads);
    stamp("host plan (admissible blocks)");
    if (rc == -3) return fail(FDPH_E_CAUSALITY);
    if (rc) return fail(FDPH_E_ARG);
    // the factors on the device leave out the Domain-F waveforms, which the FIR keeps in its own order:
    // ranges [first, first + length) of hp.fac, and what lies before each
    std::vector<std::pair<long long, long long>> cut;
    for (const SubBlock& b : hp.sbs)
        if (b.kind == SB_F) cut.push_back({(long long)b.h, (long long)b.taps * b.ns});
    std::sort(cut.begin(), cut.end());
    cut.erase(std::unique(cut.begin(), cut.end()), cut.end());
    std::vector<long long> cut_before(1, 0);
    for (const auto& c : cut) cut_before.push_back(cut_before.back() + c.second);
    auto place = [&](long long x) {   // of an offset in hp.fac
        const size_t k = std::upper_bound(cut.begin(), cut.end(), std::make_pair(x, LLONG_MAX)) - cut.begin();
        return x - cut_before[k] + (k && x < cut[k - 1].first + cut[k - 1].second ? cut[k - 1].second - (x - cut[k - 1].first) : 0);
    };
    std::vector<double> fac;
    fac.reserve(hp.fac.size() - (size_t)cut_before.back());
    {
        size_t at = 0;
        for (const auto& c : cut) {
            fac.insert(fac.end(), hp.fac.begin() + at, hp.fac.begin() + c.first);
            at = (size_t)(c.first + c.second);
        }
        fac.insert(fac.end(), hp.fac.begin() + at, hp.fac.end());
    }
    // ---- upload the far-field operator
    std::vector<SbDev> sd(hp.sbs.size());
    for (size_t q = 0; q < sd.size(); ++q) {
        const SubBlock& b = hp.sbs[q];
        const int LH = b.maxdelay - b.mindelay + 1;
        sd[q] = {b.kind, b.rank, b.r0, b.nr, b.s0, b.ns, b.L, b.LZ, b.taps, b.maxdelay, b.mindm, b.run0,
                 b.soe, b.ident, LH, place(b.f), place(b.g), b.kind == SB_F ? 0 : place(b.h), (long long)b.ring, (long long)b.zring,
                 (long long)b.dhat, (long long)b.delay, (long long)b.dm, (long long)b.ustate, (long long)b.trc,
                 (long long)b.phi, 0, b.mindelay, b.qn, (long long)b.qb};
    }
    // delayed-history form of Eq. 42 (far_mode 1): per block a history [LH][ns] of the source
    // values, recorded every step, and one gather task per (block, rank index)
    std::vector<int2> rec, gat;
    if (P->far_mode == 1)
        for (size_t q = 0; q < sd.size(); ++q) {
            sd[q].uhist = P->uhist_len;
            P->uhist_len += (long long)sd[q].LH * sd[q].ns;
            for (int j = 0; j < sd[q].ns; ++j) rec.push_back(make_int2((int)q, j));
            for (int l = 0; l < sd[q].rank; ++l) gat.push_back(make_int2((int)q, l));
        }
    P->n_rec = (int)rec.size();
    P->n_gat = (int)gat.size();
    if ((rc = upload(P, &P->rec_tasks, rec)) || (rc = upload(P, &P->gat_tasks, gat))) return fail(rc);
    // scatter warp tasks: 2^lg lanes per ring slot, 2^lg the rank rounded up to a power of two (at most
    // 32; one for identity factors), over the slots that a block of kBlk steps can reach
    std::vector<int4> sct, runs(hp.run_delay.size());
    for (size_t q = 0; q < runs.size(); ++q)
        runs[q] = make_int4(hp.run_delay[q], hp.run_len[q], hp.run_start[q], hp.src_order[hp.run_start[q]]);
    std::vector<int> last_run;   // per ring slot: the last run with delay <= the slot's offset
    P->margin = INT32_MAX;
    for (size_t q = 0; q < hp.sbs.size(); ++q) {
        const SubBlock& b = hp.sbs[q];
        P->margin = std::min(P->margin, b.mindm + b.mindelay);
        if (P->far_mode == 1) continue;
        int lg = 0;
        while ((1 << lg) < std::min(b.rank, 32)) ++lg;
        if (b.ident == 2) lg = 0;
        const int S = 32 >> lg, d1 = b.maxdelay + kBlk - 1;
        for (int d = b.mindelay; d <= d1; d += S) sct.push_back(make_int4((int)q, d, (int)last_run.size() + d - b.mindelay, lg));
        int last = b.run0;
        for (int d = b.mindelay; d <= d1; ++d) {
            while (last + 1 < b.run0 + b.nruns && hp.run_delay[last + 1] <= d) ++last;
            last_run.push_back(last);
        }
    }
    P->n_sct = (int)sct.size();
    // Eq. 39 entries, receiver-major
    std::vector<FarEnt> ents(hp.g_sb.size());
    std::vector<double> ephi(hp.interp ? hp.g_sb.size() : 0);
    for (size_t e = 0; e < ents.size(); ++e) {
        const SubBlock& b = hp.sbs[hp.g_sb[e]];
        const int il = hp.g_il[e];
        const bool tr = b.kind == SB_TR;
        ents[e] = {tr ? (long long)b.zring : (long long)b.ring, b.ident == 1 ? il : place(b.f) + (long long)il * b.rank,
                   tr ? b.LZ : b.L, hp.ints[b.dm + il], b.rank, (tr ? 1 : 0) | (b.ident == 1 ? 2 : 0)};
        if (hp.interp) ephi[e] = hp.phis[b.phi + il];
    }
    // (the lanes of a warp take entries of equal rank as far as possible)
    for (int p = 0; p < hp.n; ++p) {
        const int e0 = hp.g_ptr[p], e1 = hp.g_ptr[p + 1];
        std::vector<int> ord(e1 - e0);
        for (int e = e0; e < e1; ++e) ord[e - e0] = e;
        std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return ents[x].rank < ents[y].rank; });
        std::vector<FarEnt> es(e1 - e0);
        std::vector<double> ps(e1 - e0);
        for (int k = 0; k < e1 - e0; ++k) {
            es[k] = ents[ord[k]];
            if (hp.interp) ps[k] = ephi[ord[k]];
        }
        std::copy(es.begin(), es.end(), ents.begin() + e0);
        if (hp.interp) std::copy(ps.begin(), ps.end(), ephi.begin() + e0);
    }
    P->n_ent = (long long)ents.size();
    // FIR: the tasks of a source element in groups of 32, waveforms interleaved over a group's lanes
    std::vector<FirGroup> fir;
    std::vector<int> fdh;
    long long fh_len = 0;
    for (int p = 0; p < hp.n; ++p)
        for (int e = hp.sfir_ptr[p]; e < hp.sfir_ptr[p + 1]; e += 32) {
            FirGroup g;
            memset(&g, 0, sizeof(g));
            g.h = fh_len;
            g.src = p;
            g.first = (int)fdh.size();
            g.count = std::min(32, hp.sfir_ptr[p + 1] - e);
            for (int c = 0; c < g.count; ++c) {
                const int t = hp.sfir_q[e + c];
                const SubBlock& b = hp.sbs[hp.fir_sb[t]];
                g.taps = std::max(g.taps, b.taps);
                fdh.push_back((int)b.dhat + hp.fir_j[t]);
            }
            fh_len += (long long)g.taps * 32;
            fir.push_back(g);
        }
    P->n_fir = (int)fir.size();
    std::vector<double> fh((size_t)fh_len, 0.0);
#pragma omp parallel for schedule(static) num_threads(in.threads)
    for (long w = 0; w < (long)fir.size(); ++w) {
        const FirGroup& g = fir[w];
        const int e0 = hp.sfir_ptr[g.src] + (g.first - hp.sfir_ptr[g.src]);   // (groups keep the CSR order)
        for (int c = 0; c < g.count; ++c) {
            const int t = hp.sfir_q[e0 + c];
            const SubBlock& b = hp.sbs[hp.fir_sb[t]];
            for (int m = 0; m < b.taps; ++m) fh[(size_t)g.h + (size_t)m * 32 + c] = hp.fac[b.h + (size_t)hp.fir_j[t] * b.taps + m];
        }
    }
    if ((rc = upload(P, &P->sc_tasks, sct)) || (rc = upload(P, &P->runs, runs)) || (rc = upload(P, &P->last_run, last_run)) || (rc = upload(P, &P->ents, ents)) ||
        (rc = upload(P, &P->fir, fir)) || (rc = upload(P, &P->fir_dhat, fdh)))
        return fail(rc);
    if (hp.interp && (rc = upload(P, &P->ent_phi, ephi))) return fail(rc);
    if ((rc = upload(P, &P->perm, hp.perm)) || (rc = upload(P, &P->sbs, sd)) || (rc = upload(P, &P->ints, hp.ints)) ||
        (rc = upload(P, &P->src_order, hp.src_order)) || (rc = upload(P, &P->tr_sb, hp.tr_sb)) ||
        (rc = upload(P, &P->tr_l, hp.tr_l)) || (rc = upload(P, &P->g_ptr, hp.g_ptr)))
        return fail(rc);
    if (P->precision != FDPH_FP64) {
        std::vector<float> f(fac.begin(), fac.end());
        float* d = nullptr;
        if ((rc = upload(P, &d, f))) return fail(rc);
        P->fac = d;
        std::vector<float> h(fh.begin(), fh.end());
        float* dh = nullptr;
        if ((rc = upload(P, &dh, h))) return fail(rc);
        P->fir_h = dh;
    } else {
        double* d = nullptr;
        if ((rc = upload(P, &d, fac))) return fail(rc);
        P->fac = d;
        double* dh = nullptr;
        if ((rc = upload(P, &dh, fh))) return fail(rc);
        P->fir_h = dh;
    }
    if (hp.soe > 0 && (rc = upload(P, &P->trcoef, hp.trcoef))) return fail(rc);
    stamp("far-field upload");
    // ---- near field (device-evaluated kernel windows)
    rc = P->precision == FDPH_FP16   ? build_near_finish<float, __half>(P, in, nb)
         : P->precision == FDPH_FP32 ? build_near_finish<float, float>(P, in, nb)
                                     : build_near_finish<double, double>(P, in, nb);
    if (rc) return fail(rc);
    stamp("near field (windows, tails)");

    if ((rc = dalloc(P, &P->err, 1))) return fail(rc);
    FDPH_CUDA(cudaMemsetAsync(P->err, 0, sizeof(int), P->stream));
    // ---- state
    // (room for a whole block of steps beyond what one step reads)
    P->WD = std::max(std::max(hp.max_W + (hp.soe > 0 ? 1 : 0), hp.max_taps), 1) + kBlk - 1;
    P->WC = hp.max_W + 1 + kBlk - 1;
    if ((rc = build_recent(P))) return fail(rc);
    size_t sb = 0;
    auto st = [&](double** p, size_t cnt) {   // one copy per right-hand side
        const size_t c = std::max<size_t>(cnt, 1) * P->nrhs;
        sb += c * 8;
        return dalloc(P, p, c);
    };
    if ((rc = st(&P->Dring, (size_t)P->WD * P->N)) || (rc = st(&P->Cring, (size_t)P->WC * P->N)) ||
        (rc = st(&P->C, P->N)) || (rc = st(&P->Ccomp, P->N)) || (rc = st(&P->ring, hp.ring_len)) ||
        (rc = st(&P->zring, hp.zring_len)) || (rc = st(&P->ustate, hp.ustate_len)) ||
        (rc = st(&P->vstate, hp.vstate_len)) || (rc = st(&P->uhist, (size_t)P->uhist_len)))
        return fail(rc);
    // scratch of a block of steps: every use writes what it reads
    auto scratch = [&](double** p, size_t cnt) {
        const size_t c = std::max<size_t>(cnt, 1) * kBlk * P->nrhs;
        sb += c * 8;
        return dalloc(P, p, c);
    };
    if ((rc = scratch(&P->partial, hp.items.size() * 32)) || (rc = scratch(&P->tfar, P->N)) ||
        (rc = scratch(&P->blkD, P->N)) || (rc = scratch(&P->blkC, P->N)) || (rc = dalloc(P, &P->thist, (size_t)kBlk * P->N)))
        return fail(rc);
    {
        const size_t esz = P->precision != FDPH_FP64 ? 4 : 8;
        const size_t c = std::max<size_t>((size_t)hp.dhat_len, 1) * kBlk * P->nrhs * esz;
        unsigned char* d = nullptr;
        if ((rc = dalloc(P, &d, c))) return fail(rc);
        P->dhat = d;
        sb += c;
    }
    if (P->precision != FDPH_FP64) {   // FP32 copy of the slip-rate ring for the near-field rows
        const size_t c = (size_t)P->WD * P->N * P->nrhs;
        if ((rc = dalloc(P, &P->Dring32, c))) return fail(rc);
        sb += c * 4;
    }
    P->state_bytes = sb;
    P->partial_cap = std::max<size_t>(hp.items.size() * 32, 1);
    if ((rc = fdph_reset(P))) return fail(rc);
    fill_stats(P);
    P->st.plan_seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    *out = P;
    return FDPH_OK;
}

int fdph_reset(fdph_plan_t P) {
    if (!P) return FDPH_E_ARG;
    P->predicted = false;
    cudaSetDevice(P->device);
    double* bufs[] = {P->Dring, P->Cring, P->C, P->Ccomp, P->ring, P->zring, P->ustate, P->vstate, P->uhist};
    size_t cnt[] = {(size_t)P->WD * P->N, (size_t)P->WC * P->N, (size_t)P->N, (size_t)P->N, (size_t)P->hp.ring_len,
                    (size_t)P->hp.zring_len, (size_t)P->hp.ustate_len, (size_t)P->hp.vstate_len, (size_t)P->uhist_len};
    for (int q = 0; q < 9; ++q)   // every right-hand side: [nrhs][max(count, 1)]
        if (bufs[q])
            FDPH_CUDA(cudaMemsetAsync(bufs[q], 0, std::max<size_t>(cnt[q], 1) * P->nrhs * sizeof(double), P->stream));
    if (P->Dring32)
        FDPH_CUDA(cudaMemsetAsync(P->Dring32, 0, (size_t)P->WD * P->N * P->nrhs * sizeof(float), P->stream));
    if (P->rupture) FDPH_CUDA(cudaMemsetAsync(P->fr.slip, 0, P->N * sizeof(double), P->stream));
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    P->n = 0;
    return FDPH_OK;
}

int fdph_step(fdph_plan_t P, const double* D_n, double* T_n) {
    if (!P || !D_n || !T_n) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    if (P->n >= P->M) {
        set_error("the plan has already taken M steps");
        return FDPH_E_STATE;
    }
    return run_any(P, 1, D_n, T_n);
}

int fdph_run(fdph_plan_t P, int32_t steps, const double* D, double* T) {
    if (!P || !D || !T || steps < 0) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    if (P->n + steps > P->M) {
        set_error("run would pass step M");
        return FDPH_E_STATE;
    }
    return run_any(P, steps, D, T);
}

int fdph_run_host(fdph_plan_t P, int32_t steps, const double* D_host, double* T_host) {
    if (!P || !D_host || !T_host || steps < 0) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    if (P->n + steps > P->M) {
        set_error("run would pass step M");
        return FDPH_E_STATE;
    }
    if (steps == 0) return FDPH_OK;
    int rc;
    rc = run_host(P, steps, D_host, T_host);
    if (rc) return rc;
    return check_device_error(P);
}

int fdph_step_host(fdph_plan_t P, const double* D_n_host, double* T_n_host) {
    if (!P || !D_n_host || !T_n_host) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    const size_t row = (size_t)P->N * P->nrhs;
    if (!P->dD) {
        int rc;
        if ((rc = dalloc(P, &P->dD, row)) || (rc = dalloc(P, &P->dT, row))) return rc;
    }
    FDPH_CUDA(cudaMemcpyAsync(P->dD, D_n_host, row * sizeof(double), cudaMemcpyHostToDevice, P->stream));
    int rc = fdph_step(P, P->dD, P->dT);
    if (rc) return rc;
    FDPH_CUDA(cudaMemcpyAsync(T_n_host, P->dT, row * sizeof(double), cudaMemcpyDeviceToHost, P->stream));
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    return check_device_error(P);
}

int fdph_selftest_wait_timeout(int32_t device, int64_t polls) {
    if (polls < 1 || polls > (1LL << 24)) {
        set_error("fdph_selftest_wait_timeout: polls in [1, 2^24]");
        return FDPH_E_ARG;
    }
    FDPH_CUDA(cudaSetDevice(device));
    int* err = nullptr;
    FDPH_CUDA(cudaMalloc(&err, sizeof(int)));
    int h = 0;
    cudaError_t e = cudaMemset(err, 0, sizeof(int));
    if (e == cudaSuccess) {
        wait_selftest_kernel<<<1, 32>>>(polls, err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(&h, err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(err);
    if (e != cudaSuccess) {
        set_error(std::string("fdph_selftest_wait_timeout: ") + cudaGetErrorString(e));
        return FDPH_E_CUDA;
    }
    if (h) {
        set_error("bounded mbarrier wait gave up after " + std::to_string(polls) + " polls (self-test)");
        return FDPH_E_TIMEOUT;
    }
    return FDPH_OK;
}

int fdph_autotune(fdph_plan_t P, int32_t steps, int32_t* chunk_out) {
    if (!P || steps < 1 || steps > 1024) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    if (P->prof) {
        set_error("fdph_autotune: profiling is on");
        return FDPH_E_STATE;
    }
    if (P->hp.items.empty()) {
        if (chunk_out) *chunk_out = P->chunk;
        return FDPH_OK;
    }
    const int M = P->M;
    if (steps + 2 > M) {
        set_error("fdph_autotune: the plan has fewer than steps + 2 steps");
        return FDPH_E_ARG;
    }
    // the state is saved and restored around the trials
    size_t len = 0;
    int rc = fdph_save_state(P, nullptr, &len);
    if (rc) return rc;
    std::vector<char> saved(len);
    if ((rc = fdph_save_state(P, saved.data(), &len))) return rc;
    double *Dz = nullptr, *Tz = nullptr;
    const size_t rows = (size_t)(steps + 2) * P->N * P->nrhs;   // steps of nrhs rows of N
    if ((rc = dalloc(P, &Dz, rows)) || (rc = dalloc(P, &Tz, rows))) return rc;
    FDPH_CUDA(cudaMemsetAsync(Dz, 0, rows * sizeof(double), P->stream));
    // trials at a steady-state step index (every window full); the values stepped are irrelevant
    const int n0 = std::max(0, std::min(P->hp.max_W, M - steps - 2));
    cudaEvent_t e0, e1;
    FDPH_CUDA(cudaEventCreate(&e0));
    FDPH_CUDA(cudaEventCreate(&e1));
    const int cmax = near_max_chunk(P->nrhs, P->precision);
    const int cands[3] = {cmax, cmax / 2, cmax / 4};
    int best = P->chunk;
    float best_ms = 1e30f;
    for (int c : cands) {
        if ((rc = set_chunk_any(P, c))) break;
        P->n = n0;
        if ((rc = run_any(P, 2, Dz, Tz))) break;   // warm-up
        cudaEventRecord(e0, P->stream);
        if ((rc = run_any(P, steps, Dz, Tz))) break;
        cudaEventRecord(e1, P->stream);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best_ms) {
            best_ms = ms;
            best = c;
        }
    }
    if (!rc) rc = set_chunk_any(P, best);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    int rc2 = fdph_load_state(P, saved.data(), saved.size());
    if (rc) return rc;
    if (rc2) return rc2;
    if ((rc = check_device_error(P))) return rc;
    if (chunk_out) *chunk_out = best;
    return FDPH_OK;
}

int fdph_plan_stream(fdph_plan_t P, void** stream) {
    if (!P || !stream) return FDPH_E_ARG;
    *stream = (void*)P->stream;
    return FDPH_OK;
}

int fdph_current_step(fdph_plan_t P, int32_t* n) {
    if (!P || !n) return FDPH_E_ARG;
    *n = P->n;
    return FDPH_OK;
}

int fdph_synchronize(fdph_plan_t P) {
    if (!P) return FDPH_E_ARG;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    return check_device_error(P);
}

int fdph_get_stats(fdph_plan_t P, fdph_stats* s) {
    if (!P || !s) return FDPH_E_ARG;
    *s = P->st;
    return FDPH_OK;
}

// The arrays of a state saved at step n (n < 0: their sizes only)
struct StateArray {
    double* p;
    size_t count;                 // doubles of one right-hand side as saved
    size_t stored;                // doubles of one right-hand side in device memory
    std::vector<RingMap> rings;
};

static std::vector<StateArray> state_arrays(fdph_plan_t P, int n) {
    const HostPlan& hp = P->hp;
    std::vector<StateArray> v;
    auto ring1 = [&](double* p, int rows_dev) {
        const int rows = rows_dev - kRingRoom;
        v.push_back({p, (size_t)rows * P->N, (size_t)rows_dev * P->N, {{0, 0, rows, rows_dev, P->N, n - 1}}});
    };
    auto plain = [&](double* p, size_t c) { v.push_back({p, c, std::max<size_t>(c, 1), {}}); };
    ring1(P->Dring, P->WD);
    ring1(P->Cring, P->WC);
    plain(P->C, P->N);
    plain(P->Ccomp, P->N);
    StateArray r{P->ring, 0, (size_t)std::max<int64_t>(hp.ring_len, 1), {}}, z{P->zring, 0, (size_t)std::max<int64_t>(hp.zring_len, 1), {}};
    for (const SubBlock& b : hp.sbs) {
        if (!b.rank) continue;
        if (n >= 0) r.rings.push_back({(long long)r.count, (long long)b.ring, b.L - kRingRoom, b.L, b.rank, n - 1 + b.maxdelay});
        r.count += (size_t)(b.L - kRingRoom) * b.rank;
        if (b.kind != SB_TR) continue;
        if (n >= 0) z.rings.push_back({(long long)z.count, (long long)b.zring, b.LZ - kRingRoom, b.LZ, b.rank, n - 1 - b.mindm});
        z.count += (size_t)(b.LZ - kRingRoom) * b.rank;
    }
    v.push_back(std::move(r));
    v.push_back(std::move(z));
    plain(P->ustate, (size_t)hp.ustate_len);
    plain(P->vstate, (size_t)hp.vstate_len);
    plain(P->uhist, (size_t)P->uhist_len);
    return v;
}

// An array's saved form [nrhs][count] to or from host memory.  Rings are re-arranged on the device, staged
// in the partial sums (scratch of a block of steps, of which none is under way).
static int copy_state_array(fdph_plan_t P, const StateArray& a, char* host, bool save) {
    cudaStream_t s = P->stream;
    if (!a.count) return FDPH_OK;
    if (!save) FDPH_CUDA(cudaMemsetAsync(a.p, 0, a.stored * P->nrhs * sizeof(double), s));
    if (!a.rings.empty()) {
        if (!P->maps) {   // (the far rings are the most)
            int rc = dalloc(P, &P->maps, std::max<size_t>(P->hp.sbs.size(), 1));
            if (rc) return rc;
        }
        FDPH_CUDA(cudaMemcpyAsync(P->maps, a.rings.data(), a.rings.size() * sizeof(RingMap), cudaMemcpyHostToDevice, s));
    }
    const long long cap = (long long)P->partial_cap * kBlk * P->nrhs;
    for (int q = 0; q < P->nrhs; ++q) {
        char* h = host + q * a.count * sizeof(double);
        double* d = a.p + q * a.stored;
        if (a.rings.empty()) {
            FDPH_CUDA(cudaMemcpyAsync(save ? (void*)h : (void*)d, save ? (void*)d : (void*)h, a.count * sizeof(double),
                                      save ? cudaMemcpyDeviceToHost : cudaMemcpyHostToDevice, s));
            continue;
        }
        for (long long x0 = 0; x0 < (long long)a.count; x0 += cap) {
            const long long x1 = std::min<long long>(a.count, x0 + cap);
            const size_t bytes = (size_t)(x1 - x0) * sizeof(double);
            if (!save) FDPH_CUDA(cudaMemcpyAsync(P->partial, h + x0 * sizeof(double), bytes, cudaMemcpyHostToDevice, s));
            copy_rings_kernel<<<(int)std::min<long long>(blocks(x1 - x0, 256), 152 * 8), 256, 0, s>>>(
                P->maps, (int)a.rings.size(), x0, x1, d, P->partial, save);
            FDPH_CUDA(cudaGetLastError());
            if (save) FDPH_CUDA(cudaMemcpyAsync(h + x0 * sizeof(double), P->partial, bytes, cudaMemcpyDeviceToHost, s));
        }
    }
    return FDPH_OK;
}

int fdph_save_state(fdph_plan_t P, void* buf, size_t* len) {
    if (!P || !len) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    const std::vector<StateArray> arrays = state_arrays(P, buf ? P->n : -1);
    size_t need = sizeof(int32_t) * 2;
    for (const StateArray& a : arrays) need += a.count * P->nrhs * sizeof(double);
    if (P->rupture) need += (size_t)P->N * sizeof(double);   // the friction law's accumulated slip
    if (!buf) {
        *len = need;
        return FDPH_OK;
    }
    if (*len < need) return FDPH_E_ARG;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    char* o = (char*)buf;
    int32_t hdr[2] = {P->n, P->N};
    memcpy(o, hdr, sizeof(hdr));
    o += sizeof(hdr);
    for (const StateArray& a : arrays) {   // [nrhs][count] (a zero count stays empty)
        int rc = copy_state_array(P, a, o, true);
        if (rc) {
            cudaStreamSynchronize(P->stream);   // (no copy into the caller's buffer stays in flight)
            return rc;
        }
        o += a.count * P->nrhs * sizeof(double);
    }
    if (P->rupture) FDPH_CUDA(cudaMemcpyAsync(o, P->fr.slip, P->N * sizeof(double), cudaMemcpyDeviceToHost, P->stream));
    FDPH_CUDA(cudaStreamSynchronize(P->stream));   // the caller's buffer is complete on return
    *len = need;
    return FDPH_OK;
}

int fdph_load_state(fdph_plan_t P, const void* buf, size_t len) {
    if (!P || !buf) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    size_t need = 0;
    int rc = fdph_save_state(P, nullptr, &need);
    if (rc) return rc;
    if (len != need) {
        set_error("state buffer size does not match this plan");
        return FDPH_E_ARG;
    }
    const char* o = (const char*)buf;
    int32_t hdr[2];
    memcpy(hdr, o, sizeof(hdr));
    if (hdr[1] != P->N || hdr[0] < 0 || hdr[0] > P->M) {
        set_error("state buffer belongs to another plan");
        return FDPH_E_ARG;
    }
    o += sizeof(hdr);
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    const std::vector<StateArray> arrays = state_arrays(P, hdr[0]);   // (read by copies in flight)
    for (const StateArray& a : arrays) {
        if ((rc = copy_state_array(P, a, const_cast<char*>(o), false))) {
            cudaStreamSynchronize(P->stream);
            return rc;
        }
        o += a.count * P->nrhs * sizeof(double);
    }
    if (P->rupture)
        FDPH_CUDA(cudaMemcpyAsync(P->fr.slip, o, P->N * sizeof(double), cudaMemcpyHostToDevice, P->stream));
    if (P->Dring32) {
        const long long c = (long long)P->WD * P->N * P->nrhs;
        ring_to_float_kernel<<<blocks(c, 256), 256, 0, P->stream>>>(P->Dring, P->Dring32, c);
        FDPH_CUDA(cudaGetLastError());
    }
    FDPH_CUDA(cudaStreamSynchronize(P->stream));   // the caller may reuse the buffer on return
    P->n = hdr[0];
    return FDPH_OK;
}

// K_{ii,0} in geometry order: jump of the ramp response of each element at its own midpoint over
// [0, dt] (Eq. 4 with m = 0).  FDPH_E_STATE when the instantaneous term is not local
// (cs dt > half the shortest element: K_{ij,0} != 0 for neighbours).
static int self_coefficients(fdph_plan_t P, std::vector<double>& k0) {
    const HostPlan& hp = P->hp;
    double minlen = 1e300;
    for (int p = 0; p < P->N; ++p) minlen = std::min(minlen, hp.slen[p]);
    if (hp.cs * P->dt > 0.5 * minlen * (1.0 + 1e-12)) {
        set_error("cs dt exceeds half the shortest element; the instantaneous term is not local");
        return FDPH_E_STATE;
    }
    k0.assign(P->N, 0.0);
    for (int p = 0; p < P->N; ++p) {
        Seg sg;
        sg.ax = hp.sax[p];
        sg.ay = hp.say[p];
        sg.tx = hp.stx[p];
        sg.ty = hp.sty[p];
        sg.len = hp.slen[p];
        const Stress2 w = stress_jump(hp.px[p], hp.py[p], sg, 0.0, P->dt, hp.mu, hp.cs);
        k0[hp.perm[p]] = hp.pnx[p] * w.x + hp.pny[p] * w.y;
    }
    return FDPH_OK;
}

int fdph_rupture_init(fdph_plan_t P, const fdph_friction* f) {
    if (!P || !f || !f->tau0 || !(f->sigma_n > 0.0) || !(f->Dc > 0.0) || f->mu_d > f->mu_s ||
        (f->law != 0 && f->law != 1)) {
        set_error("fdph_rupture_init: friction with tau0, sigma_n > 0, Dc > 0, mu_d <= mu_s, law 0 or 1 required");
        return FDPH_E_ARG;
    }
    if (P->predicted) return pending_commit(P);
    if (P->nrhs != 1) {
        set_error("fdph_rupture_init: dynamic rupture takes plans of one right-hand side (nrhs = 1)");
        return FDPH_E_ARG;
    }
    std::vector<double> k0;
    int rc0 = self_coefficients(P, k0);
    if (rc0) return rc0;
    if (!P->rupture) {
        double *tau0 = nullptr, *kk = nullptr, *slip = nullptr;
        FrictionLaw* law = nullptr;
        int rc;
        if ((rc = dalloc(P, &tau0, P->N)) || (rc = dalloc(P, &kk, P->N)) || (rc = dalloc(P, &slip, P->N)) ||
            (rc = dalloc(P, &law, 1)))
            return rc;
        P->fr.law = law;
        P->fr.tau0 = tau0;
        P->fr.k0 = kk;
        P->fr.slip = slip;
    }
    // ordered after the caller's work on the plan's stream (tau0 may have been written there)
    FDPH_CUDA(cudaMemcpyAsync((void*)P->fr.tau0, f->tau0, P->N * sizeof(double), cudaMemcpyDeviceToDevice, P->stream));
    FDPH_CUDA(cudaMemcpyAsync((void*)P->fr.k0, k0.data(), P->N * sizeof(double), cudaMemcpyHostToDevice, P->stream));
    const FrictionLaw law{f->sigma_n, f->mu_s, f->mu_d, f->Dc, f->law};
    FDPH_CUDA(cudaMemcpyAsync((void*)P->fr.law, &law, sizeof(law), cudaMemcpyHostToDevice, P->stream));
    FDPH_CUDA(cudaMemsetAsync(P->fr.slip, 0, P->N * sizeof(double), P->stream));
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    P->fr.dt = P->dt;
    P->rupture = true;
    return FDPH_OK;
}

int fdph_rupture_step(fdph_plan_t P, double* D_n, double* T_n) {
    if (!P || !D_n || !T_n) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    if (!P->rupture) {
        set_error("fdph_rupture_init has not been called on this plan");
        return FDPH_E_STATE;
    }
    if (P->n >= P->M) {
        set_error("the plan has already taken M steps");
        return FDPH_E_STATE;
    }
    return P->precision != FDPH_FP64 ? rupture_steps<float>(P, 1, D_n, T_n) : rupture_steps<double>(P, 1, D_n, T_n);
}

int fdph_rupture_run(fdph_plan_t P, int32_t steps, double* D, double* T) {
    if (!P || !D || !T || steps < 0) return FDPH_E_ARG;
    if (P->predicted) return pending_commit(P);
    if (P->n + steps > P->M) {
        set_error("run would pass step M");
        return FDPH_E_STATE;
    }
    if (!P->rupture) {
        set_error("fdph_rupture_init has not been called on this plan");
        return FDPH_E_STATE;
    }
    return P->precision != FDPH_FP64 ? rupture_steps<float>(P, steps, D, T) : rupture_steps<double>(P, steps, D, T);
}

int fdph_rupture_slip(fdph_plan_t P, double* slip) {
    if (!P || !slip) return FDPH_E_ARG;
    if (!P->rupture) return FDPH_E_STATE;
    FDPH_CUDA(cudaMemcpyAsync(slip, P->fr.slip, P->N * sizeof(double), cudaMemcpyDeviceToDevice, P->stream));
    return FDPH_OK;
}

int fdph_predict(fdph_plan_t P, double* T_pred) {
    if (!P || !T_pred) return FDPH_E_ARG;
    if (P->nrhs != 1) {
        set_error("this call takes plans of one right-hand side (nrhs = 1)");
        return FDPH_E_ARG;
    }
    if (P->predicted) return pending_commit(P);
    if (P->n >= P->M) {
        set_error("the plan has already taken M steps");
        return FDPH_E_STATE;
    }
    int rc = P->precision != FDPH_FP64 ? launch_predict<float>(P, T_pred) : launch_predict<double>(P, T_pred);
    if (rc == FDPH_OK) P->predicted = true;
    return rc;
}

int fdph_commit(fdph_plan_t P, const double* D_n) {
    if (!P || !D_n) return FDPH_E_ARG;
    if (P->nrhs != 1) {
        set_error("this call takes plans of one right-hand side (nrhs = 1)");
        return FDPH_E_ARG;
    }
    if (!P->predicted) {
        set_error("fdph_commit without a preceding fdph_predict of this step");
        return FDPH_E_STATE;
    }
    int rc = P->precision != FDPH_FP64 ? launch_commit<float>(P, D_n) : launch_commit<double>(P, D_n);
    if (rc == FDPH_OK) {
        P->predicted = false;
        P->n += 1;
    }
    return rc;
}

int fdph_self(fdph_plan_t P, double* diag) {
    if (!P || !diag) return FDPH_E_ARG;
    std::vector<double> k0;
    int rc = self_coefficients(P, k0);
    if (rc) return rc;
    memcpy(diag, k0.data(), k0.size() * sizeof(double));
    return FDPH_OK;
}

int fdph_set_profiling(fdph_plan_t P, int enable) {
    if (!P) return FDPH_E_ARG;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    prof_drain(P);
    for (int k = 0; k < FDPH_NUM_KERNELS; ++k) {
        P->prof_ms[k] = 0.0;
        P->prof_n[k] = 0;
    }
    P->prof = enable != 0;
    return FDPH_OK;
}

int fdph_kernel_times(fdph_plan_t P, double* ms, int64_t* launches) {
    if (!P || !ms || !launches) return FDPH_E_ARG;
    FDPH_CUDA(cudaStreamSynchronize(P->stream));
    prof_drain(P);
    for (int k = 0; k < FDPH_NUM_KERNELS; ++k) {
        ms[k] = P->prof_ms[k];
        launches[k] = P->prof_n[k];
    }
    return FDPH_OK;
}

int fdph_batch_create(const fdph_plan_t* plans, int32_t count, fdph_batch_t* out) {
    if (!plans || !out || count < 1 || count > 1024) return FDPH_E_ARG;
    *out = nullptr;
    for (int p = 0; p < count; ++p) {
        if (!plans[p]) return FDPH_E_ARG;
        for (int q = 0; q < p; ++q)
            if (plans[q] == plans[p]) {
                set_error("fdph_batch_create: a plan appears twice");
                return FDPH_E_ARG;
            }
        if (plans[p]->device != plans[0]->device || plans[p]->precision != plans[0]->precision) {
            set_error("fdph_batch_create: plans of one batch share the device and the precision");
            return FDPH_E_ARG;
        }
        if (plans[p]->predicted) return pending_commit(plans[p]);
        if (plans[p]->nrhs != 1 || plans[p]->far_mode != 0) {
            set_error("fdph_batch_create: batches take plans of one right-hand side (nrhs = 1) and far_mode 0");
            return FDPH_E_ARG;
        }
    }
    fdph_batch_t B = new fdph_batch_s;
    B->device = plans[0]->device;
    B->precision = plans[0]->precision;
    B->plans.assign(plans, plans + count);
    for (int p = 0; p < count; ++p) B->version.push_back(plans[p]->sched_version);
    cudaSetDevice(B->device);
    if (cudaStreamCreateWithFlags(&B->hub, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&B->ev_plan, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&B->ev_hub, cudaEventDisableTiming) != cudaSuccess) {
        set_error("fdph_batch_create: cudaStreamCreate / cudaEventCreate failed");
        fdph_batch_destroy(B);
        return FDPH_E_CUDA;
    }
    *out = B;
    return FDPH_OK;
}

int fdph_batch_run(fdph_batch_t B, int32_t steps, const double* const* D, double* const* T) {
    if (!B || !D || !T || steps < 0) return FDPH_E_ARG;
    for (size_t p = 0; p < B->plans.size(); ++p)
        if (!D[p] || !T[p]) return FDPH_E_ARG;
    int rc = batch_check(B, steps);
    if (rc || steps == 0) return rc;
    cudaSetDevice(B->device);
    if ((rc = batch_join(B))) return rc;
    for (size_t p = 0; p < B->plans.size() && !rc; ++p) rc = run_any(B->plans[p], steps, D[p], T[p]);
    const int joined = batch_join(B);   // (after an error too: some plans may have been launched)
    return rc ? rc : joined;
}

int fdph_batch_rupture_run(fdph_batch_t B, int32_t steps, double* const* D, double* const* T) {
    if (!B || !D || !T || steps < 0) return FDPH_E_ARG;
    for (size_t p = 0; p < B->plans.size(); ++p) {
        if (!D[p] || !T[p]) return FDPH_E_ARG;
        if (!B->plans[p]->rupture) {
            set_error("fdph_rupture_init has not been called on a plan of the batch");
            return FDPH_E_STATE;
        }
    }
    int rc = batch_check(B, steps);
    if (rc || steps == 0) return rc;
    cudaSetDevice(B->device);
    if ((rc = batch_join(B))) return rc;
    for (size_t p = 0; p < B->plans.size() && !rc; ++p) {
        fdph_plan_t P = B->plans[p];
        rc = P->precision != FDPH_FP64 ? rupture_steps<float>(P, steps, D[p], T[p]) : rupture_steps<double>(P, steps, D[p], T[p]);
    }
    const int joined = batch_join(B);
    return rc ? rc : joined;
}

int fdph_batch_synchronize(fdph_batch_t B) {
    if (!B) return FDPH_E_ARG;
    for (fdph_plan_t P : B->plans) {
        FDPH_CUDA(cudaStreamSynchronize(P->stream));
        int rc = check_device_error(P);
        if (rc) return rc;
    }
    return FDPH_OK;
}

void fdph_batch_destroy(fdph_batch_t B) {
    if (!B) return;
    cudaSetDevice(B->device);
    if (B->hub) {   // (behind the last call's work; the plans are not touched)
        cudaStreamSynchronize(B->hub);
        cudaStreamDestroy(B->hub);
    }
    if (B->ev_plan) cudaEventDestroy(B->ev_plan);
    if (B->ev_hub) cudaEventDestroy(B->ev_hub);
    delete B;
}

void fdph_destroy(fdph_plan_t P) {
    if (!P) return;
    cudaSetDevice(P->device);
    if (P->stream) cudaStreamSynchronize(P->stream);
    prof_drain(P);
    drop_graphs(P);
    for (int k = 0; k < 2; ++k) {
        if (P->side[k]) cudaStreamDestroy(P->side[k]);
        if (P->ev_join[k]) cudaEventDestroy(P->ev_join[k]);
    }
    if (P->ev_fork) cudaEventDestroy(P->ev_fork);
    if (P->h2d) cudaStreamSynchronize(P->h2d);
    if (P->d2h) cudaStreamSynchronize(P->d2h);
    if (P->h2d) cudaStreamDestroy(P->h2d);
    if (P->d2h) cudaStreamDestroy(P->d2h);
    for (int q = 0; q < fdph_plan_s::kIoSlots; ++q) {
        if (P->ev_in[q]) cudaEventDestroy(P->ev_in[q]);
        if (P->ev_out[q]) cudaEventDestroy(P->ev_out[q]);
        if (P->ev_free[q]) cudaEventDestroy(P->ev_free[q]);
    }
    for (void* p : P->allocs) cudaFree(p);
    if (P->own_stream && P->stream) cudaStreamDestroy(P->stream);
    delete P;
}

}  // extern "C"
