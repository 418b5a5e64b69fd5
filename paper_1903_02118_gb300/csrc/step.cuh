// step.cuh -- device views of a plan and the kernels of a block of time steps.
//
// A block is up to kBlk consecutive steps n, n + 1, ..., n + nb - 1.  Where their slip rates are given
// (fdph_run, fdph_run_host) one block runs, for all its steps at once,
//   push     D -> slip-rate ring (internal order); cumulative slip C_j with a compensated (Kahan) FP64
//            sum, -> cumulative-slip ring; both also element-major for the scatter
//   fir      Domain F, formula 1 (Eq. 32): Dhat_j(n) = sum_{m < Dm_j} h_{j,m} D_{j,n-m}
//   scatter  formula 2 (Eq. 42): Tbar'_l[n + delay_j] += g_{l,j} u_j(n), one writer per ring slot;
//            u = Dhat (Domain F), dt C (Domain S, App. B.1), D (transient); the ring is the shift
//            operator M of Eq. 40 as a base-pointer increment
//   trconv   transient (App. B.3): Z_l(t) = sum_{m < Dm_tr} h^tr_m Y_l(t - m)
//   far      formula 3 (Eq. 39): Tfar_i(n) = sum_{blocks} sum_l f_{l,i} Tbar'_l[n - dm_i]
//   near     inadmissible leaves (App. E): sum_{k < W} K_{ij,k} D_{j,n-k} + Kstat_ij dt C_j(n - W)
//            (+ exponential tails), per work item into a partial-sum slot
//   gather   T_i = Tfar_i + the receiver's near partials, in the caller's element order
// so that every coefficient, factor, delay and waveform is read once per block instead of once per
// step.  A rupture block does not know its slip rates: see rup_step_kernel.
//
// Every output is summed in an order that depends on its step alone, not on the block it falls in or
// on the block's length: a march gives the same bits however it is cut into calls.
//
// Ring lengths leave room for a whole block (kBlk - 1 slots beyond what one step needs): the
// scatter of a block may run before its transient convolution and its Eq. 39 read their slots.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

static const int kBlk = 16;   // steps of one block at most

static const int kErrTimeout = 1;   // error word: a bounded wait gave up
static const int kErrIndex = 2;     // error word: an index check failed (FDPH_CHECK builds)
// Bounded-index debug build (-DFDPH_CHECK, libfdph_check.so): every ring, state, partial-sum and
// near-slice access of the step kernels is checked against the extent of its array; a failing
// check records kErrIndex in the plan's error word and skips the access (no trap: the kernel
// carries on and finishes), and the next synchronising call returns FDPH_E_CHECK.  In the normal
// build FDPH_IDX is the constant true and costs nothing.
__device__ __forceinline__ bool fdph_idx_check(bool ok, int* err) {
    if (!ok && err) atomicExch(err, kErrIndex);
    return ok;
}
#ifdef FDPH_CHECK
#define FDPH_IDX(cond, err) fdph_idx_check((cond), (err))
#else
#define FDPH_IDX(cond, err) true
#endif

struct SbDev {
    int kind, rank, r0, nr, s0, ns, L, LZ, taps, maxdelay, mindm, run0, soe, ident, LH;
    long long f, g, h, ring, zring, dhat, delay, dm, ustate, trc, phi;
    long long uhist;    // delayed-history form: [LH][ns] source values u_j of the last LH steps
    int mindelay, qn;   // qn: quantized ranges of a transient's taps (0: exact taps)
    long long qb;       // offset of their qn + 1 bounds in ints
};

struct NearDev {
    int r0, nr, s0, ns, W, sl, sla, pad;
    long long tensor, stat, tail, vstate;
};

// one near-field work item as its warp reads it (one 64-byte load)
struct __align__(16) NearTask {
    long long off;       // element offset of the item's first slice (tensor, or aux for kind 1)
    int item, k0, k1, kind, nr, ns, sl, s0, W, vstate;
    int pad[2];
};
static_assert(sizeof(NearTask) == 64, "one work item is four 16-byte loads");

// one (block, receiver) entry of Eq. 39 as its lane reads it
struct __align__(16) FarEnt {
    long long base;      // first double of the block's ring (Tbar', or Z of a transient)
    long long f;         // the receiver's factor row, or (F = I) its rank index
    int L, dm, rank;     // slots of the ring, the receiver's delay, the block's rank
    int flags;           // 1: transient (Z ring), 2: F = I
};
static_assert(sizeof(FarEnt) == 32, "one entry is two 16-byte loads");

// 32 FIR tasks of one source element (one per lane): waveforms interleaved [taps][32]
struct __align__(16) FirGroup {
    long long h;         // first waveform coefficient of the group
    int src, taps;       // source element, longest waveform of the group
    int first, count;    // the lanes' Dhat indices at fir_dhat[first + lane], lane < count
    int pad[2];
};

// near leaves that act within a block of an unknown slip rate (rupture), by receiver group
struct RecGroup {
    int r0, nr, leaf0, nleaf;
};
struct __align__(16) RecLeaf {
    long long off;       // element offset of kernel step 0 in the window slices
    long long stat;      // W < kBlk: the static tile among the aux slices; else -1
    int sl, r0, nr, s0, ns, kz, W, pad;
};
static_assert(sizeof(RecLeaf) == 48, "a leaf is three 16-byte loads");

static const int kMaxSoe = 16;
static const int kMaxRhs = 8;    // right-hand sides of one plan at most (1, 2, 4 or 8)

// which slip rates of the ring a near-field launch may use
enum { HIST_ALL = 0,      // all
       HIST_BASE = 1,     // those of steps before the launch's aligned block (n rounded down to kBlk)
       HIST_STEP = 2 };   // those of steps before n

template <class T>
struct StepArgs {
    int n, n_off, nb, hist;   // first step (+ n_off), steps of the launch, HIST_*
    int N, WD, WC;
    // graph replay: the first step is read from n_dev[0], and D_in / T_out advance by io_stride
    // elements per step past the step n_dev[1] of the call's first row (unused when n_dev is null)
    const int* n_dev;
    long long io_stride;
    double dt;
    const double* D_in;       // caller's D_n (geometry order), io_stride per step
    double* T_out;            // caller's T_n (geometry order)
    double* thist;            // [kBlk][N] gather target of a rupture block (internal order), or null
    const int* perm;          // internal -> geometry
    double* Dring;            // [WD][N]
    float* Dring32;           // [WD][N] FP32 copy of Dring (plans whose near-field rows are FP32)
    double* Cring;            // [WC][N]
    double* C;                // [N] cumulative slip (rounded sum)
    double* Ccomp;            // [N] Kahan compensation
    double *blkD, *blkC;      // D and dt C of the block's steps, [N][kBlk]; of one step [N][nrhs] (blk_pitch)
    // far field
    const SbDev* sbs;
    const T* fac;
    const int* ints;
    const int4* runs;         // {delay, sources, first in src_order, first source}
    const int* src_order;
    const int4* sc_tasks;     // scatter warp tasks {block, first slot offset, its place in last_run, log2 lanes per slot}
    const int* last_run;      // per slot offset of a block: the last run with delay <= it
    int n_sct;
    const FarEnt* ents;       // Eq. 39 entries, receiver-major
    const double* ent_phi;    // sub-step receiver delays (interpolated reading; null: rounded)
    const int* g_ptr;         // [N + 1]
    long long n_ent;
    double* tfar;             // [kBlk][N] far-field traction of each receiver
    const FirGroup* fir;
    const T* fir_h;
    const int* fir_dhat;
    int n_fir, fir_taps;      // groups; longest waveform of all
    const int* tr_sb;
    const int* tr_l;
    int n_tr;
    double* ring;
    double* zring;
    T* dhat;                  // [tasks][kBlk]; of one step [tasks][nrhs]
    long long len_ring, len_zring, len_dhat, len_ustate, len_vstate;
    // near field
    const NearTask* tasks;    // near-field work items, largest first
    int n_items;
    const void* tensor;       // near-field window slices (window storage type)
    float kinv;               // inverse of the window coefficients' storage scale (FP16: 2^-e, else 1)
    const void* stat;         // aux slices: static tiles, exponential-tail coefficients (aux storage type)
    long long len_tensor, len_aux;   // elements of tensor and stat (index checks of FDPH_CHECK builds)
    double* partial;          // [kBlk][cap_partial]: [item][32] per step
    long long cap_partial;
    const int* np_ptr;
    const int* np_idx;
    int* err;                 // device error word (1 = a bounded wait gave up)
    // exponential tails (extension; soe == 0: the paper's static cut)
    int soe;
    const double* rho;        // [soe] decay factors
    double* ustate;           // transient blocks: [rank][soe] per block
    const double* trcoef;     // transient blocks: [soe] tail coefficients per block (FP64)
    double* vstate;           // inadmissible leaves: [soe][ns] per leaf
    // right-hand sides: every time-stepping state array above is [nrhs][...] with these strides
    // (elements); the caller's rows D_n, T_n are [nrhs][N] (io_stride = nrhs N per step)
    int nrhs;
    long long rs_D, rs_C, rs_partial;
    // delayed-history form of Eq. 42 (far_mode 1)
    double* uhist;            // [blocks][LH][ns] source values
    long long len_uhist;
    const int2* rec_tasks;    // (block, source) recorded per step
    const int2* gat_tasks;    // (block, rank index) gathered per step
    int n_rec, n_gat;
    // rupture blocks
    const RecGroup* rec_groups;
    const RecLeaf* rec_leaves;
    int n_groups;
};

// ring slot of step a (a may be negative; |a| < 2^31)
__device__ __forceinline__ int wrap(int a, int L) {
    const int r = a % L;
    return r < 0 ? r + L : r;
}

template <class T>
__device__ __forceinline__ int step_index(const StepArgs<T>& a) {
    return (a.n_dev ? *a.n_dev : a.n) + a.n_off;
}

// element offset of step n's row of D_in / T_out
template <class T>
__device__ __forceinline__ long long io_offset(const StepArgs<T>& a, int n) {
    return a.n_dev ? (long long)(n - a.n_dev[1]) * a.io_stride : 0;
}

// slip rates of steps >= this are taken as zero by a near-field launch that starts at step n
template <class T>
__device__ __forceinline__ int hist_end(const StepArgs<T>& a, int n) {
    return a.hist == HIST_ALL ? n + a.nb : a.hist == HIST_BASE ? (n & ~(kBlk - 1)) : n;
}

// pitch of blkD, blkC and dhat (scratch of one launch sequence): the steps of a block side by side, or the
// right-hand sides of a single step, so that the scatter reads them together
template <class T>
__device__ __forceinline__ int blk_pitch(const StepArgs<T>& a) {
    return a.nb == 1 ? a.nrhs : kBlk;
}

// the arguments of right-hand side r
template <class T>
__device__ __forceinline__ StepArgs<T> rhs_args(const StepArgs<T>& a0, int r) {
    StepArgs<T> a = a0;
    if (r) {
        const long long rN = (long long)r * a0.N;
        if (a0.D_in) a.D_in = a0.D_in + rN;
        if (a0.T_out) a.T_out = a0.T_out + rN;
        a.Dring = a0.Dring + r * a0.rs_D;
        if (a0.Dring32) a.Dring32 = a0.Dring32 + r * a0.rs_D;
        a.Cring = a0.Cring + r * a0.rs_C;
        a.C = a0.C + rN;
        a.Ccomp = a0.Ccomp + rN;
        a.blkD = a0.blkD + (a0.nb == 1 ? r : rN * kBlk);
        a.blkC = a0.blkC + (a0.nb == 1 ? r : rN * kBlk);
        a.ring = a0.ring + r * a0.len_ring;
        a.zring = a0.zring + r * a0.len_zring;
        a.dhat = a0.dhat + (a0.nb == 1 ? r : r * a0.len_dhat);
        a.tfar = a0.tfar + rN * kBlk;
        if (a0.ustate) a.ustate = a0.ustate + r * a0.len_ustate;
        if (a0.vstate) a.vstate = a0.vstate + r * a0.len_vstate;
        a.partial = a0.partial + r * a0.rs_partial;
        if (a0.uhist) a.uhist = a0.uhist + r * a0.len_uhist;
    }
    return a;
}

// Conversions between FP32 and FP64 in integer arithmetic.  The hardware's run on the FP64 pipe, two
// lanes a clock and SM like its additions (a warp takes 15 clocks; the integer forms take 3 to 6), and
// the FP64 pipe bounds the far field and the aux slices.  Same values: exact widening, narrowing to
// nearest even; zeros here, subnormals, infinities and NaN by the hardware conversion.
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) {
    const unsigned u = __float_as_uint(x);
    if (((u >> 23) & 0xffu) - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
    if (!(u << 1)) return __hiloint2double((int)u, 0);
    return (double)x;
}
__device__ __forceinline__ double narrow(double x, double) { return x; }
__device__ __forceinline__ float narrow(double x, float) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const unsigned e = (h >> 20) & 0x7ffu;
    if (e - 897u <= 253u) {   // a normal FP32 number (or rounded up to infinity)
        unsigned v = (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29);
        const unsigned rem = l & 0x1fffffffu;
        v += rem > 0x10000000u || (rem == 0x10000000u && (v & 1u)) ? 1u : 0u;
        return __uint_as_float((h & 0x80000000u) | v);
    }
    if (!((h << 1) | l)) return __uint_as_float(h);
    return (float)x;
}

__global__ void advance_step_kernel(int* n_dev, int k) { *n_dev += k; }

__global__ void place_step_kernel(int* n_dev, int n, int first) {
    n_dev[0] = n;       // step index
    n_dev[1] = first;   // step of the call's first row of D / T
}

// Sums of B (1 or 16) columns over the lanes of a warp, each in the order of the xor butterfly
// (offsets 16, 8, 4, 2, 1).  B = 16: at each level the two halves of a pair keep one half of the
// columns each, so 16 columns take 16 additions instead of 80 (the additions are FP64, of which an
// SM does two a clock); the result of column sum_col(lane) is in lane.
template <int B>
__device__ __forceinline__ double warp_columns(double (&c)[B], int lane) {
    if constexpr (B == 1) {
        double v = c[0];
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    } else {
        static_assert(B == 16, "one or sixteen columns");
#pragma unroll
        for (int w = 8, o = 16; w; w >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < w; ++i) {
                const double send = up ? c[i] : c[i + w], keep = up ? c[i + w] : c[i];
                c[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        return c[0] + __shfl_xor_sync(0xffffffffu, c[0], 1);
    }
}

template <int B>
__device__ __forceinline__ int sum_col(int lane) {
    return B == 1 ? 0 : ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

// ---- push

// one element's slip rate d of step n (the b-th of its block) into the rings and sums
template <class T>
__device__ __forceinline__ void push_one(const StepArgs<T>& a, int p, int n, int b, double d, double& c, double& comp) {
    const size_t slot = (size_t)wrap(n, a.WD) * a.N + p;
    a.Dring[slot] = d;
    if (a.Dring32) a.Dring32[slot] = (float)d;
    const size_t at = (size_t)p * blk_pitch(a) + b;
    a.blkD[at] = d;
    // compensated running sum of the slip (units of dt)
    const double y = d - comp;
    const double t = c + y;
    comp = (t - c) - y;
    c = t;
    a.Cring[(size_t)wrap(n, a.WC) * a.N + p] = t;
    a.blkC[at] = a.dt * t;
}

template <class T>
__global__ void push_kernel(StepArgs<T> a0) {
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.N) return;
    const int n = step_index(a), e = a.perm[p];
    const double* D = a.D_in + io_offset(a, n) + e;
    double d[kBlk];
#pragma unroll
    for (int b = 0; b < kBlk; ++b) d[b] = b < a.nb ? D[b * a.io_stride] : 0.0;
    double c = a.C[p], comp = a.Ccomp[p];
#pragma unroll
    for (int b = 0; b < kBlk; ++b)
        if (b < a.nb) push_one(a, p, n + b, b, d[b], c, comp);
    a.C[p] = c;
    a.Ccomp[p] = comp;
}

// ---- Eq. 32 (FIR)

// The slip-rate history and the sums in the factor type: FP32 plans read the FP32 copy of the ring
// and add in FP32 (this GPU's FP64 rate is a small fraction of its FP32 rate, and the ~27 taps of
// a waveform lose ~2^-24 sqrt(27) relative), FP64 plans stay in FP64
template <class T>
__device__ __forceinline__ const T* fir_ring(const StepArgs<T>& a) {
    if constexpr (sizeof(T) == 4) return a.Dring32; else return a.Dring;
}

// One warp per group of 32 tasks of one source element (a task: one F block that contains it).
// The source's last taps + B - 1 slip rates go to shared memory, each lane holds the B sums of its
// task, and the waveforms are stored interleaved over the 32 lanes, so that a tap is one coalesced
// load for B multiply-adds.  (staged = false: waveforms too long for shared memory read the ring.)
constexpr int kFirWarps = 4;

template <class T, int B>
__global__ void __launch_bounds__(32 * kFirWarps) fir_kernel(StepArgs<T> a0, bool staged) {
    extern __shared__ __align__(8) unsigned char fir_smem[];
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = blockIdx.x * kFirWarps + warp;
    if (w >= a.n_fir) return;   // warp-uniform
    const FirGroup g = a.fir[w];
    const int n = step_index(a);
    const int rows = g.taps + B - 1;
    if (!FDPH_IDX(g.taps <= a.fir_taps && g.taps <= a.WD && g.src < a.N, a.err)) return;
    // slip rate of step n + B - 1 - x (zero before the march and past the block's steps)
    auto rate = [&](int x) {
        const int t = n + B - 1 - x;
        return x < rows && t >= 0 && t < n + a.nb ? fir_ring(a)[(size_t)wrap(t, a.WD) * a.N + g.src] : (T)0;
    };
    T* sd = (T*)fir_smem + (size_t)warp * (a.fir_taps + 2 * B);
    if (staged) {
        for (int x = lane; x < rows + B; x += 32) sd[x] = rate(x);
        __syncwarp();
    }
    auto d_at = [&](int x) { return staged ? sd[x] : rate(x); };
    const T* h = a.fir_h + g.h + lane;
    T s0[B], s1[B];
#pragma unroll
    for (int b = 0; b < B; ++b) s0[b] = s1[b] = 0;
    // even and odd taps in separate sums; taps in chunks of B: the 2 B - 1 slip rates that B taps of B steps need
    // sit in registers
    for (int m0 = 0; m0 < g.taps; m0 += B) {
        T x[2 * B - 1];
#pragma unroll
        for (int q = 0; q < 2 * B - 1; ++q) x[q] = d_at(min(m0 + q, rows + B - 1));
        constexpr int F = sizeof(T) == 4 ? B : B / 4;   // taps in flight together (registers)
#pragma unroll
        for (int v = 0; v < B; v += F) {
            T hm[F];
#pragma unroll
            for (int u = 0; u < F; ++u) hm[u] = m0 + v + u < g.taps ? h[(size_t)(m0 + v + u) * 32] : (T)0;
#pragma unroll
            for (int u = 0; u < F; ++u)
#pragma unroll
                for (int b = 0; b < B; ++b)
                    (u & 1 ? s1 : s0)[b] = fma(hm[u], x[B - 1 - b + v + u], (u & 1 ? s1 : s0)[b]);
        }
    }
    if (lane < g.count) {
        const long long q = a.fir_dhat[g.first + lane];
        if (FDPH_IDX((q + 1) * kBlk <= a.len_dhat, a.err)) {
#pragma unroll
            for (int b = 0; b < B; ++b) a.dhat[q * kBlk + b] = s0[b] + s1[b];
        }
    }
}

// One step of NR right-hand sides (the sums of fir_kernel): a tap is read once for all of them.  With a grid row per
// right-hand side every waveform, factor and run was read eight times: eight right-hand sides of N = 6000, one step
// 98 us here and 395 us in the scatter, now 55 and 133.
constexpr int kFirGroups = 2;   // groups of a warp, one after the other: mostly of one source, staged once

template <class T, int NR>
__global__ void __launch_bounds__(32 * kFirWarps) fir_step_kernel(StepArgs<T> a, bool staged) {
    extern __shared__ __align__(8) unsigned char fir_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = step_index(a);
    const int pitch = a.fir_taps + 2;
    T* sd = (T*)fir_smem + (size_t)warp * NR * pitch;
    int src = -1;
    for (int i = 0; i < kFirGroups; ++i) {
        const int w = (blockIdx.x * kFirWarps + warp) * kFirGroups + i;
        if (w >= a.n_fir) return;   // warp-uniform
        const FirGroup g = a.fir[w];
        if (!FDPH_IDX(g.taps <= a.fir_taps && g.taps <= a.WD && g.src < a.N, a.err)) continue;
        auto rate = [&](int x, int r) {
            const int t = n - x;
            return t >= 0 ? fir_ring(a)[r * a.rs_D + (size_t)wrap(t, a.WD) * a.N + g.src] : (T)0;
        };
        if (staged && g.src != src) {
            __syncwarp();
            for (int x = lane; x < a.fir_taps; x += 32)
#pragma unroll
                for (int r = 0; r < NR; ++r) sd[r * pitch + x] = rate(x, r);
            __syncwarp();
            src = g.src;
        }
        auto d_at = [&](int x, int r) { return staged ? sd[r * pitch + x] : rate(x, r); };
        const T* h = a.fir_h + g.h + lane;
        T s0[NR], s1[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) s0[r] = s1[r] = 0;
        int m = 0;
#pragma unroll 4
        for (; m + 1 < g.taps; m += 2) {
            const T h0 = h[(size_t)m * 32], h1 = h[(size_t)(m + 1) * 32];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                s0[r] = fma(h0, d_at(m, r), s0[r]);
                s1[r] = fma(h1, d_at(m + 1, r), s1[r]);
            }
        }
        if (m < g.taps) {
            const T h0 = h[(size_t)m * 32];
#pragma unroll
            for (int r = 0; r < NR; ++r) s0[r] = fma(h0, d_at(m, r), s0[r]);
        }
        if (lane < g.count) {
            const long long q = a.fir_dhat[g.first + lane];
            if (FDPH_IDX((q + 1) * kBlk <= a.len_dhat, a.err)) {
#pragma unroll
                for (int r = 0; r < NR; ++r) a.dhat[q * NR + r] = s0[r] + s1[r];
            }
        }
    }
}

// ---- Eq. 42

// source quantity u_j of Eq. 42 of the block's b-th step: Dhat (Domain F), dt * cumulative slip
// (Domain S, App. B.1), slip rate (transient); of a single step, of right-hand side r past the arguments' own.
// pitch: blk_pitch(a), where it is not known when the kernel is compiled
template <class T>
__device__ __forceinline__ double source_value(const StepArgs<T>& a, const SbDev& sb, int jl, int pitch, int b, int r = 0) {
    if (sb.kind == 0) return wide(a.dhat[(sb.dhat + jl) * pitch + b + r]);
    return (sb.kind == 1 ? a.blkC : a.blkD)[(size_t)(sb.s0 + jl) * pitch + b + r];
}

// Eq. 42 slot by slot: the steps of a block add to the ring slots n + mindelay ... n + nb - 1 +
// maxdelay of a sub-block; a lane owns one (slot, rank index) and collects the sources whose delay
// brings one of the block's steps there, oldest step first.  2^lg lanes per slot cover the rank
// index, so the slots of a warp are one contiguous piece of the ring, read and written once per
// block (a step-by-step scatter updates a slot once for every source).
// NR right-hand sides in one lane (kOne, one step: the factors are read once), or one per grid row (blocks).
template <class T, int NR, bool kOne>
__global__ void scatter_kernel(StepArgs<T> a0) {
    constexpr int pitch = kOne ? NR : kBlk;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    if (w >= a.n_sct) return;
    const int n = step_index(a), nb = a.nb;
    const int4 tk = a.sc_tasks[w];
    const SbDev& sb = a.sbs[tk.x];
    const int G = 1 << tk.w, lj = lane & (G - 1);
    const int d = tk.y + (lane >> tk.w);
    const int maxdelay = sb.maxdelay, rank = sb.rank, run0 = sb.run0;
    if (d > maxdelay + nb - 1) return;
    const int run = a.last_run[tk.z + (lane >> tk.w)];
    const int4 top = a.runs[run];
    if (d - top.x >= nb) return;   // no step of the block comes to this slot
    const int slot = wrap(n + d, sb.L);
    double* ring = a.ring + sb.ring + (long long)slot * rank;
    if (!FDPH_IDX(sb.ring + (long long)(slot + 1) * rank <= a.len_ring, a.err)) return;
    if (sb.ident == 2) {
        // G is the identity: column j of a slot receives source j only, once
        for (int q = run; q >= run0; --q) {
            const int4 rn = a.runs[q];
            const int b = d - rn.x;
            if (b >= nb) break;
            for (int u = lj; u < rn.y; u += G) {
                const int jl = a.src_order[rn.z + u];
                if (!FDPH_IDX(jl < rank, a.err)) continue;
#pragma unroll
                for (int r = 0; r < NR; ++r) ring[r * a.len_ring + jl] = source_value(a, sb, jl, pitch, b, r);
            }
        }
        return;
    }
    const bool fresh = d >= maxdelay;   // the slot comes into the ring's range within this block
    const T* g = a.fac + sb.g;
    for (int l = lj; l < rank; l += G) {
        double v[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) v[r] = fresh ? 0.0 : ring[r * a.len_ring + l];
        for (int q = run; q >= run0; --q) {
            const int4 rn = a.runs[q];
            const int b = d - rn.x;
            if (b >= nb) break;
            if (rn.y == 1) {
                const double gl = wide(g[(long long)rn.w * rank + l]);
#pragma unroll
                for (int r = 0; r < NR; ++r) v[r] = fma(gl, source_value(a, sb, rn.w, pitch, b, r), v[r]);
            } else {
                double s[NR];
#pragma unroll
                for (int r = 0; r < NR; ++r) s[r] = 0.0;
                for (int u = 0; u < rn.y; ++u) {
                    const int jl = a.src_order[rn.z + u];
                    const double gl = wide(g[(long long)jl * rank + l]);
#pragma unroll
                    for (int r = 0; r < NR; ++r) s[r] = fma(gl, source_value(a, sb, jl, pitch, b, r), s[r]);
                }
#pragma unroll
                for (int r = 0; r < NR; ++r) v[r] += s[r];
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) ring[r * a.len_ring + l] = v[r];
    }
}

// Delayed-history form of Eq. 42 (the gather variant of Sec. 5.3; blocks of one step): instead of
// adding g_{l,j} u_j to the future slots n + delay_j, every step records u_j(n) in the block's
// history of the last LH = maxdelay - mindelay + 1 steps and computes the one slot that the step
// completes,
//     Tbar'_l[n + mindelay] = sum_j g_{l,j} u_j(n + mindelay - delay_j),
// by causality (min(dm + delay) >= 1) a slot no evaluation of step n reads yet.
template <class T>
__global__ void record_kernel(StepArgs<T> a0) {
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= a.n_rec) return;
    const int2 t = a.rec_tasks[q];
    const SbDev& sb = a.sbs[t.x];
    a.uhist[sb.uhist + (long long)wrap(step_index(a), sb.LH) * sb.ns + t.y] = source_value(a, sb, t.y, blk_pitch(a), 0);
}

// one warp per (block, rank index l), lanes over the sources
template <class T>
__global__ void hgather_kernel(StepArgs<T> a0) {
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= a.n_gat) return;   // warp-uniform
    const int2 t = a.gat_tasks[w];
    const SbDev& sb = a.sbs[t.x];
    const int l = t.y;
    const int s = step_index(a) + sb.mindelay;
    const int* dl = a.ints + sb.delay;
    const double* u = a.uhist + sb.uhist;
    double acc = 0.0;
    if (sb.ident == 2) {   // G is the identity: rank index l is source l
        if (lane == 0) acc = u[(long long)wrap(s - dl[l], sb.LH) * sb.ns + l];
    } else {
        const T* g = a.fac + sb.g;
        for (int j = lane; j < sb.ns; j += 32)
            acc += (double)g[(long long)j * sb.rank + l] * u[(long long)wrap(s - dl[j], sb.LH) * sb.ns + j];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if (lane == 0) a.ring[sb.ring + (long long)wrap(s, sb.L) * sb.rank + l] = acc;
}

// ---- transient (App. B.3)

// One warp per (transient block, rank index), all steps of the block of steps: the lanes take the
// taps m = lane, lane + 32, ...; the B + 31 values of Y that 32 taps of B steps need are staged in
// shared memory (one load of Y per tap and block instead of one per tap and step).
constexpr int kTrWarps = 4;

template <class T, int B>
__global__ void __launch_bounds__(32 * kTrWarps) trconv_kernel(StepArgs<T> a0) {
    __shared__ double ys[kTrWarps][B + 32];
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = blockIdx.x * kTrWarps + warp;
    if (w >= a.n_tr) return;   // warp-uniform
    const int n = step_index(a), nb = a.nb;
    const SbDev& sb = a.sbs[a.tr_sb[w]];
    const int l = a.tr_l[w], rank = sb.rank, L = sb.L;
    const int t0 = n - sb.mindm;
    const double* Y = a.ring + sb.ring + l;
    if (!FDPH_IDX(sb.ring + (long long)L * rank <= a.len_ring && l < rank &&
                      sb.zring + (long long)sb.LZ * rank <= a.len_zring &&
                      (!(sb.soe + sb.qn) || sb.ustate + (long long)rank * (sb.soe + sb.qn) <= a.len_ustate), a.err))
        return;
    auto y_at = [&](int t) { return Y[(long long)wrap(t, L) * rank]; };
    double z[B];
#pragma unroll
    for (int b = 0; b < B; ++b) z[b] = 0.0;
    const int su = sb.soe + sb.qn;   // states of one rank index: exponential tail, then running sums
    if (sb.qn) {
        // quantized taps (App. A): z = sum_q hhat_q Yhat_q, Yhat_q(t) = Yhat_q(t - 1) + Y(t - b_q)
        // - Y(t - b_q+1) (Eq. A.4), the running window sums kept in the block's states
        for (int q = lane; q < sb.qn; q += 32) {
            const int b0 = a.ints[sb.qb + q], b1 = a.ints[sb.qb + q + 1];
            double* u = a.ustate + sb.ustate + (long long)l * su + sb.soe + q;
            const double hq = (double)a.fac[sb.h + q];
            double y = *u;
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (b < nb) {
                    y = y + y_at(t0 + b - b0) - y_at(t0 + b - b1);
                    z[b] = fma(hq, y, z[b]);
                }
            *u = y;
        }
    } else {
        for (int m0 = 0; m0 < sb.taps; m0 += 32) {
            // ys[x] = Y(t0 + B - 1 - m0 - x)
            for (int x = lane; x < B + 31; x += 32) {
                const int t = t0 + B - 1 - m0 - x;
                ys[warp][x] = t <= t0 + nb - 1 && t > t0 - sb.taps ? y_at(t) : 0.0;
            }
            __syncwarp();
            if (m0 + lane < sb.taps) {
                const double hm = wide(a.fac[sb.h + m0 + lane]);
#pragma unroll
                for (int b = 0; b < B; ++b) z[b] = fma(hm, ys[warp][B - 1 - b + lane], z[b]);
            }
            __syncwarp();
        }
    }
    if (lane < sb.soe) {
        // tail beyond the exact taps: U_q(t) = rho_q U_q(t - 1) + Y(t - taps), z += c_q U_q(t)
        double* u = a.ustate + sb.ustate + (long long)l * su + lane;
        const double rho = a.rho[lane], c = a.trcoef[sb.trc + lane];
        double un = *u;
#pragma unroll
        for (int b = 0; b < B; ++b)
            if (b < nb) {
                un = fma(rho, un, y_at(t0 + b - sb.taps));
                z[b] = fma(c, un, z[b]);
            }
        *u = un;
    }
    __syncwarp();
    const double s = warp_columns<B>(z, lane);
    const int b = sum_col<B>(lane);
    if ((B == 1 ? lane == 0 : !(lane & 1)) && b < nb)
        a.zring[sb.zring + (long long)wrap(t0 + b, sb.LZ) * rank + l] = s;
}

// ---- Eq. 39

// One warp per receiver: its entries (one per far block that contains it) are dealt over the lanes,
// each lane holding the B steps' sums; the B ring rows of an entry are consecutive.
template <class T, int B>
__global__ void __launch_bounds__(128) far_kernel(StepArgs<T> a0) {
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (p >= a.N) return;   // warp-uniform
    const int n = step_index(a);
    double acc[B];
#pragma unroll
    for (int b = 0; b < B; ++b) acc[b] = 0.0;
    const int e1 = a.g_ptr[p + 1];
    for (int e = a.g_ptr[p] + lane; e < e1; e += 32) {
        if (!FDPH_IDX(e < a.n_ent, a.err)) break;
        const FarEnt en = a.ents[e];
        const bool tr = en.flags & 1;
        const double* ring = (tr ? a.zring : a.ring) + en.base;
        if (!FDPH_IDX(en.base + (long long)en.L * en.rank <= (tr ? a.len_zring : a.len_ring), a.err)) continue;
        const int slot = wrap(n - en.dm, en.L);
        const double ph = a.ent_phi ? a.ent_phi[e] : 0.0;
        const bool id = en.flags & 2;
        const int l0 = id ? (int)en.f : 0, l1 = id ? l0 + 1 : en.rank;
        for (int l = l0; l < l1; ++l) {
            const double f = id ? 1.0 : wide(a.fac[en.f + l]);
#pragma unroll
            for (int b = 0; b < B; ++b) {
                int s = slot + b;   // L >= kBlk: one wrap at most
                s -= s >= en.L ? en.L : 0;
                double v = ring[(long long)s * en.rank + l];
                if (a.ent_phi) {    // exact delay dm_i + phi_i: linear interpolation with the next older step
                    const int so = s ? s - 1 : en.L - 1;
                    v = fma(ph, ring[(long long)so * en.rank + l], (1.0 - ph) * v);
                }
                acc[b] = fma(f, v, acc[b]);
            }
        }
    }
    const double s = warp_columns<B>(acc, lane);
    const int b = sum_col<B>(lane);
    if ((B == 1 ? lane == 0 : !(lane & 1)) && b < a.nb) a.tfar[(size_t)b * a.N + p] = s;
}

// ---- the steps' output: far-field traction + the receiver's near-field partial sums, 8 lanes per
// receiver, written in the caller's element order (or, for a rupture block, in internal order);
// grid (receivers, right-hand side, step)
template <class T>
__global__ void gather_kernel(StepArgs<T> a0) {
    const StepArgs<T> a = rhs_args(a0, blockIdx.y);
    const int b = blockIdx.z;
    const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, q = threadIdx.x & 7;
    double s = 0.0;
    if (p < a.N) {
        const double* part = a.partial + b * a.cap_partial;
        const int e1 = a.np_ptr[p + 1];
        for (int e = a.np_ptr[p] + q; e < e1; e += 8)
            if (FDPH_IDX(a.np_idx[e] < a.cap_partial, a.err)) s += part[a.np_idx[e]];
    }
#pragma unroll
    for (int o = 4; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (p >= a.N || q) return;
    s += a.tfar[(size_t)b * a.N + p];
    if (a.thist) {
        a.thist[(size_t)b * a.N + p] = s;
    } else {
        const int n = step_index(a);
        a.T_out[io_offset(a, n) + b * a.io_stride + a.perm[p]] = s;
    }
}

// ---- near field (App. E) on the CUDA cores: FP64 and FP32 items, FP16 windows of one right-hand side (several:
// tensor.cuh)

// Near-field storage: window slices in H; aux slices (static tile, tail coefficients) in the aux
// type (FP32 when the window is FP16: the static term multiplies the cumulative slip, so its
// coefficients keep FP32); slip-rate rows and products in the row type.
template <class H> struct NearTypes { using Aux = H; using Row = H; };
template <> struct NearTypes<__half> { using Aux = float; using Row = float; };

// 16 bytes of stored coefficients as values of the row type
__device__ __forceinline__ void unpack(const uint4& x, float (&v)[4], float) {
    v[0] = __uint_as_float(x.x);
    v[1] = __uint_as_float(x.y);
    v[2] = __uint_as_float(x.z);
    v[3] = __uint_as_float(x.w);
}
__device__ __forceinline__ void unpack(const uint4& x, double (&v)[2], double) {
    v[0] = __hiloint2double((int)x.y, (int)x.x);
    v[1] = __hiloint2double((int)x.w, (int)x.z);
}
__device__ __forceinline__ void unpack(const uint4& x, float (&v)[8], __half) {
    const unsigned u[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&u[q]));
        v[2 * q] = f.x;
        v[2 * q + 1] = f.y;
    }
}

// V consecutive entries of a shared-memory row (16-byte aligned)
template <int V>
__device__ __forceinline__ void load_row(const float* p, float (&v)[V]) {
#pragma unroll
    for (int q = 0; q < V / 4; ++q) {
        const float4 f = ((const float4*)p)[q];
        v[4 * q] = f.x;
        v[4 * q + 1] = f.y;
        v[4 * q + 2] = f.z;
        v[4 * q + 3] = f.w;
    }
}
template <int V>
__device__ __forceinline__ void load_row(const double* p, double (&v)[V]) {
    const double2 f = *(const double2*)p;
    v[0] = f.x;
    v[1] = f.y;
}

static const int kNearWarps = 4;   // work items (warps) of a near-field CTA

template <class H, int B>
struct NearCfg {
    using R = typename NearTypes<H>::Row;
    static constexpr int G = 4;                                       // window slices taken together
    static constexpr int pitch = 36;                                  // row of 32 entries, padded
    // shared memory of one warp: the rows of a window item of `chunk` slices and, past 16 slices, its sums so
    // far (FP64), or an aux item's slip rates (FP64) and one row of B steps for each of its lane groups' slices
    static constexpr size_t warp_bytes(int chunk) {
        const size_t rows = (size_t)((chunk + G - 1) / G * G + B - 1) * pitch * sizeof(R);
        const size_t win = (rows + 15) / 16 * 16 + (chunk > 16 && sizeof(R) == 4 ? (size_t)B * 32 * 8 : 0);
        const size_t aux = (size_t)B * 32 * 8 + (size_t)B * 64 * sizeof(R);
        return ((win > aux ? win : aux) + 15) / 16 * 16;
    }
};

// One warp per work item and right-hand side; lane i = receiver i, coefficients read straight from
// memory (each is used by one lane only), 16 bytes a lane.  Where the steps of a block share the
// coefficients, the products bound the kernel, so what counts is how often the slip-rate rows are
// read: window slice k of step n + b takes the row of step n + b - k, so the G slices of a group
// meet only B + G - 1 rows, each read once (a broadcast) for up to G products.
// Sums in the row type: V sources of a slice, those of two slices over all sources, the two pairs of a group, up
// to four groups; then FP64.  (A uniform slip rate cancels over the sources of a slice, not over the lags of a
// source.  With V sources x 4 slices of a load in one sum the FP32 march of N = 300 without approximation was
// 3.0e-7 off; this way it is 2.1e-7, and curved N = 4096 takes 2.23 instead of 2.17 ms per 64 steps.  One sum a
// slice: 1.9e-7, but 64 sums in registers, 2.43 ms.)  FP64: the even and the odd sources of a slice, slice by
// slice, over the item.
// FP64 plans are bound by the FP64 pipe (two multiply-adds a clock and SM; curved N = 1500 4.91 ms per 32 steps, plain march of
// N = 256 2.59 ms).  Exact products of 62-bit fixed-point numbers on the FP16 tensor cores took 1.11 and
// 0.51 ms, but cut off what lies below 2^-61 of a leaf's largest coefficient or slip rate: where only quiet
// sources of a leaf have arrived, a slip rate at 1e-12 of the largest was good to 3e-7.
// Leaves of at most 16 receivers split the warp into 32 / span lane groups that take slices (window)
// or aux slices of their own.
template <class T, class H, int B>
__global__ void __launch_bounds__(32 * kNearWarps, B == 1 ? 6 : sizeof(H) == 8 ? 3 : 4) near_block_kernel(StepArgs<T> a, int warp_bytes) {
    using C = NearCfg<H, B>;
    using R = typename C::R;
    using A = typename NearTypes<H>::Aux;
    constexpr int G = C::G, P = C::pitch;
    extern __shared__ __align__(16) unsigned char near_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * kNearWarps + warp;
    const int it = (int)(w / a.nrhs), rh = (int)(w % a.nrhs);
    if (it >= a.n_items) return;   // warp-uniform
    const NearTask tk = a.tasks[it];
    const int n = step_index(a), nb = a.nb;
    const int hend = hist_end(a, n);
    const int nr = tk.nr, ns = tk.ns;
    unsigned char* mem = near_smem + (size_t)warp * warp_bytes;
    double tot[B];
#pragma unroll
    for (int b = 0; b < B; ++b) tot[b] = 0.0;
    int span = 32;
    if (!tk.kind) {
        while (span > 1 && span / 2 >= nr) span >>= 1;
        const int ngrp = 32 / span, grp = lane / span, ri = lane - grp * span;
        const int li = ri < nr ? ri : 0;   // lanes past nr read a valid element, unused
        const int nk = tk.k1 - tk.k0;
        constexpr int V = 16 / (int)sizeof(H);
        const int nbk = (ns + V - 1) / V, ngr = (nk + G - 1) / G;
        const H* base = (const H*)a.tensor + tk.off + (size_t)li * V;
        const bool in = FDPH_IDX(tk.off + (long long)nk * tk.sl <= a.len_tensor, a.err);
        // a group's 16-byte coefficient vectors of source group jb; slices past the item are zero
        auto load = [&](int gr, int jb, uint4 (&x)[G]) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int k = gr * G + g;
                x[g] = k < nk && in ? __ldcs((const uint4*)(base + (size_t)k * tk.sl + (size_t)jb * nr * V))
                                    : make_uint4(0, 0, 0, 0);
            }
        };
        if (tk.k0 < n + nb) {   // (otherwise the item's window lies before the march)
            R* rows = (R*)mem;
            uint4 xn[G];
            if constexpr (sizeof(R) == 4 || B == 1) load(grp, 0, xn);
            // row q: slip rates of step n + B - 1 - k0 - q (zero before the march, past the steps that
            // the launch may use, and past the item's window)
            {
                const R* ring;
                if constexpr (sizeof(R) == 4) ring = a.Dring32; else ring = a.Dring;
                ring += rh * a.rs_D + tk.s0 + (lane < ns ? lane : 0);
                const int top = n + B - 1 - tk.k0, nrow = ngr * G + B - 1;
                int slot = wrap(top, a.WD);
#pragma unroll 8
                for (int q = 0; q < nrow; ++q) {
                    const int t = top - q;
                    const bool ok = t >= 0 && t < hend && q < nk + B - 1 && lane < ns;
                    rows[q * P + lane] = ok ? ring[(size_t)slot * a.N] : (R)0;
                    slot = slot ? slot - 1 : a.WD - 1;
                }
            }
            __syncwarp();
            R acc[B];
#pragma unroll
            for (int b = 0; b < B; ++b) acc[b] = 0;
            const int iters = (ngr + ngrp - 1) / ngrp;
            if constexpr (sizeof(R) == 8) {
                for (int i = 0; i < iters; ++i) {
                    const int gr = i * ngrp + grp, left = nk - gr * G;   // slices from the group's first on
                    const R* rg = rows + (size_t)min(gr, ngr - 1) * G * P;
                    if constexpr (B == 1) {   // (bound by memory: the group's loads in flight together)
                        R s[G][2];
#pragma unroll
                        for (int g = 0; g < G; ++g) s[g][0] = s[g][1] = 0;
                        for (int jb = 0; jb < nbk; ++jb) {
                            R x[G][V];
#pragma unroll
                            for (int g = 0; g < G; ++g) unpack(xn[g], x[g], R());
                            const bool wrapj = jb + 1 == nbk;
                            load(wrapj ? gr + ngrp : gr, wrapj ? 0 : jb + 1, xn);
#pragma unroll
                            for (int g = 0; g < G; ++g) {
                                R y[V];
                                load_row<V>(rg + g * P + jb * V, y);
#pragma unroll
                                for (int v = 0; v < 2; ++v) s[g][v] = fma(x[g][v], y[v], s[g][v]);
                            }
                        }
#pragma unroll
                        for (int g = 0; g < G; ++g)
                            if (g < left) acc[0] += s[g][0] + s[g][1];
                    } else {
#pragma unroll 1
                        for (int g = 0; g < min(G, left); ++g) {
                            const uint4* c = (const uint4*)(base + (size_t)(gr * G + g) * tk.sl);
                            uint4 xv = in ? __ldcs(c) : make_uint4(0, 0, 0, 0);
                            R s[2][B];
#pragma unroll
                            for (int b = 0; b < B; ++b) s[0][b] = s[1][b] = 0;
                            for (int jb = 0; jb < nbk; ++jb) {
                                R x[V];
                                unpack(xv, x, R());
                                if (jb + 1 < nbk && in) xv = __ldcs(c + (size_t)(jb + 1) * nr);
#pragma unroll
                                for (int b = 0; b < B; ++b) {
                                    if (b >= nb) break;   // (the launch's steps only: the FP64 pipe bounds)
                                    R y[V];
                                    load_row<V>(rg + (B - 1 - b + g) * P + jb * V, y);
#pragma unroll
                                    for (int v = 0; v < 2; ++v) s[v][b] = fma(x[v], y[v], s[v][b]);
                                }
                            }
#pragma unroll
                            for (int b = 0; b < B; ++b) acc[b] += s[0][b] + s[1][b];
                        }
                    }
                }
#pragma unroll
                for (int b = 0; b < B; ++b) tot[b] = acc[b];
            } else {
                double* mid = (double*)(mem + warp_bytes) - B * 32;   // the sums so far, past 16 slices
                const R ks = (R)a.kinv;   // the storage scale of the window (FP16), a power of two
                for (int i = 0; i < iters; ++i) {
                    const int gr = i * ngrp + grp;
                    const R* rg = rows + (size_t)min(gr, ngr - 1) * G * P;
                    R s[2][B];   // sums of two slices each over the sources (see above)
#pragma unroll
                    for (int b = 0; b < B; ++b) s[0][b] = s[1][b] = 0;
                    for (int jb = 0; jb < nbk; ++jb) {
                        R x[G][V];
#pragma unroll
                        for (int g = 0; g < G; ++g) {
                            if constexpr (sizeof(H) == 2) unpack(xn[g], x[g], __half());
                            else unpack(xn[g], x[g], R());
                        }
                        const bool wrapj = jb + 1 == nbk;
                        load(wrapj ? gr + ngrp : gr, wrapj ? 0 : jb + 1, xn);
#pragma unroll
                        for (int q = 0; q < B + G - 1; ++q) {
                            R y[V];
                            load_row<V>(rg + q * P + jb * V, y);
#pragma unroll
                            for (int g = 0; g < G; ++g) {
                                const int b = B - 1 - q + g;
                                if (b >= 0 && b < B) {
                                    constexpr int U = V < 4 ? V : 4;
                                    R t = x[g][0] * y[0];
#pragma unroll
                                    for (int v = 1; v < U; ++v) t = fma(x[g][v], y[v], t);
                                    if constexpr (V == 8) {
                                        R u = x[g][4] * y[4];
#pragma unroll
                                        for (int v = 5; v < V; ++v) u = fma(x[g][v], y[v], u);
                                        t += u;
                                    }
                                    s[g / 2][b] += t;
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int b = 0; b < B; ++b) acc[b] += s[0][b] + s[1][b];
                    if ((i & 3) == 3 && i + 1 < iters) {
#pragma unroll
                        for (int b = 0; b < B; ++b) {
                            const double v = wide(acc[b] * ks);
                            mid[b * 32 + lane] = i > 3 ? mid[b * 32 + lane] + v : v;
                            acc[b] = 0;
                        }
                    }
                }
#pragma unroll
                for (int b = 0; b < B; ++b) tot[b] = wide(acc[b] * ks) + (iters > 4 ? mid[b * 32 + lane] : 0.0);
            }
        }
    } else if constexpr (sizeof(H) != 2 || B == 1) {   // (those of a block of FP16 plans go to the FP32 instance)
        // aux slices: slice 0 the static tile (times C_j(n - W), it carries dt), slice 1 + q the tail
        // coefficients of term q (times the tail state V_qj(n) = rho_q V_qj(n - 1) + D_{j, n-W}, updated
        // here by its only reader).  Lane j of a lane group forms its slice's rows of the B steps.
        const int m = nr > ns ? nr : ns;
        while (span > 4 && span / 2 >= m) span >>= 1;
        const int ngrp = 32 / span, grp = lane / span, ri = lane - grp * span;
        const int li = ri < nr ? ri : 0;
        constexpr int V = 16 / (int)sizeof(A);
        const int nbk = (ns + V - 1) / V;
        const int na = tk.k1 - tk.k0;
        const bool src = ri < ns;
        const size_t col = (size_t)tk.s0 + (src ? ri : 0);
        double* dw = (double*)mem;                                     // [B][32] slip rates D(n + b - W)
        R* vr = (R*)(dw + B * 32) + (size_t)grp * B * (span + 4);      // [B][span + 4] rows of the group's slice
        const int t0 = n - tk.W;
        const bool fixed = a.hist != HIST_BASE || tk.W >= kBlk;   // (else rup_step_kernel takes the static term)
        const double* Dr = a.Dring + rh * a.rs_D + col;
        const double* Cr = a.Cring + rh * a.rs_C + col;
        double* vs = a.vstate + rh * a.len_vstate + tk.vstate + (src ? ri : 0);
        const bool in = FDPH_IDX(tk.off + (long long)na * tk.sl <= a.len_aux &&
                                     (tk.k1 <= 1 || tk.vstate + (long long)(tk.k1 - 1) * ns <= a.len_vstate),
                                 a.err);
        if (tk.k1 > 1 && grp == 0) {
#pragma unroll
            for (int b = 0; b < B; ++b)
                dw[b * 32 + ri] = b < nb && src && t0 + b >= 0 ? Dr[(size_t)wrap(t0 + b, a.WD) * a.N] : 0.0;
        }
        __syncwarp();
        const A* base = (const A*)a.stat + tk.off + (size_t)li * V;
        for (int i = 0; i < na; i += ngrp) {
            const int ai = tk.k0 + i + grp;
            const bool on = ai < tk.k1 && in;
            if (on && ai == 0) {
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const int t = min(t0 + b, hend - 1);   // (the slip by the steps that the launch may use)
                    vr[b * (span + 4) + ri] = narrow(b < nb && src && fixed && t >= 0 ? Cr[(size_t)wrap(t, a.WC) * a.N] : 0.0, R());
                }
            } else if (on) {
                const double rho = a.rho[ai - 1];
                double v = src ? vs[(size_t)(ai - 1) * ns] : 0.0;
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    if (b < nb) v = fma(rho, v, dw[b * 32 + ri]);
                    vr[b * (span + 4) + ri] = narrow(src && b < nb ? v : 0.0, R());
                }
                if (src) vs[(size_t)(ai - 1) * ns] = v;
            }
            __syncwarp();
            if (on) {
                const A* sl = base + (size_t)(i + grp) * tk.sl;
                R t[B];
#pragma unroll
                for (int b = 0; b < B; ++b) t[b] = 0;
#pragma unroll 2
                for (int jb = 0; jb < nbk; ++jb) {
                    R x[V];
                    unpack(__ldcs((const uint4*)(sl + (size_t)jb * nr * V)), x, R());
#pragma unroll
                    for (int b = 0; b < B; ++b) {
                        R y[V];
                        load_row<V>(vr + b * (span + 4) + jb * V, y);
                        R s = x[0] * y[0];
#pragma unroll
                        for (int v = 1; v < V; ++v) s = fma(x[v], y[v], s);
                        t[b] += s;
                    }
                }
                // FP64 across slices
#pragma unroll
                for (int b = 0; b < B; ++b) tot[b] += wide(t[b]);
            }
            __syncwarp();
        }
    }
    for (int o = span; o < 32; o <<= 1) {
#pragma unroll
        for (int b = 0; b < B; ++b) tot[b] += __shfl_xor_sync(0xffffffffu, tot[b], o);
    }
    if (lane < nr && FDPH_IDX((long long)tk.item * 32 + 32 <= a.cap_partial, a.err)) {
        double* out = a.partial + rh * a.rs_partial + (size_t)tk.item * 32 + lane;
#pragma unroll
        for (int b = 0; b < B; ++b)
            if (b < nb) out[b * a.cap_partial] = tot[b];
    }
}

// ---- rupture (Sec. 6.2)

// Friction law of a plan.  In device memory, like tau0: a captured graph of rupture steps replays the law
// that fdph_rupture_init last wrote, not the one it was captured with.
struct FrictionLaw {
    double sigma_n, mu_s, mu_d, Dc;
    int law;               // 0: linear slip weakening, 1: exponential (Sec. 6.2)
};

// Local friction solve (geometry order).
struct FrictionDev {
    const FrictionLaw* law;
    const double* tau0;
    const double* k0;      // instantaneous self coefficient K_{ii,0} (< 0)
    double* slip;
    double dt;
};

// One step of a rupture block.  The traction of step n with D_n = 0 is thist (everything that the
// slip rates before the step's aligned block [n0, n0 + kBlk) do, computed for the whole block
// beforehand) plus what the block's own earlier steps n0 ... n - 1 do: by causality only the kernel
// steps 1 ... n - n0 of the near leaves that a wave crosses that fast (RecLeaf: the first kz kernel
// steps of a leaf vanish), and the static term of leaves with a window shorter than a block, whole, on the
// slip C(n - W) (the far blocks and the other static and tail terms act later than kBlk steps, see
// rup_block; a share of it on the slip before the block would need C(n0 - 1), which neither the ring nor a
// saved state holds where all windows are short).  One CTA per receiver group (the disjoint maximal receiver clusters of those leaves): its
// warps take the (leaf, kernel step) units in turn, then the first warp solves the friction law and
// appends the slip rate (push).  b: the step within the launch sequence's block.
//
// The steps of a block follow one another, so the kernel's latency bounds a rupture.  It is launched
// while the step before is still running (programmatic dependent launch): what does not depend on that
// step (unit lists, the first unit's coefficients, prestress and history traction) is loaded before
// the wait.
static const int kRupThreads = 512;
static const int kRupLeaves = 32;    // leaves of a group kept in shared memory

template <class T, class H>
__global__ void __launch_bounds__(kRupThreads, sizeof(H) == 8 ? 1 : 2) rup_step_kernel(StepArgs<T> a, FrictionDev f, double* D, int b, int recent) {
    using R = typename NearTypes<H>::Row;
    constexpr int V = 16 / (int)sizeof(H), W = kRupThreads / 32;
    constexpr int NB = 32 / V;                            // 16-byte vectors of a slice per receiver
    __shared__ __align__(16) R row[W][2][36];
    __shared__ double red[W][32];
    __shared__ RecLeaf leaves[kRupLeaves];
    __shared__ FrictionLaw law;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const RecGroup g = a.rec_groups[blockIdx.x];
    const int nf = step_index(a), n = nf + b;
    const int back = recent ? n - (n & ~(kBlk - 1)) : 0;   // the block's earlier steps
    red[warp][lane] = 0.0;
    {
        constexpr int words = (int)(sizeof(RecLeaf) / 16);
        const int m = min(g.nleaf, kRupLeaves) * words;
        for (int q = threadIdx.x; q < m; q += kRupThreads) ((int4*)leaves)[q] = ((const int4*)(a.rec_leaves + g.leaf0))[q];
    }
    if (threadIdx.x == 32) law = *f.law;
    // the first warp's element
    const bool mine = warp == 0 && lane < g.nr;
    const int p = g.r0 + lane, e = mine ? a.perm[p] : 0;
    double T0 = 0.0, tau0 = 0.0, k0 = -1.0;
    if (mine) {
        T0 = a.thist[(size_t)b * a.N + p];
        tau0 = f.tau0[e];
        k0 = f.k0[e];
    }
    __syncthreads();
    auto leaf = [&](int q) -> const RecLeaf& { return q < kRupLeaves ? leaves[q] : a.rec_leaves[g.leaf0 + q]; };
    // units of a leaf: its kernel steps first, first + 1, ..., then (kernel step -1) its static term
    auto range = [&](const RecLeaf& L, int& first, int& steps) {
        first = max(L.kz, 1);
        steps = max(min(back + 1, L.W) - first, 0);
        return steps + (L.stat >= 0 && recent ? 1 : 0);
    };
    // the unit with running number r from leaf q on: its leaf (nleaf: none) and kernel step
    auto seek = [&](int& q, int r, int& k) {
        for (; q < g.nleaf; ++q) {
            int first, steps;
            const int len = range(leaf(q), first, steps);
            if (r < len) {
                k = r < steps ? first + r : -1;
                return;
            }
            r -= len;
        }
    };
    using A = typename NearTypes<H>::Aux;
    constexpr int VA = 16 / (int)sizeof(A);
    auto load_x = [&](const RecLeaf& L, int k, uint4 (&x)[NB]) {
        if (k < 0) return;   // (a static tile is read where it is used)
        const H* sl = (const H*)a.tensor + L.off + (size_t)k * L.sl + (size_t)(lane < L.nr ? lane : 0) * V;
        const bool in = FDPH_IDX(L.off + (long long)(k + 1) * L.sl <= a.len_tensor, a.err);
#pragma unroll
        for (int jb = 0; jb < NB; ++jb)
            x[jb] = in && jb * V < L.ns ? *(const uint4*)(sl + (size_t)jb * L.nr * V) : make_uint4(0, 0, 0, 0);
    };
    auto load_v = [&](const RecLeaf& L, int k) -> R {
        const int c = L.s0 + min(lane, L.ns - 1);
        R v;
        if (k < 0) {   // the slip of the steps up to n - W
            const int t = min(n - L.W, n - 1);
            v = narrow(t >= 0 ? a.Cring[(size_t)wrap(t, a.WC) * a.N + c] : 0.0, R());
        } else {
            const size_t off = (size_t)wrap(n - k, a.WD) * a.N + c;
            if constexpr (sizeof(R) == 4) v = a.Dring32[off]; else v = a.Dring[off];
        }
        return lane < L.ns ? v : (R)0;
    };
    int q = 0, k = 0;
    uint4 x[NB];
    seek(q, warp, k);
    if (q < g.nleaf) load_x(leaf(q), k, x);
    cudaGridDependencySynchronize();                 // the step before is complete
    cudaTriggerProgrammaticLaunchCompletion();
    double u = 0.0, c = 0.0, comp = 0.0;
    if (mine) {
        u = f.slip[e];
        c = a.C[p];
        comp = a.Ccomp[p];
    }
    R v = q < g.nleaf ? load_v(leaf(q), k) : (R)0;
    for (int buf = 0; q < g.nleaf; buf ^= 1) {
        row[warp][buf][lane] = v;
        __syncwarp();
        const RecLeaf& L = leaf(q);
        const int ns = L.ns, nr = L.nr, r0 = L.r0 - g.r0;
        R s = 0;
        const bool fixed = k < 0;
        if (fixed) {
            const A* sl = (const A*)a.stat + L.stat + (size_t)(lane < nr ? lane : 0) * VA;
            const bool in = FDPH_IDX(L.stat + (long long)((ns + VA - 1) / VA) * VA * nr <= a.len_aux, a.err);
            for (int jb = 0; jb * VA < ns && in; ++jb) {
                R xv[VA], y[VA];
                unpack(*(const uint4*)(sl + (size_t)jb * nr * VA), xv, R());
                load_row<VA>(&row[warp][buf][jb * VA], y);
#pragma unroll
                for (int i = 0; i < VA; ++i) s = fma(xv[i], y[i], s);
            }
        }
        // the unit W further: its slip rates are loaded meanwhile, its coefficients next
        {
            int first, steps;
            range(L, first, steps);
            seek(q, (fixed ? steps : k - first) + W, k);
        }
        if (q < g.nleaf) v = load_v(leaf(q), k);
        if (!fixed) {
#pragma unroll
            for (int jb = 0; jb < NB; ++jb) {
                if (jb * V >= ns) break;
                R xv[V], y[V];
                if constexpr (sizeof(H) == 2) unpack(x[jb], xv, __half());
                else unpack(x[jb], xv, R());
                load_row<V>(&row[warp][buf][jb * V], y);
                R t = xv[0] * y[0];
#pragma unroll
                for (int i = 1; i < V; ++i) t = fma(xv[i], y[i], t);
                s += t;
            }
            s *= (R)a.kinv;   // (the window's storage scale, a power of two)
        }
        if (q < g.nleaf) load_x(leaf(q), k, x);
        if (lane < nr && FDPH_IDX(r0 >= 0 && r0 + nr <= 32, a.err)) red[warp][r0 + lane] += wide(s);
        __syncwarp();
    }
    __syncthreads();
    if (!mine) return;
    {
        double t[W];
#pragma unroll
        for (int w = 0; w < W; ++w) t[w] = red[w][lane];
#pragma unroll
        for (int h = W / 2; h; h >>= 1)
#pragma unroll
            for (int w = 0; w < h; ++w) t[w] += t[w + h];
        T0 += t[0];
    }
    const long long off = io_offset(a, nf) + (long long)b * a.io_stride + e;
    const double tau = tau0 + T0;
    double strength;
    if (law.law == 1) {
        strength = law.sigma_n * (law.mu_d + (law.mu_s - law.mu_d) * exp(-u / law.Dc));
    } else {
        const double w = u < law.Dc ? u / law.Dc : 1.0;
        strength = law.sigma_n * (law.mu_s - (law.mu_s - law.mu_d) * w);
    }
    const double eta = -k0;
    const double d = tau > strength ? (tau - strength) / eta : 0.0;
    push_one(a, p, n, b, d, c, comp);
    D[off] = d;
    a.T_out[off] = tau + k0 * d;
    f.slip[e] = u + d * f.dt;
    a.C[p] = c;
    a.Ccomp[p] = comp;
}
