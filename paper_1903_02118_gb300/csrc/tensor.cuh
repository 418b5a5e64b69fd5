// tensor.cuh -- the near-field windows of FP16 plans with several right-hand sides on the tensor cores.
//
// One window slice is a 32 x 32 (receivers x sources) FP16 tile; with the R right-hand sides and the B
// steps of a launch it meets R B slip-rate rows: a dense (32 x 32) x (32 x R B) contraction, run as
// warp-level mma.sync m16n8k16 (FP16 inputs, FP32 accumulation).  tcgen05 tiles start at 64 rows (128 at
// full rate) that share their B operand; a slice has 32 receivers, and the leaves that share its sources
// have other windows, so the warp form is the one that fits (measured: 1034 multiply-adds a clock and SM).
//
// Neither operand is copied: the order of the 32 sources inside the contraction is free as long as both
// operands use the same one, and with source 8 t + 4 s + 2 h + {0, 1} at position (step s, half h) of
// lane t, the A fragments of lane (g, t) are exactly the stored 16 bytes (sources 8 t ... 8 t + 7 of one
// receiver, plan.h), and the B fragments of both 16-source steps are 16 contiguous bytes of a row.
//
// The slip rates go in with more digits than FP16 has: the 32 sources of a row (step, right-hand side) are split
// into two FP16 rows of x 2^sh (sh puts the largest of them in [2^13, 2^14); hi = fp16(x 2^sh), lo =
// fp16(x 2^sh - hi)), separate columns of the contraction.  A slip rate keeps 2^-22 of itself, but no less than 2^-39
// of the largest of the leaf's 32 sources: one at 1e-6 of it is good to 2e-6.  Each slice's products are scaled
// back per column by 2^-sh and added to the item's FP32 sums.  (The scale is of the leaf's own sources, found by
// the warp that stages them: one scale for a whole step's slip rates took a kernel between the push and the
// near field and lost digits where a leaf is quiet.)
#pragma once
#include "step.cuh"

// the shift sh = 14 - e that takes a row's largest |x| = f 2^e, f in [0.5, 1), to [2^13, 2^14) (e from the
// exponent field; 2^sh and 2^-sh stay normal numbers)
__device__ __forceinline__ int row_shift(unsigned m) { return min(max(14 - ((int)(m >> 23) - 126), -115), 126); }

// 2^k as a float, k in [-126, 127]
__device__ __forceinline__ float pow2f(int k) { return __uint_as_float((unsigned)(127 + k) << 23); }

__device__ __forceinline__ void mma_16816(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                          unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// c = A B: the first MMA of a sum
__device__ __forceinline__ void mma_16816_first(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                                unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// NR right-hand sides, a block of steps.  Rows in shared memory: row q of the item holds the slip
// rates of step n + S - 1 - k0 - q, S = kBlk, [q][part][right-hand side][32 sources] with
// the parts hi, lo; 8 consecutive rows are the columns of one MMA tile, so window slice k takes the tiles from
// row k - k0 on (tile = one step of 8 right-hand sides' hi or lo, of 4 with both, 2 steps of 2).
//
// Warps take 16 receivers and a share of the tiles each, and all slices of the item: the item's sums stay in
// the accumulators and are written straight out, and 16 steps of 8 right-hand sides take one pass over the
// coefficients.  With a share of the slices per warp the sums of the four warps met in shared memory and FP64
// at the end of every item, and two passes were needed: eight right-hand sides, N = 6000, 3.86 -> 3.23 ms per
// 16 steps (near field 67 us a step); four, N = 2500, 1.69 -> 1.35 ms per 32.  Bound by latency and issue slots,
// not by the tensor pipe: a slice is two 16-byte loads, then two (four) dependent MMAs and four FMAs a tile.
//
// The FP32 sum of a slice's products goes into a sum over kSum slices, that into a sum over the item.  (Against exact
// sums of the stored coefficients, plain march of N = 300, noise, four right-hand sides: one sum over the item
// 1.35e-7, kSum = 16, 8, 4: 1.18, 1.10, 1.10e-7.  Parts that meet in FP64 in the item's partial sum take four right-hand
// sides of N = 2500 from 1.36 to 1.53 ms.)
static const int kSum = 8;

template <int NR>
struct TcCfg {
    static constexpr int C = 2 * NR;                          // columns of one row q
    static constexpr int per = NR == 2 ? 2 : 1;               // steps of one tile
    static constexpr int tiles = kBlk / per;                  // accumulator tiles (hi and lo of 8 share one)
    static constexpr int warps = 4;
    static constexpr int share = tiles / 2;                   // tiles of a warp at most
    static constexpr int rows(int chunk) { return chunk + kBlk - 1; }
    static constexpr size_t row_bytes(int chunk) { return (size_t)rows(chunk) * C * 64; }
    // rows and their scales
    static constexpr size_t smem(int chunk) { return row_bytes(chunk) + (size_t)rows(chunk) * C * 4; }
};

template <int NR>
__global__ void __launch_bounds__(32 * TcCfg<NR>::warps, 4) tc_block_kernel(StepArgs<float> a, int chunk) {
    using Cf = TcCfg<NR>;
    constexpr int C = Cf::C, S = kBlk, NW = Cf::warps, T = Cf::share;
    extern __shared__ __align__(16) unsigned char tc_smem[];
    const NearTask tk = a.tasks[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = step_index(a), nb = a.nb, nr = tk.nr, ns = tk.ns;
    const int nk = tk.k0 < n + nb ? tk.k1 - tk.k0 : 0;   // (0: the item's window lies before the march)
    const int nrow = nk ? nk + S - 1 : 0;
    __half* rows = (__half*)tc_smem;
    float* scl = (float*)(tc_smem + Cf::row_bytes(chunk));
    {
        const int top = n + S - 1 - tk.k0, hend = hist_end(a, n), stop = wrap(top, a.WD);
        // warps over right-hand sides, then over rows, kAhead of them in flight (row by row the staging, not the
        // MMAs, bounded the kernel)
        constexpr int kAhead = 8, RW = NR < NW ? NR : NW, QW = NW / RW;
        const bool src = lane < ns;
        for (int r = warp % RW; r < NR; r += RW) {
            const float* ring = a.Dring32 + r * a.rs_D + tk.s0 + (src ? lane : 0);
            for (int q0 = warp / RW * kAhead; q0 < nrow; q0 += QW * kAhead) {
                float x[kAhead];
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    const int t = top - q0 - i;
                    int slot = stop - q0 - i;              // nrow <= WD: one wrap at most
                    slot += slot < 0 ? a.WD : 0;
                    const bool ok = q0 + i < nrow && t >= 0 && t < hend;
                    x[i] = ok && src ? ring[(size_t)slot * a.N] : 0.f;
                }
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    if (q0 + i >= nrow) break;
                    const int sh = row_shift(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(x[i]))));
                    const float y = x[i] * pow2f(sh);
                    const __half hi = __float2half_rn(y);
                    const float y1 = fabsf(y) <= 65504.f ? y - __half2float(hi) : 0.f;   // (an infinity has no rest)
                    const __half lo = __float2half_rn(y1);
                    __half* row = rows + (size_t)((q0 + i) * C + r) * 32 + lane;
                    row[0] = hi;
                    row[NR * 32] = lo;
                    if (lane < C / NR) scl[(q0 + i) * C + lane * NR + r] = pow2f(-sh);
                }
            }
        }
    }
    __syncthreads();
    // this warp's receivers 16 mt ... 16 mt + 15 and tiles i0 ... i0 + nt - 1 (leaves of at most 16 receivers
    // have one set of receivers: a quarter of the tiles per warp)
    const bool two = nr > 16;
    const int mt = two ? warp & 1 : 0;
    const int nt = two ? T : T / 2;
    const int i0 = (two ? warp >> 1 : warp) * nt;
    const int g = lane >> 2, t = lane & 3;
    // the 16-byte vectors (sources 8 t ... 8 t + 7) of receivers g and g + 8 of the set
    const __half* base = (const __half*)a.tensor + tk.off + ((size_t)t * nr + 16 * mt + g) * 8;
    const bool in = FDPH_IDX(tk.off + (long long)nk * tk.sl <= a.len_tensor, a.err) && 8 * t < ns;
    auto load = [&](int k, uint4 (&x)[2]) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
            x[m] = in && k < nk && 16 * mt + g + 8 * m < nr ? __ldcs((const uint4*)(base + (size_t)k * tk.sl + 64 * m))
                                                             : make_uint4(0, 0, 0, 0);
    };
    float acc[T][4];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[i][f] = 0.f;
    constexpr int D = 2;   // slices in flight
    uint4 xn[D][2];
#pragma unroll
    for (int d = 0; d < D; ++d) load(d, xn[d]);
    constexpr int parts = NR == 8 ? 2 : 1;   // (8 right-hand sides: the hi tile, then the lo tile)
    const __half* rk = rows + ((size_t)i0 * parts * 8 + g) * 32 + 8 * t;
    const float* sk = scl + i0 * parts * 8 + 2 * t;
    float sum[T][4];   // of the parts before this one
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int f = 0; f < 4; ++f) sum[i][f] = 0.f;
    for (int k0 = 0; k0 < nk; k0 += kSum) {
        for (int k = k0; k < min(k0 + kSum, nk); ++k, rk += C * 32, sk += C) {
            const uint4 x0 = xn[0][0], x1 = xn[0][1];
#pragma unroll
            for (int d = 0; d + 1 < D; ++d) {
                xn[d][0] = xn[d + 1][0];
                xn[d][1] = xn[d + 1][1];
            }
            load(k + D, xn[D - 1]);
#pragma unroll
            for (int i = 0; i < T; ++i) {
                if (i >= nt) break;   // (warp-uniform)
                float c[4];
#pragma unroll
                for (int h = 0; h < parts; ++h) {
                    const uint4 b = *(const uint4*)(rk + (size_t)(i * parts + h) * 8 * 32);
                    if (h == 0) mma_16816_first(c, x0.x, x1.x, x0.y, x1.y, b.x, b.y);
                    else mma_16816(c, x0.x, x1.x, x0.y, x1.y, b.x, b.y);
                    mma_16816(c, x0.z, x1.z, x0.w, x1.w, b.z, b.w);
                }
                const float2 s = *(const float2*)(sk + i * parts * 8);
                acc[i][0] = fmaf(c[0], s.x, acc[i][0]);
                acc[i][1] = fmaf(c[1], s.y, acc[i][1]);
                acc[i][2] = fmaf(c[2], s.x, acc[i][2]);
                acc[i][3] = fmaf(c[3], s.y, acc[i][3]);
            }
        }
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                sum[i][f] += acc[i][f];
                acc[i][f] = 0.f;
            }
    }
    const bool fits = FDPH_IDX((long long)tk.item * 32 + 32 <= a.cap_partial, a.err);
    const float ks = a.kinv;   // the window's storage scale (a power of two)
    double* out = a.partial + (size_t)tk.item * 32 + 16 * mt;
#pragma unroll
    for (int i = 0; i < T; ++i) {
        if (i >= nt) break;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            float v = sum[i][f];
            if constexpr (NR == 4) v += __shfl_xor_sync(0xffffffffu, v, 2);   // hi + lo
            if constexpr (NR == 2) v += __shfl_xor_sync(0xffffffffu, v, 1);
            const int col = 2 * t + (f & 1);          // column of the tile
            const int q = Cf::per * (i0 + i) + (NR == 2 ? col >> 2 : 0), r = col % NR, b = S - 1 - q;
            const bool mine = NR == 8 || (NR == 4 ? col < 4 : !(col & 2));
            const int row = g + 8 * (f >> 1);
            if (mine && fits && b < nb && 16 * mt + row < nr) out[r * a.rs_partial + b * a.cap_partial + row] = wide(v * ks);
        }
    }
}

// One step of NR right-hand sides: a slip-rate row meets one slice only, so the lanes split it in registers, each the
// eight sources 8 t ... 8 t + 7 of its column g that are its B fragment.  One warp per item, both sets of receivers;
// the sums of the block kernel, bit for bit.  (The block kernel's way, through shared memory, took 40 instructions a row
// and right-hand side where this takes 10: eight right-hand sides, N = 6000, 479 us against 272 a step; 490 us with the
// rows split once for all leaves that share them, which loses digits where a leaf is quiet.)
static const int kTcStepWarps = 4;

template <int NR>
__global__ void __launch_bounds__(32 * kTcStepWarps, 4) tc_step_kernel(StepArgs<float> a, int n_win) {
    const int it = blockIdx.x * kTcStepWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (it >= n_win) return;   // warp-uniform
    const NearTask tk = a.tasks[it];
    const int n = step_index(a), nr = tk.nr, ns = tk.ns;
    const int nk = tk.k0 <= n ? tk.k1 - tk.k0 : 0;   // (0: the item's window lies before the march)
    const int g = lane >> 2, t = lane & 3;
    const int r = g % NR;                            // column g: right-hand side r,
    const bool low = NR < 8 && g / NR % 2;           // hi or lo (8 right-hand sides: both, one MMA after the other)
    const __half* base = (const __half*)a.tensor + tk.off + ((size_t)t * nr + g) * 8;
    const bool in = FDPH_IDX(tk.off + (long long)nk * tk.sl <= a.len_tensor, a.err) && 8 * t < ns;
    const int top = n - tk.k0, hend = hist_end(a, n), stop = wrap(top, a.WD);
    const float* ring = a.Dring32 + r * a.rs_D + tk.s0 + 8 * t;
    constexpr int D = 2;   // slices in flight
    uint4 xn[D][4];        // receivers g, g + 8, g + 16, g + 24
    float yn[D][8];
    auto load = [&](int k, uint4 (&x)[4], float (&y)[8]) {
#pragma unroll
        for (int m = 0; m < 4; ++m)
            x[m] = in && k < nk && g + 8 * m < nr ? __ldcs((const uint4*)(base + (size_t)k * tk.sl + 64 * m)) : make_uint4(0, 0, 0, 0);
        const int tt = top - k;
        int slot = stop - k;   // nk <= WD: one wrap at most
        slot += slot < 0 ? a.WD : 0;
        const bool ok = k < nk && tt >= 0 && tt < hend;
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = ok && 8 * t + i < ns ? ring[(size_t)slot * a.N + i] : 0.f;
    };
#pragma unroll
    for (int d = 0; d < D; ++d) load(d, xn[d], yn[d]);
    float acc[2][4], sum[2][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[m][f] = sum[m][f] = 0.f;
    for (int k = 0; k < nk; ++k) {
        uint4 x[4];
        float y[8];
#pragma unroll
        for (int m = 0; m < 4; ++m) x[m] = xn[0][m];
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = yn[0][i];
#pragma unroll
        for (int d = 0; d + 1 < D; ++d) {
#pragma unroll
            for (int m = 0; m < 4; ++m) xn[d][m] = xn[d + 1][m];
#pragma unroll
            for (int i = 0; i < 8; ++i) yn[d][i] = yn[d + 1][i];
        }
        load(k + D, xn[D - 1], yn[D - 1]);
        unsigned big = 0;   // the largest of the column's 32 slip rates: those of lanes 4 g ... 4 g + 3
#pragma unroll
        for (int i = 0; i < 8; ++i) big = max(big, __float_as_uint(fabsf(y[i])));
        big = max(big, __shfl_xor_sync(0xffffffffu, big, 1));
        big = max(big, __shfl_xor_sync(0xffffffffu, big, 2));
        const int sh = row_shift(big);
        const float up = pow2f(sh), down = pow2f(-sh);
        unsigned hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float y0 = y[2 * i] * up, y1 = y[2 * i + 1] * up;
            const __half2 h = __floats2half2_rn(y0, y1);
            const float2 hf = __half22float2(h);
            const float z0 = fabsf(y0) <= 65504.f ? y0 - hf.x : 0.f, z1 = fabsf(y1) <= 65504.f ? y1 - hf.y : 0.f;
            const __half2 l = __floats2half2_rn(z0, z1);   // (an infinity has no rest)
            hi[i] = *reinterpret_cast<const unsigned*>(&h);
            lo[i] = *reinterpret_cast<const unsigned*>(&l);
        }
        // the scales of columns 2 t and 2 t + 1 (column c: lanes 4 c ...)
        const float s0 = __shfl_sync(0xffffffffu, down, 8 * t), s1 = __shfl_sync(0xffffffffu, down, 8 * t + 4);
        unsigned b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = low ? lo[i] : hi[i];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            if (m && nr <= 16) break;   // (warp-uniform)
            float c[4];
            mma_16816_first(c, x[2 * m].x, x[2 * m + 1].x, x[2 * m].y, x[2 * m + 1].y, b[0], b[1]);
            mma_16816(c, x[2 * m].z, x[2 * m + 1].z, x[2 * m].w, x[2 * m + 1].w, b[2], b[3]);
            if constexpr (NR == 8) {
                mma_16816(c, x[2 * m].x, x[2 * m + 1].x, x[2 * m].y, x[2 * m + 1].y, lo[0], lo[1]);
                mma_16816(c, x[2 * m].z, x[2 * m + 1].z, x[2 * m].w, x[2 * m + 1].w, lo[2], lo[3]);
            }
            acc[m][0] = fmaf(c[0], s0, acc[m][0]);
            acc[m][1] = fmaf(c[1], s1, acc[m][1]);
            acc[m][2] = fmaf(c[2], s0, acc[m][2]);
            acc[m][3] = fmaf(c[3], s1, acc[m][3]);
        }
        if (k % kSum == kSum - 1 || k + 1 == nk) {
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    sum[m][f] += acc[m][f];
                    acc[m][f] = 0.f;
                }
        }
    }
    const bool fits = FDPH_IDX((long long)tk.item * 32 + 32 <= a.cap_partial, a.err);
    const float ks = a.kinv;   // the window's storage scale (a power of two)
    double* out = a.partial + (size_t)tk.item * 32;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            float v = sum[m][f];
            if constexpr (NR < 8) v += __shfl_xor_sync(0xffffffffu, v, NR / 2);   // hi + lo
            const int col = 2 * t + (f & 1), row = 16 * m + g + 8 * (f >> 1);
            if (col < NR && fits && row < nr) out[col * a.rs_partial + row] = wide(v * ks);
        }
}
