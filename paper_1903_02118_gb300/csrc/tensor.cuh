// tensor.cuh -- the near-field windows of several right-hand sides on the tensor cores (FP16 window).
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
// The slip rates must not lose digits to FP16: a row (step, right-hand side) is split into two FP16 rows
// of x 2^sh (sh puts the row's largest entry in [2^13, 2^14); hi = fp16(x 2^sh), lo = fp16(x 2^sh - hi),
// 2^-22 relative, 2^-39 of the row's largest entry absolute), separate columns of the contraction, so
// that the only rounding of the FP16 path remains that of the stored coefficients.  Each slice's products
// are scaled back per column by 2^-sh and added to the item's FP32 sums.
#pragma once
#include "step.cuh"

// Dscale[slot][right-hand side] = 2^-sh of the ring's rows: sh = 14 - e for the row's largest
// |x| = f 2^e, f in [0.5, 1) (e from the exponent field; a zero or subnormal row takes the largest
// shift).  One CTA per row: the launch's nb steps, or every slot (all_slots, after a state restore).
constexpr int kRowThreads = 256;

__device__ __forceinline__ int row_shift(float m) {
    const int e = m > 0.f ? (int)((__float_as_uint(m) >> 23) & 0xffu) - 126 : -126;
    return min(max(14 - e, -100), 100);
}

// 2^k as a float, k in [-126, 127]
__device__ __forceinline__ float pow2f(int k) { return __uint_as_float((unsigned)(127 + k) << 23); }

template <class T>
__global__ void __launch_bounds__(kRowThreads) row_scale_kernel(StepArgs<T> a, int all_slots) {
    __shared__ float wmax[kRowThreads / 32];
    const int slot = all_slots ? blockIdx.x : wrap(step_index(a) + blockIdx.x, a.WD);
    const float* row = a.Dring32 + blockIdx.y * a.rs_D + (size_t)slot * a.N;
    float m = 0.f;
    for (int p = threadIdx.x; p < a.N; p += kRowThreads) m = fmaxf(m, fabsf(row[p]));
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kRowThreads / 32; ++w) m = fmaxf(m, wmax[w]);
        a.Dscale[(size_t)slot * a.nrhs + blockIdx.y] = pow2f(-row_shift(m));
    }
}

__device__ __forceinline__ void mma_16816(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                          unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

static const int kTcWarps = 4;

// NR right-hand sides, B steps of a launch.  Rows in shared memory: row q of the item holds the slip
// rates of step n + B - 1 - k0 - q, [q][hi, lo][right-hand side][32 sources]; 8 consecutive rows are the
// columns of one MMA tile, so window slice k takes the tiles from row k - k0 on, B NR / 4 of them
// (tile = one step of 8 right-hand sides' hi or lo, of 4 with both, 2 steps of 2).
template <int NR, int B>
struct TcCfg {
    static_assert((NR == 2 && B % 2 == 0) || NR == 4 || NR == 8, "whole tiles");
    static constexpr int C = 2 * NR;                        // columns of one row q
    static constexpr int tiles = NR == 8 ? B : B * NR / 4;  // accumulator tiles (hi and lo of 8 share one)
    static constexpr int rows(int chunk) { return chunk + B - 1; }
    static constexpr size_t row_bytes(int chunk) { return (size_t)rows(chunk) * C * 64; }
    // rows and their scales; afterwards the warps' sums
    static constexpr size_t smem(int chunk) {
        const size_t a = row_bytes(chunk) + (size_t)rows(chunk) * C * 4, r = (size_t)kTcWarps * B * NR * 32 * 4;
        return a > r ? a : r;
    }
};

template <int NR, int B>
__global__ void __launch_bounds__(32 * kTcWarps, 3) tc_block_kernel(StepArgs<float> a) {
    using Cf = TcCfg<NR, B>;
    constexpr int C = Cf::C;
    extern __shared__ __align__(16) unsigned char tc_smem[];
    const NearTask tk = a.tasks[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = step_index(a), nb = a.nb, nr = tk.nr, ns = tk.ns;
    const int nk = tk.k0 < n + nb ? tk.k1 - tk.k0 : 0;   // (0: the item's window lies before the march)
    const int nrow = nk ? nk + B - 1 : 0;
    __half* rows = (__half*)tc_smem;
    float* scl = (float*)(tc_smem + Cf::row_bytes(nk > 0 ? nk : 1));
    {
        const int top = n + B - 1 - tk.k0, hend = hist_end(a, n), stop = wrap(top, a.WD);
        const float* ring = a.Dring32 + tk.s0 + (lane < ns ? lane : 0);
        // (the loads of kAhead rows in flight at a time: a row is a dependent pair of loads otherwise, and
        // the staging, not the MMAs, bounded the kernel)
        constexpr int kAhead = 8;
        for (int u0 = warp * kAhead; u0 < nrow * NR; u0 += kTcWarps * kAhead) {
            float x[kAhead], sc[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                const int u = u0 + i, q = u / NR, r = u % NR, t = top - q;
                const bool ok = u < nrow * NR && t >= 0 && t < hend;
                int slot = stop - q;              // nrow <= WD: one wrap at most
                slot += slot < 0 ? a.WD : 0;
                x[i] = ok && lane < ns ? ring[r * a.rs_D + (size_t)slot * a.N] : 0.f;
                sc[i] = ok ? a.Dscale[(size_t)slot * NR + r] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                const int u = u0 + i, q = u / NR, r = u % NR;
                if (u >= nrow * NR) break;
                // 2^sh from 2^-sh: the exponents add up to that of 1
                const float y = x[i] * (sc[i] > 0.f ? __uint_as_float((254u << 23) - __float_as_uint(sc[i])) : 0.f);
                const __half hi = __float2half_rn(y);
                rows[(size_t)(q * C + r) * 32 + lane] = hi;
                rows[(size_t)(q * C + NR + r) * 32 + lane] = __float2half_rn(y - __half2float(hi));
                if (lane == 0) scl[q * C + r] = scl[q * C + NR + r] = sc[i];
            }
        }
    }
    __syncthreads();
    const int g = lane >> 2, t = lane & 3;
    // the 16-byte vectors (sources 8 t ... 8 t + 7) of receivers g, g + 8, g + 16, g + 24
    const __half* base = (const __half*)a.tensor + tk.off;
    const bool in = FDPH_IDX(tk.off + (long long)nk * tk.sl <= a.len_tensor, a.err) && 8 * t < ns;
    auto load = [&](int k, uint4 (&x)[4]) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int i = g + 8 * m;
            x[m] = in && k < nk && i < nr ? __ldcs((const uint4*)(base + (size_t)k * tk.sl + ((size_t)t * nr + i) * 8))
                                          : make_uint4(0, 0, 0, 0);
        }
    };
    float acc[Cf::tiles][2][4];
#pragma unroll
    for (int i = 0; i < Cf::tiles; ++i)
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int f = 0; f < 4; ++f) acc[i][m][f] = 0.f;
    uint4 x[4], xn[4];
    load(warp, xn);
    for (int k = warp; k < nk; k += kTcWarps) {
#pragma unroll
        for (int m = 0; m < 4; ++m) x[m] = xn[m];
        load(k + kTcWarps, xn);
        const __half* rk = rows + ((size_t)k * C + g) * 32 + 8 * t;
        const float* sk = scl + k * C + 2 * t;
#pragma unroll
        for (int i = 0; i < Cf::tiles; ++i) {
            float c[2][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int f = 0; f < 4; ++f) c[m][f] = 0.f;
            constexpr int parts = NR == 8 ? 2 : 1;   // (8 right-hand sides: the hi tile, then the lo tile)
#pragma unroll
            for (int h = 0; h < parts; ++h) {
                const uint4 b = *(const uint4*)(rk + (size_t)(i * parts + h) * 8 * 32);
#pragma unroll
                for (int m = 0; m < 2; ++m) mma_16816(c[m], x[2 * m].x, x[2 * m + 1].x, x[2 * m].y, x[2 * m + 1].y, b.x, b.y);
#pragma unroll
                for (int m = 0; m < 2; ++m) mma_16816(c[m], x[2 * m].z, x[2 * m + 1].z, x[2 * m].w, x[2 * m + 1].w, b.z, b.w);
            }
            const float2 s = *(const float2*)(sk + i * parts * 8);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                acc[i][m][0] = fmaf(c[m][0], s.x, acc[i][m][0]);
                acc[i][m][1] = fmaf(c[m][1], s.y, acc[i][m][1]);
                acc[i][m][2] = fmaf(c[m][2], s.x, acc[i][m][2]);
                acc[i][m][3] = fmaf(c[m][3], s.y, acc[i][m][3]);
            }
        }
    }
    __syncthreads();   // the rows have been read: their place takes the warps' sums
    // red[warp][step][right-hand side][receiver]
    float* red = (float*)tc_smem + (size_t)warp * B * NR * 32;
#pragma unroll
    for (int i = 0; i < Cf::tiles; ++i)
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                float v = acc[i][m][f];
                if constexpr (NR == 4) v += __shfl_xor_sync(0xffffffffu, v, 2);   // hi + lo
                if constexpr (NR == 2) v += __shfl_xor_sync(0xffffffffu, v, 1);
                const int col = 2 * t + (f & 1);          // column of the tile
                const int q = NR == 2 ? 2 * i + (col >> 2) : i, r = col % NR;
                const bool mine = NR == 8 || (NR == 4 ? col < 4 : !(col & 2));
                if (mine) red[((B - 1 - q) * NR + r) * 32 + 16 * m + g + 8 * (f >> 1)] = v;
            }
    __syncthreads();
    if (!FDPH_IDX((long long)tk.item * 32 + 32 <= a.cap_partial, a.err)) return;
    const float ks = a.kinv;   // the window's storage scale (a power of two)
    for (int u = threadIdx.x; u < nb * NR * 32; u += 32 * kTcWarps) {
        const int i = u & 31, r = (u >> 5) % NR, b = (u >> 5) / NR;
        const float* v = (const float*)tc_smem + (size_t)(b * NR + r) * 32 + i;
        double s = wide(v[0] * ks);
#pragma unroll
        for (int w = 1; w < kTcWarps; ++w) s += wide(v[(size_t)w * B * NR * 32] * ks);
        if (i < nr) a.partial[r * a.rs_partial + b * a.cap_partial + (size_t)tk.item * 32 + i] = s;
    }
}
