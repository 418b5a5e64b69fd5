// fixed.cuh -- the near field of FP64 plans: FP64 products on the FP16 tensor cores, without rounding.
//
// This GPU does two FP64 multiply-adds a clock and SM (and its FP64 MMA no more), against 1034 FP16 ones,
// so the FP64 units bounded every FP64 near field.  The products are therefore formed by the Ozaki
// scheme (Ozaki, Ogita, Oishi, Rump 2012): a coefficient and a slip rate are each a power of two, common
// to the slice (16 receivers) or the row, times a 62-bit fixed-point number, written as eight balanced
// base-256 digits d in [-128, 127],
//     x = 2^(E - 1028) sum_p d_p 2^(-8 p),  p = 0 ... 7,
// exact in FP16.  A digit product and its sum over the 32 sources and the digit pairs of one weight
// (level l = p + q, at most 8 x 32 x 2^14 = 2^22) is exact in the FP32 accumulators of the MMAs.  The
// levels 0 ... 7 of a slice are then put together: 0 ... 3 exactly as one 46-bit integer, 4 ... 7 in FP32 (a
// relative error of 2^-56 of the sum), and added to the output's FP64 sum.  Against FP64 arithmetic, which
// rounds every product and every partial sum to 2^-53, one slice is rounded twice.
//
// The coefficients are stored in that form (fx_pack_kernel: 8 bytes each, the biased fixed-point number,
// and an exponent per slice and 16 receivers); taking them apart on every read kept the integer pipe busy
// for longer than the memory.
//
// Bounds of one 32 x 32 slice and 16 steps, clocks of an SM: 288 MMAs 576, putting together 480 (FP64 pipe) + ~210
// (integer pipe), digits ~130; the FP64 multiply-adds took 7600.  One step: 8 KB from memory, ~370.
//
// Every step of this is a function of the slice and of one row, so an output does not depend on the
// columns it shares an MMA with: the single step (whose 8 columns are the 8 levels of its one row) gives
// the bits of the block of 16 (whose columns are the steps, one accumulator per level).
// Non-finite slip rates give NaN.
#pragma once
#include "step.cuh"
#include "tensor.cuh"

static const int kFxWarps = 4;
static const int kFxDigit = 80;               // bytes of one row's digit: 32 halves, padded
static const int kFxRow = 8 * kFxDigit + 16;  // bytes of a row (16 modulo 128: no bank conflicts across rows)
// biased fixed-point number of x under the common exponent E: x 2^(61 - (E - 1023)) + 128 in every byte
__device__ __forceinline__ unsigned long long fx_bytes(double x, int E) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const int e = (h >> 20) & 0x7ff;
    unsigned mh = e ? (h & 0xfffffu) | 0x100000u : 0u, ml = e ? l : 0u;   // (subnormal numbers count as zero)
    mh = (mh << 9) | (ml >> 23);
    ml <<= 9;
    const int s = E - e, s1 = min(s, 32), s2 = min(s - s1, 32);
    unsigned lo = __funnelshift_rc(ml, mh, s1), hi = __funnelshift_rc(mh, 0u, s1);
    lo = __funnelshift_rc(lo, hi, s2);
    hi = __funnelshift_rc(hi, 0u, s2);
    const unsigned long long sg = (unsigned long long)(long long)((int)h >> 31);
    return (((((unsigned long long)hi) << 32) | lo) ^ sg) - sg + 0x8080808080808080ull;
}

// the four digits in one 32-bit word of a pair of numbers, highest first, as half2 (first, second)
__device__ __forceinline__ void fx_digits(unsigned w0, unsigned w1, unsigned (&d)[4]) {
    const unsigned k = 0x64646464u;   // high byte of the halves 1024 + byte
    const unsigned top = __byte_perm(w0, w1, 0x7362), bot = __byte_perm(w0, w1, 0x5140);   // bytes 3, 2 and 1, 0 side by side
    const unsigned v[4] = {__byte_perm(top, k, 0x4342), __byte_perm(top, k, 0x4140), __byte_perm(bot, k, 0x4342),
                           __byte_perm(bot, k, 0x4140)};
    const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6480));            // 1024 + 128
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&v[q]), off);
        d[q] = *reinterpret_cast<const unsigned*>(&r);
    }
}

__device__ __forceinline__ int fx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// an integer below 2^53 in size as a double, without the FP64 pipe
__device__ __forceinline__ double fx_double(long long j) {
    const unsigned long long sg = (unsigned long long)(j >> 63), u = ((unsigned long long)j ^ sg) - sg;
    if (!u) return 0.0;
    const int z = __clzll((long long)u);
    // mantissa with its leading 1 at bit 52, which adds 1 to the exponent field
    const unsigned long long m = ((u << z) >> 11) + ((unsigned long long)(1023 + 62 - z) << 52);
    return __longlong_as_double((long long)(m | (sg & 0x8000000000000000ull)));
}

// levels 2 j and 2 j + 1 as one integer S_2j 256 + S_2j+1 (each an integer below 2^22 in size)
__device__ __forceinline__ int fx_pair(float s0, float s1) {
    const float magic = 12582912.f;   // 1.5 2^23: the sum's low bits are the integer
    return (__float_as_int(s0 + magic) - 0x4b400000) * 256 + (__float_as_int(s1 + magic) - 0x4b400000);
}

// 2^(ek + ed - 2080), the weight of levels 0 ... 3 taken as one integer; NaN for non-finite operands
__device__ __forceinline__ double fx_scale(int ek, int ed) {
    const int e = ek + ed - 2080 + 1023;
    if (ek == 0x7ff || ed == 0x7ff) return __hiloint2double(0x7ff80000, 0);
    return __hiloint2double((e <= 0 ? 0 : min(e, 0x7ff)) << 20, 0);
}

// B fragments of one 16-source step: 8 x 8 tiles of FP16 whose rows (columns of the MMA) are 16 bytes at
// the addresses of lanes 8 i ... 8 i + 7
__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], unsigned p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(p));
}
__device__ __forceinline__ void ldsm_x2(unsigned (&r)[2], unsigned p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(p));
}

template <int B>
struct FxCfg {
    static constexpr int rows(int chunk) { return chunk + B - 1 > kFxWarps * B ? chunk + B - 1 : kFxWarps * B; }
    // a row of zeros, the rows' digits, their exponents; afterwards the warps' sums
    static constexpr size_t smem(int chunk) {
        const size_t r = 128 + (size_t)rows(chunk) * (kFxRow + 4), d = (size_t)kFxWarps * B * 16 * 8;
        return r > d ? r : d;
    }
};

// Coefficients of one kind (window or aux slices) of every leaf into the stored form, in place: one CTA
// per leaf, one warp per slice and 16 receivers; ex[2 slice + tile], slices numbered over the leaves from
// first[leaf] on.
__global__ void fx_pack_kernel(double* data, int* ex, const NearDev* leaves, const long long* first, int aux, int soe) {
    const NearDev L = leaves[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int cnt = aux ? 1 + (L.tail >= 0 ? soe : 0) : L.W;
    const int pairs = (L.ns + 1) / 2;
    for (int u = warp; u < 2 * cnt; u += nw) {
        const int k = u >> 1, i0 = (u & 1) * 16, m = min(L.nr - i0, 16);   // (m <= 0: no such receivers)
        double* sl = data + (aux ? L.stat + (long long)k * L.sla : L.tensor + (long long)k * L.sl);
        int E = 0;
        for (int e = lane; e < pairs * 16; e += 32)
            if ((e & 15) < m) {
                const double2 x = *(const double2*)(sl + ((size_t)(e >> 4) * L.nr + i0 + (e & 15)) * 2);
                E = max(E, max(fx_exponent(x.x), fx_exponent(x.y)));
            }
        E = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
        for (int e = lane; e < pairs * 16; e += 32)
            if ((e & 15) < m) {
                double2* p = (double2*)(sl + ((size_t)(e >> 4) * L.nr + i0 + (e & 15)) * 2);
                const double2 x = *p;
                *(ulonglong2*)p = make_ulonglong2(fx_bytes(x.x, E), fx_bytes(x.y, E));
            }
        if (lane == 0) ex[2 * (first[blockIdx.x] + k) + (u & 1)] = E;
    }
}

// One CTA per work item and right-hand side (grid y).  Warps: two per 16-receiver tile, taking every second slice
// (leaves of at most 16 receivers: four on one tile).  Window items stage the rows of their nk + B - 1
// steps once; aux items four slices at a time, each warp forming the rows of one (static tile: C(n - W),
// tail terms: the states V_q, updated here by their only reader).
template <int B>
__global__ void __launch_bounds__(32 * kFxWarps, B == 1 ? 5 : 3) fixed_block_kernel(StepArgs<double> a, int chunk) {
    static_assert(B == 1 || B == 16, "one step (its levels in the columns of a tile) or sixteen");
    constexpr int NT = B == 1 ? 1 : 2, NL = B == 1 ? 1 : 8;   // column tiles, accumulators per tile
    extern __shared__ __align__(128) unsigned char fx_smem[];
    const NearTask tk = a.tasks[blockIdx.x];
    const int rh = blockIdx.y;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n = step_index(a), nb = a.nb, nr = tk.nr, ns = tk.ns;
    unsigned char* rows = fx_smem + 128;
    int* expo = (int*)(rows + (size_t)FxCfg<B>::rows(chunk) * kFxRow);
    if (threadIdx.x < 32) ((int*)fx_smem)[threadIdx.x] = 0;
    const int ways = nr > 16 ? 2 : 4;
    const int mt = ways == 2 ? warp & 1 : 0, first = ways == 2 ? warp >> 1 : warp;
    const bool win = !tk.kind;
    const int total = win && tk.k0 >= n + nb ? 0 : tk.k1 - tk.k0;   // (0: the item's window lies before the march)
    const int per = win ? max(total, 1) : kFxWarps;                 // slices staged together
    const unsigned long long* mat = (const unsigned long long*)(win ? a.tensor : a.stat) + tk.off;
    const int* ex = (win ? a.fx_win : a.fx_aux) + 2 * (long long)tk.slice + mt;
    const bool in = FDPH_IDX(tk.off + (long long)(tk.k1 - tk.k0) * tk.sl <= (win ? a.len_tensor : a.len_aux) &&
                                 (win || tk.k1 <= 1 || tk.vstate + (long long)(tk.k1 - 1) * ns <= a.len_vstate),
                             a.err);
    const bool src = lane < ns;
    const size_t col = (size_t)tk.s0 + (src ? lane : 0);
    const double* Dr = a.Dring + rh * a.rs_D + col;

    // a row's digits and exponent into row slot r of shared memory (x: this lane's source)
    auto put_row = [&](int r, double x) {
        const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)fx_exponent(x));
        const unsigned long long v = fx_bytes(x, E);
        unsigned d[8];
        fx_digits((unsigned)(v >> 32), 0u, *(unsigned (*)[4])&d[0]);
        fx_digits((unsigned)v, 0u, *(unsigned (*)[4])&d[4]);
        unsigned short* p = (unsigned short*)(rows + (size_t)r * kFxRow) + lane;
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q * (kFxDigit / 2)] = (unsigned short)d[q];
        if (lane == 0) expo[r] = E;
    };

    double sum[NT][4];
#pragma unroll
    for (int i = 0; i < NT; ++i)
#pragma unroll
        for (int f = 0; f < 4; ++f) sum[i][f] = 0.0;

    for (int base = 0; base < total; base += per) {
        if (base) __syncthreads();   // the rows staged before have been read
        if (win) {
            // row q: slip rates of step n + B - 1 - k0 - q
            const int top = n + B - 1 - tk.k0, hend = hist_end(a, n), stop = wrap(top, a.WD), nrow = total + B - 1;
            constexpr int kAhead = 4;
            for (int q0 = warp * kAhead; q0 < nrow; q0 += kFxWarps * kAhead) {
                double x[kAhead];
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    const int q = q0 + i, tt = top - q;
                    int slot = stop - q;
                    slot += slot < 0 ? a.WD : 0;
                    x[i] = q < nrow && src && tt >= 0 && tt < hend ? Dr[(size_t)slot * a.N] : 0.0;
                }
#pragma unroll
                for (int i = 0; i < kAhead; ++i)
                    if (q0 + i < nrow) put_row(q0 + i, x[i]);
            }
        } else if (base + warp < total) {
            const int ai = tk.k0 + base + warp, t0 = n - tk.W;
            double x[B];
            if (ai == 0) {
                const double* Cr = a.Cring + rh * a.rs_C + col;
                const bool fixed = a.hist != HIST_BASE || tk.W >= kBlk;   // (else rup_step_kernel takes the static term)
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const int tt = min(t0 + b, hist_end(a, n) - 1);   // (the slip by the steps that the launch may use)
                    x[b] = b < nb && src && fixed && tt >= 0 ? Cr[(size_t)wrap(tt, a.WC) * a.N] : 0.0;
                }
            } else {
                double* vs = a.vstate + rh * a.len_vstate + tk.vstate + (size_t)(ai - 1) * ns + (src ? lane : 0);
                const double rho = a.rho[ai - 1];
                double v = src && in ? *vs : 0.0;
#pragma unroll
                for (int b = 0; b < B; ++b)
                    x[b] = b < nb && src && t0 + b >= 0 ? Dr[(size_t)wrap(t0 + b, a.WD) * a.N] : 0.0;
#pragma unroll
                for (int b = 0; b < B; ++b)
                    if (b < nb) x[b] = v = fma(rho, v, x[b]);
                if (src && in) *vs = v;
            }
#pragma unroll
            for (int b = 0; b < B; ++b) put_row(warp * B + B - 1 - b, x[b]);
        }
        __syncthreads();
        const int cnt = min(per, total - base);
        // the slice's 16-byte pairs of sources 2 q, 2 q + 1: q = 8 s + t and 8 s + 4 + t of the 16-source steps s,
        // of receivers g and g + 8 of the tile
        auto load = [&](int k, ulonglong2 (&x)[2][2][2]) {
            const unsigned long long* sl = mat + (size_t)(base + k) * tk.sl;
            constexpr unsigned long long zero = 0x8080808080808080ull;
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int q = 8 * s + 4 * h + t, i = 16 * mt + g + 8 * r;
                        x[s][h][r] = in && k < cnt && 2 * q < ns && i < nr
                                         ? __ldcs((const ulonglong2*)(sl + ((size_t)q * nr + i) * 2))
                                         : make_ulonglong2(zero, zero);
                    }
        };
        for (int k = first; k < cnt; k += ways) {
            const int row0 = win ? k : k * B;
            ulonglong2 x[2][2][2];
            load(k, x);
            const int E = ex[2 * (base + k)];
            float acc[NL][NT][4];
#pragma unroll
            for (int l = 0; l < NL; ++l)
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                    for (int f = 0; f < 4; ++f) acc[l][i][f] = 0.f;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                unsigned A[8][4];   // digit p of (g, pair t), (g + 8, t), (g, 4 + t), (g + 8, 4 + t)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const unsigned long long v0 = x[s][h][r].x, v1 = x[s][h][r].y;
                        unsigned d[4];
                        fx_digits((unsigned)(v0 >> 32), (unsigned)(v1 >> 32), d);
#pragma unroll
                        for (int p = 0; p < 4; ++p) A[p][2 * h + r] = d[p];
                        fx_digits((unsigned)v0, (unsigned)v1, d);
#pragma unroll
                        for (int p = 0; p < 4; ++p) A[4 + p][2 * h + r] = d[p];
                    }
                const int m = lane >> 3, c = lane & 7;
                if constexpr (B == 16) {
                    // column c of tile i: row row0 + c + 8 i
                    const unsigned addr = (unsigned)__cvta_generic_to_shared(
                        rows + (size_t)(row0 + c + 8 * (m >> 1)) * kFxRow + s * 32 + (m & 1) * 16);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        unsigned b[4];
                        ldsm_x4(b, addr + q * kFxDigit);
#pragma unroll
                        for (int p = 0; p + q < 8; ++p) {
                            mma_16816(acc[p + q][0], A[p][0], A[p][1], A[p][2], A[p][3], b[0], b[1]);
                            mma_16816(acc[p + q][1], A[p][0], A[p][1], A[p][2], A[p][3], b[2], b[3]);
                        }
                    }
                } else {
                    // column l: digit l - p of the row, so that digit p of the slice adds to level l
                    const unsigned char* row = rows + (size_t)row0 * kFxRow + s * 32 + (m & 1) * 16;
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        unsigned b[2];
                        ldsm_x2(b, (unsigned)__cvta_generic_to_shared(c >= p ? row + (c - p) * kFxDigit : fx_smem));
                        mma_16816(acc[0][0], A[p][0], A[p][1], A[p][2], A[p][3], b[0], b[1]);
                    }
                }
            }
            if constexpr (B == 16) {
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    const double sc[2] = {fx_scale(E, expo[row0 + 8 * i + 2 * t]), fx_scale(E, expo[row0 + 8 * i + 2 * t + 1])};
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        const long long j = (long long)fx_pair(acc[0][i][f], acc[1][i][f]) * 65536 + fx_pair(acc[2][i][f], acc[3][i][f]);
                        const float l0 = fmaf(acc[5][i][f], 0x1p-8f, acc[4][i][f]), l1 = fmaf(acc[7][i][f], 0x1p-8f, acc[6][i][f]);
                        sum[i][f] = fma(fx_double(j), sc[f & 1], sum[i][f]);
                        sum[i][f] = fma(wide(fmaf(l1, 0x1p-16f, l0) * 0x1p-8f), sc[f & 1], sum[i][f]);
                    }
                }
            } else {
                // lane t holds levels 2 t and 2 t + 1 of receivers g and g + 8; lane t = 0 puts them together
                const double sc = fx_scale(E, expo[row0]);
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float s0 = acc[0][0][2 * r], s1 = acc[0][0][2 * r + 1];
                    const int u = t < 2 ? fx_pair(s0, s1) : __float_as_int(fmaf(s1, 0x1p-8f, s0));
                    const int v = __shfl_xor_sync(0xffffffffu, u, 1);
                    const float low = fmaf(__int_as_float(v), 0x1p-16f, __int_as_float(u)) * 0x1p-8f;   // (lanes 2)
                    const float l = __shfl_xor_sync(0xffffffffu, low, 2);
                    const long long j = (long long)u * 65536 + v;                                        // (lanes 0)
                    sum[0][r] = fma(fx_double(j), sc, sum[0][r]);
                    sum[0][r] = fma(wide(l), sc, sum[0][r]);
                }
            }
        }
    }
    __syncthreads();   // the rows have been read: their place takes the warps' sums [warp][step][16 receivers]
    double* red = (double*)fx_smem + (size_t)warp * B * 16;
    if constexpr (B == 16) {
#pragma unroll
        for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int f = 0; f < 4; ++f) red[(B - 1 - (8 * i + 2 * t + (f & 1))) * 16 + g + 8 * (f >> 1)] = sum[i][f];
    } else if (t == 0) {
        red[g] = sum[0][0];
        red[g + 8] = sum[0][1];
    }
    __syncthreads();
    if (!FDPH_IDX((long long)tk.item * 32 + 32 <= a.cap_partial, a.err)) return;
    for (int u = threadIdx.x; u < nb * 32; u += 32 * kFxWarps) {
        const int i = u & 31, b = u >> 5;
        if (i >= nr) continue;
        const double* v = (const double*)fx_smem + (size_t)(ways == 2 ? i >> 4 : 0) * B * 16 + b * 16 + (i & 15);
        double s = v[0];
        for (int w = 1; w < ways; ++w) s += v[(size_t)w * (ways == 2 ? 2 : 1) * B * 16];
        a.partial[rh * a.rs_partial + b * a.cap_partial + (size_t)tk.item * 32 + i] = s;
    }
}
