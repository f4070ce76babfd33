// Two-stage register FFT for the lengths with a two-radix plan (L = 32 ... 1024).
//
// A line of length L = RA * RB (radices 4 to 32) is transformed in two Stockham stages. In
// stage A (stride 1) task j < L/RA takes inputs j + r L/RA (r < RA) straight from global memory
// (or from the caller), applies the RA-point DFT in registers and writes output r to position
// j RA + r of a shared exchange buffer. In stage B (stride RA) task j < RA reads positions
// j + r RA (r < RB), multiplies input r by w^(j r), w = exp(sign 2 pi i / L), applies the RB-point
// DFT and holds output r = X[j + RA r] in registers, which the caller writes out. A line thus
// crosses shared memory once (one 8-byte write and one read per element); the exchange buffer
// pads every RA elements by one and every line to a pitch = 4 (mod 16) elements, so that the
// two access patterns use the minimum number of bank wavefronts for both thread mappings used
// (8 lines x 4 tasks per warp, or 32 tasks of one line per warp).
//
// Because the stage-B output of task j (X[j + RA r], r < RB) is exactly the stage-A input set
// of task j of a transform with the radices swapped (RB, RA), an inverse transform can follow a
// forward one on the same registers (the z pass chains forward, multiply, inverse).
//
// Twiddles w^(j r) come from two small shared tables, w^j (j < 32) and w^(8 m j) (m < 4, j < 32):
// w^(j r) = w^(8 floor(r/8) j) * (w^j)^(r mod 8), at most 7 multiplications from a table value.
#pragma once

#include "fft_engine.cuh"

namespace colapm {

template <int L>
struct F2;
template <> struct F2<32> { static constexpr int R1 = 8, R2 = 4; };
template <> struct F2<48> { static constexpr int R1 = 8, R2 = 6; };
template <> struct F2<64> { static constexpr int R1 = 8, R2 = 8; };
template <> struct F2<80> { static constexpr int R1 = 8, R2 = 10; };
template <> struct F2<96> { static constexpr int R1 = 8, R2 = 12; };
template <> struct F2<128> { static constexpr int R1 = 16, R2 = 8; };
template <> struct F2<160> { static constexpr int R1 = 16, R2 = 10; };
template <> struct F2<192> { static constexpr int R1 = 16, R2 = 12; };
template <> struct F2<256> { static constexpr int R1 = 16, R2 = 16; };
template <> struct F2<320> { static constexpr int R1 = 16, R2 = 20; };
template <> struct F2<384> { static constexpr int R1 = 16, R2 = 24; };
template <> struct F2<512> { static constexpr int R1 = 16, R2 = 32; };
template <> struct F2<1024> { static constexpr int R1 = 32, R2 = 32; };

// Lengths with a two-stage plan: every mesh side above 16, and half of every one above 32. The mixed ones (48, 80,
// 96, 160, 192, 320, 384) take a composite second radix (6, 10, 12, 20, 24), itself split into coprime factors in registers (prime-factor algorithm).
template <int L>
struct F2Has {
    static constexpr bool value = L == 32 || L == 48 || L == 64 || L == 80 || L == 96 || L == 128 || L == 160 || L == 192 || L == 256 || L == 320 ||
                                  L == 384 || L == 512 || L == 1024;
};

// Exchange buffer of LINES lines (8 by default) for a stage-A radix RA.
template <int L, int RA, int LINES = 8>
struct Xch {
    static constexpr int BASE = L + L / RA;
    static constexpr int PITCH = BASE + (((4 - BASE % 16) % 16) + 16) % 16;   // = 4 (mod 16)
    static constexpr int SIZE = LINES * PITCH;     // float2 elements
    __host__ __device__ __forceinline__ static int at(int c, int e) { return c * PITCH + e + e / RA; }
};

// Twiddle tables for length L: w1[j] = w^j, w8[m][j] = w^(8 m j), w = exp(-2 pi i / L). w^(j r) is w8[r >> 3][j] times a
// power of w1[j], made by a chain of products.
struct Tw2 {
    float2 w1[32];
    float2 w8[4][32];
};
// The same with the powers too, each rounded once: w[k][j] = w^(k j), k < 8, j < JN. A chain repeats the rounding of w1[j] in
// every power, and whatever it takes from a root's modulus it takes from each line alike, so that it stays in the mean of
// a P(k) bin. For the lengths whose other engine takes its roots from the full table (32, 48 and 80 points): rms error of a
// transform 9.2e-8, 9.8e-8 and 1.22e-7 by chains, 7.3e-8, 7.9e-8 and 8.7e-8 by this table, power of a line off by
// -7.9e-8, -5.9e-8 and -3.0e-8, now -3.8e-8, -3.7e-8 and 0.8e-8 (emulated on the CPU against FP64), in the same time. At 64, 160 and 192
// points it would gain as much but costs 0.4 to 1% on their meshes (spectrum of 64^3 cells 64.1 -> 66.5 us): chains there.
template <int JN>
struct Tw8 {
    static_assert(JN == 16 || JN == 32, "");
    float2 w[8][JN];
    float2 w8[4][JN];
};
template <int L>
struct TwSel {
    using type = Tw2;
};
template <> struct TwSel<32> { using type = Tw8<16>; };
template <> struct TwSel<48> { using type = Tw8<16>; };
template <> struct TwSel<80> { using type = Tw8<16>; };
template <int L>
using TwOf = typename TwSel<L>::type;

template <int L, int TWN>
__device__ __forceinline__ void load_tw2(Tw2* t, const float2* __restrict__ g, int T) {
    for (int e = threadIdx.x; e < 32 * 5; e += T) {
        const int m = e / 32, j = e % 32;
        const int idx = m == 0 ? j : ((8 * (m - 1) * j) % L);
        const float2 v = g[idx * (TWN / L)];
        if (m == 0) t->w1[j] = v; else t->w8[m - 1][j] = v;
    }
}
template <int L, int TWN, int JN>
__device__ __forceinline__ void load_tw2(Tw8<JN>* t, const float2* __restrict__ g, int T) {
    for (int e = threadIdx.x; e < JN * 12; e += T) {
        const int k = e / JN, j = e % JN;
        const float2 v = g[((k < 8 ? k : 8 * (k - 8)) * j) % L * (TWN / L)];
        if (k < 8) t->w[k][j] = v; else t->w8[k - 8][j] = v;
    }
}

// p[k] = w^(S j k), k < N <= 8.
template <int N, int S>
__host__ __device__ __forceinline__ void tw_powers(float2* p, const Tw2* t, int j) {
    float2 w1 = t->w1[j];
    if (S > 0) w1 = cconj(w1);
    p[0] = make_float2(1.0f, 0.0f);
#pragma unroll
    for (int k = 1; k < N; ++k) p[k] = cmul(p[k - 1], w1);
}
template <int N, int S, int JN>
__host__ __device__ __forceinline__ void tw_powers(float2* p, const Tw8<JN>* t, int j) {
    p[0] = make_float2(1.0f, 0.0f);
#pragma unroll
    for (int k = 1; k < N; ++k) p[k] = S > 0 ? cconj(t->w[k][j]) : t->w[k][j];
}
// Multiply v[r] by w^(S j r) for r < R (j < 32).
template <int R, int S, class TW>
__host__ __device__ __forceinline__ void twiddle2(float2* v, const TW* t, int j) {
    float2 p[8];
    tw_powers<(R < 8 ? R : 8), S>(p, t, j);
#pragma unroll
    for (int r = 1; r < R; ++r) {
        float2 w = p[r & 7];
        if (r >= 8) {
            float2 b = t->w8[r >> 3][j];
            if (S > 0) b = cconj(b);
            w = (r & 7) ? cmul(b, w) : b;
        }
        v[r] = cmul(v[r], w);
    }
}

}  // namespace colapm

#include "colapm_internal.h"
#include "launch_cache.h"

namespace colapm {

template <int L>
struct K2 {   // threads: the larger task count of the two stages (8 lines)
    static constexpr int RA = F2<L>::R1, RB = F2<L>::R2;
    static constexpr int TA = 8 * L / RA, TB = 8 * L / RB;
    static constexpr int T = TA > TB ? TA : TB;
};

__device__ __forceinline__ int sbin(int i, int L) { return i < L / 2 ? i : i - L; }

// Half-spectrum layouts (n = L/2 complex columns kx, rows y, planes z): standard [z][y][kx], or
// blocked [kx/8][y/8][z][y%8][kx%8]. In the blocked layout every tile the passes read is made of
// 512-byte runs: an x-pass tile of 8 rows is one run per 8-column block, a y-pass tile takes one
// run per group of 8 rows, and the rows of a z-pass tile are 512 bytes apart (64 bytes each; the
// 8 tiles of one row group, taken one after the other, complete every run). In the standard layout
// the rows of a z tile are 4 MB apart, every one in a different 2 MB page, which streams at about a
// third of the bandwidth.
template <int L, bool BLK>
__host__ __device__ __forceinline__ size_t hs_index(int kx, int y, int z) {
    if constexpr (BLK)
        return ((((((size_t)(kx >> 3) * (L / 8) + (y >> 3)) * L + z) << 3) + (y & 7)) << 3) + (kx & 7);
    else return ((size_t)z * L + y) * (L / 2) + kx;
}

// Distance between rows y and y + d of one column (d a multiple of 8 in the blocked layout).
template <int L, bool BLK>
__host__ __device__ __forceinline__ constexpr size_t hs_ystep(int d) {
    return BLK ? (size_t)(d / 8) * L * 64 : (size_t)d * (L / 2);
}

// Offset of row j + r STEP from row 0 of a column: what the passes add per register index. A compile-time
// multiple from row j on, except where STEP is not a multiple of 8 in the blocked layout (the mixed lengths).
template <int L, bool BLK, int STEP>
__host__ __device__ __forceinline__ size_t hs_row(int j, int r) {
    if constexpr (!BLK || STEP % 8 == 0) {
        return (BLK ? (size_t)(j >> 3) * L * 64 + (j & 7) * 8 : (size_t)j * (L / 2)) + r * hs_ystep<L, BLK>(STEP);
    } else {
        const int y = j + r * STEP;
        return (size_t)(unsigned)((y >> 3) * (L * 64) + (y & 7) * 8);
    }
}

// Stage B of a line held in exchange buffer xb (stage-A radix RA), task j < RA of line c:
// loads j + RA r, twiddles, RB-point DFT. Returns X[j + RA r] in v.
template <int L, int RA, int RB, int S, int LINES = 8, bool TRIV = false, class TW = Tw2>
__host__ __device__ __forceinline__ void stage_b(const float2* xb, const TW* tw, int c, int j, float2* v) {
#pragma unroll
    for (int r = 0; r < RB; ++r) v[r] = xb[Xch<L, RA, LINES>::at(c, j + RA * r)];
    twiddle2<RB, S>(v, tw, j);
    dft<RB, S, TRIV>(v);
}

// ---------------------------------------------------------------------------------------------
// y pass (strided columns, stride n = L/2 complex), persistent over tiles of 8 columns.
template <int L, int S, bool BLK = false>
__global__ void __launch_bounds__(K2<L>::T) k2_fy(float2* __restrict__ data, size_t fstride,
                                                   const float2* __restrict__ tw, int nfields) {
    using K = K2<L>;
    constexpr int RA = K::RA, RB = K::RB, n = L / 2, NG = n / 8, TPF = NG * L;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    auto* tws = reinterpret_cast<TwOf<L>*>(xb + Xch<L, RA>::SIZE);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, K::T);
    pdl_wait();
    __syncthreads();
    const int total = TPF * nfields;
    const int tid = threadIdx.x, c = tid & 7, j = tid >> 3;
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
        const int f = t / TPF, r0 = t % TPF;
        // rows y = j + r L/RA (stage A) and j + RA r (stage B)
        float2* g = data + (size_t)f * fstride + hs_index<L, BLK>((r0 % NG) * 8 + c, 0, r0 / NG);
        if (tid < K::TA) {
            float2 v[RA];
#pragma unroll
            for (int r = 0; r < RA; ++r) v[r] = __ldcg(g + hs_row<L, BLK, L / RA>(j, r));
            dft<RA, S>(v);
#pragma unroll
            for (int r = 0; r < RA; ++r) xb[Xch<L, RA>::at(c, j * RA + r)] = v[r];
        }
        __syncthreads();
        if (tid < K::TB) {
            float2 v[RB];
            stage_b<L, RA, RB, S>(xb, tws, c, j, v);
#pragma unroll
            for (int r = 0; r < RB; ++r) g[hs_row<L, BLK, RA>(j, r)] = v[r];
        }
        __syncthreads();
    }
}

// P(k) of a tile of C columns (k_y = ky, k_x = kx0 + c): pbuf holds |X|^2, C lines of PP floats with one word of padding per
// PER z; each of the T threads bins PER consecutive z of one line, and their mirror images L - z, which have the same
// |n| and window (win: sinc^2 along z): FP32 sums of at most 2 PER modes, then one reduction each in L2
// (fire and forget; shared-memory FP64 atomics are retry loops on which the lanes of a warp collide), over 16
// copies of the bins. What bounded the binning was the search for the next bin, which the lanes of a warp reach
// at different modes (BinWalk), and a square root and a division per mode. At 64^3, 128^3, 512^3 and 1024^3 with
// 32 to 100 bins the pass took 17, 42, 717 and 5171 us with them, 8, 16, 298 and 2109 us now (512^3
// with its tiles moved by boxes, k2_power_box: 235). Counting the modes apart, over 1/48 of the grid, took
// 460 us at 1024^3: the loops were too few and too long. Every pair of modes is divided by its own window: a factor
// per column times a table per z is faster (512^3 227 us, 1024^3 1998), but their few roundings
// stay in a bin's mean (P(k) off by 1.60, 1.77 and 2.37e-7 at 128^3, 192^3 and 384^3 instead of 1.51, 1.62 and 2.33e-7).
// |n| is summed in units of the fundamental, which is applied to the sums in FP64.
template <int L, int C, int T>
struct PowerTile {
    static constexpr int PER = L * C / (2 * T), PP = ((L + L / PER + 31) / 32) * 32 + 32 / C;   // the reads of a warp on 32 banks
    static_assert(PER * T * 2 == L * C && L % PER == 0, "the runs must cover the tile");
    __device__ __forceinline__ static int at(int c, int z) { return c * PP + z + z / PER; }
};
template <int L, int C, int T>
__device__ __forceinline__ void power_bin_tile(const float* pbuf, int kx0, int ky, const float* __restrict__ sinc2,
                                               const float* win, const int* lo, const PowerArgs& pw, double* part) {
    using P = PowerTile<L, C, T>;
    const int c = threadIdx.x % C, j = threadIdx.x / C, nx = kx0 + c, ny = sbin(ky, L);
    const float wxy = sinc2[nx] * sinc2[ky];
    const float mult = nx == 0 ? 1.0f : 2.0f, cp = mult * pw.pnorm;
    const int nxy2 = nx * nx + ny * ny, z0 = j * P::PER;
    double* psum = part + pw.nbins;
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(part + 2 * pw.nbins);
    BinWalk w;
    w.start(nxy2 + z0 * z0, lo, pw);
    float acc = 0.0f, ks = 0.0f;
    unsigned modes = 0;
    auto flush = [&]() {
        const int b = w.bin(pw.nbins);
        if (b >= 0) {
            atomicAdd(&part[b], (double)ks);
            atomicAdd(&psum[b], (double)acc);
            atomicAdd(&cnt[b], (unsigned long long)(nx == 0 ? modes : 2 * modes));
        }
        acc = 0.0f;
        ks = 0.0f;
        modes = 0;
    };
#pragma unroll
    for (int zz = 0; zz < P::PER; ++zz) {
        const int z = z0 + zz, m = L - z, n2 = nxy2 + z * z;
        const float s = pbuf[P::at(c, z)] + (z ? pbuf[P::at(c, m)] : 0.0f);
        if (w.leaves(n2)) {   // the run leaves its bin
            flush();
            w.advance(n2, pw.nbins);
        }
        const float wz = wxy * win[z];
        acc += __fdividef(cp * s, wz * wz);
        ks = fmaf(z ? 2.0f * mult : mult, sqrtf((float)n2), ks);
        modes += z ? 2 : 1;
    }
    // Few bins: all lanes of a warp end in one and would meet on the same three words. A call at 512^3 with 1, 8 and 32 bins
    // took 4011, 1697 and 1021 us without this, 1535, 1088 and 958 with it (runs that leave a bin on the
    // way still meet); from 64 bins on the lanes rarely agree, and asking them cost 1% at 100.
    const int b = w.bin(pw.nbins);
    const bool whole = T % 32 == 0 || threadIdx.x / 32 < T / 32;   // the last warp of 80 threads has 16 lanes
    if (pw.nbins < 64 && whole && __all_sync(0xffffffffu, b == __shfl_sync(0xffffffffu, b, 0))) {
        if (b < 0) return;
        double k = (double)ks, p = (double)acc;
        unsigned n = nx == 0 ? modes : 2 * modes;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            k += __shfl_xor_sync(0xffffffffu, k, o);
            p += __shfl_xor_sync(0xffffffffu, p, o);
            n += __shfl_xor_sync(0xffffffffu, n, o);
        }
        if (threadIdx.x % 32 == 0) {
            atomicAdd(&part[b], k);
            atomicAdd(&psum[b], p);
            atomicAdd(&cnt[b], (unsigned long long)n);
        }
    } else {
        flush();
    }
}
// Adds up R copies of the bins (in their order), Q results a thread at a time: R Q loads in flight.
template <int R, int Q>
__device__ __forceinline__ void power_add_copies(const PowerArgs& pw, int T) {
    const size_t copy = (size_t)3 * pw.nbins;
    for (int b0 = threadIdx.x; b0 < 2 * pw.nbins; b0 += Q * T) {
        double v[Q][R];
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) v[q][r] = __ldcg(pw.part + r * copy + min(b0 + q * T, 2 * pw.nbins - 1));
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int b = b0 + q * T;
            double s = 0.0;
#pragma unroll
            for (int r = 0; r < R; ++r) s += v[q][r];
            if (b < pw.nbins) pw.ksum[b] = pw.kfd * s;
            else if (b < 2 * pw.nbins) pw.psum[b - pw.nbins] = s;
        }
    }
    for (int b0 = threadIdx.x; b0 < pw.nbins; b0 += Q * T) {
        unsigned long long v[Q][R];
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r)
                v[q][r] = __ldcg(reinterpret_cast<const unsigned long long*>(pw.part + r * copy + 2 * pw.nbins) + min(b0 + q * T, pw.nbins - 1));
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            unsigned long long s = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) s += v[q][r];
            if (b0 + q * T < pw.nbins) pw.cnt[b0 + q * T] = s;
        }
    }
}
// The CTA that finishes last adds up the copies into the result.
__device__ __forceinline__ void power_sum_regions(const PowerArgs& pw, int T) {
    __shared__ unsigned last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(pw.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (pw.regions == kPowerRegions) power_add_copies<kPowerRegions, 1>(pw, T);
    else power_add_copies<kFewRegions, 8>(pw, T);
}
// The tables of a P(k) pass: sinc^2 along z, the thresholds.
template <int L>
__device__ __forceinline__ void power_tables(float* win, int* lo, const float* __restrict__ sinc2, const PowerArgs& pw, int T) {
    load_thresholds(lo, pw, threadIdx.x, T);
    for (int z = threadIdx.x; z < L / 2; z += T) win[z] = sinc2[z];
}
__device__ __forceinline__ double* power_region(const PowerArgs& pw) {
    return pw.part + (size_t)(blockIdx.x & (pw.regions - 1)) * 3 * pw.nbins;
}

// ---------------------------------------------------------------------------------------------
// z pass with the spectral operator fused (see k_fz in fft_kernels.cuh for the algebra):
// forward z (radices R1, R2) -> bases in registers -> inverse z (radices R2, R1) per base.
// C columns per tile: 8, or 4 (the blocked layout) to halve the shared memory per CTA.
template <int L, int MODE, int C = 8, bool DIRECT = false>
struct Z2 {
    static constexpr int R1 = F2<L>::R1, R2 = F2<L>::R2;
    static constexpr int XS = Xch<L, R1, C>::SIZE > Xch<L, R2, C>::SIZE ? Xch<L, R1, C>::SIZE : Xch<L, R2, C>::SIZE;
    static constexpr bool LPT1 = MODE == Z_LPT1 || MODE == Z_LPT1_BASES, BASES = MODE == Z_LPT1_BASES || MODE == Z_LPT2_BASES;
    static constexpr int NSAVE = LPT1 ? 2 : (MODE == Z_POWER ? 0 : 1);   // saved bases B (, C)
    // next tile via cp.async into a shared buffer, or (DIRECT) straight from global memory into the
    // stage-A registers: the smaller footprint fits three CTAs per SM at C = 4, which hides the load
    // latency better than the prefetch does with two (force z pass at 1024^3: 6.0 against 6.9 ms)
    static constexpr bool PREFETCH = !LPT1 && !DIRECT;
    static constexpr int PF = PREFETCH ? C * L : 0;                               // dense [z][C] buffer
    static constexpr int TA = C * L / R1, TB = C * L / R2, T = TA > TB ? TA : TB;
    static constexpr size_t SMEM = sizeof(float2) * ((size_t)XS * (1 + NSAVE) + PF) + sizeof(TwOf<L>);
    static constexpr int PP = PowerTile<L, C, MODE == Z_POWER ? T : L * C / 16>::PP;   // of the |X|^2 lines
    static constexpr size_t SMEM_POWER = SMEM + sizeof(float) * ((size_t)C * PP + L / 2);
    // CTAs per SM: 16 warps for the LPT bases (at most 128 registers; 256 points: 103 and 78 us without the bound, 80 and
    // 54 with it); 12 warps where a task holds 32 values, 20 (at most 102 registers) with the smaller radices
    static constexpr int MINB = DIRECT ? (R1 == 32 || R2 == 32 ? 384 / T : 640 / T) : (BASES ? 512 / T : 1);
};

template <int L, int MODE, int C = 8, bool BLK = false, bool DIRECT = false>
__global__ void __launch_bounds__(Z2<L, MODE, C, DIRECT>::T, Z2<L, MODE, C, DIRECT>::MINB)
    k2_fz(float2* __restrict__ in, ZOut out, const float2* __restrict__ tw, const float* __restrict__ sinc2, int deconv,
          float gnorm, PowerArgs pw) {
    using Z = Z2<L, MODE, C, DIRECT>;
    constexpr int R1 = Z::R1, R2 = Z::R2, n = L / 2, NG = n / C, NTILE = NG * L;
    constexpr int T = Z::T;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    float2* save = xb + Z::XS;                                   // bases B (, C), layout Xch<L,R1>
    float2* pf = xb + Z::XS * (1 + Z::NSAVE);                    // prefetched input tile [z][8]
    auto* tws = reinterpret_cast<TwOf<L>*>(pf + Z::PF);
    float* pbuf = reinterpret_cast<float*>(tws + 1);             // Z_POWER: [C][PP], then the window table, then the thresholds
    float* win = pbuf + (MODE == Z_POWER ? C * Z::PP : 0);
    int* lo = reinterpret_cast<int*>(win + (MODE == Z_POWER ? L / 2 : 0));
    pdl_trigger();
    load_tw2<L, L>(tws, tw, T);
    pdl_wait();
    double* part = nullptr;                                      // Z_POWER: the sums this CTA adds to
    if constexpr (MODE == Z_POWER) {
        power_tables<L>(win, lo, sinc2, pw, T);
        part = power_region(pw);
    }
    __syncthreads();
    const float kf = 6.283185307179586f / (float)L;
    constexpr size_t stride = BLK ? (size_t)64 : (size_t)L * n;   // distance between planes z
    // tile -> (ky, kx0); in the blocked layout the 8 ky of a row group, then the 8 / C column
    // sub-tiles of an 8-column block, are consecutive tiles (together they cover 512-byte runs)
    auto tile_of = [&](int tt, int& ky_, int& kx0_) {
        if constexpr (BLK) {
            constexpr int SUB = 8 / C;
            const int q = tt >> 3;
            ky_ = 8 * (q / (SUB * (n / 8))) + (tt & 7);
            kx0_ = ((q / SUB) % (n / 8)) * 8 + (q % SUB) * C;
        } else {
            ky_ = tt / NG;
            kx0_ = (tt % NG) * C;
        }
    };
    static_assert(!BLK || C == 8 || C == 4, "blocked layout needs 8- or 4-column tiles");
    static_assert(!BLK || MODE == Z_POWER || L < 256, "the blocked force pass of the longer lines is in fft_pair.cuh");
    const int tid = threadIdx.x, c = tid % C, j = tid / C;
    constexpr int TA = Z::TA, TB = Z::TB;   // forward stage-A / stage-B tasks
    auto prefetch = [&](int tt) {   // 16-byte cp.async.cg of rows z = 0..L-1, C columns, into pf
        int pky, pkx0;
        tile_of(tt, pky, pkx0);
        const size_t b = hs_index<L, BLK>(pkx0, pky, 0);
        constexpr int Q = C / 2;    // 16-byte pieces per row
        for (int e = tid; e < L * Q; e += T) {
            const int z = e / Q, q = e % Q;
            cp_async16_cg(pf + z * C + 2 * q, in + b + (size_t)z * stride + 2 * q);
        }
        cp_async_commit();
    };
    if constexpr (Z::PREFETCH) {
        if (blockIdx.x < NTILE) prefetch(blockIdx.x);
    }

    for (int t = blockIdx.x; t < NTILE; t += gridDim.x) {
        int ky, kx0;
        tile_of(t, ky, kx0);
        const int ny = sbin(ky, L);
        const bool nyq_y = (ky == L / 2);
        const size_t base = hs_index<L, BLK>(kx0 + c, ky, 0);
        const int nx = kx0 + c;
        float2 v[R2];   // stage-B results: X[j + R1 r] (j < R1), or the LPT1 input spectrum
        if constexpr (Z::LPT1) {
            if (tid < TB) {
#pragma unroll
                for (int r = 0; r < R2; ++r) v[r] = __ldcg(in + base + (size_t)(j + R1 * r) * stride);
            }
        } else {
            float2 a[R1];
            if constexpr (Z::PREFETCH) {
                cp_async_wait<0>();
                __syncthreads();
                if (tid < TA) {
#pragma unroll
                    for (int r = 0; r < R1; ++r) a[r] = pf[(j + r * (L / R1)) * C + c];
                }
                __syncthreads();   // prefetch buffer consumed
                if (t + (int)gridDim.x < NTILE) prefetch(t + gridDim.x);
            } else if (tid < TA) {
#pragma unroll
                for (int r = 0; r < R1; ++r) a[r] = __ldcg(in + base + (size_t)(j + r * (L / R1)) * stride);
            }
            if (tid < TA) {
                dft<R1, -1>(a);
#pragma unroll
                for (int r = 0; r < R1; ++r) xb[Xch<L, R1, C>::at(c, j * R1 + r)] = a[r];
            }
            __syncthreads();
            if (tid < TB) stage_b<L, R1, R2, -1, C>(xb, tws, c, j, v);
        }

        if constexpr (MODE == Z_POWER) {
            // |X|^2 in z order, then the bins (power_bin_tile)
            if (tid < TB) {
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    const int z = j + R1 * r;
                    pbuf[PowerTile<L, C, T>::at(c, z)] = fmaf(v[r].x, v[r].x, v[r].y * v[r].y);
                }
            }
            __syncthreads();
            if (!nyq_y) power_bin_tile<L, C, T>(pbuf, kx0, ky, sinc2, win, lo, pw, part);
            continue;
        } else {
            // bases: A = g X, B = k_z A (, C = k_z^2 A); g = gnorm / (k^2 [W^d]), 0 on excluded modes
            if (tid < TB) {
                const int nxy2 = nx * nx + ny * ny;                                   // per column
                const float wxy = MODE == Z_FORCE && deconv ? sinc2[nx] * sinc2[ky] : 1.0f;
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    const int z = j + R1 * r;
                    const int nz = sbin(z, L);
                    const int n2 = nxy2 + nz * nz;   // 0 only at k = 0
                    float w = 1.0f;
                    if (MODE == Z_FORCE && deconv) {
                        w = wxy * sinc2[z];
                        if (deconv == 2) w *= w;
                    }
                    // fast division (within 2 ulp; k^2 W is far from the range where it flushes)
                    const float g = !nyq_y && z != L / 2 && n2 != 0 ? __fdividef(gnorm, kf * kf * (float)n2 * w) : 0.0f;
                    v[r] = cscale(v[r], g);
                    const float kz = kf * (float)nz;
                    save[Xch<L, R1, C>::at(c, j + R1 * r)] = cscale(v[r], kz);
                    if constexpr (Z::NSAVE == 2) save[Z::XS + Xch<L, R1, C>::at(c, j + R1 * r)] = cscale(v[r], kz * kz);
                }
            }
            __syncthreads();   // forward exchange buffer free
            const float kyv = kf * (float)ny;
            const float kxv = kf * (float)nx;
            const float sg = MODE == Z_LPT2 ? -out.vscale : out.vscale;
            constexpr int NB = Z::NSAVE + 1;
#pragma unroll 1
            for (int bi = 0; bi < NB; ++bi) {
                // inverse stage A (radix R2) on base bi held by task j < R1
                if (tid < TB) {
                    if (bi > 0) {
#pragma unroll
                        for (int r = 0; r < R2; ++r) v[r] = save[(bi - 1) * Z::XS + Xch<L, R1, C>::at(c, j + R1 * r)];
                    }
                    dft<R2, +1>(v);
#pragma unroll
                    for (int r = 0; r < R2; ++r) xb[Xch<L, R2, C>::at(c, j * R2 + r)] = v[r];
                }
                __syncthreads();
                if (tid < TA) {   // inverse stage B (radix R1), task j < R2: outputs at j + R2 r
                    float2 u[R1];
                    stage_b<L, R2, R1, +1, C>(xb, tws, c, j, u);
#pragma unroll
                    for (int r = 0; r < R1; ++r) {
                        const size_t o = base + (size_t)(j + R2 * r) * stride;
                        const float2 a = u[r];
                        const float2 ia = make_float2(-a.y, a.x);   // i * a
                        if (MODE == Z_FORCE && BLK) {   // bases only; k2_fy_force applies i k_x, i k_y, i
                            out.p[bi == 0 ? 0 : 2][o] = a;
                        } else if (Z::BASES) {
                            out.p[bi][o] = a;
                        } else if (bi == 0) {
                            out.p[0][o] = cscale(ia, sg * kxv);
                            out.p[1][o] = cscale(ia, sg * kyv);
                            if constexpr (MODE == Z_LPT1) {
                                out.p[3][o] = cscale(a, kxv * kxv);
                                out.p[4][o] = cscale(a, kyv * kyv);
                                out.p[6][o] = cscale(a, kxv * kyv);
                            }
                        } else if (bi == 1) {
                            out.p[2][o] = cscale(ia, sg);
                            if constexpr (MODE == Z_LPT1) {
                                out.p[7][o] = cscale(a, kxv);
                                out.p[8][o] = cscale(a, kyv);
                            }
                        } else {
                            out.p[5][o] = a;
                        }
                    }
                }
                __syncthreads();
            }
        }
    }
    if constexpr (MODE == Z_POWER) {
        power_sum_regions(pw, T);
    }
}

// ---------------------------------------------------------------------------------------------
// Inverse y pass of the force in the blocked layout. The z pass leaves the two inverse-z bases
// A' = IFFT_z(g X) in field 0 and B' = IFFT_z(k_z g X) in field 2 (k_x and k_y are constant along
// a z line, so the three force spectra are i k_x A', i k_y A' and i B'). Per 8-column tile this
// kernel makes the three y transforms from the two inputs:
//   F_z = i IFFT_y(B')         -> field 2 (in place)
//   F_y = i IFFT_y(k_y A')     -> field 1
//   F_x = i k_x IFFT_y(A')     -> field 0 (in place; A' is read twice, the second time from L2)
// It reads 8 bytes per cell instead of the 12 of three separate spectra. (512 and 1024 points: k2_fy_box.)
template <int L, bool BLK>
__global__ void __launch_bounds__(K2<L>::T) k2_fy_force(float2* __restrict__ data, size_t fstride,
                                                        const float2* __restrict__ tw, float sg) {
    using K = K2<L>;
    constexpr int RA = K::RA, RB = K::RB, n = L / 2, NG = n / 8, TPF = NG * L;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    auto* tws = reinterpret_cast<TwOf<L>*>(xb + Xch<L, RA>::SIZE);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, K::T);
    pdl_wait();
    __syncthreads();
    const float kf = 6.283185307179586f / (float)L;
    const int tid = threadIdx.x, c = tid & 7, j = tid >> 3;
    for (int t = blockIdx.x; t < TPF; t += gridDim.x) {
        const int kx = (t % NG) * 8 + c;
        const size_t off = hs_index<L, BLK>(kx, 0, t / NG);
        const float kxv = kf * (float)kx;
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            const float2* src = data + (pass == 0 ? 2 * fstride : 0) + off;
            float2* dst = data + (pass == 0 ? 2 : (pass == 1 ? 1 : 0)) * fstride + off;
            if (tid < K::TA) {
                float2 v[RA];
#pragma unroll
                for (int r = 0; r < RA; ++r) {
                    const int y = j + r * (L / RA);
                    v[r] = __ldcg(src + hs_row<L, BLK, L / RA>(j, r));
                    if (pass == 1) v[r] = cscale(v[r], kf * (float)sbin(y, L));
                }
                dft<RA, +1>(v);
#pragma unroll
                for (int r = 0; r < RA; ++r) xb[Xch<L, RA>::at(c, j * RA + r)] = v[r];
            }
            __syncthreads();
            if (tid < K::TB) {
                float2 u[RB];
                stage_b<L, RA, RB, +1>(xb, tws, c, j, u);
                const float sc = pass == 2 ? sg * kxv : sg;
#pragma unroll
                for (int r = 0; r < RB; ++r) dst[hs_row<L, BLK, RA>(j, r)] = make_float2(-sc * u[r].y, sc * u[r].x);
            }
            __syncthreads();
        }
    }
}

// Inverse y pass of the first-order LPT: six spectra from the three bases A, B, C of the z pass (see launch_fy_lpt). The
// x and y derivatives of one base differ by factors constant along a z line, so the passes carry 4 + 12, 12 + 24
// and 24 + 16 bytes per cell (the x pass makes nine rows of them) instead of 4 + 36, 36 + 36 and 36 + 36.
template <int L>
__global__ void __launch_bounds__(K2<L>::T) k2_fy_lpt(const float2* bases, float2* __restrict__ dst, size_t fstride,
                                                      const float2* __restrict__ tw) {
    using K = K2<L>;
    constexpr int RA = K::RA, RB = K::RB, n = L / 2, NG = n / 8, TPF = NG * L;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    auto* tws = reinterpret_cast<TwOf<L>*>(xb + Xch<L, RA>::SIZE);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, K::T);
    pdl_wait();
    __syncthreads();
    const float kf = 6.283185307179586f / (float)L;
    const int tid = threadIdx.x, c = tid & 7, j = tid >> 3;
    for (int t = blockIdx.x; t < TPF; t += gridDim.x) {
        const size_t off = hs_index<L, false>((t % NG) * 8 + c, 0, t / NG);
#pragma unroll 1
        for (int f = 0; f < 6; ++f) {   // A, k_y A, k_y^2 A, B, k_y B, C
            const float2* src = bases + (f < 3 ? 0 : (f < 5 ? 1 : 2)) * fstride + off;
            const int power = f < 3 ? f : (f == 4 ? 1 : 0);
            if (tid < K::TA) {
                float2 v[RA];
#pragma unroll
                for (int r = 0; r < RA; ++r) {
                    v[r] = __ldcg(src + hs_row<L, false, L / RA>(j, r));   // a base's second and third time from L2
                    const float ky = kf * (float)sbin(j + r * (L / RA), L);
                    if (power) v[r] = cscale(v[r], power == 1 ? ky : ky * ky);
                }
                dft<RA, +1>(v);
#pragma unroll
                for (int r = 0; r < RA; ++r) xb[Xch<L, RA>::at(c, j * RA + r)] = v[r];
            }
            __syncthreads();
            if (tid < K::TB) {
                float2 u[RB];
                stage_b<L, RA, RB, +1>(xb, tws, c, j, u);
                float2* d = dst + f * fstride + off;
#pragma unroll
                for (int r = 0; r < RB; ++r) d[hs_row<L, false, RA>(j, r)] = u[r];
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------------------------
// x passes on rows of n complex (the N = 2n real rows), 8 rows per tile.
template <int n>
struct X2 {
    static constexpr int RA = F2<n>::R1, RB = F2<n>::R2;
    static constexpr int TA = 8 * n / RA, TB = 8 * n / RB, T = TA > TB ? TA : TB;
    static constexpr size_t SMEM = sizeof(float2) * (size_t)Xch<n, RA>::SIZE + sizeof(TwOf<n>);
    static constexpr bool SPLIT = n != 128 && n != 256;   // forward: the half spectrum inside stage B (see k2_fx_fwd)
    // inverse: plus a dense [8][n] staging buffer for the cp.async prefetch of the rows
    static constexpr size_t SMEM_INV = SMEM + sizeof(float2) * 8 * (size_t)n;
};

// forward r2c: in = int64 density pairs (I64, converted to rho * scale - 1) or float reals.
// zero (optional): the int64 input itself, cleared as it is read (the next deposit then needs no memset).
template <int n, bool I64, bool BLK = false>
__global__ void __launch_bounds__(X2<n>::T) k2_fx_fwd(const void* in_, float2* __restrict__ out,
                                                       const float2* __restrict__ tw, float scale, int* err,
                                                       int nitems, unsigned long long* zero) {
    using X = X2<n>;
    constexpr int RA = X::RA, RB = X::RB, N = 2 * n;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    auto* tws = reinterpret_cast<TwOf<n>*>(xb + Xch<n, RA>::SIZE);
    pdl_trigger();
    load_tw2<n, N>(tws, tw, X::T);
    pdl_wait();
    __syncthreads();
    const int tid = threadIdx.x;
    bool over = false;
    for (int t = blockIdx.x; t < nitems; t += gridDim.x) {
        const size_t row0 = (size_t)t * 8;
        if (tid < X::TA) {   // stage A: line c, task j (j fastest)
            const int c = tid / (n / RA), j = tid % (n / RA);
            float2 v[RA];
            if constexpr (I64) {
                // all loads first: the clearing stores go through another pointer to the same memory
                ulonglong2 q[RA];
#pragma unroll
                for (int r = 0; r < RA; ++r) q[r] = __ldcs(reinterpret_cast<const ulonglong2*>(in_) + (row0 + c) * n + j + r * (n / RA));
                if (zero) {
#pragma unroll
                    for (int r = 0; r < RA; ++r)
                        __stcs(reinterpret_cast<ulonglong2*>(zero) + (row0 + c) * n + j + r * (n / RA), make_ulonglong2(0ull, 0ull));
                }
#pragma unroll
                for (int r = 0; r < RA; ++r) {
                    over |= ((q[r].x | q[r].y) >> 63) != 0;
                    v[r] = make_float2(fmaf((float)(long long)q[r].x, scale, -1.0f),
                                       fmaf((float)(long long)q[r].y, scale, -1.0f));
                }
            } else {
#pragma unroll
                for (int r = 0; r < RA; ++r) v[r] = __ldcg(reinterpret_cast<const float2*>(in_) + (row0 + c) * n + j + r * (n / RA));
            }
            dft<RA, -1>(v);
#pragma unroll
            for (int r = 0; r < RA; ++r) xb[Xch<n, RA>::at(c, j * RA + r)] = v[r];
        }
        __syncthreads();
        // The half spectrum X[k] from Z[k] and Z[n-k]: inside stage B (partner values by warp shuffle;
        // one barrier and one shared round trip fewer), or in a separate loop over the exchange buffer. Blocked
        // layout, us with one / the other: n = 32 5.5 / 5.9, 48 8.4 / 8.9, 64 9.5 / 11.6, 80 14.9 / 18.4, 96 20.6 /
        // 27.4, 160 111 / 287, 192 186 / 461, 512 3400 / 3800; but 128 162 / 60, and 256 about 790 / 440: there
        // all CTAs write the same few blocks at once, a power of two apart, and wait for them.
        if constexpr (X::SPLIT) {
            if (tid < X::TB) {   // stage B: Z[j + RA r], then X[k] for the same k = j + RA r
                static_assert(32 % RA == 0 && X::TB % 32 == 0, "the partner of a task must be in its warp");
                const int c = tid / RA, j = tid % RA;
                float2 v[RB];
                stage_b<n, RA, RB, -1>(xb, tws, c, j, v);
                // X[k] needs Z[n - k] too: for j > 0 that is element RB - 1 - r of task RA - j (same
                // line, same warp); for j = 0 it is this task's own element (RB - r) mod RB
                const int lane = threadIdx.x & 31;
                const int partner = (lane & ~(RA - 1)) | ((RA - j) & (RA - 1));
                const int y = (int)((row0 + c) % N), z = (int)((row0 + c) / N);
    #pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const float bx = __shfl_sync(0xffffffffu, v[RB - 1 - r].x, partner);
                    const float by = __shfl_sync(0xffffffffu, v[RB - 1 - r].y, partner);
                    const float2 a = v[r], b = j == 0 ? v[(RB - r) % RB] : make_float2(bx, by);
                    const int k = j + RA * r;
                    // X[k] from Z[k] = a, Z[n-k] = b; w^k = exp(-2 pi i k / N) = tw[k]
                    const float2 bc = cconj(b);
                    const float2 E = cscale(cadd(a, bc), 0.5f);
                    const float2 d = csub(a, bc);
                    out[hs_index<N, BLK>(k, y, z)] = cadd(E, cmul(tw[k], make_float2(0.5f * d.y, -0.5f * d.x)));
                }
            }
            __syncthreads();   // exchange buffer free for the next tile's stage A
        } else {
            if (tid < X::TB) {   // stage B in place: Z[j + RA r]
                const int c = tid / RA, j = tid % RA;
                float2 v[RB];
                stage_b<n, RA, RB, -1>(xb, tws, c, j, v);
    #pragma unroll
                for (int r = 0; r < RB; ++r) xb[Xch<n, RA>::at(c, j + RA * r)] = v[r];
            }
            __syncthreads();
            constexpr int H = n / 2 + 1;
            for (int e = tid; e < 8 * H; e += X::T) {
                const int c = e / H, k = e % H, k2 = (n - k) % n;
                const float2 a = xb[Xch<n, RA>::at(c, k)], b = xb[Xch<n, RA>::at(c, k2)];
                const int y = (int)((row0 + c) % N), z = (int)((row0 + c) / N);
                {   // X[k] from Z[k] = a, Z[n-k] = b; w^k = exp(-2 pi i k / N) = tw[k]
                    const float2 bc = cconj(b);
                    const float2 E = cscale(cadd(a, bc), 0.5f);
                    const float2 d = csub(a, bc);
                    out[hs_index<N, BLK>(k, y, z)] = cadd(E, cmul(tw[k], make_float2(0.5f * d.y, -0.5f * d.x)));
                }
                if (k != 0 && k2 != k) {
                    const float2 ac = cconj(a);
                    const float2 E = cscale(cadd(b, ac), 0.5f);
                    const float2 d = csub(b, ac);
                    out[hs_index<N, BLK>(k2, y, z)] = cadd(E, cmul(tw[k2], make_float2(0.5f * d.y, -0.5f * d.x)));
                }
            }
            __syncthreads();
        }
    }
    if constexpr (I64) {
        if (over) atomicOr(err, 1);
    }
}

// inverse c2r in place on `nfields` arrays; the next tile's rows are prefetched into a dense
// [8][n] staging buffer with 16-byte cp.async as soon as stage A has read the current one, so the
// copy overlaps stage B. With BLK the spectra are read in the blocked layout and the real rows
// written to `dst` (same field stride), a separate array; otherwise dst == data and the pass is in
// place.
template <int n, bool BLK = false>
__global__ void __launch_bounds__(X2<n>::T, 3) k2_fx_inv(float2* __restrict__ data, size_t fstride,
                                                       const float2* __restrict__ tw, int items_per_field,
                                                       int nfields, float2* __restrict__ dst) {
    using X = X2<n>;
    constexpr int RA = X::RA, RB = X::RB, N = 2 * n, T = X::T;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    auto* tws = reinterpret_cast<TwOf<n>*>(xb + Xch<n, RA>::SIZE);
    float2* stg = reinterpret_cast<float2*>(tws + 1);   // [8][n]
    pdl_trigger();
    load_tw2<n, N>(tws, tw, T);
    pdl_wait();
    const int tid = threadIdx.x;
    const int nitems = items_per_field * nfields;
    auto gptr = [&](int t) { return dst + (size_t)(t / items_per_field) * fstride + (size_t)(t % items_per_field) * 8 * n; };
    auto prefetch = [&](int t) {
        float2* d = stg;
        if constexpr (BLK) {   // 8 rows of one plane (one row group): a 512-byte run per 8-column block
            const int row0 = (t % items_per_field) * 8, y0 = row0 % N, z = row0 / N;
            const float2* g = data + (size_t)(t / items_per_field) * fstride;
            for (int e = tid; e < 8 * n / 2; e += T) {
                const int q = e & 3, c = (e >> 2) & 7, kxb = e >> 5;
                cp_async16_cg(d + c * n + kxb * 8 + 2 * q, g + hs_index<N, true>(kxb * 8 + 2 * q, y0 + c, z));
            }
        } else {
            const float2* g = data + (size_t)(t / items_per_field) * fstride + (size_t)(t % items_per_field) * 8 * n;
            for (int e = tid; e < 8 * n / 2; e += T) cp_async16_cg(d + 2 * e, g + 2 * e);
        }
        cp_async_commit();
    };
    if (blockIdx.x < nitems) prefetch(blockIdx.x);
    for (int t = blockIdx.x; t < nitems; t += gridDim.x) {
        float2* d = gptr(t);
        const float2* rows = stg;
        cp_async_wait<0>();
        __syncthreads();
        // stage A reads its inputs Z'[k] = E + i O straight from the staged rows, with
        // E = X[k] + conj X[n-k], O = (X[k] - conj X[n-k]) conj w^k and X[n] = 0
        const int ca = tid / (n / RA), ja = tid % (n / RA);
        if (tid < X::TA) {
            const float2* row = rows + ca * n;
            float2 v[RA];
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                const int k = ja + r * (n / RA);
                const float2 xk = row[k];
                const float2 xm = row[k == 0 ? 0 : n - k];
                const float2 xc = k == 0 ? make_float2(0.0f, 0.0f) : cconj(xm);
                const float2 E = cadd(xk, xc);
                const float2 O = cmul(csub(xk, xc), cconj(tw[k]));
                v[r] = make_float2(E.x - O.y, E.y + O.x);
            }
            dft<RA, +1>(v);
#pragma unroll
            for (int r = 0; r < RA; ++r) xb[Xch<n, RA>::at(ca, ja * RA + r)] = v[r];
        }
        __syncthreads();
        if (t + (int)gridDim.x < nitems) prefetch(t + gridDim.x);   // staging free: overlaps stage B
        if (tid < X::TB) {
            const int c = tid / RA, j = tid % RA;
            float2 u[RB];
            stage_b<n, RA, RB, +1>(xb, tws, c, j, u);
#pragma unroll
            for (int r = 0; r < RB; ++r) d[(size_t)c * n + j + RA * r] = u[r];
        }
        // no barrier: the next tile's stage A writes xb only after the wait + barrier at its top
    }
    cp_async_wait<0>();
}

// Inverse x pass of the first-order LPT and the second-order source (see launch_fx_lpt): nine c2r transforms per row from six
// spectra, 8 rows per tile, each spectrum's rows staged by cp.async while the one before is transformed. The six second
// derivatives stay in registers, where a thread holds the same cells of each row; they were stored (24 bytes
// per cell), read by a pass that formed the source, and written and read once more: at 256^3 the x pass and the
// source pass took 281 and 71 us, this one 225 (1.8 TB/s: bound by the exchanges of nine transforms per row and their
// barriers, at 12 to 16 warps per SM), with the y pass 273 and now 121, the z pass 139 and 80; the initial conditions
// of 256^3 particles as a whole went from 1122 to 914 us.
template <int n>
__global__ void __launch_bounds__(X2<n>::T, (X2<n>::RB >= 16 ? 3 : 4) * 128 / X2<n>::T)
    k2_fx_lpt(const float2* spec, size_t fstride, float2* __restrict__ psi, float2* __restrict__ src,
              const float2* __restrict__ tw, int nitems, float vscale) {
    using X = X2<n>;
    constexpr int RA = X::RA, RB = X::RB, N = 2 * n, T = X::T;
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    auto* tws = reinterpret_cast<TwOf<n>*>(xb + Xch<n, RA>::SIZE);
    float2* stg = reinterpret_cast<float2*>(tws + 1);   // [8][n]
    pdl_trigger();
    load_tw2<n, N>(tws, tw, T);
    pdl_wait();
    const int tid = threadIdx.x;
    const float kf = 6.283185307179586f / (float)N;
    // order of the spectra: xx first, then yy and zz (the products), then the mixed ones
    constexpr int NS = 6;
    constexpr int FIELD[NS] = {0, 2, 5, 1, 3, 4};   // A, k_y^2 A, C, k_y A, B, k_y B
    auto prefetch = [&](int t, int f) {
        const float2* g = spec + (size_t)f * fstride + (size_t)t * 8 * n;
        for (int e = tid; e < 8 * n / 2; e += T) cp_async16_cg(stg + 2 * e, g + 2 * e);
        cp_async_commit();
    };
    // c2r of the staged rows times (1, k_x or k_x^2) [times i vscale]: u = real pairs at j + RA r of line c
    const int ca = tid / (n / RA), ja = tid % (n / RA), c = tid / RA, j = tid % RA;
    auto transform = [&](int power, bool vec, float2* u) {
        if (tid < X::TA) {
            const float2* row = stg + ca * n;
            auto factor = [&](int k, float2 x) {
                const float kx = kf * (float)k;
                const float f = (power == 0 ? 1.0f : (power == 1 ? kx : kx * kx)) * (vec ? vscale : 1.0f);
                return vec ? make_float2(-f * x.y, f * x.x) : cscale(x, f);
            };
            float2 v[RA];
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                const int k = ja + r * (n / RA);
                const float2 xk = factor(k, row[k]);
                const float2 xc = k == 0 ? make_float2(0.0f, 0.0f) : cconj(factor(n - k, row[k == 0 ? 0 : n - k]));
                const float2 E = cadd(xk, xc);
                const float2 O = cmul(csub(xk, xc), cconj(tw[k]));
                v[r] = make_float2(E.x - O.y, E.y + O.x);
            }
            dft<RA, +1>(v);
#pragma unroll
            for (int r = 0; r < RA; ++r) xb[Xch<n, RA>::at(ca, ja * RA + r)] = v[r];
        }
        __syncthreads();
        if (tid < X::TB) stage_b<n, RA, RB, +1>(xb, tws, c, j, u);
    };
    if (blockIdx.x < nitems) prefetch(blockIdx.x, FIELD[0]);
    for (int t = blockIdx.x; t < nitems; t += gridDim.x) {
        const size_t out = ((size_t)t * 8 + c) * n + j;
        float2 S[RB], D[RB];   // the source so far; xx, then xx + yy
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            cp_async_wait<0>();
            __syncthreads();   // the staged rows are complete, the exchange buffer free
            const int f = FIELD[s];
            float2 u[RB];
            if (f == 0 || f == 1 || f == 3) {   // a displacement component from the same spectrum
                transform(f == 0 ? 1 : 0, true, u);
                if (tid < X::TB) {
                    float2* d = psi + (size_t)(f == 0 ? 0 : (f == 1 ? 1 : 2)) * fstride + out;
#pragma unroll
                    for (int r = 0; r < RB; ++r) d[RA * r] = u[r];
                }
                __syncthreads();   // the exchange buffer has been read
            }
            transform(f == 0 ? 2 : (f == 1 || f == 3 ? 1 : 0), false, u);
            // every thread has passed the barrier after the last read of the staged rows
            if (s + 1 < NS) prefetch(t, FIELD[s + 1 < NS ? s + 1 : 0]);
            else if (t + (int)gridDim.x < nitems) prefetch(t + gridDim.x, FIELD[0]);
            if (tid < X::TB) {
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    if (s == 0) {
                        D[r] = u[r];
                    } else if (s == 1) {
                        S[r] = make_float2(D[r].x * u[r].x, D[r].y * u[r].y);
                        D[r] = cadd(D[r], u[r]);
                    } else if (s == 2) {
                        S[r] = make_float2(fmaf(D[r].x, u[r].x, S[r].x), fmaf(D[r].y, u[r].y, S[r].y));
                    } else {
                        S[r] = make_float2(fmaf(-u[r].x, u[r].x, S[r].x), fmaf(-u[r].y, u[r].y, S[r].y));
                    }
                }
            }
        }
        if (tid < X::TB) {
#pragma unroll
            for (int r = 0; r < RB; ++r) src[out + RA * r] = S[r];
        }
    }
    cp_async_wait<0>();
}

}  // namespace colapm
