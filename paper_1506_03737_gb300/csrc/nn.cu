// Learned displacement correction: a 3 -> 16 -> 16 -> 16 -> 3 network of periodic 3x3x3
// convolutions with ReLU between layers, trained and applied on the GPU by the kernels in this
// file (BF16 tensor-core products, FP32 accumulation, FP32 master weights, Adam).
//
// The paper has no learned component. The network maps the final displacement field Psi of a
// coarse, few-step COLA run (3 channels on the Lagrangian grid) to a correction dPsi toward a
// fine-mesh, many-step run from the same seed; plain COLA stays the fallback.
//
// Layout
//   activations  bf16 [n + 2][n + 2][n + 2][16] ([z][y][x], 32 B per voxel) with the periodic images around
//                the box stored, so that the halo of any tile is one box of the array: voxel x sits at
//                x + 1, its image at n + 1 (x = 0) or 0 (x = n - 1), likewise y and z; whoever writes a
//                voxel writes its images. Channels 0..7 and 8..15 are two 16-byte halves, which swap
//                places where (stored x >> 2) & 1, so that rows copied as they are into shared memory are
//                read by ldmatrix without bank conflicts (8 consecutive voxels, one half)
//   3 channels   the same with 8 channels (16 B per voxel, the rest zero): the packed input and the
//                gradient at the network output
//   weights      bf16 [tap][c_out 16][c_in 16], tap = (dz+1) 9 + (dy+1) 3 + (dx+1)
//   master       fp32 [layer][28][16][16]: taps 0..26 = W[tap][o][i], slot 27 holds the bias in i = 0
//
// Every convolution (forward of each layer, backward-data of layers 2..4) is one implicit GEMM:
// with mma.sync (k_conv, the default), or on the tcgen05 tensor cores (k_conv_tc, engine 1, grid side
// a multiple of 128). With 16 channels each tcgen05.mma (M = 128 voxels, N = 16, K = 16) reads a 4 KB
// operand from shared memory for 65,536 FLOP, which bounds it by shared-memory bandwidth; measured at
// 128^3 it is slower than the mma.sync kernel.
//
//   forward        out[v][o]  = b[o] + sum_tap sum_i W[tap][o][i] a[v + d_tap][i]
//   backward-data  da[u][i]   = sum_tap sum_o W[tap][o][i] dz[u - d_tap][o]
//                             = forward with W'[tap][i][o] = W[26 - tap][o][i], no bias
//   weight grad    dW[tap][o][i] = sum_v dz[v][o] a[v + d_tap][i];  db[o] = sum_v dz[v][o]
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/colapm.h"
#include "../../include/colapm_nn.h"
#include "colapm_internal.h"
#include "launch_cache.h"
#include "tma.cuh"

namespace colapm {
namespace nn {
namespace {

constexpr int C = 16;                          // padded channel count
constexpr int TX = 16, TY = 8;                 // output tile 16 x 8 x TZ voxels (TZ = 8, or 2 on small grids)
constexpr int HX = TX + 2, HY = TY + 2;
constexpr int CONV_TZ = 8;                      // planes of a k_conv tile
constexpr int SLOTS = 28;                      // 27 taps + bias
constexpr int LAYERS = 4;
constexpr int LSIZE = SLOTS * C * C;           // 7168 master slots per layer
constexpr int CIN[LAYERS] = {3, 16, 16, 16};
constexpr int COUT[LAYERS] = {16, 16, 16, 3};

enum Epi { EPI_RELU = 0, EPI_OUT = 1, EPI_MASK = 2 };

struct ConvArgs {
    const __nv_bfloat16* in;     // input voxels (k_conv_tc; k_conv takes them through its tensor map)
    const __nv_bfloat16* w;      // [27][16][16]
    const float* bias;           // [16] or null
    int n;
    __nv_bfloat16* out;          // EPI_RELU / EPI_MASK: 16 channels; EPI_OUT with target: dz, 8 channels
    const __nv_bfloat16* mask;   // EPI_MASK: the layer input whose ReLU gates the gradient
    float* y;                    // EPI_OUT: [n^3][3] = base + oscale * net
    const float* base;           // EPI_OUT: optional [n^3][3]
    float oscale;
    const float* target;         // EPI_OUT training: [n^3][3] physical; normalised by tscale
    float tscale, gscale;        // gscale = 2 / (3 n^3)
    double* loss;                // sum of squared normalised errors
    bool wide;                   // EPI_OUT: y, base and target start at multiples of 16 bytes
    int* err;                    // bit 4: a bounded wait gave up
};

// Four consecutive floats of a caller's array, as one access where it is aligned.
__device__ __forceinline__ float4 load4(const float* p, bool wide) {
    return wide ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
__device__ __forceinline__ void store4(float* p, float4 v, bool wide) {
    if (wide) {
        *reinterpret_cast<float4*>(p) = v;
    } else {
        p[0] = v.x;
        p[1] = v.y;
        p[2] = v.z;
        p[3] = v.w;
    }
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t addr, uint32_t& r0, uint32_t& r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t addr, uint32_t& r0, uint32_t& r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Place of half `k` (0: channels 0..7, 1: channels 8..15) of a voxel stored at x: its 16-byte slot.
__host__ __device__ __forceinline__ int half_slot(int x, int k) { return k ^ ((x >> 2) & 1); }

// Index of voxel (x, y, z) in the stored array, and a call f(index) for each of its periodic images there.
__device__ __forceinline__ size_t voxel(int n, int x, int y, int z) {
    return ((size_t)(z + 1) * (n + 2) + (y + 1)) * (n + 2) + (x + 1);
}
// Distance to the image along an axis: n on the low face, -n on the high one, 0 inside.
__device__ __forceinline__ int image_of(int x, int n) { return x == 0 ? n : (x == n - 1 ? -n : 0); }
template <class F>
__device__ __forceinline__ void at_images(int n, size_t v, int ox, int oy, int oz, F f) {   // v: the voxel's index
#pragma unroll 1
    for (int m = (ox ? 1 : 0) | (oy ? 2 : 0) | (oz ? 4 : 0), k = m; k; k = (k - 1) & m)   // the subsets of its faces
        f(v + (ptrdiff_t)(k & 1 ? ox : 0) + (ptrdiff_t)(n + 2) * ((k & 2 ? oy : 0) + (ptrdiff_t)(n + 2) * (k & 4 ? oz : 0)));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n" ::);
    asm volatile("cp.async.wait_group 0;\n" ::);
}

template <int TZ>
__device__ __forceinline__ void tile_origin(int t, int n, int& x0, int& y0, int& z0) {
    const int tx = n / TX, ty = n / TY;
    x0 = (t % tx) * TX;
    y0 = ((t / tx) % ty) * TY;
    z0 = (t / (tx * ty)) * TZ;
}

// Byte offsets into the dynamic shared memory of k_conv.
template <int EPI, int TZ, int VB>
struct ConvSmem {
    static constexpr uint32_t HALO = HX * HY * (TZ + 2) * VB;
    static constexpr uint32_t W = HALO;                             // weights [tap][16][16]
    static constexpr uint32_t AUX = W + 27 * C * 32;                // output tile (EPI_MASK: first the mask tile)
    static constexpr uint32_t AUXB = TX * TY * TZ * (EPI == EPI_OUT ? 12 : 32);
    static constexpr uint32_t BAR = AUX + AUXB;                     // one barrier of the halo, one per warp
    static constexpr size_t BYTES = BAR + 8 * (1 + TZ);
};

// Implicit-GEMM convolution, persistent over tiles of 16 x 8 x TZ voxels; warp w makes output plane z = w.
// M = 16 consecutive x voxels per mma, N = output channels (NT n-tiles of 8), K = 16 input channels of
// one tap (VB = 16: the upper 8 are zero and are not stored).
//
// What bounds it: the mma.sync rate (1024 FMA per clock and SM, measured: 600 TFLOP/s), 49 us for a
// 16-channel layer at 128^3. Each operand row (hz, hy, dx) is therefore read once per plane offset dz and used
// for the three dy that need it (rows hy, hy - 1 and hy - 2 of the output), with the nine weights of dz
// in registers: 30 operand loads per 144 products instead of 72. In that order every output still gets its taps
// as (dz, dy, dx) from first to last, so the sums are the same bit for bit as tap by tap. The halo of the
// next tile is fetched by one TMA box while this one's outputs are written, and the second CTA of
// the SM computes while this one waits. At 128^3 a hidden layer takes 73-75 us (65% of the mma.sync rate; what is left
// is the start and end of each tile) against 95 us with one operand load per product pair and per-thread 16-byte
// copies, a backward one 79 against 133, the output layer 64 against 122 (153 with the loss). Row by row bulk copies
// instead of the box took 89-95 us (about 130 cycles each), 4-plane tiles at three CTAs per SM 86 us.
template <int NT, int EPI, int TZ, int VB>
__global__ void __launch_bounds__(32 * TZ, TZ == 8 ? 2 : 4)
    k_conv(ConvArgs a, const __grid_constant__ CUtensorMap halo, const __grid_constant__ CUtensorMap out,
           const __grid_constant__ CUtensorMap mask) {
    using S = ConvSmem<EPI, TZ, VB>;
    extern __shared__ __align__(1024) uint8_t sm[];
    const int n = a.n;
    const int ntiles = (n / TX) * (n / TY) * (n / TZ);
    const int lane = threadIdx.x & 31, tz = threadIdx.x >> 5;
    const int g = lane >> 2, q = lane & 3;
    const uint32_t hb = smem_u32(sm), wb = hb + S::W, aux = hb + S::AUX + tz * (TX * TY * 32),
                   bar = hb + S::BAR, mbar = bar + 8 + 8 * tz;
    pdl_trigger();
    if (threadIdx.x == 0) {
        for (int b = 0; b < 1 + TZ; ++b) mbar_init(bar + 8 * b);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_wait();
    for (int j = threadIdx.x; j < 27 * C * 2; j += 32 * TZ) {   // weights, swizzled with the row index
        const int row = j >> 1, k = j & 1;
        cp_async16(wb + row * 32 + (half_slot(row, k) << 4), a.w + row * C + k * 8);
    }
    cp_async_wait_all();
    __syncthreads();
    // a run of consecutive tiles, so that every CTA has its share of those on the faces of the box, which
    // write images too (dealt out round robin, one CTA had the same place in x every time)
    const int tend = (int)((long long)ntiles * (blockIdx.x + 1) / gridDim.x);
    int t = (int)((long long)ntiles * blockIdx.x / gridDim.x), x0, y0, z0;
    tile_origin<TZ>(t, n, x0, y0, z0);
    auto load_halo = [&]() {   // stored voxel x0 is the left neighbour of x0
        mbar_expect(bar, S::HALO);
        box_load(hb, halo, x0 * (VB / 8), y0, z0, bar);
    };
    auto load_mask = [&]() {   // this warp's plane of the mask tile
        mbar_expect(mbar, TX * TY * 32);
        box_load(aux, mask, (x0 + 1) * 4, y0 + 1, z0 + 1 + tz, mbar);
    };
    if (threadIdx.x == 0) load_halo();

    // ldmatrix roles: A rows (voxels) and halves; B rows (output channels) and halves
    const int ar = (lane & 7) + 8 * ((lane >> 3) & 1), ak = lane >> 4;
    const int bn = (lane & 7) + 8 * (lane >> 4), bk = (lane >> 3) & 1;
    uint32_t aoff[3];   // this lane's operand row for each dx (stored x0 is a multiple of 16)
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
        aoff[dx] = hb + tz * (HY * HX * VB) + (ar + dx) * VB + (VB == 32 ? half_slot(ar + dx, ak) << 4 : 0);
    const uint32_t boff = wb + bn * 32 + (half_slot(bn, bk) << 4);
    double lsum = 0.0;   // loss: the sum over this lane's tiles

    uint32_t phase = 0;
    for (; t < tend; ++t, phase ^= 1) {
        bool ok = mbar_wait(bar, phase);
        if (!ok) ok = (atomicOr(a.err, 4), mbar_wait(bar, phase), false);   // flag it, let the copies land, stop
        if (!__syncthreads_and(ok)) break;
        if (EPI != EPI_OUT && lane == 0) {
            box_stores_read();   // the previous tile's outputs have left the buffer
            if (EPI == EPI_MASK) load_mask();
        }
        constexpr int NPRE = EPI == EPI_OUT ? TX * TY * 3 / 128 : 1;
        float4 pre[NPRE];   // EPI_OUT: the tile of target or base, in flight during the products
        if (EPI == EPI_OUT) {
            const float* src = a.target ? a.target : a.base;
#pragma unroll
            for (int i = 0; i < NPRE; ++i) {
                const int e = 4 * (lane + 32 * i);
                const size_t at = (((size_t)(z0 + tz) * n + y0 + e / (TX * 3)) * n + x0) * 3 + e % (TX * 3);
                pre[i] = src ? load4(src + at, a.wide) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
        }
        float acc[TY][NT][4];
#pragma unroll
        for (int m = 0; m < TY; ++m)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[m][j][e] = 0.0f;
#pragma unroll 1
        for (int dz = 0; dz < 3; ++dz) {
            uint32_t b[9][2 * NT];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                if (NT == 2) ldsm_x4(boff + (dz * 9 + k) * (C * 32), b[k]);
                else ldsm_x2(boff + (dz * 9 + k) * (C * 32), b[k][0], b[k][1]);
            }
            const uint32_t zo = dz * (HY * HX * VB);
#pragma unroll
            for (int hy = 0; hy < HY; ++hy) {
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    uint32_t f[4];
                    if (VB == 32) {
                        ldsm_x4(aoff[dx] + zo + hy * (HX * VB), f);
                    } else {
                        ldsm_x2(aoff[dx] + zo + hy * (HX * VB), f[0], f[1]);
                        f[2] = f[3] = 0u;
                    }
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const int m = hy - dy;
                        if (m < 0 || m >= TY) continue;
#pragma unroll
                        for (int j = 0; j < NT; ++j) mma_bf16(acc[m][j], f, b[3 * dy + dx][2 * j], b[3 * dy + dx][2 * j + 1]);
                    }
                }
            }
        }
        __syncthreads();   // the halo has been read
        const int cx = x0, cy = y0, cz = z0;
        if (t + 1 < tend) {
            tile_origin<TZ>(t + 1, n, x0, y0, z0);
            if (threadIdx.x == 0) load_halo();
        }
        if (EPI == EPI_RELU || EPI == EPI_MASK) {
            if (EPI == EPI_MASK && !mbar_wait(mbar, phase)) {
                atomicOr(a.err, 4);   // flag it and let the copy land
                mbar_wait(mbar, phase);
            }
            float bia[NT][2];
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) bia[j][e] = EPI == EPI_RELU ? a.bias[8 * j + 2 * q + e] : 0.0f;
            __syncwarp();
            uint8_t* tile = sm + S::AUX + tz * (TX * TY * 32);   // voxels as they are stored, from x0 + 1
#pragma unroll
            for (int m = 0; m < TY; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        float u0 = acc[m][j][2 * h], u1 = acc[m][j][2 * h + 1];
                        __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(
                            tile + (m * TX + g + 8 * h) * 32 + half_slot(g + 1, j) * 16 + 4 * q);
                        if (EPI == EPI_RELU) {
                            u0 = fmaxf(u0 + bia[j][0], 0.0f);
                            u1 = fmaxf(u1 + bia[j][1], 0.0f);
                        } else {   // the mask's value lies where the output goes
                            const __nv_bfloat162 mk = *p;
                            u0 = __bfloat162float(mk.x) > 0.0f ? u0 : 0.0f;
                            u1 = __bfloat162float(mk.y) > 0.0f ? u1 : 0.0f;
                        }
                        *p = __floats2bfloat162_rn(u0, u1);
                    }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) box_store(out, (cx + 1) * 4, cy + 1, cz + tz + 1, aux);
            // images of the voxels on the faces of the box (n voxels away: the same half slots, n a multiple of 16).
            // Per axis a set of shifts: 0, +n on the low face, -n on the high one
            const int z = cz + tz;
            const unsigned mx = 1u | (cx == 0 ? 2u : 0u) | (cx + TX == n ? 4u : 0u),
                           my = 1u | (cy == 0 ? 2u : 0u) | (cy + TY == n ? 4u : 0u),
                           mz = 1u | (z == 0 ? 2u : 0u) | (z + 1 == n ? 4u : 0u);
            if ((mx | my | mz) != 1u)
                for (unsigned uz = mz; uz; uz &= uz - 1)
                    for (unsigned uy = my; uy; uy &= uy - 1)
                        for (unsigned ux = mx; ux; ux &= ux - 1) {
                            const unsigned lowz = uz & -uz, lowy = uy & -uy, lowx = ux & -ux;
                            if ((lowx | lowy | lowz) == 1u) continue;   // the voxels themselves
                            const int nx = lowx == 1u ? TX : 1, ny = lowy == 1u ? TY : 1;
                            const int lx = lowx == 4u ? TX - 1 : 0, ly = lowy == 4u ? TY - 1 : 0;
                            const size_t v0 = voxel(n, cx + (lowx == 1u ? 0 : (lowx == 2u ? n : -n)),
                                                    cy + (lowy == 1u ? 0 : (lowy == 2u ? n : -n)),
                                                    z + (lowz == 1u ? 0 : (lowz == 2u ? n : -n)));
                            for (int e = lane; e < 2 * nx * ny; e += 32) {
                                const int x = lx + ((e >> 1) & (nx - 1)), y = ly + (nx == 1 ? e >> 1 : e / (2 * TX));
                                reinterpret_cast<uint4*>(a.out)[2 * (v0 + (size_t)y * (n + 2) + x) + (e & 1)] =
                                    reinterpret_cast<const uint4*>(tile)[2 * (y * TX + x) + (e & 1)];
                            }
                        }
            __syncwarp();
        } else {   // EPI_OUT: channels 0..2 through shared memory, so that rows leave as whole 192-byte runs
            float* so = reinterpret_cast<float*>(sm + S::AUX) + tz * (TX * TY * 3);
            if (q < 2) {
                const float c0 = a.bias[2 * q], c1 = q == 0 ? a.bias[1] : 0.0f;
#pragma unroll
                for (int m = 0; m < TY; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float* p = so + (m * TX + g + 8 * h) * 3 + 2 * q;
                        p[0] = acc[m][0][2 * h] + c0;
                        if (q == 0) p[1] = acc[m][0][2 * h + 1] + c1;
                    }
            }
            __syncwarp();
            float ls = 0.0f, lc = 0.0f;   // the tile's squares: their sum and its rounding errors
#pragma unroll
            for (int k = 0; k < NPRE; ++k) {   // four values a lane: rows are 48 values, all multiples of 4
                const int e = 4 * (lane + 32 * k);
                const size_t i = (((size_t)(cz + tz) * n + cy + e / (TX * 3)) * n + cx) * 3 + e % (TX * 3);
                const float4 u4 = *reinterpret_cast<const float4*>(so + e);
                const float u[4] = {u4.x, u4.y, u4.z, u4.w}, q4[4] = {pre[k].x, pre[k].y, pre[k].z, pre[k].w};
                float yv[4], g4[4], d4[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float b = !a.target ? q4[m] : (a.base ? a.base[i + m] : 0.0f);
                    yv[m] = b + a.oscale * u[m];
                    if (a.target) {
                        const float d = u[m] - q4[m] * a.tscale;
                        g4[m] = a.gscale * d;
                        d4[m] = d;
                        const float p = __fmul_rn(d, d), pe = fmaf(d, d, -p), s = __fadd_rn(ls, p), z = __fsub_rn(s, ls);
                        lc += (__fsub_rn(ls, __fsub_rn(s, z)) + __fsub_rn(p, z)) + pe;
                        ls = s;
                    }
                }
                store4(a.y + i, make_float4(yv[0], yv[1], yv[2], yv[3]), a.wide);
                if (a.target) {
                    *reinterpret_cast<float4*>(so + e) = make_float4(g4[0], g4[1], g4[2], g4[3]);
                    pre[k] = make_float4(d4[0], d4[1], d4[2], d4[3]);
                }
            }
            if (a.target) {
                // Twelve squares as an exact sum of floats (Knuth's two-sum and the product's error by fma), then one
                // FP64 addition, of which the GPU does few. Where the sum is not well inside the range of a
                // float, in which the errors are floats too, and for infinities and NaN, the squares in FP64.
                if (ls >= 0x1p-48f && ls < 0x1p120f) {
                    lsum += (double)ls + (double)lc;
                } else {
#pragma unroll
                    for (int k = 0; k < NPRE; ++k) {
                        const float4 d = pre[k];
                        lsum += ((double)d.x * d.x + (double)d.y * d.y) + ((double)d.z * d.z + (double)d.w * d.w);
                    }
                }
                __syncwarp();
                for (int e = lane; e < TX * TY; e += 32) {
                    const __nv_bfloat162 b01 = __floats2bfloat162_rn(so[3 * e], so[3 * e + 1]);
                    const __nv_bfloat162 b2z = __floats2bfloat162_rn(so[3 * e + 2], 0.0f);
                    const uint4 u = make_uint4(*reinterpret_cast<const uint32_t*>(&b01), *reinterpret_cast<const uint32_t*>(&b2z), 0u, 0u);
                    const int x = cx + e % TX, y = cy + e / TX, z = cz + tz;
                    const size_t v = voxel(n, x, y, z);
                    reinterpret_cast<uint4*>(a.out)[v] = u;
                    at_images(n, v, image_of(x, n), image_of(y, n), image_of(z, n),
                              [&](size_t i) { reinterpret_cast<uint4*>(a.out)[i] = u; });
                }
            }
            __syncwarp();   // the outputs have been read before the next tile's are written
        }
    }
    if (EPI != EPI_OUT && lane == 0) box_stores_read();   // shared memory stays until it has been read
    if (EPI == EPI_OUT && a.target) {
#pragma unroll
        for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0 && lsum != 0.0) atomicAdd(a.loss, lsum);
    }
}

// Byte offsets into the dynamic shared memory of k_wgrad: two buffers of (activation halo, dz tile); at the
// end the per-group sums take their place.
template <int TZ, int VA, int VD>
struct WgradSmem {
    static constexpr uint32_t HALO = HX * HY * (TZ + 2) * VA;
    static constexpr uint32_t BUF = HALO + TX * TY * TZ * VD;
    static constexpr uint32_t SUMS = (TZ / 2) * LSIZE * 4;
    static constexpr uint32_t BAR = 2 * BUF > SUMS ? 2 * BUF : SUMS;
    static constexpr size_t BYTES = BAR + 16;
};

// Per-CTA partial weight gradients of one layer over a static round-robin share of the tiles:
// part[blockIdx.x][slot][o][i]. A warp takes one plane offset dz (9 taps, all accumulators in
// registers) and two output planes of the tile: 3 x TZ / 2 warps. K = the 16 voxels of an x row.
// ACT_A = false: M = output channels (dz rows), N = input channels; true (the last layer, whose 3 output
// channels fit one n-tile): M = input channels, N = output channels.
//
// What bounds it: the mma.sync rate (49 us per 16-channel layer at 128^3). Stepping over the halo rows hy, a
// warp loads the three shifted activation rows (dx) and one dz row, and uses them with the last three dz rows
// (dy): 18 products for 4 operand loads, against 7 for 4.5 when each warp walked its own taps. The next
// tile arrives in the other buffer meanwhile, as two TMA boxes. At 128^3 a 16-channel layer takes
// 67 us (75% of that rate) against 170 us, the first and the last layer 41 and 43.
template <bool ACT_A, int NT, int TZ, int VA, int VD>
__global__ void __launch_bounds__(32 * 3 * (TZ / 2), 1)
    k_wgrad(const __grid_constant__ CUtensorMap act, const __grid_constant__ CUtensorMap dz, int n,
            float* __restrict__ part, int* err) {
    using S = WgradSmem<TZ, VA, VD>;
    constexpr int NTHR = 32 * 3 * (TZ / 2);
    extern __shared__ __align__(1024) uint8_t sm[];
    const int ntiles = (n / TX) * (n / TY) * (n / TZ);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int zo = w % 3, grp = w / 3;                                      // plane offset, planes 2 grp and 2 grp + 1
    const int g = lane >> 2, q = lane & 3;
    const uint32_t sb = smem_u32(sm), bar = sb + S::BAR;
    if (threadIdx.x == 0) {
        mbar_init(bar);
        mbar_init(bar + 8);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    auto load = [&](int t, int buf) {   // halo of the activations and dz of tile t
        int x0, y0, z0;
        tile_origin<TZ>(t, n, x0, y0, z0);
        const uint32_t d = sb + buf * S::BUF, b = bar + 8 * buf;
        mbar_expect(b, S::BUF);
        box_load(d, act, x0 * (VA / 8), y0, z0, b);
        box_load(d + S::HALO, dz, (x0 + 1) * (VD / 8), y0 + 1, z0 + 1, b);
    };
    // Operand rows are voxels (K), read transposed. As A (M = channels): matrices (lo channels, voxels 0-7),
    // (hi, 0-7), (lo, 8-15), (hi, 8-15). As B (N = channels): (lo, 0-7), (lo, 8-15), (hi, 0-7), (hi, 8-15).
    const int a_v = (lane & 7) + 8 * (lane >> 4), a_k = (lane >> 3) & 1;
    const int b_v = (lane & 7) + 8 * ((lane >> 3) & 1), b_k = lane >> 4;
    const int act_v = ACT_A ? a_v : b_v, act_k = ACT_A ? a_k : b_k;
    const int dz_v = ACT_A ? b_v : a_v, dz_k = ACT_A ? b_k : a_k;
    uint32_t ao[3];
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
        ao[dx] = (VA == 32 ? (act_v + dx) * 32 + (half_slot(act_v + dx, act_k) << 4) : (((lane & 15) + dx) * 16)) +
                 zo * (HY * HX * VA);
    const uint32_t dof = S::HALO + (VD == 32 ? dz_v * 32 + (half_slot(dz_v + 1, dz_k) << 4) : (lane & 15) * 16);
    const uint32_t ones = 0x3F803F80u;                                      // bf16 pair (1, 1)
    const uint32_t ones4[4] = {ones, ones, ones, ones};

    float acc[9][NT][4], accb[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int s = 0; s < 9; ++s)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[s][j][e] = 0.0f;

    if (threadIdx.x == 0 && (int)blockIdx.x < ntiles) load(blockIdx.x, 0);
    int it = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++it) {
        const int buf = it & 1;
        if (threadIdx.x == 0 && t + (int)gridDim.x < ntiles) load(t + gridDim.x, buf ^ 1);
        bool ok = mbar_wait(bar + 8 * buf, (it >> 1) & 1);
        if (!ok) ok = (atomicOr(err, 4), mbar_wait(bar + 8 * buf, (it >> 1) & 1), false);
        if (!__syncthreads_and(ok)) {   // let the other buffer's copies land too, then stop
            if (t + (int)gridDim.x < ntiles) mbar_wait(bar + 8 * (buf ^ 1), ((it + 1) >> 1) & 1);
            return;
        }
        const uint32_t base = sb + buf * S::BUF;
#pragma unroll 1
        for (int pl = 0; pl < 2; ++pl) {
            const uint32_t ab = base + (2 * grp + pl) * (HY * HX * VA);
            const uint32_t db = base + dof + (2 * grp + pl) * (TY * TX * VD);
            uint32_t d[TY][4];
#pragma unroll
            for (int hy = 0; hy < HY; ++hy) {
                if (hy < TY) {
                    if (VD == 32) {
                        ldsm_x4_t(db + hy * (TX * VD), d[hy]);
                    } else {   // 8 channels: two matrices, voxels 0-7 and 8-15
                        ldsm_x2_t(db + hy * (TX * VD), d[hy][0], d[hy][1]);
                        d[hy][2] = d[hy][3] = 0u;
                    }
                    if (zo == 1) {   // bias: the sum of dz
                        if (ACT_A) mma_bf16(accb, ones4, d[hy][0], d[hy][1]);
                        else mma_bf16(accb, d[hy], ones, ones);
                    }
                }
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    uint32_t f[4];
                    if (VA == 32) ldsm_x4_t(ab + ao[dx] + hy * (HX * VA), f);
                    else ldsm_x2_t(ab + ao[dx] + hy * (HX * VA), f[0], f[1]);
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const int m = hy - dy;   // output row of the tap (dz, dy, dx) that reads halo row hy
                        if (m < 0 || m >= TY) continue;
#pragma unroll
                        for (int j = 0; j < NT; ++j) {
                            if (ACT_A) mma_bf16(acc[3 * dy + dx][j], f, d[m][0], d[m][1]);
                            else mma_bf16(acc[3 * dy + dx][j], d[m], f[2 * j], f[2 * j + 1]);
                        }
                    }
                }
            }
        }
        __syncthreads();   // this buffer has been read
    }
    // sums of the groups, then over the groups in a fixed order
    float* sums = reinterpret_cast<float*>(sm);
    float* mine = sums + (size_t)grp * LSIZE;
    auto put = [&](int slot, int m, int k, float v) { mine[slot * C * C + (ACT_A ? k * C + m : m * C + k)] = v; };
    for (int e = threadIdx.x; e < (TZ / 2) * LSIZE; e += NTHR) sums[e] = 0.0f;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 9; ++s)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) put(zo * 9 + s, g + 8 * (e >> 1), 8 * j + 2 * q + (e & 1), acc[s][j][e]);
    if (zo == 1) {   // db[o] in column 0 of slot 27: from column 0 (M = o), or from row 0 (N = o)
        if (ACT_A) {
            if (g == 0) {
                put(27, 0, 2 * q, accb[0]);
                put(27, 0, 2 * q + 1, accb[1]);
            }
        } else if (q == 0) {
            put(27, g, 0, accb[0]);
            put(27, g + 8, 0, accb[2]);
        }
    }
    __syncthreads();
    float* p = part + (size_t)blockIdx.x * LSIZE;
    for (int e = threadIdx.x; e < LSIZE; e += NTHR) {
        float s = sums[e];
#pragma unroll
        for (int k = 1; k < TZ / 2; ++k) s += sums[(size_t)k * LSIZE + e];
        p[e] = s;
    }
}

// ---------------------------------------------------------------------------------------------
// The same convolution on the 5th-generation tensor cores (tcgen05), for grids whose side is a
// multiple of 128. A CTA computes TC_ROWS output x-rows of 128 voxels; for each row and tap one
// tcgen05.mma (M = 128 voxels, N = 16 output channels, K = 16 input channels, BF16 x BF16 -> FP32)
// accumulates into the row's 16 TMEM columns. The halo is staged as two K-half planes (channels
// 0..7 and 8..15, 16 bytes per voxel), which is the no-swizzle K-major core-matrix layout: 8
// consecutive voxels x 16 bytes form one 128-byte core matrix, LBO = the plane distance (K),
// SBO = 128 bytes (next 8 voxels). A tap's operand is the row of 128 halo voxels shifted by the
// tap, i.e. a descriptor start offset. Weights: [tap][K half][16 outputs][8 inputs] (512 B a tap).
// One thread issues the MMAs and commits them to an mbarrier; after a bounded wait the four warps
// read their TMEM lanes (lane = voxel) with tcgen05.ld and run the same epilogues as k_conv.
constexpr int TC_TY = 2, TC_TZ = 2, TC_ROWS = TC_TY * TC_TZ;
constexpr int TC_HX = 130, TC_HY = TC_TY + 2, TC_HZ = TC_TZ + 2;
constexpr int TC_HALO = TC_HX * TC_HY * TC_HZ;                    // 2080 voxels
constexpr uint32_t TC_PLANE = TC_HALO * 16;                       // bytes per K-half plane
constexpr uint32_t TC_W = 27 * 512;                               // weight bytes
constexpr size_t TC_SMEM = 2 * (size_t)TC_PLANE + TC_W + 128;     // + mbarrier and TMEM address
constexpr uint32_t TC_COLS = TC_ROWS * 16;                        // TMEM columns (power of two)
// kind::f16 instruction descriptor: FP32 D (bits 4-5), BF16 A and B (bits 7-9, 10-12), both
// K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((16u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);   // no swizzle, base offset 0
}

// Stage the halo of tile t into the two K-half planes with 16-byte cp.async.
// An 8-channel input (in8) fills the first plane; the second is zero and is cleared once by the caller.
__device__ __forceinline__ void tc_stage(uint32_t sbase, const __nv_bfloat16* __restrict__ in, int n, int t, bool in8) {
    const int txn = n / 128, tyn = n / TC_TY;
    const int x0 = (t % txn) * 128, y0 = ((t / txn) % tyn) * TC_TY, z0 = (t / (txn * tyn)) * TC_TZ;
    // thread t copies the 16-byte pieces t, t + 128, ... of each of the 16 rows: the same place in every row
    const int vb = in8 ? 16 : 32, pieces = in8 ? TC_HX : 2 * TC_HX;
    const size_t ys = (size_t)(n + 2) * vb, zs = ys * (n + 2);
    const char* base = reinterpret_cast<const char*>(in) + (size_t)z0 * zs + (size_t)y0 * ys + (size_t)x0 * vb;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int j = threadIdx.x + 128 * i;
        if (j >= pieces) break;
        const int hx = in8 ? j : j >> 1, k = in8 ? 0 : j & 1;
        const char* src = base + (size_t)hx * vb + (in8 ? 0 : half_slot(hx, k) * 16);
        const uint32_t dst = sbase + k * TC_PLANE + hx * 16;
#pragma unroll
        for (int row = 0; row < TC_HY * TC_HZ; ++row)
            cp_async16(dst + row * (TC_HX * 16), src + (row / TC_HY) * zs + (row % TC_HY) * ys);
    }
    asm volatile("cp.async.commit_group;\n" ::);
}

// Persistent over tiles: weights, TMEM and the mbarrier are set up once per CTA. Per tile: wait for
// the staged halo, issue the 27 x TC_ROWS MMAs (one thread), wait for them, start staging the next
// tile's halo (the MMAs no longer read shared memory), then read TMEM and write the outputs.
template <int EPI>
__global__ void __launch_bounds__(128) k_conv_tc(ConvArgs a, bool in8) {
    extern __shared__ __align__(1024) uint8_t sm[];
    uint8_t* wsm = sm + 2 * TC_PLANE;
    uint64_t* mbar = reinterpret_cast<uint64_t*>(wsm + TC_W);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);
    const int n = a.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int txn = n / 128, tyn = n / TC_TY;
    const int ntiles = txn * tyn * (n / TC_TZ);
    const uint32_t sbase = smem_u32(sm);
    for (int j = tid; j < 27 * C * 2; j += 128) {     // weights [tap][K half][out][8]
        const int tap = j >> 5, o = (j >> 1) & 15, k = j & 1;
        cp_async16(sbase + 2 * TC_PLANE + tap * 512 + k * 256 + o * 16, a.w + (tap * C + o) * C + k * 8);
    }
    if (in8)
        for (uint32_t j = tid; j < TC_PLANE / 16; j += 128)
            *reinterpret_cast<uint4*>(sm + TC_PLANE + j * 16) = make_uint4(0u, 0u, 0u, 0u);
    if (blockIdx.x < ntiles) tc_stage(sbase, a.in, n, blockIdx.x, in8);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                     "r"(TC_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t taddr = *tslot;
    const uint64_t a_desc0 = tc_desc(sbase, TC_PLANE, 128), b_desc0 = tc_desc(sbase + 2 * TC_PLANE, 256, 128);
    bool ok = true;
    double lsum = 0.0;
    int it = 0;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++it) {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the tensor cores read these bytes
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (tid == 0) {
#pragma unroll 1
            for (int r = 0; r < TC_ROWS; ++r) {
                const int ry = r % TC_TY, rz = r / TC_TY;
                // descriptor start addresses count 16-byte units: adding a voxel index moves by one voxel
                const uint64_t arow = a_desc0 + (uint64_t)(((rz + 1) * TC_HY + (ry + 1)) * TC_HX + 1);
#pragma unroll
                for (int tap = 0; tap < 27; ++tap) {
                    const int off = (tap / 9 - 1) * TC_HY * TC_HX + ((tap / 3) % 3 - 1) * TC_HX + (tap % 3 - 1);
                    asm volatile(
                        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(taddr + r * 16),
                        "l"(arow + (uint64_t)(int64_t)off), "l"(b_desc0 + (uint64_t)(tap * 32)), "r"(TC_IDESC), "r"(tap));
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                             smem_u32(mbar))
                         : "memory");
        }
        uint32_t done = 0;
        for (long long i = 0; i < SPIN_LIMIT && !done; ++i) {
            asm volatile(
                "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(smem_u32(mbar)), "r"(it & 1)
                : "memory");
        }
        if (!done) {
            if (tid == 0 && a.err) atomicOr(a.err, 4);
            ok = false;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (!__syncthreads_and(done)) break;
        if (t + (int)gridDim.x < ntiles) tc_stage(sbase, a.in, n, t + gridDim.x, in8);   // overlaps the epilogue
        const int x0 = (t % txn) * 128, y0 = ((t / txn) % tyn) * TC_TY, z0 = (t / (txn * tyn)) * TC_TZ;
#pragma unroll 1
        for (int r = 0; r < TC_ROWS; ++r) {
            uint32_t q[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]),
                  "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
                : "r"(taddr + ((uint32_t)(32 * warp) << 16) + r * 16));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            const int ry = r % TC_TY, rz = r / TC_TY;
            const int vx = x0 + 32 * warp + lane, vy = y0 + ry, vz = z0 + rz;
            const size_t v = ((size_t)vz * n + vy) * n + vx, vs = voxel(n, vx, vy, vz);
            float acc[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) acc[c] = __uint_as_float(q[c]);
            if (EPI == EPI_RELU || EPI == EPI_MASK) {
                uint32_t pk[8];
                if (EPI == EPI_MASK) {
                    const uint4* mp = reinterpret_cast<const uint4*>(a.mask + vs * C);
                    const uint4 m0 = mp[half_slot(lane + 1, 0)], m1 = mp[half_slot(lane + 1, 1)];
                    const uint32_t mw[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const __nv_bfloat162 mk = *reinterpret_cast<const __nv_bfloat162*>(&mw[c]);
                        const float v0 = __bfloat162float(mk.x) > 0.0f ? acc[2 * c] : 0.0f;
                        const float v1 = __bfloat162float(mk.y) > 0.0f ? acc[2 * c + 1] : 0.0f;
                        const __nv_bfloat162 b = __floats2bfloat162_rn(v0, v1);
                        pk[c] = *reinterpret_cast<const uint32_t*>(&b);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const __nv_bfloat162 b = __floats2bfloat162_rn(fmaxf(acc[2 * c] + a.bias[2 * c], 0.0f),
                                                                       fmaxf(acc[2 * c + 1] + a.bias[2 * c + 1], 0.0f));
                        pk[c] = *reinterpret_cast<const uint32_t*>(&b);
                    }
                }
                auto put = [&](size_t i) {
                    uint4* op = reinterpret_cast<uint4*>(a.out) + 2 * i;
                    op[half_slot(lane + 1, 0)] = make_uint4(pk[0], pk[1], pk[2], pk[3]);   // stored at lane + 1 (mod 8)
                    op[half_slot(lane + 1, 1)] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                };
                put(vs);
                at_images(n, vs, image_of(vx, n), image_of(vy, n), image_of(vz, n), put);
            } else {   // EPI_OUT: channels 0..2
                float dzv[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float val = acc[c] + a.bias[c];
                    a.y[v * 3 + c] = (a.base ? a.base[v * 3 + c] : 0.0f) + a.oscale * val;
                    dzv[c] = 0.0f;
                    if (a.target) {
                        const float d = val - a.target[v * 3 + c] * a.tscale;
                        lsum += (double)d * d;
                        dzv[c] = a.gscale * d;
                    }
                }
                if (a.target) {
                    const __nv_bfloat162 b01 = __floats2bfloat162_rn(dzv[0], dzv[1]);
                    const __nv_bfloat162 b2z = __floats2bfloat162_rn(dzv[2], 0.0f);
                    const uint4 u = make_uint4(*reinterpret_cast<const uint32_t*>(&b01), *reinterpret_cast<const uint32_t*>(&b2z), 0u, 0u);
                    reinterpret_cast<uint4*>(a.out)[vs] = u;
                    at_images(n, vs, image_of(vx, n), image_of(vy, n), image_of(vz, n),
                              [&](size_t i) { reinterpret_cast<uint4*>(a.out)[i] = u; });
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");   // TMEM reads done before the next MMAs
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (EPI == EPI_OUT && a.target) {
#pragma unroll
        for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0 && lsum != 0.0) atomicAdd(a.loss, lsum);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(TC_COLS));
}

__device__ __forceinline__ bool real_slot(int l, int slot, int o, int i) {
    constexpr int cin[LAYERS] = {3, 16, 16, 16}, cout[LAYERS] = {16, 16, 16, 3};
    if (o >= cout[l]) return false;
    return slot < 27 ? i < cin[l] : i == 0;
}

// Sum the per-CTA partials of every layer in a fixed order: grad[l][slot][o][i]. 32 slots per block, the
// partials dealt over RG_Y rows of threads (a column of 304 sums one after the other took 23 us).
constexpr int RG_Y = 32;
__global__ void __launch_bounds__(32 * RG_Y) k_reduce_grads(const float* part, int nparts, float* __restrict__ grad) {
    pdl_trigger();
    pdl_wait();
    __shared__ float sh[RG_Y][33];
    const int idx = blockIdx.x * 32 + threadIdx.x;   // LAYERS * LSIZE is a multiple of 32
    const int l = idx / LSIZE, r = idx % LSIZE;
    const int slot = r / (C * C), o = (r / C) % C, i = r % C;
    const bool real = real_slot(l, slot, o, i);
    float s = 0.0f;
    if (real)
        for (int b = threadIdx.y; b < nparts; b += RG_Y) s += part[((size_t)l * nparts + b) * LSIZE + r];
    sh[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0) {
        s = 0.0f;
#pragma unroll
        for (int k = 0; k < RG_Y; ++k) s += sh[k][threadIdx.x];
        grad[idx] = real ? s : 0.0f;
    }
}

// Adam on the FP32 master copy, then the BF16 forward and flipped-transposed weights and the bias. No update after a wait that
// gave up (err), until that has been reported: the partial gradients are then not all written.
__global__ void k_adam(float* __restrict__ wm, float* __restrict__ m1, float* __restrict__ m2,
                       const float* grad, float lr, float b1, float b2, float eps, float c1, float c2,
                       int update, __nv_bfloat16* __restrict__ wf, __nv_bfloat16* __restrict__ wt,
                       float* __restrict__ bias, const int* err) {
    pdl_trigger();
    pdl_wait();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= LAYERS * LSIZE) return;
    const int l = idx / LSIZE, r = idx % LSIZE;
    const int slot = r / (C * C), o = (r / C) % C, i = r % C;
    float w = wm[idx];
    if (update && !*err && real_slot(l, slot, o, i)) {
        const float g = grad[idx];
        const float m = b1 * m1[idx] + (1.0f - b1) * g;
        const float v = b2 * m2[idx] + (1.0f - b2) * g * g;
        m1[idx] = m;
        m2[idx] = v;
        w -= lr * (m / c1) / (sqrtf(v / c2) + eps);
        wm[idx] = w;
    }
    if (slot < 27) {
        const __nv_bfloat16 wb = __float2bfloat16_rn(w);
        wf[((size_t)l * 27 + slot) * C * C + o * C + i] = wb;
        wt[((size_t)l * 27 + (26 - slot)) * C * C + i * C + o] = wb;
    } else if (i == 0) {
        bias[l * C + o] = w;
    }
}

// x[v][c] = bf16(psi[v][c] / s_in) for c < 3, zero for the other five channels; one thread per stored voxel.
__global__ void k_pack_input(const float* psi, int n, float inv_s, __nv_bfloat16* __restrict__ x) {
    pdl_trigger();
    pdl_wait();
    const int m = n + 2, row = blockIdx.x * blockDim.y + threadIdx.y;   // stored row (z, y)
    if (row >= m * m) return;
    int y = row % m - 1, z = row / m - 1;
    y += y < 0 ? n : (y >= n ? -n : 0);
    z += z < 0 ? n : (z >= n ? -n : 0);
    const float* src = psi + ((size_t)z * n + y) * n * 3;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const int gx = i == 0 ? n - 1 : (i == n + 1 ? 0 : i - 1);
        const __nv_bfloat162 p01 = __floats2bfloat162_rn(src[3 * gx] * inv_s, src[3 * gx + 1] * inv_s);
        const __nv_bfloat162 p2z = __floats2bfloat162_rn(src[3 * gx + 2] * inv_s, 0.0f);
        reinterpret_cast<uint4*>(x)[(size_t)row * m + i] =
            make_uint4(*reinterpret_cast<const uint32_t*>(&p01), *reinterpret_cast<const uint32_t*>(&p2z), 0u, 0u);
    }
}

}  // namespace
}  // namespace nn
}  // namespace colapm

using namespace colapm::nn;

struct colapm_nn {
    int n = 0;
    size_t nv = 0;
    colapm_nn_config cfg{};
    cudaStream_t stream = nullptr;
    int steps = 0;
    int nparts = 0;                    // CTAs of a weight gradient (one per SM at most)
    int sms = 0;
    bool small = false;                // tiles of 2 planes instead of 8
    // device
    __nv_bfloat16* act[LAYERS] = {};   // act[0] = packed input (8 channels), act[l] = output of layer l (l = 1..3)
    __nv_bfloat16* dz[2] = {};         // gradient ping-pong
    // TMA boxes of each array: halo and plane of a k_conv tile, halo and tile of k_wgrad
    struct Maps { CUtensorMap halo, whalo, wtile, plane; } m_act[LAYERS], m_dz[2], m_dz_out;
    __nv_bfloat16* dz_out = nullptr;   // gradient at the network output (8 channels, 0..2 used)
    float* y = nullptr;                // scratch output [n^3][3]
    float* wm = nullptr;               // master [4][28][16][16], then the error word
    float* m1 = nullptr;
    float* m2 = nullptr;
    float* grad = nullptr;
    float* part = nullptr;             // [4][nparts][28][16][16]
    __nv_bfloat16* wf = nullptr;       // [4][27][16][16]
    __nv_bfloat16* wt = nullptr;
    float* bias = nullptr;             // [4][16]
    double* loss = nullptr;
    int* err = nullptr;                // device error word (bit 4: a bounded wait gave up, in either engine): after wm, to be read with it
    bool use_tc = false;               // tcgen05 convolutions (grid side a multiple of 128)
    long long launches = 0;
};

namespace {

#define NN_CK(x)                                  \
    do {                                          \
        if ((x) != cudaSuccess) {                 \
            (void)cudaGetLastError();             \
            return COLAPM_E_CUDA;                 \
        }                                         \
    } while (0)

// Tiles of 16 x 8 x TZ voxels. TZ = 8 gives the least halo; a grid with fewer of them than half the SMs (side
// 32 and less) is cut into planes of 2, so that up to four times as many SMs work on it: forward / training
// step at side 32 in 35 / 110 us against 43 / 135 us with TZ = 8, at side 16 in 39 / 112 against 49 / 137, but
// at side 48 (108 tiles of 8 planes) in 45 / 138 against 43 / 138.
int tiles_of(int n, int tz) { return (n / TX) * (n / TY) * (n / tz); }

template <int NT, int EPI, int TZ, int VB>
cudaError_t launch_conv(const colapm_nn* c, const ConvArgs& a, const CUtensorMap& halo, const CUtensorMap& out, const CUtensorMap& mask) {
    using S = ConvSmem<EPI, TZ, VB>;
    static colapm::GridCache cache;
    int grid = 0;
    cudaError_t e = colapm::cached_grid(cache, k_conv<NT, EPI, TZ, VB>, 32 * TZ, S::BYTES, &grid);
    if (e) return e;
    return colapm::launch_dep(true, k_conv<NT, EPI, TZ, VB>, std::min(tiles_of(c->n, TZ), grid), 32 * TZ, S::BYTES, c->stream, a, halo,
                              out, mask);
}

// VB: bytes per voxel of the input (16: the packed input or the output gradient).
template <int NT, int EPI, int VB>
cudaError_t conv(colapm_nn* c, ConvArgs a, const colapm_nn::Maps& in, const colapm_nn::Maps& out, const colapm_nn::Maps& mask) {
    a.err = c->err;
    ++c->launches;
    if (c->use_tc) {
        const int tiles = (c->n / 128) * (c->n / TC_TY) * (c->n / TC_TZ);
        static colapm::GridCache cache;
        int grid = 0;
        cudaError_t e = colapm::cached_grid(cache, k_conv_tc<EPI>, 128, TC_SMEM, &grid);
        if (e) return e;
        k_conv_tc<EPI><<<std::min(tiles, grid), 128, TC_SMEM, c->stream>>>(a, VB == 16);
        return cudaGetLastError();
    }
    return c->small ? launch_conv<NT, EPI, 2, VB>(c, a, in.halo, out.plane, mask.plane)
                    : launch_conv<NT, EPI, CONV_TZ, VB>(c, a, in.halo, out.plane, mask.plane);
}

template <bool ACT_A, int NT, int TZ, int VA, int VD>
cudaError_t launch_wgrad(colapm_nn* c, const CUtensorMap& dz, int l) {
    using S = WgradSmem<TZ, VA, VD>;
    static colapm::GridCache cache;
    int grid = 0;   // only the shared-memory attribute: the CTAs are the network's partials
    cudaError_t e = colapm::cached_grid(cache, k_wgrad<ACT_A, NT, TZ, VA, VD>, 96 * (TZ / 2), S::BYTES, &grid);
    if (e) return e;
    return colapm::launch_dep(true, k_wgrad<ACT_A, NT, TZ, VA, VD>, c->nparts, 96 * (TZ / 2), S::BYTES, c->stream, c->m_act[l].whalo,
                              dz, c->n, c->part + (size_t)l * c->nparts * LSIZE, c->err);
}

template <bool ACT_A, int NT, int VA, int VD>
cudaError_t wgrad(colapm_nn* c, const CUtensorMap& dz, int l) {
    ++c->launches;
    return c->small ? launch_wgrad<ACT_A, NT, 2, VA, VD>(c, dz, l) : launch_wgrad<ACT_A, NT, 8, VA, VD>(c, dz, l);
}

// Report (and clear) a device-side error of the network's kernels, whose word has been read.
int report_err(colapm_nn* c, int h) {
    if (!h) return COLAPM_OK;
    (void)cudaMemsetAsync(c->err, 0, sizeof(int), c->stream);
    return COLAPM_E_TIMEOUT;
}
// The same; synchronises.
int check_err(colapm_nn* c) {
    int h = 0;
    if (cudaMemcpyAsync(&h, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
        cudaStreamSynchronize(c->stream) != cudaSuccess) {
        (void)cudaGetLastError();
        return COLAPM_E_CUDA;
    }
    return report_err(c, h);
}

// Weights (padded master layout) -> bf16 copies and bias, with no update.
cudaError_t publish(colapm_nn* c) {
    const int total = LAYERS * LSIZE;
    k_adam<<<(total + 255) / 256, 256, 0, c->stream>>>(c->wm, c->m1, c->m2, c->grad, 0.f, 0.f, 0.f, 0.f, 1.f, 1.f, 0,
                                                       c->wf, c->wt, c->bias, c->err);
    ++c->launches;
    return cudaGetLastError();
}

// Forward through all four layers; with `target`, also the output gradient and the loss sum.
cudaError_t forward(colapm_nn* c, const float* psi, float* y, const float* base, const float* target) {
    const size_t nv = c->nv;
    const int rows = (c->n + 2) * (c->n + 2), bx = c->n >= 62 ? 64 : 32;
    ++c->launches;
    cudaError_t e = colapm::launch_dep(true, k_pack_input, (rows + 3) / 4, dim3(bx, 4), 0, c->stream, psi, c->n, 1.0f / c->cfg.s_in,
                                       c->act[0]);
    if (e) return e;
    for (int l = 0; l < 3; ++l) {
        ConvArgs a{};
        a.in = c->act[l];
        a.w = c->wf + (size_t)l * 27 * C * C;
        a.bias = c->bias + l * C;
        a.n = c->n;
        a.out = c->act[l + 1];
        const auto &in = c->m_act[l], &out = c->m_act[l + 1];
        e = l == 0 ? conv<2, EPI_RELU, 16>(c, a, in, out, out) : conv<2, EPI_RELU, 32>(c, a, in, out, out);
        if (e) return e;
    }
    ConvArgs a{};
    a.in = c->act[3];
    a.w = c->wf + (size_t)3 * 27 * C * C;
    a.bias = c->bias + 3 * C;
    a.n = c->n;
    a.y = y;
    a.base = base;
    a.oscale = c->cfg.s_out;
    a.wide = (reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(base) | reinterpret_cast<uintptr_t>(target)) % 16 == 0;
    if (target) {
        a.target = target;
        a.tscale = 1.0f / c->cfg.s_out;
        a.gscale = (float)(2.0 / (3.0 * (double)nv));
        a.loss = c->loss;
        a.out = c->dz_out;
    }
    return conv<1, EPI_OUT, 32>(c, a, c->m_act[3], c->m_dz_out, c->m_dz_out);
}

// Backward through all layers into per-CTA partials, then the fixed-order reduction into grad.
cudaError_t backward(colapm_nn* c) {
    cudaError_t e;
    const __nv_bfloat16* g = c->dz_out;
    const colapm_nn::Maps* gm = &c->m_dz_out;
    for (int l = 3; l >= 0; --l) {
        e = l == 3 ? wgrad<true, 1, 32, 16>(c, gm->wtile, l)
                   : (l == 0 ? wgrad<false, 1, 16, 32>(c, gm->wtile, l) : wgrad<false, 2, 32, 32>(c, gm->wtile, l));
        if (e) return e;
        if (l == 0) break;
        ConvArgs a{};
        a.in = g;
        a.w = c->wt + (size_t)l * 27 * C * C;
        a.n = c->n;
        a.mask = c->act[l];
        a.out = c->dz[l & 1];
        const colapm_nn::Maps* om = &c->m_dz[l & 1];
        e = l == 3 ? conv<2, EPI_MASK, 16>(c, a, *gm, *om, c->m_act[l]) : conv<2, EPI_MASK, 32>(c, a, *gm, *om, c->m_act[l]);
        if (e) return e;
        g = c->dz[l & 1];
        gm = om;
    }
    ++c->launches;
    return colapm::launch_dep(true, k_reduce_grads, LAYERS * LSIZE / 32, dim3(32, RG_Y), 0, c->stream, c->part, c->nparts, c->grad);
}

// Tensor maps of a stored array of (n + 2)^3 voxels of vb bytes, as 8-byte elements.
bool encode_maps(colapm_nn::Maps& m, void* p, int n, int vb, bool small) {
    const cuuint64_t e = vb / 8, s = n + 2, dims[3] = {s * e, s, s}, strides[2] = {s * vb, s * s * vb};
    auto box = [&](CUtensorMap* map, cuuint32_t x, cuuint32_t y, cuuint32_t z) {
        const cuuint32_t b[3] = {(cuuint32_t)(x * e), y, z};
        return colapm::encode_box3(map, p, dims, strides, b);
    };
    const int cz = small ? 2 : CONV_TZ, wz = small ? 2 : 8;
    return box(&m.halo, HX, HY, cz + 2) && box(&m.whalo, HX, HY, wz + 2) && box(&m.wtile, TX, TY, wz) && box(&m.plane, TX, TY, 1);
}

// Flat parameter order: per layer W[27][cout][cin] then b[cout].
template <class F>
void for_each_param(F f) {
    size_t k = 0;
    for (int l = 0; l < LAYERS; ++l) {
        for (int t = 0; t < 27; ++t)
            for (int o = 0; o < COUT[l]; ++o)
                for (int i = 0; i < CIN[l]; ++i) f(k++, (size_t)l * LSIZE + (t * C + o) * C + i);
        for (int o = 0; o < COUT[l]; ++o) f(k++, (size_t)l * LSIZE + (27 * C + o) * C);
    }
}

// He-normal initial weights from a host splitmix64 stream and Box-Muller; biases start at zero.
void init_weights(std::vector<float>& flat, unsigned long long seed) {
    unsigned long long s = seed;
    auto next = [&]() {
        unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    auto unif = [&]() { return ((double)(next() >> 11) + 0.5) * (1.0 / 9007199254740992.0); };
    size_t k = 0;
    for (int l = 0; l < LAYERS; ++l) {
        const double sd = std::sqrt(2.0 / (27.0 * CIN[l]));
        for (int j = 0; j < 27 * COUT[l] * CIN[l]; ++j) {
            const double r = std::sqrt(-2.0 * std::log(unif())), th = 6.283185307179586 * unif();
            flat[k++] = (float)(sd * r * std::cos(th));
        }
        for (int o = 0; o < COUT[l]; ++o) flat[k++] = 0.0f;
    }
}

int upload_params(colapm_nn* c, const float* flat) {
    std::vector<float> pad((size_t)LAYERS * LSIZE, 0.0f);
    for_each_param([&](size_t k, size_t slot) { pad[slot] = flat[k]; });
    NN_CK(cudaMemcpyAsync(c->wm, pad.data(), pad.size() * sizeof(float), cudaMemcpyHostToDevice, c->stream));
    NN_CK(publish(c));
    NN_CK(cudaStreamSynchronize(c->stream));
    return COLAPM_OK;
}

bool device_ptr(const void* p) {
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" {

void colapm_nn_default_config(colapm_nn_config* cfg) {
    if (!cfg) return;
    cfg->s_in = 1.0f;
    cfg->s_out = 1.0f;
    cfg->lr = 1e-3f;
    cfg->beta1 = 0.9f;
    cfg->beta2 = 0.999f;
    cfg->eps = 1e-8f;
    cfg->engine = 0;
    cfg->seed = 1;
}

int colapm_nn_create(int n, const colapm_nn_config* cfg, void* stream, colapm_nn** out) {
    if (!out) return COLAPM_E_ARG;
    *out = nullptr;
    if (!cfg || n < 16 || n > 1024 || n % 16 != 0 || !(cfg->s_in > 0.0f) || !(cfg->s_out > 0.0f) ||
        !(cfg->lr >= 0.0f) || !(cfg->beta1 >= 0.0f && cfg->beta1 < 1.0f) || !(cfg->beta2 >= 0.0f && cfg->beta2 < 1.0f) ||
        !(cfg->eps > 0.0f) || cfg->engine < 0 || cfg->engine > 1)
        return COLAPM_E_ARG;
    colapm_nn* c = new (std::nothrow) colapm_nn;
    if (!c) return COLAPM_E_NOMEM;
    c->n = n;
    c->nv = (size_t)n * n * n;
    c->cfg = *cfg;
    c->stream = static_cast<cudaStream_t>(stream);
    auto fail = [&](int code) {
        colapm_nn_destroy(c);
        return code;
    };
    int dev = 0;
    if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev)) return fail(COLAPM_E_CUDA);
    c->small = 2 * tiles_of(n, 8) < c->sms;
    c->nparts = std::min(tiles_of(n, c->small ? 2 : 8), c->sms * (c->small ? 2 : 1));
    const size_t abytes = (size_t)(n + 2) * (n + 2) * (n + 2) * C * sizeof(__nv_bfloat16);
    bool ok = true;
    for (int l = 0; l < LAYERS; ++l) ok = ok && cudaMalloc(&c->act[l], l == 0 ? abytes / 2 : abytes) == cudaSuccess;
    ok = ok && cudaMalloc(&c->dz[0], abytes) == cudaSuccess && cudaMalloc(&c->dz[1], abytes) == cudaSuccess &&
         cudaMalloc(&c->dz_out, abytes / 2) == cudaSuccess && cudaMalloc(&c->y, c->nv * 3 * sizeof(float)) == cudaSuccess;
    const size_t ps = (size_t)LAYERS * LSIZE * sizeof(float);
    ok = ok && cudaMalloc(&c->wm, ps + sizeof(int)) == cudaSuccess && cudaMalloc(&c->m1, ps) == cudaSuccess &&
         cudaMalloc(&c->m2, ps) == cudaSuccess && cudaMalloc(&c->grad, ps) == cudaSuccess &&
         cudaMalloc(&c->part, ps * c->nparts) == cudaSuccess &&
         cudaMalloc(&c->wf, (size_t)LAYERS * 27 * C * C * sizeof(__nv_bfloat16)) == cudaSuccess &&
         cudaMalloc(&c->wt, (size_t)LAYERS * 27 * C * C * sizeof(__nv_bfloat16)) == cudaSuccess &&
         cudaMalloc(&c->bias, LAYERS * C * sizeof(float)) == cudaSuccess &&
         cudaMalloc(&c->loss, sizeof(double)) == cudaSuccess;
    if (!ok) {
        (void)cudaGetLastError();
        return fail(COLAPM_E_NOMEM);
    }
    c->err = reinterpret_cast<int*>(c->wm + LAYERS * LSIZE);
    for (int l = 0; l < LAYERS; ++l) ok = ok && encode_maps(c->m_act[l], c->act[l], n, l == 0 ? 16 : 32, c->small);
    ok = ok && encode_maps(c->m_dz[0], c->dz[0], n, 32, c->small) && encode_maps(c->m_dz[1], c->dz[1], n, 32, c->small) &&
         encode_maps(c->m_dz_out, c->dz_out, n, 16, c->small);
    if (!ok) return fail(COLAPM_E_CUDA);
    c->use_tc = cfg->engine == 1 && n % 128 == 0;
    if (cudaMemsetAsync(c->err, 0, sizeof(int), c->stream) ||
        cudaMemsetAsync(c->m1, 0, ps, c->stream) ||
        cudaMemsetAsync(c->m2, 0, ps, c->stream) || cudaMemsetAsync(c->grad, 0, ps, c->stream))
        return fail(COLAPM_E_CUDA);
    std::vector<float> flat(COLAPM_NN_PARAMS);
    init_weights(flat, cfg->seed);
    const int r = upload_params(c, flat.data());
    if (r) return fail(r);
    *out = c;
    return COLAPM_OK;
}

int colapm_nn_destroy(colapm_nn* c) {
    if (!c) return COLAPM_OK;
    (void)cudaStreamSynchronize(c->stream);
    for (auto* p : c->act) cudaFree(p);
    cudaFree(c->dz[0]);
    cudaFree(c->dz[1]);
    cudaFree(c->dz_out);
    cudaFree(c->y);
    for (float* p : {c->wm, c->m1, c->m2, c->grad, c->part, c->bias}) cudaFree(p);
    cudaFree(c->wf);
    cudaFree(c->wt);
    cudaFree(c->loss);
    (void)cudaGetLastError();
    delete c;
    return COLAPM_OK;
}

int colapm_nn_set_params(colapm_nn* c, const float* params) {
    if (!c || !params) return COLAPM_E_ARG;
    NN_CK(cudaStreamSynchronize(c->stream));
    return upload_params(c, params);
}

int colapm_nn_get_params(colapm_nn* c, float* params) {
    if (!c || !params) return COLAPM_E_ARG;
    std::vector<float> pad((size_t)LAYERS * LSIZE + 1);   // the parameters and the error word
    NN_CK(cudaMemcpyAsync(pad.data(), c->wm, pad.size() * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
    NN_CK(cudaStreamSynchronize(c->stream));
    int h;
    std::memcpy(&h, &pad[(size_t)LAYERS * LSIZE], sizeof(h));
    if (int r = report_err(c, h)) return r;
    for_each_param([&](size_t k, size_t slot) { params[k] = pad[slot]; });
    return COLAPM_OK;
}

int colapm_nn_forward(colapm_nn* c, const float* psi, float* out, int add) {
    if (!c || !psi || !out || !device_ptr(psi) || !device_ptr(out) || psi == out) return COLAPM_E_ARG;
    NN_CK(forward(c, psi, out, add ? psi : nullptr, nullptr));
    return COLAPM_OK;
}

static int grads_impl(colapm_nn* c, const float* psi, const float* target, double* loss) {
    if (!c || !psi || !target || !device_ptr(psi) || !device_ptr(target)) return COLAPM_E_ARG;
    NN_CK(cudaMemsetAsync(c->loss, 0, sizeof(double), c->stream));
    NN_CK(forward(c, psi, c->y, nullptr, target));
    NN_CK(backward(c));
    if (loss) {
        double h = 0.0;
        NN_CK(cudaMemcpyAsync(&h, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        NN_CK(cudaStreamSynchronize(c->stream));
        *loss = h / (3.0 * (double)c->nv);
        return check_err(c);
    }
    return COLAPM_OK;
}

int colapm_nn_grads(colapm_nn* c, const float* psi, const float* target, float* grads, double* loss) {
    int r = grads_impl(c, psi, target, loss);
    if (r) return r;
    if (grads) {
        std::vector<float> pad((size_t)LAYERS * LSIZE);
        NN_CK(cudaMemcpyAsync(pad.data(), c->grad, pad.size() * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
        NN_CK(cudaStreamSynchronize(c->stream));
        for_each_param([&](size_t k, size_t slot) { grads[k] = pad[slot]; });
        return check_err(c);
    }
    return COLAPM_OK;
}

int colapm_nn_train_step(colapm_nn* c, const float* psi, const float* target, double* loss) {
    int r = grads_impl(c, psi, target, nullptr);
    if (r) return r;
    ++c->steps;
    const float c1 = 1.0f - std::pow(c->cfg.beta1, (float)c->steps);
    const float c2 = 1.0f - std::pow(c->cfg.beta2, (float)c->steps);
    const int total = LAYERS * LSIZE;
    ++c->launches;
    NN_CK(colapm::launch_dep(true, k_adam, (total + 255) / 256, 256, 0, c->stream, c->wm, c->m1, c->m2, c->grad, c->cfg.lr,
                             c->cfg.beta1, c->cfg.beta2, c->cfg.eps, c1, c2, 1, c->wf, c->wt, c->bias, c->err));
    if (loss) {
        double h = 0.0;
        NN_CK(cudaMemcpyAsync(&h, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        NN_CK(cudaStreamSynchronize(c->stream));
        *loss = h / (3.0 * (double)c->nv);
        return check_err(c);
    }
    return COLAPM_OK;
}

int colapm_nn_steps(colapm_nn* c) { return c ? c->steps : COLAPM_E_ARG; }

long long colapm_nn_launches(colapm_nn* c) { return c ? c->launches : (long long)COLAPM_E_ARG; }

int colapm_nn_sync(colapm_nn* c) {
    if (!c) return COLAPM_E_ARG;
    return check_err(c);
}

}  // extern "C"
