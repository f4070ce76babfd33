// Passes of the blocked layout whose tiles are moved by TMA boxes (force and P(k) along z, force along y), and, for 1024
// (32 x 32) and 512 points (16 x 32), 32-point transforms on pairs of lanes.
//
// The two-stage z pass gives every radix-32 task to one thread, which then holds 32 complex
// values: with the saved base in shared memory that allows 12 warps per SM. Here a task is split
// over a pair of threads (h = 0, 1), each holding 16 values, so that twice as many warps fit.
// A 32-point DFT of a pair is a radix-2 step between the two threads and a 16-point DFT in each:
//
//  - decimation in time (inputs r = 2m + h, thread h; the DIT form): each thread transforms its
//    16 inputs (E = DFT16 of the even inputs in thread 0, O = of the odd ones in thread 1), then
//    X[k] = E[k] + W^k O[k] and X[k + 16] = E[k] - W^k O[k] (W = exp(S 2 pi i / 32)). Thread h
//    finishes k = i + 8h (i < 8): it needs the other thread's E[k] or O[k] for those k, so each
//    sends 8 values. Thread h ends with outputs r = i + 8h + 16e in slot q = i + 8e.
//  - decimation in frequency (inputs in that same distribution, r = i + 8h + 16e): the first
//    butterfly pairs r = k and k + 16, both in the same thread: Y0[k] = x[k] + x[k + 16],
//    Y1[k] = (x[k] - x[k + 16]) W^k. Thread 0 then collects Y0 (k < 16) and thread 1 Y1, 8 values
//    each way, and a 16-point DFT gives X[2m + h] in slot m.
//
// Every branch on h is a select between two values computed by both threads, so a warp never
// diverges. Each exchange is split into a `send` half (what this thread gives its partner) and a
// `finish` half (given what it received) per butterfly index, so that a host program can emulate
// a pair with the kernel's own arithmetic.
#pragma once

#include "fft2.cuh"
#include "tma.cuh"

namespace colapm {

__host__ __device__ __forceinline__ float2 csel(bool p, float2 a, float2 b) { return p ? a : b; }

// Output r of the DIT form held in slot q by thread h.
__host__ __device__ __forceinline__ int pair_dit_r(int q, int h) { return (q & 7) + 8 * h + 16 * (q >> 3); }

// DIT, one butterfly index i < 8 at a time: v = DFT16 of this thread's 16 inputs (E for h = 0,
// O for h = 1). dit_send gives the partner E[i + 8] (h = 0) or O[i] (h = 1); dit_finish, given the
// partner's value, leaves X[i + 8h] in v[i] and X[i + 8h + 16] in v[i + 8]. Index i touches only
// v[i] and v[i + 8], so the pairs can be exchanged one at a time.
__host__ __device__ __forceinline__ float2 pair_dit_send(const float2* v, int h, int i) {
    return csel(h != 0, v[i], v[i + 8]);
}
template <int S>
__host__ __device__ __forceinline__ void pair_dit_finish(float2* v, int h, int i, float2 recv) {
    const float2 e = csel(h != 0, recv, v[i]);       // E[i + 8h]
    const float2 o = csel(h != 0, v[i + 8], recv);   // O[i + 8h]
    const float2 w = csel(h != 0, root<32, S>(i + 8), root<32, S>(i));
    const float2 t = cmul(o, w);
    v[i] = cadd(e, t);       // X[i + 8h]
    v[i + 8] = csub(e, t);   // X[i + 8h + 16]
}

// DIF, one index i < 8 at a time: v holds x[r] for r = pair_dit_r(q, h) in slot q. dif_send makes
// the butterfly of k = i + 8h (Y0[k] = x[k] + x[k + 16] in v[i], Y1[k] = (x[k] - x[k + 16]) W^k
// in v[i + 8]) and gives the partner Y1[i] (h = 0) or Y0[i + 8] (h = 1); dif_finish puts the
// partner's value in place, so that v holds Y_h[0..15]; pair_dif_dft then leaves X[2m + h] in v[m].
template <int S>
__host__ __device__ __forceinline__ float2 pair_dif_send(float2* v, int h, int i) {
    const float2 a = v[i], b = v[i + 8];
    const float2 w = csel(h != 0, root<32, S>(i + 8), root<32, S>(i));
    v[i] = cadd(a, b);
    v[i + 8] = cmul(csub(a, b), w);
    return csel(h != 0, v[i], v[i + 8]);
}
__host__ __device__ __forceinline__ void pair_dif_finish(float2* v, int h, int i, float2 recv) {
    v[i] = csel(h != 0, recv, v[i]);              // Y_h[i]
    v[i + 8] = csel(h != 0, v[i + 8], recv);      // Y_h[i + 8]
}
template <int S>
__host__ __device__ __forceinline__ void pair_dif_dft(float2* v) { dft<16, S, true>(v); }

// Twiddles of stage B for task j, inputs r = 2m + h: v[m] *= w^(S j r), w = exp(-2 pi i / L), from
// the tables w^(8 M j) (M = r >> 3 = m >> 2) and the powers w^(k j), k = r & 7 = 2 (m & 3) + h. The force passes
// take the powers from a table (Tw8): as products of w^2j they are further off than the chain of a thread that holds
// the whole task (512 points: rms error of a transform 1.42e-7 against 1.33e-7, with the table 1.14e-7; force at 512^3 4.07e-7,
// 4.06e-7, now 3.82e-7 in the same time). P(k) keeps the products (512^3: 2.24e-7; 2.34e-7 with the table, which
// takes more of a line's power; 2.27e-7 by one thread per task).
template <int S>
__host__ __device__ __forceinline__ void pair_powers(float2* q, const Tw2* t, int j, int h) {
    float2 w1 = t->w1[j];
    if (S > 0) w1 = cconj(w1);
    const float2 w2 = cmul(w1, w1);
    q[0] = csel(h != 0, w1, make_float2(1.0f, 0.0f));
#pragma unroll
    for (int i = 1; i < 4; ++i) q[i] = cmul(q[i - 1], w2);
}
template <int S, int JN>
__host__ __device__ __forceinline__ void pair_powers(float2* q, const Tw8<JN>* t, int j, int h) {
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = S > 0 ? cconj(t->w[2 * i + h][j]) : t->w[2 * i + h][j];
}
template <int S, class TW>
__host__ __device__ __forceinline__ void pair_twiddle(float2* v, const TW* t, int j, int h) {
    float2 q[4];
    pair_powers<S>(q, t, j, h);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        float2 w = q[m & 3];
        if (m >= 4) {
            float2 b = t->w8[m >> 2][j];
            if (S > 0) b = cconj(b);
            w = cmul(b, w);
        }
        v[m] = cmul(v[m], w);
    }
}

#ifdef __CUDACC__
__device__ __forceinline__ float2 pair_swap(float2 a) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, 16), __shfl_xor_sync(0xffffffffu, a.y, 16));
}
// The exchanges on the device: every send first, then the shuffles, then every finish (the same
// arithmetic as index by index; measured faster than interleaving them at 2 CTAs per SM).
template <int S>
__device__ __forceinline__ void pair_dit(float2* v, int h) {
    float2 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = pair_dit_send(v, h, i);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = pair_swap(x[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) pair_dit_finish<S>(v, h, i, x[i]);
}
template <int S>
__device__ __forceinline__ void pair_dif(float2* v, int h) {
    float2 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = pair_dif_send<S>(v, h, i);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = pair_swap(x[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) pair_dif_finish(v, h, i, x[i]);
    pair_dif_dft<S>(v);
}

// ---------------------------------------------------------------------------------------------
// Force z pass, 1024-point lines, blocked layout, 4-column tiles, 256 threads: thread
// c = tid & 3, h = (tid >> 4) & 1, j = the other bits is half h of task j of column c. The partner is
// lane ^ 16, so that the 16 lanes of a shared-memory phase are 4 columns x 4 tasks of one half: with the
// exchange buffer's pitch (4 mod 16) they fall on 16 different 8-byte banks (as lane ^ 4 the halves met two
// by two: 4.93 ms per pass at 1024^3, then 4.59, and 3.39 with the boxes below). The chain is that of k2_fz<1024, Z_FORCE, 4, true>: forward
// z (stage A DIT from global memory, exchange, stage B DIT), the Green's function with CIC deconvolution,
// the saved base B = k_z A in shared memory, and two inverse z transforms (stage A DIF, exchange, stage B
// DIT) written as the bases A' (field 0) and B' (field 2).
constexpr int PZ_T = 256;

// Tile t of the blocked layout: its columns (ky, kx0 .. kx0 + 3) as in k2_fz, and its place in the tensor maps.
template <int L>
__device__ __forceinline__ void pair_tile(int t, int& ky, int& kx0) {
    constexpr int n = L / 2;
    const int q = t >> 3;
    ky = 8 * (q / (2 * (n / 8))) + (t & 7);
    kx0 = ((q / 2) % (n / 8)) * 8 + (q % 2) * 4;
}

// The tile buffer: [z][4 columns] dense in shared memory, moved by boxes of 256 z each. Through the L1 data path
// a 32-byte row costs a whole wavefront, in each direction, which was what bounded the pass (71% busy at
// 512^3); the boxes bypass it, and the tile after this one arrives while the second base is transformed.
template <int L>
__device__ __forceinline__ void pair_load(float2* buf, const CUtensorMap& map, int t, uint32_t bar) {
    int ky, kx0;
    pair_tile<L>(t, ky, kx0);
    mbar_expect(bar, L * 32);
#pragma unroll
    for (int z = 0; z < L; z += 256)
        box_load(smem_u32(buf + 4 * z), map, (ky & 7) * 8 + (kx0 & 7), z, (kx0 >> 3) * (L / 8) + (ky >> 3), bar);
}
template <int L>
__device__ __forceinline__ void pair_store(const float2* buf, const CUtensorMap& map, int ky, int kx0) {
#pragma unroll
    for (int z = 0; z < L; z += 256)
        box_store(map, (ky & 7) * 8 + (kx0 & 7), z, (kx0 >> 3) * (L / 8) + (ky >> 3), smem_u32(buf + 4 * z));
}
// Green's function with the CIC window at index z of a column: gnorm / (k^2 W^d), 0 on excluded modes (nxy2 and wxy: the
// column's nx^2 + ny^2 and window factor). A table of it per z in shared memory took the L1 that the window
// factors live in, and was slower.
template <int L>
__device__ __forceinline__ float green_at(int z, int nz, int nxy2, float wxy, bool nyq_y, const float* __restrict__ sinc2,
                                          int deconv, float gnorm) {
    const float kf = 6.283185307179586f / (float)L;
    const int n2 = nxy2 + nz * nz;   // 0 only at k = 0
    float w = 1.0f;
    if (deconv) {
        w = wxy * sinc2[z];
        if (deconv == 2) w *= w;
    }
    // fast division (within 2 ulp; k^2 W is far from the range where it flushes)
    return !nyq_y && z != L / 2 && n2 != 0 ? __fdividef(gnorm, kf * kf * (float)n2 * w) : 0.0f;
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

template <int MINB>
__global__ void __launch_bounds__(PZ_T, MINB)
    k2_fz_pair(const __grid_constant__ CUtensorMap f0, const __grid_constant__ CUtensorMap f2, const float2* __restrict__ tw,
               const float* __restrict__ sinc2, int deconv, float gnorm, int* err) {
    constexpr int L = 1024, R = 32, n = L / 2, C = 4, NTILE = (n / C) * L;
    using X = Xch<L, R, C>;
    extern __shared__ __align__(128) float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    float2* save = xb + X::SIZE;   // the saved base, then the tile of the second output
    float2* buf = save + X::SIZE;  // the input tile, then that of the first output
    static_assert(X::SIZE * sizeof(float2) % 128 == 0 && X::SIZE >= L * C, "box copies start at multiples of 128 bytes");
    auto* tws = reinterpret_cast<Tw8<32>*>(buf + L * C);
    const uint32_t bar = smem_u32(tws + 1);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, PZ_T);
    if (threadIdx.x == 0) {
        mbar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_wait();
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.x < NTILE) pair_load<L>(buf, f0, blockIdx.x, bar);
    const float kf = 6.283185307179586f / (float)L;
    const int tid = threadIdx.x, c = tid & 3, h = (tid >> 4) & 1, j = ((tid >> 2) & 3) + 4 * (tid >> 5);
    uint32_t phase = 0;
    for (int t = blockIdx.x; t < NTILE; t += gridDim.x, phase ^= 1) {
        int ky, kx0;
        pair_tile<L>(t, ky, kx0);
        const int ny = sbin(ky, L), nx = kx0 + c;
        const bool nyq_y = ky == L / 2;
        float2 v[16];
        // forward stage A: inputs z = j + 32 r, r = 2m + h
        bool ok = mbar_wait(bar, phase);
        if (!ok) {   // flag it, let the copy land, stop
            atomicOr(err, 4);
            mbar_wait(bar, phase);
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = buf[(j + R * (2 * m + h)) * C + c];
        dft<16, -1, true>(v);
        pair_dit<-1>(v, h);
#pragma unroll
        for (int q = 0; q < 16; ++q) xb[X::at(c, j * R + pair_dit_r(q, h))] = v[q];
        if (tid == 0) box_stores_read();   // the last tile's second output has left `save`
        if (!__syncthreads_and(ok)) break;
        // forward stage B: inputs j + 32 r, r = 2m + h; outputs X[j + 32 r], r = pair_dit_r(q, h)
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = xb[X::at(c, j + R * (2 * m + h))];
        pair_twiddle<-1>(v, tws, j, h);
        dft<16, -1, true>(v);
        pair_dit<-1>(v, h);
        // bases: A = g X, B = k_z A; g = gnorm / (k^2 W^d), 0 on excluded modes
        {
            const int nxy2 = nx * nx + ny * ny;
            const float wxy = deconv ? sinc2[nx] * sinc2[ky] : 1.0f;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int z = j + R * pair_dit_r(q, h), nz = sbin(z, L);
                v[q] = cscale(v[q], green_at<L>(z, nz, nxy2, wxy, nyq_y, sinc2, deconv, gnorm));
                save[X::at(c, z)] = cscale(v[q], kf * (float)nz);
            }
        }
        __syncthreads();   // forward exchange buffer free
#pragma unroll 1
        for (int bi = 0; bi < 2; ++bi) {
            if (bi > 0) {
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = save[X::at(c, j + R * pair_dit_r(q, h))];
            }
            // inverse stage A (DIF): outputs 2m + h of task j
            pair_dif<+1>(v, h);
#pragma unroll
            for (int m = 0; m < 16; ++m) xb[X::at(c, j * R + 2 * m + h)] = v[m];
            if (bi > 0 && tid == 0) {   // the first output has left the tile buffer: the next tile
                box_stores_read();
                if (t + (int)gridDim.x < NTILE) pair_load<L>(buf, f0, t + gridDim.x, bar);
            }
            __syncthreads();
            // inverse stage B: inputs j + 32 r, r = 2m + h; outputs z = j + 32 pair_dit_r(q, h)
#pragma unroll
            for (int m = 0; m < 16; ++m) v[m] = xb[X::at(c, j + R * (2 * m + h))];
            pair_twiddle<+1>(v, tws, j, h);
            dft<16, +1, true>(v);
            pair_dit<+1>(v, h);
            float2* dst = bi == 0 ? buf : save;
#pragma unroll
            for (int q = 0; q < 16; ++q) dst[(j + R * pair_dit_r(q, h)) * C + c] = v[q];
            fence_async_smem();
            __syncthreads();   // the output tile is complete, the exchange buffer free for the next base / tile
            if (tid == 0) pair_store<L>(dst, bi == 0 ? f0 : f2, ky, kx0);
        }
    }
    if (tid == 0) box_stores_done();
}

// ---------------------------------------------------------------------------------------------
// The same pass for 512-point lines (L = 16 x 32): the radix-16 stages keep one thread per task, the radix-32 ones
// use a pair, so that all 128 threads of a 4-column tile work in every stage with 16 values each. With one
// thread per task the radix-32 stages left half of the threads waiting at the barrier and held 32
// values: 530 us at 512^3 with 3 CTAs per SM, 457 with 4, 364 with the boxes (500 with 5, 587 with 6: more tiles in flight
// only queue for the L1 data path, which is 71% busy; a 32-byte row of the mesh costs it as much as
// 128 bytes of shared memory).
constexpr int PZ5_T = 128, PZ5_MINB = 4;

static __global__ void __launch_bounds__(PZ5_T, PZ5_MINB)
    k2_fz_pair512(const __grid_constant__ CUtensorMap f0, const __grid_constant__ CUtensorMap f2, const float2* __restrict__ tw,
                  const float* __restrict__ sinc2, int deconv, float gnorm, int* err) {
    constexpr int L = 512, RA = 16, RB = 32, n = L / 2, C = 4, NTILE = (n / C) * L;
    using XF = Xch<L, RA, C>;   // forward exchange (and the saved base)
    using XI = Xch<L, RB, C>;   // inverse exchange
    constexpr int XS = XF::SIZE > XI::SIZE ? XF::SIZE : XI::SIZE;
    static_assert(XS * sizeof(float2) % 128 == 0 && XF::SIZE * sizeof(float2) % 128 == 0 && XF::SIZE >= L * C, "box copies");
    extern __shared__ __align__(128) float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    float2* save = xb + XS;            // the saved base, then the tile of the second output
    float2* buf = save + XF::SIZE;     // the input tile, then that of the first output
    auto* tws = reinterpret_cast<Tw8<32>*>(buf + L * C);
    const uint32_t bar = smem_u32(tws + 1);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, PZ5_T);
    if (threadIdx.x == 0) {
        mbar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_wait();
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.x < NTILE) pair_load<L>(buf, f0, blockIdx.x, bar);
    const float kf = 6.283185307179586f / (float)L;
    const int tid = threadIdx.x, c = tid & 3;
    const int ja = tid >> 2;                                                              // radix-16 task (32 of them)
    const int h = (tid >> 4) & 1, jb = ((tid >> 2) & 3) + 4 * (tid >> 5);                 // half of a radix-32 task (16)
    uint32_t phase = 0;
    for (int t = blockIdx.x; t < NTILE; t += gridDim.x, phase ^= 1) {
        int ky, kx0;
        pair_tile<L>(t, ky, kx0);
        const int ny = sbin(ky, L), nx = kx0 + c;
        const bool nyq_y = ky == L / 2;
        float2 v[16];
        // forward stage A: inputs z = ja + 32 r
        bool ok = mbar_wait(bar, phase);
        if (!ok) {   // flag it, let the copy land, stop
            atomicOr(err, 4);
            mbar_wait(bar, phase);
        }
#pragma unroll
        for (int r = 0; r < RA; ++r) v[r] = buf[(ja + RB * r) * C + c];
        dft<RA, -1, true>(v);
#pragma unroll
        for (int r = 0; r < RA; ++r) xb[XF::at(c, ja * RA + r)] = v[r];
        if (tid == 0) box_stores_read();   // the last tile's second output has left `save`
        if (!__syncthreads_and(ok)) break;
        // forward stage B: inputs jb + 16 r, r = 2m + h; outputs X[jb + 16 r], r = pair_dit_r(q, h)
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = xb[XF::at(c, jb + RA * (2 * m + h))];
        pair_twiddle<-1>(v, tws, jb, h);
        dft<16, -1, true>(v);
        pair_dit<-1>(v, h);
        // bases: A = g X, B = k_z A; g = gnorm / (k^2 W^d), 0 on excluded modes
        const int nxy2 = nx * nx + ny * ny;
        const float wxy = deconv ? sinc2[nx] * sinc2[ky] : 1.0f;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int z = jb + RA * pair_dit_r(q, h), nz = sbin(z, L);
            v[q] = cscale(v[q], green_at<L>(z, nz, nxy2, wxy, nyq_y, sinc2, deconv, gnorm));
            save[XF::at(c, z)] = cscale(v[q], kf * (float)nz);
        }
        __syncthreads();   // forward exchange buffer free
#pragma unroll 1
        for (int bi = 0; bi < 2; ++bi) {
            if (bi > 0) {
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = save[XF::at(c, jb + RA * pair_dit_r(q, h))];
            }
            // inverse stage A (radix 32, DIF): outputs 2m + h of task jb
            pair_dif<+1>(v, h);
#pragma unroll
            for (int m = 0; m < 16; ++m) xb[XI::at(c, jb * RB + 2 * m + h)] = v[m];
            if (bi > 0 && tid == 0) {   // the first output has left the tile buffer: the next tile
                box_stores_read();
                if (t + (int)gridDim.x < NTILE) pair_load<L>(buf, f0, t + gridDim.x, bar);
            }
            __syncthreads();
            // inverse stage B (radix 16): inputs and outputs ja + 32 r
            stage_b<L, RB, RA, +1, C, true>(xb, tws, c, ja, v);
            float2* dst = bi == 0 ? buf : save;
#pragma unroll
            for (int r = 0; r < RA; ++r) dst[(ja + RB * r) * C + c] = v[r];
            fence_async_smem();
            __syncthreads();   // the output tile is complete, the exchange buffer free for the next base / tile
            if (tid == 0) pair_store<L>(dst, bi == 0 ? f0 : f2, ky, kx0);
        }
    }
    if (tid == 0) box_stores_done();
}
constexpr size_t PZ5_SMEM =
    sizeof(float2) * ((size_t)(Xch<512, 16, 4>::SIZE > Xch<512, 32, 4>::SIZE ? Xch<512, 16, 4>::SIZE : Xch<512, 32, 4>::SIZE) +
                      Xch<512, 16, 4>::SIZE + 512 * 4) + sizeof(Tw8<32>) + 8;

// ---------------------------------------------------------------------------------------------
// The same pass for lines of 256, 320 and 384 points, one thread per task, tiles of 4 columns moved by boxes as above
// (one box of all 256 z, two halves above). With loads and stores through L1 (k2_fz) the pass took 52, 127 and
// 221 us on these meshes, with boxes 41, 105 and 155. The shorter lines stay with k2_fz: their meshes live in L2, and a box
// costs more than it saves (128^3: 9.9 us against 10.9).
template <int L>
struct ZBox {
    static constexpr int C = 4;                                    // columns
    static constexpr int R1 = F2<L>::R1, R2 = F2<L>::R2;
    static constexpr int TA = C * L / R1, TB = C * L / R2, T = TA > TB ? TA : TB;
    using XF = Xch<L, R1, C>;
    using XI = Xch<L, R2, C>;
    static constexpr int up(int n) { return (n + 15) / 16 * 16; }  // to 128 bytes
    static constexpr int XS = up(XF::SIZE > XI::SIZE ? XF::SIZE : XI::SIZE), SV = up(XF::SIZE), BOXZ = L <= 256 ? L : L / 2;
    static constexpr size_t SMEM = sizeof(float2) * ((size_t)XS + SV + L * C) + sizeof(Tw2) + 8;
    static constexpr int MINB = 512 / T;
};

template <int L>
__global__ void __launch_bounds__(ZBox<L>::T, ZBox<L>::MINB)
    k2_fz_box(const __grid_constant__ CUtensorMap f0, const __grid_constant__ CUtensorMap f2, const float2* __restrict__ tw,
              const float* __restrict__ sinc2, int deconv, float gnorm, int* err) {
    using Z = ZBox<L>;
    using XF = typename Z::XF;
    using XI = typename Z::XI;
    constexpr int C = Z::C, R1 = Z::R1, R2 = Z::R2, n = L / 2, NTILE = (n / C) * L;
    extern __shared__ __align__(128) float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    float2* save = xb + Z::XS;         // the saved base, then the tile of the second output
    float2* buf = save + Z::SV;        // the input tile, then that of the first output
    Tw2* tws = reinterpret_cast<Tw2*>(buf + L * C);
    const uint32_t bar = smem_u32(tws + 1);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, Z::T);
    if (threadIdx.x == 0) {
        mbar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_wait();
    __syncthreads();
    auto load = [&](int t) {
        int ky, kx0;
        pair_tile<L>(t, ky, kx0);
        mbar_expect(bar, L * C * 8);
#pragma unroll
        for (int z = 0; z < L; z += Z::BOXZ)
            box_load(smem_u32(buf + C * z), f0, (ky & 7) * 8 + (kx0 & 7), z, (kx0 >> 3) * (L / 8) + (ky >> 3), bar);
    };
    const int tid = threadIdx.x, c = tid % C, j = tid / C;
    const float kf = 6.283185307179586f / (float)L;
    if (tid == 0 && blockIdx.x < NTILE) load(blockIdx.x);
    uint32_t phase = 0;
    for (int t = blockIdx.x; t < NTILE; t += gridDim.x, phase ^= 1) {
        int ky, kx0;
        pair_tile<L>(t, ky, kx0);
        const int ny = sbin(ky, L), nx = kx0 + c;
        bool ok = mbar_wait(bar, phase);
        if (!ok) {   // flag it, let the copy land, stop
            atomicOr(err, 4);
            mbar_wait(bar, phase);
        }
        float2 v[R2];
        if (tid < Z::TA) {   // forward stage A: inputs z = j + r L / R1
            float2 a[R1];
#pragma unroll
            for (int r = 0; r < R1; ++r) a[r] = buf[(j + r * (L / R1)) * C + c];
            dft<R1, -1, true>(a);
#pragma unroll
            for (int r = 0; r < R1; ++r) xb[XF::at(c, j * R1 + r)] = a[r];
        }
        if (tid == 0) box_stores_read();   // the last tile's second output has left `save`
        if (!__syncthreads_and(ok)) break;
        if (tid < Z::TB) {   // forward stage B, then the bases A = g X (kept) and B = k_z A (saved)
            stage_b<L, R1, R2, -1, C, true>(xb, tws, c, j, v);
            const int nxy2 = nx * nx + ny * ny;
            const float wxy = deconv ? sinc2[nx] * sinc2[ky] : 1.0f;
#pragma unroll
            for (int r = 0; r < R2; ++r) {
                const int z = j + R1 * r, nz = sbin(z, L);
                v[r] = cscale(v[r], green_at<L>(z, nz, nxy2, wxy, ky == L / 2, sinc2, deconv, gnorm));
                save[XF::at(c, z)] = cscale(v[r], kf * (float)nz);
            }
        }
        __syncthreads();   // forward exchange buffer free
#pragma unroll 1
        for (int bi = 0; bi < 2; ++bi) {
            if (tid < Z::TB) {   // inverse stage A (radix R2)
                if (bi > 0) {
#pragma unroll
                    for (int r = 0; r < R2; ++r) v[r] = save[XF::at(c, j + R1 * r)];
                }
                dft<R2, +1, true>(v);
#pragma unroll
                for (int r = 0; r < R2; ++r) xb[XI::at(c, j * R2 + r)] = v[r];
            }
            if (bi > 0 && tid == 0) {   // the first output has left the tile buffer: the next tile
                box_stores_read();
                if (t + (int)gridDim.x < NTILE) load(t + gridDim.x);
            }
            __syncthreads();
            float2* dst = bi == 0 ? buf : save;
            if (tid < Z::TA) {   // inverse stage B (radix R1): outputs z = j + R2 r
                float2 u[R1];
                stage_b<L, R2, R1, +1, C, true>(xb, tws, c, j, u);
#pragma unroll
                for (int r = 0; r < R1; ++r) dst[(j + R2 * r) * C + c] = u[r];
            }
            fence_async_smem();
            __syncthreads();   // the output tile is complete, the exchange buffer free for the next base / tile
            if (tid == 0) {
#pragma unroll
                for (int z = 0; z < L; z += Z::BOXZ)
                    box_store(bi == 0 ? f0 : f2, (ky & 7) * 8 + (kx0 & 7), z, (kx0 >> 3) * (L / 8) + (ky >> 3),
                              smem_u32(dst + C * z));
            }
        }
    }
    if (tid == 0) box_stores_done();
}

// ---------------------------------------------------------------------------------------------
// Inverse y pass of the force (k2_fy_force in fft2.cuh) with tiles of 4 columns moved by boxes: A' of the tile is read once
// for its two transforms, B' arrives while the second one's stage B runs, the next tile's A' during the third one's.
// What bounded k2_fy_force was latency: 16 warps per SM at 127 registers and no load in flight while a tile is
// transformed (66 to 69% of the DRAM's cycles). From 512 points on the pass went from 512 to 464 us and, at 1024, from 3.93
// to 3.81 ms (84% of the copy bandwidth); below, the boxes lose: 53 -> 59, 111 -> 115 and 186 -> 195 us at 256, 320, 384.
#define COLAPM_FOR_FY_BOX_SIZES(X) X(512) X(1024)
template <int L>
struct FyBox {
    static constexpr int C = 4, R1 = F2<L>::R1, R2 = F2<L>::R2;
    static constexpr bool PA = R1 == 32, PB = R2 == 32;                                  // stages on pairs
    static constexpr int TA = C * L / R1 * (PA ? 2 : 1), TB = C * L / R2 * (PB ? 2 : 1), T = TA > TB ? TA : TB;
    using X = Xch<L, R1, C>;
    static constexpr int XS = (X::SIZE + 15) / 16 * 16;   // to 128 bytes
    static constexpr size_t SMEM = sizeof(float2) * ((size_t)XS + 2 * L * C) + sizeof(Tw8<32>) + 8;
    static constexpr int MINB = 512 / T;
};

template <int L>
__global__ void __launch_bounds__(FyBox<L>::T, FyBox<L>::MINB)
    k2_fy_box(const __grid_constant__ CUtensorMap f0, const __grid_constant__ CUtensorMap f1, const __grid_constant__ CUtensorMap f2,
              const float2* __restrict__ tw, int* err) {
    using Z = FyBox<L>;
    using X = typename Z::X;
    constexpr int C = Z::C, R1 = Z::R1, R2 = Z::R2, T = Z::T, n = L / 2, NTILE = (n / C) * L;
    extern __shared__ __align__(128) float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    float2* in = xb + Z::XS;            // [y][4]: A', then B'
    float2* ob = in + L * C;            // the tile of each output
    auto* tws = reinterpret_cast<Tw8<32>*>(ob + L * C);
    const uint32_t bar = smem_u32(tws + 1);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, T);
    if (threadIdx.x == 0) {
        mbar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_wait();
    __syncthreads();
    // tile t: columns kx0 .. kx0 + 3 of plane z; the two halves of a block on neighbouring CTAs
    auto load = [&](int t, const CUtensorMap& f) {
        const int q = t % (n / C);
        mbar_expect(bar, L * C * 8);
        box_load4(smem_u32(in), f, (q & 1) * 4, 0, t / (n / C), (q >> 1) * (L / 8), bar);
    };
    const int tid = threadIdx.x, c = tid & 3;
    const int js = tid >> 2, h = (tid >> 4) & 1, jp = ((tid >> 2) & 3) + 4 * (tid >> 5);   // task alone, or half of one
    const float kf = 6.283185307179586f / (float)L;
    if (tid == 0 && blockIdx.x < NTILE) load(blockIdx.x, f0);
    uint32_t phase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < NTILE && ok; t += gridDim.x) {
        const int q = t % (n / C), z = t / (n / C);
        const float kxv = kf * (float)(4 * q + c);
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {   // F_y from k_y A', F_x from A', F_z from B'
            if (pass != 1) {
                ok = mbar_wait(bar, phase);
                if (!ok) {   // flag it, let the copy land, stop
                    atomicOr(err, 4);
                    mbar_wait(bar, phase);
                }
                phase ^= 1;
            }
            auto value = [&](int y) {
                const float2 a = in[y * C + c];
                return pass == 0 ? cscale(a, kf * (float)sbin(y, L)) : a;
            };
            if constexpr (Z::PA) {
                float2 v[16];
#pragma unroll
                for (int m = 0; m < 16; ++m) v[m] = value(jp + (L / R1) * (2 * m + h));
                dft<16, +1, true>(v);
                pair_dit<+1>(v, h);
#pragma unroll
                for (int i = 0; i < 16; ++i) xb[X::at(c, jp * R1 + pair_dit_r(i, h))] = v[i];
            } else if (tid < Z::TA) {
                float2 v[R1];
#pragma unroll
                for (int r = 0; r < R1; ++r) v[r] = value(js + r * (L / R1));
                dft<R1, +1, true>(v);
#pragma unroll
                for (int r = 0; r < R1; ++r) xb[X::at(c, js * R1 + r)] = v[r];
            }
            if (tid == 0) box_stores_read();   // the output before has left `ob`
            ok = __syncthreads_and(ok);        // the tile has been read as well
            if (!ok) break;
            if (tid == 0) {
                if (pass == 1) load(t, f2);
                if (pass == 2 && t + (int)gridDim.x < NTILE) load(t + gridDim.x, f0);
            }
            const float sc = pass == 1 ? kxv : 1.0f;
            if constexpr (Z::PB) {
                float2 v[16];
#pragma unroll
                for (int m = 0; m < 16; ++m) v[m] = xb[X::at(c, jp + R1 * (2 * m + h))];
                pair_twiddle<+1>(v, tws, jp, h);
                dft<16, +1, true>(v);
                pair_dit<+1>(v, h);
#pragma unroll
                for (int i = 0; i < 16; ++i) ob[(jp + R1 * pair_dit_r(i, h)) * C + c] = make_float2(-sc * v[i].y, sc * v[i].x);
            } else if (tid < Z::TB) {
                float2 v[R2];
                stage_b<L, R1, R2, +1, C, true>(xb, tws, c, js, v);
#pragma unroll
                for (int r = 0; r < R2; ++r) ob[(js + R1 * r) * C + c] = make_float2(-sc * v[r].y, sc * v[r].x);
            }
            fence_async_smem();
            __syncthreads();   // the output tile is complete, the exchange buffer free
            if (tid == 0) {
                const CUtensorMap& f = pass == 0 ? f1 : (pass == 1 ? f0 : f2);
                box_store4(f, (q & 1) * 4, 0, z, (q >> 1) * (L / 8), smem_u32(ob));
            }
        }
    }
    if (tid == 0) box_stores_done();
}

// ---------------------------------------------------------------------------------------------
// P(k) z pass of the blocked layout at 256, 384 and 512 points: 4-column tiles by boxes, stages as in the passes above
// (the radix-32 ones on pairs), |X|^2 into shared memory, power_bin_tile. The next tile arrives during stage B and
// the binning, which bounds the pass (one search and one flush per run, three reductions in L2 each). Against
// k2_fz: 49 -> 46, 115 -> 112 and 287 -> 228 us at 256, 384 and 512 points (100 bins; before every mode had its own window,
// with which it takes 235 at 512). Not at 320 (68 -> 69), and not at
// 1024: its stages need 256 threads, and runs of 8 modes then double the reductions (1.98 -> 3.11 ms; binning by
// half of the threads 2.07; the same at 512 points 259 us).
template <int L>
struct PowBox {
    static constexpr int C = 4, R1 = F2<L>::R1, R2 = F2<L>::R2;
    static constexpr bool PA = R1 == 32, PB = R2 == 32;                                  // stages on pairs
    static constexpr int TA = C * L / R1 * (PA ? 2 : 1), TB = C * L / R2 * (PB ? 2 : 1), T = TA > TB ? TA : TB;
    using X = Xch<L, R1, C>;
    static constexpr int BOXZ = ZBox<L>::BOXZ > 256 ? 256 : ZBox<L>::BOXZ;
    static constexpr size_t SMEM = sizeof(float2) * ((size_t)L * C + X::SIZE) + sizeof(Tw2) +
                                   sizeof(float) * ((size_t)C * PowerTile<L, C, T>::PP + L / 2) + 8;   // then the thresholds
    static constexpr int MINB = 512 / T;
};

template <int L>
__global__ void __launch_bounds__(PowBox<L>::T, PowBox<L>::MINB)
    k2_power_box(const __grid_constant__ CUtensorMap f0, const float2* __restrict__ tw, const float* __restrict__ sinc2, PowerArgs pw,
                 int* err) {
    using Z = PowBox<L>;
    using X = typename Z::X;
    using P = PowerTile<L, Z::C, Z::T>;
    constexpr int C = Z::C, R1 = Z::R1, R2 = Z::R2, T = Z::T, NTILE = (L / 2 / C) * L;
    extern __shared__ __align__(128) float4 smem4[];
    float2* buf = reinterpret_cast<float2*>(smem4);
    float2* xb = buf + L * C;
    Tw2* tws = reinterpret_cast<Tw2*>(xb + X::SIZE);
    const uint32_t bar = smem_u32(tws + 1);
    float* pbuf = reinterpret_cast<float*>(tws + 1) + 2;
    float* win = pbuf + C * P::PP;
    int* lo = reinterpret_cast<int*>(win + L / 2);
    pdl_trigger();
    load_tw2<L, L>(tws, tw, T);
    if (threadIdx.x == 0) {
        mbar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    pdl_wait();
    power_tables<L>(win, lo, sinc2, pw, T);
    double* part = power_region(pw);
    __syncthreads();
    auto load = [&](int t) {
        int ky, kx0;
        pair_tile<L>(t, ky, kx0);
        mbar_expect(bar, L * C * 8);
#pragma unroll
        for (int z = 0; z < L; z += Z::BOXZ)
            box_load(smem_u32(buf + C * z), f0, (ky & 7) * 8 + (kx0 & 7), z, (kx0 >> 3) * (L / 8) + (ky >> 3), bar);
    };
    const int tid = threadIdx.x, c = tid & 3;
    const int js = tid >> 2, h = (tid >> 4) & 1, jp = ((tid >> 2) & 3) + 4 * (tid >> 5);   // task alone, or half of one
    if (tid == 0 && blockIdx.x < NTILE) load(blockIdx.x);
    uint32_t phase = 0;
    for (int t = blockIdx.x; t < NTILE; t += gridDim.x, phase ^= 1) {
        int ky, kx0;
        pair_tile<L>(t, ky, kx0);
        bool ok = mbar_wait(bar, phase);
        if (!ok) {   // flag it, let the copy land, stop
            atomicOr(err, 4);
            mbar_wait(bar, phase);
        }
        if constexpr (Z::PA) {
            float2 v[16];
#pragma unroll
            for (int m = 0; m < 16; ++m) v[m] = buf[(jp + (L / R1) * (2 * m + h)) * C + c];
            dft<16, -1, true>(v);
            pair_dit<-1>(v, h);
#pragma unroll
            for (int q = 0; q < 16; ++q) xb[X::at(c, jp * R1 + pair_dit_r(q, h))] = v[q];
        } else if (tid < Z::TA) {
            float2 v[R1];
#pragma unroll
            for (int r = 0; r < R1; ++r) v[r] = buf[(js + r * (L / R1)) * C + c];
            dft<R1, -1, true>(v);
#pragma unroll
            for (int r = 0; r < R1; ++r) xb[X::at(c, js * R1 + r)] = v[r];
        }
        if (!__syncthreads_and(ok)) break;   // the tile has been read; the last tile's values have been binned
        if (tid == 0 && t + (int)gridDim.x < NTILE) load(t + gridDim.x);
        if constexpr (Z::PB) {
            float2 v[16];
#pragma unroll
            for (int m = 0; m < 16; ++m) v[m] = xb[X::at(c, jp + R1 * (2 * m + h))];
            pair_twiddle<-1>(v, tws, jp, h);
            dft<16, -1, true>(v);
            pair_dit<-1>(v, h);
#pragma unroll
            for (int q = 0; q < 16; ++q) pbuf[P::at(c, jp + R1 * pair_dit_r(q, h))] = fmaf(v[q].x, v[q].x, v[q].y * v[q].y);
        } else if (tid < Z::TB) {
            float2 v[R2];
            stage_b<L, R1, R2, -1, C, true>(xb, tws, c, js, v);
#pragma unroll
            for (int r = 0; r < R2; ++r) pbuf[P::at(c, js + R1 * r)] = fmaf(v[r].x, v[r].x, v[r].y * v[r].y);
        }
        __syncthreads();
        if (ky != L / 2) power_bin_tile<L, C, T>(pbuf, kx0, ky, sinc2, win, lo, pw, part);
    }
    power_sum_regions(pw, T);
}

template <int MINB>
struct PairZ {
    static constexpr size_t SMEM = sizeof(float2) * (2 * (size_t)Xch<1024, 32, 4>::SIZE + 1024 * 4) + sizeof(Tw8<32>) + 8;
};
#endif

}  // namespace colapm
