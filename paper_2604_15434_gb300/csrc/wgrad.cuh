// wgrad.cuh -- the weight and bias gradient of the U-Net's 3x3x3 periodic convolution:
//   dW[tap][ci][co] = sum_v x[v + tap][ci] dy[v][co],  db[co] = sum_v dy[v][co].
//
// A contraction over voxels with 16 to 96 channels on both sides.  Each input voxel takes part in
// all 27 taps, so what bounds it is how often the operands are read: one launch per tap and chunk
// of voxels read x and dy 27 times through L2 (5 TB/s, 0.77 ms for 16 -> 16 channels at 128^3).
// Here a block stages them once: it walks its chunk of 8192 voxels row by row with the input rows
// in a shared ring (copies two steps ahead).  Where the chunks fill the chip (KX = 3) it takes the
// rows of three planes and all 27 taps, warp (kz, ky) owning the three x taps; on small levels
// (KX = 1) one plane and the nine taps of one kz, warp (ky, kx) owning one, which makes three
// times the blocks.  Per 16 voxels of a row a warp loads its shifted A fragments (16 input channels
// x 16 voxels; the tap is an address offset) and the row's B fragments (16 voxels x CO outputs)
// with transposing ldmatrix and keeps its sums in registers until the block is done.  Shared
// memory holds [8-channel half][voxel] x 16 bytes, so the eight rows of an ldmatrix matrix are 128
// contiguous bytes.
//
// The chunk and the order in it are part of the accuracy: the tensor core's FP32 accumulation
// truncates, so an error of 1e-5 of the gradient grows with the length of the chain; 8192 voxels
// (512 products) is what the per-tap kernel used, and up to 128^3 the order is the same as well.
// (Columns marched in z with chunks cut to the number of blocks took 1.03 ms for the ten layers
// where this takes 1.6, but moved the gradient by up to 2e-5.)
//
// No pipe is full now (16 and 48 -> 16 channels at 128^3: tensor 34 and 40%, issue 47 and 54%, L1 51 and
// 60%; one m16n8k16 per six cycles and SM): it is the latency of ldmatrix and mma.sync at 15 to 23 warps
// per SM.  The tcgen05 shapes gain little at these channel counts: their M of 64 or 128 rows is 3 or
// 6 z taps of 16 channels, read again from shared memory for every in-plane tap.
// Measured at 128^3: 48 -> 16 channels 2.82 -> 0.42 ms, 96 -> 32 at 64^3 1.33 -> 0.23 ms, all ten
// layers with their biases and reductions 9.3 -> 1.7 ms of a 12.0 ms training step.
#pragma once

#include <cuda_bf16.h>

namespace pmeft {

constexpr int kWgMin = 16;        // smallest level
constexpr int kWgChunk = 8192;    // voxels per block
constexpr int kWgStep = 128;      // voxels per step: G = 128 / W rows of W = min(n, 128) voxels
constexpr int kWgThreads = 288;   // nine warps
constexpr int kWgDepth = 3;       // steps in the ring: the one being read and two arriving

// input rows in the ring: a step reads G + 2, each later one adds G
__host__ __device__ inline int wgrad_slots(int W) { return kWgDepth * (kWgStep / W) + 2; }
inline size_t wgrad_smem(int n, int CO, int KX)
{
    const int W = n < kWgStep ? n : kWgStep;
    return (size_t)KX * wgrad_slots(W) * (W + 2) * 32 + (size_t)kWgDepth * kWgStep * CO * 2;
}

__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// Grid (chunks, ci/16 * 3/KX, co/CO): the second index is the ci slice, for KX = 1 (ci slice, kz);
// chunks = n^3 / 8192 (at least one).  part[chunk][27][ci][co] and, from the blocks of index 0,
// bpart[chunk][co] receive the block's sums.  n a power of two of at least 16; x_ld, x_off, dy_ld,
// dy_off multiples of 8 (16-byte copies).
template <int CO, int KX>
__global__ void __launch_bounds__(kWgThreads, KX == 1 ? 4 : (CO == 16 ? 3 : 2))
    k_wgrad(const __nv_bfloat16* __restrict__ x, int x_ld, int x_off, const __nv_bfloat16* __restrict__ dy, int dy_ld,
            int dy_off, int n, int ci, int co, float* __restrict__ part, float* __restrict__ bpart)
{
    extern __shared__ __align__(128) unsigned char wg_raw[];
    constexpr int NT = CO / 8, DB = NT * kWgStep * 16, D = kWgDepth;  // DB: bytes of a dy slot
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // this warp's taps: (kz, ky) and kx .. kx + KX - 1; the planes staged start at z + kz0 - 1
    const int kz = KX == 3 ? warp / 3 : blockIdx.y % 3, ky = KX == 3 ? warp % 3 : warp / 3,
              kx = KX == 3 ? 0 : warp % 3, kz0 = KX == 3 ? 0 : kz, m = n - 1;
    const int W = n < kWgStep ? n : kWgStep, G = kWgStep / W, SL = wgrad_slots(W);  // row width, rows a step, ring
    const int lgW = 31 - __clz(W), w2 = W + 2;
    const unsigned RB = (unsigned)w2 * 32u;  // bytes of a ring row
    const unsigned sx = (unsigned)__cvta_generic_to_shared(wg_raw), PB = (unsigned)SL * RB,
                   sd = sx + (unsigned)KX * PB;  // PB: bytes of a plane's ring
    const int ci0 = (KX == 3 ? blockIdx.y : blockIdx.y / 3) * 16, co0 = blockIdx.z * CO;
    const bool bias = blockIdx.y == 0;
    // the chunk: rows row0 .. row0 + per (y fastest, then z) of the x segment from x0
    const int total_rows = n * n, per = min(kWgChunk / W, total_rows), chunks_per_seg = total_rows / per;
    const int x0 = ((int)blockIdx.x / chunks_per_seg) * W, row0 = ((int)blockIdx.x % chunks_per_seg) * per;

    float acc[KX][NT][4], bsum[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        bsum[j] = 0.f;
#pragma unroll
        for (int k = 0; k < KX; ++k)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[k][j][q] = 0.f;
    }
    // ldmatrix row of this lane: matrix lane / 8, row lane % 8
    const int mi = lane >> 3, mr = lane & 7;
    const unsigned la = (unsigned)((mi & 1) * w2 + (mi >> 1) * 8 + mr + kx) * 16u;  // A: channel half, voxel half, tap
    const unsigned lb = (unsigned)((mi >> 1) * kWgStep + (mi & 1) * 8 + mr) * 16u;  // B: channel group, voxel half

    // this thread's pieces of a step's G new input rows (at most 288 per plane: row, half, voxel)
    int pk[KX], pl[KX];
    unsigned pd[KX];
    const __nv_bfloat16* xsrc[KX];
#pragma unroll
    for (int i = 0; i < KX; ++i) {
        const int e = t + kWgThreads * i, pieces = 2 * G * w2, r = e % pieces, pr = r % (2 * w2), half = pr >= w2;
        pl[i] = e / pieces;
        pk[i] = pl[i] < KX ? r / (2 * w2) : G;
        pd[i] = sx + (unsigned)pl[i] * PB + (unsigned)(pr * 16);
        xsrc[i] = x + (size_t)((x0 - 1 + pr - half * w2) & m) * x_ld + x_off + ci0 + half * 8;
    }
    // rows y = q - 1 for q in [q0, q0 + cnt) (cnt <= G) of the planes around z, into ring rows q mod SL
    auto load_x = [&](int z, int q0, int cnt) {
#pragma unroll
        for (int i = 0; i < KX; ++i) {
            if (pk[i] >= cnt) continue;
            const int q = q0 + pk[i];
            const size_t v = ((size_t)((z + kz0 + pl[i] - 1) & m) * n + ((q - 1) & m)) * n;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(pd[i] + (unsigned)(q % SL) * RB),
                         "l"(xsrc[i] + v * x_ld));
        }
    };
    // the step's 128 voxels of dy from row `row` on, into slot sl
    auto load_d = [&](int row, int sl) {
        for (int e = t; e < NT * kWgStep; e += kWgThreads) {
            const int g = e % NT, p = e / NT;  // a voxel's channel groups side by side
            const size_t v = (size_t)(row + (p >> lgW)) * n + x0 + (p & (W - 1));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sd + (unsigned)(sl * DB + (g * kWgStep + p) * 16)),
                         "l"(dy + v * dy_ld + dy_off + co0 + g * 8));
        }
    };
    // step `s` of the chunk into the ring, one copy group (empty past the end of its plane's rows)
    auto issue = [&](int s, int last) {
        if (s <= last) {
            const int row = row0 + s * G;
            load_x(row / n, (row & m) + 2, G);
            load_d(row, s % D);
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    const int steps = per / G;
    int last = -1;  // last step of the plane in the ring
    for (int s = 0; s < steps; ++s) {
        const int row = row0 + s * G, y = row & m;
        if (s > last) {  // first step of a plane: its two leading rows, then the steps ahead
            last = min(steps - 1, s + (n - y) / G - 1);
            __syncthreads();  // the previous plane's last rows are read
            for (int q = 0; q < 2; q += G) load_x(row / n, y + q, min(G, 2));
            for (int d = 0; d < D - 1; ++d) issue(s + d, last);
        }
        asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 2) : "memory");
        __syncthreads();  // this step's rows landed; the last step is done with its rows
        issue(s + D - 1, last);
        const int qs = (y + ky) % SL;
        const unsigned bd = sd + (unsigned)((s % D) * DB) + lb, ax = sx + (unsigned)(kz - kz0) * PB + la;
#pragma unroll (KX == 1 ? 4 : 2)
        for (int gi = 0; gi < kWgStep / 16; ++gi) {
            const int rr = (gi * 16) >> lgW, xx = (gi * 16) & (W - 1);
            const int q = qs + rr < SL ? qs + rr : qs + rr - SL;
            unsigned b[NT / 2][4];
#pragma unroll
            for (int j = 0; j < NT / 2; ++j) ldsm_x4_t(b[j], bd + (unsigned)(2 * j * kWgStep + gi * 16) * 16u);
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                unsigned a[4];
                ldsm_x4_t(a, ax + (unsigned)q * RB + (unsigned)(xx + k) * 16u);
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const unsigned bj[2] = {b[j / 2][2 * (j & 1)], b[j / 2][2 * (j & 1) + 1]};
                    mma_bf16(acc[k][j], a, bj);
                }
            }
            if (bias && gi == warp) {  // each of eight warps adds up one group of voxels
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const unsigned w = b[j / 2][2 * (j & 1) + h];
                        bsum[j] += __uint_as_float(w << 16) + __uint_as_float(w & 0xffff0000u);
                    }
            }
        }
    }
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int k = 0; k < KX; ++k) {
        const int tap = (kz * 3 + ky) * 3 + kx + k;
        float* dst = part + (((size_t)blockIdx.x * 27 + tap) * ci + ci0) * co + co0;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const int c = j * 8 + 2 * t4;
            *reinterpret_cast<float2*>(dst + (size_t)g * co + c) = make_float2(acc[k][j][0], acc[k][j][1]);
            *reinterpret_cast<float2*>(dst + (size_t)(g + 8) * co + c) = make_float2(acc[k][j][2], acc[k][j][3]);
        }
    }
    if (!bias) return;
    __shared__ float sbias[8][CO];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        bsum[j] += __shfl_xor_sync(0xffffffffu, bsum[j], 1);
        bsum[j] += __shfl_xor_sync(0xffffffffu, bsum[j], 2);
        if (t4 == 0 && warp < 8) sbias[warp][j * 8 + g] = bsum[j];
    }
    __syncthreads();
    if (t < CO) {
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) v += sbias[q][t];
        bpart[(size_t)blockIdx.x * co + co0 + t] = v;
    }
}

// grad[i] += sum over `rows` of partials[row][i], i < count, in a fixed order: a block takes 32
// consecutive i, its eight warps an eighth of the rows each (coalesced, eight loads in flight),
// and adds the eight sums.  A thread per i alone left most of the chip idle: 41 us a call, now 5.
__global__ void __launch_bounds__(256) k_sum_rows_add(const float* __restrict__ partials, int rows, int count,
                                                      float* __restrict__ grad)
{
    __shared__ float sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const int r0 = (int)((long long)rows * w / 8), r1 = (int)((long long)rows * (w + 1) / 8);
    float s = 0.f;
    if (i < count) {
        const float* p = partials + i;
#pragma unroll 8
        for (int r = r0; r < r1; ++r) s += p[(size_t)r * count];
    }
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && i < count) {
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) v += sh[q][lane];
        grad[i] += v;
    }
}

}  // namespace pmeft
