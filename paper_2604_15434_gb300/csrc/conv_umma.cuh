// conv_umma.cuh -- the U-Net's 3x3x3 periodic convolution on the fifth-generation tensor cores:
// tcgen05.mma (BF16 x BF16 -> FP32) with the accumulator in tensor memory.
//
// Implicit GEMM per output tile of M = 128 voxels (8 in x, 16 in y, one z plane): D[128 x NT]
// = sum over taps and 16-channel input chunks of A[128 x 16] B[16 x NT], where the A rows are
// the tile's voxels shifted by the tap and B is the tap's weight block.  Both operands sit in
// shared memory in the K-major, unswizzled layout of the tensor core's descriptors: 8 rows of
// 16 bytes (8 BF16 k-values) form a 128-byte core matrix; the leading byte offset steps to the
// next 8 k, the stride byte offset to the next 8 rows.
//   A: a block marches an 8 x 16 column of tiles up z.  It keeps up to eight patch planes (10 x 18
//      voxels, periodic) in a ring, each as [chunk][k-half][y][x] x 16 bytes: eight consecutive
//      x of one patch row are a core matrix, the next y row is the next one (stride 160 bytes),
//      so the A operand of a tap is the plane z + dz with its start moved by (dy, dx); no data is
//      copied per tap, and each input plane is loaded once per column (plus two halo planes
//      per work item) instead of three times.
//   B: the layer's weights for NT output channels, resident for the block's lifetime, as
//      [in-plane tap][chunk][k-half][z tap][co] x 16 bytes (stride 128 bytes per 8 outputs).
// Roles: three warps copy input planes, one thread watches the barriers, one issues MMAs, two groups of
// four warps read finished output planes back in turn; they meet only at mbarriers, so copies, tensor
// core and epilogue run at their own pace.  What bounds it is shared memory: an MMA of N = 48 reads 4 KB
// of A and 1.5 KB of B and takes 57 cycles, one of N = 96 78.  The tensor pipe is busy 28% of the time for
// 16 -> 16 channels at 256^3, 35 for 48 -> 16, 43 for 32 -> 32 at 128^3; for 16 -> 16 at 128^3 17 to 20 (18 when
// the same warps did everything in turn, plane by plane, in 85 us a layer; now 64).  Moving the window of output
// planes costs the tensor core some 500 cycles more per input plane, which a second block on the SM
// fills where two fit (16 -> 16 channels at 256^3: one block 0.52 ms, two 0.36).
// Before -> now: 256^3 16 -> 16 channels 0.41 -> 0.36 ms, 48 -> 16 1.36 -> 0.80; 128^3 96 -> 32 0.79 -> 0.54,
// 32 -> 32 0.17 -> 0.12; the warm start of a 256^3 box with the passes fused below 5.2 -> 3.6 ms.  The epilogue
// reads a data gradient's ReLU mask as two 16-byte loads: 16 -> 48 channels at 128^3 0.195 -> 0.118 ms.
#pragma once

#include <cuda_bf16.h>

#include "internal.cuh"

namespace pmeft {

constexpr int kUmTX = 8, kUmTY = 16;                       // output tile (x, y), one z plane
constexpr int kUmPX = kUmTX + 2, kUmPY = kUmTY + 2;
constexpr int kUmPP = kUmPX * kUmPY;                       // 180 voxels per patch plane
constexpr int kUmEpi = 128, kUmLoad = 96;                  // threads of an epilogue group, copying threads
constexpr int kUmThreads = 2 * kUmEpi + 64 + kUmLoad;      // warps 0-3 and 4-7 (epilogue), 8 (MMA issue), 9-11
                                                           // (copies), 12 (lookout)
// Bound on a wait, in polls.  A poll is a shared-memory round trip at least (some 30 cycles; try_wait may sleep
// longer), so 2^22 of them are 60 ms or more.  The longest wait of a working launch is for the MMAs of the
// planes in flight: at most eight planes of 54 MMAs of 78 cycles, 34 k cycles or 16 us.
constexpr long long kUmSpin = 1ll << 22;

__device__ __forceinline__ uint32_t um_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading / stride byte offsets (all >> 4),
// the descriptor version 1 (bits 46-47), no swizzle (bits 61-63 = 0)
__device__ __forceinline__ uint64_t um_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A and B BF16 (bits 7-9
// and 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 in bits 17-22, M >> 4 in bits 24-28
constexpr uint32_t um_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void um_mma(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum));
}

__device__ __forceinline__ void um_commit(uint64_t* mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(um_smem(mbar))
                 : "memory");
}

__device__ __forceinline__ bool um_try_wait(uint64_t* mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(um_smem(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void um_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void um_cp16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}

// zero 16 FP32 columns of this warp's 32 tensor-memory lanes
__device__ __forceinline__ void um_st16_zero(uint32_t taddr)
{
    const uint32_t z = 0u;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n" ::"r"(taddr),
        "r"(z)
        : "memory");
}

__device__ __forceinline__ void um_arrive(uint64_t* mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(um_smem(mbar)) : "memory");
}

// BPS blocks share an SM's 512 tensor-memory columns; the output planes of NT columns each that a block
// holds, a power of two
template <int NT, int BPS>
constexpr int um_planes()
{
    return (NT <= 16 ? 32 : (NT <= 32 ? 16 : 8)) / BPS;
}

constexpr int kUmMaxSlots = 8;  // input planes in flight
// barriers: full and done per input slot, accumulator full and empty per output plane
constexpr int kUmBars = 2 * kUmMaxSlots + 2 * 32;

// dynamic shared memory of k_conv3d_umma for Cin input channels, NT outputs and `slots` patch planes:
// the resident weights, the planes, the barriers, the tensor-memory address, a failure flag, biases
constexpr size_t umma_smem(int nt, int cin, int slots)
{
    return (size_t)9 * (cin / 16) * 2 * 3 * nt * 16 + (size_t)slots * (cin / 16) * kUmPP * 32 + kUmBars * 8 + 16 + nt * 4;
}

// shared memory for each of `blocks` blocks on an SM (1 KB per block is the system's)
inline size_t umma_budget(int blocks) { return (size_t)(228 / blocks - 1) * 1024; }

// Output channels per launch (16, 32, 48 or 64) of a layer of ci inputs and co outputs: the widest slice
// whose resident weights fit beside two patch planes; 0 where the kernel does not take the layer.  fused:
// a launch with an UmmaFuse, whose one instantiation has 16.
constexpr int umma_slice(int ci, int co, bool fused)
{
    if (ci % 16 != 0 || co % 16 != 0) return 0;
    int nt = fused ? 16 : co;
    while ((nt > 64 || umma_smem(nt, ci, 2) > (size_t)227 * 1024) && nt % 32 == 0) nt /= 2;
    return nt <= 64 && umma_smem(nt, ci, 2) <= (size_t)227 * 1024 ? nt : 0;
}

// Where a convolution's input comes from and what else its epilogue makes (forward passes that keep
// no activations for a backward pass; null / 0 otherwise).
struct UmmaFuse {
    // the first up_chunks 16-channel chunks come from `up` on the grid of half the size (nearest
    // upsampling: voxel v reads its parent), the rest from `in`; the upsampled tensor is never stored
    const __nv_bfloat16* up = nullptr;
    int up_ld = 0, up_chunks = 0;
    // the input holds 8 channels per voxel; the chunk's other 8 are zero
    bool half = false;
    // T[v] = sum_c head[c] y[v][c] + head[16] of the rounded outputs y (NT = 16) instead of storing them
    const float* head = nullptr;
    double* T = nullptr;
};

// out[v][out_off + co0 + c] = act(sum_tap sum_ci in[v + tap][ci] W[tap][ci][co0 + c] + bias[co0 + c]),
// c < NT (NT <= 64), optionally times (mask[v][mask_off + co0 + c] > 0); bias may be null (no bias
// term).  wt: the packed weights [tap][Cin/16][Cout][16] of the whole layer (Cout outputs).
// Work item: an 8 x 16 column of outputs over zl planes (zl divides n, at most um_planes<NT, BPS>()).
//
// The block walks the input planes p = zs - 1 .. zs + zl of its column.  Input plane p feeds output
// planes p - 1, p, p + 1 through the z taps 2, 1, 0, so for each in-plane tap (dy, dx) and chunk one MMA
// of N = 3 NT (B = the three z taps' weight blocks side by side) adds its A operand, read once from
// shared memory, into all three outputs.  Output plane z keeps NT tensor-memory columns at slot z - zs,
// so the three are neighbours; at the ends of the column the window is cut to the planes that exist.
// Every MMA accumulates: the epilogue zeroes a slot as it empties it.
//
//   copying warps   wait done(slot) of the slot's last plane, copy plane p, arrive full(slot)
//   lookout         wait full(slot) and empty(p + 1) in order, publish the number of planes that are ready
//   MMA thread      read that number (one plane ahead of its use), issue plane p's MMAs, commit
//                   done(slot) and acc(p - 1), which plane p completes
//   epilogue warps  wait acc(z), read slot z, zero it, arrive empty(z), store plane z (each group every
//                   other plane)
//
// err (nullable): set to 1 if a wait gave up (bounded polls; every role then leaves, what is not
// written stays unwritten).
template <int NT, int BPS, bool FUSE>
__global__ void __launch_bounds__(kUmThreads, BPS)
    k_conv3d_umma(const __nv_bfloat16* __restrict__ in, int in_ld, int in_off, int Cin,
                  const __nv_bfloat16* __restrict__ wt, int Cout, int co0, const float* __restrict__ bias,
                  __nv_bfloat16* __restrict__ out, int out_ld, int out_off, int n, int zl, int slots, int relu,
                  const __nv_bfloat16* __restrict__ mask, int mask_ld, int mask_off, int* __restrict__ err,
                  UmmaFuse fuse)
{
    static_assert(NT % 16 == 0 && NT >= 16 && NT <= 64, "N = 3 NT of a kind::f16 MMA with M = 128");
    constexpr uint32_t kUmCols = 512 / BPS;
    extern __shared__ __align__(128) unsigned char um_raw[];
    const int kch = Cin / 16;
    const uint32_t slot_bytes = (uint32_t)kch * 2 * kUmPP * 16;
    unsigned char* sW = um_raw;                                      // [9][kch][2][3 NT] x 16 B
    unsigned char* sP = sW + (size_t)9 * kch * 2 * 3 * NT * 16;      // [slot][kch][2][PY][PX] x 16 B
    uint64_t* full = reinterpret_cast<uint64_t*>(sP + (size_t)slots * slot_bytes);
    uint64_t* done = full + kUmMaxSlots;
    uint64_t* acc = done + kUmMaxSlots;   // [32]
    uint64_t* empty = acc + 32;           // [32]
    uint32_t* tslot = reinterpret_cast<uint32_t*>(empty + 32);
    volatile int* failed = reinterpret_cast<volatile int*>(tslot + 1);
    uint32_t* ready = tslot + 2;  // input planes of this block ready for the tensor core so far
    float* sBias = reinterpret_cast<float*>(tslot + 4);  // [NT]
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t sW_s = um_smem(sW), sP_s = um_smem(sP);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(um_smem(tslot)),
                     "r"(kUmCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (t == 0) {
        *failed = 0;
        *ready = 0;
        for (int q = 0; q < kUmMaxSlots; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(um_smem(full + q)), "r"(kUmLoad));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(um_smem(done + q)), "r"(1));
        }
        for (int q = 0; q < 32; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(um_smem(acc + q)), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(um_smem(empty + q)), "r"(kUmEpi));
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");  // visible to the tensor core's arrive
    }
    if (bias)
        for (int c = t; c < NT; c += kUmThreads) sBias[c] = bias[co0 + c];
    // resident weights: 16-byte piece (tap9, chunk, half, group, c) = output co0 + c of the z tap 2 - group
    // at in-plane tap tap9 = dy * 3 + dx
    const int wpieces = 9 * kch * 2 * 3 * NT;
    for (int q = t; q < wpieces; q += kUmThreads) {
        const int c = q % NT, r = q / NT;  // r = ((tap9 * kch + ch) * 2 + half) * 3 + group
        const int g = r % 3, r2 = r / 3, half = r2 & 1, tc = r2 >> 1;
        const int tap9 = tc / kch, ch = tc - tap9 * kch, tap27 = (2 - g) * 9 + tap9;
        um_cp16(sW_s + (uint32_t)q * 16u, wt + (((size_t)tap27 * kch + ch) * Cout + co0 + c) * 16 + half * 8);
    }
    if (FUSE && fuse.half)  // the upper 8 channels of every slot, never written again
        for (int q = t; q < slots * kUmPP; q += kUmThreads)
            *reinterpret_cast<uint4*>(sP + (size_t)(q / kUmPP) * slot_bytes + (size_t)(kUmPP + q % kUmPP) * 16) =
                make_uint4(0u, 0u, 0u, 0u);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // visible to the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tslot;
    if (warp < 4) {  // every output slot starts at zero
        for (int c = 0; c < um_planes<NT, BPS>() * NT; c += 16) um_st16_zero(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c);
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");

    const int m = n - 1;
    const int tx = n / kUmTX, ty = n / kUmTY, nzs = n / zl;
    const long long items = (long long)tx * ty * nzs;
    // a bounded wait for the completion of a barrier's phase; false once any role has given up
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        for (long long it = 0; it < kUmSpin; ++it) {
            if (um_try_wait(bar, parity)) return true;
            if (*failed) return false;
        }
        *failed = 1;
        return false;
    };
    int slot = 0;            // input slot of the next plane and the parity of its use
    uint32_t round = 0;
    uint32_t use = 0;        // parity of this item's use of the output slots
    auto next_slot = [&]() {
        if (++slot == slots) {
            slot = 0;
            round ^= 1u;
        }
    };

    if (warp == 12) {
        // ---- lookout: a barrier poll costs the MMA thread some 200 cycles beside the operand reads, so this
        // thread polls and the MMA thread loads a counter whose value it needs one plane later
        if (lane == 0) {
            bool ok = true;
            uint32_t count = 0;
            for (long long item = blockIdx.x; item < items && ok; item += gridDim.x, use ^= 1u)
                for (int r = -1; r <= zl && ok; ++r) {
                    ok = wait(full + slot, round);
                    if (ok && r + 1 < zl) ok = wait(empty + (r + 1), use ^ 1u);
                    if (ok) asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(um_smem(ready)), "r"(++count) : "memory");
                    next_slot();
                }
        }
    } else if (warp >= 9) {
        // ---- copies: this thread's voxels of a plane, 48 voxels x 2 halves per pass; up to `lag` planes are
        // in flight behind the newest, then handed over in order
        const int lt = t - (2 * kUmEpi + 32), half = lt & 1;
        const int lag = slots >= 6 ? 4 : (slots >= 4 ? 2 : 1);  // less than slots: the tensor core keeps one
        int flying = 0, oldest = 0;
        auto hand_over = [&]() {
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            um_arrive(full + oldest);
            if (++oldest == slots) oldest = 0;
            --flying;
        };
        bool ok = true;
        for (long long item = blockIdx.x; item < items && ok; item += gridDim.x) {
            const int x0 = (int)(item % tx) * kUmTX, y0 = (int)((item / tx) % ty) * kUmTY,
                      zs = (int)(item / ((long long)tx * ty)) * zl;
            int off[4], offu[4];  // of the voxel in a plane, and of its parent in a coarse plane
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int v = (lt >> 1) + 48 * i, py = v / kUmPX, px = v - py * kUmPX;
                const int y = (y0 - 1 + py) & m, x = (x0 - 1 + px) & m;
                off[i] = v < kUmPP && !(FUSE && fuse.half && half) ? (y * n + x) * in_ld + in_off + half * 8 : -1;
                if (FUSE) offu[i] = ((y >> 1) * (n >> 1) + (x >> 1)) * fuse.up_ld + half * 8;
            }
            for (int p = zs - 1; p <= zs + zl; ++p) {
                ok = wait(done + slot, round ^ 1u);  // the tensor core is done with the slot's last plane
                if (!ok) break;
                const __nv_bfloat16* src = in + (size_t)(p & m) * n * n * in_ld;
                const __nv_bfloat16* srcu = FUSE ? fuse.up + (size_t)((p & m) >> 1) * (n >> 1) * (n >> 1) * fuse.up_ld : nullptr;
                const int upc = FUSE ? fuse.up_chunks : 0;
                const uint32_t dst = sP_s + (uint32_t)slot * slot_bytes + (uint32_t)(half * kUmPP + (lt >> 1)) * 16u;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (off[i] < 0) continue;
                    for (int ch = 0; ch < upc; ++ch)
                        um_cp16(dst + (uint32_t)(ch * 2 * kUmPP + 48 * i) * 16u, srcu + offu[i] + ch * 16);
                    for (int ch = upc; ch < kch; ++ch)
                        um_cp16(dst + (uint32_t)(ch * 2 * kUmPP + 48 * i) * 16u,
                                src + off[i] + (ch - upc) * 16);
                }
                asm volatile("cp.async.commit_group;\n" ::);
                ++flying;
                if (flying > lag) {
                    if (lag == 4) asm volatile("cp.async.wait_group 4;\n" ::: "memory");
                    else if (lag == 2) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
                    else asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                    hand_over();
                }
                next_slot();
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        while (flying > 0) hand_over();
    } else if (warp == 8) {
        if (lane == 0) {
            // ---- MMA issue
            // descriptors of the first A and B core matrices; the others differ only in the start
            // address field (addresses below 256 KB, so adding (offset >> 4) never carries out of it)
            const uint64_t dA0 = um_desc(sP_s, kUmPP * 16, kUmPX * 16);
            const uint64_t dB0 = um_desc(sW_s, 3 * NT * 16, 128);
            bool ok = true;
            int last = -1;  // input slot and parity of the last plane issued
            uint32_t last_round = 0;
            uint32_t have = 0, mine = 0;  // planes known to be ready, planes issued
            auto load_ready = [&]() {
                uint32_t v;
                asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(um_smem(ready)) : "memory");
                return v;
            };
            for (long long item = blockIdx.x; item < items && ok; item += gridDim.x) {
                for (int r = -1; r <= zl; ++r) {  // input plane zs + r, outputs r - 1 .. r + 1 of this column
                    for (long long it = 0; have <= mine && ok; ++it) {
                        have = load_ready();
                        ok = it < kUmSpin && !*failed;
                    }
                    if (!ok) {
                        *failed = 1;
                        break;
                    }
                    ++mine;
                    const uint32_t ahead = load_ready();  // used at the next plane
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const int z0 = max(r - 1, 0), z1 = min(r + 1, zl - 1);
                    const uint32_t idesc = um_idesc(128, (z1 - z0 + 1) * NT), d = tmem + (uint32_t)(z0 * NT);
                    const uint64_t ab = dA0 + (uint64_t)((uint32_t)slot * (slot_bytes >> 4));
                    const uint64_t bb = dB0 + (uint64_t)((z0 - (r - 1)) * NT);
                    const uint64_t bstep = (uint64_t)(kch * 2 * 3 * NT);  // one in-plane tap of B, 16-byte units
                    for (int ch = 0; ch < kch; ++ch) {
                        const uint64_t ac = ab + (uint64_t)(ch * 2 * kUmPP);
                        const uint64_t bc = bb + (uint64_t)(ch * 2 * 3 * NT);
#pragma unroll
                        for (int tap9 = 0; tap9 < 9; ++tap9) {
                            const int dy = tap9 / 3, dx = tap9 % 3;
                            um_mma(d, ac + (uint64_t)(dy * kUmPX + dx), bc + (uint64_t)tap9 * bstep, idesc, 1u);
                        }
                    }
                    um_commit(done + slot);
                    if (r >= 1) um_commit(acc + (r - 1));
                    last = slot;
                    last_round = round;
                    next_slot();
                    have = ahead;
                }
            }
            // the MMAs in flight end before the tensor memory is released (bounded, also after a failure)
            if (last >= 0)
                for (long long it = 0; it < kUmSpin; ++it)
                    if (um_try_wait(done + last, last_round)) break;
        }
    } else {
        // ---- epilogue: row warp * 32 + lane of an output plane is voxel (x0 + row % 8, y0 + row / 8)
        const int row = t & (kUmEpi - 1), group = warp >> 2;
        float hw[FUSE ? 17 : 1];
        if (FUSE && fuse.T)
#pragma unroll
            for (int q = 0; q < 17; ++q) hw[FUSE ? q : 0] = fuse.head[q];
        bool ok = true;
        for (long long item = blockIdx.x; item < items && ok; item += gridDim.x, use ^= 1u) {
            const int x0 = (int)(item % tx) * kUmTX, y0 = (int)((item / tx) % ty) * kUmTY,
                      zs = (int)(item / ((long long)tx * ty)) * zl;
            const size_t v0 = ((size_t)zs * n + y0 + (row >> 3)) * n + x0 + (row & 7);
            for (int z = group; z < zl; z += 2) {
                ok = wait(acc + z, use);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t ts = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(z * NT);
                float d[NT];
#pragma unroll
                for (int c0 = 0; c0 < NT; c0 += 16) {
                    float d16[16];
                    um_ld16(ts + (uint32_t)c0, d16);
                    um_st16_zero(ts + (uint32_t)c0);
#pragma unroll
                    for (int q = 0; q < 16; ++q) d[c0 + q] = d16[q];
                }
                asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                um_arrive(empty + z);
                const size_t v = v0 + (size_t)z * n * n;
#pragma unroll
                for (int c0 = 0; c0 < NT; c0 += 16) {
                    __align__(16) __nv_bfloat16 o[16];
                    __align__(16) __nv_bfloat16 mk[16];
                    if (mask) {
                        const uint4* src = reinterpret_cast<const uint4*>(mask + v * mask_ld + mask_off + co0 + c0);
                        reinterpret_cast<uint4*>(mk)[0] = src[0];
                        reinterpret_cast<uint4*>(mk)[1] = src[1];
                    }
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        float y = bias ? d[c0 + q] + sBias[c0 + q] : d[c0 + q];  // no bias in the backward-data convolution
                        if (relu) y = fmaxf(y, 0.f);
                        if (mask && !(__bfloat162float(mk[q]) > 0.f)) y = 0.f;
                        o[q] = __float2bfloat16(y);
                    }
                    if (FUSE && fuse.T) {  // the head's sum, in its own kernel's order
                        float h = hw[FUSE ? 16 : 0];
#pragma unroll
                        for (int q = 0; q < 16; ++q) h += hw[FUSE ? q : 0] * __bfloat162float(o[q]);
                        fuse.T[v] = (double)h;
                        continue;
                    }
                    uint4* dst = reinterpret_cast<uint4*>(out + v * out_ld + out_off + co0 + c0);
                    dst[0] = reinterpret_cast<const uint4*>(o)[0];
                    dst[1] = reinterpret_cast<const uint4*>(o)[1];
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (t == 0 && *failed && err) atomicExch(err, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kUmCols));
}

}  // namespace pmeft
