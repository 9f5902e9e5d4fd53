// coarse_cluster.cuh -- the levels 32^3 .. 4^3 of the FP32 inner V-cycle in one launch: a cluster of
// 16 blocks whose shared memories hold all of them (included by mg.cu; uses its device functions).
//
// On these levels a kernel runs 2 to 10 us for well under 1 us of work: some forty launches per
// V-cycle, each with its launch gap, its loads from L2 and, for the residuals, a reduction through
// global memory.  Here block r of the cluster owns planes 2r, 2r + 1 of the 32^3 level and plane r
// of the 16^3 level, with a ghost plane on either side; the 8^3 and 4^3 levels live in block 0.
// A thread owns an x pair (a red and a black cell) of each plane, whose background coefficients,
// weights and right-hand sides stay in registers (32^3) or shared memory.  A half-sweep reads one copy of the
// iterate and writes the pair (new value, partner's old value) to the other copy, its own and the
// neighbour block's ghost plane (distributed shared memory), so one cluster barrier per half-sweep
// separates everything.  The sums of a level's gauge shift go to every block's shared memory at the
// barrier that ends the restriction.  Arithmetic per cell is that of half_sweep_cell, residual_cell,
// fas_rhs_cell and prolong_children; the sums are FP64, as those of the level-by-level kernels.
//
// One launch takes 55 us (the launches it replaces took some 160 us of a V-cycle): 12 on each side
// of it for the 32^3 sweeps, 14 for the coarsest solve.  What bounds it is latency: a few hundred
// dependent instructions per evaluation, fetched from L2 the first time (so every loop that can
// stay rolled does), and a barrier after each.
#pragma once

#include <cooperative_groups.h>

namespace pmeft {

constexpr int kClBlocks = 16, kClThreads = 512;

struct ClusterParams {
    float* u;             // 32^3 iterate, updated in place
    const float* f;       // its right-hand side
    const float* bg;      // its background
    const uint8_t* kmask;
    const int* active;    // null, or 0 once the box has converged: the launch does nothing
    float nu, kap, lsat_c;
    double nu_d, kap_d, eta;
    int npre, npost, coarse_sweeps;
};

// what a cell keeps through the cycle: the background's second and cross differences, kappa and
// L_sat with the cell's weight, the right-hand side
struct ClCell {
    float Xb, Yb, Zb, bxy, bxz, byz, kc, lsat, f;
};

struct ClSmem {
    float u32[2][4][1024];  // planes 2r - 1 .. 2r + 2
    float bg32[4][1024];
    float r32[2][1024];
    float u16[2][3][256], ur16[3][256], bg16[3][256];  // planes r - 1 .. r + 1
    float rs16[256], d8[3][64];  // d8: the 8^3 corrections around this block's plane
    ClCell c16[256];
    // block 0; h8: the 16^3 planes' parts of the 8^3 cells (iterate, raw residual, background)
    float h8[3][2][512];
    uint8_t hc8[2][512], hn8[2][512];
    float u8[2][512], ur8[512], bg8[512], r8[512], e8[512];
    ClCell c8[512];
    float u4[64], ur4[64], bg4[64], f4[64];
    CoarsestSmem<float> cs;
    double wsum[128], csum[2][kClBlocks];  // csum, ccnt: of the 32^3 and of the 16^3 level
    int wcnt[kClThreads / 32], ccnt[2][kClBlocks];
    float gm;
    uint8_t km32[2][1024], fl32[2][1024], km16[256], nun16[256], km8[512], fl8[512], km4[64];
};

// named directly wherever it is used (a reference to it, captured by the kernel's lambdas, would turn
// every access into a generic one)
extern __shared__ ClSmem cl_s[];

__device__ __forceinline__ ClCell cl_cell(const Stencil<float>& b, float kap, float lsat_c, int k)
{
    ClCell c;
    c.Xb = b.ax - 2.f * b.c0;
    c.Yb = b.ay - 2.f * b.c0;
    c.Zb = b.az - 2.f * b.c0;
    c.bxy = b.exy;
    c.bxz = b.exz;
    c.byz = b.eyz;
    const float w = k >= 8 ? 0.f : (float)(8 - k) * 0.125f;
    c.kc = kap * w;
    c.lsat = c.kc != 0.f ? lsat_c / w : 0.f;
    c.f = 0.f;
    return c;
}

// local_eval<float, true> from the cell's constants
__device__ __forceinline__ Local<float> cl_eval(const Stencil<float>& s, const ClCell& b, float ih2, float nu, float rhs)
{
    const float X = s.ax - 2.f * s.c0, Y = s.ay - 2.f * s.c0, Z = s.az - 2.f * s.c0;
    Local<float> o;
    const float L1 = X + Y + Z;
    float q2 = 2.f * (X * Y + Y * Z + Z * X) - 0.125f * (s.exy * s.exy + s.exz * s.exz + s.eyz * s.eyz);
    q2 += 2.f * (b.Xb * (Y + Z) + b.Yb * (X + Z) + b.Zb * (X + Y)) -
          0.25f * (b.bxy * s.exy + b.bxz * s.exz + b.byz * s.eyz);
    o.L = (L1 + (b.Xb + b.Yb + b.Zb)) * ih2;
    o.g = b.kc != 0.f ? b.lsat - o.L : 0.f;
    const float nu1 = nu * ih2, kap1 = b.kc * ih2 * ih2;
    o.G = nu1 * L1 - kap1 * q2 - rhs;
    o.Ep = (-6.f * nu + 8.f * b.kc * o.L) * ih2;
    o.P = -24.f * kap1;
    o.D = o.Ep * o.Ep - 4.f * o.P * o.G;
    return o;
}

// the red (q = 0) or black cell of a pair kept in registers
__device__ __forceinline__ ClCell cl_pick(const ClCell (&k)[2], int q)
{
    ClCell c;
    c.Xb = q ? k[1].Xb : k[0].Xb;
    c.Yb = q ? k[1].Yb : k[0].Yb;
    c.Zb = q ? k[1].Zb : k[0].Zb;
    c.bxy = q ? k[1].bxy : k[0].bxy;
    c.bxz = q ? k[1].bxz : k[0].bxz;
    c.byz = q ? k[1].byz : k[0].byz;
    c.kc = q ? k[1].kc : k[0].kc;
    c.lsat = q ? k[1].lsat : k[0].lsat;
    c.f = q ? k[1].f : k[0].f;
    return c;
}

// the residual of a coarse cell (residual_cell without the finest level's floored piece)
__device__ __forceinline__ float cl_resid(const Local<float>& o, float nu, bool& fl)
{
    fl = (o.P != 0.f) && (o.D < 0.f);
    return fl ? nu * o.g : -o.G;
}

// load_stencil on an N x N plane and the planes below and above it
template <int N>
__device__ __forceinline__ Stencil<float> cl_stencil(const float* lo, const float* at, const float* hi, int i, int j)
{
    const int ip = (i + 1) & (N - 1), im = (i - 1) & (N - 1), r = j * N, rp = ((j + 1) & (N - 1)) * N,
              rm = ((j - 1) & (N - 1)) * N;
    Stencil<float> s;
    s.c0 = at[r + i];
    s.ax = at[r + ip] + at[r + im];
    s.ay = at[rp + i] + at[rm + i];
    s.az = hi[r + i] + lo[r + i];
    s.exy = at[rp + ip] - at[rm + ip] - at[rp + im] + at[rm + im];
    s.exz = hi[r + ip] - lo[r + ip] - hi[r + im] + lo[r + im];
    s.eyz = hi[rp + i] - lo[rp + i] - hi[rm + i] + lo[rm + i];
    return s;
}

// The four children in one fine plane of coarse column (I, J): near and far are the coarse planes
// of weight 3/4 and 1/4 (prolong_children's order); put(dy, dx, value).
template <int N, typename D, typename Put>
__device__ __forceinline__ void cl_prolong_plane(int I, int J, D&& d, Put&& put)
{
    const int xs[3] = {(I - 1) & (N - 1), I, (I + 1) & (N - 1)}, ys[3] = {(J - 1) & (N - 1), J, (J + 1) & (N - 1)};
    auto mix = [](float near, float far) { return 0.75f * near + 0.25f * far; };
    float py[2][2][2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {  // near, far
        float px[3][2];
#pragma unroll
        for (int jy = 0; jy < 3; ++jy) {
            const float v0 = d(k, ys[jy] * N + xs[0]), v1 = d(k, ys[jy] * N + xs[1]), v2 = d(k, ys[jy] * N + xs[2]);
            px[jy][0] = mix(v1, v0);
            px[jy][1] = mix(v1, v2);
        }
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) py[k][dy][dx] = mix(px[1][dx], px[dy ? 2 : 0][dx]);
    }
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int dx = 0; dx < 2; ++dx) put(dy, dx, mix(py[0][dy][dx], py[1][dy][dx]));
}

__global__ void __launch_bounds__(kClThreads, 1) k_coarse_cluster(ClusterParams P)
{
    namespace cg = cooperative_groups;
    if (P.active && *P.active == 0) return;  // every block alike, before any barrier
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), t = threadIdx.x, lane = t & 31, wid = t >> 5;
    ClSmem* below = cl.map_shared_rank(&cl_s[0], (rank + kClBlocks - 1) % kClBlocks);  // owns plane 2r - 1
    ClSmem* above = cl.map_shared_rank(&cl_s[0], (rank + 1) % kClBlocks);
    const float sp = P.nu >= 0.f ? -1.f : 1.f;
    auto floor_of = [&](int n) {  // the smoother's floor on the discriminant
        const double s = P.eta * 6.0 * fabs(P.nu_d) * ((double)n * (double)n);
        return (float)(s * s);
    };
    const float Df32 = floor_of(32), Df16 = floor_of(16), Df8 = floor_of(8);

    // this thread's pairs on the 32^3 level: planes 2r + p, row j, cells 2m and 2m + 1; (j + p) & 1 is the
    // x parity of the red cell
    const int j32 = t >> 4, m32 = t & 15, pair32 = j32 * 32 + 2 * m32;
    float2 f32[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) f32[p] = *reinterpret_cast<const float2*>(P.f + (2 * rank + p) * 1024 + pair32);

    // ---- the 32^3 level: this block's planes and their ghosts
#pragma unroll
    for (int e = t; e < 4 * 1024; e += kClThreads) {
        const int q = e >> 10, c = e & 1023, z = (2 * rank - 1 + q) & 31;
        cl_s[0].u32[0][q][c] = P.u[z * 1024 + c];
        cl_s[0].bg32[q][c] = P.bg[z * 1024 + c];
    }
    for (int e = t; e < 2 * 1024; e += kClThreads) cl_s[0].km32[e >> 10][e & 1023] = P.kmask[2 * rank * 1024 + e];
    __syncthreads();
    ClCell k32[2][2];  // [plane][red, black]
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = 2 * m32 + (((j32 + p) & 1) ^ q), c = j32 * 32 + i;
            k32[p][q] = cl_cell(cl_stencil<32>(cl_s[0].bg32[p], cl_s[0].bg32[p + 1], cl_s[0].bg32[p + 2], i, j32), P.kap,
                                P.lsat_c, cl_s[0].km32[p][c]);
            k32[p][q].f = (i & 1) ? f32[p].y : f32[p].x;
        }
    int b32 = 0, b16 = 0, b8 = 0;  // current copy of each level's iterate
    cl.sync();  // every block of the cluster runs: its shared memory may be written
    auto sweep32 = [&]() {
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            float2 w[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const ClCell k = cl_pick(k32[p], q);
                const int x = ((j32 + p) & 1) ^ q, i = 2 * m32 + x;
                const Stencil<float> s = cl_stencil<32>(cl_s[0].u32[b32][p], cl_s[0].u32[b32][p + 1], cl_s[0].u32[b32][p + 2], i, j32);
                const float other = cl_s[0].u32[b32][p + 1][pair32 + (x ^ 1)];
                const float v = s.c0 + local_update(cl_eval(s, k, 1024.f, P.nu, k.f), sp, Df32, 1024.f);
                w[p] = x ? make_float2(other, v) : make_float2(v, other);
            }
            b32 ^= 1;
            *reinterpret_cast<float2*>(&cl_s[0].u32[b32][1][pair32]) = w[0];
            *reinterpret_cast<float2*>(&cl_s[0].u32[b32][2][pair32]) = w[1];
            *reinterpret_cast<float2*>(&below->u32[b32][3][pair32]) = w[0];
            *reinterpret_cast<float2*>(&above->u32[b32][0][pair32]) = w[1];
            cl.sync();
        }
    };
    // the 16^3 level: threads 0 .. 127, plane r
    const int j16 = t >> 3, m16 = t & 7, pair16 = j16 * 16 + 2 * m16, par16 = (j16 + rank) & 1;
    auto sweep16 = [&]() {
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            if (t < 128) {
                const int x = par16 ^ q, i = 2 * m16 + x;
                const ClCell k = cl_s[0].c16[j16 * 16 + i];
                const Stencil<float> s = cl_stencil<16>(cl_s[0].u16[b16][0], cl_s[0].u16[b16][1], cl_s[0].u16[b16][2], i, j16);
                const float other = cl_s[0].u16[b16][1][pair16 + (x ^ 1)];
                const float v = s.c0 + local_update(cl_eval(s, k, 256.f, P.nu, k.f), sp, Df16, 256.f);
                const float2 w = x ? make_float2(other, v) : make_float2(v, other);
                const int o = b16 ^ 1;
                *reinterpret_cast<float2*>(&cl_s[0].u16[o][1][pair16]) = w;
                *reinterpret_cast<float2*>(&below->u16[o][2][pair16]) = w;
                *reinterpret_cast<float2*>(&above->u16[o][0][pair16]) = w;
            }
            b16 ^= 1;
            cl.sync();
        }
    };
    // the 8^3 level: threads 0 .. 255 of block 0
    const int k8 = t >> 5, j8 = (t >> 2) & 7, m8 = t & 3, par8 = (j8 + k8) & 1;
    auto stencil8 = [&](const float* u, int i, int j, int k) {
        return cl_stencil<8>(u + ((k - 1) & 7) * 64, u + k * 64, u + ((k + 1) & 7) * 64, i, j);
    };
    auto sweep8 = [&]() {
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            if (t < 256) {
                const int x = par8 ^ q, i = 2 * m8 + x, c = k8 * 64 + j8 * 8 + i;
                const ClCell k = cl_s[0].c8[c];
                const Stencil<float> s = stencil8(cl_s[0].u8[b8], i, j8, k8);
                cl_s[0].u8[b8 ^ 1][c ^ 1] = cl_s[0].u8[b8][c ^ 1];
                cl_s[0].u8[b8 ^ 1][c] = s.c0 + local_update(cl_eval(s, k, 64.f, P.nu, k.f), sp, Df8, 64.f);
            }
            b8 ^= 1;
            __syncthreads();
        }
    };
    // a block's residual sum and unfloored count into wsum/wcnt[0]: `count` values in shared memory (a
    // multiple of 128) and each thread's unfloored cells in.  FP64 additions, 16 cycles each per warp and SM,
    // are what it costs: four warps and then one add up columns, so that there is one shuffle tree and not one per warp.
    auto block_sum = [&](const float* v, int count, int unfl) {
        const int n = __reduce_add_sync(0xffffffffu, unfl);
        if (lane == 0) cl_s[0].wcnt[wid] = n;
        __syncthreads();
        if (t < 128) {
            double s = f2d_bits(v[t]);
#pragma unroll 4
            for (int i = t + 128; i < count; i += 128) s += f2d_bits(v[i]);
            cl_s[0].wsum[t] = s;
        }
        __syncthreads();
        if (wid == 0) {
            const double a = warp_sum((cl_s[0].wsum[lane] + cl_s[0].wsum[lane + 32]) +
                                      (cl_s[0].wsum[lane + 64] + cl_s[0].wsum[lane + 96]));
            const int c = __reduce_add_sync(0xffffffffu, lane < kClThreads / 32 ? cl_s[0].wcnt[lane] : 0);
            if (lane == 0) {
                cl_s[0].wsum[0] = a;
                cl_s[0].wcnt[0] = c;
            }
        }
        __syncthreads();
    };
    // the cluster's sums (csum, ccnt of this block, written by every block before the last cluster
    // barrier) to the gauge shift; ends with a block barrier
    auto cluster_gm = [&](int l) {
        if (wid == 0) {
            const double a = warp_sum(lane < kClBlocks ? cl_s[0].csum[l][lane] : 0.0);
            const int n = __reduce_add_sync(0xffffffffu, lane < kClBlocks ? cl_s[0].ccnt[l][lane] : 0);
            if (lane == 0) cl_s[0].gm = n > 0 ? (float)(a / (double)n) : 0.f;
        }
        __syncthreads();
    };
    auto share_sums = [&](int l) {
        if (t < kClBlocks) {
            ClSmem* o = cl.map_shared_rank(&cl_s[0], t);
            o->csum[l][rank] = cl_s[0].wsum[0];
            o->ccnt[l][rank] = cl_s[0].wcnt[0];
        }
    };

    // The V-cycle, each level's sweeps written once and run on the way down (leg 0) and up (leg 1): the
    // code is read from L2 as it is first run, and a second copy of it cost as much as its sweeps.
#pragma unroll 1
    for (int leg32 = 0; leg32 < 2; ++leg32) {
#pragma unroll 1
        for (int s = 0; s < (leg32 ? P.npost : P.npre); ++s) sweep32();
        if (leg32) break;
        {
            int un = 0;
#pragma unroll 1
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const ClCell k = cl_pick(k32[p], q);
                    const int i = 2 * m32 + (((j32 + p) & 1) ^ q), c = j32 * 32 + i;
                    const Stencil<float> s =
                        cl_stencil<32>(cl_s[0].u32[b32][p], cl_s[0].u32[b32][p + 1], cl_s[0].u32[b32][p + 2], i, j32);
                    bool fl;
                    const float r = cl_resid(cl_eval(s, k, 1024.f, P.nu, k.f), P.nu, fl);
                    cl_s[0].r32[p][c] = r;
                    cl_s[0].fl32[p][c] = fl;
                    un += !fl;
                }
            block_sum(cl_s[0].r32[0], 2048, un);
            share_sums(0);
            if (t < 256) {  // plane r of the 16^3 level; the gauge term waits for the sums
                const int I = t & 15, J = t >> 4;
                float su = 0.f, sr = 0.f, sb = 0.f;
                int cnt = 0, nun = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int c = (2 * J + ((q >> 1) & 1)) * 32 + 2 * I + (q & 1), z = q >> 2;
                    const bool fl = cl_s[0].fl32[z][c] != 0;
                    su += cl_s[0].u32[b32][z + 1][c];
                    sr += cl_s[0].r32[z][c];
                    sb += cl_s[0].bg32[z + 1][c];
                    cnt += fl ? 8 : min((int)cl_s[0].km32[z][c], 8);
                    nun += !fl;
                }
                su *= 0.125f;
                sb *= 0.125f;
                cl_s[0].rs16[t] = sr * 0.125f;
                cl_s[0].nun16[t] = (uint8_t)nun;
                cl_s[0].km16[t] = (uint8_t)((cnt + 4) >> 3);
                cl_s[0].u16[0][1][t] = cl_s[0].ur16[1][t] = su;
                cl_s[0].bg16[1][t] = sb;
                below->u16[0][2][t] = below->ur16[2][t] = su;
                below->bg16[2][t] = sb;
                above->u16[0][0][t] = above->ur16[0][t] = su;
                above->bg16[0][t] = sb;
            }
            cl.sync();
            cluster_gm(0);
            if (t < 256) {
                const int i = t & 15, j = t >> 4;
                ClCell k = cl_cell(cl_stencil<16>(cl_s[0].bg16[0], cl_s[0].bg16[1], cl_s[0].bg16[2], i, j), P.kap, P.lsat_c, cl_s[0].km16[t]);
                const Stencil<float> s = cl_stencil<16>(cl_s[0].u16[0][0], cl_s[0].u16[0][1], cl_s[0].u16[0][2], i, j);
                k.f = cl_eval(s, k, 256.f, P.nu, 0.f).G + (cl_s[0].rs16[t] - cl_s[0].gm * (float)cl_s[0].nun16[t] * 0.125f);
                cl_s[0].c16[t] = k;
            }
            __syncthreads();
        }
#pragma unroll 1
        for (int leg16 = 0; leg16 < 2; ++leg16) {
#pragma unroll 1
            for (int s = 0; s < (leg16 ? P.npost : P.npre); ++s) sweep16();
            if (leg16) break;
            {
                // the residual; each thread's pair and the row below it (eight lanes on) are the plane's four
                // children of an 8^3 cell, whose part goes to block 0
                float sr = 0.f, su = 0.f, sb = 0.f;
                int un = 0, cnt = 0;
                if (t < 128) {
#pragma unroll 1
                    for (int q = 0; q < 2; ++q) {
                        const int i = 2 * m16 + (par16 ^ q), c = j16 * 16 + i;
                        const ClCell k = cl_s[0].c16[c];
                        const Stencil<float> s = cl_stencil<16>(cl_s[0].u16[b16][0], cl_s[0].u16[b16][1], cl_s[0].u16[b16][2], i, j16);
                        bool fl;
                        const float r = cl_resid(cl_eval(s, k, 256.f, P.nu, k.f), P.nu, fl);
                        cl_s[0].rs16[c] = r;
                        sr += r;
                        su += s.c0;
                        sb += cl_s[0].bg16[1][c];
                        un += !fl;
                        cnt += fl ? 8 : min((int)cl_s[0].km16[c], 8);
                    }
                    sr += __shfl_down_sync(0xffffffffu, sr, 8);
                    su += __shfl_down_sync(0xffffffffu, su, 8);
                    sb += __shfl_down_sync(0xffffffffu, sb, 8);
                    cnt += __shfl_down_sync(0xffffffffu, cnt, 8);
                    const int n2 = un + __shfl_down_sync(0xffffffffu, un, 8);
                    if (!(j16 & 1)) {
                        ClSmem* o = cl.map_shared_rank(&cl_s[0], 0);
                        const int h = rank & 1, c = (rank >> 1) * 64 + (j16 >> 1) * 8 + m16;
                        o->h8[0][h][c] = su;
                        o->h8[1][h][c] = sr;
                        o->h8[2][h][c] = sb;
                        o->hc8[h][c] = (uint8_t)cnt;
                        o->hn8[h][c] = (uint8_t)n2;
                    }
                }
                block_sum(cl_s[0].rs16, 256, un);
                share_sums(1);
                cl.sync();
            }
            if (rank == 0) {
                cluster_gm(1);
                if (t < 512) {
                    const float su = 0.125f * (cl_s[0].h8[0][0][t] + cl_s[0].h8[0][1][t]);
                    const int cnt = cl_s[0].hc8[0][t] + cl_s[0].hc8[1][t], nun = cl_s[0].hn8[0][t] + cl_s[0].hn8[1][t];
                    cl_s[0].u8[0][t] = cl_s[0].ur8[t] = su;
                    cl_s[0].bg8[t] = 0.125f * (cl_s[0].h8[2][0][t] + cl_s[0].h8[2][1][t]);
                    cl_s[0].r8[t] = 0.125f * (cl_s[0].h8[1][0][t] + cl_s[0].h8[1][1][t]) - cl_s[0].gm * (float)nun * 0.125f;
                    cl_s[0].km8[t] = (uint8_t)((cnt + 4) >> 3);
                }
                __syncthreads();
                if (t < 512) {
                    const int i = t & 7, j = (t >> 3) & 7, k = t >> 6;
                    ClCell c = cl_cell(stencil8(cl_s[0].bg8, i, j, k), P.kap, P.lsat_c, cl_s[0].km8[t]);
                    c.f = cl_eval(stencil8(cl_s[0].u8[0], i, j, k), c, 64.f, P.nu, 0.f).G + cl_s[0].r8[t];
                    cl_s[0].c8[t] = c;
                }
                __syncthreads();
#pragma unroll 1
                for (int leg8 = 0; leg8 < 2; ++leg8) {
#pragma unroll 1
                    for (int s = 0; s < (leg8 ? P.npost : P.npre); ++s) sweep8();
                    if (leg8) break;
                    int un = 0;
                    if (t < 512) {
                        const int i = t & 7, j = (t >> 3) & 7, k = t >> 6;
                        const ClCell c = cl_s[0].c8[t];
                        bool fl;
                        const float r = cl_resid(cl_eval(stencil8(cl_s[0].u8[b8], i, j, k), c, 64.f, P.nu, c.f), P.nu, fl);
                        cl_s[0].r8[t] = r;
                        cl_s[0].fl8[t] = fl;
                        un = !fl;
                    }
                    block_sum(cl_s[0].r8, 512, un);
                    if (t < 64) {  // the 4^3 level
                        const float gm = cl_s[0].wcnt[0] > 0 ? (float)(cl_s[0].wsum[0] / (double)cl_s[0].wcnt[0]) : 0.f;
                        const int I = t & 3, J = (t >> 2) & 3, K = t >> 4;
                        float su = 0.f, sr = 0.f, sb = 0.f;
                        int cnt = 0;
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int c = (2 * K + (q >> 2)) * 64 + (2 * J + ((q >> 1) & 1)) * 8 + 2 * I + (q & 1);
                            const bool fl = cl_s[0].fl8[c] != 0;
                            su += cl_s[0].u8[b8][c];
                            sr += fl ? cl_s[0].r8[c] : cl_s[0].r8[c] - gm;
                            sb += cl_s[0].bg8[c];
                            cnt += fl ? 8 : min((int)cl_s[0].km8[c], 8);
                        }
                        su *= 0.125f;
                        cl_s[0].u4[t] = cl_s[0].ur4[t] = su;
                        cl_s[0].bg4[t] = sb * 0.125f;
                        cl_s[0].f4[t] = sr * 0.125f;
                        cl_s[0].km4[t] = (uint8_t)((cnt + 4) >> 3);
                    }
                    __syncthreads();
                    if (t < 64) {
                        const int i = t & 3, j = (t >> 2) & 3, k = t >> 4;
                        auto st = [&](const float* u) {
                            return cl_stencil<4>(u + ((k - 1) & 3) * 16, u + k * 16, u + ((k + 1) & 3) * 16, i, j);
                        };
                        const ClCell c = cl_cell(st(cl_s[0].bg4), P.kap, P.lsat_c, cl_s[0].km4[t]);
                        cl_s[0].f4[t] += cl_eval(st(cl_s[0].u4), c, 16.f, P.nu, 0.f).G;
                    }
                    __syncthreads();
                    coarsest_block<float, true>(cl_s[0].u4, cl_s[0].f4, 1.f, cl_s[0].km4, cl_s[0].bg4, 4, 16.0, P.nu_d, P.kap_d, P.eta, P.coarse_sweeps,
                                                false, cl_s[0].cs, K64{});
                    __syncthreads();
                    // 4^3 -> 8^3
                    if (t < 128) {
                        const int K8 = t >> 4, I = t & 3, J = (t >> 2) & 3, K = K8 >> 1, far = (K + (K8 & 1 ? 1 : -1)) & 3;
                        cl_prolong_plane<4>(
                            I, J, [&](int k, int c) { return cl_s[0].u4[(k ? far : K) * 16 + c] - cl_s[0].ur4[(k ? far : K) * 16 + c]; },
                            [&](int dy, int dx, float v4) { cl_s[0].u8[b8][K8 * 64 + (2 * J + dy) * 8 + 2 * I + dx] += v4; });
                    }
                    __syncthreads();
                }
                if (t < 512) cl_s[0].e8[t] = cl_s[0].u8[b8][t] - cl_s[0].ur8[t];
            }
            cl.sync();
            // 8^3 -> 16^3: this block's plane and, alike in the neighbours, its ghosts.  The three coarse
            // planes K0 .. K0 + 2 that they read come over once (reading them in place left block 0's shared
            // memory serving 52 k single loads, 5 us).
            const int K0 = ((rank + 16 - 2) >> 1) & 7;  // coarse plane of fine plane r - 2, the lowest one read
            if (t < 192) cl_s[0].d8[t >> 6][t & 63] = cl.map_shared_rank(&cl_s[0], 0)->e8[((K0 + (t >> 6)) & 7) * 64 + (t & 63)];
            __syncthreads();
            if (t < 192) {
                const int q = t >> 6, I = t & 7, J = (t >> 3) & 7, z = (rank - 1 + q) & 15, K = z >> 1,
                far = (K + (z & 1 ? 1 : -1)) & 7;
                cl_prolong_plane<8>(
                    I, J, [&](int k, int c) { return cl_s[0].d8[((k ? far : K) - K0) & 7][c]; },
                    [&](int dy, int dx, float v) { cl_s[0].u16[b16][q][(2 * J + dy) * 16 + 2 * I + dx] += v; });
            }
            __syncthreads();
        }
        {  // 16^3 -> 32^3: planes 2r - 1 .. 2r + 2 from coarse planes r - 1 .. r + 1
            const int I = t & 15, J = (t >> 4) & 15;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = (t >> 8) + 2 * h;
                const int near = (q + 1) >> 1, far = q == 0 ? 1 : (q == 1 ? 0 : (q == 2 ? 2 : 1));
                cl_prolong_plane<16>(
                    I, J, [&](int k, int c) { return cl_s[0].u16[b16][k ? far : near][c] - cl_s[0].ur16[k ? far : near][c]; },
                    [&](int dy, int dx, float v) { cl_s[0].u32[b32][q][(2 * J + dy) * 32 + 2 * I + dx] += v; });
            }
        }
        __syncthreads();
    }
    for (int e = t; e < 2 * 1024; e += kClThreads) P.u[2 * rank * 1024 + e] = cl_s[0].u32[b32][1 + (e >> 10)][e & 1023];
    cl.sync();  // no block leaves while another may still write its ghost planes
}

// Whether the cluster fits this device (asked once per context).
static bool cluster_available(pm_ctx* c)
{
    if (c->cluster_ok < 0) {
        c->cluster_ok = 0;
        int active = 0;
        cudaLaunchConfig_t lc{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim = {kClBlocks, 1, 1};
        lc.gridDim = dim3(kClBlocks);
        lc.blockDim = dim3(kClThreads);
        lc.dynamicSmemBytes = sizeof(ClSmem);
        lc.attrs = at;
        lc.numAttrs = 1;
        if (cudaFuncSetAttribute(k_coarse_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClSmem)) ==
                cudaSuccess &&
            cudaFuncSetAttribute(k_coarse_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&active, k_coarse_cluster, &lc) == cudaSuccess && active > 0)
            c->cluster_ok = 1;
        cudaGetLastError();
    }
    return c->cluster_ok == 1;
}

}  // namespace pmeft
