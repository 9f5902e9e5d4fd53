// cell64.cuh -- the local equation of a cell in FP64 (Eq. chi_discrete, Sec. 3.2.1, 3.3) with as
// few FP64 instructions as its rounding allows, and the FP64 half-sweep built on it.
//
// GB300's FP64 pipe takes 16 cycles per warp instruction and SM (1/58 of the FP32 rate), so the
// FP64 cycle is bound by the number of FP64 instructions per cell (the pipe is 85% busy at
// 128^3), not by memory.  local_eval / local_update spend 89-94 of them on an updated cell
// and 63 on a residual: the level's constants recomputed per cell, three divisions of which a
// cell needs one, products that a fused multiply-add absorbs.  Here the level's constants come in
// precomputed (K64, KW64), the products are fused and one division serves
// every branch.  The arithmetic is FP64 throughout, rounding at the same places or fewer.
#pragma once

#include "internal.cuh"

namespace pmeft {

// What the screening weight w of a cell scales: with kap1 = w kappa/h^4, the factors -2 kap1 of
// T, 8 kap1 of h^2 L in dN/dc, 96 kap1 = -4P of G in the discriminant, and L_sat/w.
struct KW64 {
    double m2, p8, p96, lsat;
};

// A level's constants: nu, 1/h^2, nu/h^2, -6 nu/h^2, h^2/6, the floor on the discriminant,
// -sgn nu, and the factors of an unmasked cell.
struct K64 {
    double nu, ih2, nu1, ep0, h2o6, Df, sp;
    KW64 w1;
};

inline K64 make_k64(int n, double nu, double kap, double eta)
{
    K64 k;
    const double ih2 = (double)n * (double)n;
    const double sqDf = eta * 6.0 * (nu < 0.0 ? -nu : nu) * ih2, kap1 = kap * ih2 * ih2;
    k.nu = nu;
    k.ih2 = ih2;
    k.nu1 = nu * ih2;
    k.ep0 = -6.0 * nu * ih2;
    k.h2o6 = 1.0 / (6.0 * ih2);
    k.Df = sqDf * sqDf;
    k.sp = nu >= 0.0 ? -1.0 : 1.0;
    k.w1 = KW64{-2.0 * kap1, 8.0 * kap1, 96.0 * kap1, kap != 0.0 ? 0.75 * nu * (1.0 - eta) / kap : 0.0};
    return k;
}

// The factors of every mask value k (weight (8 - k)/8, none from 8 on), filled by the block's
// first nine threads; the caller synchronises.
__device__ __forceinline__ void fill_kw64(KW64 (&tab)[9], const K64& k)
{
    const int q = threadIdx.x;
    if (q < 9) {
        const double w = (double)(8 - q) * 0.125;
        tab[q] = KW64{k.w1.m2 * w, k.w1.p8 * w, k.w1.p96 * w, q < 8 ? k.w1.lsat / w : 0.0};
    }
}

struct Eval64 {
    double G, Ep, D, L1;  // N - rhs, dN/dc, the discriminant, h^2 L
};

// N(chi) - rhs at a cell and its local quadratic:
// h^4 q2 = 2 (XY + YZ + ZX) - (exy^2 + exz^2 + eyz^2)/8 = 2 T, N = nu1 L1 - 2 kap1 T.
__device__ __forceinline__ Eval64 eval64(const Stencil<double>& s, double nu1, double ep0, const KW64& w, double rhs)
{
    const double X = fma(-2.0, s.c0, s.ax), Y = fma(-2.0, s.c0, s.ay), Z = fma(-2.0, s.c0, s.az);
    const double XY = X + Y;
    Eval64 o;
    o.L1 = XY + Z;
    const double E = fma(s.exy, s.exy, fma(s.exz, s.exz, s.eyz * s.eyz));
    const double T = fma(-0.0625, E, fma(Z, XY, X * Y));
    o.G = fma(w.m2, T, fma(nu1, o.L1, -rhs));
    o.Ep = fma(w.p8, o.L1, ep0);
    o.D = fma(w.p96, o.G, o.Ep * o.Ep);
    return o;
}

// a < b for b >= +0 on the integer pipe, false for a NaN of either sign: among the negative values' high
// words, those above -infinity's are NaNs (the NaN that an operation makes here has its sign set; a is the
// result of one, so a NaN is quiet and its high word says so).  -0, which a discriminant is only where it
// underflows, counts as negative.
__device__ __forceinline__ bool below64(double a, double b)
{
    return __double_as_longlong(a) < __double_as_longlong(b) && (unsigned)__double2hiint(a) <= 0xfff00000u;
}
__device__ __forceinline__ bool screened64(const KW64& w) { return (__double_as_longlong(w.m2) << 1) != 0; }

// L_sat - L, the floored gap
__device__ __forceinline__ double gap64(const Eval64& o, double ih2, double lsat) { return fma(-ih2, o.L1, lsat); }

// The correction of local_update: the root continuing the linear solution, or the floored root.
__device__ __forceinline__ double update64(const Eval64& o, const K64& k, const KW64& w)
{
    double num = -o.G, den = o.Ep;
    if (screened64(w)) {
        if (below64(o.D, k.Df)) return -gap64(o, k.ih2, w.lsat) * k.h2o6;
        const double sq = sqrt(o.D), ssq = k.sp < 0.0 ? -sq : sq;
        // Ep and ssq of one sign (by their sign bits): -2G/(Ep + ssq), else, and for Ep = 0 of either sign,
        // the other form
        if ((__double2hiint(o.Ep) ^ (__double2hiint(k.sp) & (int)0x80000000)) > 0) {
            num = -2.0 * o.G;
            den = o.Ep + ssq;
        } else {
            num = ssq - o.Ep;
            den = 24.0 * w.m2;  // 2P
        }
    }
    return num / den;
}

// The residual of a cell: f + lam - N, or nu (L_sat - L) where D is below Dfl (the floor on the
// finest level, 0 on coarse ones; see residual_cell).  fl: the floored piece was taken.
__device__ __forceinline__ double resid64(const Eval64& o, const K64& k, const KW64& w, double Dfl, bool& fl)
{
    fl = screened64(w) && below64(o.D, Dfl);
    return fl ? k.nu * gap64(o, k.ih2, w.lsat) : -o.G;
}

// A residual value's share of the five sums (residual_cell): per-thread FP32, as there.
__device__ __forceinline__ void resid_sums(double rv, bool fl, float (&fa)[5])
{
    const float d = (float)rv;
    if (!isfinite(d)) {
        fa[4] += 1.f;
    } else {
        fa[0] += d;
        fa[2] += d * d;
        if (!fl) {
            fa[1] += d;
            fa[3] += 1.f;
        }
    }
}

// One colour half-sweep of an FP64 level (half_sweep_cell's semantics), one cell per thread:
// grid * block >= n^3/2 threads.  At 128^3 a launch took 0.190 ms with local_eval's 91 FP64
// instructions per cell, 0.112 ms with these 50 or so.  Small levels are launched in blocks of 32
// to 128 threads, so that every SM's FP64 pipe gets a share: 256-thread blocks put a 16^3 or 8^3
// half-sweep's 2048 or 256 cells on eight SMs or one (7.5 us a launch, now 4.5; what is left
// there is the latency of the dependent FP64 chain).
template <bool MASK>
__global__ void __launch_bounds__(256) k_half_sweep64(const double* __restrict__ own, const double* __restrict__ oth,
                                                      double* __restrict__ out, const double* __restrict__ F,
                                                      double fscale, double lam, const uint8_t* __restrict__ kmask,
                                                      int n, int lg, int colour, K64 k,
                                                      const double* __restrict__ lamp)
{
    __shared__ KW64 tab[9];
    if (MASK) {
        fill_kw64(tab, k);
        __syncthreads();
    }
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (size_t)n * n * (n >> 1)) return;
    if (lamp) lam += *lamp;
    const int m = (int)(t & (size_t)((n >> 1) - 1));  // n is a power of two
    const size_t row = t >> (lg - 1);
    const int j = (int)(row & (size_t)(n - 1)), kz = (int)(row >> lg);
    const int i = 2 * m + ((j + kz + colour) & 1);
    const size_t c = row * n + i;
    const Stencil<double> s = load_stencil(own, oth, i, j, kz, n);
    const KW64 w = MASK ? tab[min((int)kmask[c], 8)] : k.w1;
    const Eval64 o = eval64(s, k.nu1, k.ep0, w, fma(fscale, F[c], lam));
    out[c] = s.c0 + update64(o, k, w);
}

// The FP64 residual of a level below 64^3 and its block sums (one cell per thread).
__global__ void __launch_bounds__(256) k_residual64(const double* __restrict__ u, const double* __restrict__ F,
                                                    double fscale, double lam, const uint8_t* __restrict__ kmask,
                                                    int n, int lg, K64 k, double Dfl, double* __restrict__ r,
                                                    uint8_t* __restrict__ sat, double* __restrict__ partials,
                                                    float* __restrict__ rplain, float* __restrict__ chi32,
                                                    float* __restrict__ gap32, const double* __restrict__ lamp,
                                                    double* __restrict__ fin_out)
{
    __shared__ KW64 tab[9];
    fill_kw64(tab, k);
    __syncthreads();
    if (lamp) lam += *lamp;
    float fa[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < (size_t)n * n * n) {
        const int i = (int)(c & (size_t)(n - 1));
        const size_t row = c >> lg;
        const int j = (int)(row & (size_t)(n - 1)), kz = (int)(row >> lg);
        const Stencil<double> s = load_stencil(u, u, i, j, kz, n);
        const KW64 w = tab[kmask ? min((int)kmask[c], 8) : 0];
        const Eval64 o = eval64(s, k.nu1, k.ep0, w, fma(fscale, F[c], lam));
        bool fl;
        const double rv = resid64(o, k, w, Dfl, fl);
        if (r) r[c] = rv;
        if (sat) sat[c] = fl ? 1 : 0;
        if (rplain) {  // the FP32 copies of the defect-correction loop (residual_cell, MIXED)
            rplain[c] = (float)(-o.G);
            chi32[c] = (float)s.c0;
            gap32[c] = screened64(w) ? (float)gap64(o, k.ih2, w.lsat) : 0.f;
        }
        resid_sums(rv, fl, fa);
    }
    block_sums<5>(fa, partials, fin_out);
}

// The FP64 residual of a level from 64^3 up, marching up z: a block of 32 x 8 threads keeps three
// planes of its 32 x 8 tile and their one-cell halo in a shared ring, so each iterate value is
// read from global memory once per block instead of once per stencil point.  Grid (n/32, n/8,
// n/nz).  0.275 -> 0.156 ms at 128^3 with the arithmetic above (63 -> 33 FP64 instructions per
// cell), 14.8 -> 8.6 ms for the confirming residual of a 512^3 mixed solve.  MIXED (precision 2)
// also writes the FP32 copies of the defect-correction loop.
constexpr int kR64TX = 32, kR64TY = 8;
template <bool WRITE_R, bool MIXED, bool MASK>
__global__ void __launch_bounds__(256) k_residual64_zm(const double* __restrict__ u, const double* __restrict__ F,
                                                       double fscale, double lam, const uint8_t* __restrict__ kmask,
                                                       int n, int nz, K64 k, double Dfl, double* __restrict__ r,
                                                       uint8_t* __restrict__ sat, double* __restrict__ partials,
                                                       float* __restrict__ rplain, float* __restrict__ chi32,
                                                       float* __restrict__ gap32, const double* __restrict__ lamp,
                                                       double* __restrict__ fin_out)
{
    constexpr int WX = kR64TX + 2, WY = kR64TY + 2, PL = WX * WY;
    __shared__ double ring[3][PL];
    __shared__ KW64 tab[9];
    if (MASK) fill_kw64(tab, k);  // read after the first plane's barrier
    if (lamp) lam += *lamp;
    const int m = n - 1;
    const int x0 = blockIdx.x * kR64TX, y0 = blockIdx.y * kR64TY, z0 = blockIdx.z * nz;
    const int t = threadIdx.x, tx = t & (kR64TX - 1), ty = t / kR64TX;
    const size_t plane = (size_t)n * n;
    auto load = [&](int z, int slot) {
        const size_t zo = (size_t)(z & m) * plane;
        for (int e = t; e < PL; e += 256) {
            const int xx = e % WX, yy = e / WX;
            ring[slot][e] = u[zo + (size_t)((y0 - 1 + yy) & m) * n + ((x0 - 1 + xx) & m)];
        }
    };
    float fa[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    load(z0 - 1, 0);
    load(z0, 1);
    const int cl = (ty + 1) * WX + tx + 1;
    for (int s = 0; s < nz; ++s) {
        const int z = z0 + s;
        load(z + 1, (s + 2) % 3);
        const size_t c = (size_t)z * plane + (size_t)(y0 + ty) * n + (x0 + tx);
        const double f = F[c];
        __syncthreads();
        const double* pm = ring[s % 3];        // plane z - 1
        const double* pc = ring[(s + 1) % 3];  // plane z
        const double* pp = ring[(s + 2) % 3];  // plane z + 1
        Stencil<double> st;
        st.c0 = pc[cl];
        st.ax = pc[cl + 1] + pc[cl - 1];
        st.ay = pc[cl + WX] + pc[cl - WX];
        st.az = pp[cl] + pm[cl];
        st.exy = pc[cl + 1 + WX] - pc[cl + 1 - WX] - pc[cl - 1 + WX] + pc[cl - 1 - WX];
        st.exz = pp[cl + 1] - pm[cl + 1] - pp[cl - 1] + pm[cl - 1];
        st.eyz = pp[cl + WX] - pm[cl + WX] - pp[cl - WX] + pm[cl - WX];
        const KW64 w = MASK ? tab[min((int)kmask[c], 8)] : k.w1;
        const Eval64 o = eval64(st, k.nu1, k.ep0, w, fma(fscale, f, lam));
        bool fl;
        const double rv = resid64(o, k, w, Dfl, fl);
        if (WRITE_R) {
            r[c] = rv;
            sat[c] = fl ? 1 : 0;
        }
        if (MIXED) {
            rplain[c] = (float)(-o.G);
            chi32[c] = (float)st.c0;
            gap32[c] = screened64(w) ? (float)gap64(o, k.ih2, w.lsat) : 0.f;
        }
        resid_sums(rv, fl, fa);
        __syncthreads();  // the slot of plane z - 1 is refilled next step
    }
    block_sums<5>(fa, partials, blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z), fin_out);
}

}  // namespace pmeft
