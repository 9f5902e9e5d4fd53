// pm.cu -- particle-mesh steps around the chi solve (arXiv 2604.15434, Sec. 3.1, 3.5, 3.6):
// CIC deposit in 2^40 fixed point, the FFT Poisson solve of Eq. phipsi_mod, the five-point
// gradient of Psi = Psi_N + (alpha_B - alpha_M) chi interpolated to particles (Eq. force),
// and one kick-drift.
#include <cmath>

#include "internal.cuh"

namespace pmeft {

// Cell-centred CIC weights of one coordinate; every operation rounded as written
// (no contraction) so that the weights are identical on every machine.
__device__ __forceinline__ void cic_1d(double x, int n, int& i0, int& i1, double& w0, double& w1)
{
    const double u = __dmul_rn(x, (double)n);
    const double s = __dsub_rn(u, 0.5);
    const double fl = floor(s);
    const double d = __dsub_rn(s, fl);
    const int i = (int)fl;
    i0 = i & (n - 1);
    i1 = (i + 1) & (n - 1);
    w0 = __dsub_rn(1.0, d);
    w1 = d;
}

// ---------------------------------------------------------------- CIC weights on the integer pipe
//
// GB300's FP64 pipe takes 16 cycles per warp instruction and SM, and the 46 FP64 instructions of a
// deposited particle (products, floors and conversions) kept it 86% busy while the memory system
// idled.  The integer pipes do the same in fixed point: with s = x n - 1/2 (the one FP64 operation
// left per axis), the weights d = s - floor(s) and 1 - d are 63-bit fractions of s's mantissa.

// One axis: cell indices and the two weights times 2^63.  ok: s in (-1, 4096) and not a NaN, which takes in
// every x in [0, 1) (n <= 4096) and some outside, whose cells wrap as cic_1d's do; exact: s >= 1, so that d
// and 1 - d are exact (they are in cic_1d as well).
struct CicFixed {
    int i0, i1;
    unsigned long long w0, w1;
    bool ok, exact;
};
__device__ __forceinline__ CicFixed cic_fixed(double x, int n)
{
    CicFixed r;
    const double s = __fma_rn(x, (double)n, -0.5);  // x n is exact (n a power of two): cic_1d's s
    const unsigned long long b = (unsigned long long)__double_as_longlong(s);
    const int e = (int)((b >> 52) & 0x7ff) - 1023;
    const bool neg = (long long)b < 0;
    const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const int sh = e + 11;  // |s| 2^63 = m 2^sh
    const unsigned long long f =
        (sh >= 0 ? m << (sh & 63) : (sh > -64 ? m >> (-sh & 63) : 0ull)) & 0x7fffffffffffffffull;
    const int i = e >= 0 ? (int)(m >> ((52 - e) & 63)) : 0;
    r.ok = neg ? e <= -1 : e < 12;  // s = -1/2 has e = -1
    r.exact = e >= 0;
    r.w1 = neg ? 0x8000000000000000ull - f : f;
    r.w0 = 0x8000000000000000ull - r.w1;
    const int fl = neg ? -1 : i;
    r.i0 = fl & (n - 1);
    r.i1 = (fl + 1) & (n - 1);
    return r;
}

// Particle p's eight contributions in the order of the corners c = (x, y, z) bits, each
// round((w_x w_y) w_z 2^40) with every operation rounded as written.
__device__ __forceinline__ void cic_contributions(double px, double py, double pz, int n, long long (&q)[8])
{
    int i[2];
    double wx[2], wy[2], wz[2];
    cic_1d(px, n, i[0], i[1], wx[0], wx[1]);
    cic_1d(py, n, i[0], i[1], wy[0], wy[1]);
    cic_1d(pz, n, i[0], i[1], wz[0], wz[1]);
    for (int c = 0; c < 8; ++c)
        q[c] = __double2ll_rn(__dmul_rn(__dmul_rn(__dmul_rn(wx[c & 1], wy[(c >> 1) & 1]), wz[c >> 2]), 1099511627776.0));
}

// The deposit, bit for bit cic_contributions: the fixed-point product of the three weights carries
// 61 fraction bits; it differs from the twice rounded FP64 product by at most 2^-52 of itself plus
// four units (weights not exact, s < 1: 5 x 2^-53 more), so its rounding to 40 bits is the same
// unless it lies that near a tie.  Those particles (1 in 2000) and any whose coordinate is not `ok` take
// the FP64 form.  256^3 particles: 1.44 -> 0.46 ms; what is left is the eight 64-bit reductions (L1 72% of
// its throughput, L2's atomic unit 54%, FP64 pipe 44% at 128^3).
__global__ void __launch_bounds__(256) k_deposit(const double* __restrict__ pos, long long np, int n,
                                                 unsigned long long* __restrict__ acc)
{
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const double px = pos[p], py = pos[np + p], pz = pos[2 * np + p];
    const CicFixed x = cic_fixed(px, n), y = cic_fixed(py, n), z = cic_fixed(pz, n);
    int ix[2] = {x.i0, x.i1}, iy[2] = {y.i0, y.i1}, iz[2] = {z.i0, z.i1};
    const unsigned wide = x.exact && y.exact && z.exact ? 8u : 2048u;
    bool redo = !(x.ok && y.ok && z.ok);
    long long q[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const unsigned long long wxy = __umul64hi((c & 1) ? x.w1 : x.w0, (c >> 1) ? y.w1 : y.w0);  // 2^62
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const unsigned long long w = __umul64hi(wxy, e ? z.w1 : z.w0);  // 2^61
            const unsigned slack = (unsigned)(w >> 52) + wide, r = (unsigned)w & 0x1fffffu;
            redo |= r - (0x100000u - slack) <= 2u * slack;
            q[4 * e + c] = (long long)((w + 0x100000ull) >> 21);
        }
    }
    if (redo) {
        cic_contributions(px, py, pz, n, q);
        double w0, w1;  // the indices of a coordinate outside [0, 1) as well
        cic_1d(px, n, ix[0], ix[1], w0, w1);
        cic_1d(py, n, iy[0], iy[1], w0, w1);
        cic_1d(pz, n, iz[0], iz[1], w0, w1);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c)
        atomicAdd(&acc[((size_t)iz[c >> 2] * n + iy[(c >> 1) & 1]) * n + ix[c & 1]], (unsigned long long)q[c]);
}

// delta = acc 2^-40 (n^3/np) - 1, rounded after the product and after the difference; a negative
// accumulator means the int64 capacity (2^23 particles at full weight in one cell) was exceeded.
// Bound by the FP64 pipe: an accumulator below 2^52 becomes a double by setting the exponent bits
// of 2^52 + a (no conversion), the power of two joins the factor c = 2^-40 n^3/np, and where n^3/np
// is a power of two itself (POW2: the product is exact) one fused multiply-add does it all.
// 256^3 cells: 0.128 -> 0.047 ms.
template <bool POW2>
__global__ void __launch_bounds__(256) k_density(const long long* __restrict__ acc, size_t cells, double c,
                                                 double* __restrict__ delta, int* __restrict__ flag)
{
    const double two52 = 4503599627370496.0;
    const double k = -(two52 * c) - 1.0;  // exact for the c that POW2 is used with
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < cells; t += (size_t)gridDim.x * blockDim.x) {
        const long long a = acc[t];
        if (a < 0) flag[0] = 1;
        double v;
        if ((unsigned long long)a < (1ull << 52)) {
            const double up = __longlong_as_double(a | 0x4330000000000000ll);  // 2^52 + a
            v = POW2 ? __fma_rn(up, c, k) : __dsub_rn(__dmul_rn(__dsub_rn(up, two52), c), 1.0);
        } else {
            v = __dsub_rn(__dmul_rn((double)a, c), 1.0);
        }
        delta[t] = v;
    }
}

// Multiply the spectrum by fac / lambda_k with lambda_k = -(4/h^2) sum sin^2(pi m/n), the
// 7-point Laplacian's eigenvalues; the zero mode is set to 0.  Also folds in 1/n^3.  Each
// block first tabulates sin^2(pi m/n), m <= n/2, in shared memory.  A thread takes |kz|, |ky|, kx and the
// up to four modes (+-kz, +-ky, kx) that share the factor: one division for the four, with the
// operations and so the bits of a mode by itself.  256^3: 0.244 ms with a division and two 64-bit index
// divisions per mode, 0.122 so (270 MB there and back); the solve 3.77 -> 3.65 ms, the rest cuFFT's.
__global__ void __launch_bounds__(256) k_green(double2* __restrict__ spec, int n, double fac)
{
    extern __shared__ double s2[];  // [n/2 + 1]
    const int nh = n / 2 + 1;
    for (int m = threadIdx.x; m < nh; m += blockDim.x) {
        const double sm = sinpi((double)m / n);
        s2[m] = sm * sm;
    }
    __syncthreads();
    const size_t total = (size_t)nh * nh * nh;
    const double h2inv = (double)n * (double)n;
    const double scale = fac * (1.0 / ((double)n * (double)n * (double)n));
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int mx = (int)(t % nh);
        const size_t row = t / nh;
        const int ay = (int)(row % nh), az = (int)(row / nh);
        const bool two_y = ay != 0 && ay != n - ay, two_z = az != 0 && az != n - az;
        const size_t y1 = (size_t)(n - ay) * nh, y0 = (size_t)ay * nh, z0 = (size_t)az * n * nh + mx,
                     z1 = (size_t)(n - az) * n * nh + mx;
        double2 v[4];
        v[0] = spec[z0 + y0];
        if (two_y) v[1] = spec[z0 + y1];
        if (two_z) v[2] = spec[z1 + y0];
        if (two_y && two_z) v[3] = spec[z1 + y1];
        const double g = scale / (-4.0 * h2inv * (s2[mx] + s2[ay] + s2[az]));
        spec[z0 + y0] = t == 0 ? make_double2(0.0, 0.0) : make_double2(v[0].x * g, v[0].y * g);
        if (two_y) spec[z0 + y1] = make_double2(v[1].x * g, v[1].y * g);
        if (two_z) spec[z1 + y0] = make_double2(v[2].x * g, v[2].y * g);
        if (two_y && two_z) spec[z1 + y1] = make_double2(v[3].x * g, v[3].y * g);
    }
}

// k_green in FP32 (the start fields' solve): the same eigenvalues, zero mode and 1/n^3
__global__ void k_green32(float2* __restrict__ spec, int n, float fac)
{
    const int nh = n / 2 + 1;
    const size_t total = (size_t)n * n * nh;
    const float h2inv = (float)n * (float)n;
    const float scale = fac / ((float)n * (float)n * (float)n);
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int mx = (int)(t % nh);
        const size_t row = t / nh;
        const int my = (int)(row % n), mz = (int)(row / n);
        const float sx = sinpif((float)mx / n), sy = sinpif((float)my / n), sz = sinpif((float)mz / n);
        const float lam = -4.f * h2inv * (sx * sx + sy * sy + sz * sz);
        float2 v = spec[t];
        if (t == 0) {
            v = make_float2(0.f, 0.f);
        } else {
            const float g = scale / lam;
            v.x *= g;
            v.y *= g;
        }
        spec[t] = v;
    }
}

__global__ void k_d2f(const double* __restrict__ x, size_t total, float* __restrict__ y)
{
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += (size_t)gridDim.x * blockDim.x)
        y[c] = (float)x[c];
}

__global__ void k_f2d(const float* __restrict__ x, size_t total, double* __restrict__ y)
{
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += (size_t)gridDim.x * blockDim.x)
        y[c] = (double)x[c];
}

// Psi = psiN + xi chi on the grid, rounded as written; psi may be psiN.
__global__ void __launch_bounds__(256) k_psi_total(const double* psiN, const double* __restrict__ chi, double xi,
                                                   size_t total, double* psi)
{
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += (size_t)gridDim.x * blockDim.x)
        psi[c] = __dadd_rn(psiN[c], __dmul_rn(xi, chi[c]));
}

// The grid force up to its scale: G = 8 (f+1 - f-1) - (f+2 - f-2) per axis (FOUR; else f+1 - f-1) of
// the potential, periodic, one cell per thread; -grad Psi is G times -n/12 (-n/2), a factor the
// interpolation applies.  g holds (Gx, Gy, Gz, 0) per cell, 32 bytes, so that a particle's corner
// is one aligned 256-bit load.  Bound by FP64 instructions: three per component where the scaled
// difference took four (0.40 -> 0.295 ms at 256^3).  (A z-marching block that formed Psi itself
// recomputed it on its halo, 2.9 instructions per cell instead of 2: 0.43 ms against 0.37 for the
// two kernels.)
template <bool FOUR>
__global__ void __launch_bounds__(256) k_grad(const double* __restrict__ psi, int n, int lg, double* __restrict__ g)
{
    const int m = n - 1;
    const size_t total = (size_t)n * n * n;
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(c & (size_t)m), j = (int)((c >> lg) & (size_t)m), k = (int)(c >> (2 * lg));
        const double* row = psi + (c - i);
        const double* col = psi + (((size_t)k << (2 * lg)) + i);
        const double* pil = psi + (((size_t)j << lg) + i);
        auto x = [&](int d) { return row[(i + d) & m]; };
        auto y = [&](int d) { return col[(size_t)((j + d) & m) << lg]; };
        auto z = [&](int d) { return pil[(size_t)((k + d) & m) << (2 * lg)]; };
        double gx = x(1) - x(-1), gy = y(1) - y(-1), gz = z(1) - z(-1);
        if (FOUR) {
            gx = fma(8.0, gx, x(-2) - x(2));
            gy = fma(8.0, gy, y(-2) - y(2));
            gz = fma(8.0, gz, z(-2) - z(2));
        }
        double2* o = reinterpret_cast<double2*>(g + 4 * c);
        o[0] = make_double2(gx, gy);
        o[1] = make_double2(gz, 0.0);
    }
}

// f 2^-63 as a double (correctly rounded but for exact ties), f <= 2^63: the integer pipe's conversion
__device__ __forceinline__ double fixed_to_double(unsigned long long f)
{
    if (f == 0) return 0.0;
    const int lz = __clzll((long long)f);
    const unsigned long long m = f << lz;  // top bit set
    return __longlong_as_double((long long)(((unsigned long long)(1022 - lz) << 52) + (m >> 11) + ((m >> 10) & 1)));
}

// four doubles of one 32-byte aligned cell
__device__ __forceinline__ void ld_cell(const double* p, double& a, double& b, double& c)
{
    double unused;
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(unused) : "l"(p));
}

// The force at each particle: the grid force at the 8 CIC corners weighted by the corners' CIC
// weights (the deposit's adjoint), times `scale`.  Bound by FP64 instructions (39 per particle where
// eight weights, three-component sums and the weights' floors and conversions took 54): the weights
// come from the integer pipe, the x-y weights serve both z planes, and the scale rides on the z
// weights.  256^3 particles: 1.64 -> 1.19 ms.
__global__ void __launch_bounds__(256) k_interp_force(const double* __restrict__ g, int n, double scale,
                                                      const double* __restrict__ pos, long long np,
                                                      double* __restrict__ acc)
{
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    int ix[2], iy[2], iz[2];
    double wx[2], wy[2], wz[2];
    auto axis = [&](double x, int (&i)[2], double (&w)[2]) {
        const CicFixed f = cic_fixed(x, n);
        if (f.ok) {
            i[0] = f.i0;
            i[1] = f.i1;
            w[0] = fixed_to_double(f.w0);
            w[1] = fixed_to_double(f.w1);
        } else {
            cic_1d(x, n, i[0], i[1], w[0], w[1]);
        }
    };
    axis(pos[p], ix, wx);
    axis(pos[np + p], iy, wy);
    axis(pos[2 * np + p], iz, wz);
    double s[2][3];
    const double w4[4] = {wx[0] * wy[0], wx[1] * wy[0], wx[0] * wy[1], wx[1] * wy[1]};
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            double a, b, d;
            ld_cell(g + 4 * (((size_t)iz[e] * n + iy[c >> 1]) * n + ix[c & 1]), a, b, d);
            s[e][0] = c ? fma(w4[c], a, s[e][0]) : w4[c] * a;
            s[e][1] = c ? fma(w4[c], b, s[e][1]) : w4[c] * b;
            s[e][2] = c ? fma(w4[c], d, s[e][2]) : w4[c] * d;
        }
    const double z0 = wz[0] * scale, z1 = wz[1] * scale;
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k * np + p] = fma(z1, s[1][k], z0 * s[0][k]);
}

// v += g dt; x = frac(x + v dt), each product and sum rounded as written.  Four FP64 instructions per
// coordinate (the wrap is entered only where the bits of x say x < 0 or x >= 1) and 40 bytes of HBM
// traffic; four coordinates per thread in flight (50 M coordinates: 0.68 -> 0.39 ms).
__global__ void __launch_bounds__(256) k_kick_drift(double* __restrict__ pos, double* __restrict__ vel,
                                                    const double* __restrict__ acc, long long total, double dt)
{
    const long long i0 = (long long)blockIdx.x * 1024 + threadIdx.x;
    double a[4], v[4], x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const long long i = i0 + 256 * k;
        if (i >= total) break;
        a[k] = acc[i];
        v[k] = vel[i];
        x[k] = pos[i];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const long long i = i0 + 256 * k;
        if (i >= total) break;
        v[k] = __dadd_rn(v[k], __dmul_rn(a[k], dt));
        vel[i] = v[k];
        x[k] = __dadd_rn(x[k], __dmul_rn(v[k], dt));
        if ((unsigned)__double2hiint(x[k]) >= 0x3ff00000u) {  // negative, >= 1 or not a number
            x[k] = __dsub_rn(x[k], floor(x[k]));
            if (x[k] >= 1.0) x[k] = 0.0;
        }
        pos[i] = x[k];
    }
}

// out = s * x (+ y), each product and sum rounded as written
__global__ void k_scale_add(const double* __restrict__ x, double s, const double* __restrict__ y, size_t total,
                            double* __restrict__ out)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const double v = __dmul_rn(s, x[i]);
        out[i] = y ? __dadd_rn(y[i], v) : v;
    }
}

static void scale_add(pm_ctx* ctx, const double* x, double s, const double* y, size_t total, double* out)
{
    ctx->begin(PM_K_PM, false, 0);
    k_scale_add<<<grid_for(ctx, total), kThreads, 0, ctx->stream>>>(x, s, y, total, out);
    ctx->end();
}

pm_status deposit(pm_ctx* ctx, const double* pos, long long np, int n, long long* acc)
{
    const size_t cells = (size_t)n * n * n;
    PM_CUDA(cudaMemsetAsync(acc, 0, cells * sizeof(long long), ctx->stream));
    ctx->begin(PM_K_PM, false, 0);
    k_deposit<<<(unsigned)((np + kThreads - 1) / kThreads), kThreads, 0, ctx->stream>>>(pos, np, n,
                                                                                       (unsigned long long*)acc);
    ctx->end();
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

static void launch_density(cudaStream_t s, int grid, const long long* acc, size_t cells, long long np, double* delta,
                           int* flag)
{
    // fused form: n^3/np a power of two (the product exact) and its constant -(2^12 n^3/np) - 1 too
    const double fac = (double)cells / (double)np, c = fac * 9.094947017729282379150390625e-13;  // 2^-40
    int ex = 0;
    if (std::frexp(fac, &ex) == 0.5 && ex >= -8 && ex <= 30)
        k_density<true><<<grid, kThreads, 0, s>>>(acc, cells, c, delta, flag);
    else
        k_density<false><<<grid, kThreads, 0, s>>>(acc, cells, c, delta, flag);
}

// ctx->flag[0] is zero between calls (cleared here after an overflow)
pm_status density(pm_ctx* ctx, const long long* acc, int n, long long np, double* delta)
{
    const size_t cells = (size_t)n * n * n;
    ctx->begin(PM_K_PM, false, 0);
    launch_density(ctx->stream, grid_for(ctx, cells), acc, cells, np, delta, ctx->flag);
    ctx->end();
    int* hflag = reinterpret_cast<int*>(ctx->host_out + 63);
    PM_CUDA(cudaMemcpyAsync(hflag, ctx->flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    PM_CUDA(cudaStreamSynchronize(ctx->stream));
    if (*hflag) {
        PM_CUDA(cudaMemsetAsync(ctx->flag, 0, sizeof(int), ctx->stream));
        ctx->set_error("fixed-point deposit overflow (more than 2^23 particles in one cell)");
        return PM_ERR_OVERFLOW;
    }
    return PM_OK;
}

pm_status poisson(pm_ctx* ctx, const double* delta, int n, double fac, double* psi)
{
    Workspace* w = nullptr;
    PM_TRY(get_workspace(ctx, n, &w));
    PM_TRY(ensure_fft(ctx, w));
    ctx->prof.launches[PM_K_PM] += 2;  // the two cuFFT executions (library kernels)
    if (cufftExecD2Z(w->plan_r2c, (cufftDoubleReal*)delta, (cufftDoubleComplex*)w->spec) != CUFFT_SUCCESS) {
        ctx->set_error("cufftExecD2Z failed");
        return PM_ERR_CUDA;
    }
    ctx->begin(PM_K_PM, false, 0);
    const size_t nh = n / 2 + 1;
    k_green<<<grid_for(ctx, nh * nh * nh), kThreads, nh * sizeof(double), ctx->stream>>>(w->spec, n, fac);
    ctx->end();
    if (cufftExecZ2D(w->plan_c2r, (cufftDoubleComplex*)w->spec, (cufftDoubleReal*)psi) != CUFFT_SUCCESS) {
        ctx->set_error("cufftExecZ2D failed");
        return PM_ERR_CUDA;
    }
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

pm_status poisson32(pm_ctx* ctx, const double* delta, int n, double fac, double* psi)
{
    Workspace* w = nullptr;
    PM_TRY(get_workspace(ctx, n, &w));
    PM_TRY(ensure_fft32(ctx, w));
    const size_t cells = (size_t)n * n * n;
    ctx->begin(PM_K_PM, false, 0);
    k_d2f<<<grid_for(ctx, cells), kThreads, 0, ctx->stream>>>(delta, cells, w->buf32);
    ctx->end();
    ctx->prof.launches[PM_K_PM] += 2;  // the two cuFFT executions (library kernels)
    if (cufftExecR2C(w->plan_r2c32, (cufftReal*)w->buf32, (cufftComplex*)w->spec32) != CUFFT_SUCCESS) {
        ctx->set_error("cufftExecR2C failed");
        return PM_ERR_CUDA;
    }
    ctx->begin(PM_K_PM, false, 0);
    k_green32<<<grid_for(ctx, (size_t)n * n * (n / 2 + 1)), kThreads, 0, ctx->stream>>>(w->spec32, n, (float)fac);
    ctx->end();
    if (cufftExecC2R(w->plan_c2r32, (cufftComplex*)w->spec32, (cufftReal*)w->buf32) != CUFFT_SUCCESS) {
        ctx->set_error("cufftExecC2R failed");
        return PM_ERR_CUDA;
    }
    ctx->begin(PM_K_PM, false, 0);
    k_f2d<<<grid_for(ctx, cells), kThreads, 0, ctx->stream>>>(w->buf32, cells, psi);
    ctx->end();
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

// g = -grad(psiN + xi chi) at each particle (Eq. force, Sec. 3.5.2; psiN alone when chi is null): the
// total potential (in the workspace's psi, in place where psiN is that) and its gradient on the grid
// (workspace: [n^3][4]), then the CIC interpolation of the grid force.
pm_status interp_force(pm_ctx* ctx, const double* psiN, const double* chi, double xi, int n, const double* pos,
                       long long np, double* acc)
{
    Workspace* w = nullptr;
    PM_TRY(get_workspace(ctx, n, &w));
    const size_t cells = (size_t)n * n * n;
    if (!w->grad) PM_CUDA(cudaMalloc(&w->grad, 4 * cells * sizeof(double)));
    const double* psi = psiN;
    if (chi) {
        if (!w->psi) PM_CUDA(cudaMalloc(&w->psi, cells * sizeof(double)));
        ctx->begin(PM_K_PM, false, 0);
        k_psi_total<<<grid_for(ctx, cells), kThreads, 0, ctx->stream>>>(psiN, chi, xi, cells, w->psi);
        ctx->end();
        psi = w->psi;
    }
    const bool four = ctx->prm.grad_order != 2;
    const int lg = __builtin_ctz(n);
    ctx->begin(PM_K_PM, false, 0);
    if (four) k_grad<true><<<grid_for(ctx, cells), kThreads, 0, ctx->stream>>>(psi, n, lg, w->grad);
    else k_grad<false><<<grid_for(ctx, cells), kThreads, 0, ctx->stream>>>(psi, n, lg, w->grad);
    ctx->end();
    ctx->begin(PM_K_PM, false, 0);
    k_interp_force<<<(unsigned)((np + kThreads - 1) / kThreads), kThreads, 0, ctx->stream>>>(
        w->grad, n, four ? -(double)n / 12.0 : -(double)n * 0.5, pos, np, acc);
    ctx->end();
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

pm_status kick_drift(pm_ctx* ctx, double* pos, double* vel, const double* acc, long long np, double dt)
{
    ctx->begin(PM_K_PM, false, 0);
    k_kick_drift<<<(unsigned)((3 * np + 1023) / 1024), kThreads, 0, ctx->stream>>>(pos, vel, acc, 3 * np, dt);
    ctx->end();
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

// Launchers on a bare stream (no context), used by the allocation-free deposit.
static int grid_on(int sms, size_t work)
{
    size_t blocks = (work + kThreads - 1) / kThreads, cap = (size_t)(sms > 0 ? sms : 152) * 16;
    return (int)(blocks < 1 ? 1 : (blocks > cap ? cap : blocks));
}

void launch_deposit_on(cudaStream_t s, const double* pos, long long np, int n, unsigned long long* acc)
{
    k_deposit<<<(unsigned)((np + kThreads - 1) / kThreads), kThreads, 0, s>>>(pos, np, n, acc);
}

void launch_density_on(cudaStream_t s, int sms, const long long* acc, int n, long long np, double* delta, int* flag)
{
    const size_t cells = (size_t)n * n * n;
    launch_density(s, grid_on(sms, cells), acc, cells, np, delta, flag);
}

}  // namespace pmeft

using namespace pmeft;

static pm_status check_common(pm_ctx* ctx, int n)
{
    if (!ctx) return PM_ERR_INVALID_ARG;
    if (!valid_n(n)) {
        ctx->set_error("n must be a power of two >= 8");
        return PM_ERR_INVALID_ARG;
    }
    if (cudaSetDevice(ctx->device) != cudaSuccess) return PM_ERR_CUDA;
    return PM_OK;
}

extern "C" pm_status pm_deposit_cic_fixed(pm_ctx* ctx, const double* pos, long long np, int n, long long* acc)
{
    PM_TRY(check_common(ctx, n));
    if (!pos || !acc || np < 1) {
        ctx->set_error("pm_deposit_cic: null buffer or np < 1");
        return PM_ERR_INVALID_ARG;
    }
    return deposit(ctx, pos, np, n, acc);
}

extern "C" pm_status pm_deposit_cic(pm_ctx* ctx, const double* pos, long long np, int n, double* delta)
{
    PM_TRY(check_common(ctx, n));
    if (!pos || !delta || np < 1) {
        ctx->set_error("pm_deposit_cic: null buffer or np < 1");
        return PM_ERR_INVALID_ARG;
    }
    Workspace* w = nullptr;
    PM_TRY(get_workspace(ctx, n, &w));
    if (!w->acc) PM_CUDA(cudaMalloc(&w->acc, (size_t)n * n * n * sizeof(long long)));
    PM_TRY(deposit(ctx, pos, np, n, w->acc));
    return density(ctx, w->acc, n, np, delta);
}

extern "C" pm_status poisson_solve(pm_ctx* ctx, const double* delta, int n, double a, double alpha_M0, double* psi_N)
{
    PM_TRY(check_common(ctx, n));
    if (!delta || !psi_N || delta == psi_N || !(a > 0.0)) {
        ctx->set_error("poisson_solve: null or aliased buffer, or a <= 0");
        return PM_ERR_INVALID_ARG;
    }
    pm_coeffs cf;
    coefficients(0.0, alpha_M0, a, ctx->prm.omega_m0, ctx->prm.include_dot_alphaB, &cf);
    return poisson(ctx, delta, n, cf.poisson_fac, psi_N);
}

extern "C" pm_status force_interp(pm_ctx* ctx, const double* psi_N, const double* phi, int n, double alpha_B0,
                                  double alpha_M0, double a, const double* pos, long long np, double* acc)
{
    PM_TRY(check_common(ctx, n));
    if (!psi_N || !pos || !acc || np < 1 || !(a > 0.0)) {
        ctx->set_error("force_interp: null buffer, np < 1 or a <= 0");
        return PM_ERR_INVALID_ARG;
    }
    pm_coeffs cf;
    coefficients(alpha_B0, alpha_M0, a, ctx->prm.omega_m0, ctx->prm.include_dot_alphaB, &cf);
    return interp_force(ctx, psi_N, phi, cf.xi, n, pos, np, acc);
}

extern "C" pm_status pm_step(pm_ctx* ctx, double* pos, double* vel, long long np, int n, double alpha_B0,
                             double alpha_M0, double a, double dt, double tol, double* phi_state, pm_solve_info* info)
{
    PM_TRY(check_common(ctx, n));
    if (!pos || !vel || !phi_state || np < 1 || !(a > 0.0) || !(tol > 0.0)) {
        ctx->set_error("pm_step: null buffer, np < 1, a <= 0 or tol <= 0");
        return PM_ERR_INVALID_ARG;
    }
    Workspace* w = nullptr;
    PM_TRY(get_workspace(ctx, n, &w));
    const size_t cells = (size_t)n * n * n;
    if (!w->acc) PM_CUDA(cudaMalloc(&w->acc, cells * sizeof(long long)));
    if (!w->delta) PM_CUDA(cudaMalloc(&w->delta, cells * sizeof(double)));
    if (!w->psi) PM_CUDA(cudaMalloc(&w->psi, cells * sizeof(double)));
    pm_coeffs cf;
    coefficients(alpha_B0, alpha_M0, a, ctx->prm.omega_m0, ctx->prm.include_dot_alphaB, &cf);
    PM_TRY(deposit(ctx, pos, np, n, w->acc));
    PM_TRY(density(ctx, w->acc, n, np, w->delta));
    PM_TRY(poisson(ctx, w->delta, n, cf.poisson_fac, w->psi));
    if (ctx->prm.linear_eft) {
        // linearised equations: nu L chi = xi S and L Psi_N = S, so chi = (xi / nu) Psi_N
        if (cf.nu == 0.0 && cf.xi != 0.0) {
            ctx->set_error("pm_step: nu = 0, the linearised chi equation is degenerate");
            return PM_ERR_INVALID_ARG;
        }
        scale_add(ctx, w->psi, cf.xi != 0.0 ? cf.xi / cf.nu : 0.0, nullptr, cells, phi_state);
        if (info) *info = pm_solve_info{};
    } else {
        pm_status st = mg_solve(ctx, w->delta, n, cf, tol, phi_state, info);
        if (st != PM_OK) return st;
    }
    // the acceleration goes into the (now free) fixed-point grid's storage when it fits
    double* acc = nullptr;
    const size_t need = (size_t)3 * np * sizeof(double);
    if (need <= cells * sizeof(long long)) {
        acc = (double*)w->acc;
    } else {
        PM_CUDA(cudaMallocAsync(&acc, need, ctx->stream));
    }
    PM_TRY(interp_force(ctx, w->psi, phi_state, cf.xi, n, pos, np, acc));
    PM_TRY(kick_drift(ctx, pos, vel, acc, np, dt));
    if ((void*)acc != (void*)w->acc) PM_CUDA(cudaFreeAsync(acc, ctx->stream));
    PM_CUDA(cudaStreamSynchronize(ctx->stream));
    return PM_OK;
}

// ------------------------------------------------------------------ several steps

// supercomoving time per unit scale factor: dt~/da = 1 / (a^3 E(a)), E^2 = Om a^-3 + 1 - Om
static double dtda(double a, double om) { return 1.0 / (a * a * a * std::sqrt(om / (a * a * a) + 1.0 - om)); }
static double dadt(double a, double om) { return a * a * a * std::sqrt(om / (a * a * a) + 1.0 - om); }

extern "C" pm_status pm_run(pm_ctx* ctx, double* pos, double* vel, long long np, int n, double alpha_B0,
                            double alpha_M0, double a_start, double a_end, int nsteps, double tol,
                            double* phi_state, pm_solve_info* info)
{
    PM_TRY(check_common(ctx, n));
    if (!(a_start > 0.0) || !(a_end >= a_start) || nsteps < 1) {
        ctx->set_error("pm_run: need 0 < a_start <= a_end and nsteps >= 1");
        return PM_ERR_INVALID_ARG;
    }
    const double om = ctx->prm.omega_m0;
    // total supercomoving time by composite Simpson in a (4096 intervals), equal steps in it
    const int K = 4096;
    const double ha = (a_end - a_start) / K;
    double T = dtda(a_start, om) + dtda(a_end, om);
    for (int k = 1; k < K; ++k) T += (k & 1 ? 4.0 : 2.0) * dtda(a_start + k * ha, om);
    T *= ha / 3.0;
    const double dt = T / nsteps;
    double a = a_start;
    pm_solve_info local{};
    for (int s = 0; s < nsteps; ++s) {
        PM_TRY(pm_step(ctx, pos, vel, np, n, alpha_B0, alpha_M0, a, dt, tol, phi_state, info ? info : &local));
        // advance a over the step: classical Runge-Kutta on da/dt~ = a^3 E(a), 8 substeps
        const double hs = dt / 8.0;
        for (int q = 0; q < 8; ++q) {
            const double k1 = dadt(a, om), k2 = dadt(a + 0.5 * hs * k1, om), k3 = dadt(a + 0.5 * hs * k2, om),
                         k4 = dadt(a + hs * k3, om);
            a += hs * (k1 + 2.0 * k2 + 2.0 * k3 + k4) / 6.0;
        }
    }
    return PM_OK;
}

extern "C" pm_status lensing_potential(pm_ctx* ctx, const double* psi_N, const double* chi, int n, double alpha_B0,
                                       double alpha_M0, double a, double* Phi)
{
    PM_TRY(check_common(ctx, n));
    if (!psi_N || !chi || !Phi || !(a > 0.0)) {
        ctx->set_error("lensing_potential: null buffer or a <= 0");
        return PM_ERR_INVALID_ARG;
    }
    pm_coeffs cf;
    coefficients(alpha_B0, alpha_M0, a, ctx->prm.omega_m0, ctx->prm.include_dot_alphaB, &cf);
    scale_add(ctx, chi, cf.alpha_B, psi_N, (size_t)n * n * n, Phi);
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}
