// PM (long-range) part of the TreePM split (Sec. 2.1-2.2 step 1; Table 2 rows "density
// assignment", "FFT", "convolution", "force interpolation").
//
// The PP part is Newton's law times g_P3M (Eq. 1-2), i.e. Newton's law minus the force
// between two S2 clouds of radius eta; the PM part carries exactly that cloud-cloud force:
//   phi_k = G(k) rho_k,  G(k) = -4 pi S(k eta)^2 / (k^2 W(k)^2),  k = 0 removed,
// with S(xi) = 12 (2 - 2 cos xi - xi sin xi)/xi^4 and W the assignment window (CIC p = 2,
// TSC p = 3, divided out once for the assignment and once for the interpolation).  The
// acceleration is -i k phi_k per component (Nyquist components zeroed), transformed back
// and interpolated with the assignment weights.  Grid points sit at x = j L/n (periodic).
//
// G is tabulated once per (n, L, r_cut, scheme) in FP64 over |k_x|, |k_y|, k_z (the
// (n/2+1)^3 table the paper also keeps, Sec. 3.2.5), with 1/Delta^3 (mass -> density)
// and 1/n^3 (unnormalised inverse FFT) folded in.  The FFTs are cuFFT (FP32).
#include <cufft.h>

#include "common.cuh"
#include "pm.cuh"

namespace greem {

struct PmGeom {
    int n;             // grid points per side
    int scheme;        // 0 CIC, 1 TSC
    double L;
    double inv_delta;  // n / L
    int pow2_e;        // L = 2^pow2_e, or kNotPow2
    int log2n;         // n = 2^log2n, or -1
};

// Integer grid index and fractional part of x * n / L (x wrapped into [0, L)).
__device__ __forceinline__ void grid_coord(double x, const PmGeom &g, int &i, float &f)
{
    x = wrap_pos_fast(x, g.L);
    if (g.pow2_e != kNotPow2 && g.log2n >= 0) {
        // exact: x n/L = fixed52(x) * 2^(log2n - 52)
        const long long q = fixed52(x, g.pow2_e);
        const int sh = 52 - g.log2n;
        i = (int)(q >> sh);
        f = __ll2float_rn(q & ((1ll << sh) - 1)) * __int_as_float((127 - sh) << 23);
    } else {
        const double s = x * g.inv_delta;
        const double fl = floor(s);
        i = (int)fl;
        f = (float)(s - fl);
    }
    if (i >= g.n) {  // x * n / L rounded up to n
        i -= g.n;
    }
}

// Per-axis weights: CIC (i, i+1) with (1-f, f); TSC (i-1, i, i+1) about the nearest point.
template <int SCHEME>
__device__ __forceinline__ void axis_weights(int i, float f, int n, int (&idx)[3], float (&w)[3])
{
    if (SCHEME == 0) {
        idx[0] = i;
        idx[1] = i + 1 == n ? 0 : i + 1;
        w[0] = 1.0f - f;
        w[1] = f;
        idx[2] = 0;
        w[2] = 0.0f;
    } else {
        int c = i;
        float d = f;
        if (f >= 0.5f) {
            c = i + 1 == n ? 0 : i + 1;
            d = f - 1.0f;
        }
        idx[0] = c == 0 ? n - 1 : c - 1;
        idx[1] = c;
        idx[2] = c + 1 == n ? 0 : c + 1;
        const float a = 0.5f - d, b = 0.5f + d;
        w[0] = 0.5f * a * a;
        w[1] = 0.75f - d * d;
        w[2] = 0.5f * b * b;
    }
}

__device__ __forceinline__ void red_v4(float *p, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ void red_v2(float *p, float a, float b)
{
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}

// Bound by the atomics' sectors.  Particles of a row in order (a set that keeps its grid
// order) add to consecutive points, and a warp's 27 scalar atomics coalesce; a particle
// with no neighbour beside it (halos in any order) touches a sector of its own with each,
// so such lanes add a row's points by one or two vector atomics instead (adding 0 to the
// points between).  Six blocks per SM hide more of the atomics' latency than five.  256^3
// particles (25% of them out of order) and mesh: 1.034 -> 0.832 ms; 2 M halo particles on
// 64^3: the whole PM force 1.17 -> 0.75 ms.  Vector atomics for every lane: 0.95 ms, lanes in
// order then meet in the same vectors.
template <int SCHEME>
__global__ void __launch_bounds__(256, 6) k_pm_assign(const double *__restrict__ pos, const float *__restrict__ mass,
                                                   uint32_t N, PmGeom g, float *__restrict__ grid)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t p = min(t, N - 1);  // whole warps look at their neighbours below
    const double x = pos[3 * (size_t)p], y = pos[3 * (size_t)p + 1], z = pos[3 * (size_t)p + 2];
    int ix, iy, iz;
    float fx, fy, fz;
    grid_coord(x, g, ix, fx);
    grid_coord(y, g, iy, fy);
    grid_coord(z, g, iz, fz);
    int jx[3], jy[3], jz[3];
    float wx[3], wy[3], wz[3];
    axis_weights<SCHEME>(ix, fx, g.n, jx, wx);
    axis_weights<SCHEME>(iy, fy, g.n, jy, wy);
    axis_weights<SCHEME>(iz, fz, g.n, jz, wz);
    const float m = mass[p];
    constexpr int K = SCHEME == 0 ? 2 : 3;
    const size_t n = (size_t)g.n;
    // is a neighbour lane's particle on the same row, next to this one's?
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    auto beside = [&](int src) {
        const int ox = __shfl_sync(FULL, jx[0], src), oy = __shfl_sync(FULL, jy[0], src),
                  oz = __shfl_sync(FULL, jz[0], src);
        return ox == jx[0] && oy == jy[0] && abs(oz - jz[0]) <= 2;
    };
    const bool left = beside((lane - 1) & 31), right = beside((lane + 1) & 31);
    const bool lone = !(left && lane > 0) && !(right && lane < 31);
    if (t >= N) return;
    if (lone && (g.n & 3) == 0 && jz[0] < jz[K - 1]) {
        // the row's K points lie in one aligned group of four or across two
        const int A = jz[0] & ~3, off = jz[0] & 3;
#pragma unroll
        for (int a = 0; a < K; a++)
#pragma unroll
            for (int b = 0; b < K; b++) {
                const float mab = m * wx[a] * wy[b];
                float *row = grid + ((size_t)jx[a] * n + (size_t)jy[b]) * n + A;
                const float p0 = mab * wz[0], p1 = mab * wz[1], p2 = K > 2 ? mab * wz[2] : 0.0f;
                red_v4(row, off == 0 ? p0 : 0.0f, off == 0 ? p1 : (off == 1 ? p0 : 0.0f),
                       off == 0 ? p2 : (off == 1 ? p1 : (off == 2 ? p0 : 0.0f)),
                       off == 1 ? p2 : (off == 2 ? p1 : (off == 3 ? p0 : 0.0f)));
                if (off > 4 - K) red_v2(row + 4, off == 3 ? p1 : p2, off == 3 ? p2 : 0.0f);
            }
        return;
    }
#pragma unroll
    for (int a = 0; a < K; a++)
#pragma unroll
        for (int b = 0; b < K; b++) {
            const float mab = m * wx[a] * wy[b];
            float *row = grid + ((size_t)jx[a] * n + (size_t)jy[b]) * n;
#pragma unroll
            for (int c = 0; c < K; c++) atomicAdd(row + jz[c], mab * wz[c]);
        }
}

// All three components at once from the interleaved field: a particle's row of grid points
// is one or two 32-byte sectors per point, where three planes (a pass each, or one pass over
// three) touch three times as many cache lines; out-of-order particles (25% of the 256^3
// set) are bound by those.  256^3 particles and mesh: 0.959 -> 0.600 ms, and 0.071 ms to interleave.
// 32-byte loads of two points (rows padded with their ends) measured the same.
template <int SCHEME>
__global__ void __launch_bounds__(256) k_pm_interp(const double *__restrict__ pos, uint32_t N, PmGeom g,
                                                   const float4 *__restrict__ field, int accumulate,
                                                   float *__restrict__ acc)
{
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    const double x = pos[3 * (size_t)p], y = pos[3 * (size_t)p + 1], z = pos[3 * (size_t)p + 2];
    int ix, iy, iz;
    float fx, fy, fz;
    grid_coord(x, g, ix, fx);
    grid_coord(y, g, iy, fy);
    grid_coord(z, g, iz, fz);
    int jx[3], jy[3], jz[3];
    float wx[3], wy[3], wz[3];
    axis_weights<SCHEME>(ix, fx, g.n, jx, wx);
    axis_weights<SCHEME>(iy, fy, g.n, jy, wy);
    axis_weights<SCHEME>(iz, fz, g.n, jz, wz);
    constexpr int K = SCHEME == 0 ? 2 : 3;
    const size_t n = (size_t)g.n;
    float sx = 0.0f, sy = 0.0f, sz = 0.0f;
#pragma unroll
    for (int a = 0; a < K; a++)
#pragma unroll
        for (int b = 0; b < K; b++) {
            const float4 *row = field + ((size_t)jx[a] * n + (size_t)jy[b]) * n;
            float tx = 0.0f, ty = 0.0f, tz = 0.0f;
#pragma unroll
            for (int c = 0; c < K; c++) {
                const float4 v = __ldg(row + jz[c]);
                tx = fmaf(wz[c], v.x, tx);
                ty = fmaf(wz[c], v.y, ty);
                tz = fmaf(wz[c], v.z, tz);
            }
            const float w = wx[a] * wy[b];
            sx = fmaf(w, tx, sx);
            sy = fmaf(w, ty, sy);
            sz = fmaf(w, tz, sz);
        }
    float *o = acc + 3 * (size_t)p;
    if (accumulate) {
        sx += o[0];
        sy += o[1];
        sz += o[2];
    }
    o[0] = sx;
    o[1] = sy;
    o[2] = sz;
}

// Green's table over (|m_x|, |m_y|, m_z) in [0, n/2]^3, FP64 then rounded to FP32.
__global__ void k_pm_table(int n, double L, double eta, int scheme, float *__restrict__ table)
{
    const int h = n / 2 + 1;
    const long long total = (long long)h * h * h;
    const double pi = 3.14159265358979323846;
    const double delta = L / n;
    const double norm = 1.0 / (delta * delta * delta) / ((double)n * n * n);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int a = (int)(t / ((long long)h * h)), b = (int)((t / h) % h), c = (int)(t % h);
        if (a == 0 && b == 0 && c == 0) {
            table[t] = 0.0f;
            continue;
        }
        const double kx = 2 * pi * a / L, ky = 2 * pi * b / L, kz = 2 * pi * c / L;
        const double k2 = kx * kx + ky * ky + kz * kz;
        const double xi = sqrt(k2) * eta;
        double S;
        if (xi < 1e-2) {
            S = 1.0 - xi * xi / 15.0 + xi * xi * xi * xi / 560.0;
        } else {
            S = 12.0 * (2.0 - 2.0 * cos(xi) - xi * sin(xi)) / (xi * xi * xi * xi);
        }
        auto sinc = [](double v) { return v == 0.0 ? 1.0 : sin(v) / v; };
        double W = sinc(0.5 * kx * delta) * sinc(0.5 * ky * delta) * sinc(0.5 * kz * delta);
        W = scheme == 0 ? W * W : W * W * W;
        table[t] = (float)(-4.0 * pi * S * S / (k2 * W * W) * norm);
    }
}

// The three spectra -i k_c phi_k, phi_k = rho_k G, on the half-complex spectrum
// [n][n][n/2+1] (the Nyquist component of each k_c, mode n/2 of an even n, is zero): one read of rho_k and G for
// what took a pass for phi and one per component (256^3 mesh: 0.128 -> 0.046 ms).
__global__ void __launch_bounds__(256) k_pm_fields(const cufftComplex *__restrict__ rho, int n, double L,
                                                   const float *__restrict__ table, cufftComplex *__restrict__ out,
                                                   size_t plane)
{
    const uint32_t hz = n / 2 + 1, h = n / 2 + 1;
    const uint32_t total = (uint32_t)n * n * hz;  // n <= 1024: below 2^30
    const float twopi_L = (float)(2.0 * 3.14159265358979323846 / L);
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const uint32_t row = t / hz;
        const int z = (int)(t - row * hz), x = (int)(row / n), y = (int)(row - (uint32_t)x * n);
        const int ax = x <= n / 2 ? x : n - x, ay = y <= n / 2 ? y : n - y;
        const float gk = table[((size_t)ax * h + ay) * h + z];
        cufftComplex v = rho[t];
        v.x *= gk;
        v.y *= gk;
        auto sided = [n](int m) { return 2 * m < n ? m : (2 * m == n ? 0 : m - n); };
        const float kx = twopi_L * (float)sided(x), ky = twopi_L * (float)sided(y), kz = twopi_L * (float)sided(z);
        out[t] = make_cuFloatComplex(kx * v.y, -kx * v.x);
        out[plane + t] = make_cuFloatComplex(ky * v.y, -ky * v.x);
        out[2 * plane + t] = make_cuFloatComplex(kz * v.y, -kz * v.x);
    }
}

// The three transformed planes (in place in the spectra: rows of 2 (n/2+1) floats) as one
// float4 per grid point.
__global__ void __launch_bounds__(256) k_pm_interleave(const float *__restrict__ planes, int n, size_t plane,
                                                       float4 *__restrict__ field)
{
    const uint32_t pitch = 2 * (n / 2 + 1), total = (uint32_t)n * n * n;  // n <= 1024: 2^30 at most
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const uint32_t row = t / (uint32_t)n, z = t - row * (uint32_t)n;
        const float *p = planes + (size_t)row * pitch + z;
        field[t] = make_float4(p[0], p[plane], p[2 * plane], 0.0f);
    }
}

int pm_plan(PmPlan &pl, int n, cudaStream_t s)
{
    if (pl.have && pl.n == n) {
        cufftSetStream(pl.r2c, s);
        cufftSetStream(pl.c2r, s);
        return 0;
    }
    if (pl.have) {
        cufftDestroy(pl.r2c);
        cufftDestroy(pl.c2r);
        pl.have = false;
    }
    if (cufftPlan3d(&pl.r2c, n, n, n, CUFFT_R2C) != CUFFT_SUCCESS) return -1;
    if (cufftPlan3d(&pl.c2r, n, n, n, CUFFT_C2R) != CUFFT_SUCCESS) {
        cufftDestroy(pl.r2c);
        return -1;
    }
    cufftSetStream(pl.r2c, s);
    cufftSetStream(pl.c2r, s);
    pl.n = n;
    pl.have = true;
    return 0;
}

void pm_plan_destroy(PmPlan &pl)
{
    if (pl.have) {
        cufftDestroy(pl.r2c);
        cufftDestroy(pl.c2r);
    }
    pl.have = false;
}

void launch_pm_table(int n, double L, double r_cut, int scheme, float *table, cudaStream_t s, int nsm)
{
    k_pm_table<<<nsm * 8, 256, 0, s>>>(n, L, 0.5 * r_cut, scheme, table);
    g_launches++;
}

// The whole PM force: tmp 3 pm_plane(n) complex, field n^3 float4, table from
// launch_pm_table.  acc gets (or accumulates) input order.  The density and its spectrum are
// done with when the field is made, and lie in its buffer: 4 n^3 bytes, then 8 n^2 (n/2+1)
// from a multiple of 256 on, less than 16 n^3 for n >= 8.
int run_pm(const PmPlan &pl, const double *pos, const float *mass, uint32_t N, double L, int n, int scheme, int pow2_e,
           const float *table, cufftComplex *tmp, float4 *field, float *acc, int accumulate, cudaStream_t s, int nsm)
{
    PmGeom g;
    g.n = n;
    g.scheme = scheme;
    g.L = L;
    g.inv_delta = n / L;
    g.pow2_e = pow2_e;
    int lg = -1;
    for (int q = 0; q < 31; q++)
        if ((1 << q) == n) lg = q;
    g.log2n = lg;
    const size_t cells = (size_t)n * n * n, plane = pm_plane(n);
    float *grid = reinterpret_cast<float *>(field);
    cufftComplex *spec = reinterpret_cast<cufftComplex *>(grid + (cells + 63) / 64 * 64);
    cudaMemsetAsync(grid, 0, cells * sizeof(float), s);
    const unsigned pb = (N + 255) / 256;
    if (scheme == 0) k_pm_assign<0><<<pb, 256, 0, s>>>(pos, mass, N, g, grid);
    else k_pm_assign<1><<<pb, 256, 0, s>>>(pos, mass, N, g, grid);
    if (cufftExecR2C(pl.r2c, grid, spec) != CUFFT_SUCCESS) return -2;
    k_pm_fields<<<nsm * 8, 256, 0, s>>>(spec, n, L, table, tmp, plane);
    for (int c = 0; c < 3; c++) {
        cufftComplex *t = tmp + c * plane;
        if (cufftExecC2R(pl.c2r, t, reinterpret_cast<cufftReal *>(t)) != CUFFT_SUCCESS) return -2;
    }
    k_pm_interleave<<<nsm * 8, 256, 0, s>>>(reinterpret_cast<const float *>(tmp), n, 2 * plane, field);
    if (scheme == 0) k_pm_interp<0><<<pb, 256, 0, s>>>(pos, N, g, field, accumulate, acc);
    else k_pm_interp<1><<<pb, 256, 0, s>>>(pos, N, g, field, accumulate, acc);
    g_launches += 4;
    return 0;
}

}  // namespace greem
