// flb_lb.cu -- populations outside the time step: equilibrium initialisation,
// the velocity of a drawn D2Q9 start, and the copies between padded and interior
// fields.
//
// Storage: populations are SoA planes [q][N] holding the POST-collision
// deviations fbar*_i - w_i rho0 at their origin site (not yet streamed).  A step
// pulls fbar_i(r, t) = stored_i(r - c_i), relaxes at r and stores the new
// post-collision values at r into the other buffer.
//
// Collision (D2Q9 in flb_step2d.cu, D3Q19 in flb_site3d.cuh, D3Q15 in
// flb_site15.cuh), written per opposite pair (c, -c) of velocities: with
// s = fbar_c + fbar_-c and d = fbar_c - fbar_-c the hydrodynamic moments are
// sums of s (mass, stress) and d (momentum).  Post-collision
//   fbar*_i = w_i [ rho + 3 A.c_i + 9/2 B:Q_i + sum_ghost e_k(c_i) g_k ],
//   A = j + F,  B = S + omega_s dev(X) + omega_b iso(X) + (1 - omega_s/2) dev(T)
//       + (1 - omega_b/2) iso(T) + (stress noise),  X = -S + rho v v,
//   T = v F + F v,  v = (j + F/2)/rho                              (Eq. bab)
// and every stress and ghost mode k receives sqrt(mu_n b_k (1 - gamma_k^2)) g_k,
// mu_n = rho kT / c_s^2 (thermalisation of all modes, Sec. III / adhikari2005).
// The ghost vectors e_k are the w-orthogonal (Gram-Schmidt) completions of the
// monomials c^2 c_a, c_a(c_b^2 - c_g^2), c^4, c^2(3c_x^2 - c^2), c^2(c_y^2 - c_z^2)
// (D3Q19) and c^2 c_a, c^4 (D2Q9), written out per velocity pair.
#include <algorithm>

#include "flb_internal.cuh"

namespace flb {

template <typename T>
__device__ __forceinline__ float ldpop(const T *p, long long i);
template <>
__device__ __forceinline__ float ldpop<float>(const float *p, long long i) { return __ldg(p + i); }
template <>
__device__ __forceinline__ float ldpop<__half>(const __half *p, long long i) { return __half2float(p[i]); }

template <typename T>
__device__ __forceinline__ void stpop(T *p, long long i, float v);
template <>
__device__ __forceinline__ void stpop<float>(float *p, long long i, float v) { p[i] = v; }
template <>
__device__ __forceinline__ void stpop<__half>(__half *p, long long i, float v) { p[i] = __float2half_rn(v); }

// Pull of the 9 populations of site (x, y) from the stored post-collision
// planes: fbar_i(r) = stored_i(r - c_i).
template <typename T>
__device__ __forceinline__ void pull9(const T *fi, const Geom &g, int x, int y, float f[9])
{
    const int xm = x == 0 ? g.nx - 1 : x - 1, xp = x == g.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? g.ny - 1 : y - 1, yp = y == g.ny - 1 ? 0 : y + 1;
    const long long N = g.n;
    f[0] = ldpop(fi, g.sidx(x, y, 0));
    f[1] = ldpop(fi, 1 * N + g.sidx(xm, y, 0));
    f[2] = ldpop(fi, 2 * N + g.sidx(xp, y, 0));
    f[3] = ldpop(fi, 3 * N + g.sidx(x, ym, 0));
    f[4] = ldpop(fi, 4 * N + g.sidx(x, yp, 0));
    f[5] = ldpop(fi, 5 * N + g.sidx(xm, ym, 0));
    f[6] = ldpop(fi, 6 * N + g.sidx(xp, yp, 0));
    f[7] = ldpop(fi, 7 * N + g.sidx(xm, yp, 0));
    f[8] = ldpop(fi, 8 * N + g.sidx(xp, ym, 0));
}

// Second-order equilibrium fbar = w rho (1 + 3 c.u + 9/2 (c.u)^2 - 3/2 u^2) of a
// given (rho, u) field, stored as post-collision deviations at the origin site:
// stored_i(r) = fbar_i(r + c_i) - w_i rho0.  rho and u are padded planes (rho may be null).
__constant__ int8_t kEq19[19][3] = {{0, 0, 0},  {1, 0, 0},   {-1, 0, 0}, {0, 1, 0},  {0, -1, 0},
                                    {0, 0, 1},  {0, 0, -1},  {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                                    {-1, 1, 0}, {1, 0, 1},   {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                                    {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
__constant__ int8_t kEq15[15][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0},  {0, 1, 0},   {0, -1, 0},
                                    {0, 0, 1},  {0, 0, -1}, {1, 1, 1},   {-1, -1, -1}, {1, 1, -1},
                                    {-1, -1, 1}, {1, -1, 1}, {-1, 1, -1}, {1, -1, -1}, {-1, 1, 1}};
__constant__ int8_t kEq9[9][3] = {{0, 0, 0}, {1, 0, 0}, {-1, 0, 0}, {0, 1, 0}, {0, -1, 0},
                                  {1, 1, 0}, {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0}};

// Velocity u = (sum fbar c)/rho of the D2Q9 populations at a.fout, streamed (the
// equilibrium start's; a step forms its own in flb_step2d.cu).
template <typename T>
__global__ void __launch_bounds__(256) vel_d2q9_kernel(const LBArgs a)
{
    const Geom &g = a.g;
    const long long site = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= g.n) return;
    const int x = (int)(site % g.nx);
    const int y = (int)(site / g.nx);
    float f[9];
    pull9((const T *)a.fout, g, x, y, f);
    const float drho = f[0] + (((f[1] + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8])));
    // planes (5,6) +-(1,1), (7,8) +-(1,-1)
    const float jx = (f[1] - f[2]) + ((f[5] - f[6]) + (f[7] - f[8]));
    const float jy = (f[3] - f[4]) + ((f[5] - f[6]) - (f[7] - f[8]));
    const float irho = 1.0f / (a.rho0 + drho);
    store_padded(a.u, g, x, y, 0, jx * irho, 1);
    store_padded(a.u + g.pn, g, x, y, 0, jy * irho, 1);
}

template <typename T>
__global__ void init_eq_kernel(const Geom g, int q, const float *__restrict__ rho, const float *__restrict__ u,
                               float rho0, T *__restrict__ fout)
{
    const long long site = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= g.n) return;
    const int x = (int)(site % g.nx);
    const int y = (int)((site / g.nx) % g.ny);
    const int z = (int)(site / ((long long)g.nx * g.ny));
    for (int i = 0; i < q; ++i) {
        const int8_t *c = q == 19 ? kEq19[i] : q == 15 ? kEq15[i] : kEq9[i];
        const long long pi = g.pidx(x + c[0], y + c[1], z + c[2]);
        const float r = rho ? rho[pi] : rho0;
        const float ux = u[pi], uy = u[g.pn + pi], uz = g.dim == 3 ? u[2 * g.pn + pi] : 0.f;
        const float cu = c[0] * ux + c[1] * uy + c[2] * uz;
        const float u2 = ux * ux + uy * uy + uz * uz;
        const float l2 = (float)(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
        const float w = q == 19   ? (l2 == 0.f ? 1.f / 3.f : l2 == 1.f ? 1.f / 18.f : 1.f / 36.f)
                        : q == 15 ? (l2 == 0.f ? 2.f / 9.f : l2 == 1.f ? 1.f / 9.f : 1.f / 72.f)
                                  : (l2 == 0.f ? 4.f / 9.f : l2 == 1.f ? 1.f / 9.f : 1.f / 36.f);
        stpop(fout, (long long)i * g.n + site, w * ((r - rho0) + r * (3.f * cu + 4.5f * cu * cu - 1.5f * u2)));
    }
}

// Padded plane (every ghost column, row and plane included) from an interior
// field [N], x fastest: each padded cell takes its periodic image.
__global__ void pad_kernel(const Geom g, const float *__restrict__ in, float *__restrict__ out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.pn) return;
    const int xp = (int)(i % g.px), yp = (int)((i / g.px) % g.py), zp = (int)(i / ((long long)g.px * g.py));
    const int x = ((xp - GX) % g.nx + g.nx) % g.nx, y = ((yp - GY) % g.ny + g.ny) % g.ny;
    const int z = g.dim == 3 ? ((zp - g.gz) % g.nz + g.nz) % g.nz : 0;
    out[i] = in[x + (long long)g.nx * (y + (long long)g.ny * z)];
}

// The interiors of padded fields, site-major, one after the other: p0 (if given), then
// the planes pn apart from p1.  Field blockIdx.z; a block takes 64 columns of four
// rows at a time, so a site's index costs no division.  (One launch per field with 64-bit divisions took 562 us a field at 512^3, 0.28 of
// the copy bandwidth.)
__global__ void __launch_bounds__(256) unpad_kernel(const Geom g, const float *__restrict__ p0, const float *__restrict__ p1,
                                                    float *__restrict__ out)
{
    const int f = blockIdx.z;
    const float *src = p0 && f == 0 ? p0 : p1 + (long long)(f - (p0 ? 1 : 0)) * g.pn;
    float *dst = out + (long long)f * g.n;
    const int x = blockIdx.x * 64 + (threadIdx.x & 63);
    if (x >= g.nx) return;
    for (int row = blockIdx.y * 4 + (threadIdx.x >> 6); row < g.ny * g.nz; row += gridDim.y * 4) {
        const int y = row % g.ny, z = row / g.ny;
        dst[(long long)row * g.nx + x] = __ldg(src + g.pidx32(x, y, z));
    }
}

// psi (may be null) and the nu components of u (may be null) to out, [field][N]
cudaError_t launch_unpad(const Geom &g, const float *psi, const float *u, int nu, float *out, cudaStream_t st)
{
    const int nf = (psi ? 1 : 0) + (u ? nu : 0);
    const dim3 grid((g.nx + 63) / 64, (unsigned)std::min<long long>(((long long)g.ny * g.nz + 3) / 4, 16384), nf);
    unpad_kernel<<<grid, 256, 0, st>>>(g, psi, u, out);
    return cudaGetLastError();
}

cudaError_t launch_pad(const Geom &g, const float *interior, float *padded, cudaStream_t st)
{
    pad_kernel<<<(unsigned)((g.pn + 255) / 256), 256, 0, st>>>(g, interior, padded);
    return cudaGetLastError();
}

cudaError_t launch_init_eq(const Geom &g, int q, int storage, const float *rho, const float *u, float rho0, void *f,
                           cudaStream_t st)
{
    const unsigned grid = (unsigned)((g.n + 255) / 256);
    if (storage == FLB_F16_DEV) init_eq_kernel<__half><<<grid, 256, 0, st>>>(g, q, rho, u, rho0, (__half *)f);
    else init_eq_kernel<float><<<grid, 256, 0, st>>>(g, q, rho, u, rho0, (float *)f);
    return cudaGetLastError();
}

cudaError_t launch_vel2(const LBArgs &a, int storage, cudaStream_t st)
{
    const int bs = 256;
    const unsigned grid = (unsigned)((a.g.n + bs - 1) / bs);
    if (storage == FLB_F16_DEV) vel_d2q9_kernel<__half><<<grid, bs, 0, st>>>(a);
    else vel_d2q9_kernel<float><<<grid, bs, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace flb
