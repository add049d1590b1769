// flb_psi3c.cu -- one Runge-Kutta stage of the order-parameter equation (Sec. V)
// by small 3D tiles: the finite-difference and naive schemes and every Laplacian at
// all sizes, and the finite-volume scheme on boxes where the z-marching kernel of
// flb_psi3d.cu leaves the chip idle.
//
// A marching block works through its planes one after the other, 2 us a plane, and
// fills a pipeline of 8 planes first: a 64^3 box has 8 columns, so
// whatever the chunk a stage costs 20 us or more (142 us with 64-plane chunks).  Here
// a block owns 32 x 8 x 4 (16 x 8 x 4) sites and its threads walk whole columns of
// each region in registers, so that a stage is a chain of two or three phases:
//   noise  the normals of tile + 1 into shared memory, before the wait for the
//          kernel in front (they depend on nothing);
//   (mu)   mu of the stage input on tile + 2 (FV) or + 1 (FD), unless the step has
//          written it for the force (MU_IN);
//   (J)    FV: the flux M grad mu - u psi on tile + 1;
//   out    the increment and the stage output.
// psi, mu, u and E are read through L1 where they are used, without staging: what
// bounds a small box is the latency of the chain, a large one instruction issue
// (the FD noise above all: 13 normals on twice the sites, 1036 instructions per site at 72% of the
// slots; FV 707 and 452 at 64^3, at 52 and 43%).  Heun steps, marching with the best chunk and here, both in
// stream order: 64^3 FV 65.6 and 56 us, 32^3 FD 50 and 37; with launches overlapped and the
// polynomial normals 38.5 and 22.  96^3 FV with the Patra-Karttunen Laplacian 257 us with
// one thread per site and a launch per field, 109 here.
//
// The FV stages take the same explicitly rounded operations in the same order as
// psi3_fv_tma_block (per-plane partial sums included), so a field has the same bits
// whichever kernel wrote it.
#include "flb_psi3d.cuh"

namespace flb {

namespace {

// A block's tile of sites.
template <int X_, int Y_, int Z_>
struct Tile3 {
    static constexpr int CX = X_, CY = Y_, CZ = Z_, NT = 2 * CX * CY;  // NT: threads, two per output column, each CZ/2 planes
    static constexpr int CW1 = CX + 2, CH1 = CY + 2, CP1 = CW1 * CH1;  // flux and noise columns: tile + 1
    static constexpr int CW2 = CX + 4, CH2 = CY + 4;                   // FV mu columns: tile + 2
};
#define FLB_TILE3(T)                                                                                        \
    constexpr int CX = T::CX, CY = T::CY, CZ = T::CZ, NT = T::NT, CW1 = T::CW1, CH1 = T::CH1, CP1 = T::CP1, \
                  CW2 = T::CW2, CH2 = T::CH2;                                                               \
    (void)CX, (void)CY, (void)CZ, (void)NT, (void)CW1, (void)CH1, (void)CP1, (void)CW2, (void)CH2

struct CubeArgs {
    Psi3Args a;
    const float *mu;  // MU_IN: mu of the stage input, 2 ghost layers
    int naive;        // the naive noise (Sec. III) instead of FD's link noise
    float s1, s2, s3; // FD: sqrt(2 kT M a_l) of the face, edge and corner half-links
    float sd;         // naive: sqrt(2 kT M)
};

// Sums of one plane of a field at p (row pitch Y): the centre, the four in-plane faces,
// the four in-plane diagonals.
struct Plane3 {
    F1 a, b, d;
};
__device__ __forceinline__ Plane3 plane3(const float *p, int Y)
{
    auto at = [&](int o) { return F1{p[o]}; };
    Plane3 r;
    r.a = at(0);
    r.b = (at(-1) + at(1)) + (at(-Y) + at(Y));
    r.d = (at(-1 - Y) + at(1 - Y)) + (at(-1 + Y) + at(1 + Y));
    return r;
}

// mu on the columns of a region (tile + H) from psi in global memory, planes
// z0 - H .. z0 + nzt + H - 1, into smu [CZ + 2H][CY + 2H][CX + 2H].
template <class T, int H, bool W, bool FD>
__device__ __forceinline__ void form_mu(const Psi3Args &a, int x0, int y0, int z0, int nzt, float *smu)
{
    FLB_TILE3(T);
    constexpr int WX = CX + 2 * H, WY = CY + 2 * H;
    static_assert(WX * WY <= NT, "one thread per column of the region");
    const Geom &g = a.g;
    const int k = threadIdx.x, lx = k % WX, ly = k / WX;
    const int x = x0 - H + lx, y = y0 - H + ly;
    if (k >= WX * WY || x >= g.nx + H || y >= g.ny + H) return;
    const int Y = g.px, Z = g.px * g.py;
    const float k22 = a.K * (1.0f / 22.0f);
    const float *p = a.psi + g.pidx32(x, y, z0 - H - 1);
    Plane3 q0 = plane3(p, Y), q1 = plane3(p + Z, Y);
    // planes past a ragged box repeat its last one (loads stay unconditional, so that
    // those of all planes are in flight together); what they form is not used
#pragma unroll
    for (int j = 0; j < CZ + 2 * H; ++j) {
        const Plane3 q2 = plane3(p + min(j + 2, nzt + 2 * H + 1) * Z, Y);
        const F1 n1 = q1.b + (q0.a + q2.a), n2 = FD ? (q1.d + q0.b) + q2.b : q1.d + (q0.b + q2.b), n3 = q0.d + q2.d;
        const float ps = q1.a.v;
        smu[(j * WY + ly) * WX + lx] =
            W ? a.A * ps + a.B * ps * ps * ps - a.K * ((a.lw.c1 * n1.v + a.lw.c2 * n2.v) + (a.lw.c3 * n3.v + a.lw.c0 * ps))
            : FD ? a.A * ps + a.B * ps * ps * ps - k22 * (6.f * n1.v + 3.f * n2.v + n3.v - 80.f * ps)
                 : mu_so_v<F1>(a.A, a.B, k22, q1.a, n1, n2, n3).v;
        q0 = q1;
        q1 = q2;
    }
}

// The output of a stage at (x, y, z) from the increment D and the noise increment
// eta, pv the stage input there (Sec. V; operations and order as in
// psi3_fv_tma_block).
// e: the accumulator E there (later stages).
template <bool FIRST>
__device__ __forceinline__ void stage_out(const Psi3Args &a, int x, int y, int z, F1 pv, F1 e, F1 D, F1 eta)
{
    const Geom &g = a.g;
    const int si = x + g.nx * (y + g.ny * z);
    F1 out;
    if (!FIRST) {
        if (a.rk4 == 4) {
            out = vfma(D, 1.f / 6.f, e);
        } else if (a.rk4) {  // stages 2 and 3
            const F1 n{a.Dn[si]}, b{a.base[g.pidx32(x, y, z)]};
            a.E[si] = vfma(D, 1.f / 3.f, e).v;
            out = a.rk4 == 2 ? vfma(D + n, 0.5f, b) : (b + D) + n;
        } else {
            out = vfma(D, 0.5f, e);
        }
    } else if (a.rk4) {
        a.E[si] = vfma(D, 1.f / 6.f, pv + eta).v;
        a.Dn[si] = eta.v;
        out = vfma(D + eta, 0.5f, pv);
    } else {
        if (a.heun) a.E[si] = (vfma(D, 0.5f, pv) + eta).v;
        out = (pv + D) + eta;
    }
    store_padded(a.out, g, x, y, z, out.v, 3);
}

// ---------------------------------------------------------------------------
// Finite volume (operators of D3Q19, or of D3Q15 with Q15; see psi3_fv_tma_block).
// ---------------------------------------------------------------------------
// 12 (24) div of the vector planes v (each [CZ + 2][CH1][CW1]) by per-plane sums:
// what plane p gives to the divergence at p - 1, p and p + 1.
struct Div3 {
    F1 lo, mid, hi;
};
template <class T, bool Q15>
__device__ __forceinline__ Div3 div3(const float *v, int JN, int c)
{
    constexpr int Y = T::CW1;
    auto X = [&](int o) { return F1{v[c + o]}; };
    auto Yv = [&](int o) { return F1{v[JN + c + o]}; };
    auto Zv = [&](int o) { return F1{v[2 * JN + c + o]}; };
    const F1 hxy = (X(1) - X(-1)) + (Yv(Y) - Yv(-Y));
    const F1 dg = ((X(1 + Y) + Yv(1 + Y)) - (X(-1 - Y) + Yv(-1 - Y))) + ((X(1 - Y) - Yv(1 - Y)) - (X(-1 + Y) - Yv(-1 + Y)));
    const F1 zc = Zv(0);
    Div3 r;
    if (Q15) {
        const F1 c4 = (Zv(1 + Y) + Zv(1 - Y)) + (Zv(-1 + Y) + Zv(-1 - Y));
        r.lo = vfma(zc, 8.f, dg) + c4;
        r.mid = hxy;
        r.hi = vfma(zc, -8.f, dg - c4);
    } else {
        const F1 z4 = (Zv(1) + Zv(-1)) + (Zv(Y) + Zv(-Y));
        r.lo = vfma(zc, 2.f, hxy) + z4;
        r.mid = vfma(hxy, 2.f, dg);
        r.hi = vfma(zc, -2.f, hxy - z4);
    }
    return r;
}
// the divergence at a plane from its own and its neighbours' sums
template <bool Q15>
__device__ __forceinline__ F1 div_sum(const Div3 &below, const Div3 &own, const Div3 &above)
{
    return (Q15 ? vfma(own.mid, 8.f, below.hi) : below.hi + own.mid) + above.lo;
}

// shared memory of a block (floats)
template <class T, int NOISE, bool MU_IN>
__host__ __device__ constexpr int cube_fv_floats()
{
    return (T::CZ + 2) * T::CP1 * (NOISE ? 6 : 3) + (MU_IN ? 0 : (T::CZ + 4) * T::CW2 * T::CH2);
}

// The noise of the block's nodes (tile + 1) into sX, [3][CZ + 2][CH1][CW1].
template <class T, int NOISE>
__device__ __forceinline__ void cube_fv_noise(const Psi3Args &a, int x0, int y0, int z0, float *sX)
{
    FLB_TILE3(T);
    constexpr int JN = (CZ + 2) * CP1;
    const Geom &g = a.g;
    const float sdx = sqrtf(2.0f * a.kT * a.M);
    for (int k = threadIdx.x; k < JN; k += NT) {
        const int lx = k % CW1, ly = (k / CW1) % CH1, lz = k / CP1;
        const int x = x0 - 1 + lx, y = y0 - 1 + ly, z = z0 - 1 + lz;
        if (x > g.nx || y > g.ny || z > g.nz) continue;
        float G[4];
        const uint32_t id = (uint32_t)(wrapi(x, g.nx) + g.nx * (wrapi(y, g.ny) + g.ny * wrapi(z, g.nz)));
        normals<2, false, true, NOISE == 2>(a.key, a.step, id, 1u, 0u, G, sdx);
        sX[k] = G[0];
        sX[JN + k] = G[1];
        sX[2 * JN + k] = G[2];
    }
}

// The rest of a stage on the tile at (x0, y0, z0); the noise, if any, is in sX.
template <class T, bool FIRST, int NOISE, bool MU_IN, bool Q15, bool W>
__device__ __forceinline__ void cube_fv_stage(const Psi3Args &a, const float *mu, int x0, int y0, int z0, float *sJ,
                                              const float *sX, float *smu)
{
    FLB_TILE3(T);
    constexpr int JN = (CZ + 2) * CP1;
    const Geom &g = a.g;
    const int nzt = min(CZ, g.nz - z0);
    const int tx = threadIdx.x % CX, ty = (threadIdx.x / CX) % CY, zh = (threadIdx.x / (CX * CY)) * (CZ / 2);
    const bool act = x0 + tx < g.nx && y0 + ty < g.ny && zh < nzt;
    float e_pre[CZ / 2];  // a later stage's accumulator, in flight meanwhile
#pragma unroll
    for (int j = 0; j < CZ / 2; ++j)
        e_pre[j] = !FIRST && act ? a.E[x0 + tx + g.nx * (y0 + ty + g.ny * min(z0 + zh + j, g.nz - 1))] : 0.f;
    if (!MU_IN) {
        form_mu<T, 2, W, false>(a, x0, y0, z0, nzt, smu);
        __syncthreads();
    }
    {  // flux columns
        static_assert(CP1 <= NT, "one thread per flux column");
        const int k = threadIdx.x, lx = k % CW1, ly = k / CW1, x = x0 - 1 + lx, y = y0 - 1 + ly;
        if (k < CP1 && x <= g.nx && y <= g.ny) {
            const int Y = MU_IN ? g.px : CW2, Z = MU_IN ? g.px * g.py : CW2 * CH2;
            const int pi = g.pidx32(x, y, z0 - 1), pz = g.px * g.py;
            const float *m0 = MU_IN ? mu + (pi - pz) : smu + (lx + 1) + CW2 * (ly + 1);
            const float mg = a.M * (Q15 ? 1.0f / 24.0f : 1.0f / 12.0f);
            F1 G0[3], G1[3];
#pragma unroll
            for (int j = 0; j < CZ + 4; ++j) {
                const float *m = m0 + (MU_IN ? min(j, nzt + 3) : j) * Z;
                auto at = [&](int o) { return F1{m[o]}; };
                const F1 mxp = at(1), mxm = at(-1), myp = at(Y), mym = at(-Y);
                const F1 mpp = at(1 + Y), mpm = at(1 - Y), mmp = at(-1 + Y), mmm = at(-1 - Y);
                const F1 ex = mxp - mxm, ey = myp - mym;
                const F1 Dx = (mpp + mpm) - (mmp + mmm), Dy = (mpp + mmp) - (mpm + mmm);
                F1 gx, gy, gz;
                if (Q15) {
                    const F1 Zq = vfma(at(0), 8.f, (mpp + mpm) + (mmp + mmm));
                    if (j >= 2) {
                        gx = G0[0] + Dx;
                        gy = G0[1] + Dy;
                        gz = G0[2] + Zq;
                    }
                    if (j >= 1) {
                        G0[0] = vfma(ex, 8.f, G1[0]);
                        G0[1] = vfma(ey, 8.f, G1[1]);
                        G0[2] = G1[2];
                    }
                    G1[0] = Dx;
                    G1[1] = Dy;
                    G1[2] = Zq * -1.0f;
                } else {
                    const F1 Zp = vfma(at(0), 2.f, (mxp + mxm) + (myp + mym));
                    if (j >= 2) {
                        gx = G0[0] + ex;
                        gy = G0[1] + ey;
                        gz = G0[2] + Zp;
                    }
                    if (j >= 1) {
                        G0[0] = G1[0] + vfma(ex, 2.f, Dx);
                        G0[1] = G1[1] + vfma(ey, 2.f, Dy);
                        G0[2] = G1[2];
                    }
                    G1[0] = ex;
                    G1[1] = ey;
                    G1[2] = Zp * -1.0f;
                }
                if (j >= 2) {  // the flux of plane z0 - 1 + (j - 2)
                    F1 jx = gx * mg, jy = gy * mg, jz = gz * mg;
                    if (a.advect) {
                        const int o = pi + min(j - 2, nzt + 1) * pz;
                        const F1 npv = F1{a.psi[o]} * -1.0f;
                        jx = vfma(F1{a.u[o]}, npv, jx);
                        jy = vfma(F1{a.u[g.pn + o]}, npv, jy);
                        jz = vfma(F1{a.u[2 * g.pn + o]}, npv, jz);
                    }
                    float *J = sJ + (j - 2) * CP1 + k;
                    J[0] = jx.v;
                    J[JN] = jy.v;
                    J[2 * JN] = jz.v;
                }
            }
        }
    }
    __syncthreads();
    {  // output columns, planes zh .. zh + CZ/2 - 1 of the tile
        const int x = x0 + tx, y = y0 + ty;
        if (!act) return;
        constexpr float DIV = Q15 ? 1.0f / 24.0f : 1.0f / 12.0f;
        int c = (tx + 1) + CW1 * (ty + 1) + CP1 * zh;
        Div3 d0, d1, n0, n1;
        d0 = div3<T, Q15>(sJ, JN, c);
        d1 = div3<T, Q15>(sJ, JN, c + CP1);
        if (NOISE) {
            n0 = div3<T, Q15>(sX, JN, c);
            n1 = div3<T, Q15>(sX, JN, c + CP1);
        }
        c += 2 * CP1;
#pragma unroll
        for (int j = 0; j < CZ / 2; ++j, c += CP1) {
            const int z = z0 + zh + j;
            const Div3 d2 = div3<T, Q15>(sJ, JN, c);
            const F1 D = vmul_sep(div_sum<Q15>(d0, d1, d2), DIV);
            F1 eta = F1{0.f};
            if (NOISE) {
                const Div3 n2 = div3<T, Q15>(sX, JN, c);
                eta = vmul_sep(div_sum<Q15>(n0, n1, n2), DIV);
                n0 = n1;
                n1 = n2;
            }
            d0 = d1;
            d1 = d2;
            if (zh + j >= nzt) break;
            const F1 pv{FIRST ? a.psi[g.pidx32(x, y, z)] : 0.f};
            stage_out<FIRST>(a, x, y, z, pv, F1{e_pre[j]}, D, eta);
        }
    }
}

template <class T, bool FIRST, int NOISE, bool MU_IN, bool Q15, bool W>
__global__ void __launch_bounds__(T::NT) psi3_fv_cube_kernel(const CubeArgs ca)
{
    constexpr int JN = (T::CZ + 2) * T::CP1;
    extern __shared__ float csm[];
    float *sJ = csm, *sX = sJ + 3 * JN, *smu = sX + (NOISE ? 3 * JN : 0);  // smu: [CZ + 4][CH2][CW2] unless MU_IN
    const int x0 = blockIdx.x * T::CX, y0 = blockIdx.y * T::CY, z0 = blockIdx.z * T::CZ;
    pdl_trigger();
    if (NOISE) cube_fv_noise<T, NOISE>(ca.a, x0, y0, z0, sX);
    pdl_wait();
    cube_fv_stage<T, FIRST, NOISE, MU_IN, Q15, W>(ca.a, ca.mu, x0, y0, z0, sJ, sX, smu);
}

// ---------------------------------------------------------------------------
// Finite difference and the naive contrast: D = M lap mu - div_CD(u psi).
// ---------------------------------------------------------------------------
// half-links: x, y, z, (1,1,0), (1,-1,0), (1,0,1), (1,0,-1), (0,1,1), (0,1,-1),
// (1,1,1), (1,1,-1), (1,-1,1), (1,-1,-1): eta(r) = sum_l [zeta_l(r - c_l) - zeta_l(r)]
__device__ constexpr int8_t kCubeL[13][3] = {{1, 0, 0},  {0, 1, 0},  {0, 0, 1},  {1, 1, 0}, {1, -1, 0},
                                             {1, 0, 1},  {1, 0, -1}, {0, 1, 1},  {0, 1, -1}, {1, 1, 1},
                                             {1, 1, -1}, {1, -1, 1}, {1, -1, -1}};

// Without noise, 512 threads go three blocks an SM (40 registers; with 43 two, and at 512^3 a later
// stage with another Laplacian takes 2.30 ms instead of 1.75).  0: no bound.
template <class T, bool FIRST, int NOISE, bool MU_IN, bool W>
__global__ void __launch_bounds__(T::NT, NOISE == 0 && T::NT == 512 ? 3 : 0) psi3_fd_cube_kernel(const CubeArgs ca)
{
    FLB_TILE3(T);
    constexpr int ZN = (CZ + 2) * CP1;
    extern __shared__ float csm[];
    float *smu = csm;                                   // [CZ + 2][CH1][CW1] unless MU_IN
    float *sZ = csm + (MU_IN ? 0 : ZN);                 // 13 (naive 3) normals on tile + 1
    const Psi3Args &a = ca.a;
    const Geom &g = a.g;
    const int x0 = blockIdx.x * CX, y0 = blockIdx.y * CY, z0 = blockIdx.z * CZ;
    const int nzt = min(CZ, g.nz - z0);
    pdl_trigger();
    if (NOISE) {
        for (int k = threadIdx.x; k < ZN; k += NT) {
            const int lx = k % CW1, ly = (k / CW1) % CH1, lz = k / CP1;
            const int x = x0 - 1 + lx, y = y0 - 1 + ly, z = z0 - 1 + lz;
            if (x > g.nx || y > g.ny || z > g.nz) continue;
            const uint32_t id = (uint32_t)(wrapi(x, g.nx) + g.nx * (wrapi(y, g.ny) + g.ny * wrapi(z, g.nz)));
            if (ca.naive) {
                float G[4];
                normals<2, false, false, NOISE == 2>(a.key, a.step, id, 1u, 0u, G);
#pragma unroll
                for (int l = 0; l < 3; ++l) sZ[l * ZN + k] = G[l];
            } else {
                if (lx == CW1 - 1) continue;  // no half-link points to -x: the last column is not read
                float G[14];
                normals<4, false, false, NOISE == 2>(a.key, a.step, id, 1u, 0u, G);
                normals<3, false, false, NOISE == 2>(a.key, a.step, id, 1u, 1u, G + 8);
#pragma unroll
                for (int l = 0; l < 13; ++l) sZ[l * ZN + k] = (l < 3 ? ca.s1 : (l < 9 ? ca.s2 : ca.s3)) * G[l];
            }
        }
    }
    pdl_wait();
    const int tx = threadIdx.x % CX, ty = (threadIdx.x / CX) % CY, zh = (threadIdx.x / (CX * CY)) * (CZ / 2);
    const int x = x0 + tx, y = y0 + ty;
    const bool act = x < g.nx && y < g.ny && zh < nzt;
    float e_pre[CZ / 2];  // a later stage's accumulator, in flight while mu is formed
#pragma unroll
    for (int j = 0; j < CZ / 2; ++j)
        e_pre[j] = !FIRST && act ? a.E[x + g.nx * (y + g.ny * min(z0 + zh + j, g.nz - 1))] : 0.f;
    if (!MU_IN) form_mu<T, 1, W, true>(a, x0, y0, z0, nzt, smu);
    if (NOISE || !MU_IN) __syncthreads();
    if (!act) return;
    const int Y = MU_IN ? g.px : CW1, Z = MU_IN ? g.px * g.py : CP1;
    const float *m = MU_IN ? ca.mu + g.pidx32(x, y, z0 + zh - 1) : smu + (tx + 1) + CW1 * (ty + 1) + CP1 * zh;
    Plane3 q0 = plane3(m, Y), q1 = plane3(m + Z, Y);
#pragma unroll
    for (int j = 0; j < CZ / 2; ++j) {
        const int z = z0 + zh + j;
        if (zh + j >= nzt) break;
        const Plane3 q2 = plane3(m + (j + 2) * Z, Y);
        const float n1 = (q1.b + (q0.a + q2.a)).v, n2 = ((q1.d + q0.b) + q2.b).v, n3 = (q0.d + q2.d).v;
        float D = W ? a.M * ((a.lw.c1 * n1 + a.lw.c2 * n2) + (a.lw.c3 * n3 + a.lw.c0 * q1.a.v))
                    : a.M * ((1.0f / 22.0f) * (6.f * n1 + 3.f * n2 + n3 - 80.f * q1.a.v));
        q0 = q1;
        q1 = q2;
        const int pi = g.pidx32(x, y, z);
        if (a.advect) {
            const int sy = g.px, sz = g.px * g.py;
            const float *u = a.u + pi, *v = u + g.pn, *w = v + g.pn, *p = a.psi + pi;
            const float adv = (u[1] * p[1] - u[-1] * p[-1]) +
                              (v[sy] * p[sy] - v[-sy] * p[-sy]) +
                              (w[sz] * p[sz] - w[-sz] * p[-sz]);
            D -= 0.5f * adv;
        }
        float eta = 0.f;
        if (NOISE) {
            const int c = (tx + 1) + CW1 * (ty + 1) + CP1 * (zh + j + 1);
            if (ca.naive) {
                eta = 0.5f * ca.sd * ((sZ[c + 1] - sZ[c - 1]) + (sZ[ZN + c + CW1] - sZ[ZN + c - CW1]) +
                                      (sZ[2 * ZN + c + CP1] - sZ[2 * ZN + c - CP1]));
            } else {
                float own = 0.f, in0 = 0.f, up = 0.f, dn = 0.f;
#pragma unroll
                for (int l = 0; l < 13; ++l) {
                    own += sZ[l * ZN + c];
                    const float v = sZ[l * ZN + c - kCubeL[l][0] - CW1 * kCubeL[l][1] - CP1 * kCubeL[l][2]];
                    if (kCubeL[l][2] == 0) in0 += v;
                    else if (kCubeL[l][2] > 0) up += v;
                    else dn += v;
                }
                eta = (up + (in0 - own)) + dn;
            }
        }
        const F1 own{FIRST ? a.psi[pi] : 0.f};
        stage_out<FIRST>(a, x, y, z, own, F1{e_pre[j]}, F1{D}, F1{eta});
    }
}

template <class K>
cudaError_t go(K k, const CubeArgs &ca, dim3 grid, int threads, int floats, cudaStream_t st)
{
    const int smem = (int)sizeof(float) * floats;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e != cudaSuccess ? e : launch_pdl(k, grid, threads, smem, st, PDL_BLOCKS, ca);
}

template <class T, bool FIRST, int NOISE, bool MU_IN, bool W>
cudaError_t go_fd(const CubeArgs &ca, dim3 grid, cudaStream_t st)
{
    const int zn = (T::CZ + 2) * T::CP1;
    return go(psi3_fd_cube_kernel<T, FIRST, NOISE, MU_IN, W>, ca, grid, T::NT,
              zn * ((MU_IN ? 0 : 1) + (NOISE ? (ca.naive ? 3 : 13) : 0)), st);
}
template <class T, bool FIRST, int NOISE, bool MU_IN, bool Q15, bool W>
cudaError_t go_fv(const CubeArgs &ca, dim3 grid, cudaStream_t st)
{
    return go(psi3_fv_cube_kernel<T, FIRST, NOISE, MU_IN, Q15, W>, ca, grid, T::NT, cube_fv_floats<T, NOISE, MU_IN>(), st);
}

template <class T, bool MU_IN, bool W>
cudaError_t first_fd(const CubeArgs &ca, int noise, dim3 g, cudaStream_t st)
{
    return noise == 2 ? go_fd<T, true, 2, MU_IN, W>(ca, g, st)
           : noise    ? go_fd<T, true, 1, MU_IN, W>(ca, g, st)
                      : go_fd<T, true, 0, MU_IN, W>(ca, g, st);
}
template <class T, bool MU_IN, bool Q15, bool W>
cudaError_t first_fv(const CubeArgs &ca, int noise, dim3 g, cudaStream_t st)
{
    return noise == 2 ? go_fv<T, true, 2, MU_IN, Q15, W>(ca, g, st)
           : noise    ? go_fv<T, true, 1, MU_IN, Q15, W>(ca, g, st)
                      : go_fv<T, true, 0, MU_IN, Q15, W>(ca, g, st);
}

template <class T, bool W>
cudaError_t fd_cube(const CubeArgs &ca, bool first, int noise, dim3 g, cudaStream_t st)
{
    if (!first) return go_fd<T, false, 0, false, W>(ca, g, st);
    if (ca.mu) return first_fd<T, true, W>(ca, noise, g, st);
    return first_fd<T, false, W>(ca, noise, g, st);
}

template <class T, bool Q15>
cudaError_t fv_cube(const CubeArgs &ca, bool first, int noise, dim3 g, cudaStream_t st)
{
    const bool w = ca.a.lap_w;
    if (!first) return w ? go_fv<T, false, 0, false, Q15, true>(ca, g, st)
                         : go_fv<T, false, 0, false, Q15, false>(ca, g, st);
    if (ca.mu) return first_fv<T, true, Q15, false>(ca, noise, g, st);
    if (w) return first_fv<T, false, Q15, true>(ca, noise, g, st);
    return first_fv<T, false, Q15, false>(ca, noise, g, st);
}

template <class T>
cudaError_t tile_cube(const CubeArgs &ca, int scheme, int q, bool first, int noise, cudaStream_t st)
{
    const Geom &g = ca.a.g;
    const dim3 grid((g.nx + T::CX - 1) / T::CX, (g.ny + T::CY - 1) / T::CY, (g.nz + T::CZ - 1) / T::CZ);
    if (scheme == FLB_FV) return q == 15 ? fv_cube<T, true>(ca, first, noise, grid, st) : fv_cube<T, false>(ca, first, noise, grid, st);
    return ca.a.lap_w ? fd_cube<T, true>(ca, first, noise, grid, st) : fd_cube<T, false>(ca, first, noise, grid, st);
}

// 32 x 8 x 4 tiles (halo factors 3.4 and 2.0 for mu and flux, rows of a full warp)
// where they make a block for two SMs in three and do not idle in x; 16 x 8 x 4 else.
// A Heun step at 64^3 took 65.7 us with 16-wide tiles and 56.1 us with 32-wide ones, FD at
// 160^3 495 and 467 us; at 32^3 (64 or 32 blocks) both 38 us.  Taller and deeper tiles (16 x 16 x 4, 16 x 8 x 8,
// 32 x 8 x 8) were level or slower up to 96^3, FD at any size.
bool wide_tile(const Geom &g)
{
    const int wide = (g.nx + 31) / 32, narrow = (g.nx + 15) / 16;
    const long long rows = (long long)((g.ny + 7) / 8) * ((g.nz + 3) / 4);
    return wide * rows >= 100 && 20 * wide <= 11 * narrow;
}

}  // namespace

cudaError_t launch_psi3_cube(const Psi3Args &a, int scheme, int q, bool first, int noise, const float *mu_in,
                             cudaStream_t st)
{
    CubeArgs ca;
    ca.a = a;
    ca.mu = first ? mu_in : nullptr;
    ca.naive = scheme == FLB_NAIVE;
    const float v = 2.0f * a.kT * a.M;
    ca.sd = sqrtf(v);
    ca.s1 = sqrtf(v * (a.lap_w ? a.lw.c1 : 6.f / 22.f));
    ca.s2 = sqrtf(v * (a.lap_w ? a.lw.c2 : 3.f / 22.f));
    ca.s3 = sqrtf(v * (a.lap_w ? a.lw.c3 : 1.f / 22.f));
    return wide_tile(a.g) ? tile_cube<Tile3<32, 8, 4>>(ca, scheme, q, first, noise, st)
                          : tile_cube<Tile3<16, 8, 4>>(ca, scheme, q, first, noise, st);
}

}  // namespace flb
