// flb_step2d.cu -- the D2Q9 time step in one launch for the fluid and one per
// Runge-Kutta stage of psi (a Heun step is three launches).
//
//   lb2_kernel        forms mu (or the stress sigma) of psi^n on the block's tile + 1
//                     in shared memory, the force density from it, pulls the nine
//                     populations, relaxes them with noise (Sec. IV, App. B) and
//                     stores the post-collision populations.
//   psi2_kernel FIRST pulls the just-written populations on tile + 1, forms the
//                     velocity (sum fbar c + F/2)/rho of the new fluid state there
//                     (Gauss-Seidel coupling, Sec. VI), draws the step's noise and
//                     takes the first stage; the velocity is stored for the later
//                     stages and for the observables.
//   psi2_kernel       a later stage: mu of the stage input, its increment, the output.
//
// What bounds them: the populations go through HBM twice read and once written
// (108 B/site; a step moves 134 at 2048^2), but a large box is bound by
// instruction issue (65% of the slots in lb2_kernel, 78 and 86% in the two stages; 454, 683 and 262
// instructions per site): a 2048^2 FD Heun step takes 204 us (383 us with one thread per
// site and one launch per field; 226 with a later stage's velocities and accumulator loaded
// where they are used, 213 with u psi in shared memory instead of u).  A small one is bound by
// latency, so what counts is the number of launches and what each has to wait for: 64^2
// takes 7.7 us a step (28.8 us with eight launches; 14.4 with these three in stream
// order).
#include "flb_internal.cuh"

namespace flb {

namespace {

template <typename T>
__device__ __forceinline__ float ldp(const T *p);
template <>
__device__ __forceinline__ float ldp<float>(const float *p) { return *p; }
template <>
__device__ __forceinline__ float ldp<__half>(const __half *p) { return __half2float(*p); }
__device__ __forceinline__ void stp(float *p, float v) { *p = v; }
__device__ __forceinline__ void stp(__half *p, float v) { *p = __float2half_rn(v); }

// The nine populations of site (x, y) from the post-collision planes at f
// (n sites each): fbar_i(r) = stored_i(r - c_i).  Planes: 0 rest; (1,2) +-x,
// (3,4) +-y, (5,6) +-(1,1), (7,8) +-(1,-1).
template <typename T>
__device__ __forceinline__ void pull9(const T *f, long long n, int nx, int ny, int x, int y, float v[9])
{
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    const int r0 = nx * y, rm = nx * (y == 0 ? ny - 1 : y - 1), rp = nx * (y == ny - 1 ? 0 : y + 1);
    v[0] = ldp(f + (r0 + x));
    v[1] = ldp(f + n + (r0 + xm));
    v[2] = ldp(f + 2 * n + (r0 + xp));
    v[3] = ldp(f + 3 * n + (rm + x));
    v[4] = ldp(f + 4 * n + (rp + x));
    v[5] = ldp(f + 5 * n + (rm + xm));
    v[6] = ldp(f + 6 * n + (rp + xp));
    v[7] = ldp(f + 7 * n + (rp + xm));
    v[8] = ldp(f + 8 * n + (rm + xp));
}

// Planar Laplacian with axis and diagonal weights w at c of a plane of row pitch P.
template <int P>
__device__ __forceinline__ float lap2(const float *f, int c, const LapW &w)
{
    const float n1 = f[c + 1] + f[c - 1] + f[c + P] + f[c - P];
    const float n2 = f[c + P + 1] + f[c - P - 1] + f[c - P + 1] + f[c + P - 1];
    return (w.c1 * n1 + w.c2 * n2) + w.c0 * f[c];
}

// Load the psi region tile + H (row pitch TX + 2H) of the block at (x0, y0); cells
// past a ragged box's ghost frame repeat its last column or row and are not used.
template <int TX, int TY, int H, int NT>
__device__ __forceinline__ void load_psi2(const Geom &g, const float *psi, int x0, int y0, float *s)
{
    constexpr int W = TX + 2 * H, N = W * (TY + 2 * H);
#pragma unroll
    for (int j = 0; j < (N + NT - 1) / NT; ++j) {
        const int k = (int)threadIdx.x + j * NT;
        if (k < N) {
            const int x = min(x0 - H + k % W, g.nx + GX - 1), y = min(y0 - H + k / W, g.ny + GY - 1);
            s[k] = psi[(x + GX) + g.px * (y + GY)];
        }
    }
}

// mu on tile + H from psi on tile + H + 1.
template <int TX, int TY, int H, int NT>
__device__ __forceinline__ void form_mu2(const float *sps, float *smu, float A, float B, float K, const LapW &lw)
{
    constexpr int W = TX + 2 * H, N = W * (TY + 2 * H), PW = W + 2;
#pragma unroll
    for (int j = 0; j < (N + NT - 1) / NT; ++j) {
        const int k = (int)threadIdx.x + j * NT;
        if (k < N) {
            const int c = (k % W + 1) + PW * (k / W + 1);
            const float p = sps[c];
            smu[k] = A * p + B * p * p * p - K * lap2<PW>(sps, c, lw);
        }
    }
}

// The order-parameter stress (Sec. IV, Eq. muf), planes xx, yy, xy, on tile + H:
// sigma_ab = K g_a g_b + delta_ab [A/2 psi^2 + 3B/4 psi^4 - K psi lap_SO psi - K/2 |g|^2].
template <int TX, int TY, int H, int NT>
__device__ __forceinline__ void form_sigma2(const float *sps, float *sg, float A, float B, float K)
{
    constexpr int W = TX + 2 * H, N = W * (TY + 2 * H), PW = W + 2;
    const LapW so{-3.f, 0.5f, 0.25f, 0.f};
#pragma unroll
    for (int j = 0; j < (N + NT - 1) / NT; ++j) {
        const int k = (int)threadIdx.x + j * NT;
        if (k < N) {
            const int c = (k % W + 1) + PW * (k / W + 1);
            const float p = sps[c], p2 = p * p;
            const float gx = 0.5f * (sps[c + 1] - sps[c - 1]), gy = 0.5f * (sps[c + PW] - sps[c - PW]);
            const float iso = 0.5f * A * p2 + 0.75f * B * p2 * p2 - K * p * lap2<PW>(sps, c, so) -
                              0.5f * K * (gx * gx + gy * gy);
            sg[k] = K * gx * gx + iso;
            sg[N + k] = K * gy * gy + iso;
            sg[2 * N + k] = K * gx * gy;
        }
    }
}

// the links of D2Q9
__device__ constexpr int8_t kLink9[8][2] = {{1, 0}, {-1, 0}, {0, 1}, {0, -1}, {1, 1}, {-1, -1}, {1, -1}, {-1, 1}};

// Force density at offset c of the mu plane (pitch P; or of the three stress
// planes of PN values): F = -psi grad mu with the central difference (kind 0) or
// the FV gradient [4 (mu(+x) - mu(-x)) + diagonals]/12 (kind 1), or -div sigma (kind 2).
template <int P, int PN>
__device__ __forceinline__ void force2(const float *m, int c, float ps, int kind, float &Fx, float &Fy)
{
    if (kind == 2) {
        const float *yy = m + PN, *xy = m + 2 * PN;
        Fx = -0.5f * ((m[c + 1] - m[c - 1]) + (xy[c + P] - xy[c - P]));
        Fy = -0.5f * ((xy[c + 1] - xy[c - 1]) + (yy[c + P] - yy[c - P]));
        return;
    }
    const float dx = m[c + 1] - m[c - 1], dy = m[c + P] - m[c - P];
    if (kind == 1) {
        const float pp = m[c + 1 + P], pm = m[c + 1 - P], mp = m[c - 1 + P], mm = m[c - 1 - P];
        Fx = -ps * (1.0f / 12.0f) * (4.f * dx + ((pp + pm) - (mp + mm)));
        Fy = -ps * (1.0f / 12.0f) * (4.f * dy + ((pp - pm) + (mp - mm)));
    } else {
        Fx = -ps * 0.5f * dx;
        Fy = -ps * 0.5f * dy;
    }
}

// ---------------------------------------------------------------------------
// Collide-stream of the sites s[l] of the lanes of V (their nine populations f
// and force density), the lanes in ok stored.  As on D3Q19 (flb_site3d.cuh) the
// stress is carried as Q = 4.5 B and the ghosts as h6 = g6/3, h7 = g7/3,
// h8 = 2 g8/9, with a.rq and a.nq in these units, so that
//   f_i = w_i [drho + 3 c_i.(j + F) + 4.5 (c_i c_i - I/3):B + ghosts]
// needs no further scale factors.  Noise order: bulk c^2 - 2/3, c_x^2 - c_y^2,
// c_x c_y, c_x(c^2 - 4/3), c_y(c^2 - 4/3), c^4-type ghost (2/9, -4/9 axes, 8/9 diagonals).
// ---------------------------------------------------------------------------
template <class V, typename T, bool GHOST_RELAX>
__device__ __forceinline__ void collide9(const LBArgs &a, const uint32_t *s, const bool *ok, const V f[9], const V n[6],
                                         V Fx, V Fy)
{
    constexpr int L = V::L;
    V sp[5], dp[5];
#pragma unroll
    for (int p = 1; p <= 4; ++p) {
        sp[p] = f[2 * p - 1] + f[2 * p];
        dp[p] = f[2 * p - 1] - f[2 * p];
    }
    const V s34 = sp[3] + sp[4];
    const V drho = f[0] + ((sp[1] + sp[2]) + s34);
    const V jx = dp[1] + (dp[3] + dp[4]), jy = dp[2] + (dp[3] - dp[4]);
    const V third = drho * (1.0f / 3.0f);
    const V Sxx = sp[1] + s34 - third, Syy = sp[2] + s34 - third, Sxy = sp[3] - sp[4];
    const V rho = drho + a.rho0;
    float ir[L];
#pragma unroll
    for (int l = 0; l < L; ++l) ir[l] = 1.0f / rho.lane(l);
    const V irho = vmake<V>(ir);
    const V vx = vfma(Fx, 0.5f, jx) * irho, vy = vfma(Fy, 0.5f, jy) * irho;
    const V cFx = Fx * a.rq[2], cFy = Fy * a.rq[2];
    const V wr = rho * a.rq[1];
    const V hx = vfma(wr, vx, cFx), hy = vfma(wr, vy, cFy);
    V Qxx = vfma(Sxx, a.rq[0], vx * (hx + cFx));
    V Qyy = vfma(Syy, a.rq[0], vy * (hy + cFy));
    V Qxy = vfma(Sxy, a.rq[0], vfma(vy, hx, vx * cFy));
    if (a.iso) {  // the trace relaxes at its own rate
        const V isoq = vfma(vfma(rho, vfma(vy, vy, vx * vx), (Sxx + Syy) * -1.0f), a.rq[3],
                            vfma(vy, Fy, vx * Fx) * a.rq[4]);
        Qxx = Qxx + isoq;
        Qyy = Qyy + isoq;
    }
    V h6 = V::bc(0.f), h7 = V::bc(0.f), h8 = V::bc(0.f);
    if (GHOST_RELAX) {  // gamma_g m_k / b_k in the units above (1/b = 27/2, 27/2, 81/16)
        const V gg = V::bc(a.gamma_g);
        h6 = gg * ((dp[3] + dp[4]) * 3.0f - dp[1] * 1.5f);
        h7 = gg * ((dp[3] - dp[4]) * 3.0f - dp[2] * 1.5f);
        h8 = gg * (f[0] * 0.25f + (s34 - (sp[1] + sp[2]) * 0.5f));
    }
    if (a.kT > 0.f) {
        const V mun = rho * a.k3T;
        float sq[L];
#pragma unroll
        for (int l = 0; l < L; ++l) sq[l] = sqrtf(mun.lane(l));
        const V sc = vmake<V>(sq);
        const V m0 = n[0] * a.nq[0], m1 = n[1] * a.nq[1];
        Qxx = vfma(m0 + m1, sc, Qxx);
        Qyy = vfma(m0 - m1, sc, Qyy);
        Qxy = vfma(n[2] * a.nq[2], sc, Qxy);
        h6 = vfma(n[3] * a.nq[3], sc, h6);
        h7 = vfma(n[4] * a.nq[4], sc, h7);
        h8 = vfma(n[5] * a.nq[5], sc, h8);
    }
    T *fo[L];
#pragma unroll
    for (int l = 0; l < L; ++l) fo[l] = (T *)a.fout + s[l];
    auto store = [&](int i, V v) {
#pragma unroll
        for (int l = 0; l < L; ++l)
            if (ok[l]) stp(fo[l] + i * a.g.n, v.lane(l));
    };
    const V tr = Qxx + Qyy;
    const V d = vfma(tr, -1.0f / 3.0f, drho);
    store(0, (d + h8) * (4.0f / 9.0f));
    constexpr float w1 = 1.0f / 9.0f, w2 = 1.0f / 36.0f;
    const V ax = (jx + Fx) * 3.0f, ay = (jy + Fy) * 3.0f;
    const V da = vfma(h8, -2.0f, d), dd = vfma(h8, 4.0f, d) + tr;
    const V Ex = da + Qxx, Ey = da + Qyy, Ox = ax - h6, Oy = ay - h7;
    store(1, (Ex + Ox) * w1);
    store(2, (Ex - Ox) * w1);
    store(3, (Ey + Oy) * w1);
    store(4, (Ey - Oy) * w1);
    const V E5 = vfma(Qxy, 2.0f, dd), E7 = vfma(Qxy, -2.0f, dd);
    const V O5 = vfma(h6 + h7, 2.0f, ax + ay), O7 = vfma(h6 - h7, 2.0f, ax - ay);
    store(5, (E5 + O5) * w2);
    store(6, (E5 - O5) * w2);
    store(7, (E7 + O7) * w2);
    store(8, (E7 - O7) * w2);
}

// The same for populations stored as FP16 deviations, one site, in the order of one
// kernel per phase and one thread per site: a last bit here moves roundings to 16 bits and with
// them psi by up to 4e-4 of itself in 200 steps (FP32 storage: 2e-6), so FP16 runs keep
// that order, here and in psi2_kernel's F16 branches.  G: the site's unit normals.
template <bool GHOST_RELAX>
__device__ __forceinline__ void collide9_f16(const LBArgs &a, uint32_t site, const float *f, const float *G, float Fx,
                                             float Fy)
{
    __half *fo = (__half *)a.fout;
    const long long N = a.g.n;
    float s[5], d[5];
#pragma unroll
    for (int p = 1; p <= 4; ++p) {
        s[p] = f[2 * p - 1] + f[2 * p];
        d[p] = f[2 * p - 1] - f[2 * p];
    }
    const float drho = f[0] + ((s[1] + s[2]) + (s[3] + s[4]));
    const float jx = d[1] + (d[3] + d[4]);
    const float jy = d[2] + (d[3] - d[4]);
    const float third = drho * (1.0f / 3.0f);
    const float Sxx = s[1] + (s[3] + s[4]) - third;
    const float Syy = s[2] + (s[3] + s[4]) - third;
    const float Sxy = s[3] - s[4];

    const float rho = a.rho0 + drho;
    const float irho = 1.0f / rho;
    const float vx = (jx + 0.5f * Fx) * irho, vy = (jy + 0.5f * Fy) * irho;

    const float ws = a.omega_s, wb = a.omega_b;
    const float cs = 1.0f - 0.5f * ws, cb = 1.0f - 0.5f * wb;
    const float Xxx = rho * vx * vx - Sxx, Xyy = rho * vy * vy - Syy;
    const float trX2 = 0.5f * (Xxx + Xyy);
    const float Txx = 2.f * vx * Fx, Tyy = 2.f * vy * Fy;
    const float trT2 = 0.5f * (Txx + Tyy);
    const float isoB = (wb - ws) * trX2 + (cb - cs) * trT2;
    float Bxx = Sxx + ws * Xxx + cs * Txx + isoB;
    float Byy = Syy + ws * Xyy + cs * Tyy + isoB;
    float Bxy = Sxy + ws * (rho * vx * vy - Sxy) + cs * (vx * Fy + Fx * vy);
    const float Ax = jx + Fx, Ay = jy + Fy;

    float g6 = 0.f, g7 = 0.f, g8 = 0.f;
    if (GHOST_RELAX) {
        const float gg = a.gamma_g;
        const float m6 = -(1.f / 3.f) * d[1] + (2.f / 3.f) * (d[3] + d[4]);
        const float m7 = -(1.f / 3.f) * d[2] + (2.f / 3.f) * (d[3] - d[4]);
        const float m8 = (2.f / 9.f) * f[0] - (4.f / 9.f) * (s[1] + s[2]) + (8.f / 9.f) * (s[3] + s[4]);
        g6 = gg * m6 * 13.5f;          // 1/b = 27/2
        g7 = gg * m7 * 13.5f;
        g8 = gg * m8 * (81.f / 16.f);  // 1/b = 81/16
    }
    if (a.kT > 0.f) {
        const float sq = sqrtf(3.0f * rho * a.kT);
        float n[6];
#pragma unroll
        for (int t = 0; t < 6; ++t) n[t] = sq * a.namp[t] * G[t];
        const float two9 = 2.0f / 9.0f;
        Bxx += two9 * (n[0] + n[1]);
        Byy += two9 * (n[0] - n[1]);
        Bxy += (1.0f / 9.0f) * n[2];
        g6 += n[3];
        g7 += n[4];
        g8 += n[5];
    }
    const float e0 = 1.5f * (Bxx + Byy);  // 9/2 trB/3
    stp(fo + site, (4.f / 9.f) * (drho - e0 + (2.f / 9.f) * g8));
    const float w1 = 1.f / 9.f, w2 = 1.f / 36.f;
    float E, O;
    E = drho + 4.5f * Bxx - e0 - (4.f / 9.f) * g8;
    O = 3.f * Ax - (1.f / 3.f) * g6;
    stp(fo + 1 * N + site, w1 * (E + O));
    stp(fo + 2 * N + site, w1 * (E - O));
    E = drho + 4.5f * Byy - e0 - (4.f / 9.f) * g8;
    O = 3.f * Ay - (1.f / 3.f) * g7;
    stp(fo + 3 * N + site, w1 * (E + O));
    stp(fo + 4 * N + site, w1 * (E - O));
    E = drho + 4.5f * (Bxx + Byy + 2.f * Bxy) - e0 + (8.f / 9.f) * g8;
    O = 3.f * (Ax + Ay) + (2.f / 3.f) * (g6 + g7);
    stp(fo + 5 * N + site, w2 * (E + O));
    stp(fo + 6 * N + site, w2 * (E - O));
    E = drho + 4.5f * (Bxx + Byy - 2.f * Bxy) - e0 + (8.f / 9.f) * g8;
    O = 3.f * (Ax - Ay) + (2.f / 3.f) * (g6 - g7);
    stp(fo + 7 * N + site, w2 * (E + O));
    stp(fo + 8 * N + site, w2 * (E - O));
}

// V = F2: a thread works the sites (x, y) and (x, y + TY/2) in packed FP32.
template <int TX, int TY, class V, typename T, bool GHOST_RELAX>
__global__ void __launch_bounds__(TX *TY / V::L) lb2_kernel(const LBArgs a, const Psi2Args p)
{
    constexpr int L = V::L, NT = TX * TY / L, MN = (TX + 2) * (TY + 2);
    __shared__ float sps[(TX + 4) * (TY + 4)], smu[3 * MN];
    const Geom &g = a.g;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX, x = x0 + tx;
    bool ok[L];
    uint32_t s[L];
    const int xc = min(x, g.nx - 1);  // off the box: a site of it, not stored
    int yc[L];
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const int y = y0 + ty + l * (TY / 2);
        ok[l] = x < g.nx && y < g.ny;
        yc[l] = min(y, g.ny - 1);
        s[l] = (uint32_t)(xc + g.nx * yc[l]);
    }
    pdl_trigger();
    constexpr bool F16 = sizeof(T) == 2;
    V n[6];  // unit normals, drawn while the kernel before this one ends
    float G[6];
    if (a.kT > 0.f) {
        if constexpr (F16) normals<3, false, false, true>(a.key, a.step, s[0], 0u, 0u, G);
        else lane_block<6, false>(a.key, a.step, s, 0u, V::bc(1.0f), n);
    }
    pdl_wait();
    V f[9];  // in flight while mu is formed
    {
        float fl[L][9];
#pragma unroll
        for (int l = 0; l < L; ++l) pull9((const T *)a.fin, g.n, g.nx, g.ny, xc, yc[l], fl[l]);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float t[L];
#pragma unroll
            for (int l = 0; l < L; ++l) t[l] = fl[l][i];
            f[i] = vmake<V>(t);
        }
    }
    float Fx[L], Fy[L];
#pragma unroll
    for (int l = 0; l < L; ++l) Fx[l] = Fy[l] = 0.f;
    if (a.coupling & FLB_COUPLE_FORCE) {
        load_psi2<TX, TY, 2, NT>(g, a.psi, x0, y0, sps);
        __syncthreads();
        if (a.force_kind == 2) form_sigma2<TX, TY, 1, NT>(sps, smu, p.A, p.B, p.K);
        else form_mu2<TX, TY, 1, NT>(sps, smu, p.A, p.B, p.K, p.lw);
        __syncthreads();
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const int yy = ty + l * (TY / 2);
            force2<TX + 2, MN>(smu, (tx + 1) + (TX + 2) * (yy + 1), sps[(tx + 2) + (TX + 4) * (yy + 2)], a.force_kind,
                               Fx[l], Fy[l]);
        }
    }
    if constexpr (F16) {
        static_assert(!F16 || L == 1, "one site per thread");
        float f1[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f1[i] = f[i].lane(0);
        if (ok[0]) collide9_f16<GHOST_RELAX>(a, s[0], f1, G, Fx[0], Fy[0]);
    } else {
        collide9<V, T, GHOST_RELAX>(a, s, ok, f, n, vmake<V>(Fx), vmake<V>(Fy));
    }
}

// ---------------------------------------------------------------------------
// One Runge-Kutta stage of psi on a TX x TY tile.
//   FD, naive: D = M lap mu - div_CD(u psi)      (Sec. V.A)
//   FV:        D = (2/c_s^2) sum_i w_i c_i . (J(r) + J(r + c_i))/2 with
//              J = M grad mu - u psi              (Sec. V.B; the J(r) terms cancel)
// The noise increment eta of the step (held fixed over its stages, Sec. V) from
// the normals of every point of tile + 1 (counter: the point's site id, Philox
// stream 1, block 0):
//   FD: sum_l sqrt(2 kT M a_l) [zeta_l(r - c_l) - zeta_l(r)] over the half-links
//       (1,0), (0,1), (1,1), (1,-1), a_l the Laplacian's axis and diagonal weights;
//   FV: the divergence above of xi, two N(0, 2 kT M) per node;
//   naive (Sec. III): (1/2) sum_a [xi_a(r + e_a) - xi_a(r - e_a)].
// s1 holds u (FD) or J (FV) on tile + 1, sz the normals there.
// ---------------------------------------------------------------------------
template <int TX, int TY, int NT, typename T, bool FV, bool FIRST, bool NOISE>
__global__ void __launch_bounds__(NT) psi2_kernel(const Psi2Args a)
{
    static_assert(FIRST || !NOISE, "the noise is drawn in the first stage");
    constexpr bool F16 = sizeof(T) == 2;  // see collide9_f16
    constexpr int MH = FIRST || FV ? 2 : 1, PH = MH + 1;          // mu and psi regions: tile + MH, + PH
    constexpr int W1 = TX + 2, N1 = W1 * (TY + 2);
    constexpr int WM = TX + 2 * MH, NM = WM * (TY + 2 * MH), WP = TX + 2 * PH, NP = WP * (TY + 2 * PH);
    constexpr int NZ = NOISE ? (FV ? 2 : 4) : 0;
    constexpr int J1 = (N1 + NT - 1) / NT;  // points of tile + 1 per thread
    extern __shared__ float sm2[];
    float *sps = sm2, *smu = sps + NP, *s1 = smu + NM, *sz = s1 + 2 * N1, *sg = sz + NZ * N1;  // sg: stress form
    const Geom &g = a.g;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const bool force = FIRST && (a.coupling & FLB_COUPLE_FORCE);
    const bool advect = (a.coupling & FLB_COUPLE_ADVECT) != 0;
    // points of tile + 1 outside the box and its first ghost layer are skipped
    auto point = [&](int k, int &lx, int &ly) {
        lx = k % W1 - 1;
        ly = k / W1 - 1;
        return k < N1 && x0 + lx <= g.nx && y0 + ly <= g.ny;
    };
    pdl_trigger();
    if (NOISE) {  // depends on nothing: drawn while the kernel before this one ends
#pragma unroll
        for (int j = 0; j < J1; ++j) {
            const int k = (int)threadIdx.x + j * NT;
            int lx, ly;
            if (!point(k, lx, ly)) continue;
            float G[4];
            normals<2, false, false, F16>(a.key, a.step, (uint32_t)(wrapi(x0 + lx, g.nx) + g.nx * wrapi(y0 + ly, g.ny)), 1u, 0u, G);
#pragma unroll
            for (int t = 0; t < NZ; ++t) sz[t * N1 + k] = G[t];
        }
    }
    pdl_wait();
    float f0[9];
    if (FIRST && J1 == 1) {  // one point per thread: its populations are in flight while mu is formed
        int lx, ly;
        if (point(threadIdx.x, lx, ly))
            pull9((const T *)a.f, g.n, g.nx, g.ny, wrapi(x0 + lx, g.nx), wrapi(y0 + ly, g.ny), f0);
    }
    // a later stage's velocities and accumulator, in flight while mu is formed
    constexpr int J0 = (TX * TY + NT - 1) / NT;
    float uxy[J1][2], e_pre[J0];
    if (!FIRST) {
#pragma unroll
        for (int j = 0; j < J1; ++j) {
            int lx, ly;
            const bool in = advect && point((int)threadIdx.x + j * NT, lx, ly);
            const int o = in ? (x0 + lx + GX) + g.px * (y0 + ly + GY) : 0;
            uxy[j][0] = in ? a.u[o] : 0.f;
            uxy[j][1] = in ? a.u[g.pn + o] : 0.f;
        }
#pragma unroll
        for (int j = 0; j < J0; ++j) {
            const int k = (int)threadIdx.x + j * NT, x = x0 + k % TX, y = y0 + k / TX;
            e_pre[j] = k < TX * TY && x < g.nx && y < g.ny ? a.E[x + g.nx * y] : 0.f;
        }
    }
    load_psi2<TX, TY, PH, NT>(g, a.psi, x0, y0, sps);
    __syncthreads();
    form_mu2<TX, TY, MH, NT>(sps, smu, a.A, a.B, a.K, a.lw);
    if (FIRST && force && a.force_kind == 2) form_sigma2<TX, TY, MH, NT>(sps, sg, a.A, a.B, a.K);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < J1; ++j) {
        const int k = (int)threadIdx.x + j * NT;
        int lx, ly;
        if (!point(k, lx, ly)) continue;
        const int x = x0 + lx, y = y0 + ly;
        const int cm = (lx + MH) + WM * (ly + MH);
        const float ps = sps[(lx + PH) + WP * (ly + PH)];
        float ux = 0.f, uy = 0.f;
        if (FIRST) {
            float f[9];
            if (J1 == 1)
                for (int i = 0; i < 9; ++i) f[i] = f0[i];
            else
                pull9((const T *)a.f, g.n, g.nx, g.ny, wrapi(x, g.nx), wrapi(y, g.ny), f);
            const float drho = f[0] + (((f[1] + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8])));
            const float jx = (f[1] - f[2]) + ((f[5] - f[6]) + (f[7] - f[8]));
            const float jy = (f[3] - f[4]) + ((f[5] - f[6]) - (f[7] - f[8]));
            float Fx = 0.f, Fy = 0.f;
            if (force) force2<WM, NM>(a.force_kind == 2 ? sg : smu, cm, ps, a.force_kind, Fx, Fy);
            const float irho = 1.0f / (a.rho0 + drho);
            ux = (jx + 0.5f * Fx) * irho;
            uy = (jy + 0.5f * Fy) * irho;
            if (lx >= 0 && lx < TX && ly >= 0 && ly < TY && x < g.nx && y < g.ny) {
                store_padded(a.u, g, x, y, 0, ux, 1);
                store_padded(a.u + g.pn, g, x, y, 0, uy, 1);
            }
        } else {
            ux = uxy[j][0];
            uy = uxy[j][1];
        }
        const float px = advect ? ux * ps : 0.f, py = advect ? uy * ps : 0.f;
        if (FV && F16) {
            float gx = 0.f, gy = 0.f;
#pragma unroll
            for (int l = 0; l < 8; ++l) {
                const float m = __fmul_rn(l < 4 ? 1.f / 9.f : 1.f / 36.f, smu[cm + kLink9[l][0] + WM * kLink9[l][1]]);
                gx = __fmaf_rn((float)kLink9[l][0], m, gx);
                gy = __fmaf_rn((float)kLink9[l][1], m, gy);
            }
            const float m3 = 3.f * a.M, jx = __fmul_rn(m3, gx), jy = __fmul_rn(m3, gy);
            s1[k] = advect ? __fmaf_rn(-ux, ps, jx) : jx;
            s1[N1 + k] = advect ? __fmaf_rn(-uy, ps, jy) : jy;
        } else if (FV) {
            const float dx = smu[cm + 1] - smu[cm - 1], dy = smu[cm + WM] - smu[cm - WM];
            const float pp = smu[cm + 1 + WM], pm = smu[cm + 1 - WM], mp = smu[cm - 1 + WM], mm = smu[cm - 1 - WM];
            s1[k] = a.M * ((1.f / 12.f) * (4.f * dx + ((pp + pm) - (mp + mm)))) - px;
            s1[N1 + k] = a.M * ((1.f / 12.f) * (4.f * dy + ((pp - pm) + (mp - mm)))) - py;
        } else {
            s1[k] = ux;
            s1[N1 + k] = uy;
        }
    }
    __syncthreads();
    // (2/c_s^2) link-average divergence of the pair of planes v on tile + 1
    auto div_fv = [&](const float *v, int c) {
        const float *vy = v + N1;
        const float ax = (v[c + 1] - v[c - 1]) + (vy[c + W1] - vy[c - W1]);
        const float dg = ((v[c + 1 + W1] + vy[c + 1 + W1]) - (v[c - 1 - W1] + vy[c - 1 - W1])) +
                         ((v[c + 1 - W1] - vy[c + 1 - W1]) - (v[c - 1 + W1] - vy[c - 1 + W1]));
        return (1.f / 12.f) * (4.f * ax + dg);
    };
#pragma unroll
    for (int j = 0; j < J0; ++j) {
        const int k = (int)threadIdx.x + j * NT;
        const int tx = k % TX, ty = k / TX, x = x0 + tx, y = y0 + ty;
        if (k >= TX * TY || x >= g.nx || y >= g.ny) continue;
        const int c = (tx + 1) + W1 * (ty + 1);
        const int cp = (tx + PH) + WP * (ty + PH);
        float D, eta = 0.f;
        if (FV && F16) {
            const float *vy = s1 + N1;
            float acc = 0.f;
#pragma unroll
            for (int l = 0; l < 8; ++l) {
                const int o = c + kLink9[l][0] + W1 * kLink9[l][1];
                const float cx = kLink9[l][0], cy = kLink9[l][1];
                const float lx = __fadd_rn(s1[c], s1[o]), ly = __fadd_rn(vy[c], vy[o]);
                acc = __fmaf_rn(l < 4 ? 1.f / 9.f : 1.f / 36.f, __fmaf_rn(cx, lx, cy * ly), acc);
            }
            D = __fmul_rn(3.f, acc);
        } else if (FV) {
            D = div_fv(s1, c);
        } else {
            D = a.M * lap2<WM>(smu, (tx + MH) + WM * (ty + MH), a.lw);
            if (advect) {
                const float *v = s1 + N1;
                float adv = s1[c + 1] * sps[cp + 1] - s1[c - 1] * sps[cp - 1];
                adv += v[c + W1] * sps[cp + WP] - v[c - W1] * sps[cp - WP];
                D -= 0.5f * adv;
            }
        }
        if (NOISE) {
            if (FV && F16) {
                const float *zx = sz, *zy = sz + N1;
                const float ox = zx[c], oy = zy[c];
                const float ax = ((ox + zx[c + 1]) - (ox + zx[c - 1])) + ((oy + zy[c + W1]) - (oy + zy[c - W1]));
                const float dg = ((ox + zx[c + W1 + 1]) + (oy + zy[c + W1 + 1])) -
                                 ((ox + zx[c - W1 - 1]) + (oy + zy[c - W1 - 1])) +
                                 ((ox + zx[c - W1 + 1]) - (oy + zy[c - W1 + 1])) -
                                 ((ox + zx[c + W1 - 1]) - (oy + zy[c + W1 - 1]));
                eta = 3.f * a.amp[0] * ((1.f / 9.f) * ax + (1.f / 36.f) * dg);
            } else if (FV) {
                eta = a.amp[0] * div_fv(sz, c);
            } else if (a.scheme == FLB_NAIVE) {
                eta = 0.5f * a.amp[0] * ((sz[c + 1] - sz[c - 1]) + (sz[N1 + c + W1] - sz[N1 + c - W1]));
            } else {
                eta = a.amp[1] * ((sz[c - 1] - sz[c]) + (sz[N1 + c - W1] - sz[N1 + c])) +
                      a.amp[2] * ((sz[2 * N1 + c - 1 - W1] - sz[2 * N1 + c]) + (sz[3 * N1 + c - 1 + W1] - sz[3 * N1 + c]));
            }
        }
        const int site = x + g.nx * y;
        const float ps = sps[cp];
        float out;
        if (a.integrator == FLB_RK4) {  // k_s = D_s + eta with eta fixed over the step
            if (FIRST) {
                out = ps + 0.5f * (D + eta);
                a.E[site] = ps + eta + D * (1.f / 6.f);
                a.eta[site] = eta;
            } else if (a.stage == 4) {
                out = e_pre[j] + D * (1.f / 6.f);
            } else {
                out = a.base[(x + GX) + g.px * (y + GY)] + (a.stage == 2 ? 0.5f : 1.f) * (D + a.eta[site]);
                a.E[site] = e_pre[j] + D * (1.f / 3.f);
            }
        } else if (FIRST) {
            out = ps + D + eta;
            if (a.integrator == FLB_HEUN) a.E[site] = ps + 0.5f * D + eta;
        } else {
            out = e_pre[j] + 0.5f * D;
        }
        store_padded(a.out, g, x, y, 0, out, 3);
    }
}

// Tiles: 32 x 16 where two blocks per SM of them cover the chip, else 16 x 8: a
// small box then has four times the blocks, each with one point per thread, and its
// latency is what a step costs.
// Every launch overlaps (launch_pdl): Heun steps, overlapped and in stream order, 256^2 11.2 and 16.6 us,
// 1024^2 54.5 and 63.7, 2048^2 205 and 214, 2560^2 314 and 323, 3072^2 442 and 451, 4096^2, the largest box,
// 768 and 777.
constexpr long long PDL_ALWAYS = 1LL << 62;
bool small_box2(const Geom &g) { return (long long)g.nx * g.ny < 304LL * 512; }

template <int TX, int TY, int NT, typename T, bool FV, bool FIRST, bool NOISE>
cudaError_t go_psi2(const Psi2Args &a, cudaStream_t st)
{
    constexpr int MH = FIRST || FV ? 2 : 1, PH = MH + 1;
    constexpr int N1 = (TX + 2) * (TY + 2), NM = (TX + 2 * MH) * (TY + 2 * MH), NP = (TX + 2 * PH) * (TY + 2 * PH);
    const bool stress = FIRST && (a.coupling & FLB_COUPLE_FORCE) && a.force_kind == 2;
    const size_t smem = sizeof(float) * (size_t)(NP + NM + (2 + (NOISE ? (FV ? 2 : 4) : 0)) * N1 + (stress ? 3 * NM : 0));
    const dim3 grid((a.g.nx + TX - 1) / TX, (a.g.ny + TY - 1) / TY);
    return launch_pdl(psi2_kernel<TX, TY, NT, T, FV, FIRST, NOISE>, grid, NT, smem, st, PDL_ALWAYS, a);
}

template <typename T, bool FV, bool FIRST, bool NOISE>
cudaError_t tile_psi2(const Psi2Args &a, cudaStream_t st)
{
    return small_box2(a.g) ? go_psi2<16, 8, 256, T, FV, FIRST, NOISE>(a, st)
                           : go_psi2<32, 16, 256, T, FV, FIRST, NOISE>(a, st);
}

template <bool FV>
cudaError_t scheme_psi2(const Psi2Args &a, int storage, bool noise, cudaStream_t st)
{
    if (storage == FLB_F16_DEV) {
        if (a.stage > 1) return tile_psi2<__half, FV, false, false>(a, st);
        return noise ? tile_psi2<__half, FV, true, true>(a, st) : tile_psi2<__half, FV, true, false>(a, st);
    }
    if (a.stage > 1) return tile_psi2<float, FV, false, false>(a, st);
    return noise ? tile_psi2<float, FV, true, true>(a, st) : tile_psi2<float, FV, true, false>(a, st);
}

template <int TX, int TY, class V, typename T>
cudaError_t go_lb2(const LBArgs &a, const Psi2Args &p, cudaStream_t st)
{
    constexpr int NT = TX * TY / V::L;
    const dim3 grid((a.g.nx + TX - 1) / TX, (a.g.ny + TY - 1) / TY);
    return a.gamma_g != 0.0f ? launch_pdl(lb2_kernel<TX, TY, V, T, true>, grid, NT, 0, st, PDL_ALWAYS, a, p)
                             : launch_pdl(lb2_kernel<TX, TY, V, T, false>, grid, NT, 0, st, PDL_ALWAYS, a, p);
}

}  // namespace

cudaError_t launch_lb2(const LBArgs &a, const Psi2Args &p, int storage, cudaStream_t st)
{
    if (storage == FLB_F16_DEV)
        return small_box2(a.g) ? go_lb2<16, 8, F1, __half>(a, p, st) : go_lb2<32, 8, F1, __half>(a, p, st);
    return small_box2(a.g) ? go_lb2<16, 8, F1, float>(a, p, st) : go_lb2<32, 16, F2, float>(a, p, st);
}

cudaError_t launch_psi2(const Psi2Args &a, int storage, bool noise, cudaStream_t st)
{
    return a.scheme == FLB_FV ? scheme_psi2<true>(a, storage, noise, st) : scheme_psi2<false>(a, storage, noise, st);
}

}  // namespace flb
