// flb_obs.cu -- observables of Sec. VI of arXiv:1104.0078 reduced on the device:
// conserved totals and velocity variance (FP64, deterministic two-pass
// reduction), the static structure factor <|psi~(q)|^2> by a separable direct
// DFT accumulated in FP64, and the capillary spectrum of the two psi = 0
// surfaces of a slab (linear interpolation of the zero in every column).
#include "flb_obs.cuh"

namespace flb {

constexpr int RED_BS = 256;

template <typename T>
__device__ __forceinline__ float ldv(const T *p, long long i);
template <>
__device__ __forceinline__ float ldv<float>(const float *p, long long i) { return p[i]; }
template <>
__device__ __forceinline__ float ldv<__half>(const __half *p, long long i) { return __half2float(p[i]); }

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Pass 1: every block reduces a grid-stride share of the sites into NRED doubles:
// {sum dev, sum j_x, sum j_y, sum j_z, sum psi, sum u_x^2, sum u_y^2, sum u_z^2, non-finite count}.
template <typename T>
__global__ void __launch_bounds__(RED_BS) totals_kernel(const Geom g, int q, const T *__restrict__ f,
                                                        const float *__restrict__ psi, const float *__restrict__ u,
                                                        double *__restrict__ partial)
{
    double acc[NRED];
#pragma unroll
    for (int k = 0; k < NRED; ++k) acc[k] = 0.0;
    const long long N = g.n;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(s % g.nx), y = (int)((s / g.nx) % g.ny), z = (int)(s / ((long long)g.nx * g.ny));
        float m = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
        int bad = 0;
        float fi[19];
        for (int i = 0; i < q; ++i) {
            fi[i] = ldv(f, (long long)i * N + s);
            bad |= !isfinite(fi[i]);
        }
        if (q == 19) {
            m = fi[0];
            for (int i = 1; i < 19; ++i) m += fi[i];
            jx = (fi[1] - fi[2]) + (fi[7] - fi[8]) + (fi[9] - fi[10]) + (fi[11] - fi[12]) + (fi[13] - fi[14]);
            jy = (fi[3] - fi[4]) + (fi[7] - fi[8]) - (fi[9] - fi[10]) + (fi[15] - fi[16]) + (fi[17] - fi[18]);
            jz = (fi[5] - fi[6]) + (fi[11] - fi[12]) - (fi[13] - fi[14]) + (fi[15] - fi[16]) - (fi[17] - fi[18]);
        } else if (q == 15) {
            m = fi[0];
            for (int i = 1; i < 15; ++i) m += fi[i];
            // corner pairs (7,8) +(1,1,1), (9,10) +(1,1,-1), (11,12) +(1,-1,1), (13,14) +(1,-1,-1)
            const float d4 = fi[7] - fi[8], d5 = fi[9] - fi[10], d6 = fi[11] - fi[12], d7 = fi[13] - fi[14];
            jx = (fi[1] - fi[2]) + (d4 + d5) + (d6 + d7);
            jy = (fi[3] - fi[4]) + (d4 + d5) - (d6 + d7);
            jz = (fi[5] - fi[6]) + (d4 - d5) + (d6 - d7);
        } else {
            m = fi[0];
            for (int i = 1; i < 9; ++i) m += fi[i];
            jx = (fi[1] - fi[2]) + (fi[5] - fi[6]) + (fi[7] - fi[8]);
            jy = (fi[3] - fi[4]) + (fi[5] - fi[6]) - (fi[7] - fi[8]);
        }
        const long long pi = g.pidx(x, y, z);
        const float ps = psi[pi];
        const float ux = u[pi], uy = u[g.pn + pi], uz = g.dim == 3 ? u[2 * g.pn + pi] : 0.f;
        bad |= !isfinite(ps) | !isfinite(ux) | !isfinite(uy) | !isfinite(uz);
        acc[0] += m;
        acc[1] += jx;
        acc[2] += jy;
        acc[3] += jz;
        acc[4] += ps;
        acc[5] += (double)ux * ux;
        acc[6] += (double)uy * uy;
        acc[7] += (double)uz * uz;
        acc[8] += bad;
    }
    __shared__ double sh[RED_BS / 32][NRED];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NRED; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) sh[wid][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < NRED) {
        double t = 0.0;
        for (int w = 0; w < RED_BS / 32; ++w) t += sh[w][threadIdx.x];
        partial[(long long)blockIdx.x * NRED + threadIdx.x] = t;
    }
}

// Pass 2: one block of a warp per sum adds the nk sums of every first-pass block,
// each lane its own share and then the lanes, in a fixed order.  (One thread per
// sum, its loads one behind the other, took 77 us for 1024 blocks; this takes 7.)
__global__ void __launch_bounds__(32 * NMSQ) final_kernel(const double *__restrict__ partial, int nblocks, int nk,
                                                         double *__restrict__ out)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
    for (int b = lane; b < nblocks; b += 32) t += partial[(long long)b * nk + k];
    t = warp_sum(t);
    if (lane == 0) out[k] = t;
}

cudaError_t launch_totals(const Geom &g, int q, int storage, const void *f, const float *psi, const float *u,
                          double *partial, int nblocks, double *out, cudaStream_t s)
{
    if (storage == FLB_F16_DEV)
        totals_kernel<__half><<<nblocks, RED_BS, 0, s>>>(g, q, (const __half *)f, psi, u, partial);
    else
        totals_kernel<float><<<nblocks, RED_BS, 0, s>>>(g, q, (const float *)f, psi, u, partial);
    final_kernel<<<1, 32 * NRED, 0, s>>>(partial, nblocks, NRED, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Per-mode mean squares (Sec. III: every non-conserved mode carries
// <m_k^2> = (rho kT / c_s^2) b_k in equilibrium): each site pulls its physical
// populations fbar_i(r) = stored_i(r - c_i) (deviations from w_i rho0), projects
// them on the moment basis and adds m_k^2 in FP64; blocks reduce as for the totals.
// ---------------------------------------------------------------------------
__constant__ int8_t kMsq19[19][3] = {{0, 0, 0},  {1, 0, 0},   {-1, 0, 0}, {0, 1, 0},  {0, -1, 0},
                                     {0, 0, 1},  {0, 0, -1},  {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                                     {-1, 1, 0}, {1, 0, 1},   {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                                     {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
__constant__ int8_t kMsq15[15][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0},  {0, 1, 0},   {0, -1, 0},
                                     {0, 0, 1},  {0, 0, -1}, {1, 1, 1},   {-1, -1, -1}, {1, 1, -1},
                                     {-1, -1, 1}, {1, -1, 1}, {-1, 1, -1}, {1, -1, -1}, {-1, 1, 1}};
__constant__ int8_t kMsq9[9][3] = {{0, 0, 0}, {1, 0, 0}, {-1, 0, 0}, {0, 1, 0}, {0, -1, 0},
                                   {1, 1, 0}, {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0}};

template <typename T>
__global__ void __launch_bounds__(RED_BS) mode_msq_kernel(const Geom g, const ModeBasis B, const T *__restrict__ f,
                                                          double *__restrict__ partial)
{
    const int q = B.q;
    double acc[NMSQ];
#pragma unroll
    for (int k = 0; k < NMSQ; ++k) acc[k] = 0.0;
    const long long N = g.n;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(s % g.nx), y = (int)((s / g.nx) % g.ny), z = (int)(s / ((long long)g.nx * g.ny));
        float d[19];
        int bad = 0;
        for (int i = 0; i < q; ++i) {
            const int8_t *c = q == 19 ? kMsq19[i] : q == 15 ? kMsq15[i] : kMsq9[i];
            const long long src =
                g.sidx(wrapi(x - c[0], g.nx), wrapi(y - c[1], g.ny), g.dim == 3 ? wrapi(z - c[2], g.nz) : 0);
            d[i] = ldv(f, (long long)i * N + src);
            bad |= !isfinite(d[i]);
        }
        for (int k = 0; k < q; ++k) {
            float m = 0.f;
            for (int i = 0; i < q; ++i) m = fmaf(B.E[k * q + i], d[i], m);
            acc[k] += (double)m * m;
        }
        acc[NMSQ - 1] += bad;
    }
    __shared__ double sh[RED_BS / 32][NMSQ];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NMSQ; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) sh[wid][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < NMSQ) {
        double t = 0.0;
        for (int w = 0; w < RED_BS / 32; ++w) t += sh[w][threadIdx.x];
        partial[(long long)blockIdx.x * NMSQ + threadIdx.x] = t;
    }
}

cudaError_t launch_mode_msq(const Geom &g, int storage, const ModeBasis &B, const void *f, double *partial,
                            int nblocks, double *out, cudaStream_t s)
{
    if (storage == FLB_F16_DEV)
        mode_msq_kernel<__half><<<nblocks, RED_BS, 0, s>>>(g, B, (const __half *)f, partial);
    else
        mode_msq_kernel<float><<<nblocks, RED_BS, 0, s>>>(g, B, (const float *)f, partial);
    final_kernel<<<1, 32 * NMSQ, 0, s>>>(partial, nblocks, NMSQ, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Separable DFT.  Axis lists: index j of an axis of length n with window kmax
// (K = 2 kmax + 1 < n) is k = j for j <= kmax and n - (K - j) otherwise; with
// K = n every k is kept.  The field is real, so the component at -k is the
// conjugate of that at k: the x pass forms k_x = 0 .. Kx/2 only (nu = Kx/2 + 1 of
// them, the width of X1 and X2), the other passes work on those, and the last one
// writes each |.|^2 at both places.
// ---------------------------------------------------------------------------
// list index of -k for the list index j of k
__device__ __forceinline__ int conj_partner(int j, int n, int K) { return j == 0 ? 0 : (K >= n ? n - j : K - j); }

__device__ __forceinline__ float2 twiddle(int k, int x, int n)
{
    // e^{-2 pi i k x / n}, argument reduced exactly in integers first
    const int m = (int)(((long long)k * x) % n);
    float s, c;
    sincospif(2.0f * (float)m / (float)n, &s, &c);
    return make_float2(c, -s);
}

// Longest axis: the twiddle tables e^{-2 pi i m / n}, m < n, sit in shared memory;
// each output walks its phase index m = k x mod n by additions.
constexpr int TW_MAX = 4096;

// X1[(z*ny + y)*nu + j] = sum_x in(x,y,z) e^{-2 pi i j x / nx}, one output per thread,
// in NP partial sums over x mod NP (independent chains).
template <int NP>
__global__ void dft_x_kernel(DftArgs a)
{
    extern __shared__ float2 tw[];
    for (int m = threadIdx.x; m < a.nx; m += blockDim.x) tw[m] = twiddle(1, m, a.nx);
    __syncthreads();
    const int nu = a.Kx / 2 + 1;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long tot = (long long)nu * a.ny * a.nz;
    if (t >= tot) return;
    const int k = (int)(t % nu);
    const long long row = t / nu;  // z*ny + y
    const float *src = a.in + a.off + (row % a.ny) * a.sy + (row / a.ny) * a.sz;
    float re[NP] = {}, im[NP] = {};
    int m = 0, x = 0;
#pragma unroll 8 / NP
    for (; x + NP <= a.nx; x += NP) {
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const float v = __ldg(src + x + u);
            const float2 w = tw[m];
            re[u] = fmaf(v, w.x, re[u]);
            im[u] = fmaf(v, w.y, im[u]);
            m += k;
            if (m >= a.nx) m -= a.nx;
        }
    }
    for (; x < a.nx; ++x) {
        const float v = __ldg(src + x);
        const float2 w = tw[m];
        re[0] = fmaf(v, w.x, re[0]);
        im[0] = fmaf(v, w.y, im[0]);
        m += k;
        if (m >= a.nx) m -= a.nx;
    }
    a.X1[t] = NP == 4 ? make_float2((re[0] + re[1]) + (re[2] + re[NP - 1]), (im[0] + im[1]) + (im[2] + im[NP - 1]))
                      : make_float2(re[0], im[0]);
}

// The same X1 for windows of nu <= 18, as a small matrix product over blocks of
// rows.  A block builds the table e^{-2 pi i m / nx} once; chunks of DXR_CX columns
// of its rows are copied into two shared-memory buffers by cp.async (the next chunk
// in flight while the current one is summed), and the chunk's twiddles
// e^{-2 pi i k x / nx} (k x reduced mod nx exactly, as twiddle() does) are taken from
// the table.  S threads share a row, each summing every S-th column of a chunk, and
// add up at the end: 1 where 128-row blocks cover the chip, else 8 (2048 rows of
// 2048 with nu = 17 in 16 blocks would keep 16 SMs busy).
constexpr int DXR_NT = 128, DXR_CX = 32;

// dynamic shared memory of dft_x_rows_kernel<NUP, S> for rows of n
template <int NUP, int S>
constexpr size_t dxr_smem(int n)
{
    constexpr int R = DXR_NT / S;
    return R * sizeof(long long) + DXR_CX * NUP * sizeof(float2) + 2 * R * (DXR_CX + 1) * sizeof(float) + n * sizeof(float2);
}

template <int NUP, int S>
__global__ void __launch_bounds__(DXR_NT) dft_x_rows_kernel(DftArgs a, long long nrows)
{
    constexpr int R = DXR_NT / S, PS = R * (DXR_CX + 1);
    extern __shared__ __align__(16) unsigned char dsm[];
    long long *roff = reinterpret_cast<long long *>(dsm);                          // [R]
    float2 *Wc = reinterpret_cast<float2 *>(roff + R);                               // [DXR_CX][NUP]
    float *P = reinterpret_cast<float *>(Wc + DXR_CX * NUP);                        // [2][R][DXR_CX + 1]
    float2 *tw = reinterpret_cast<float2 *>(P + 2 * PS);                             // [n]
    const int n = a.nx, nu = a.Kx / 2 + 1, t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int row = t / S, sl = t % S;
    const int nch = (n + DXR_CX - 1) / DXR_CX;
    const long long r0 = (long long)blockIdx.x * R;
    for (int m = t; m < n; m += DXR_NT) tw[m] = twiddle(1, m, n);
    if (t < R) roff[t] = r0 + t < nrows ? a.off + ((r0 + t) % a.ny) * a.sy + ((r0 + t) / a.ny) * a.sz : -1;
    __syncthreads();
    // this thread's copies of chunk c: rows wp, wp + 4, ..., column x0 + lane
    auto stage = [&](int c) {
        float *buf = P + (c & 1) * PS;
        const int x = c * DXR_CX + lane;
        for (int rr = wp; rr < R; rr += DXR_NT / 32) {
            const long long o = roff[rr];
            const bool ok = o >= 0 && x < n;
            cp_async4(buf + rr * (DXR_CX + 1) + lane, a.in + (ok ? o + x : 0), ok ? 4 : 0);
        }
    };
    stage(0);
    cp_async_commit();
    float re[NUP], im[NUP];
#pragma unroll
    for (int j = 0; j < NUP; ++j) re[j] = im[j] = 0.f;
    for (int c = 0; c < nch; ++c) {
        if (c + 1 < nch) stage(c + 1);
        cp_async_commit();
        const int x0 = c * DXR_CX;
        for (int e = t; e < DXR_CX * NUP; e += DXR_NT) {
            const int i = e / NUP, j = e % NUP, x = x0 + i;
            Wc[e] = (j < nu && x < n) ? tw[(int)(((long long)j * x) % n)] : make_float2(0.f, 0.f);
        }
        cp_async_wait1();  // this thread's copies of chunk c have landed
        __syncthreads();   // everyone's copies of chunk c, and the chunk's twiddles
        const float *Pc = P + (c & 1) * PS + row * (DXR_CX + 1);
        const int cx = min(DXR_CX, n - x0);
        for (int i = sl; i < cx; i += S) {
            const float v = Pc[i];
#pragma unroll
            for (int j = 0; j < NUP; j += 2) {
                const float4 w = *reinterpret_cast<const float4 *>(&Wc[i * NUP + j]);
                re[j] = fmaf(v, w.x, re[j]);
                im[j] = fmaf(v, w.y, im[j]);
                re[j + 1] = fmaf(v, w.z, re[j + 1]);
                im[j + 1] = fmaf(v, w.w, im[j + 1]);
            }
        }
        __syncthreads();  // chunk c's buffer and twiddles are free again
    }
#pragma unroll
    for (int o = S / 2; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < NUP; ++j) {
            re[j] += __shfl_xor_sync(0xffffffffu, re[j], o);
            im[j] += __shfl_xor_sync(0xffffffffu, im[j], o);
        }
    if (sl == 0 && r0 + row < nrows) {
        float2 *o = a.X1 + (r0 + row) * nu;
#pragma unroll
        for (int j = 0; j < NUP; ++j)
            if (j < nu) o[j] = make_float2(re[j], im[j]);
    }
}

// The y and z passes: DFT along the middle axis of in[outer][n][C], columns
// (outer, c) to lanes, out[outer][K][C].  The components at k and -k share their
// products: with A = sum v_x c, B = sum v_y s, C = sum v_y c, D = sum v_x s,
//   X(k) = (A + B) + i (C - D),  X(-k) = (A - B) + i (C + D),
// so a thread carries PP such pairs.  The NS warps of a pair group take every NS-th
// term and are added in order at the end; a block has PB groups.
//   ACC: the sums' type (float in the y pass, double in the z pass).
//   LAST: instead of `out`, S += scale |X|^2 (and the snapshot) at k and at the conjugate place.
// The z pass is bound by the FP64 pipe (4 products a term and pair): one warp per
// output, without the pairs and the symmetry, took 515 us for all of a 64^3 box, and
// this 55; the window passes of a 512^3 box (|k| <= 8) 68 + 65 us, here 26 + 38; one
// thread per output took 664 us for the y pass of a 2048^2 box (|k| <= 16), here 76.
struct AxisArgs {
    const float2 *in;
    float2 *out;
    int outer, n, C, K;
    DftArgs d;  // LAST: S, scale, snap and the lists
};

template <class ACC>
struct Pair2;
template <>
struct Pair2<float> { using T = float2; };
template <>
struct Pair2<double> { using T = double2; };

template <class ACC, int PP, int NS, int PB, bool LAST>
__global__ void __launch_bounds__(32 * NS * PB) dft_axis_kernel(const AxisArgs a)
{
    using A2 = typename Pair2<ACC>::T;
    extern __shared__ __align__(16) unsigned char asm_[];
    A2 *tw = reinterpret_cast<A2 *>(asm_);                 // [n] (cos, sin)
    ACC *red = reinterpret_cast<ACC *>(tw + a.n);          // [PB][NS][4 PP][32]
    const int n = a.n;
    for (int m = threadIdx.x; m < n; m += blockDim.x) {
        const float2 w = twiddle(1, m, n);
        tw[m].x = w.x;
        tw[m].y = -w.y;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, pg = wp / NS, sl = wp % NS;
    const long long col = (long long)blockIdx.x * 32 + lane;
    const bool act = col < (long long)a.outer * a.C;
    const int o = act ? (int)(col / a.C) : 0, c = act ? (int)(col % a.C) : 0;
    const int npair = a.K / 2 + 1, p0 = (blockIdx.y * PB + pg) * PP;
    ACC acc[PP][4];
    int m[PP], step[PP];
#pragma unroll
    for (int q = 0; q < PP; ++q) {
        const int k = min(p0 + q, npair - 1);
        acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0;
        m[q] = (int)(((long long)k * sl) % n);
        step[q] = (int)(((long long)k * NS) % n);
    }
    const float2 *src = a.in + (long long)o * n * a.C + c;
    if (p0 < npair) {
#pragma unroll 4
        for (int r = sl; r < n; r += NS) {
            const float2 v = __ldg(src + (long long)r * a.C);
            const ACC vx = v.x, vy = v.y;
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                const A2 w = tw[m[q]];
                acc[q][0] += vx * w.x;
                acc[q][1] += vy * w.y;
                acc[q][2] += vy * w.x;
                acc[q][3] += vx * w.y;
                m[q] += step[q];
                if (m[q] >= n) m[q] -= n;
            }
        }
    }
    if (NS > 1) {
        ACC *mine = red + (pg * NS + sl) * (4 * PP) * 32 + lane;
#pragma unroll
        for (int q = 0; q < PP; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) mine[(4 * q + e) * 32] = acc[q][e];
        __syncthreads();
        if (sl != 0) return;
        const ACC *all = red + pg * NS * (4 * PP) * 32 + lane;
#pragma unroll
        for (int q = 0; q < PP; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                ACC t = all[(4 * q + e) * 32];
                for (int w = 1; w < NS; ++w) t += all[(w * 4 * PP + 4 * q + e) * 32];
                acc[q][e] = t;
            }
    }
    if (!act) return;
#pragma unroll
    for (int q = 0; q < PP; ++q) {
        const int j = p0 + q;
        if (j >= npair) break;
        const int jm = conj_partner(j, n, a.K);
        const ACC re[2] = {acc[q][0] + acc[q][1], acc[q][0] - acc[q][1]};
        const ACC im[2] = {acc[q][2] - acc[q][3], acc[q][2] + acc[q][3]};
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int jk = s ? jm : j;
            if (s && jm == j) break;
            if (!LAST) {
                a.out[((long long)o * a.K + jk) * a.C + c] = make_float2((float)re[s], (float)im[s]);
                continue;
            }
            const DftArgs &d = a.d;
            const int nu = d.Kx / 2 + 1, jx = c % nu;
            // planar fields end with the y pass (columns jx), others with the z pass (columns jx + nu jy)
            const int jy = d.nz == 1 ? jk : c / nu, jz = d.nz == 1 ? 0 : jk;
            const double val = d.scale * ((double)re[s] * re[s] + (double)im[s] * im[s]);
            const long long e = ((long long)jz * d.Ky + jy) * d.Kx + jx;
            if (d.S) d.S[e] += val;
            if (d.snap) d.snap[e] = make_float2((float)re[s], (float)im[s]);
            const int jxm = conj_partner(jx, d.nx, d.Kx);
            if (jxm == jx) continue;  // -k is another column's
            const long long em = ((long long)conj_partner(jz, d.nz, d.Kz) * d.Ky + conj_partner(jy, d.ny, d.Ky)) * d.Kx + jxm;
            if (d.S) d.S[em] += val;
            if (d.snap) d.snap[em] = make_float2((float)re[s], -(float)im[s]);
        }
    }
}

template <class ACC, int PP, int NS, int PB, bool LAST>
cudaError_t go_axis(const AxisArgs &a, long long groups, cudaStream_t s)
{
    const int npair = a.K / 2 + 1;
    const size_t smem = sizeof(ACC) * (2 * (size_t)a.n + (NS > 1 ? (size_t)PB * NS * 4 * PP * 32 : 0));
    auto k = dft_axis_kernel<ACC, PP, NS, PB, LAST>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<dim3((unsigned)groups, (unsigned)((npair + PP * PB - 1) / (PP * PB))), 32 * NS * PB, smem, s>>>(a);
    return cudaGetLastError();
}

// Four pairs a block (two groups of two pairs, four warps each) where that makes two
// blocks per SM, else one pair and eight warps: a short list of columns on a long axis is
// spread over as many SMs as it can.
template <class ACC, bool LAST>
cudaError_t launch_axis(const AxisArgs &a, cudaStream_t s)
{
    const long long groups = ((long long)a.outer * a.C + 31) / 32;
    return groups * ((a.K / 2 + 4) / 4) >= 304 ? go_axis<ACC, 2, 4, 2, LAST>(a, groups, s)
                                               : go_axis<ACC, 1, 8, 1, LAST>(a, groups, s);
}

// Dynamic structure factor: correlate the newest Fourier components with those
// of the nlag - 1 samples before them, in FP64.
__global__ void dyn_corr_kernel(const float2 *__restrict__ ring, int L, int slot, int nlag, long long K,
                                double *__restrict__ acc, double scale)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= K) return;
    const float2 c = ring[(long long)slot * K + t];
    int s = slot;
    for (int l = 0; l < nlag; ++l) {
        const float2 p = ring[(long long)s * K + t];
        acc[(long long)l * K + t] += scale * ((double)c.x * p.x + (double)c.y * p.y);
        s = s == 0 ? L - 1 : s - 1;
    }
}

cudaError_t launch_dyn_corr(const float2 *ring, int L, int slot, int nlag, long long K, double *acc, double scale,
                            cudaStream_t s)
{
    const int bs = 256;
    dyn_corr_kernel<<<(unsigned)((K + bs - 1) / bs), bs, 0, s>>>(ring, L, slot, nlag, K, acc, scale);
    return cudaGetLastError();
}

// The y pass of a planar field in a fixed order of summation, one output (j, jy) per
// thread in NP partial sums over y mod NP: S += scale |X|^2 at k and at its conjugate place.  For
// the interface heights: their mean is 10^3 times what the spectrum shows, so its small
// components carry the rounding of this order, which is therefore part of the result.
template <int NP>
__global__ void __launch_bounds__(128) dft_y_planar_kernel(DftArgs a)
{
    extern __shared__ float2 tw[];
    for (int m = threadIdx.x; m < a.ny; m += blockDim.x) tw[m] = twiddle(1, m, a.ny);
    __syncthreads();
    const int nu = a.Kx / 2 + 1, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nu * a.Ky) return;
    const int jx = t % nu, jy = t / nu;
    const int k = (a.Ky >= a.ny || jy <= a.Ky / 2) ? jy : a.ny - (a.Ky - jy);
    const float2 *src = a.X1 + jx;
    float re4[NP] = {}, im4[NP] = {};
    int m = 0, y = 0;
    auto add = [&](int u, float2 v) {
        const float2 w = tw[m];
        re4[u] += v.x * w.x - v.y * w.y;
        im4[u] += v.x * w.y + v.y * w.x;
        m += k;
        if (m >= a.ny) m -= a.ny;
    };
    constexpr int B = 16;  // loads in flight
    for (; y + B <= a.ny; y += B) {
        float2 v[B];
#pragma unroll
        for (int u = 0; u < B; ++u) v[u] = __ldg(src + (long long)(y + u) * nu);
#pragma unroll
        for (int u = 0; u < B; ++u) add(u % NP, v[u]);
    }
    for (; y + NP <= a.ny; y += NP)
#pragma unroll
        for (int u = 0; u < NP; ++u) add(u, __ldg(src + (long long)(y + u) * nu));
    for (; y < a.ny; ++y) add(0, __ldg(src + (long long)y * nu));
    const double re = NP == 4 ? (re4[0] + re4[1]) + (re4[2] + re4[NP - 1]) : re4[0];
    const double im = NP == 4 ? (im4[0] + im4[1]) + (im4[2] + im4[NP - 1]) : im4[0];
    const double val = a.scale * (re * re + im * im);
    a.S[(long long)jy * a.Kx + jx] += val;
    const int jxm = conj_partner(jx, a.nx, a.Kx);
    if (jxm != jx) a.S[(long long)conj_partner(jy, a.ny, a.Ky) * a.Kx + jxm] += val;
}

template <int NUP>
cudaError_t go_rows(const DftArgs &a, cudaStream_t s)
{
    const long long rows = (long long)a.ny * a.nz;
    auto go = [&](auto k, int per, size_t smem) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k<<<(unsigned)((rows + per - 1) / per), DXR_NT, smem, s>>>(a, rows);
        return cudaGetLastError();
    };
    return rows >= 152 * DXR_NT || a.ordered ? go(dft_x_rows_kernel<NUP, 1>, DXR_NT, dxr_smem<NUP, 1>(a.nx))
                                : go(dft_x_rows_kernel<NUP, 8>, DXR_NT / 8, dxr_smem<NUP, 8>(a.nx));
}

// kernels launched by launch_dft_accumulate
int dft_launches(const DftArgs &a) { return a.nz == 1 ? 2 : 3; }

cudaError_t launch_dft_accumulate(const DftArgs &a, cudaStream_t s)
{
    if (a.nx > TW_MAX || a.ny > TW_MAX || a.nz > TW_MAX) return cudaErrorInvalidValue;
    const int nu = a.Kx / 2 + 1;
    cudaError_t e;
    if (nu <= 2) e = go_rows<2>(a, s);
    else if (nu <= 4) e = go_rows<4>(a, s);
    else if (nu <= 6) e = go_rows<6>(a, s);
    else if (nu <= 10) e = go_rows<10>(a, s);
    else if (nu <= 18) e = go_rows<18>(a, s);
    else {
        const int bs = 256;
        const unsigned grid = (unsigned)(((long long)nu * a.ny * a.nz + bs - 1) / bs);
        if (a.ordered) dft_x_kernel<1><<<grid, bs, sizeof(float2) * a.nx, s>>>(a);
        else dft_x_kernel<4><<<grid, bs, sizeof(float2) * a.nx, s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    if (a.ordered) {  // planar; one chain for small windows, four for others
        const unsigned grid = (unsigned)((nu * a.Ky + 127) / 128);
        if (a.Kx * a.Ky <= 1024) dft_y_planar_kernel<1><<<grid, 128, sizeof(float2) * a.ny, s>>>(a);
        else dft_y_planar_kernel<4><<<grid, 128, sizeof(float2) * a.ny, s>>>(a);
        return cudaGetLastError();
    }
    const AxisArgs y{a.X1, a.X2, a.nz, a.ny, nu, a.Ky, a};
    if (a.nz == 1) return launch_axis<float, true>(y, s);
    e = launch_axis<float, false>(y, s);
    if (e != cudaSuccess) return e;
    return launch_axis<double, true>(AxisArgs{a.X2, nullptr, 1, a.nz, a.Ky * nu, a.Kz, a}, s);
}

// Heights of the two psi = 0 surfaces of a slab normal to z: in every column the
// first sign change in z in [0, nz/2) and in [nz/2, nz) (the next node wrapping
// periodically), located by linear interpolation; a half-column without a sign
// change reports the centre of its half.
__global__ void heights_kernel(const Geom g, const float *__restrict__ psi, float *__restrict__ h)
{
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long ncol = (long long)g.nx * g.ny;
    if (c >= ncol) return;
    const int x = (int)(c % g.nx), y = (int)(c / g.nx);
    const int half = g.nz / 2;
    for (int part = 0; part < 2; ++part) {
        const int lo = part == 0 ? 0 : half, hi = part == 0 ? half : g.nz;
        float hv = 0.5f * (float)(lo + hi);
        for (int z = lo; z < hi; ++z) {
            const float v0 = psi[g.pidx(x, y, z)], v1 = psi[g.pidx(x, y, z + 1 == g.nz ? 0 : z + 1)];
            if ((v0 < 0.f) != (v1 < 0.f)) {
                hv = (float)z + v0 / (v0 - v1);
                break;
            }
        }
        h[part * ncol + c] = hv;
    }
}

cudaError_t launch_heights(const Geom &g, const float *psi, float *h, cudaStream_t s)
{
    const long long ncol = (long long)g.nx * g.ny;
    heights_kernel<<<(unsigned)((ncol + 255) / 256), 256, 0, s>>>(g, psi, h);
    return cudaGetLastError();
}

}  // namespace flb

namespace flb {

__constant__ int8_t kWin19[19][3] = {{0, 0, 0},  {1, 0, 0},   {-1, 0, 0}, {0, 1, 0},  {0, -1, 0},
                                     {0, 0, 1},  {0, 0, -1},  {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                                     {-1, 1, 0}, {1, 0, 1},   {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                                     {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
__constant__ int8_t kWin15[15][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0},  {0, 1, 0},   {0, -1, 0},
                                     {0, 0, 1},  {0, 0, -1}, {1, 1, 1},   {-1, -1, -1}, {1, 1, -1},
                                     {-1, -1, 1}, {1, -1, 1}, {-1, 1, -1}, {1, -1, -1}, {-1, 1, 1}};
__constant__ int8_t kWin9[9][3] = {{0, 0, 0}, {1, 0, 0}, {-1, 0, 0}, {0, 1, 0}, {0, -1, 0},
                                   {1, 1, 0}, {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0}};

// Gather the physical (streamed) population deviations and psi of a periodic window.
template <typename T>
__global__ void window_kernel(const Geom g, int q, const T *__restrict__ f, const float *__restrict__ psi, int x0,
                              int y0, int z0, int wx, int wy, int wz, float *__restrict__ out)
{
    const long long W = (long long)wx * wy * wz;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= W) return;
    const int x = (x0 + (int)(k % wx)) % g.nx;
    const int y = (y0 + (int)((k / wx) % wy)) % g.ny;
    const int z = (z0 + (int)(k / ((long long)wx * wy))) % g.nz;
    for (int i = 0; i < q; ++i) {
        const int8_t *c = q == 19 ? kWin19[i] : q == 15 ? kWin15[i] : kWin9[i];
        const long long src = g.sidx(wrapi(x - c[0], g.nx), wrapi(y - c[1], g.ny), g.dim == 3 ? wrapi(z - c[2], g.nz) : 0);
        out[(long long)i * W + k] = ldv(f, (long long)i * g.n + src);
    }
    out[(long long)q * W + k] = psi[g.pidx(x, y, z)];
}

cudaError_t launch_window(const Geom &g, int q, int storage, const void *f, const float *psi, int x0, int y0, int z0,
                          int wx, int wy, int wz, float *out, cudaStream_t s)
{
    const long long W = (long long)wx * wy * wz;
    const unsigned grid = (unsigned)((W + 255) / 256);
    if (storage == FLB_F16_DEV)
        window_kernel<__half><<<grid, 256, 0, s>>>(g, q, (const __half *)f, psi, x0, y0, z0, wx, wy, wz, out);
    else
        window_kernel<float><<<grid, 256, 0, s>>>(g, q, (const float *)f, psi, x0, y0, z0, wx, wy, wz, out);
    return cudaGetLastError();
}

}  // namespace flb
