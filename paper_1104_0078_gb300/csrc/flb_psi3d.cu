// flb_psi3d.cu -- one Runge-Kutta stage of the order-parameter equation (Sec. V.B
// of arXiv:1104.0078, finite volume) on a 3D box, fused in one pass with z-marching
// (2.5D) blocking: large boxes, and the batched mode.  The finite-difference and
// naive schemes, other Laplacians than SO and small boxes run flb_psi3c.cu.
//
// A block owns a TX x TY column tile and a chunk of planes.  Rolling rings of planes
// in shared memory hold psi (tile + 3 ghost cells), the chemical potential
// mu = A psi + B psi^3 - K lap_SO psi (tile + 2), the node flux J = M grad mu - u psi
// and the node noise xi (tile + 1); the stage output at plane z is formed from the three
// flux planes z-1, z, z+1.  Nothing but psi, u and the Heun accumulator touches
// HBM.  The psi and velocity planes arrive by TMA (cp.async.bulk.tensor) two
// planes ahead of use.
//
//   grad mu = (1/c_s^2) sum_i w_i c_i mu(r + c_i)
//   D(r)    = (1/c_s^2) sum_i w_i c_i . J(r + c_i)
//             (the link average (J(r) + J(r+c_i))/2 of Eq. fvflux with
//              the 2/c_s^2 divergence; sum_i w_i c_i = 0 removes J(r)),
//   xi_a ~ N(0, 2 kT M) per node and component.
// Stage 1 writes psi* = psi + D + eta and (Heun) E = psi + D/2 + eta; stage 2
// writes psi^{n+1} = E + D(psi*)/2 (the noise is held fixed over the step).
#include <cudaTypedefs.h>

#include <type_traits>

#include "flb_psi3d.cuh"

namespace flb {

struct TmaArgs {
    Psi3Args a;
    int *status;
};

// MU_IN: stage 1 reads mu of its input from mu_map instead of forming it; Q15:
// the FV operators of D3Q15
// 256 threads, each on point pairs (y, y + H/2) of every region in packed FP32 (F2)
using StageV = F2;
template <int STAGE, int NOISE, bool RK, bool MU_IN, bool Q15 = false>
__global__ void __launch_bounds__(block_threads<StageV, MU_IN>(), 2) psi3_fv_tma_kernel(const __grid_constant__ CUtensorMap psi_map,
                                                                   const __grid_constant__ CUtensorMap u_map,
                                                                   const __grid_constant__ CUtensorMap mu_map,
                                                                   const TmaArgs ta)
{
    extern __shared__ __align__(1024) float tsmem[];
    pdl_trigger();
    pdl_wait();
    // the fields were stored by threads of the launches in front and come by TMA
    if (threadIdx.x == 0) asm volatile("fence.proxy.async.global;" ::: "memory");
    psi3_fv_tma_block<STAGE, NOISE, false, false, RK, MU_IN, Q15, StageV>(&psi_map, &u_map, ta.a, ta.status, blockIdx.x,
                                                                     blockIdx.y, blockIdx.z, tsmem, &mu_map);
}

// batched: block b of the launch works on L.psi[b]; MU_IN: stage 1 reads mu of
// psi^n from the replica's mu field (every replica's step formed it)
template <int STAGE, int NOISE, bool MU_IN = false, bool Q15 = false>
__global__ void __launch_bounds__(block_threads<StageV, MU_IN>(), 2) psi3_fv_tma_batch_kernel(const BatchLists L)
{
    extern __shared__ __align__(1024) float tsmem[];
    __shared__ Psi3Args sa;
    const BatchBlock b = L.psi[blockIdx.x];
    const BatchRep &r = L.reps[b.rep];
    const long long ds = *L.dstep;
    if (threadIdx.x == 0) psi_batch_args(r, ds, STAGE, sa);
    __syncthreads();
    const CUtensorMap *pm = STAGE == 1 ? &r.map_psi[(int)(ds & 1)] : &r.map_psis;
    psi3_fv_tma_block<STAGE, NOISE, false, true, false, MU_IN, Q15, StageV>(pm, &r.map_u, sa, L.status, b.bx, b.by, b.bz,
                                                                       tsmem, &r.map_mu);
}

__global__ void advance_kernel(long long *dstep) { *dstep += 1; }

cudaError_t launch_lb3_batch(const BatchLists &L, int storage, bool ghost, bool force, cudaStream_t st);
cudaError_t launch_lb15_batch(const BatchLists &L, int storage, bool ghost, bool force, cudaStream_t st);

template <bool Q15>
static cudaError_t batch_psi(const BatchLists &L, bool heun, int noise, bool mu_in, cudaStream_t st)
{
    const size_t sm = sizeof(float) * (size_t)fv_smem_floats<StageV>();
    const size_t smm = sizeof(float) * (size_t)fv_mu_smem_floats<StageV>();
    const size_t nb = sizeof(float) * FV_NOISE_FLOATS;
    auto go = [&](auto kernel, size_t bytes, int nt) {
        cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (r != cudaSuccess) return r;
        kernel<<<L.npsi, nt, bytes, st>>>(L);
        return cudaGetLastError();
    };
    constexpr int n1 = block_threads<StageV, true>(), nn = block_threads<StageV, false>();
    cudaError_t e = mu_in ? (noise == 2 ? go(psi3_fv_tma_batch_kernel<1, 2, true, Q15>, smm + nb, n1)
                                 : noise ? go(psi3_fv_tma_batch_kernel<1, 1, true, Q15>, smm + nb, n1)
                                         : go(psi3_fv_tma_batch_kernel<1, 0, true, Q15>, smm, n1))
                          : (noise == 2 ? go(psi3_fv_tma_batch_kernel<1, 2, false, Q15>, sm + nb, nn)
                                 : noise ? go(psi3_fv_tma_batch_kernel<1, 1, false, Q15>, sm + nb, nn)
                                         : go(psi3_fv_tma_batch_kernel<1, 0, false, Q15>, sm, nn));
    if (e != cudaSuccess || !heun) return e;
    return go(psi3_fv_tma_batch_kernel<2, 0, false, Q15>, sm, nn);
}

cudaError_t launch_batch_psi(const BatchLists &L, bool heun, int noise, bool mu_in, bool q15, cudaStream_t st)
{
    return q15 ? batch_psi<true>(L, heun, noise, mu_in, st) : batch_psi<false>(L, heun, noise, mu_in, st);
}

cudaError_t launch_batch_step(const BatchLists &L, int storage, bool ghost, bool force, int scheme_fv, bool heun,
                              int noise, bool mu_in, bool q15, cudaStream_t st)
{
    if (!scheme_fv) return cudaErrorNotSupported;
    cudaError_t e = q15 ? launch_lb15_batch(L, storage, ghost, force, st)
                        : launch_lb3_batch(L, storage, ghost, force, st);
    if (e != cudaSuccess) return e;
    return launch_batch_psi(L, heun, noise, mu_in, q15, st);
}

cudaError_t launch_batch_advance(const BatchLists &L, cudaStream_t st)
{
    advance_kernel<<<1, 1, 0, st>>>(const_cast<long long *>(L.dstep));
    return cudaGetLastError();
}

cudaError_t encode_tensor_map_f32(CUtensorMap *map, const void *base, int rank, const uint64_t *dims,
                                  const uint64_t *strides_bytes, const uint32_t *box)
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !p)
            return cudaErrorNotSupported;
        fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    cuuint64_t d[5], str[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        bx[i] = box[i];
        es[i] = 1;
        if (i > 0) str[i - 1] = strides_bytes[i - 1];
    }
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<void *>(base), d, str, bx,
                          es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

static cudaError_t launch_fv_tma(const Psi3Args &a, int q, int stage, int noise, const float *mu_in, int *status,
                                 cudaStream_t st)
{
    const Geom &g = a.g;
    CUtensorMap pm, um;
    const uint64_t pd[3] = {(uint64_t)g.px, (uint64_t)g.py, (uint64_t)g.pz};
    const uint64_t ps[2] = {(uint64_t)g.px * 4, (uint64_t)g.px * g.py * 4};
    const uint32_t pb[3] = {(uint32_t)TB_X, (uint32_t)H3Y, 1};
    cudaError_t e = encode_tensor_map_f32(&pm, a.psi, 3, pd, ps, pb);
    if (e != cudaSuccess) return e;
    const uint64_t ud[4] = {(uint64_t)g.px, (uint64_t)g.py, (uint64_t)g.pz, 3};
    const uint64_t us[3] = {(uint64_t)g.px * 4, (uint64_t)g.px * g.py * 4, (uint64_t)g.pn * 4};
    const uint32_t ub[4] = {(uint32_t)TB_X, (uint32_t)H1Y, 1, 3};
    e = encode_tensor_map_f32(&um, a.u, 4, ud, us, ub);
    if (e != cudaSuccess) return e;
    CUtensorMap mm = pm;  // unused unless stage 1 reads mu
    const bool mu = stage == 1 && mu_in != nullptr;
    if (mu) {
        const uint32_t mb[3] = {(uint32_t)TB_X, (uint32_t)H2Y, 1};
        e = encode_tensor_map_f32(&mm, mu_in, 3, pd, ps, mb);
        if (e != cudaSuccess) return e;
    }
    TmaArgs ta;
    ta.a = a;
    ta.status = status;
    const dim3 grid((g.nx + PS_TX - 1) / PS_TX, (g.ny + PS_TY - 1) / PS_TY, (g.nz + a.zc - 1) / a.zc);
    const size_t sm = sizeof(float) * (size_t)fv_smem_floats<StageV>();
    auto go = [&](auto kernel, size_t bytes) {
        cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (r != cudaSuccess) return r;
        return launch_pdl(kernel, grid, mu ? block_threads<StageV, true>() : block_threads<StageV, false>(), bytes, st, PDL_BLOCKS, pm, um, mm, ta);
    };
    const size_t smn = sm + sizeof(float) * FV_NOISE_FLOATS;
    const size_t smm = sizeof(float) * (size_t)fv_mu_smem_floats<StageV>(), smmn = smm + sizeof(float) * FV_NOISE_FLOATS;
    // one kernel per stage, RK4 or not (its branches cost registers), mu given or not,
    // noise (0, 1, 2) and lattice
    auto stage1 = [&](auto rk, auto mi, auto q15) {
        constexpr bool RK = decltype(rk)::value, MU = decltype(mi)::value, Q15 = decltype(q15)::value;
        const size_t bytes = MU ? smm : sm, bytes_n = MU ? smmn : smn;
        return noise == 2 ? go(psi3_fv_tma_kernel<1, 2, RK, MU, Q15>, bytes_n)
               : noise    ? go(psi3_fv_tma_kernel<1, 1, RK, MU, Q15>, bytes_n)
                          : go(psi3_fv_tma_kernel<1, 0, RK, MU, Q15>, bytes);
    };
    auto lattice = [&](auto q15) {
        constexpr bool Q15 = decltype(q15)::value;
        using Yes = std::true_type;
        using No = std::false_type;
        if (stage == 2) return a.rk4 ? go(psi3_fv_tma_kernel<2, 0, true, false, Q15>, sm)
                                     : go(psi3_fv_tma_kernel<2, 0, false, false, Q15>, sm);
        if (a.rk4) return mu ? stage1(Yes(), Yes(), q15) : stage1(Yes(), No(), q15);
        return mu ? stage1(No(), Yes(), q15) : stage1(No(), No(), q15);
    };
    return q == 15 ? lattice(std::true_type()) : lattice(std::false_type());
}

cudaError_t launch_psi3(const Geom &g, int scheme, int q, int stage, int noise, const float *psi, const float *u,
                        float *out, float *E, float A, float B, float K, float M, float kT, int advect, int heun,
                        const PhiloxKey &key, int64_t step, int zc, int rk4, const float *base, float *Dn,
                        const float *mu_in, int *status, cudaStream_t st, const LapW *lw)
{
    // the marching stage is the FV one with SO's Laplacian
    if (zc != 0 && (zc < PS_ZC_MIN || scheme != FLB_FV || lw)) return cudaErrorInvalidValue;
    Psi3Args a;
    a.lap_w = lw ? 1 : 0;
    a.lw = lw ? *lw : LapW{0.f, 0.f, 0.f, 0.f};
    a.rk4 = rk4;
    a.base = base;
    a.Dn = Dn;
    a.g = g;
    a.psi = psi;
    a.u = u;
    a.out = out;
    a.E = E;
    a.A = A;
    a.B = B;
    a.K = K;
    a.M = M;
    a.kT = kT;
    a.advect = advect;
    a.heun = heun;
    a.zc = zc;
    a.key = key;
    a.step = step;
    return zc == 0 ? launch_psi3_cube(a, scheme, q, stage == 1, noise, mu_in, st)
                   : launch_fv_tma(a, q, stage, noise, mu_in, status, st);
}

}  // namespace flb
