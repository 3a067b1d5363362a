// vgrad_f64.cu -- adjoint of the region-I term: gradient of E_I = sum gamma_{mu nu} V_{mu nu}
// (Eq. 9) with respect to the QM centres, the MM image positions and the MM charges, FP64.
//
// Per primitive pair the density is folded into Hermite coefficients once,
//   D0_tuv = sum_ab g_ab E^x_t E^y_u E^z_v,   Dx_tuv = sum_ab g_ab E'^x_t E^y_u E^z_v, ...
// with g_ab the density element (plus its mirror) times the pair prefactor and
//   E'^{ij}_t = dE^{ij}_t / dX_AB = 2a E^{i+1,j}_t - i E^{i-1,j}_t - (a/p) E^{ij}_{t-1}.
// Moving A shifts P by a/p, so with e_a = sum D0_tuv R_{tuv + 1_a} and d_a = sum Da_tuv R_tuv
// (recomputed for every charge, never stored):
//   dI/dA_a = d_a + (a/p) e_a,   dI/dB_a = -d_a + (b/p) e_a,   dI/dC_a = -e_a,
// and E contains -q_C I.  The d_a enter only through sum_C q_C d_a(C) = sum Da_tuv W_tuv with
// W_tuv = sum_C q_C R_tuv, so the sweep accumulates the charge sums and Da is formed and contracted
// once per pair after it (contract_dA).
//
// Bound: the FP64 pipe, 2 lanes per clock and SM, 85-91% busy, with 7-8% of the issue slots used: the
// kernel's time is its count of FP64 instructions.  So the tensors R are never formed: D0 and W are
// kept as solid-harmonic components (harm.cuh), per charge one recursion of (L+1)^2 harmonics, one
// multiply-add per harmonic for the value, the charge sum and each gradient component (these with
// the coefficients N of the differentiated harmonics, one order lower).  FP64 instructions per
// (warp, charge) on a 60-atom active site, setup included: (s,s) 30, (p,p) 77, (d,s) 87, (d,p) 141,
// (d,d) 262.  Coefficients and sums of the high classes spill to local memory ((f,f): 4.7 KB
// stores), which the idle load pipe carries.  Adjoint sweep against the Hermite recursion with its
// contractions: active site 78.3 -> 60.9 ms, a 150-atom site with f shells 412 -> 242 ms, a QM
// water 1.35 -> 0.82 ms (untuned handles).
//
// Per-pair sums over charges stay in registers; per-charge sums over the
// 32 primitive pairs of a tile use a warp butterfly and go to shared-memory accumulators that
// are flushed to global memory once per block.
#include <algorithm>

#include "harm.cuh"
#include "pp_tile.cuh"

namespace qmmm {

template <int LA, int LB>
struct VgradF64 {
    static cudaError_t run(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                           int ch_end, const double *boys, const double *dm, double *gqm, double *gchg, int *err,
                           int nblk, int threads, int nslice,
                           cudaStream_t st);
};

#ifdef QMMM_SPLIT_CLASS  // one angular class per compilation

template <int LA, int LB, int NT>
__global__ void __launch_bounds__(NT, 1)
k_vgrad_f64(BasisDev bd, RegionDev rg, int pp_begin, int pp_end, int ch_begin, int ch_end,
            const double *__restrict__ boys, const double *__restrict__ dm, double *__restrict__ gqm,
            double *__restrict__ gchg, int *err)
{
    constexpr int L = LA + LB, NH = nherm(L), NG = nhgrad(L) + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    {
        // this block row's slice of the charge chunk (gridDim.y > 1 spreads small systems over more SMs)
        const int per = (ch_end - ch_begin + (int)gridDim.y - 1) / (int)gridDim.y;
        ch_begin += (int)blockIdx.y * per;
        ch_end = min(ch_end, ch_begin + per);
    }
    if (ch_begin >= ch_end) return;
    const int nch = ch_end - ch_begin;
    double4_32a *chg = reinterpret_cast<double4_32a *>(smem_raw);
    double *acc = reinterpret_cast<double *>(smem_raw + (size_t)nch * sizeof(double4_32a));
    for (int k = threadIdx.x; k < 4 * nch; k += blockDim.x) acc[k] = 0.0;
    if (!stage_to_smem(chg, rg.chg + ch_begin, (unsigned)(nch * sizeof(double4_32a)), &bar, err)) return;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int ntile = (pp_end - pp_begin + 31) >> 5;
    for (int tile = blockIdx.x * nwarp + warp; tile < ntile; tile += gridDim.x * nwarp) {
        const PPLane pl = load_pp(bd, pp_begin + tile * 32 + lane, pp_end);
        const double aop = pl.a * pl.ip, bop = pl.b * pl.ip;
        // the density-folded Hermite coefficients as harmonic ones, their gradients, and the charge
        // sums S (harm.cuh); unit: the unit of the harmonic factors
        const double unit = HALF_SQRT_PI * sqrt(pl.ip);
        double M[NH], Nx[NG], Ny[NG], Nz[NG], S[NH];
        {
            double D0[NH];
            fold_density<LA, LB>(pl, bd, dm, D0);
#pragma unroll
            for (int k = 0; k < NH; ++k) D0[k] *= unit;
            harm_fold<L>(D0, M);
            harm_grad<L>(M, Nx, Ny, Nz);
        }
#pragma unroll
        for (int k = 0; k < NH; ++k) S[k] = 0.0;

        double sex = 0, sey = 0, sez = 0;
        for (int c = 0; c < rg.ncls; ++c) {
            const int lo = max(__ldg(rg.cls_off + c), ch_begin) - ch_begin;
            const int hi = min(__ldg(rg.cls_off + c + 1), ch_end) - ch_begin;
            if (lo >= hi) continue;
            const double kap = __ldg(rg.cls_kappa + c);
            const double rho = kap > 0.0 ? pl.p * (kap / (pl.p + kap)) : pl.p;
            const double c0 = sqrt(rho) / HALF_SQRT_PI;
            const double rfar = harm_tmax(L + 1) / rho;
            for (int j = lo; j < hi; ++j) {
                const double4_32a ch = chg[j];
                const double X = pl.P[0] - ch.x, Y = pl.P[1] - ch.y, Z = pl.P[2] - ch.z;
                const double r2 = X * X + Y * Y + Z * Z;
                const bool far = harm_far(r2, rfar);
                double e0, ex, ey, ez;
                const double q = ch.w;
                if (__all_sync(FULL, far)) {
                    double F[L + 1];
                    const double y = harm_rsqrt(r2), y2 = y * y;
                    F[0] = y;
#pragma unroll
                    for (int l = 1; l <= L; ++l) F[l] = F[l - 1] * y2;
                    harm_eval<L, false>(M, Nx, Ny, Nz, F, 0.0, 0.0, y2, X, Y, Z, r2, q, S, e0, ex, ey, ez);
                } else {
                    double F[L + 2], E0;
                    boys_hat<L + 1>(far, r2, rho, c0, F, E0, boys);
                    harm_eval<L, true>(M, Nx, Ny, Nz, F, E0, rho, 0.0, X, Y, Z, r2, q, S, e0, ex, ey, ez);
                }
                sex += q * ex; sey += q * ey; sez += q * ez;
                // per-charge sums over the 32 primitive pairs of (e_x, e_y, e_z, e_0), whose
                // factors (q, q, q, -1) in (dE/dC, dE/dq) are applied when the block's sums leave:
                // halve the four values twice (each lane keeps one component summed over 4
                // lanes), then a 3-step butterfly; lane 8c ends with component c.  6 FP64
                // additions instead of 4 full warp sums (20).
                {
                    const bool up = lane & 16;
                    double k0 = up ? ez : ex, k1 = up ? e0 : ey;
                    const double s0 = up ? ex : ez, s1 = up ? ey : e0;
                    k0 += __shfl_xor_sync(FULL, s0, 16);
                    k1 += __shfl_xor_sync(FULL, s1, 16);
                    const bool up8 = lane & 8;
                    double k = up8 ? k1 : k0;
                    k += __shfl_xor_sync(FULL, up8 ? k0 : k1, 8);
                    k += __shfl_xor_sync(FULL, k, 4);
                    k += __shfl_xor_sync(FULL, k, 2);
                    k += __shfl_xor_sync(FULL, k, 1);
                    if ((lane & 7) == 0) atomicAdd(acc + 4 * j + (((lane >> 4) << 1) | ((lane >> 3) & 1)), k);
                }
            }
        }
        double sd[3];
        {
            double W[NH];
            harm_unfold<L>(S, W);
#pragma unroll
            for (int k = 0; k < NH; ++k) W[k] *= unit;
            contract_dA<LA, LB>(pl, bd, dm, W, sd);
        }
        // dE/dA = -(sd + a/p se), dE/dB = sd - b/p se
        double g[6] = {-(sd[0] + aop * sex), -(sd[1] + aop * sey), -(sd[2] + aop * sez),
                       sd[0] - bop * sex, sd[1] - bop * sey, sd[2] - bop * sez};
        bool take[5], head;
        seg_setup(pl.active ? pl.s : -1 - lane, lane, take, head);
#pragma unroll
        for (int k = 0; k < 6; ++k) g[k] = seg_reduce(g[k], take);
        if (head && pl.active) {
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                atomicAdd(gqm + 3 * pl.atomA + x, g[x]);
                atomicAdd(gqm + 3 * pl.atomB + x, g[3 + x]);
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 4 * nch; k += blockDim.x) {
        const double v = (k & 3) < 3 ? chg[k >> 2].w * acc[k] : -acc[k];
        if (v != 0.0) atomicAdd(gchg + 4 * (size_t)ch_begin + k, v);
    }
}

template <int LA, int LB, int NT>
static cudaError_t launch_nt(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                             int ch_end, const double *boys, const double *dm, double *gqm, double *gchg, int *err,
                             int nblk, int threads, int nslice, cudaStream_t st)
{
    const int nper = (ch_end - ch_begin + nslice - 1) / nslice;  // charges per slice
    const size_t smem = std::max((size_t)nper * (sizeof(double4_32a) + 4 * sizeof(double)), SWEEP_SMEM_MIN);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_vgrad_f64<LA, LB, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(CHUNK_GRAD * (sizeof(double4_32a) + 4 * sizeof(double))));
        if (e != cudaSuccess) return e;
        attr = true;
    }
        k_vgrad_f64<LA, LB, NT><<<dim3(nblk, nslice), threads, smem, st>>>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys,
                                                                  dm, gqm, gchg, err);
    return cudaGetLastError();
}

template <int LA, int LB>
cudaError_t VgradF64<LA, LB>::run(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                                  int ch_end, const double *boys, const double *dm, double *gqm, double *gchg,
                                  int *err,
                                  int nblk, int threads, int nslice,
                                  cudaStream_t st)
{
    constexpr int W = sweep_wide_threads(SW_VGRAD_F64, class_of(LA, LB));
    if constexpr (W > 0)
        if (threads == W)
            return launch_nt<LA, LB, W>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys, dm, gqm, gchg, err, nblk, threads,
                                        nslice, st);
    return launch_nt<LA, LB, 256>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys, dm, gqm, gchg, err, nblk, threads,
                                  nslice, st);
}

template struct VgradF64<la_of_class(QMMM_SPLIT_CLASS), lb_of_class(QMMM_SPLIT_CLASS)>;

#else  // the dispatcher

cudaError_t launch_vgrad_f64(const BasisDev &b, const RegionDev &r, int cls, int pp_begin, int pp_end,
                             int ch_begin, int ch_end, const double *boys, const double *dm, double *gqm,
                             double *gchg, int *err, int nblk, int threads, int nslice, cudaStream_t st)
{
    if (pp_end <= pp_begin || ch_end <= ch_begin) return cudaSuccess;
    return dispatch_class<VgradF64>(cls, b, r, pp_begin, pp_end, ch_begin, ch_end, boys, dm, gqm, gchg, err, nblk, threads, nslice, st);
}

#endif

}  // namespace qmmm
