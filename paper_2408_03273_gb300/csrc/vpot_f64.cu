// vpot_f64.cu -- region-I one-electron matrix of Eq. 9 in FP64 (McMurchie-Davidson).
//
//   V_{ab} = - sum_{C in I} q_C (2 pi/p) sqrt(kappa_C/(p+kappa_C)) c_a c_b K_AB
//            sum_tuv E^x_t E^y_u E^z_v R_tuv(rho_C, P - C)
//
// A warp owns 32 primitive pairs of one angular class; the block stages a chunk of region-I
// charges (x, y, z, q) into shared memory with one TMA bulk copy, every lane sweeps all of them
// (shared-memory broadcast) and accumulates W_tuv = sum_C q_C s_C R_tuv in registers, as
// solid-harmonic components (harm.cuh).  The bound is the FP64 pipe (90% busy, 8% of the issue
// slots used), so the kernel's time is its count of FP64 instructions: per (warp, charge) 13, 21,
// 37, 61, 94, 135, 182 for L = 0..6, setup included (150-atom site with f shells; a 60-atom site within
// 1.5%).  V sweep against the Hermite recursion: active site 33.5 -> 24.4 ms, a 150-atom site with f
// shells 147 -> 104 ms, a QM water 0.43 -> 0.33 ms (untuned handles).  Charges are grouped by Gaussian width so that rho is formed once per
// (primitive pair, width class).
//
// The sweep leaves the sums of every pair and charge slice; k_pair_V adds the slices in a fixed order
// and contracts them with E once per primitive pair, in blocks of 32 pairs x the components of shell
// A (in the sweep this was one lane's chain, some 1 500 FP64 instructions for (d,d) and 6 000 for (f,f),
// once per slice, into one partial V per slice: sweep of 17 atoms with f shells 1.18 -> 0.70 ms, of a QM
// water 0.205 -> 0.138 ms, of the 60-atom site 19.8 -> 19.7 ms).  Primitive pairs of a
// shell pair are summed by a segmented warp-shuffle reduction and the head lane adds the block into
// the lower triangle of V (mirrored at the end).  A shell pair spans at most two tiles when it has at most
// 32 primitive pairs, so at most two additions per chunk of charges reach any element: with one chunk the
// result does not depend on scheduling.
#include <algorithm>

#include "harm.cuh"
#include "pair_block.cuh"
#include "pp_tile.cuh"

namespace qmmm {

template <int LA, int LB>
struct VpotF64 {
    static cudaError_t run(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                           int ch_end, const double *boys, double *V, int *err, int nblk, int threads, int nslice,
                           double *sums, cudaStream_t st);
};

#ifdef QMMM_SPLIT_CLASS  // one angular class per compilation

template <int LA, int LB, int NT>
__global__ void __launch_bounds__(NT, 1)
k_vpot_f64(BasisDev bd, RegionDev rg, int pp_begin, int pp_end, int ch_begin, int ch_end,
           const double *__restrict__ boys, double *__restrict__ sums, int *err)
{
    constexpr int L = LA + LB, NH = nherm(L);
    const size_t np = pp_end - pp_begin;
    sums += (size_t)blockIdx.y * NH * np;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    double4_32a *chg = reinterpret_cast<double4_32a *>(smem_raw);
    {
        // this block row's slice of the charge chunk (gridDim.y > 1 spreads small systems over more SMs)
        const int per = (ch_end - ch_begin + (int)gridDim.y - 1) / (int)gridDim.y;
        ch_begin += (int)blockIdx.y * per;
        ch_end = min(ch_end, ch_begin + per);
    }
    const int nch = max(ch_end - ch_begin, 0);  // (an empty last slice leaves zero sums)
    if (nch > 0 && !stage_to_smem(chg, rg.chg + ch_begin, (unsigned)(nch * sizeof(double4_32a)), &bar, err)) return;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int ntile = (pp_end - pp_begin + 31) >> 5;
    for (int tile = blockIdx.x * nwarp + warp; tile < ntile; tile += gridDim.x * nwarp) {
        const PPLane pl = load_pp(bd, pp_begin + tile * 32 + lane, pp_end);
        double S[NH];  // harmonic sums (harm.cuh)
#pragma unroll
        for (int k = 0; k < NH; ++k) S[k] = 0.0;

        for (int c = 0; c < rg.ncls; ++c) {
            const int lo = max(__ldg(rg.cls_off + c), ch_begin) - ch_begin;
            const int hi = min(__ldg(rg.cls_off + c + 1), ch_end) - ch_begin;
            if (lo >= hi) continue;
            const double kap = __ldg(rg.cls_kappa + c);
            const double rho = kap > 0.0 ? pl.p * (kap / (pl.p + kap)) : pl.p;
            const double c0 = sqrt(rho) / HALF_SQRT_PI;
            const double rfar = harm_tmax(L) / rho;
            for (int j = lo; j < hi; ++j) {
                const double4_32a ch = chg[j];
                const double X = pl.P[0] - ch.x, Y = pl.P[1] - ch.y, Z = pl.P[2] - ch.z;
                const double r2 = X * X + Y * Y + Z * Z;
                const bool far = harm_far(r2, rfar);
                if (__all_sync(FULL, far)) {
                    harm_add_far<L>(S, ch.w, X, Y, Z, r2);
                } else {
                    double F[L + 1], E0;
                    boys_hat<L>(far, r2, rho, c0, F, E0, boys);
                    harm_add<L, true>(S, F, E0, rho, ch.w, X, Y, Z, r2);
                }
            }
        }
        if (pl.active)
#pragma unroll
            for (int k = 0; k < NH; ++k) sums[k * np + tile * 32 + lane] = S[k];
    }
}

template <int LA, int LB>
__global__ void __launch_bounds__(32 * ncart(LA))
k_pair_V(BasisDev bd, int pp_begin, int pp_end, const double *__restrict__ sums, int nslice, double *__restrict__ V)
{
    using Sh = PairShape<LA, LB>;
    constexpr int L = Sh::L, NH = Sh::NH, NA = Sh::NA, NB = Sh::NB, T = Sh::T;
    extern __shared__ double sm[][32];
    double(*S)[32] = sm + Sh::NF, (*W)[32] = S + NH;
    const int lane = threadIdx.x, ia = threadIdx.y, i = pp_begin + blockIdx.x * 32 + lane;
    const size_t np = pp_end - pp_begin, ip = min(blockIdx.x * 32 + lane, (int)np - 1);
    const PPLane pl = load_pp(bd, i, pp_end);
    constexpr int TD = (LA + 1) * (LB + 1) * (T + 1);
    for (int d = ia; d < 3; d += NA) {
        const double xa = d == 0 ? pl.P[0] - pl.A[0] : d == 1 ? pl.P[1] - pl.A[1] : pl.P[2] - pl.A[2];
        const double xb = d == 0 ? pl.P[0] - pl.B[0] : d == 1 ? pl.P[1] - pl.B[1] : pl.P[2] - pl.B[2];
        hermite_table<LA, LB, T>(sm + d * TD, lane, xa, xb, 0.5 * pl.ip);
    }
    for (int k = ia; k < NH; k += NA) {
        double s = 0.0;
        for (int sl = 0; sl < nslice; ++sl) s += sums[((size_t)sl * NH + k) * np + ip];
        S[k][lane] = s;
        W[k][lane] = 0.0;
    }
    __syncthreads();
    // harmonic sums -> Hermite sums, a warp per Hermite index at a time
    for (int e = 0; e < HT.tend[L]; ++e) {
        const HarmEntry &t = HT.t[e];
        if (t.herm % NA == ia) W[t.herm][lane] += t.c * S[harm_off(L, t.k) + t.lm][lane];
    }
    __syncthreads();
    int a3[3] = {0, 0, 0};
    cart_of(LA, ia, a3);
    const double coef = -TWO_PI * pl.ip * pl.cab * HALF_SQRT_PI * sqrt(pl.ip);
    bool take[5], head;
    seg_setup(pl.active ? pl.s : -1 - lane, lane, take, head);
    const bool self = pl.sp.shA == pl.sp.shB;  // a shell with itself: one triangle
#pragma unroll 1
    for (int ib = 0; ib < NB; ++ib) {
        int b3[3] = {0, 0, 0};
        cart_of(LB, ib, b3);
        // E_t vanishes beyond t = i + j: bounds uniform over the warp
        const int lx = a3[0] + b3[0], ly = a3[1] + b3[1], lz = a3[2] + b3[2];
        const double(*row[3])[32];
#pragma unroll
        for (int d = 0; d < 3; ++d) row[d] = sm + d * TD + (a3[d] * (LB + 1) + b3[d]) * (T + 1);
        double Ez[L + 1], v = 0.0;
#pragma unroll
        for (int t = 0; t <= L; ++t) Ez[t] = t <= lz ? row[2][t][lane] : 0.0;
#pragma unroll 1
        for (int t = 0; t <= lx; ++t) {
            double h = 0.0;
#pragma unroll 1
            for (int u = 0; u <= ly; ++u) {
                double w = 0.0;
#pragma unroll
                for (int z = 0; z <= L; ++z)
                    if (z <= lz) w = fma(Ez[z], W[hidx(t, u, z)][lane], w);
                h = fma(row[1][u][lane], w, h);
            }
            v = fma(row[0][t][lane], h, v);
        }
        v = seg_reduce(coef * v, take);
        if (head && pl.active && (!self || ia <= ib))
            atomicAdd(V + lower_index(pl.sp.aoA + ia, pl.sp.aoB + ib, bd.nao), v);
    }
}

template <int LA, int LB, int NT>
static cudaError_t launch_nt(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                             int ch_end, const double *boys, double *sums, int *err, int nblk, int threads, int nslice,
                             cudaStream_t st)
{
    const int per = (ch_end - ch_begin + nslice - 1) / nslice;
    const size_t smem = std::max((size_t)per * sizeof(double4_32a), SWEEP_SMEM_MIN);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_vpot_f64<LA, LB, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(CHUNK_F64 * sizeof(double4_32a)));
        if (e != cudaSuccess) return e;
        attr = true;
    }
    k_vpot_f64<LA, LB, NT><<<dim3(nblk, nslice), threads, smem, st>>>(bd, rg, pp_begin, pp_end, ch_begin, ch_end,
                                                                      boys, sums, err);
    return cudaGetLastError();
}

template <int LA, int LB>
cudaError_t VpotF64<LA, LB>::run(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                                 int ch_end, const double *boys, double *V, int *err, int nblk, int threads,
                                 int nslice, double *sums, cudaStream_t st)
{
    using Sh = PairShape<LA, LB>;
    constexpr size_t smem = Sh::VS * 32 * sizeof(double);
    static bool attr = false;
    cudaError_t e;
    if (!attr) {
        if ((e = cudaFuncSetAttribute(k_pair_V<LA, LB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
            cudaSuccess)
            return e;
        attr = true;
    }
    constexpr int W = sweep_wide_threads(SW_VPOT_F64, class_of(LA, LB));
    bool wide = false;
    if constexpr (W > 0)
        if (threads == W) {
            wide = true;
            e = launch_nt<LA, LB, W>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys, sums, err, nblk, threads, nslice,
                                     st);
        }
    if (!wide)
        e = launch_nt<LA, LB, 256>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys, sums, err, nblk, threads, nslice,
                                   st);
    if (e != cudaSuccess) return e;
    k_pair_V<LA, LB><<<(pp_end - pp_begin + 31) / 32, dim3(32, Sh::NA), smem, st>>>(bd, pp_begin, pp_end, sums, nslice,
                                                                                    V);
    return cudaGetLastError();
}

template struct VpotF64<la_of_class(QMMM_SPLIT_CLASS), lb_of_class(QMMM_SPLIT_CLASS)>;

#else  // the dispatcher

cudaError_t launch_vpot_f64(const BasisDev &b, const RegionDev &r, int cls, int pp_begin, int pp_end,
                            int ch_begin, int ch_end, const double *boys, double *V, int *err, int nblk,
                            int threads, int nslice, double *sums, cudaStream_t st)
{
    if (pp_end <= pp_begin || ch_end <= ch_begin) return cudaSuccess;
    return dispatch_class<VpotF64>(cls, b, r, pp_begin, pp_end, ch_begin, ch_end, boys, V, err, nblk, threads, nslice,
                                   sums, st);
}

#endif

}  // namespace qmmm
