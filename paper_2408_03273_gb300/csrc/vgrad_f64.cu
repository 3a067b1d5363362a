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
// W_tuv = sum_C q_C R_tuv, so the sweep accumulates the charge sums and Da is contracted with them once
// per pair after it.  Three kernels per class:
//   k_pair_fold      D0 of every primitive pair, as solid-harmonic coefficients M (block: 32 pairs x the
//                    Cartesian components of shell A);
//   k_vgrad_f64      the sweep: M in, charge gradients and the pairs' charge sums out;
//   k_pair_contract  Da . W and the pair gradients onto the atoms (blocks as k_pair_fold).
// With the fold and the contraction in the sweep, one lane did them all for its pair, once per charge
// slice: some 7 000 FP64 instructions for a (d,d) pair and 30 000 for (f,f), a chain that set the time
// of small systems.  Sweep of a QM water 0.53 -> 0.34 ms, of 17 atoms with f shells 4.31 -> 2.05 ms; of the
// 60- and the 150-atom site, which hide the chain, unchanged (45 and 194 ms).
//
// Bound: the FP64 pipe, 2 lanes per clock and SM, 88-90% busy on the SMs that hold a block and 85-86% over
// a whole sweep, with 7-8% of the issue slots used: the kernel's time is its count of FP64
// instructions.  So the tensors R are never formed: D0 and W are kept as solid-harmonic components
// (harm.cuh), per charge one recursion of (L+1)^2 harmonics, one multiply-add per harmonic for the
// value, the charge sum and each gradient component (these with the coefficients N of the
// differentiated harmonics, one order lower).  FP64 instructions per (warp, charge) for L = 0..6, setup
// included: 31, 46, 83, 138, 214, 310, 423 (150-atom site with f shells; a 60-atom site within 1.5%).
// Coefficients and sums of the high classes spill to local memory ((f,f): 2.9 KB stores), which the
// idle load pipe carries.  Adjoint sweep against the Hermite recursion with its
// contractions: active site 78.3 -> 60.9 ms, a 150-atom site with f shells 412 -> 242 ms, a QM
// water 1.35 -> 0.82 ms (untuned handles).
//
// Per-pair sums over charges stay in registers; per-charge sums over the
// 32 primitive pairs of a tile use a warp butterfly and go to shared-memory accumulators that
// are flushed to global memory once per block.
#include <algorithm>

#include "harm.cuh"
#include "pair_block.cuh"
#include "pp_tile.cuh"

namespace qmmm {

template <int LA, int LB>
struct VgradF64 {
    static cudaError_t run(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                           int ch_end, const double *boys, const double *dm, double *gqm, double *gchg, int *err,
                           int nblk, int threads, int nslice, double *pairs, cudaStream_t st);
};

#ifdef QMMM_SPLIT_CLASS  // one angular class per compilation

// ---------------------------------------------------------------------------------------------
// Per-pair algebra: blocks as in pair_block.cuh
// ---------------------------------------------------------------------------------------------
// M[k npair + i]: harmonic coefficients of pair i, in the sweep's units; the charge sums are cleared
template <int LA, int LB>
__global__ void __launch_bounds__(32 * ncart(LA))
k_pair_fold(BasisDev bd, int pp_begin, int pp_end, const double *__restrict__ dm, double *__restrict__ pairs)
{
    using Sh = PairShape<LA, LB>;
    constexpr int L = Sh::L, NH = Sh::NH, NA = Sh::NA, NB = Sh::NB, T = Sh::T, KR = Sh::KR;
    extern __shared__ double sm[][32];
    double(*dsum)[32] = sm + (Sh::FS - NH);
    const int lane = threadIdx.x, ia = threadIdx.y, i = pp_begin + blockIdx.x * 32 + lane;
    const size_t np = pp_end - pp_begin, ip = blockIdx.x * 32 + lane;
    const PPLane pl = load_pp(bd, i, pp_end);
    constexpr int TD = (LA + 1) * (LB + 1) * (T + 1);
    for (int d = ia; d < 3; d += NA) {
        const double xa = d == 0 ? pl.P[0] - pl.A[0] : d == 1 ? pl.P[1] - pl.A[1] : pl.P[2] - pl.A[2];
        const double xb = d == 0 ? pl.P[0] - pl.B[0] : d == 1 ? pl.P[1] - pl.B[1] : pl.P[2] - pl.B[2];
        hermite_table<LA, LB, T>(sm + d * TD, lane, xa, xb, 0.5 * pl.ip);
    }
    __syncthreads();
    int a3[3] = {0, 0, 0};
    cart_of(LA, ia, a3);
    double D[NH];
#pragma unroll
    for (int k = 0; k < NH; ++k) D[k] = 0.0;
    const double unit = HALF_SQRT_PI * sqrt(pl.ip);
#pragma unroll 1
    for (int ib = 0; ib < NB; ++ib) {
        int b3[3] = {0, 0, 0};
        cart_of(LB, ib, b3);
        const double g = unit * pair_density(pl, bd, dm, ia, ib);
        // E_t vanishes beyond t = i + j: bounds uniform over the warp
        const int lx = a3[0] + b3[0], ly = a3[1] + b3[1], lz = a3[2] + b3[2];
        double E[3][L + 1];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int t = 0; t <= L; ++t) E[d][t] = sm[d * TD + (a3[d] * (LB + 1) + b3[d]) * (T + 1) + t][lane];
#pragma unroll
        for (int t = 0; t <= L; ++t) {
            if (t > lx) continue;
            const double gx = g * E[0][t];
#pragma unroll
            for (int u = 0; u <= L - t; ++u) {
                if (u > ly) continue;
                const double gxy = gx * E[1][u];
#pragma unroll
                for (int v = 0; v <= L - t - u; ++v)
                    if (v <= lz) D[hidx(t, u, v)] = fma(gxy, E[2][v], D[hidx(t, u, v)]);
            }
        }
    }
    // sum over the components of A, KR Hermite indices at a time
#pragma unroll
    for (int k0 = 0; k0 < NH; k0 += KR) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KR; ++k)
            if (k0 + k < NH) sm[ia * KR + k][lane] = D[k0 + k < NH ? k0 + k : 0];
        __syncthreads();
        for (int k = ia; k < KR && k0 + k < NH; k += NA) {
            double s = 0.0;
            for (int w = 0; w < NA; ++w) s += sm[w * KR + k][lane];
            dsum[k0 + k][lane] = s;
        }
    }
    __syncthreads();
    if (i >= pp_end) return;
    // change of basis: a harmonic component's entries are consecutive in the table
    double m = 0.0;
    for (int e = 0; e < HT.tend[L]; ++e) {
        const HarmEntry &t = HT.t[e];
        const int j = harm_off(L, t.k) + t.lm;
        if (j % NA != ia) continue;
        m += t.c * dsum[t.herm][lane];
        if (e + 1 == HT.tend[L] || HT.t[e + 1].k != t.k || HT.t[e + 1].lm != t.lm) {
            pairs[j * np + ip] = m;
            m = 0.0;
        }
    }
    for (int k = ia; k < NH + 3; k += NA) pairs[(NH + k) * np + ip] = 0.0;
}

// The pairs' gradients from the charge sums: d_a = sum_ab g_ab sum_tuv E'^a_tuv W_tuv with
// E'_t = dE^{ij}_t / dX_AB = (b/p) E^{ij}_{t-1} - 2b E^{i,j+1}_t + j E^{i,j-1}_t in direction a, then
// dE/dA = -(d + a/p se), dE/dB = d - b/p se, se = sum_C q_C e(C)
template <int LA, int LB>
__global__ void __launch_bounds__(32 * ncart(LA))
k_pair_contract(BasisDev bd, int pp_begin, int pp_end, const double *__restrict__ dm, const double *__restrict__ pairs,
                double *__restrict__ gqm)
{
    using Sh = PairShape<LA, LB>;
    constexpr int L = Sh::L, NH = Sh::NH, NA = Sh::NA, NB = Sh::NB, T = Sh::T;
    extern __shared__ double sm[][32];
    double(*W)[32] = sm + Sh::NC, (*dsum)[32] = W + NH;
    const int lane = threadIdx.x, ia = threadIdx.y, i = pp_begin + blockIdx.x * 32 + lane;
    const size_t np = pp_end - pp_begin, ip = min(blockIdx.x * 32 + lane, (int)np - 1);
    const PPLane pl = load_pp(bd, i, pp_end);
    constexpr int TD = (LA + 1) * (LB + 2) * (T + 1);
    for (int d = ia; d < 3; d += NA) {
        const double xa = d == 0 ? pl.P[0] - pl.A[0] : d == 1 ? pl.P[1] - pl.A[1] : pl.P[2] - pl.A[2];
        const double xb = d == 0 ? pl.P[0] - pl.B[0] : d == 1 ? pl.P[1] - pl.B[1] : pl.P[2] - pl.B[2];
        hermite_table<LA, LB + 1, T>(sm + d * TD, lane, xa, xb, 0.5 * pl.ip);
    }
    // harmonic sums -> W (a warp per Hermite index at a time)
    for (int k = ia; k < NH; k += NA) W[k][lane] = 0.0;
    for (int e = 0; e < HT.tend[L]; ++e) {
        const HarmEntry &t = HT.t[e];
        if (t.herm % NA == ia) W[t.herm][lane] += t.c * __ldg(pairs + (NH + harm_off(L, t.k) + t.lm) * np + ip);
    }
    __syncthreads();
    int a3[3] = {0, 0, 0};
    cart_of(LA, ia, a3);
    double dx = 0.0, dy = 0.0, dz = 0.0;
#pragma unroll 1
    for (int ib = 0; ib < NB; ++ib) {
        int b3[3] = {0, 0, 0};
        cart_of(LB, ib, b3);
        const double g = pair_density(pl, bd, dm, ia, ib);
        // E_t and E'_t vanish beyond t = i + j: bounds uniform over the warp, tables read as they are
        const int lx = a3[0] + b3[0], ly = a3[1] + b3[1], lz = a3[2] + b3[2];
        const double(*row[3])[32];
#pragma unroll
        for (int d = 0; d < 3; ++d) row[d] = sm + d * TD + (a3[d] * (LB + 2) + b3[d]) * (T + 1);
        auto deriv = [&](int d, int t) {
            double e = -2.0 * pl.b * row[d][T + 1 + t][lane];
            if (b3[d] > 0) e += (double)b3[d] * row[d][t - (T + 1)][lane];
            if (t > 0) e += pl.b * pl.ip * row[d][t - 1][lane];
            return e;
        };
        double Ez[L + 1], dEz[L + 1], dEy[L + 1];
#pragma unroll
        for (int t = 0; t <= L; ++t) {
            if (t <= lz) {
                Ez[t] = row[2][t][lane];
                dEz[t] = deriv(2, t);
            }
            if (t <= ly) dEy[t] = deriv(1, t);
        }
        double sx = 0.0, sy = 0.0, sz = 0.0;
#pragma unroll 1
        for (int t = 0; t <= lx; ++t) {
            double h = 0.0, hy = 0.0, hz = 0.0;
#pragma unroll
            for (int u = 0; u <= L; ++u) {
                if (u > ly) continue;
                double w = 0.0, wz = 0.0;
#pragma unroll
                for (int v = 0; v <= L - u; ++v)
                    if (v <= lz) {
                        const double x = W[hidx(t, u, v)][lane];
                        w = fma(Ez[v], x, w);
                        wz = fma(dEz[v], x, wz);
                    }
                const double Ey = row[1][u][lane];
                h = fma(Ey, w, h);
                hy = fma(dEy[u], w, hy);
                hz = fma(Ey, wz, hz);
            }
            const double Ex = row[0][t][lane];
            sx = fma(deriv(0, t), h, sx);
            sy = fma(Ex, hy, sy);
            sz = fma(Ex, hz, sz);
        }
        dx = fma(g, sx, dx);
        dy = fma(g, sy, dy);
        dz = fma(g, sz, dz);
    }
    dsum[3 * ia][lane] = dx;
    dsum[3 * ia + 1][lane] = dy;
    dsum[3 * ia + 2][lane] = dz;
    __syncthreads();
    if (ia > 0) return;
    const double unit = HALF_SQRT_PI * sqrt(pl.ip), aop = pl.a * pl.ip, bop = pl.b * pl.ip;
    bool take[5], head;
    seg_setup(pl.active ? pl.s : -1 - lane, lane, take, head);
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        double d = 0.0;
        for (int w = 0; w < NA; ++w) d += dsum[3 * w + x][lane];
        d *= unit;
        const double se = pl.active ? pairs[(2 * NH + x) * np + ip] : 0.0;
        const double gA = seg_reduce(-(d + aop * se), take), gB = seg_reduce(d - bop * se, take);
        if (head && pl.active) {
            atomicAdd(gqm + 3 * pl.atomA + x, gA);
            atomicAdd(gqm + 3 * pl.atomB + x, gB);
        }
    }
}

template <int LA, int LB, int NT>
__global__ void __launch_bounds__(NT, 1)
k_vgrad_f64(BasisDev bd, RegionDev rg, int pp_begin, int pp_end, int ch_begin, int ch_end,
            const double *__restrict__ boys, double *__restrict__ pairs, double *__restrict__ gchg, int *err)
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
        // the density-folded coefficients (k_pair_fold), their gradients, and the charge sums S
        const size_t np = pp_end - pp_begin, ip = min(tile * 32 + lane, (int)np - 1);
        double M[NH], Nx[NG], Ny[NG], Nz[NG], S[NH];
#pragma unroll
        for (int k = 0; k < NH; ++k) M[k] = pl.active ? pairs[k * np + ip] : 0.0;
        harm_grad<L>(M, Nx, Ny, Nz);
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
        if (pl.active) {
#pragma unroll
            for (int k = 0; k < NH; ++k) atomicAdd(pairs + (NH + k) * np + ip, S[k]);
            atomicAdd(pairs + 2 * NH * np + ip, sex);
            atomicAdd(pairs + (2 * NH + 1) * np + ip, sey);
            atomicAdd(pairs + (2 * NH + 2) * np + ip, sez);
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
                             int ch_end, const double *boys, double *pairs, double *gchg, int *err, int nblk,
                             int threads, int nslice, cudaStream_t st)
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
                                                                       pairs, gchg, err);
    return cudaGetLastError();
}

template <int LA, int LB>
cudaError_t VgradF64<LA, LB>::run(const BasisDev &bd, const RegionDev &rg, int pp_begin, int pp_end, int ch_begin,
                                  int ch_end, const double *boys, const double *dm, double *gqm, double *gchg,
                                  int *err, int nblk, int threads, int nslice, double *pairs, cudaStream_t st)
{
    using Sh = PairShape<LA, LB>;
    constexpr size_t row = 32 * sizeof(double);
    static bool attr = false;
    cudaError_t e;
    if (!attr) {
        if ((e = cudaFuncSetAttribute(k_pair_fold<LA, LB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(Sh::FS * row))) != cudaSuccess ||
            (e = cudaFuncSetAttribute(k_pair_contract<LA, LB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(Sh::CS * row))) != cudaSuccess)
            return e;
        attr = true;
    }
    const int tiles = (pp_end - pp_begin + 31) / 32;
    k_pair_fold<LA, LB><<<tiles, dim3(32, Sh::NA), Sh::FS * row, st>>>(bd, pp_begin, pp_end, dm, pairs);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    constexpr int W = sweep_wide_threads(SW_VGRAD_F64, class_of(LA, LB));
    bool wide = false;
    if constexpr (W > 0)
        if (threads == W) {
            wide = true;
            e = launch_nt<LA, LB, W>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys, pairs, gchg, err, nblk, threads,
                                     nslice, st);
        }
    if (!wide)
        e = launch_nt<LA, LB, 256>(bd, rg, pp_begin, pp_end, ch_begin, ch_end, boys, pairs, gchg, err, nblk, threads,
                                   nslice, st);
    if (e != cudaSuccess) return e;
    k_pair_contract<LA, LB><<<tiles, dim3(32, Sh::NA), Sh::CS * row, st>>>(bd, pp_begin, pp_end, dm, pairs, gqm);
    return cudaGetLastError();
}

template struct VgradF64<la_of_class(QMMM_SPLIT_CLASS), lb_of_class(QMMM_SPLIT_CLASS)>;

#else  // the dispatcher

cudaError_t launch_vgrad_f64(const BasisDev &b, const RegionDev &r, int cls, int pp_begin, int pp_end,
                             int ch_begin, int ch_end, const double *boys, const double *dm, double *gqm,
                             double *gchg, int *err, int nblk, int threads, int nslice, double *pairs, cudaStream_t st)
{
    if (pp_end <= pp_begin || ch_end <= ch_begin) return cudaSuccess;
    return dispatch_class<VgradF64>(cls, b, r, pp_begin, pp_end, ch_begin, ch_end, boys, dm, gqm, gchg, err, nblk,
                                    threads, nslice, pairs, st);
}

#endif

}  // namespace qmmm
