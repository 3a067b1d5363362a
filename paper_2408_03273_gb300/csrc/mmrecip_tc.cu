// mmrecip_tc.cu -- the MM side of the reciprocal Ewald sum (SI, "Multipolar Ewald", long-range
// part, differentiated for the adjoint) on the tensor cores:
//
//   dE/dq_i += sum_G Re[A(G) e^{-iG.R_i}],   dE/dR_i += q_i sum_G G Im[A(G) e^{-iG.R_i}]
//
// over the half space of the kmax cube, with A(G) = 2 g(G) sum_j e^{iG.R_j} (Q_j + i G.mu_j
// - 1/2 G.theta_j.G) from the QM multipoles and the separable phase e^{-iG.R} = X(n_x) Y(n_y) Z(n_z).
// Over (n_y, n_z) the sum is a product of two matrices followed by a short contraction:
//
//   T_k[i, n_x] = sum_{n_y, n_z} C_k[n_x, n_y, n_z] Y_i(n_y) Z_i(n_z),   C_0 = A, C_1 = G_y A, C_2 = G_z A,
//   dE/dq_i = Re sum X_i T_0,  f_x = sum G_x Im(X_i T_0),  f_y = sum Im(X_i T_1),  f_z = sum Im(X_i T_2).
//
// The phases of +n and -n are conjugate, so the product is taken over real functions: per axis
// cos(2 pi n u), n = 0..k, and sin(2 pi n u), n = 1..k, and K = (2 ky + 1)(2 kz + 1) products of one of
// each, their complex coefficients B_k the sums of the four C_k(+-n_y, +-n_z) with factors 1, -i, i.
// Over complex phases K was twice as long and an entry cost two multiplications.  Sum of a 150-atom
// site (kmax 24, 200 001 charges), mixed path: 4.36 -> 2.64 ms with the real functions, -> 2.02 ms with the
// z rows resident in shared memory and the y rows of a chunk in one copy; FP64 path 14.9 -> 8.0 ms.
// Bound: the producers' integer work and barrier round trips per chunk (FP64 path, 60-atom site: 0.97 ms,
// tensor pipe 22% busy, issue slots 35%).
//
// A operand (M = 128 charges x K): the products of the charges' real phases, digitised on chip from
// fixed-point phase rows staged by TMA; B operand (N = 112 rows (k, n_x, re/im) x K): B_k divided
// by a power of two per (k, n_x) so that |B| <= 1, digitised once per call into the shared-memory
// layout.  Digits as for the structure factor (tc_digits.cuh).  FP64 path: seven planes per operand
// (48-bit fixed point), 28 plane pairs per K-step into FP32 accumulators in tensor memory, five
// accumulators (levels 0..3 kept apart, 4..6 merged), so at most 96 N rows per tile.  Mixed path:
// five planes (34-bit operands, 15 plane pairs) and three accumulators (levels 0 and 1 apart, 2..4
// merged: the merged sum's FP32 rounding is about 2^-31 of level 0's scale), so 160 rows per tile
// and the three channels of kx <= 25 take a single N tile: the A operand is digitised once and no
// N row beyond the 6 (kx + 1) in use is computed.  Against the double-float CUDA-core kernel the
// mixed path's sum differs by 9e-10 (dE/dq: 1.6e-9; active site, kmax 16) and 5.5e-9 (7.3e-9; large site,
// kmax 24) of the largest MM gradient component, a tenth or less of the mixed path's error against
// FP64; the FP64 sum from the CUDA cores' by 1.7e-13 (3.4e-13) and 1.1e-12 (1.6e-12).  Level 0
// is exact for any input while 4096 N_y N_z < 2^24 (kmax <= 31) and beyond that unless the
// row-normalised coefficients, which decay as exp(-G^2/4 alpha^2), sum to more than 2^11 in
// magnitude; levels 1 to 3 are sums of random-sign digit products, typically 2^17 or less.  The epilogue
// (one thread per charge) combines the levels exactly in 64-bit integers, applies the row scales
// and contracts with X_i(n_x) in FP64.
#include <algorithm>

#include "device_common.cuh"
#include "qmmm_internal.h"
#include "tc_common.cuh"
#include "tc_digits.cuh"

namespace qmmm {

namespace {
using namespace tcd;
constexpr int MM = 128;                 // charges per tile (MMA M)
constexpr int NRMAX = 256;              // N rows (channel k, n_x, re/im) of one tile, a multiple of 16
constexpr int KC = 16;                  // K entries per chunk
constexpr int YR = 3;                   // y rows that a chunk of 16 entries can touch (N_z >= 8)
constexpr int NSTGMAX = 3;              // pipeline depth (2 when three stages do not fit)
constexpr int NACCMAX = 5;              // accumulators: levels 0 .. nacc-2 exact, the rest merged
constexpr int NPROD = 16;               // producer warps
constexpr int NGRP = 2;                 // groups of producer warps, taking the chunks in turn
constexpr int NTHR = (NPROD + 3) * 32;  // + MMA warp + phase loader + B plane loader
constexpr int NYB = 4;                  // buffers of y rows, one chunk's each
constexpr uint32_t CMK = 128;                    // byte step between core matrices along K
constexpr uint32_t CMN = (KC / 8) * 128;         // byte step between 8-row groups
constexpr uint32_t APL = MM * KC * 2;            // A plane bytes per chunk
constexpr uint32_t RSTR = MM * 8 + 16;           // bytes of one phase row (128 charges, int2) with its padding:
                                                 // 16 lanes that read four charges of four rows meet 32
                                                 // distinct banks; global memory holds the rows the same way
constexpr uint32_t YBUF = YR * RSTR;             // a chunk's y rows
constexpr size_t SMEM_MAX = 232448;
__host__ __device__ inline uint32_t mmr_bpl(int nr) { return (uint32_t)nr * KC * 2; }  // B plane bytes
__host__ __device__ inline uint32_t mmr_stage(int nr, int np) { return np * (APL + mmr_bpl(nr)); }
__host__ inline size_t mmr_smem(int nr, int nstg, int NZ, int np)
{
    return nstg * (size_t)mmr_stage(nr, np) + (size_t)NZ * RSTR + NYB * YBUF + 256;
}
// fixed-point width of an operand with NP planes, and the balanced input w of a value at 2^(bits + shift)
__host__ __device__ constexpr int mmr_bits(int np) { return 6 + 7 * (np - 1); }
template <int NP>
__device__ __forceinline__ long long fixw_n(long long v, int shift)
{
    return (v + (1ll << (shift - 1)) + (bal<NP>() << shift)) >> shift;
}

struct MmrArgs {
    const unsigned char *Yt, *Zt;  // per charge tile NY + 2 and NZ rows of RSTR bytes: split 2^61 fixed
                                   // point, cos rows, then sin rows
    const uint32_t *bpl;   // B planes per chunk (NP * BPL bytes)
    const double *cscale;  // [3][NX] power-of-two row scales
    const double *mm_xyz, *mm_q;
    double *dq, *dR;
    int *err;
    int nmm, NX, NY, NZ, nent, nchunk;
    int nr, nr_last, cpt, nstg;  // N rows of a tile and of the last tile, channels per tile, stages
    int nacc;                  // accumulators (3 or 5)
    double box0;
};
}  // namespace

// Mixed-path epilogue of one charge (row i of the tile) in double-float arithmetic on the FP32
// pipes: the FP64 pipe (2 FMAs per clock and SM) took about a tenth of the kernel's time for the
// level join, the row scales and the contraction with X_i(n_x), while the MMA pipeline of the SM
// stood idle.  The exact levels and the merged one join by error-free two-sums (all terms are
// FP32 values), the row scales are powers of two (exact), the phases X_i(n_x) come from an FP64
// start and step and a double-float recurrence; about 44 significant bits throughout, against
// the 34-bit operands of the sum.
__device__ __forceinline__ void mmr_epilogue_df(const MmrArgs &a, uint32_t tl, int NR, int kfirst, int nk, bool act,
                                                int i)
{
    double sn, cs;
    sincospi(-2.0 * (act ? a.mm_xyz[3 * i] : 0.0) / a.box0, &sn, &cs);
    const c2 step{f2_from(cs), f2_from(sn)};
    c2 X{f2{1.0f, 0.0f}, f2{0.0f, 0.0f}};
    const f2 g1 = f2_from(6.283185307179586476925 / a.box0);  // G_x per unit n_x
    float ph = 0.0f, pl = 0.0f;                               // sum_nx Re(X T_0)
    float fh[3] = {0.0f, 0.0f, 0.0f}, fl[3] = {0.0f, 0.0f, 0.0f};  // sum_nx Im(X T_k), tile channel kl
    for (int nx = 0; nx < a.NX; ++nx) {
#pragma unroll
        for (int kl = 0; kl < 3; ++kl) {
            if (kl >= nk) break;
            const int k = kfirst + kl, col = 2 * (kl * a.NX + nx);
            uint32_t v[NACCMAX][2];
#pragma unroll
            for (int acc = 0; acc < NACCMAX; ++acc) {
                v[acc][0] = v[acc][1] = 0u;
                if (acc < a.nacc)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                                 : "=r"(v[acc][0]), "=r"(v[acc][1])
                                 : "r"(tl + acc * NR + col)
                                 : "memory");
            }
            tc::tmem_wait_ld();
            const float sc = (float)(__ldg(a.cscale + k * a.NX + nx) * 0x1p-12);  // a power of two
            f2 t[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float h = __uint_as_float(v[0][r]), l = 0.0f;
#pragma unroll
                for (int acc = 1; acc < NACCMAX; ++acc)
                    if (acc < a.nacc) df_add(h, l, __uint_as_float(v[acc][r]));
                t[r] = f2_fast2sum(h * sc, l * sc);
            }
            if (k == 0) {
                f2_mac(ph, pl, X.re, t[0]);
                f2_mac(ph, pl, f2_neg(X.im), t[1]);
                const f2 u = f2_add(f2_mul(X.re, t[1]), f2_mul(X.im, t[0]));
                f2_mac(fh[kl], fl[kl], f2_mul(g1, f2{(float)nx, 0.0f}), u);
            } else {
                f2_mac(fh[kl], fl[kl], X.re, t[1]);
                f2_mac(fh[kl], fl[kl], X.im, t[0]);
            }
        }
        X = c2_mul(X, step);
    }
    if (act) {
        // each channel belongs to exactly one N tile: no two CTAs write the same output
        const double q = a.mm_q[i];
        if (kfirst == 0) a.dq[i] += f2_to(ph, pl);
#pragma unroll
        for (int kl = 0; kl < 3; ++kl)
            if (kl < nk) a.dR[3 * i + kfirst + kl] += q * f2_to(fh[kl], fl[kl]);
    }
}

// grid (mtiles, N tiles), NTHR threads, mmr_smem() dynamic shared memory; chunk ch uses buffer set
// ch % nstg.  NP digit planes per operand: 7 (48-bit operands, FP64 class) on the FP64 path, 5
// (34-bit) on the mixed path.
template <int NP>
__global__ void __launch_bounds__(NTHR, 1) k_mm_recip_tc(MmrArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    // the last N tile may hold fewer channels and rows; the smem layout follows its own NR
    const int NSTG = a.nstg, NR = (int)blockIdx.y + 1 == (int)gridDim.y ? a.nr_last : a.nr;
    const uint32_t BPL = mmr_bpl(NR), STG = mmr_stage(NR, NP);
    unsigned char *zrows = sm + NSTG * STG, *ybuf = zrows + a.NZ * RSTR;
    // per stage: full (producers), bfull (B copy), empty (MMA done); per y buffer: yfull (copy), yempty
    // (producers have read it); zfull; done
    uint64_t *bars = reinterpret_cast<uint64_t *>(ybuf + NYB * YBUF);
    uint64_t *full = bars, *bfull = bars + NSTGMAX, *empty = bars + 2 * NSTGMAX;
    uint64_t *yfull = bars + 3 * NSTGMAX, *yempty = yfull + NYB, *zfull = yempty + NYB, *done = zfull + 1;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * MM;
    // N tile blockIdx.y: channels [kfirst, kfirst + nk), its own B planes
    const int kfirst = blockIdx.y * a.cpt, nk = min(a.cpt, 3 - kfirst);
    const uint32_t *bpl = a.bpl + (size_t)blockIdx.y * a.nchunk * (NP * mmr_bpl(a.nr) / 4);

    if (threadIdx.x == 0) {
        for (int k = 0; k < NSTGMAX; ++k) {
            mbar_init(&full[k], NPROD / NGRP);
            mbar_init(&bfull[k], 1);
            mbar_init(&empty[k], 1);
        }
        for (int k = 0; k < NYB; ++k) {
            mbar_init(&yfull[k], 1);
            mbar_init(&yempty[k], NPROD / NGRP);
        }
        mbar_init(zfull, 1);
        mbar_init(done, 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == NPROD) {
        tc::tmem_alloc(tslot, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *tslot;
    auto give_up = [&]() {
        *abort = 1;
        atomicOr(a.err, DEVERR_TIMEOUT);
    };

    if (warp < NPROD) {
        // ---------------- producers: A planes, 128 charges x 16 entries per chunk ----------------
        // groups of 8 charges x 4 pairs of entries (32 distinct banks)
        constexpr int AJ = 32 * NGRP / NPROD;
        const int grp = warp / (NPROD / NGRP), gw = warp % (NPROD / NGRP);
        int e_m[AJ], e_k[AJ];
        uint32_t e_off[AJ];
#pragma unroll
        for (int j = 0; j < AJ; ++j) {
            const int combo = gw * AJ + j, rg = combo >> 1, cg = combo & 1;
            e_m[j] = rg * 8 + (lane >> 2);
            e_k[j] = 2 * (cg * 4 + (lane & 3));
            e_off[j] = rg * CMN + cg * CMK + (lane >> 2) * 16 + (lane & 3) * 4;
        }
        int z0 = grp * KC % a.NZ;  // z index of the chunk's first entry
        for (int ch = grp; ch < a.nchunk; ch += NGRP, z0 = (z0 + NGRP * KC) % a.NZ) {
            const int st = ch % NSTG, u = ch / NSTG, yb = ch % NYB;
            if ((ch >= NSTG && !tc::mbar_wait_thread(&empty[st], (u - 1) & 1, abort)) ||
                (ch == grp && !tc::mbar_wait_thread(zfull, 0, abort)) ||
                !tc::mbar_wait_thread(&yfull[yb], (ch / NYB) & 1, abort)) {
                give_up();
                break;
            }
            unsigned char *sA = sm + st * STG;
            const unsigned char *yrows = ybuf + yb * YBUF;
            const int p0 = ch * KC;
#pragma unroll
            for (int j = 0; j < AJ; ++j) {
                const int m = e_m[j];
                PlanesN<NP> pl[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = e_k[j] + h, z = z0 + k;
                    const int y = (z >= a.NZ) + (z >= 2 * a.NZ);  // y row of the entry, from the chunk's first
                    const int2 ys = *reinterpret_cast<const int2 *>(yrows + y * RSTR + m * 8);
                    const int2 zs = *reinterpret_cast<const int2 *>(zrows + (z - y * a.NZ) * RSTR + m * 8);
                    constexpr int SH = 60 - mmr_bits(NP);
                    long long w = bal<NP>();  // the digits of 0
                    if (m0 + m < a.nmm && p0 + k < a.nent) w = fixw_n<NP>(rmul61(ys, zs), SH);
                    pl[h] = planes_n<NP>(w);
                }
#pragma unroll
                for (int s = 0; s < NP; ++s)
                    *reinterpret_cast<uint32_t *>(sA + s * APL + e_off[j]) = pack_bf16(pl[0].p[s], pl[1].p[s]);
            }
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive(&yempty[yb]);
                tc::mbar_arrive(&full[st]);
            }
        }
    } else if (warp == NPROD) {
        if (lane == 0) {
            // ---------------- MMA issue: NP (NP + 1) / 2 plane pairs per chunk ----------------
            const uint32_t idesc = tc::idesc_bf16_f32(MM, NR);
            for (int ch = 0; ch < a.nchunk; ++ch) {
                const int st = ch % NSTG, u = ch / NSTG;
                if (!tc::mbar_wait_thread(&full[st], u & 1, abort) || !tc::mbar_wait_thread(&bfull[st], u & 1, abort)) {
                    give_up();
                    break;
                }
                tc::fence_after_sync();
                const uint32_t sA = smem_addr(sm + st * STG), sB = sA + NP * APL;
#pragma unroll
                for (int s = 0; s < NP; ++s)
#pragma unroll
                    for (int t = 0; t < NP - s; ++t) {
                        const int acc = s + t < a.nacc - 1 ? s + t : a.nacc - 1;
                        const uint32_t first = (ch == 0 && s == 0 && t == acc);
                        const uint64_t ad = tc::smem_desc(sA + s * APL, CMK, CMN);
                        const uint64_t bd = tc::smem_desc(sB + t * BPL, CMK, CMN);
                        tc::mma_bf16(tbase + acc * NR, ad, bd, idesc, first ? 0u : 1u);
                    }
                tc::commit(&empty[st]);
            }
            tc::commit(done);
        }
    } else if (warp == NPROD + 1) {
        if (lane == 0) {
            // ---------------- phase loader: every z row once, then the y rows of each chunk ----------------
            // few large copies: with one copy per row of a chunk (19 of 1 KB) their issue set the time of
            // a chunk (mixed sum of a 150-atom site 2.44 ms, with these copies 2.02)
            int issued = 0;
            mbar_arrive_expect_tx(zfull, a.NZ * RSTR);
            for (uint32_t o = 0; o < a.NZ * RSTR; o += 65536)
                bulk_g2s(zrows + o, a.Zt + (size_t)blockIdx.x * a.NZ * RSTR + o, min(65536u, a.NZ * RSTR - o), zfull);
            for (int ch = 0; ch < a.nchunk; ++ch) {
                const int yb = ch % NYB, u = ch / NYB;
                if (ch >= NYB && !tc::mbar_wait_thread(&yempty[yb], (u - 1) & 1, abort)) {
                    give_up();
                    break;
                }
                mbar_arrive_expect_tx(&yfull[yb], YBUF);
                bulk_g2s(ybuf + yb * YBUF, a.Yt + ((size_t)blockIdx.x * (a.NY + YR - 1) + ch * KC / a.NZ) * RSTR, YBUF,
                         &yfull[yb]);
                issued = ch + 1;
            }
            // copies possibly still in flight (after a give-up): wait for them to land, bounded in time
            // only (not cut short by the abort flag), before the block may leave
            tc::mbar_drain(zfull, 0);
            for (int ch = issued > NYB ? issued - NYB : 0; ch < issued; ++ch)
                tc::mbar_drain(&yfull[ch % NYB], (ch / NYB) & 1);
        }
    } else if (lane == 0) {
        // ---------------- B plane loader ----------------
        int issued = 0;
        for (int ch = 0; ch < a.nchunk; ++ch) {
            const int st = ch % NSTG, u = ch / NSTG;
            if (ch >= NSTG && !tc::mbar_wait_thread(&empty[st], (u - 1) & 1, abort)) {
                give_up();
                break;
            }
            mbar_arrive_expect_tx(&bfull[st], NP * BPL);
            bulk_g2s(sm + st * STG + NP * APL, bpl + (size_t)ch * (NP * BPL / 4), NP * BPL, &bfull[st]);
            issued = ch + 1;
        }
        for (int ch = issued > NSTG ? issued - NSTG : 0; ch < issued; ++ch)
            tc::mbar_drain(&bfull[ch % NSTG], (ch / NSTG) & 1);
    }

    // ---------------- epilogue: one thread per charge (warps 0..3) ----------------
    if (warp < 4) {
        if (!tc::mbar_wait_thread(done, 0, abort)) {
            give_up();
            // the MMA thread commits `done` on every path: wait for it (bounded in time only), so
            // that no MMA still writes tensor memory when it is freed below
            tc::mbar_drain(done, 0);
        } else {
            tc::fence_after_sync();
            const int row = 32 * warp + lane, i = m0 + row;
            const uint32_t tl = tbase + ((uint32_t)(32 * warp) << 16);
            const bool act = i < a.nmm;
            if constexpr (NP == MMR_NP_MIXED) {
                mmr_epilogue_df(a, tl, NR, kfirst, nk, act, i);
            } else {
            double sn, cs;
            sincospi(-2.0 * (act ? a.mm_xyz[3 * i] : 0.0) / a.box0, &sn, &cs);
            double xr = 1.0, xi = 0.0;
            double pot = 0.0;
            double f[3] = {0.0, 0.0, 0.0};  // sum_nx Im(X T_k) (channel 0 weighted by G_x)
            for (int nx = 0; nx < a.NX; ++nx) {
                const double gx = 6.283185307179586476925 * nx / a.box0;
                for (int kl = 0; kl < nk; ++kl) {
                    const int k = kfirst + kl, col = 2 * (kl * a.NX + nx);
                    uint32_t v[NACCMAX][2];
#pragma unroll
                    for (int acc = 0; acc < NACCMAX; ++acc) {
                        v[acc][0] = v[acc][1] = 0u;
                        if (acc < a.nacc)
                            asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                                         : "=r"(v[acc][0]), "=r"(v[acc][1])
                                         : "r"(tl + acc * NR + col)
                                         : "memory");
                    }
                    tc::tmem_wait_ld();
                    double t2[2];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        // exact levels 0 .. nacc-2 in units of 2^-21, then the merged rest
                        long long ex = 0;
#pragma unroll
                        for (int l = 0; l < NACCMAX - 1; ++l)
                            if (l < a.nacc - 1)
                                ex += __float2ll_rn(__uint_as_float(v[l][r]) * (float)(1 << (7 * l))) << (21 - 7 * l);
                        t2[r] = fma((double)ex, 0x1p-21, (double)__uint_as_float(v[a.nacc - 1][r]));
                    }
                    const double sc = __ldg(a.cscale + k * a.NX + nx) * 0x1p-12;
                    const double tr = t2[0] * sc, ti = t2[1] * sc;
                    if (k == 0) pot += xr * tr - xi * ti;
                    f[k] += (k == 0 ? gx : 1.0) * (xr * ti + xi * tr);
                }
                const double nr = xr * cs - xi * sn;
                xi = xr * sn + xi * cs;
                xr = nr;
            }
            if (act) {
                // each channel belongs to exactly one N tile: no two CTAs write the same output
                const double q = a.mm_q[i];
                if (kfirst == 0) a.dq[i] += pot;
                for (int kl = 0; kl < nk; ++kl) a.dR[3 * i + kfirst + kl] += q * f[kfirst + kl];
            }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == NPROD) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tbase, 512);
    }
}

// The charges' real phases along y and z, per tile of 128 charges: row r = 0..k holds cos(2 pi r u), row
// k + n sin(2 pi n u), split 2^61 fixed point, RSTR bytes apart; the y rows of a tile are followed by
// YR - 1 that only pad the last chunks' copies.  One thread per (axis, charge): the step from FP64
// sincospi, the recurrence in fixed point.
__global__ void k_mmr_phases(EwaldDev e, unsigned char *Yt, unsigned char *Zt)
{
    const long long item = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= 2ll * e.nmm) return;
    const int d = 1 + (int)(item / e.nmm), i = (int)(item - (long long)(d - 1) * e.nmm);
    const int k = e.kmax[d], rows = 2 * k + (d == 1 ? YR : 1);
    unsigned char *col = (d == 1 ? Yt : Zt) + (size_t)(i / MM) * rows * RSTR + (i % MM) * 8;
    const double u = e.mm_xyz[3 * i + d] / e.box[d];
    double sn, cs;
    sincospi(2.0 * u, &sn, &cs);
    const long long sr = fix61(cs), si = fix61(sn);
    long long pr = fix61(1.0), pi = 0;
    for (int n = 0; n <= k; ++n) {
        *reinterpret_cast<int2 *>(col + (size_t)n * RSTR) = split61r(pr);
        if (n > 0) *reinterpret_cast<int2 *>(col + (size_t)(k + n) * RSTR) = split61r(pi);
        const long long nr = (mul61(pr, sr) - mul61(pi, si)) * 2;
        const long long ni = (mul61(pr, si) + mul61(pi, sr)) * 2;
        pr = nr;
        pi = ni;
    }
}

// channel k of the B operand at dense index (n_x, iy, iz): C_0 = A, C_1 = G_y A, C_2 = A_z
__device__ __forceinline__ double2 mmr_channel(const double2 *A, const double2 *Az, int k, size_t idx, double gy)
{
    if (k == 2) return Az[idx];
    const double2 c = A[idx];
    return k == 1 ? make_double2(gy * c.x, gy * c.y) : c;
}

// Coefficient B_k of the product of real phase functions p = (ry, rz) at n_x: the sum over the signs of
// (n_y, n_z) of C_k times 1 for a cosine, -i (n > 0) or i (n < 0) for a sine
__device__ __forceinline__ double2 mmr_coef(const EwaldDev &e, const double2 *A, const double2 *Az, int k, int nx, int p)
{
    const int ky = e.kmax[1], kz = e.kmax[2], NY = 2 * ky + 1, NZ = 2 * kz + 1;
    const int ry = p / NZ, rz = p - ry * NZ;
    const bool siny = ry > ky, sinz = rz > kz;
    const int ny = siny ? ry - ky : ry, nz = sinz ? rz - kz : rz;
    double2 s = make_double2(0.0, 0.0);
    for (int sy = ny ? -1 : 1; sy <= 1; sy += 2)
        for (int sz = nz ? -1 : 1; sz <= 1; sz += 2) {
            const double gy = 6.283185307179586476925 * (sy * ny) / e.box[1];
            double2 c = mmr_channel(A, Az, k, ((size_t)nx * NY + sy * ny + ky) * NZ + sz * nz + kz, gy);
            if (siny) c = sy > 0 ? make_double2(c.y, -c.x) : make_double2(-c.y, c.x);
            if (sinz) c = sz > 0 ? make_double2(c.y, -c.x) : make_double2(-c.y, c.x);
            s.x += c.x;
            s.y += c.y;
        }
    return s;
}

// cscale[k NX + n_x] = 2^e >= max over the entries of |Re B_k|, |Im B_k| (1 where B_k vanishes);
// one block per (k, n_x)
__global__ void __launch_bounds__(256) k_mmr_scale(EwaldDev e, const double2 *A, const double2 *Az, double *cscale)
{
    __shared__ double ws[8];
    const int NX = e.kmax[0] + 1, NY = 2 * e.kmax[1] + 1, NZ = 2 * e.kmax[2] + 1;
    const int k = blockIdx.x / NX, nx = blockIdx.x % NX;
    double m = 0.0;
    for (int t = threadIdx.x; t < NY * NZ; t += 256) {
        const double2 c = mmr_coef(e, A, Az, k, nx, t);
        m = fmax(m, fmax(fabs(c.x), fabs(c.y)));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = 0.0;
        for (int w = 0; w < 8; ++w) r = fmax(r, ws[w]);
        int ex = 0;
        if (r > 0.0) frexp(r, &ex);
        cscale[blockIdx.x] = r > 0.0 ? ldexp(1.0, ex) : 1.0;
    }
}

// B planes of one N tile (channels [kfirst, kfirst + nk)), per chunk of 16 entries, in the
// shared-memory layout: row (k, n_x, 0) holds Re B_k / cscale, row (k, n_x, 1) Im B_k / cscale.  A warp
// writes 8 rows x 4 pairs of entries: 128 contiguous bytes of each plane.
template <int NP>
__global__ void k_mmr_bplanes(EwaldDev e, const double2 *A, const double2 *Az, const double *cscale, int kfirst,
                              int nk, int nr, int nchunk, uint32_t *bpl)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per = (long long)nr * (KC / 2);  // (row, pair of entries) items of one chunk
    if (t >= per * nchunk) return;
    const int ch = (int)(t / per), it = (int)(t - (long long)ch * per);
    const int NX = e.kmax[0] + 1, nent = (2 * e.kmax[1] + 1) * (2 * e.kmax[2] + 1);
    const int lane = it & 31, grp = it >> 5;
    const int j = (grp & 1) * 4 + (lane & 3), n = (grp >> 1) * 8 + (lane >> 2);
    long long w0 = bal<NP>(), w1 = bal<NP>();
    if (n < 2 * nk * NX) {
        const int kl = n / (2 * NX), nx = (n % (2 * NX)) >> 1, r = n & 1, k = kfirst + kl;
        // over the power-of-two scale (exact), to fixed point
        const double sc = (double)(1ll << mmr_bits(NP)) / cscale[k * NX + nx];
        const int p = ch * KC + 2 * j;
        if (p < nent) {
            const double2 c = mmr_coef(e, A, Az, k, nx, p);
            w0 += __double2ll_rn((r ? c.y : c.x) * sc);
        }
        if (p + 1 < nent) {
            const double2 c = mmr_coef(e, A, Az, k, nx, p + 1);
            w1 += __double2ll_rn((r ? c.y : c.x) * sc);
        }
    }
    const PlanesN<NP> p0 = planes_n<NP>(w0), p1 = planes_n<NP>(w1);
    const uint32_t words = mmr_bpl(nr) / 4;
    uint32_t *dst = bpl + (size_t)ch * NP * words + ((n >> 3) * CMN + (j >> 2) * CMK + (n & 7) * 16 + (j & 3) * 4) / 4;
#pragma unroll
    for (int s = 0; s < NP; ++s) dst[(size_t)s * words] = pack_bf16(p0.p[s], p1.p[s]);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
// nacc accumulators (levels 0 .. nacc-2 exact) of at most 512 / nacc columns each: the channels
// take as few N tiles as fit (FP64 path: 5, 96 rows; mixed path: 3, 160 rows)
void tc_mmr_shape(const EwaldDev &e, int nacc, int np, MmrShape &sh)
{
    sh.np = np;
    const int NX = e.kmax[0] + 1, NY = 2 * e.kmax[1] + 1, NZ = 2 * e.kmax[2] + 1;
    sh.nacc = nacc;
    sh.mtiles = (e.nmm + MM - 1) / MM;
    sh.nent = NY * NZ;
    sh.nchunk = (sh.nent + KC - 1) / KC;
    const int maxr = std::min(NRMAX, 512 / nacc / 16 * 16);  // N rows that fit nacc accumulators
    int cpt = 3;  // channels per N tile: 2 cpt NX rows
    while (cpt > 1 && 2 * cpt * NX > maxr) --cpt;
    sh.cpt = cpt;
    sh.ntiles = (3 + cpt - 1) / cpt;
    sh.nr = (2 * cpt * NX + 15) / 16 * 16;
    sh.nr_last = (2 * (3 - (sh.ntiles - 1) * cpt) * NX + 15) / 16 * 16;
    // a chunk of 16 entries touches at most YR y rows from N_z = 8
    sh.supported = sh.nr <= maxr && NZ >= 8 && mmr_smem(sh.nr, 2, NZ, np) <= SMEM_MAX;
    sh.nstg = mmr_smem(sh.nr, 3, NZ, np) <= SMEM_MAX ? 3 : 2;
    sh.phase_bytes = (size_t)sh.mtiles * (NY + YR - 1 + NZ) * RSTR;
    sh.bplane_words = ((size_t)(sh.ntiles - 1) * mmr_bpl(sh.nr) + mmr_bpl(sh.nr_last)) * sh.nchunk * np / 4;
}

template <int NP>
static cudaError_t mm_recip_np(const EwaldDev &e, const MmrShape &sh, const MmrBuf &b, const double2 *A,
                               const double2 *Az, const unsigned char *Yt, const unsigned char *Zt, double *dq,
                               double *dR, int *err, cudaStream_t st);

cudaError_t launch_mm_recip_tc(const EwaldDev &e, const MmrShape &sh, const MmrBuf &b, const double2 *A,
                               const double2 *Az, double *dq, double *dR, int *err, cudaStream_t st)
{
    if (e.nmm == 0) return cudaSuccess;
    cudaError_t rc;
    const int NX = e.kmax[0] + 1, NY = 2 * e.kmax[1] + 1;
    unsigned char *Yt = b.phase, *Zt = Yt + (size_t)sh.mtiles * (NY + YR - 1) * RSTR;
    k_mmr_phases<<<(unsigned)((2ll * e.nmm + 255) / 256), 256, 0, st>>>(e, Yt, Zt);
    if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    k_mmr_scale<<<3 * NX, 256, 0, st>>>(e, A, Az, b.cscale);
    if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    if (sh.np == MMR_NP_FP64) return mm_recip_np<MMR_NP_FP64>(e, sh, b, A, Az, Yt, Zt, dq, dR, err, st);
    if (sh.np == MMR_NP_MIXED) return mm_recip_np<MMR_NP_MIXED>(e, sh, b, A, Az, Yt, Zt, dq, dR, err, st);
    return cudaErrorInvalidValue;
}

// B planes and the MMA kernel with NP planes per operand
template <int NP>
static cudaError_t mm_recip_np(const EwaldDev &e, const MmrShape &sh, const MmrBuf &b, const double2 *A,
                               const double2 *Az, const unsigned char *Yt, const unsigned char *Zt, double *dq,
                               double *dR, int *err, cudaStream_t st)
{
    cudaError_t rc;
    const int NX = e.kmax[0] + 1, NY = 2 * e.kmax[1] + 1, NZ = 2 * e.kmax[2] + 1;
    const size_t smem = mmr_smem(sh.nr, sh.nstg, NZ, NP);
    static size_t at = 0;
    if (smem > at) {
        if ((rc = cudaFuncSetAttribute((const void *)k_mm_recip_tc<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem)) != cudaSuccess)
            return rc;
        at = smem;
    }
    const size_t tile_words = (size_t)sh.nchunk * NP * mmr_bpl(sh.nr) / 4;
    for (int tl = 0; tl < sh.ntiles; ++tl) {
        const int kfirst = tl * sh.cpt, nk = std::min(sh.cpt, 3 - kfirst);
        const int nr = tl + 1 == sh.ntiles ? sh.nr_last : sh.nr;
        const long long n = (long long)nr * (KC / 2) * sh.nchunk;
        k_mmr_bplanes<NP><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(e, A, Az, b.cscale, kfirst, nk, nr,
                                                                        sh.nchunk, b.bpl + tl * tile_words);
        if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    }
    MmrArgs a;
    a.Yt = Yt;
    a.Zt = Zt;
    a.bpl = b.bpl;
    a.cscale = b.cscale;
    a.mm_xyz = e.mm_xyz;
    a.mm_q = e.mm_q;
    a.dq = dq;
    a.dR = dR;
    a.err = err;
    a.nmm = e.nmm;
    a.NX = NX;
    a.NY = NY;
    a.NZ = NZ;
    a.nent = sh.nent;
    a.nchunk = sh.nchunk;
    a.nr = sh.nr;
    a.nr_last = sh.nr_last;
    a.cpt = sh.cpt;
    a.nstg = sh.nstg;
    a.nacc = sh.nacc;
    a.box0 = e.box[0];
    k_mm_recip_tc<NP><<<dim3(sh.mtiles, sh.ntiles), NTHR, smem, st>>>(a);
    if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    return cudaSuccess;
}

}  // namespace qmmm
