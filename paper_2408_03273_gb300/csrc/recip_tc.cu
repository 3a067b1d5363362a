// recip_tc.cu -- the MM structure factor of the reciprocal Ewald sum (SI, "Multipolar Ewald",
// long-range part) on the tensor cores.
//
// S(G) = sum_i q_i exp(i G.R_i) over the half space n_x >= 0 of the cube |n_c| <= kmax, with
// separable phases.  The phases of +n and -n are conjugate, so the sums are taken over real
// functions, per axis cos(2 pi n u), n = 0..k, and sin(2 pi n u), n = 1..k:
//
//   R[(rx, ry), rz] = sum_i a_i(rx, ry) z_i(rz),   a_i = q_i X_i(rx) Y_i(ry),  z_i = Z_i(rz),
//
// a product of two real matrices over the charges, from which S at (n_x, +-n_y, +-n_z) is eight of R
// with signs (k_sf_tc_combine).  Over complex phases both operands had re and im rows per charge:
// twice the products, two N tiles (and so twice the digitising) beyond kz = 19 and two
// multiplications per entry of A.  k_sf_tc on a 150-atom site (kmax 24, 200 001 charges): 4.07 -> 2.01 ms;
// the producers' integer work is the bound (60-atom site: 0.31 ms, tensor pipe 29% busy, issue slots 42%).
//
// The product is D[line, rz] = sum_k A[line, k] B[rz, k], k the charge.  The tensor cores multiply BF16
// operands exactly and accumulate in FP32, so the FP64-class product is built from exact pieces (an
// Ozaki-type split): every operand element,
// a 48-bit fixed-point number v (|v| <= 2^48, scaled by 1/max|q| for A), is written as seven
// balanced digit planes, a leading one and six of base 128,
//     v 2^-48 = 2^-6 sum_{s<7} p_s,   p_0 in [-64, 64],  p_s in [-64, 63] 2^-7s (s >= 1),
// each p_s exact in BF16 (at most 7 significant bits).  Products of planes with s + t = l carry
// the weight 2^-7l; for l <= 3 each level has its own FP32 accumulator in tensor memory and stays
// an exact integer multiple of 2^-7l over a K block of 1024 terms ((l + 1) 4096 * 1024 <= 2^24),
// levels 4..6 are added in FP32 at the end, rounding near 2^-52 of the leading level, and
// the pairs with s + t >= 7 (weight <= 2^-49) are dropped: 28 plane pairs.  Each CTA (a 128-line
// tile, an N tile and a block of 1024 charges) writes five partials; a second kernel sums
// the exact levels over the charge blocks in 64-bit integers and combines them in FP64.
//
// Kernels, in order: per-block max |q|; fixed-point phase rows (one sincospi pair per charge and
// axis, the recurrence in integers); the B digit planes (the z phases are shared by every line
// tile, so they are digitised once, straight into the shared-memory layout of the MMA); the MMA
// kernel; the reduction over charge blocks; S from R.  In the MMA kernel one warp stages the B planes
// and the phase rows of the next chunk of 32 charges with TMA bulk copies, 16 producer warps build the
// A planes of a chunk (an outer product formed on chip: nothing of it goes to HBM), one thread
// issues a chunk's tcgen05.mma (2 K-steps x 28 plane pairs), double-buffered through
// mbarriers, and the epilogue reads tensor memory with tcgen05.ld.
#include <algorithm>

#include "device_common.cuh"
#include "qmmm_internal.h"
#include "tc_common.cuh"
#include "tc_digits.cuh"

namespace qmmm {

namespace {
using namespace tcd;
constexpr int TCM = 128;               // lines per tile (MMA M)
constexpr int TCND = tcd::ND;           // digit planes
constexpr int TCKC = 32;               // K entries (charges) per chunk: two MMA K-steps
constexpr int TCNCH = 32;              // chunks per charge block
constexpr int NSTAGE = 2;              // pipeline depth (A, B and phase-row buffers)
constexpr int TCCPB = TCKC * TCNCH;    // charges per CTA (K block of 1024)
constexpr int TCNACC = 5;              // partials per CTA: levels 0..3 exact, levels 4..6 merged
constexpr int TCPROD = 16;             // producer warps
constexpr int TCGRP = 2;               // groups of producer warps, taking the chunks in turn
constexpr int TCTHREADS = (TCPROD + 3) * 32;  // + the MMA warp, the phase loader, the B plane loader
constexpr uint32_t A_PLANE = TCM * TCKC * 2;  // bytes per A digit plane of a chunk
constexpr uint32_t CM_K = 128;                // byte step between core matrices along K
constexpr uint32_t CM_MN = (TCKC / 8) * 128;  // byte step between 8-row groups
constexpr size_t TC_SMEM_MAX = 232448;           // 227 KB per CTA
constexpr int BMAX_CH = 4096;                    // charges per block of the max |q| reduction

__host__ __device__ inline uint32_t tc_bplane_bytes(int ntr) { return (uint32_t)ntr * TCKC * 2; }
__host__ __device__ inline uint32_t tc_stage_bytes(int ntr) { return TCND * (A_PLANE + tc_bplane_bytes(ntr)); }
// Phase rows of one chunk for the A operand: the x rows that a tile of 128 lines touches and every y
// row, 32 charges of 8 bytes each.  The row stride in shared memory puts the eight lanes of a
// 16-byte access (two rows, four pairs of charges) on 32 distinct banks.
// Global memory holds the rows of a chunk the same way, so that two copies bring them all.
constexpr uint32_t RSTR = TCKC * 8 + 64;
__host__ __device__ inline int tc_xrows(int NY) { return (TCM - 1) / NY + 2; }
__host__ __device__ inline uint32_t tc_pbuf_bytes(int NY) { return (uint32_t)(tc_xrows(NY) + NY) * RSTR; }
__host__ inline size_t tc_smem_bytes(int ntr, int NY, bool staged)
{
    return NSTAGE * ((size_t)tc_stage_bytes(ntr) + (staged ? (size_t)tc_pbuf_bytes(NY) : 0)) + 256;
}

struct TcSfArgs {
    const unsigned char *qx, *py;  // per chunk NX and NY rows of RSTR bytes: split 2^61 fixed point, cos
                                   // rows, then sin rows
    const uint32_t *bpl;  // B planes, per (block, chunk, N tile): TCND * bplane bytes
    int *part;            // per CTA: [5][ntr][128]
    int *err;
    int nmm, NX, NY, NL;
    int ntiles, ntr, mtiles;
};
}  // namespace

// grid (mtiles, nkb * ntiles), TCTHREADS threads, tc_smem_bytes() dynamic shared memory.  STAGED:
// the A phase rows of each chunk come through shared memory (TMA bulk copies); otherwise the
// producers read them from global memory.  The B planes always come by bulk copy.  Chunk ch uses
// buffer set ch % NSTAGE; its barriers complete once per use, phase parity (ch / NSTAGE) & 1.
template <bool STAGED>
__global__ void __launch_bounds__(TCTHREADS, 1) k_sf_tc(TcSfArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    const int ntr = a.ntr, NY = a.NY;
    const uint32_t b_plane = tc_bplane_bytes(ntr), stage = tc_stage_bytes(ntr), bbytes = TCND * b_plane;
    const uint32_t pbytes = STAGED ? tc_pbuf_bytes(NY) : 0;
    unsigned char *pbuf0 = sm + NSTAGE * stage;
    // per stage: full (producers), bfull (B copy), pfull (phase copy), empty (MMA done); then done
    uint64_t *bars = reinterpret_cast<uint64_t *>(pbuf0 + NSTAGE * pbytes);
    uint64_t *full = bars, *bfull = bars + NSTAGE, *pfull = bars + 2 * NSTAGE, *empty = bars + 3 * NSTAGE;
    uint64_t *done = bars + 4 * NSTAGE;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt = blockIdx.x, kb = blockIdx.y / a.ntiles, nt = blockIdx.y % a.ntiles;
    const int rx0 = mt * TCM / NY, xrows = tc_xrows(NY);  // first x row of the tile, rows reserved

    if (threadIdx.x == 0) {
        for (int k = 0; k < NSTAGE; ++k) {
            mbar_init(&full[k], TCPROD / TCGRP);
            mbar_init(&bfull[k], 1);
            mbar_init(&pfull[k], 1);
            mbar_init(&empty[k], 1);
        }
        mbar_init(done, 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == TCPROD) {
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

    if (warp < TCPROD) {
        // ---------------- producers: A digit planes of one chunk ----------------
        // 128 lines x 32 charges in groups of 8 rows x 4 pairs of charges (32 distinct banks); the
        // line indices of a thread are the same for every chunk
        constexpr int NCG = TCKC / 8, NW = TCPROD / TCGRP, AJ = 16 * NCG / NW;
        const int grp = warp / NW, gw = warp % NW;
        int a_x[AJ], a_y[AJ], a_c[AJ];
        uint32_t a_off[AJ];
#pragma unroll
        for (int j = 0; j < AJ; ++j) {
            const int combo = gw + j * NW, rg = combo / NCG, cg = combo % NCG;
            const int r = rg * 8 + (lane >> 2), line = mt * TCM + r;
            a_c[j] = 2 * (cg * 4 + (lane & 3));
            a_x[j] = line < a.NL ? line / NY : -1;
            a_y[j] = line < a.NL ? line - a_x[j] * NY : 0;
            a_off[j] = rg * CM_MN + cg * CM_K + (lane >> 2) * 16 + (lane & 3) * 4;
        }
        for (int ch = grp; ch < TCNCH; ch += TCGRP) {
            const int st = ch % NSTAGE, u = ch / NSTAGE;
            if (ch >= NSTAGE && !tc::mbar_wait_thread(&empty[st], (u - 1) & 1, abort)) {
                give_up();
                break;
            }
            if (STAGED && !tc::mbar_wait_thread(&pfull[st], u & 1, abort)) {
                give_up();
                break;
            }
            unsigned char *sA = sm + st * stage;
            const int c0 = kb * TCCPB + ch * TCKC, cmax = a.nmm - c0;
#pragma unroll
            for (int j = 0; j < AJ; ++j) {
                const int c = a_c[j];
                long long w0 = BAL, w1 = BAL;  // the digits of 0
                if (a_x[j] >= 0 && c < cmax) {
                    int4 x, y;  // two charges
                    if (STAGED) {
                        const unsigned char *rows = pbuf0 + st * pbytes + c * 8;
                        x = *reinterpret_cast<const int4 *>(rows + (a_x[j] - rx0) * RSTR);
                        y = *reinterpret_cast<const int4 *>(rows + (xrows + a_y[j]) * RSTR);
                    } else {
                        const size_t gc = (size_t)(kb * TCNCH + ch);
                        x = __ldg(reinterpret_cast<const int4 *>(a.qx + (gc * a.NX + a_x[j]) * RSTR + c * 8));
                        y = __ldg(reinterpret_cast<const int4 *>(a.py + (gc * NY + a_y[j]) * RSTR + c * 8));
                    }
                    w0 = fixw(rmul61(make_int2(x.x, x.y), make_int2(y.x, y.y)), 12);
                    if (c + 1 < cmax) w1 = fixw(rmul61(make_int2(x.z, x.w), make_int2(y.z, y.w)), 12);
                }
                const Planes p0 = planes(w0), p1 = planes(w1);
#pragma unroll
                for (int s = 0; s < TCND; ++s)
                    *reinterpret_cast<uint32_t *>(sA + s * A_PLANE + a_off[j]) = pack_bf16(p0.p[s], p1.p[s]);
            }
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&full[st]);
        }
    } else if (warp == TCPROD) {
        if (lane == 0) {
            // ---------------- MMA issue: one thread, 28 plane pairs per K-step ----------------
            // The B planes lie one after the other in shared memory and the accumulators of the
            // levels in tensor memory, so plane s of A meets planes t, t + 1, .. of B in one MMA of
            // several times ntr columns, into levels s + t, s + t + 1, ..: a third of the MMAs, A read
            // from shared memory that much less.
            const int most = 256 / ntr;
            for (int ch = 0; ch < TCNCH; ++ch) {
                const int st = ch % NSTAGE, u = ch / NSTAGE;
                if (!tc::mbar_wait_thread(&full[st], u & 1, abort) || !tc::mbar_wait_thread(&bfull[st], u & 1, abort)) {
                    give_up();
                    break;
                }
                tc::fence_after_sync();
                const uint32_t sA = smem_addr(sm + st * stage), sB = sA + TCND * A_PLANE;
#pragma unroll 1
                for (int kk = 0; kk < TCKC / 16; ++kk)
#pragma unroll 1
                    for (int s = 0; s < TCND; ++s) {
                        const uint64_t ad = tc::smem_desc(sA + s * A_PLANE + kk * 2 * CM_K, CM_K, CM_MN);
                        for (int t = 0; t < TCND - s; t += most) {
                            const int np = min(most, TCND - s - t);
                            const uint64_t bd = tc::smem_desc(sB + t * b_plane + kk * 2 * CM_K, CM_K, CM_MN);
                            tc::mma_bf16(tbase + (s + t) * ntr, ad, bd, tc::idesc_bf16_f32(TCM, np * ntr),
                                         ch == 0 && kk == 0 && s == 0 ? 0u : 1u);
                        }
                    }
                tc::commit(&empty[st]);
            }
            tc::commit(done);
        }
    } else if (warp == TCPROD + 1) {
        if (STAGED && lane == 0) {
            // ---------------- phase loader: the x and y rows of chunk ch ----------------
            // a thread of its own, so that the rows need not wait for the MMAs as the B planes do
            const int nxr = min(a.NX - 1, (mt * TCM + TCM - 1) / NY) - rx0 + 1;
            int issued = 0;
            for (int ch = 0; ch < TCNCH; ++ch) {
                const int st = ch % NSTAGE, u = ch / NSTAGE;
                const size_t gc = (size_t)kb * TCNCH + ch;
                // the producers have finished chunk ch - NSTAGE: its phase rows are no longer read
                if (ch >= NSTAGE && !tc::mbar_wait_thread(&full[st], (u - 1) & 1, abort)) {
                    give_up();
                    break;
                }
                unsigned char *dst = pbuf0 + st * pbytes;
                mbar_arrive_expect_tx(&pfull[st], (nxr + NY) * RSTR);
                bulk_g2s(dst, a.qx + (gc * a.NX + rx0) * RSTR, nxr * RSTR, &pfull[st]);
                bulk_g2s(dst + xrows * RSTR, a.py + gc * NY * RSTR, NY * RSTR, &pfull[st]);
                issued = ch + 1;
            }
            // copies possibly still in flight (after a give-up): wait for them to land, bounded in
            // time only (not cut short by the abort flag), before the block may leave
            for (int ch = issued > NSTAGE ? issued - NSTAGE : 0; ch < issued; ++ch)
                tc::mbar_drain(&pfull[ch % NSTAGE], (ch / NSTAGE) & 1);
        }
    } else if (lane == 0) {
        // ---------------- B plane loader ----------------
        int issued = 0;
        for (int ch = 0; ch < TCNCH; ++ch) {
            const int st = ch % NSTAGE, u = ch / NSTAGE;
            // the MMA has finished chunk ch - NSTAGE: the B area of the buffer set is free
            if (ch >= NSTAGE && !tc::mbar_wait_thread(&empty[st], (u - 1) & 1, abort)) {
                give_up();
                break;
            }
            const uint32_t *src = a.bpl + ((size_t)(kb * TCNCH + ch) * a.ntiles + nt) * (bbytes / 4);
            mbar_arrive_expect_tx(&bfull[st], bbytes);
            bulk_g2s(sm + st * stage + TCND * A_PLANE, src, bbytes, &bfull[st]);
            issued = ch + 1;
        }
        for (int ch = issued > NSTAGE ? issued - NSTAGE : 0; ch < issued; ++ch)
            tc::mbar_drain(&bfull[ch % NSTAGE], (ch / NSTAGE) & 1);
    }

    // ---------------- epilogue: tensor memory -> per-CTA partials (warps 0..7) ----------------
    if (warp < 8) {
        if (!tc::mbar_wait_thread(done, 0, abort)) {
            give_up();
            // the MMA thread commits `done` on every path: wait for it (bounded in time only), so
            // that no MMA still writes tensor memory when it is freed below
            tc::mbar_drain(done, 0);
        } else {
            tc::fence_after_sync();
            const int q = warp & 3, half = warp >> 2, row = 32 * q + lane;
            int *dst = a.part + (size_t)((kb * a.ntiles + nt) * a.mtiles + mt) * (TCNACC * ntr * TCM);
            const int cw = ntr / 2;
            const uint32_t tl = tbase + ((uint32_t)(32 * q) << 16);
            for (int acc = 0; acc < TCNACC; ++acc)
                for (int cb = half * cw; cb < half * cw + cw; cb += 8) {
                    float v[8];
                    tc::tmem_ld8(tl + acc * ntr + cb, v);
                    tc::tmem_wait_ld();
                    const float sc = acc < TCNACC - 1 ? (float)(1 << (7 * acc)) : 1.0f;
                    if (acc == TCNACC - 1) {  // the last levels together
#pragma unroll
                        for (int l = TCNACC; l < TCND; ++l) {
                            float x[8];
                            tc::tmem_ld8(tl + l * ntr + cb, x);
                            tc::tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 8; ++k) v[k] += x[k];
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int w = acc < TCNACC - 1 ? __float2int_rn(v[k] * sc) : __float_as_int(v[k]);
                        dst[((size_t)acc * ntr + cb + k) * TCM + row] = w;
                    }
                }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == TCPROD) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tbase, 512);
    }
}

// B digit planes of every (charge block, chunk, N tile), in the shared-memory layout of one stage:
// row rz holds the charges' z phases.  One thread per (row, pair of charges); a warp covers 8 rows x
// 4 pairs, i.e. 128 contiguous bytes of each plane.
__global__ void k_tc_bplanes(const unsigned char *pz, int nmm, int NZ, int ntiles, int ntr, long long nitems,
                             uint32_t *bpl)
{
    const long long item = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= nitems) return;
    const int per = ntr * (TCKC / 2);  // items of one (block, chunk, N tile)
    const long long grp = item / per;
    const int it = (int)(item - grp * per);
    const int nt = (int)(grp % ntiles), chunk = (int)(grp / ntiles);  // chunk over all blocks
    constexpr int NCG = TCKC / 8;  // groups of 4 pairs
    const int ln = it & 31, combo = it >> 5;
    const int j = (combo % NCG) * 4 + (ln & 3), n = (combo / NCG) * 8 + (ln >> 2);
    const int rz = nt * ntr + n, ci = chunk * TCKC + 2 * j;
    long long w0 = BAL, w1 = BAL;
    if (rz < NZ && ci < nmm) {
        const int4 z = __ldg(reinterpret_cast<const int4 *>(pz + ((size_t)chunk * NZ + rz) * RSTR + 16 * j));
        w0 = fixw(join61(z.x, z.y), 13);
        if (ci + 1 < nmm) w1 = fixw(join61(z.z, z.w), 13);
    }
    const Planes p0 = planes(w0), p1 = planes(w1);
    const uint32_t b_words = tc_bplane_bytes(ntr) / 4;
    uint32_t *dst = bpl + (size_t)grp * (TCND * b_words) +
                    ((n >> 3) * CM_MN + (j >> 2) * CM_K + (n & 7) * 16 + (j & 3) * 4) / 4;
#pragma unroll
    for (int s = 0; s < TCND; ++s) dst[(size_t)s * b_words] = pack_bf16(p0.p[s], p1.p[s]);
}

// R[rz NL + line] from the partials: grid (mtiles, NZ), 4 x 128 threads: a row of the line tile per
// thread, the charge blocks split over the four thread groups and added in a fixed order
constexpr int RED_G = 4;
__device__ __forceinline__ double max_of(const double *bmax, int n)
{
    double m = 0.0;
    for (int k = 0; k < n; ++k) m = fmax(m, bmax[k]);
    return m > 0.0 ? m : 1.0;
}
__global__ void __launch_bounds__(TCM *RED_G) k_sf_tc_reduce(const int *part, int nkb, int ntiles, int ntr,
                                                            int mtiles, int NL, const double *bmax, int nbmax,
                                                            double *R)
{
    __shared__ long long sI[RED_G - 1][TCNACC - 1][TCM];
    __shared__ double sF[RED_G - 1][TCM];
    const int mt = blockIdx.x, rz = blockIdx.y, row = threadIdx.x & (TCM - 1), g = threadIdx.x / TCM;
    const int line = mt * TCM + row;
    const int nt = rz / ntr, nl = rz - nt * ntr;
    long long I[TCNACC - 1] = {};
    double F = 0.0;
    if (line < NL)
        for (int kb = g; kb < nkb; kb += RED_G) {
            const int *p = part + (size_t)((kb * ntiles + nt) * mtiles + mt) * (TCNACC * ntr * TCM);
#pragma unroll
            for (int acc = 0; acc < TCNACC - 1; ++acc) I[acc] += p[((size_t)acc * ntr + nl) * TCM + row];
            F += (double)__int_as_float(p[((size_t)(TCNACC - 1) * ntr + nl) * TCM + row]);
        }
    if (g > 0) {
        for (int acc = 0; acc < TCNACC - 1; ++acc) sI[g - 1][acc][row] = I[acc];
        sF[g - 1][row] = F;
    }
    __syncthreads();
    if (g > 0 || line >= NL) return;
    for (int h = 0; h < RED_G - 1; ++h) {
        for (int acc = 0; acc < TCNACC - 1; ++acc) I[acc] += sI[h][acc][row];
        F += sF[h][row];
    }
    for (int acc = TCNACC - 2; acc >= 0; --acc) F += ldexp((double)I[acc], -7 * acc);
    R[(size_t)rz * NL + line] = max_of(bmax, nbmax) * 0x1p-12 * F;
}

// S at (n_x, n_y, n_z) from the real sums: (c_x + i s_x)(c_y + i s_y)(c_z + i s_z), where the sine of a
// negative index is minus that of its magnitude and the sine of index 0 vanishes
__global__ void k_sf_tc_combine(const double *R, int kx, int ky, int kz, double2 *S)
{
    const int NY = 2 * ky + 1, NZ = 2 * kz + 1, NL = (2 * kx + 1) * NY;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (kx + 1) * NY * NZ) return;
    const int nx = k / (NY * NZ), ny = (k / NZ) % NY - ky, nz = k % NZ - kz, ay = abs(ny), az = abs(nz);
    auto at = [&](bool sx, bool sy, bool sz) {
        if ((sx && nx == 0) || (sy && ny == 0) || (sz && nz == 0)) return 0.0;
        const double v = R[(size_t)(sz ? kz + az : az) * NL + (size_t)(sx ? kx + nx : nx) * NY + (sy ? ky + ay : ay)];
        return ((sy && ny < 0) != (sz && nz < 0)) ? -v : v;
    };
    S[k] = make_double2(at(0, 0, 0) - at(0, 1, 1) - at(1, 0, 1) - at(1, 1, 0),
                        at(1, 0, 0) + at(0, 1, 0) + at(0, 0, 1) - at(1, 1, 1));
}

// bmax[b] = max |q_i| over charges [b BMAX_CH, (b + 1) BMAX_CH)
__global__ void __launch_bounds__(256) k_absmax(const double *q, int n, double *bmax)
{
    __shared__ double ws[8];
    const int i0 = blockIdx.x * BMAX_CH;
    double m = 0.0;
#pragma unroll 4
    for (int k = threadIdx.x; k < BMAX_CH; k += 256)
        if (i0 + k < n) m = fmax(m, fabs(q[i0 + k]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = 0.0;
        for (int w = 0; w < 8; ++w) r = fmax(r, ws[w]);
        bmax[blockIdx.x] = r;
    }
}

// fixed-point phase rows, qx = (q_i / max|q|) X_i, py = Y_i, pz = Z_i, per chunk of 32 charges: row r = 0..k
// cos(2 pi r u), row k + n sin(2 pi n u), split 2^61, RSTR bytes apart; one thread per (axis, charge): the
// step from FP64 sincospi, the recurrence in 2^61 fixed point (each step rounds within 2^-60; at
// most kmax steps)
__global__ void k_tc_phases(EwaldDev e, const double *bmax, int nbmax, unsigned char *qx, unsigned char *py,
                            unsigned char *pz)
{
    const long long item = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= 3ll * e.nmm) return;
    const int d = (int)(item / e.nmm), i = (int)(item - (long long)d * e.nmm), k = e.kmax[d];
    unsigned char *col = (d == 0 ? qx : d == 1 ? py : pz) + (size_t)(i / TCKC) * (2 * k + 1) * RSTR + (i % TCKC) * 8;
    const double u = e.mm_xyz[3 * i + d] / e.box[d];
    double sn, cs;
    sincospi(2.0 * u, &sn, &cs);
    const long long sr = fix61(cs), si = fix61(sn);
    long long pr = fix61(d == 0 ? e.mm_q[i] / max_of(bmax, nbmax) : 1.0), pi = 0;
    for (int n = 0; n <= k; ++n) {
        *reinterpret_cast<int2 *>(col + (size_t)n * RSTR) = split61r(pr);
        if (n > 0) *reinterpret_cast<int2 *>(col + (size_t)(k + n) * RSTR) = split61r(pi);
        const long long nr = (mul61(pr, sr) - mul61(pi, si)) * 2;  // 2^60 -> 2^61
        const long long ni = (mul61(pr, si) + mul61(pi, sr)) * 2;
        pr = nr;
        pi = ni;
    }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
void tc_sf_shape(const EwaldDev &e, TcShape &sh)
{
    const int NX = 2 * e.kmax[0] + 1, NY = 2 * e.kmax[1] + 1, NZ = 2 * e.kmax[2] + 1;
    sh.NL = NX * NY;
    sh.mtiles = (sh.NL + TCM - 1) / TCM;
    // N tiles of at most 64 rows: seven accumulators (448 columns) fit in tensor memory, and two
    // pipeline stages with their phase rows in shared memory up to ky = 45 (narrower N tiles: for every
    // ky; 64 rows: kz 24..31 and from 48 on).  Beyond that the producers read the rows from global memory
    sh.ntiles = (NZ + 63) / 64;
    sh.ntr = ((NZ + sh.ntiles - 1) / sh.ntiles + 15) / 16 * 16;
    sh.nkb = (e.nmm + TCCPB - 1) / TCCPB;
    sh.nbmax = (e.nmm + BMAX_CH - 1) / BMAX_CH;
    sh.part_ints = (size_t)sh.nkb * sh.ntiles * sh.mtiles * TCNACC * sh.ntr * TCM;
    // phase rows for whole charge blocks (the bulk copies of the last block stay in bounds)
    sh.phase_bytes = (size_t)sh.nkb * TCNCH * (NX + NY + NZ) * RSTR;
    sh.bplane_words = (size_t)sh.nkb * TCNCH * sh.ntiles * TCND * tc_bplane_bytes(sh.ntr) / 4;
    sh.real_sums = (size_t)sh.NL * NZ;
    sh.staged = tc_smem_bytes(sh.ntr, NY, true) <= TC_SMEM_MAX;
}

cudaError_t launch_structure_factor_tc(const EwaldDev &e, const TcShape &sh, const TcBuf &b, double2 *S, int *err,
                                       cudaStream_t st)
{
    if (e.nmm == 0) return cudaMemsetAsync(S, 0, sizeof(double2) * (size_t)ewald_dense_size(e), st);
    cudaError_t rc;
    const int NX = 2 * e.kmax[0] + 1, NY = 2 * e.kmax[1] + 1, NZ = 2 * e.kmax[2] + 1;
    k_absmax<<<sh.nbmax, 256, 0, st>>>(e.mm_q, e.nmm, b.bmax);
    if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    const size_t nch = (size_t)sh.nkb * TCNCH;  // chunks
    unsigned char *qx = b.phase, *py = qx + nch * NX * RSTR, *pz = py + nch * NY * RSTR;
    {
        const long long n = 3ll * e.nmm;
        k_tc_phases<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(e, b.bmax, sh.nbmax, qx, py, pz);
        if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    }
    {
        const long long n = (long long)sh.nkb * TCNCH * sh.ntiles * sh.ntr * (TCKC / 2);
        k_tc_bplanes<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(pz, e.nmm, NZ, sh.ntiles, sh.ntr, n, b.bpl);
        if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    }
    {
        const size_t smem = tc_smem_bytes(sh.ntr, NY, sh.staged);
        const void *fn = sh.staged ? (const void *)k_sf_tc<true> : (const void *)k_sf_tc<false>;
        static size_t attr[2] = {0, 0};
        if (smem > attr[sh.staged]) {
            if ((rc = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
                return rc;
            attr[sh.staged] = smem;
        }
        TcSfArgs a;
        a.qx = qx;
        a.py = py;
        a.bpl = b.bpl;
        a.part = b.part;
        a.err = err;
        a.nmm = e.nmm;
        a.NX = NX;
        a.NY = NY;
        a.NL = sh.NL;
        a.ntiles = sh.ntiles;
        a.ntr = sh.ntr;
        a.mtiles = sh.mtiles;
        const dim3 grid(sh.mtiles, sh.nkb * sh.ntiles);
        if (sh.staged)
            k_sf_tc<true><<<grid, TCTHREADS, smem, st>>>(a);
        else
            k_sf_tc<false><<<grid, TCTHREADS, smem, st>>>(a);
        if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    }
    k_sf_tc_reduce<<<dim3(sh.mtiles, NZ), TCM * RED_G, 0, st>>>(b.part, sh.nkb, sh.ntiles, sh.ntr, sh.mtiles, sh.NL,
                                                               b.bmax, sh.nbmax, b.R);
    const int n = ewald_dense_size(e);
    k_sf_tc_combine<<<(n + 255) / 256, 256, 0, st>>>(b.R, e.kmax[0], e.kmax[1], e.kmax[2], S);
    return cudaGetLastError();
}

}  // namespace qmmm
