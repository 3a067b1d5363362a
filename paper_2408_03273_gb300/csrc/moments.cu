// moments.cu -- overlap-type moment integrals about the atom centres and what is built from
// them: Mulliken charge/dipole/quadrupole (SI, "Multipolar Ewald"), the region-II Fock term of
// Eqs. 11-14 and the multipole Pulay gradient of Eq. 15.
//
// Everything goes through the Hermite expansion of the pair density g_a g_b = sum E^x_t E^y_u E^z_v
// Lambda_tuv: a polynomial of order n about any centre only sees t + u + v <= n (in one direction
// int Lambda_t (x-K)^e = M^e_t,  M^0 = (1), M^1 = (X_PK, 1), M^2 = (X_PK^2 + h, 2 X_PK, 2),
// M^3 = (X_PK^3 + 3 h X_PK, 3 X_PK^2 + 3 h, 6 X_PK, 6),  h = 1/(2p)), so
//   * the multipoles of both atoms follow from D_tuv = sum_ab gamma_ab E^x_t E^y_u E^z_v, ten sums per
//     pair (twenty for octupoles), by a change of basis once per pair;
//   * with the local potential polynomial W_k(r) = sum_c w_c v_k,c O_c(r - R_k) of atom k (w = 1, or
//     2 for the off-diagonal theta components) and H^k_tuv = int Lambda_tuv W_k, the Fock element
//     F_{mu nu} = -1/2 (<mu|W_{k(mu)}|nu> + <mu|W_{k(nu)}|nu>) is -1/2 sum E E E (H^A + H^B)_tuv;
//   * E_II = sum_k Z_k v_k,0 - sum_{mu in k, nu} gamma_{nu mu} <mu|W_k|nu> moves with the basis: moving B
//     by d moves P by b/p and changes E by -dE/dX_AB, and <a|W_A|b> only depends on B - A, so
//       dE_II/dA = -dE_II/dB = sum_tuv D_tuv (b/p H^A - a/p H^B)_{tuv + 1_d} - sum_tuv D'_d,tuv (H^A + H^B)_tuv,
//       dE^{ij}_t/dX_AB = (b/p) E^{ij}_{t-1} - 2b E^{i,j+1}_t + j E^{i,j-1}_t.
// The sums over the Cartesian components cost 20 FP64 instructions per component for the
// multipoles, 20 for the Fock term and 50 for the gradient, where forming ten operator integrals
// about each centre took about 80, 20 and 350.  The kernels are bound by the FP64 pipe (2 lanes per
// clock and SM), on small systems by one warp's chain of FP64 instructions.  qmmm_ewald (multipoles)
// on a QM water 0.25 -> 0.12 ms, on a 60-atom site 0.58 -> 0.33 ms, on a 150-atom site with f shells
// 2.9 -> 1.3 ms; the multipoles with their gradient in qmmm_forces on the 150-atom site, 14.5 -> 9.5 ms
// for everything outside the sweep.
// A density that is not symmetric counts gamma_{nu mu} for mu's atom, as the definitions have it: the
// difference to the transpose is carried in sums of its own, formed only where it is not zero.
#include "pp_tile.cuh"

namespace qmmm {

__host__ __device__ constexpr int op_x(int c) { return c == 1 ? 1 : c == 4 ? 2 : (c == 5 || c == 6) ? 1 : 0; }
__host__ __device__ constexpr int op_y(int c) { return c == 2 ? 1 : c == 7 ? 2 : (c == 5 || c == 8) ? 1 : 0; }
__host__ __device__ constexpr int op_z(int c) { return c == 3 ? 1 : c == 9 ? 2 : (c == 6 || c == 8) ? 1 : 0; }
// Exponents of the octupole components xxx, xxy, xxz, xyy, xyz, xzz, yyy, yyz, yzz, zzz
__host__ __device__ constexpr int o3_x(int c) { return c == 0 ? 3 : c <= 2 ? 2 : c <= 5 ? 1 : 0; }
__host__ __device__ constexpr int o3_z(int c)
{
    return c == 9 ? 3 : (c == 5 || c == 8) ? 2 : (c == 2 || c == 4 || c == 7) ? 1 : 0;
}
__host__ __device__ constexpr int o3_y(int c) { return 3 - o3_x(c) - o3_z(c); }

// 1-D moments M^e_t about a centre at distance X from P
template <int ORD>
struct Mom1 {
    double m[ORD + 1][ORD + 1];
    __device__ __forceinline__ Mom1(double X, double h)
    {
        const double X2 = X * X;
        m[0][0] = 1.0;
        if constexpr (ORD >= 1) {
            m[1][0] = X;
            m[1][1] = 1.0;
        }
        if constexpr (ORD >= 2) {
            m[2][0] = X2 + h;
            m[2][1] = 2.0 * X;
            m[2][2] = 2.0;
        }
        if constexpr (ORD >= 3) {
            m[3][0] = X * (X2 + 3.0 * h);
            m[3][1] = 3.0 * (X2 + h);
            m[3][2] = 6.0 * X;
            m[3][3] = 6.0;
        }
    }
};

// H^k_tuv, t + u + v <= 2, of the potential polynomial of atom k (phi: its 20 Taylor components) at
// displacement X = P - R_k
__device__ __forceinline__ void potential_hermite(const double *__restrict__ phi, const double (&X)[3], double h,
                                                  double (&H)[10])
{
    const double xx = phi[4], xy = phi[5], xz = phi[6], yy = phi[7], yz = phi[8], zz = phi[9];
    const double lx = xx * X[0] + xy * X[1] + xz * X[2], ly = xy * X[0] + yy * X[1] + yz * X[2],
                 lz = xz * X[0] + yz * X[1] + zz * X[2];
    H[0] = phi[0] + X[0] * (phi[1] + lx) + X[1] * (phi[2] + ly) + X[2] * (phi[3] + lz) + h * (xx + yy + zz);
    H[hidx(1, 0, 0)] = phi[1] + 2.0 * lx;
    H[hidx(0, 1, 0)] = phi[2] + 2.0 * ly;
    H[hidx(0, 0, 1)] = phi[3] + 2.0 * lz;
    H[hidx(2, 0, 0)] = 2.0 * xx;
    H[hidx(0, 2, 0)] = 2.0 * yy;
    H[hidx(0, 0, 2)] = 2.0 * zz;
    H[hidx(1, 1, 0)] = 2.0 * xy;
    H[hidx(1, 0, 1)] = 2.0 * xz;
    H[hidx(0, 1, 1)] = 2.0 * yz;
}

// Block (32, NA): lane = primitive pair, warp = Cartesian component of shell A.  The warps first
// share the pair's setup (1-D Hermite tables per direction, prefactor, potentials) through shared
// memory, then each sweeps the components of shell B, and the sums over the components of A meet
// in shared memory again: one setup and one set of atomics per pair whatever its component count,
// and short chains for a pair of high angular momentum.
// ORD: 2 multipoles to the quadrupole (out: mult), 3 octupoles (out: oct).
template <int LA, int LB, int ORD, bool FOCK, bool PULAY>
struct MomShape {
    static constexpr int NA = ncart(LA), NB = ncart(LB), LBP = PULAY ? LB + 1 : LB;
    static constexpr int TM = LA + LB < ORD ? LA + LB : ORD;  // highest Hermite order that occurs
    static constexpr int ND = nherm(TM);
    static constexpr int NT = 3 * (LA + 1) * (LBP + 1) * (TM + 1);  // table doubles per lane
    static constexpr int NR = ND + (PULAY ? 3 : 0);                 // sums per lane and warp
    static constexpr int NP = (FOCK || PULAY) ? 21 : 1;  // coefficient, H^A + H^B, H^B
    static constexpr int NS = (NT > NA * NR ? NT : NA * NR) + NP;
};

template <int LA, int LB, int ORD, bool MULT, bool FOCK, bool PULAY>
__global__ void __launch_bounds__(32 * ncart(LA))
k_moments(BasisDev bd, int pp_begin, int pp_end, const double *__restrict__ dm, const double *__restrict__ phi,
          double *__restrict__ mult, double *__restrict__ F, double *__restrict__ gqm)
{
    using Sh = MomShape<LA, LB, ORD, FOCK, PULAY>;
    constexpr int NA = Sh::NA, NB = Sh::NB, LBP = Sh::LBP, TM = Sh::TM, ND = Sh::ND, NR = Sh::NR;
    extern __shared__ double sm[][32];
    double(*pairc)[32] = sm + (Sh::NS - Sh::NP);
    auto tab = [](int d, int a, int b, int t) { return ((d * (LA + 1) + a) * (LBP + 1) + b) * (TM + 1) + t; };
    const int lane = threadIdx.x, ia = threadIdx.y;
    const int i = pp_begin + blockIdx.x * 32 + lane;
    const bool active = i < pp_end;
    const uint32_t code = __ldg(bd.pp + (active ? i : pp_end - 1));
    const int s = (int)(code >> 8), ka = (code >> 4) & 15, kb = code & 15;
    const SPair sp = bd.sp[s];
    const int pa = __ldg(bd.shell_off + sp.shA) + ka, pb = __ldg(bd.shell_off + sp.shB) + kb;
    const int atomA = __ldg(bd.shell_atom + sp.shA), atomB = __ldg(bd.shell_atom + sp.shB);
    const double a = __ldg(bd.exps + pa), b = __ldg(bd.exps + pb), ip = 1.0 / (a + b), h = 0.5 * ip;
    double XA[3], XB[3];  // P - A, P - B
    double ab2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double A = bd.qm_xyz[3 * atomA + d], B = bd.qm_xyz[3 * atomB + d];
        const double P = (a * A + b * B) * ip;
        XA[d] = P - A;
        XB[d] = P - B;
        ab2 += (A - B) * (A - B);
    }
    const bool mirror = sp.shA != sp.shB, two = atomA != atomB;

    // setup: tasks 0..2 the tables of one direction, 3 the prefactor, 4 the potentials
    for (int task = ia; task < 5; task += NA) {
        if (task < 3) {
            const double xa = task == 0 ? XA[0] : task == 1 ? XA[1] : XA[2];
            const double xb = task == 0 ? XB[0] : task == 1 ? XB[1] : XB[2];
            // E_0 by its two-term recursion, E_t = h/t (i E^{i-1,j}_{t-1} + j E^{i,j-1}_{t-1})
            double E[LA + 1][LBP + 1][TM + 1];
            E[0][0][0] = 1.0;
#pragma unroll
            for (int k = 0; k <= LA; ++k)
#pragma unroll
                for (int j = 0; j <= LBP; ++j) {
#pragma unroll
                    for (int t = 1; t <= TM; ++t) {
                        double e = 0.0;
                        if (k > 0) e += (double)k * E[k > 0 ? k - 1 : 0][j][t - 1];
                        if (j > 0) e += (double)j * E[k][j > 0 ? j - 1 : 0][t - 1];
                        E[k][j][t] = (k + j > 0) ? (h * (1.0 / t)) * e : 0.0;
                    }
                    double e1 = 0.0;  // E_1 of (k, j), whatever TM
                    if constexpr (TM >= 1) e1 = E[k][j][TM >= 1 ? 1 : 0];
                    else if (j > 0) e1 = h * j * E[k][j > 0 ? j - 1 : 0][0];
                    if (k == 0 && j < LBP) E[0][j < LBP ? j + 1 : 0][0] = xb * E[0][j][0] + e1;
                    if (k < LA) E[k < LA ? k + 1 : 0][j][0] = xa * E[k][j][0] + e1;
                }
#pragma unroll
            for (int k = 0; k <= LA; ++k)
#pragma unroll
                for (int j = 0; j <= LBP; ++j)
#pragma unroll
                    for (int t = 0; t <= TM; ++t) sm[tab(task, k, j, t)][lane] = E[k][j][t];
        } else if (task == 3) {
            const double spp = PI * ip;
            pairc[0][lane] = active ? __ldg(bd.ncoef + pa) * __ldg(bd.ncoef + pb) * exp(-a * b * ip * ab2) * spp * sqrt(spp)
                                    : 0.0;
        } else if constexpr (FOCK || PULAY) {
            double HA[10], HB[10];
            potential_hermite(phi + 20 * (size_t)atomA, XA, h, HA);
            potential_hermite(phi + 20 * (size_t)atomB, XB, h, HB);
#pragma unroll
            for (int k = 0; k < 10; ++k) {
                pairc[1 + k][lane] = HA[k] + HB[k];
                pairc[11 + k][lane] = HB[k];
            }
        }
    }
    __syncthreads();

    const double coef = pairc[0][lane];
    bool take[5], head;
    seg_setup(active ? s : -1 - lane, lane, take, head);
    int a3[3] = {0, 0, 0};
    {
        int k = 0;
#pragma unroll
        for (int x = LA; x >= 0; --x)
#pragma unroll
            for (int y = LA - x; y >= 0; --y, ++k)
                if (k == ia) {
                    a3[0] = x;
                    a3[1] = y;
                    a3[2] = LA - x - y;
                }
    }
    constexpr int NH2 = nherm(TM < 2 ? TM : 2);
    double Hs[10], Hb[10];
    if constexpr (FOCK || PULAY) {
#pragma unroll
        for (int k = 0; k < NH2; ++k) {
            Hs[k] = pairc[1 + k][lane];
            Hb[k] = pairc[11 + k][lane];
        }
    }
    double D[ND], Dd[ND], g[3] = {0.0, 0.0, 0.0}, gd[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < ND; ++k) D[k] = Dd[k] = 0.0;
    bool skew = false;  // a density element differs from its transpose
    const size_t r = sp.aoA + ia;
#pragma unroll 1
    for (int ib = 0; ib < NB; ++ib) {
        int b3[3] = {0, 0, 0};
        {
            int k = 0;
#pragma unroll
            for (int x = LB; x >= 0; --x)
#pragma unroll
                for (int y = LB - x; y >= 0; --y, ++k)
                    if (k == ib) {
                        b3[0] = x;
                        b3[1] = y;
                        b3[2] = LB - x - y;
                    }
        }
        const size_t c = sp.aoB + ib;
        double E[3][TM + 1], gm = 0.0, delta = 0.0;
        if (MULT || PULAY) {
            if (active) {
                gm = dm[c * bd.nao + r];
                delta = dm[r * bd.nao + c] - gm;
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int t = 0; t <= TM; ++t) E[d][t] = sm[tab(d, a3[d], b3[d], t)][lane];
        const bool odd = (MULT || PULAY) && __any_sync(FULL, delta != 0.0);
        skew |= odd;
        if (MULT || PULAY) {
#pragma unroll
            for (int t = 0; t <= TM; ++t) {
                const double gx = gm * E[0][t];
#pragma unroll
                for (int u = 0; u <= TM - t; ++u) {
                    const double gxy = gx * E[1][u];
#pragma unroll
                    for (int v = 0; v <= TM - t - u; ++v) D[hidx(t, u, v)] += gxy * E[2][v];
                }
            }
            if (odd) {
#pragma unroll
                for (int t = 0; t <= TM; ++t)
#pragma unroll
                    for (int u = 0; u <= TM - t; ++u)
#pragma unroll
                        for (int v = 0; v <= TM - t - u; ++v) Dd[hidx(t, u, v)] += delta * E[0][t] * E[1][u] * E[2][v];
            }
        }
        if constexpr (FOCK || PULAY) {
            // sum_tuv E^x_t E^y_u E^z_v H_tuv, innermost direction first
            double hxy[TM + 1][TM + 1], hx[TM + 1], f = 0.0;
#pragma unroll
            for (int t = 0; t <= TM; ++t) {
                hx[t] = 0.0;
#pragma unroll
                for (int u = 0; u <= TM - t; ++u) {
                    hxy[t][u] = 0.0;
#pragma unroll
                    for (int v = 0; v <= TM - t - u; ++v) hxy[t][u] += E[2][v] * Hs[hidx(t, u, v)];
                    hx[t] += E[1][u] * hxy[t][u];
                }
                f += E[0][t] * hx[t];
            }
            if constexpr (FOCK) {
                const double v = seg_reduce(-0.5 * coef * f, take);
                // a shell with itself: one triangle and its mirror, equal bit for bit
                if (head && active && (mirror || ia <= ib)) {
                    atomicAdd(F + r * bd.nao + c, v);
                    if (mirror || ia < ib) atomicAdd(F + c * bd.nao + r, v);
                }
            }
            if constexpr (PULAY) {
                // dE^{ij}_t / dX_AB in each direction
                double dE[3][TM + 1];
#pragma unroll
                for (int d = 0; d < 3; ++d)
#pragma unroll
                    for (int t = 0; t <= TM; ++t) {
                        double e = -2.0 * b * sm[tab(d, a3[d], b3[d] + 1, t)][lane];
                        if (b3[d] > 0) e += (double)b3[d] * sm[tab(d, a3[d], b3[d] - 1, t)][lane];
                        if (t > 0) e += b * ip * E[d][t > 0 ? t - 1 : 0];
                        dE[d][t] = e;
                    }
                double dx = 0.0, dy = 0.0, dz = 0.0;
#pragma unroll
                for (int t = 0; t <= TM; ++t) {
                    double sy = 0.0, sz = 0.0;
#pragma unroll
                    for (int u = 0; u <= TM - t; ++u) {
                        double hz = 0.0;
#pragma unroll
                        for (int v = 0; v <= TM - t - u; ++v) hz += dE[2][v] * Hs[hidx(t, u, v)];
                        sy += dE[1][u] * hxy[t][u];
                        sz += E[1][u] * hz;
                    }
                    dx += dE[0][t] * hx[t];
                    dy += E[0][t] * sy;
                    dz += E[0][t] * sz;
                }
                g[0] += gm * dx;
                g[1] += gm * dy;
                g[2] += gm * dz;
                if (odd) {
#pragma unroll
                    for (int t = 0; t <= TM; ++t)
#pragma unroll
                        for (int u = 0; u <= TM - t; ++u)
#pragma unroll
                            for (int v = 0; v <= TM - t - u; ++v) {
                                const double H = delta * Hb[hidx(t, u, v)];
                                gd[0] += H * dE[0][t] * E[1][u] * E[2][v];
                                gd[1] += H * E[0][t] * dE[1][u] * E[2][v];
                                gd[2] += H * E[0][t] * E[1][u] * dE[2][v];
                            }
                }
            }
        }
    }
    // sums over the components of A (warps 0, 1, 2, as far as there are, need the totals): the
    // density's part, then the antisymmetric rest if there is one
    auto total = [&](double (&d)[ND], double (&v)[3]) {
        if constexpr (NA > 1) {
            __syncthreads();
#pragma unroll
            for (int k = 0; k < ND; ++k) sm[ia * NR + k][lane] = d[k];
            if constexpr (PULAY) {
#pragma unroll
                for (int k = 0; k < 3; ++k) sm[ia * NR + ND + k][lane] = v[k];
            }
            __syncthreads();
            if (ia >= 3) return;
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                double x = 0.0;
                for (int w = 0; w < NA; ++w) x += sm[w * NR + k][lane];
                if (k < ND) d[k < ND ? k : 0] = x;
                else v[k < ND ? 0 : k - ND] = x;
            }
        }
    };
    const bool rest = __syncthreads_or(skew);
    total(D, g);
    if (rest) total(Dd, gd);
    if (ia >= 3) return;

    if constexpr (MULT) {
        // about A from D (warp 0), about B from D plus the antisymmetric rest (warp 1, or 0 again)
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            if (ia != (NA > 1 ? side : 0)) continue;
            if (side && rest) {
#pragma unroll
                for (int k = 0; k < ND; ++k) D[k] += Dd[k];
            }
            const Mom1<ORD> mx(side ? XB[0] : XA[0], h), my(side ? XB[1] : XA[1], h), mz(side ? XB[2] : XA[2], h);
            const int at = side ? atomB : atomA;
#pragma unroll
            for (int k = 0; k < 10; ++k) {
                const int ox = ORD == 2 ? op_x(k) : o3_x(k), oy = ORD == 2 ? op_y(k) : o3_y(k),
                          oz = ORD == 2 ? op_z(k) : o3_z(k);
                double m = 0.0;
#pragma unroll
                for (int t = 0; t <= ox; ++t)
#pragma unroll
                    for (int u = 0; u <= oy; ++u)
#pragma unroll
                        for (int v = 0; v <= oz; ++v)
                            if (t + u + v <= TM)
                                m += mx.m[ox][t] * my.m[oy][u] * mz.m[oz][v] * D[t + u + v <= TM ? hidx(t, u, v) : 0];
                const double v = seg_reduce(side && !mirror ? 0.0 : -coef * m, take);
                if (head && active && (!side || mirror)) atomicAdd(mult + 10 * at + k, v);
            }
        }
    }
    if constexpr (PULAY) {
        if (ia != (NA > 1 ? 2 : 0)) return;
        double HA[10], HB[10], K[10];
        potential_hermite(phi + 20 * (size_t)atomA, XA, h, HA);
        potential_hermite(phi + 20 * (size_t)atomB, XB, h, HB);
        if (MULT && NA == 1 && rest) {  // this warp's D was B's
#pragma unroll
            for (int k = 0; k < ND; ++k) D[k] -= Dd[k];
        }
        // D (b/p H^A - a/p H^B) raised once per direction; the antisymmetric rest only meets H^B
#pragma unroll
        for (int k = 0; k < 10; ++k) K[k] = b * ip * HA[k] - a * ip * HB[k];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double v = -g[d], w = -gd[d];
#pragma unroll
            for (int k = 0; k < (TM >= 1 ? 4 : 1); ++k) {
                const int t = k == 1, u = k == 2, z = k == 3;
                const int up = hidx(t + (d == 0), u + (d == 1), z + (d == 2));
                v += D[hidx(t, u, z)] * K[up];
                if (rest) w -= Dd[hidx(t, u, z)] * (a * ip * HB[up]);
            }
            v = seg_reduce(two ? coef * (v + w) : 0.0, take);
            if (head && active && two) {
                atomicAdd(gqm + 3 * atomA + d, v);
                atomicAdd(gqm + 3 * atomB + d, -v);
            }
        }
    }
}

template <int LA, int LB, int ORD, bool MULT, bool FOCK, bool PULAY>
static cudaError_t launch_mom(const BasisDev &bd, int pp_begin, int pp_end, const double *dm, const double *phi,
                              double *mult, double *F, double *gqm, cudaStream_t st)
{
    const size_t smem = (size_t)MomShape<LA, LB, ORD, FOCK, PULAY>::NS * 32 * sizeof(double);
    auto kern = k_moments<LA, LB, ORD, MULT, FOCK, PULAY>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<(pp_end - pp_begin + 31) / 32, dim3(32, ncart(LA)), smem, st>>>(bd, pp_begin, pp_end, dm, phi, mult, F, gqm);
    return cudaGetLastError();
}

template <int LA, int LB>
struct Octupoles {
    static cudaError_t run(const BasisDev &bd, int pp_begin, int pp_end, const double *dm, double *oct,
                           cudaStream_t st)
    {
        return launch_mom<LA, LB, 3, true, false, false>(bd, pp_begin, pp_end, dm, nullptr, oct, nullptr, nullptr, st);
    }
};

cudaError_t launch_octupoles(const BasisDev &b, int cls, int pp_begin, int pp_end, const double *dm, double *oct,
                             cudaStream_t st)
{
    if (pp_end <= pp_begin) return cudaSuccess;
    return dispatch_class<Octupoles>(cls, b, pp_begin, pp_end, dm, oct, st);
}

template <int LA, int LB>
struct Moments {
    static cudaError_t run(const BasisDev &bd, int pp_begin, int pp_end, const double *dm, const double *phi,
                           double *mult, double *F, double *gqm, int mode, cudaStream_t st)
    {
        switch (mode) {
        case MOM_MULT: return launch_mom<LA, LB, 2, true, false, false>(bd, pp_begin, pp_end, dm, phi, mult, F, gqm, st);
        case MOM_MULT | MOM_FOCK:
            return launch_mom<LA, LB, 2, true, true, false>(bd, pp_begin, pp_end, dm, phi, mult, F, gqm, st);
        case MOM_MULT | MOM_PULAY:
            return launch_mom<LA, LB, 2, true, false, true>(bd, pp_begin, pp_end, dm, phi, mult, F, gqm, st);
        case MOM_PULAY: return launch_mom<LA, LB, 2, false, false, true>(bd, pp_begin, pp_end, dm, phi, mult, F, gqm, st);
        case MOM_PULAY | MOM_FOCK:
            return launch_mom<LA, LB, 2, false, true, true>(bd, pp_begin, pp_end, dm, phi, mult, F, gqm, st);
        default: return cudaErrorInvalidValue;
        }
    }
};

cudaError_t launch_moments(const BasisDev &b, int cls, int pp_begin, int pp_end, const double *dm,
                           const double *phi, double *mult, double *F, double *gqm, int mode, cudaStream_t st)
{
    if (pp_end <= pp_begin) return cudaSuccess;
    return dispatch_class<Moments>(cls, b, pp_begin, pp_end, dm, phi, mult, F, gqm, mode, st);
}

}  // namespace qmmm
