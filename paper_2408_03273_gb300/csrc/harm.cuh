// harm.cuh -- Hermite integrals in solid harmonics.
//
// A Hermite tensor of order N is x^t y^u z^v applied as a differential operator, and every
// homogeneous polynomial splits into harmonic ones: x^t y^u z^v = sum_k r^2k sum_m t_klm Y_lm with
// l = N - 2k.  On the radial function B(r) = F_0(rho r^2) of the region-I integrals the two factors
// act separately (Hobson's theorem for a harmonic polynomial, and the Laplacian of erf(r)/r, a
// Gaussian):
//   Y_lm(d) B          = (-2 rho)^l F_l(T) Y_lm(P - C),                            T = rho |P - C|^2,
//   Y_lm(d) lap^k B    = (-2 rho)^(l+k) p_kl(T) e^-T Y_lm(P - C),                  k >= 1,
//   p_1l = 1,  p_2l = 3 + 2l - 2T,  p_3l = p_30 - p_30' ... (p_k,l+1 = p_kl - p_kl').
// So a (primitive pair, charge) needs the (L+1)^2 solid harmonics and one factor per l instead of
// the C(L+3,3) Hermite tensors and their C(L+4,4)-term recursion, and the k >= 1 terms vanish with
// e^-T: they are formed only for charges close to the pair (a sixth of the (warp, charge) steps of
// the benchmark's active sites).  The change of basis happens once per pair.
//
// Units.  With sqrt(kappa / (p + kappa)) = sqrt(rho / p) in front, B's factors in units of
// sqrt(pi) / (2 sqrt(p)) are
//   k = 0:  (-1)^l (2l-1)!! F'_l,      F'_l = 2 / sqrt(pi) rho^(l+1/2) 2^l F_l / (2l-1)!!  -> r^-(2l+1),
//   k >= 1: (-2)^(l+k) p_kl E_(l+k),   E_j = 2 / sqrt(pi) rho^(j+1/2) e^-T,
// the constants folded into the change of basis: for a distant charge the factors are those of a
// point charge, with neither rho nor T in them, whatever its width.
#pragma once
#include "device_common.cuh"

namespace qmmm {

constexpr int HARM_L = 2 * LMAX;  // highest order of a sweep's Hermite tensors

// Solid harmonics of order l: index l^2 (m = 0), l^2 + 2m - 1 (cosine), l^2 + 2m (sine),
// normalised to leading coefficient 1 in z: Y_lm = z Y_l-1,m - c r^2 Y_l-2,m with
// c = ((l-1)^2 - m^2) / (4 (l-1)^2 - 1), started from Y_mm = Re, Im (x + iy)^m.
__host__ __device__ constexpr double harm_c(int l, int m)  // coefficient that gives Y_l+1 from Y_l, Y_l-1
{
    return (double)(l * l - m * m) / (double)(4 * l * l - 1);
}
// Storage of the harmonic components of an order-L Hermite tensor: power k of the Laplacian, then
// the harmonic index of order l <= L - 2k; nherm(L) in all.
__host__ __device__ constexpr int harm_off(int L, int k)
{
    int o = 0;
    for (int i = 0; i < k; ++i) o += (L - 2 * i + 1) * (L - 2 * i + 1);
    return o;
}

struct HarmEntry {
    double c;                   // t_klm times the constant of the radial factor of (k, l)
    unsigned char herm, k, lm;  // Hermite index, Laplacian power, harmonic index
};
struct HarmGrad {
    double c;
    unsigned char dir, lm, lm1;  // d Y_lm / d(dir) += c Y_lm1
};
constexpr int HARM_NT = 362, HARM_NG = 158;
struct HarmTables {
    HarmEntry t[HARM_NT] = {};
    HarmGrad g[HARM_NG] = {};
    int nt = 0, ng = 0;
    int tend[HARM_L + 1] = {};  // entries of Hermite orders <= N
    int gend[HARM_L + 1] = {};  // gradient entries of harmonics l <= N
};

// Coefficients by the Fischer product <p, q> = p(d) q, under which the components r^2k Y_lm are
// orthogonal: t = <x^t y^u z^v, r^2k Y_lm> / <r^2k Y_lm, r^2k Y_lm>.
constexpr HarmTables make_harm_tables()
{
    constexpr int ND = (HARM_L + 1) * (HARM_L + 2) / 2;  // monomials of the highest degree
    HarmTables H;
    double y[(HARM_L + 1) * (HARM_L + 1)][ND] = {};
    // monomial x^(d-b) y^(b-v) z^v of degree d: index b(b+1)/2 + v, b = u + v
    double fact[HARM_L + 1] = {1.0};
    for (int i = 1; i <= HARM_L; ++i) fact[i] = i * fact[i - 1];
    y[0][0] = 1.0;
    for (int l = 1; l <= HARM_L; ++l) {
        for (int m = 0; m <= l; ++m)
            for (int s = 0; s < (m ? 2 : 1); ++s) {
                double *out = y[l * l + (m ? 2 * m - 1 + s : 0)];
                if (m == l) {  // (x + iy)^l = (x + iy) (x + iy)^(l-1)
                    const double *re = y[(l - 1) * (l - 1) + (l > 1 ? 2 * l - 3 : 0)];
                    const double *im = y[(l - 1) * (l - 1) + (l > 1 ? 2 * l - 2 : 0)];
                    for (int b = 0, i = 0; b < l; ++b)
                        for (int v = 0; v <= b; ++v, ++i) {
                            const double r = re[i], q = l > 1 ? im[i] : 0.0;
                            out[i] += s ? q : r;                          // times x
                            out[(b + 1) * (b + 2) / 2 + v] += s ? r : -q;  // times y
                        }
                } else {
                    const double *p1 = y[(l - 1) * (l - 1) + (m ? 2 * m - 1 + s : 0)];
                    for (int b = 0, i = 0; b < l; ++b)
                        for (int v = 0; v <= b; ++v, ++i) out[(b + 1) * (b + 2) / 2 + v + 1] += p1[i];  // times z
                    if (m <= l - 2) {
                        const double *p2 = y[(l - 2) * (l - 2) + (m ? 2 * m - 1 + s : 0)];
                        const double c = harm_c(l - 1, m);
                        for (int b = 0, i = 0; b < l - 1; ++b)
                            for (int v = 0; v <= b; ++v, ++i) {  // times r^2
                                out[i] -= c * p2[i];
                                out[(b + 2) * (b + 3) / 2 + v] -= c * p2[i];
                                out[(b + 2) * (b + 3) / 2 + v + 2] -= c * p2[i];
                            }
                    }
                }
            }
    }
    for (int N = 0; N <= HARM_L; ++N) {
        for (int k = 0; 2 * k <= N; ++k) {
            const int l = N - 2 * k;
            for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) {
                double p[ND] = {};
                for (int i = 0; i < (l + 1) * (l + 2) / 2; ++i) p[i] = y[lm][i];
                for (int r = 0; r < k; ++r) {  // times r^2, in place from the top
                    double q[ND] = {};
                    const int d = l + 2 * r;
                    for (int b = 0, i = 0; b <= d; ++b)
                        for (int v = 0; v <= b; ++v, ++i) {
                            q[i] += p[i];
                            q[(b + 2) * (b + 3) / 2 + v] += p[i];
                            q[(b + 2) * (b + 3) / 2 + v + 2] += p[i];
                        }
                    for (int i = 0; i < ND; ++i) p[i] = q[i];
                }
                double norm = 0.0;
                for (int b = 0, i = 0; b <= N; ++b)
                    for (int v = 0; v <= b; ++v, ++i) norm += fact[N - b] * fact[b - v] * fact[v] * p[i] * p[i];
                for (int b = 0, i = 0; b <= N; ++b)
                    for (int v = 0; v <= b; ++v, ++i)
                        if (p[i] > 1e-12 || p[i] < -1e-12) {
                            HarmEntry &e = H.t[H.nt++];
                            // with the constant part of the radial factor
                            double rad = 1.0;
                            for (int j = 1; k == 0 && j <= l; ++j) rad *= -(2 * j - 1);
                            for (int j = 0; k > 0 && j < l + k; ++j) rad *= -2.0;
                            e.c = rad * fact[N - b] * fact[b - v] * fact[v] * p[i] / norm;
                            e.herm = (unsigned char)hidx(N - b, b - v, v);
                            e.k = (unsigned char)k;
                            e.lm = (unsigned char)lm;
                        }
            }
        }
        H.tend[N] = H.nt;
    }
    for (int l = 0; l <= HARM_L; ++l) {
        for (int lm = l * l; l > 0 && lm < (l + 1) * (l + 1); ++lm)
            for (int dir = 0; dir < 3; ++dir)
                for (int lm1 = (l - 1) * (l - 1); lm1 < l * l; ++lm1) {
                    double s = 0.0, norm = 0.0;
                    for (int b = 0, i = 0; b <= l - 1; ++b)
                        for (int v = 0; v <= b; ++v, ++i) {
                            const int t = l - 1 - b, u = b - v;
                            const double w = fact[t] * fact[u] * fact[v] * y[lm1][i];
                            const int up = dir == 0 ? i : (b + 1) * (b + 2) / 2 + v + (dir == 2 ? 1 : 0);
                            const double mult = dir == 0 ? t + 1 : dir == 1 ? u + 1 : v + 1;
                            s += w * mult * y[lm][up];
                            norm += w * y[lm1][i];
                        }
                    s /= norm;
                    if (s > 1e-12 || s < -1e-12) {
                        HarmGrad &e = H.g[H.ng++];
                        e.c = s;
                        e.dir = (unsigned char)dir;
                        e.lm = (unsigned char)lm;
                        e.lm1 = (unsigned char)lm1;
                    }
                }
        H.gend[l] = H.ng;
    }
    return H;
}


#ifdef __CUDACC__
static __constant__ HarmTables HT = make_harm_tables();
#else
static const HarmTables HT = make_harm_tables();
#endif

// Above this T the relative weight of e^-T in F_M (the regularised upper gamma function
// Q(M + 1/2, T)) is below 1e-17, and so is that of the Gaussian (k >= 1) terms.
__host__ __device__ constexpr double harm_tmax(int M)
{
    constexpr double T[9] = {37.0, 41.5, 45.0, 48.0, 51.0, 53.5, 56.0, 58.5, 59.9};
    return T[M];
}

// 1 / sqrt(r2): hardware estimate (about 2^-20) and one third-order Householder step,
// y (1 + h/2 + 3 h^2/8) with h = 1 - r2 y^2
__host__ __device__ __forceinline__ double harm_rsqrt(double r2)
{
    double y;
#ifdef __CUDA_ARCH__
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(r2));
#else
    y = (float)(1.0 / sqrt(r2));
#endif
    const double h = fma(-r2 * y, y, 1.0);
    return fma(y * h, fma(h, 0.375, 0.5), y);
}

// A charge is distant if the high word of r2 exceeds that of the limit: the words order
// non-negative doubles (a NaN counts as distant and never indexes the Boys table), and the integer
// comparison stays off the FP64 pipe.
__device__ __forceinline__ bool harm_far(double r2, double limit)
{
    return (unsigned)__double2hiint(r2) > (unsigned)__double2hiint(limit);
}

// F'_m, m = 0..M, and E_0 (0 for a distant charge) of a pair with rho, c0 = 2 sqrt(rho / pi);
// far: T = rho r2 above harm_tmax(M).  F^_m = 2^m F_m / (2m-1)!! by the table's Taylor expansion and
// F^_(m-1) = T F^_m + e^-T 2^(m-1) / (2m-1)!!.
template <int M>
__host__ __device__ __forceinline__ void boys_hat(bool far, double r2, double rho, double c0, double (&F)[M + 1],
                                                  double &E0, const double *__restrict__ tab)
{
    constexpr double TOP[9] = {1.0, 2.0, 4.0 / 3, 8.0 / 15, 16.0 / 105, 32.0 / 945, 64.0 / 10395, 128.0 / 135135,
                               256.0 / 2027025};  // 2^M / (2M-1)!!
    if (!far) {
        const double T = rho * r2;
#ifdef __CUDA_ARCH__
        const int k = __double2int_rn(T * BOYS_INV_STEP);
#else
        const int k = (int)(T * BOYS_INV_STEP + 0.5);
#endif
        const double x = (double)k * BOYS_STEP - T;  // -(T - T_k)
        const double2 *row = reinterpret_cast<const double2 *>(tab + ((size_t)M * BOYS_NROW_D + k) * BOYS_ROW_D);
        const double2 c01 = row[0], c23 = row[1], c45 = row[2], c6e = row[3];
        double f = fma(c6e.x, x, c45.y);
        f = fma(f, x, c45.x);
        f = fma(f, x, c23.y);
        f = fma(f, x, c23.x);
        f = fma(f, x, c01.y);
        f = fma(f, x, c01.x);
        F[M] = TOP[M] * f;
        // e^-T = e^-T_k e^x, |x| <= 0.05: 8-term Taylor series of e^x
        const double ex = 1.0 + x * (1.0 + x * (0.5 + x * (1.0 / 6.0 + x * (1.0 / 24.0 + x * (1.0 / 120.0 +
                          x * (1.0 / 720.0 + x * (1.0 / 5040.0)))))));
        const double e = c6e.y * ex;
#pragma unroll
        for (int m = M; m > 0; --m) F[m - 1] = fma(T, F[m], e * (TOP[m] * 0.5));
        double s = c0;
#pragma unroll
        for (int m = 0; m <= M; ++m) {
            F[m] *= s;
            s *= rho;
        }
        E0 = c0 * e;
    } else {
        const double y = harm_rsqrt(r2), y2 = y * y;
        F[0] = y;
#pragma unroll
        for (int m = 0; m < M; ++m) F[m + 1] = F[m] * y2;
        E0 = 0.0;
    }
}

// visit(l, index, Y_lm(X, Y, Z)) for every harmonic of order <= L, column by column in m so that
// only two members of a column are live
template <int L, typename V>
__host__ __device__ __forceinline__ void harm_walk(double X, double Y, double Z, double r2, V visit)
{
    double re = 1.0, im = 0.0;
#pragma unroll
    for (int m = 0; m <= L; ++m) {
        if (m == 1) {
            re = X;
            im = Y;
        } else if (m > 1) {
            const double t = fma(X, re, -(Y * im));
            im = fma(X, im, Y * re);
            re = t;
        }
        double c1 = re, s1 = im, c0 = 0.0, s0 = 0.0;
#pragma unroll
        for (int l = m; l <= L; ++l) {
            visit(l, l * l + (m ? 2 * m - 1 : 0), c1);
            if (m) visit(l, l * l + 2 * m, s1);
            if (l == L) continue;
            if (l == m) {
                c0 = c1;
                s0 = s1;
                c1 = m ? Z * c1 : Z;
                s1 = Z * s1;
            } else {
                const double w = harm_c(l, m) * r2;
                const double c = fma(Z, c1, (l == 1 && m == 0) ? -w : -(w * c0)), s = fma(Z, s1, -(w * s0));
                c0 = c1;
                s0 = s1;
                c1 = c;
                s1 = s;
            }
        }
    }
}

// radial polynomials p_kl(T) of the Gaussian terms, k = 2, 3
__host__ __device__ __forceinline__ double harm_p2(int l, double T) { return fma(-2.0, T, 3.0 + 2 * l); }
__host__ __device__ __forceinline__ double harm_p3(int l, double T)
{
    return l == 0 ? fma(fma(4.0, T, -20.0), T, 15.0) : fma(fma(4.0, T, -28.0), T, 35.0);
}

// The factors of one charge in the sums S_klm += q (radial factor) Y_lm; NEAR: with the Gaussian
// terms, E[j] = E_j.
template <int L, bool NEAR>
struct HarmSum {
    double qF[L + 1], qE[L + 1], T;
    __host__ __device__ __forceinline__ HarmSum(const double *F, const double *E, double T_, double q) : T(T_)
    {
#pragma unroll
        for (int l = 0; l <= L; ++l) qF[l] = q * F[l];
        if constexpr (NEAR) {
#pragma unroll
            for (int j = 1; j < L; ++j) qE[j] = q * E[j];
        }
    }
    __host__ __device__ __forceinline__ void add(double (&S)[nherm(L)], int l, int i, double y) const
    {
        S[i] = i == 0 ? S[i] + qF[0] : fma(qF[l], y, S[i]);
        if constexpr (NEAR) {
            if (l <= L - 2) S[harm_off(L, 1) + i] = fma(qE[l + 1], y, S[harm_off(L, 1) + i]);
            if (l <= L - 4) S[harm_off(L, 2) + i] = fma(qE[l + 2] * harm_p2(l, T), y, S[harm_off(L, 2) + i]);
            if (l <= L - 6) S[harm_off(L, 3) + i] = fma(qE[l + 3] * harm_p3(l, T), y, S[harm_off(L, 3) + i]);
        }
    }
};
// E_1 .. E_L from E_0
template <int L>
__host__ __device__ __forceinline__ void harm_powers(double E0, double rho, double (&E)[L + 1])
{
    E[0] = E0;
#pragma unroll
    for (int j = 1; j <= L; ++j) E[j] = E[j - 1] * rho;
}

// One charge into the sums S: its harmonic components at the pair (V sweep)
template <int L, bool NEAR>
__host__ __device__ __forceinline__ void harm_add(double (&S)[nherm(L)], const double *F, double E0, double rho, double q,
                                                  double X, double Y, double Z, double r2)
{
    double E[L + 1];
    if constexpr (NEAR) harm_powers<L>(E0, rho, E);
    const HarmSum<L, NEAR> s(F, E, NEAR ? rho * r2 : 0.0, q);
    harm_walk<L>(X, Y, Z, r2, [&](int l, int i, double y) { s.add(S, l, i, y); });
}
// the same for a charge distant from every pair of the warp: factors q r^-(2l+1)
template <int L>
__host__ __device__ __forceinline__ void harm_add_far(double (&S)[nherm(L)], double q, double X, double Y, double Z,
                                                      double r2)
{
    const double y = harm_rsqrt(r2), y2 = y * y;
    double qF[L + 1];
    qF[0] = q * y;
#pragma unroll
    for (int l = 1; l <= L; ++l) qF[l] = qF[l - 1] * y2;
    harm_walk<L>(X, Y, Z, r2, [&](int l, int i, double v) { S[i] = i == 0 ? fma(q, y, S[i]) : fma(qF[l], v, S[i]); });
}

// components of the gradient arrays: per Laplacian power k the harmonics of order l <= L - 2k - 1
__host__ __device__ constexpr int hgrad_off(int L, int k)
{
    int o = 0;
    for (int i = 0; i < k; ++i) o += L > 2 * i ? (L - 2 * i) * (L - 2 * i) : 0;
    return o;
}
__host__ __device__ constexpr int nhgrad(int L) { return hgrad_off(L, L / 2 + 1); }

// e0 = sum M_klm (radial) Y_lm, the value of a pair's Hermite multipole at a charge, and its
// gradient with respect to P - C; the same harmonics add the charge to the sums S (harm_add).  Not
// NEAR: the charge is distant from every pair of the warp, F'_(l+1) = F'_l / r2 =: F'_l y2.
template <int L, bool NEAR>
__host__ __device__ __forceinline__ void harm_eval(const double (&M)[nherm(L)], const double (&Nx)[nhgrad(L) + 1],
                                                   const double (&Ny)[nhgrad(L) + 1], const double (&Nz)[nhgrad(L) + 1],
                                                   const double *F, double E0, double rho, double y2, double X, double Y,
                                                   double Z, double r2, double q, double (&S)[nherm(L)], double &e0,
                                                   double &ex, double &ey, double &ez)
{
    double E[L + 1];
    if constexpr (NEAR) harm_powers<L>(E0, rho, E);
    const double T = NEAR ? rho * r2 : 0.0;
    const HarmSum<L, NEAR> s(F, E, T, q);
    // per l: value and gradient sums of the Laplacian powers k = 0, 1, 2
    double h[L + 1], kx[L + 1], ky[L + 1], kz[L + 1];
    double h1[L + 1], x1[L + 1], y1[L + 1], z1[L + 1], h2[L + 1], x2[L + 1], y2k[L + 1], z2[L + 1];
#pragma unroll
    for (int l = 0; l <= L; ++l)
        h[l] = kx[l] = ky[l] = kz[l] = h1[l] = x1[l] = y1[l] = z1[l] = h2[l] = x2[l] = y2k[l] = z2[l] = 0.0;
    harm_walk<L>(X, Y, Z, r2, [&](int l, int i, double y) {
        s.add(S, l, i, y);
        h[l] = i == 0 ? M[0] : fma(M[i], y, h[l]);
        if (l < L) {
            kx[l + 1] = i == 0 ? Nx[i] : fma(Nx[i], y, kx[l + 1]);
            ky[l + 1] = i == 0 ? Ny[i] : fma(Ny[i], y, ky[l + 1]);
            kz[l + 1] = i == 0 ? Nz[i] : fma(Nz[i], y, kz[l + 1]);
        }
        if constexpr (NEAR) {
            if (l <= L - 2) h1[l] = fma(M[harm_off(L, 1) + i], y, h1[l]);
            if (l <= L - 3) {
                const int j = hgrad_off(L, 1) + i;
                x1[l + 1] = fma(Nx[j], y, x1[l + 1]);
                y1[l + 1] = fma(Ny[j], y, y1[l + 1]);
                z1[l + 1] = fma(Nz[j], y, z1[l + 1]);
            }
            if (l <= L - 4) h2[l] = fma(M[harm_off(L, 2) + i], y, h2[l]);
            if (l <= L - 5) {
                const int j = hgrad_off(L, 2) + i;
                x2[l + 1] = fma(Nx[j], y, x2[l + 1]);
                y2k[l + 1] = fma(Ny[j], y, y2k[l + 1]);
                z2[l + 1] = fma(Nz[j], y, z2[l + 1]);
            }
        }
    });
    // e = sum_l F'_l k_l - X sum_l (2l+1) F'_(l+1) h_l (minus sign: the constants' (-1)^l)
    double w;
    e0 = F[0] * h[0];
    w = NEAR ? F[1] * h[0] : e0;
    ex = ey = ez = 0.0;
#pragma unroll
    for (int l = 1; l <= L; ++l) {
        if constexpr (NEAR) {
            e0 = fma(F[l], h[l], e0);
            w = fma((2 * l + 1) * F[l + 1], h[l], w);
        } else {
            const double t = F[l] * h[l];
            e0 += t;
            w = fma((double)(2 * l + 1), t, w);
        }
        ex = fma(F[l], kx[l], ex);
        ey = fma(F[l], ky[l], ey);
        ez = fma(F[l], kz[l], ez);
    }
    if constexpr (!NEAR) w *= y2;
    if constexpr (NEAR) {
        double w2 = 0.0;  // Gaussian terms of sum_kl E_(l+k+1) p_k,l+1 h_kl
#pragma unroll
        for (int l = 0; l <= L - 2; ++l) {
            e0 = fma(E[l + 1], h1[l], e0);
            w2 = fma(E[l + 2], h1[l], w2);
            if (l > 0) {
                ex = fma(E[l + 1], x1[l], ex);
                ey = fma(E[l + 1], y1[l], ey);
                ez = fma(E[l + 1], z1[l], ez);
            }
            if (l <= L - 4) {
                const double p = E[l + 2] * harm_p2(l, T);
                e0 = fma(p, h2[l], e0);
                w2 = fma(E[l + 3 > L ? L : l + 3] * harm_p2(l + 1, T), h2[l], w2);
                if (l > 0) {
                    ex = fma(p, x2[l], ex);
                    ey = fma(p, y2k[l], ey);
                    ez = fma(p, z2[l], ez);
                }
            }
        }
        if constexpr (L >= 6) {
            const double m3 = M[harm_off(L, 3)];
            e0 = fma(E[3] * harm_p3(0, T), m3, e0);
            w2 = fma(E[4] * harm_p3(1, T), m3, w2);
        }
        w = fma(2.0, w2, w);
    }
    ex = fma(-X, w, ex);
    ey = fma(-Y, w, ey);
    ez = fma(-Z, w, ez);
}

// gradient coefficients: sum_lm M_klm d Y_lm / da = sum N^a_k,lm1 Y_lm1
template <int L>
__device__ __forceinline__ void harm_grad(const double (&M)[nherm(L)], double (&Nx)[nhgrad(L) + 1],
                                                   double (&Ny)[nhgrad(L) + 1], double (&Nz)[nhgrad(L) + 1])
{
    double in[nherm(L)], out[3][nhgrad(L) + 1];
#pragma unroll
    for (int i = 0; i < nherm(L); ++i) in[i] = M[i];
    for (int i = 0; i <= nhgrad(L); ++i) out[0][i] = out[1][i] = out[2][i] = 0.0;
#pragma unroll 1
    for (int k = 0; 2 * k < L; ++k)
#pragma unroll 1
        for (int i = 0; i < HT.gend[L - 2 * k]; ++i) {
            const HarmGrad &g = HT.g[i];
            out[g.dir][hgrad_off(L, k) + g.lm1] += g.c * in[harm_off(L, k) + g.lm];
        }
#pragma unroll
    for (int i = 0; i <= nhgrad(L); ++i) {
        Nx[i] = out[0][i];
        Ny[i] = out[1][i];
        Nz[i] = out[2][i];
    }
}

}  // namespace qmmm
