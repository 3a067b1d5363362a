"""The solid-harmonic form of the Hermite integrals (csrc/harm.cuh) against the Hermite recursion in
extended precision, on the CPU: the header's host code, compiled by nvcc, no GPU call.

Tolerance: the Boys table's Taylor remainder, (0.05)^7 / 7! F_(M+7) / F_M <= 1.5e-13 * 0.45, and
rounding (a few 1e-15) over the change of basis, relative to the largest component of an order (of
the summed magnitudes for the contracted value and gradient): 1e-13.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_03273_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "harm.cuh"
using namespace qmmm;
typedef long double ld;
static const HarmTables H = make_harm_tables();
static void boys(ld T, int M, ld *F)
{
    const ld e = expl(-T);
    if (T < 70) {
        ld term = 1.0L / (2 * M + 1), s = term;
        for (int i = 1; term > 1e-24L * s; ++i) s += term *= 2 * T / (2 * M + 2 * i + 1);
        F[M] = e * s;
        for (int m = M; m > 0; --m) F[m - 1] = (2 * T * F[m] + e) / (2 * m - 1);
    } else {
        F[0] = sqrtl(acosl(-1.0L) / T) / 2 * erfl(sqrtl(T));
        for (int m = 0; m < M; ++m) F[m + 1] = ((2 * m + 1) * F[m] - e) / (2 * T);
    }
}
static void hermite(int L, ld rho, const double *d, ld *R)
{
    ld F[16];
    boys(rho * ((ld)d[0] * d[0] + (ld)d[1] * d[1] + (ld)d[2] * d[2]), L, F);
    for (int n = L; n >= 0; --n) {
        for (int k = L - n; k >= 1; --k)
            for (int t = k; t >= 0; --t)
                for (int u = k - t; u >= 0; --u) {
                    const int v = k - t - u, a = t ? 0 : u ? 1 : 2, p = a == 0 ? t : a == 1 ? u : v;
                    ld r = d[a] * R[hidx(t - (a == 0), u - (a == 1), v - (a == 2))];
                    if (p > 1) r += (p - 1) * R[hidx(t - 2 * (a == 0), u - 2 * (a == 1), v - 2 * (a == 2))];
                    R[hidx(t, u, v)] = r;
                }
        R[0] = powl(-2 * rho, n) * F[n];
    }
}
static std::vector<double> tab;
static double worst = 0;
static void see(ld got, ld ref, ld scale, int L, const char *what)
{
    const double e = scale > 0 ? (double)(fabsl(got - ref) / scale) : (double)fabsl(got);
    if (!(e <= worst)) worst = e;
    if (!(e <= 1e-13)) {
        printf("L=%d %s: got %Lg ref %Lg scale %Lg\n", L, what, got, ref, scale);
        exit(1);
    }
}
template <int L>
static void one(double rho, const double *d, double q)
{
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], T = rho * r2, c0 = sqrt(rho) / HALF_SQRT_PI;
    ld R[286];
    hermite(L + 1, rho, d, R);
    double F[L + 2], E0, D[nherm(L)], S[nherm(L)] = {}, S2[nherm(L)] = {}, M[nherm(L)] = {}, N[3][nhgrad(L) + 1] = {};
    const bool far = T > harm_tmax(L + 1);
    boys_hat<L + 1>(far, r2, rho, c0, F, E0, tab.data());
    if (far) harm_add_far<L>(S, q, d[0], d[1], d[2], r2);
    else harm_add<L, true>(S, F, E0, rho, q, d[0], d[1], d[2], r2);
    const ld unit = 1 / (ld)c0;
    ld W[nherm(L)] = {};
    for (int i = 0; i < nherm(L); ++i) D[i] = drand48() - 0.5;
    for (int i = 0; i < H.tend[L]; ++i) {
        const int j = harm_off(L, H.t[i].k) + H.t[i].lm;
        W[H.t[i].herm] += unit * H.t[i].c * S[j];
        M[j] += (double)unit * H.t[i].c * D[H.t[i].herm];
    }
    for (int k = 0; 2 * k < L; ++k)
        for (int i = 0; i < H.gend[L - 2 * k]; ++i)
            N[H.g[i].dir][hgrad_off(L, k) + H.g[i].lm1] += H.g[i].c * M[harm_off(L, k) + H.g[i].lm];
    for (int n = 0; n <= L; ++n) {
        ld top = 0;
        for (int i = nherm(n - 1); i < nherm(n); ++i) top = fmaxl(top, fabsl(q * R[i]));
        for (int i = nherm(n - 1); i < nherm(n); ++i) see(W[i], q * R[i], top, L, "sum");
    }
    double e0, ex, ey, ez;
    if (far) harm_eval<L, false>(M, N[0], N[1], N[2], F, 0.0, 0.0, F[1] / F[0], d[0], d[1], d[2], r2, q, S2, e0, ex, ey, ez);
    else harm_eval<L, true>(M, N[0], N[1], N[2], F, E0, rho, 0.0, d[0], d[1], d[2], r2, q, S2, e0, ex, ey, ez);
    ld v = 0, va = 0, g[3] = {}, ga = 0;
    for (int t = 0; t <= L; ++t)
        for (int u = 0; t + u <= L; ++u)
            for (int w = 0; t + u + w <= L; ++w) {
                const ld c = D[hidx(t, u, w)];
                const ld x[4] = {c * R[hidx(t, u, w)], c * R[hidx(t + 1, u, w)], c * R[hidx(t, u + 1, w)], c * R[hidx(t, u, w + 1)]};
                v += x[0];
                va += fabsl(x[0]);
                for (int a = 0; a < 3; ++a) g[a] += x[a + 1], ga += fabsl(x[a + 1]);
            }
    see(e0, v, va, L, "value");
    see(ex, g[0], ga, L, "x");
    see(ey, g[1], ga, L, "y");
    see(ez, g[2], ga, L, "z");
    for (int i = 0; i < nherm(L); ++i) see(S2[i], S[i], fabsl(S[i]), L, "sum beside value");
}
template <int L>
static void all()
{
    for (int it = 0; it < 4000; ++it) {
        const double rho = exp(drand48() * 9 - 4.6);  // 0.01 .. 80
        double d[3], n = 0;
        for (double &x : d) x = drand48() - 0.5, n += x * x;
        // distances from on top of the pair to far away; every tenth at the near / far limit
        const double r = it % 10 ? exp(drand48() * 8 - 4) : sqrt(harm_tmax(L + 1) / rho) * (1 + 2e-6 * (drand48() - 0.5));
        for (double &x : d) x *= r / sqrt(n);
        if (it % 97 == 0) d[0] = d[1] = 0;
        if (it % 101 == 0) d[0] = d[1] = d[2] = 0;
        one<L>(rho, d, it % 7 ? drand48() - 0.5 : 0.0);
    }
}
int main()
{
    tab.assign((size_t)BOYS_MAXM * BOYS_NROW_D * BOYS_ROW_D, 0.0);
    for (int k = 0; k < BOYS_NROW_D; ++k) {
        ld F[16];
        boys(k * 0.1L, 15, F);
        for (int M = 0; M < BOYS_MAXM; ++M) {
            double *row = &tab[((size_t)M * BOYS_NROW_D + k) * BOYS_ROW_D];
            ld fact = 1;
            for (int j = 0; j < BOYS_TAYLOR_D; ++j) row[j] = (double)(F[M + j] / (fact *= j ? j : 1));
            row[BOYS_ROW_D - 1] = (double)expl(-k * 0.1L);
        }
    }
    all<0>(), all<1>(), all<2>(), all<3>(), all<4>(), all<5>(), all<6>();
    printf("worst %.2e\n", worst);
    return 0;
}
"""


def test_harmonics_match_hermite_recursion(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "harm.cu", tmp_path / "harm"
    src.write_text(SRC)
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-I" + CSRC, str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
