"""The near and far branches of the FP64 sweeps at their own limits (csrc/harm.cuh): the V sweep
changes to point-charge factors at harm_tmax(L), the adjoint at harm_tmax(L + 1), and a distant charge
of a warp with a near one takes the near branch with point-charge factors and no Gaussian terms.  Each
against the Hermite recursion in extended precision, on the CPU, with the helpers and the tolerance
(Boys table, rounding; what is dropped above harm_tmax weighs less than 1e-17) of test_harm.py."""
import os
import shutil
import subprocess

import pytest

from test_harm import CSRC, SRC

SRC_LIMITS = SRC[:SRC.index("template <int L>\nstatic void one")] + r"""
#include <cstring>
static bool distant(double r2, double limit)  // the kernels' comparison of high words
{
    unsigned long long a, b;
    memcpy(&a, &r2, 8);
    memcpy(&b, &limit, 8);
    return (unsigned)(a >> 32) > (unsigned)(b >> 32);
}
static int nfar = 0, nnear = 0;
template <int L>
static void one(double rho, const double *d, double q)
{
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], c0 = sqrt(rho) / HALF_SQRT_PI;
    const ld unit = 1 / (ld)c0;
    ld R[286];
    hermite(L + 1, rho, d, R);
    auto sums = [&](const double *S, const char *what) {
        ld W[nherm(L)] = {};
        for (int i = 0; i < H.tend[L]; ++i) W[H.t[i].herm] += unit * H.t[i].c * S[harm_off(L, H.t[i].k) + H.t[i].lm];
        for (int n = 0; n <= L; ++n) {
            ld top = 0;
            for (int i = nherm(n - 1); i < nherm(n); ++i) top = fmaxl(top, fabsl(q * R[i]));
            for (int i = nherm(n - 1); i < nherm(n); ++i) see(W[i], q * R[i], top, L, what);
        }
    };
    {  // V sweep
        const bool far = distant(r2, harm_tmax(L) / rho);
        (far ? nfar : nnear)++;
        double F[L + 1], E0, S[nherm(L)] = {};
        boys_hat<L>(far, r2, rho, c0, F, E0, tab.data());
        harm_add<L, true>(S, F, E0, rho, q, d[0], d[1], d[2], r2);
        sums(S, "V, in a warp with near charges");
        if (far) {
            double S2[nherm(L)] = {};
            harm_add_far<L>(S2, q, d[0], d[1], d[2], r2);
            sums(S2, "V, every lane far");
        }
    }
    {  // adjoint: a lane of a warp with near charges
        const bool far = distant(r2, harm_tmax(L + 1) / rho);
        double F[L + 2], E0, D[nherm(L)], M[nherm(L)] = {}, N[3][nhgrad(L) + 1] = {}, S[nherm(L)] = {}, e0, e[3];
        for (double &x : D) x = drand48() - 0.5;
        for (int i = 0; i < H.tend[L]; ++i) M[harm_off(L, H.t[i].k) + H.t[i].lm] += (double)unit * H.t[i].c * D[H.t[i].herm];
        for (int k = 0; 2 * k < L; ++k)
            for (int i = 0; i < H.gend[L - 2 * k]; ++i)
                N[H.g[i].dir][hgrad_off(L, k) + H.g[i].lm1] += H.g[i].c * M[harm_off(L, k) + H.g[i].lm];
        boys_hat<L + 1>(far, r2, rho, c0, F, E0, tab.data());
        harm_eval<L, true>(M, N[0], N[1], N[2], F, E0, rho, 0.0, d[0], d[1], d[2], r2, q, S, e0, e[0], e[1], e[2]);
        sums(S, "adjoint sums");
        ld v = 0, va = 0, g[3] = {}, ga = 0;
        for (int t = 0; t <= L; ++t)
            for (int u = 0; t + u <= L; ++u)
                for (int w = 0; t + u + w <= L; ++w) {
                    const ld c = D[hidx(t, u, w)];
                    const ld x[4] = {c * R[hidx(t, u, w)], c * R[hidx(t + 1, u, w)], c * R[hidx(t, u + 1, w)],
                                     c * R[hidx(t, u, w + 1)]};
                    v += x[0], va += fabsl(x[0]);
                    for (int a = 0; a < 3; ++a) g[a] += x[a + 1], ga += fabsl(x[a + 1]);
                }
        see(e0, v, va, L, "value");
        for (int a = 0; a < 3; ++a) see(e[a], g[a], ga, L, "gradient");
    }
}
template <int L>
static void all()
{
    for (int it = 0; it < 2000; ++it) {
        const double rho = exp(drand48() * 9 - 4.6);  // 0.01 .. 80
        double d[3], n = 0;
        for (double &x : d) x = drand48() - 0.5, n += x * x;
        const double lim = it % 2 ? harm_tmax(L) : harm_tmax(L + 1);
        // within 2e-6 of a limit, within a factor of 2, or anywhere beyond it
        const double s = it % 4 < 2 ? 1 + 2e-6 * (drand48() - 0.5) : it % 4 == 2 ? 0.5 + drand48() : exp(4 * drand48());
        for (double &x : d) x *= sqrt(lim / rho) * s / sqrt(n);
        one<L>(rho, d, drand48() - 0.5);
    }
}
""" + SRC[SRC.index("int main()"):].replace('printf("worst %.2e\\n", worst);',
                                            'printf("worst %.2e far %d near %d\\n", worst, nfar, nnear);')


def test_branches_at_their_limits(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "limits.cu", tmp_path / "limits"
    src.write_text(SRC_LIMITS)
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-I" + CSRC, str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    far, near = int(r.stdout.split()[3]), int(r.stdout.split()[5])
    assert far > 2000 and near > 2000
