// pair_block.cuh -- the per-pair algebra around the FP64 sweeps: blocks of (32, NA) threads, lane =
// primitive pair, warp = Cartesian component of shell A.  The warps share the pair's 1-D Hermite
// tables through shared memory.
#pragma once
#include "device_common.cuh"

namespace qmmm {

// E^{ij}_t of one direction for i <= LA, j <= JB, t <= T into tab[((i (JB + 1) + j) (T + 1) + t)][lane]:
// E_0 by its two-term recursion, E_t = h/t (i E^{i-1,j}_{t-1} + j E^{i,j-1}_{t-1}), h = 1/(2p)
template <int LA, int JB, int T>
__device__ __forceinline__ void hermite_table(double (*tab)[32], int lane, double xa, double xb, double h)
{
    auto at = [](int i, int j, int t) { return (i * (JB + 1) + j) * (T + 1) + t; };
    for (int i = 0; i <= LA; ++i)
        for (int j = 0; j <= JB; ++j) {
            double e = 1.0;
            if (j > 0) e = xb * tab[at(i, j - 1, 0)][lane] + (T > 0 ? tab[at(i, j - 1, T > 0 ? 1 : 0)][lane] : 0.0);
            else if (i > 0) e = xa * tab[at(i - 1, 0, 0)][lane] + (T > 0 ? tab[at(i - 1, 0, T > 0 ? 1 : 0)][lane] : 0.0);
            tab[at(i, j, 0)][lane] = e;
            for (int t = 1; t <= T; ++t) {
                double s = 0.0;
                if (i > 0) s += i * tab[at(i - 1, j, t - 1)][lane];
                if (j > 0) s += j * tab[at(i, j - 1, t - 1)][lane];
                tab[at(i, j, t)][lane] = h / t * s;
            }
        }
}

template <int LA, int LB>
struct PairShape {
    static constexpr int L = LA + LB, NH = nherm(L), NA = ncart(LA), NB = ncart(LB);
    // Hermite order needed: E_1 also where L = 0 (the derivative of (s, s))
    static constexpr int T = L > 0 ? L : 1;
    static constexpr int NF = 3 * (LA + 1) * (LB + 1) * (T + 1);  // table doubles per lane: fold
    static constexpr int NC = 3 * (LA + 1) * (LB + 2) * (T + 1);  // contraction (shell B up to LB + 1)
    static constexpr int KR = NH < 28 ? NH : 28;                  // components summed over warps at a time
    // shared doubles per lane: density fold, gradient contraction, V contraction
    static constexpr int FS = (NF > NA * KR ? NF : NA * KR) + NH, CS = NC + NH + 3 * NA, VS = NF + 2 * NH;
};
__device__ __forceinline__ void cart_of(int l, int k, int (&c)[3])
{
    int i = 0;
    for (int x = l; x >= 0; --x)
        for (int y = l - x; y >= 0; --y, ++i)
            if (i == k) {
                c[0] = x;
                c[1] = y;
                c[2] = l - x - y;
            }
}

}  // namespace qmmm
