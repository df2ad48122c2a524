// sscn_rho.cuh -- one radial line of the axially symmetric form solved in FP64
// by a pair of lanes (k_sweep_rho, and the FP64 branch of k_inc_rho).
#pragma once

#include <cuda_runtime.h>

#include "sscn_internal.h"
#include "sscn_line.cuh"

namespace gp {

constexpr int kPrefetchR = 4;

__device__ __forceinline__ double2 shfl_pair(double2 v, int pair)
{
    v.x = __shfl_xor_sync(0xffffffffu, v.x, pair);
    v.y = __shfl_xor_sync(0xffffffffu, v.y, pair);
    return v;
}

// row[0 .. m - 1]: the line, swept in place; wl: m entries of scratch.  Unknown
// j = 1 .. m sits at stored index j - 1.  Top lane: j = 1 .. kmid - 1, bottom
// lane: j = m .. kmid + 1, the top lane closes the middle row.  pair: the lanes'
// distance; before(p, i): psi at i ahead of the sweep.  Every lane of the warp
// calls this; `active` marks those with a line.
template <int MODE, typename Before>
__device__ __forceinline__ void solve_rho(double2 *row, double2 *wl, const RadialTables &rt, int m, bool active,
                                          bool top, int pair, Before before)
{
    const int kmid = (m + 1) >> 1;
    const int len = top ? kmid - 1 : m - kmid;
    const double2 *cp = top ? rt.cp_top : rt.cp_bot;
    const double2 *mult = top ? rt.mult_top : rt.mult_bot;
    const double *kk = top ? rt.ka_top : rt.kc_bot;
    double2 d = make_double2(0.0, 0.0);
    if (active) {
        for (int t0 = 0; t0 < len; t0 += kPrefetchR) {
            double2 pv[kPrefetchR];
#pragma unroll
            for (int q = 0; q < kPrefetchR; ++q)
                if (t0 + q < len) pv[q] = row[top ? t0 + q : m - 1 - t0 - q];
#pragma unroll
            for (int q = 0; q < kPrefetchR; ++q) {
                const int t = t0 + q;
                if (t < len) {
                    const int i = top ? t : m - 1 - t;
                    const double2 p = before(pv[q], i);
                    row[i] = p;
                    d = LineOps<double, MODE>{kk[t]}.fwd(p, d, mult[t]);
                    wl[i] = d;
                }
            }
        }
    }
    const double2 other = shfl_pair(d, pair);
    double2 vk = make_double2(0.0, 0.0);
    if (active && top) {
        const int i = kmid - 1;
        const double2 pk = before(row[i], i);
        // kappa (a_k d'_{k-1} + c_k e_{k+1}) as kappa^ q with |kappa| folded into q
        const double2 q = make_double2(fma(rt.ka_mid, d.x, rt.kc_mid * other.x),
                                       fma(rt.ka_mid, d.y, rt.kc_mid * other.y));
        vk = LineOps<double, MODE>{1.0}.fwd(pk, q, rt.mid);
        row[i] = LineOps<double, MODE>::out(vk, pk);
    }
    const double2 vpair = shfl_pair(vk, pair);
    double2 v = top ? vk : vpair;
    if (active) {
        for (int t0 = len - 1; t0 >= 0; t0 -= kPrefetchR) {
            double2 wv[kPrefetchR], lv[kPrefetchR];
#pragma unroll
            for (int q = 0; q < kPrefetchR; ++q)
                if (t0 - q >= 0) {
                    const int i = top ? t0 - q : m - 1 - t0 + q;
                    wv[q] = wl[i];
                    lv[q] = row[i];
                }
#pragma unroll
            for (int q = 0; q < kPrefetchR; ++q) {
                const int t = t0 - q;
                if (t >= 0) {
                    const int i = top ? t : m - 1 - t;
                    v = LineOps<double, MODE>{0.0}.back(wv[q], cp[t], v);
                    row[i] = LineOps<double, MODE>::out(v, lv[q]);
                }
            }
        }
    }
}

}  // namespace gp
