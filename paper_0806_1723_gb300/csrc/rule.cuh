// Sums of a sphere quadrature (Gauss-Legendre rings in cos(theta), uniform phi) against the 25
// real harmonics, factorised ring by ring: y_lm = f_lm(theta) cos(m phi) or f_l|m| sin(|m| phi).
#pragma once

#include "internal.cuh"

namespace lasto {

// F[row][c] = sum_b V[row][b] g_c(b), g_0 = 1, g_{2m-1} = cos(m phi_b), g_{2m} = sin(m phi_b)
// (trig[b] = cos, sin of phi_b; m phi_b is phi at (m b) mod np).  All threads of the block call;
// V complete before, F complete after a barrier.
template <int NT>
__device__ __forceinline__ void rule_rings(const double* V, int rows, int np, const double* trig, double* F)
{
    for (int t = threadIdx.x; t < 9 * rows; t += NT) {
        const int row = t / 9, c = t - 9 * row, m = (c + 1) >> 1, sn = c > 0 && (c & 1) == 0;
        const double* v = V + row * np;
        double acc = 0.0;
        if (m == 0) {
            for (int b = 0; b < np; b++) acc += v[b];
        } else {
            for (int b = 0, p = 0; b < np; b++) {
                acc = fma(v[b], trig[2 * p + sn], acc);
                p += m;
                while (p >= np) p -= np;
            }
        }
        F[t] = acc;
    }
}

// sum over the rings r0 .. r0 + rows - 1 of w f_lm F[.][c(m)]
__device__ __forceinline__ double rule_lm(const SphereRule& q, const double* F, int r0, int rows, int lm)
{
    const int l = l_of_lm(lm), ms = lm - l * l - l, m = ms < 0 ? -ms : ms;
    const int c = m == 0 ? 0 : ms > 0 ? 2 * m - 1 : 2 * m;
    double acc = 0.0;
    for (int r = 0; r < rows; r++) acc = fma(q.wf[r0 + r][rule_slot(l, m)], F[9 * r + c], acc);
    return acc;
}

}  // namespace lasto
