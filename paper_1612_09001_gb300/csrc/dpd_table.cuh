// Derivation of the per-tap coefficient tables (layouts in dpd_internal.h) from the
// stacked coefficient vector of Sec. 2.2, for the kernels that produce coefficients.
#pragma once

#include "dpd_internal.h"

namespace dpd {

// Thread i of a block with at least B * T threads: (tap, order) pair i; thread 0 also
// the constant.  h(j) is coefficient j; adj (the adjoint table) may be null.
template <class H>
__device__ __forceinline__ void wl_table_entry(H h, int i, int Bp, int Bq, int T, int B, float *__restrict__ tab,
                                               float *__restrict__ adj)
{
    if (i < T * B) {
        const int k = i / B, m = i % B;
        const float2 A = (m < Bp) ? h(m * T + k) : make_float2(0.f, 0.f);          // h_{2m+1,k}
        const float2 C = (m < Bq) ? h((Bp + m) * T + k) : make_float2(0.f, 0.f);   // hbar_{2m+1,k}
        tab[wl_index(B, k, m, 0)] = A.x + C.x;      // P0 = Re(A+C)
        tab[wl_index(B, k, m, 1)] = -(A.y - C.y);   // P1 = -Im(A-C)
        tab[wl_index(B, k, m, 2)] = A.y + C.y;      // P2 = Im(A+C)
        tab[wl_index(B, k, m, 3)] = A.x - C.x;      // P3 = Re(A-C)
        if (adj) {
            // {P0, P3} multiplies the gradient sample {c, d}, {P2, P1} its swap
            // {d, c}: conj(h) g + hbar conj(g) = {P0 c + P2 d, P3 d + P1 c}.
            float *q = adj + 4 * (k * B + m);
            q[0] = A.x + C.x;
            q[1] = A.x - C.x;
            q[2] = A.y + C.y;
            q[3] = C.y - A.y;
        }
    }
    if (i == 0) {
        const float2 c = h((Bp + Bq) * T);
        tab[4 * B * T] = c.x;
        tab[4 * B * T + 1] = c.y;
    }
}

}  // namespace dpd
