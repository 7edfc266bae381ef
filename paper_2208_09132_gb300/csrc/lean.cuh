// lean.cuh -- equilibria from factor tables, for the "lean" face-store shapes of
// the CDUGKS step (arXiv:2208.09132, Sec. 2.1; D = 2 and 3, velocity grids with
// no node at xi_a = 0).
//
// The equilibria (eqs. geq, beq) are products of separable factors: the Maxwellian
// of a place is rho (2 pi RT)^{-D/2} prod_b exp(-(xi_b - u_b)^2 / 2RT), and the
// per-axis factors of every cell (and, with face tables, face) are formed in double
// by the FP64 kernels (write_factors: W update, face constants, init) into tables.
// A point's g_eq is then D - 1 multiplications of table entries -- no exponential
// per point, and the exponent is exact to double rounding at any Mach number.
// Sweep A of these shapes is usweep.cuh's with TAB, sweep B bflux.cuh's (with face
// tables: XF).
#pragma once

#include "kernels.cuh"

namespace cdg {

// Factor-table rows of the current chunk (aligned velocity grids: nv1_0 a
// multiple of VC, so a chunk's four velocities share k1, k2): the first row of
// its axis-0 block and its rows of axes 1 and 2, direct and with the axis
// mirrored (k -> n - 1 - k).  Advanced chunk by chunk without divisions.
struct LeanRows {
    int c0, k1, k2;               // chunk index along axis 0 (of nv1_0 / VC), k1, k2
    int r0, r1, r2, r0m, r1m, r2m;
};
__device__ __forceinline__ void lean_rows_set(const Geo& g, LeanRows& R) {
    const int n0c = g.nv1[0] / VC;
    R.r0 = R.c0 * VC;
    R.r0m = (n0c - 1 - R.c0) * VC;
    R.r1 = g.xrow[1] + R.k1;
    R.r1m = g.xrow[1] + g.nv1[1] - 1 - R.k1;
    R.r2 = g.xrow[2] + R.k2;
    R.r2m = g.xrow[2] + g.nv1[2] - 1 - R.k2;
}
// g_eq of the four lanes of chunk vt at table place `item` (n places), with the
// velocity components of the mirror axes (bits of refl) reflected.  Aligned
// grids: one vector and one or two scalar loads (rows of R); otherwise each
// lane's indices are found from its velocity number.
template <typename T, int D>
__device__ __forceinline__ void lean_geq4(const Geo& g, const T* __restrict__ X, long long n, long long item,
                                          int refl, int vt, const LeanRows& R, T (&ge)[VC]) {
    const size_t nn = (size_t)n, it = (size_t)item;
    if (g.xal) {
        const int r0 = (refl & 1) ? R.r0m : R.r0;
        const int r1 = (refl & 2) ? R.r1m : R.r1;
        T x0[VC];
        Chunk<T>::load(X + (size_t)r0 * nn + VC * it, x0);      // = xaddr(g, n, r0, item), r0 a multiple of VC
        const T x1 = __ldg(X + (size_t)r1 * nn + it);
        T x2 = T(1);
        if (D == 3) x2 = __ldg(X + (size_t)((refl & 4) ? R.r2m : R.r2) * nn + it);
        const T pr = lean_pair<T, D>(x1, x2);
#pragma unroll
        for (int v = 0; v < VC; ++v) ge[v] = ((refl & 1) ? x0[VC - 1 - v] : x0[v]) * pr;
    } else {
        const int nv = g.nv1[0] * g.nv1[1] * g.nv1[2];
#pragma unroll
        for (int v = 0; v < VC; ++v) {
            const int i = vt * VC + v;
            ge[v] = T(0);
            if (i < nv) {
                int k0 = i % g.nv1[0], k1 = (i / g.nv1[0]) % g.nv1[1], k2 = i / (g.nv1[0] * g.nv1[1]);
                if (refl & 1) k0 = g.nv1[0] - 1 - k0;
                if (refl & 2) k1 = g.nv1[1] - 1 - k1;
                if (refl & 4) k2 = g.nv1[2] - 1 - k2;
                const T x2 = D == 3 ? __ldg(X + xaddr(g, n, g.xrow[2] + k2, item)) : T(1);
                ge[v] = lean_geq<T, D>(__ldg(X + xaddr(g, n, k0, item)), __ldg(X + xaddr(g, n, g.xrow[1] + k1, item)),
                                       x2);
            }
        }
    }
}

}  // namespace cdg
