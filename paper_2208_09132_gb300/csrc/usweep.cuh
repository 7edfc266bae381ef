// usweep.cuh -- sweep A of the face-store shapes (two relaxation times,
// upwind-cell reconstruction; D = 1, 2, 3; any boundary; any velocity grid):
// every cell forms the face values it is upwind of.
//
// For one velocity a cell is upwind of exactly one face per axis: its right
// face where xi_a > 0, its left one where xi_a < 0.  So a thread per owned cell
// takes phibar+ of its cell and of its 2D axis neighbours, one limited slope
// vector (eq. VanLeer), and writes D face values (eq. relation) -- no slope is
// formed twice anywhere, and the halo a tile needs is one layer of phibar+
// without corners.  (Owning the left faces instead, as sweeps B and the fused
// sweeps do, needs phibar+ on a two-cell halo and the slopes of a layer around
// the tile: on an 8 x 8 x 4 tile 2.7 phibar+ and 1.5 slopes per point against
// 2.0 and 1.0 here.)
//
// The face moments (eqs. rhobar-rhoEbar) are summed per cell and side: what
// left cells add to a face and what right cells add to it are separate partial
// sums, the *slots* of the face constants' fixed-order sum.  So that a thread
// sums one side per axis in registers, the chunks are visited in order of their
// signs (a *visit* is a chunk with its sign per axis).  A chunk whose lanes
// differ in sign along an axis stores either side's lanes and sums the right
// cells' side apart, in shared memory; in 3D that is axis 0 only, a chunk mixed
// along another axis (velocity rows that are not whole chunks) is visited once
// per pattern of those axes.  A node at xi_a = 0 counts half to either side (the
// mean of the one-sided values, R-h) and its stored value, which no flux takes,
// is the right cell's.  Per velocity group and axis there is a slot for each
// sign the group's visits have.
//
// Boundaries: the halo is mapped by resolve().  On a grid without Dirichlet
// ends a ghost is an image of a cell with all its neighbours.  Periodic ends:
// the face at both ends gets the one value.  Specular ends: the ghost's face
// value at xi is its cell's at the mirrored velocity, so the cell stores it
// there as well, and the face moments are the cell's doubled, without the
// normal momentum.  With a Dirichlet end (whose ghosts along one axis differ
// from the images of their neighbours' ghosts), and between walls on a grid whose
// middle node rounds to one side of 0 (it is its own image, of the same sign), the
// end tiles form the ghosts' values after the sweep (edge_pass).
//
// What bounds it: in FP32 instruction issue and latency at 16 warps per SM, then the
// 8 B read and 8 D B written per point; in FP64 the FP64 pipe.  Against left-face
// owners, ms per launch: FP32 3D 48^3 cells x 24^3 velocities 39.8 -> 14.2 (3.4 TB/s
// of its 32 B per point), 45 x 37 x 29 x 14^3 between walls 7.3 -> 2.9, 2D 256^2 x
// 32^2 0.615 -> 0.402 (4.0 TB/s), 100^2 x 101^2 with nodes at 0 1.71 -> 0.81; FP64
// 2D 256^2 x 32^2 13.0 -> 8.7 (1D 8192 x 129 0.137 -> 0.152, at 7 groups instead of 17).
#pragma once

#include "kernels.cuh"
#include "lean.cuh"
#include "pack.cuh"

namespace cdg {

// Flags of a visit record: the main side per axis (plus: left cells, of their
// right faces), mixed axes (main side plus; the rest minus), the lanes stored.
__host__ __device__ constexpr int visit_class(int flags) { return flags & 63; }
__host__ __device__ constexpr int visit_plus(int flags, int a) { return (flags >> a) & 1; }
__host__ __device__ constexpr int visit_mixed(int flags, int a) { return (flags >> (3 + a)) & 1; }
__host__ __device__ constexpr int visit_lanes(int flags, int a) { return (flags >> (8 + 4 * a)) & 15; }
__host__ __device__ constexpr int visit_minus_lanes(int flags, int a) { return (int)((unsigned)flags >> (20 + 4 * a)) & 15; }
// Axes a visit may be mixed along.
__host__ __device__ constexpr int mixed_axes(int D) { return D == 3 ? 1 : D; }

template <typename T, int D, int T0_, int T1_, int T2_, bool TAB, bool SK = false>
struct USmem {
    using TL = Tile<D, T0_, T1_, T2_, 1>;
    static constexpr int NT = TL::NT, BOX = TL::BOX;
    static constexpr int NH = 2 * TL::NPL;                       // halo cells: one layer, no corners
    static constexpr int KH = (NH + NT - 1) / NT;                // per thread
    static constexpr int NCV = TAB ? 2 : EqPack<T, D, SK>::NV;        // packed constants of a cell
    static constexpr size_t nP = (size_t)2 * 2 * BOX;            // phibar+, two chunks in flight
    // per thread and cell of it: the constants, (TAB) the axis-0 factors, the next visit's phi*
    static constexpr int NS = NCV + (TAB ? 1 : 0) + 2;
    static constexpr size_t nCC = (size_t)NS * (1 + KH) * NT;
    // visit records staged ahead, and of the mixed axes' other side the g values of a visit and the sums
    static constexpr int RING = 8;
    static constexpr size_t rec_bytes = 4 * kVisitInts + kVisitVecs * sizeof(V4<T>);
    static constexpr size_t mix_bytes = (size_t)mixed_axes(D) * NT * ((2 + D) * sizeof(Kahan<T>) + sizeof(V4<T>));
    static constexpr size_t bytes = (nP + nCC) * sizeof(V4<T>) + RING * rec_bytes + mix_bytes;
    // 3D instances without mixed visits keep the cells' numbers there instead, for
    // the registers; the others in registers, for the size: two CTAs of up to 97
    // KB leave L1 60 KB, larger ones 28 KB (the mixed sweep 11.9 -> 13.7 ps per point)
    static constexpr size_t cell_bytes = (size_t)(1 + KH) * NT * sizeof(int2);
    static_assert(D < 3 || cell_bytes <= mix_bytes, "the cells fit");
    static size_t bytes_of(const Geo& g) { return g.mixed ? bytes : bytes - mix_bytes + (D == 3 ? cell_bytes : 0); }
};
// The geometry and buffers of a batch member, copied to shared memory at the
// start of an item (a reference into the table costs a global load per use, a
// copy per thread its stack).
template <typename T>
struct URec {
    Geo g;
    Bufs<T> b;
    __device__ __forceinline__ void load(const Inst<T>& in, int c) {
        static_assert(sizeof(Geo) % 4 == 0 && sizeof(Bufs<T>) % 4 == 0, "copied in words");
        const int* sg = reinterpret_cast<const int*>(&in.g);
        const int* sb = reinterpret_cast<const int*>(&in.b[c]);
        for (int i = threadIdx.x; i < (int)(sizeof(Geo) / 4); i += blockDim.x) reinterpret_cast<int*>(&g)[i] = sg[i];
        for (int i = threadIdx.x; i < (int)(sizeof(Bufs<T>) / 4); i += blockDim.x) reinterpret_cast<int*>(&b)[i] = sb[i];
        __syncthreads();
    }
};

// CTAs per SM: what shared memory, threads and registers (128 in FP32, 168 in
// FP64, or more) allow.
template <typename T, int D, int T0_, int T1_, int T2_, bool TAB, bool SK = false>
struct UOcc {
    static constexpr size_t per = USmem<T, D, T0_, T1_, T2_, TAB, SK>::bytes + 1024;
    static constexpr int NT = T0_ * T1_ * T2_;
    static constexpr int by_smem = (int)((228 * 1024) / per);
    static constexpr int by_regs = 65536 / (NT * (sizeof(T) == 8 ? 168 : 128));
    static constexpr int v = by_smem < by_regs ? by_smem : by_regs;
    static constexpr int value = v < 1 ? 1 : (v > 8 ? 8 : v);
};

// phibar+ of the cell with coordinates q (ghosts included) for the four
// velocities of one chunk, straight from global memory (end cells only).
template <typename T, int D, bool TAB, bool NOSRC, bool SK, bool PRE>
__device__ __noinline__ void phibar_at(const Geo& g, const Bufs<T>& bf, int q0, int q1, int q2, int vt,
                                          const T* __restrict__ vr, T (&pg)[VC], T (&pb)[VC]) {
    int q[3] = {q0, q1, q2};
    int refl;
    bool dir;
    resolve<D>(g, q, refl, dir);
    const long long c = cell_index(g, q);
    if (PRE && !dir) {             // formed by the pre-pass
#pragma unroll
        for (int v = 0; v < VC; ++v) {
            const int i = vt * VC + v, is = refl ? bf.refl[refl * g.Nvp + i] : i;
            pg[v] = bf.phibar[phi_addr(g, c, is, 0)];
            pb[v] = bf.phibar[phi_addr(g, c, is, 1)];
        }
        return;
    }
    const CellC<T>& cs = dir ? bf.cellc0[c] : bf.cellc[c];
    T u[D];
#pragma unroll
    for (int a = 0; a < D; ++a) u[a] = (refl & (1 << a)) ? -cs.u[a] : cs.u[a];
    T ge[VC];
    if constexpr (TAB) {
        LeanRows R = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        if (g.xal) {
            const int n0c = g.nv1[0] / VC;
            R.c0 = vt % n0c;
            R.k1 = (vt / n0c) % g.nv1[1];
            R.k2 = vt / (n0c * g.nv1[1]);
            lean_rows_set(g, R);
        }
        lean_geq4<T, D>(g, dir ? bf.xc0 : bf.xc, g.Nc, c, refl, vt, R, ge);
    }
    const T hL = g.consts<T>().ceb;
#pragma unroll
    for (int v = 0; v < VC; ++v) {
        T z = -cs.hu2, be;
        if constexpr (SK) {
            T c2 = T(0), cq = T(0);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const T d = vr[a * VC + v] - u[a];
                c2 = fma(d, d, c2);
                cq = fma((refl & (1 << a)) ? -cs.sq[a] : cs.sq[a], d, cq);
            }
            shakhov_point<T, D>(cs.pref * Num<T>::expo(cs.cexp * c2), c2, cq, cs.cexp * Num<T>::irt_scale(),
                                vr[3 * VC + v], cs.eb, hL, cs.e2, ge[v], be);
        } else if constexpr (!TAB) {
            T c2 = T(0);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const T d = vr[a * VC + v] - u[a];
                c2 = fma(d, d, c2);
            }
            ge[v] = cs.pref * Num<T>::expo(cs.cexp * c2);
        }
        if constexpr (!SK) be = (vr[3 * VC + v] + cs.eb) * ge[v];
        if (dir) {                 // Dirichlet ghost: the equilibrium of its initial state
            pg[v] = ge[v];
            pb[v] = be;
            continue;
        }
#pragma unroll
        for (int a = 0; a < D; ++a) z = fma(vr[a * VC + v], u[a], z);
        const int i = vt * VC + v, is = refl ? bf.refl[refl * g.Nvp + i] : i;
        phibar_plus<T, NOSRC>(ge[v], be, bf.phi_in[phi_addr(g, c, is, 0)], bf.phi_in[phi_addr(g, c, is, 1)],
                              NOSRC ? T(0) : z, cs.kp_g, cs.kp_b, cs.kp_s, pg[v], pb[v]);
    }
}

// The faces that the ghosts beyond one end of a tile (axis a, side 0 low /
// 1 high) are upwind of: their values for every visit of the group, stored and
// summed into the group's slot of that side.  Every thread of the CTA calls it,
// one (end cell, visit) pair per thread and round; the end cells' threads add
// the visits' moments in order.  Not inlined: kept out of the sweep's registers
// and code.
template <typename T, int D, typename TL, bool TAB, bool NOSRC, bool SK, bool PRE>
__device__ __noinline__ void edge_pass(const Geo& g, const Bufs<T>& bf, int org0, int org1, int org2, int a, int side, int j0,
                                       int j1, int slot, T* red) {
    constexpr int NM = 2 + D, NT = TL::NT;
    const int plane = TL::plane(a), vpr = NT / plane;      // visits per round
    const int t = threadIdx.x, p = t % plane, dj = t / plane;
    int l[3] = {0, 0, 0};
    if (a == 0) { l[1] = p % TL::T1; l[2] = p / TL::T1; }
    else if (a == 1) { l[0] = p % TL::T0; l[2] = p / TL::T0; }
    else { l[0] = p % TL::T0; l[1] = p / TL::T0; }
    int q[3] = {org0 + l[0], org1 + l[1], org2 + l[2]};
    q[a] = side ? g.n[a] - 1 : 0;
    bool on = dj < vpr;
#pragma unroll
    for (int b = 0; b < D; ++b) on = on && q[b] < g.n[b];
    q[a] += side;
    const long long f = on ? face_index(g, a, q) : 0;      // the end face
    if (!side) q[a] = -1;                                  // the ghost
    Kahan<T> acc[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) acc[m].zero();
    for (int jb = j0; jb < j1; jb += vpr) {
        const int j = jb + dj;
        T sm[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) sm[m] = T(0);
        const int flags = on && j < j1 ? __ldg(bf.vint + (size_t)kVisitInts * j + 1) : 0;
        // (a low ghost is upwind where xi_a > 0)
        const bool other = side && visit_mixed(flags, a);
        if (on && j < j1 && (visit_plus(flags, a) != side || other)) {
            const int vt = __ldg(bf.vint + (size_t)kVisitInts * j);
            const T* vr = bf.vrec + (size_t)j * (kVisitVecs * VC);
            T base[2][VC], ctr[2][VC], hsa[2][VC];
            phibar_at<T, D, TAB, NOSRC, SK, PRE>(g, bf, q[0], q[1], q[2], vt, vr, base[0], base[1]);
#pragma unroll
            for (int v = 0; v < VC; ++v) {
                ctr[0][v] = base[0][v];
                ctr[1][v] = base[1][v];
            }
#pragma unroll 1
            for (int e = 0; e < D; ++e) {
                T lo[2][VC], hi[2][VC];
                phibar_at<T, D, TAB, NOSRC, SK, PRE>(g, bf, q[0] - (e == 0), q[1] - (e == 1), q[2] - (e == 2), vt, vr, lo[0], lo[1]);
                phibar_at<T, D, TAB, NOSRC, SK, PRE>(g, bf, q[0] + (e == 0), q[1] + (e == 1), q[2] + (e == 2), vt, vr, hi[0], hi[1]);
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int v = 0; v < VC; ++v) {
                        const T hs = vanleer1(ctr[k][v] - lo[k][v], hi[k][v] - ctr[k][v]);
                        base[k][v] = fma(vr[(4 + e) * VC + v], hs, base[k][v]);
                        if (e == a) hsa[k][v] = hs;
                    }
            }
            const int st = other ? visit_minus_lanes(flags, a) : visit_lanes(flags, a);
            T* dst = bf.face[a] + ((size_t)vt * (size_t)g.nf[a] + (size_t)f) * (2 * VC);
#pragma unroll
            for (int v = 0; v < VC; ++v) {
                const T vg = side ? base[0][v] - hsa[0][v] : base[0][v] + hsa[0][v];
                const T vb = side ? base[1][v] - hsa[1][v] : base[1][v] + hsa[1][v];
                if ((st >> v) & 1) {
                    dst[v] = vg;
                    dst[VC + v] = vb;
                }
                const T w = vr[((other ? 10 : 7) + a) * VC + v], wg = w * vg;
                sm[0] = Ar<T>::add(sm[0], wg);
#pragma unroll
                for (int b = 0; b < D; ++b) sm[1 + b] = fma(vr[b * VC + v], wg, sm[1 + b]);
                sm[1 + D] = fma(w, vb, sm[1 + D]);
            }
        }
        __syncthreads();                                   // the last round's sums are read
#pragma unroll
        for (int m = 0; m < NM; ++m) red[m * NT + t] = sm[m];
        __syncthreads();
        if (dj == 0)
            for (int i = 0; i < vpr && jb + i < j1; ++i)
#pragma unroll
                for (int m = 0; m < NM; ++m) acc[m].add(red[m * NT + i * plane + p]);
    }
    if (dj == 0 && on && slot >= 0)
#pragma unroll
        for (int m = 0; m < NM; ++m) bf.wf[a][((size_t)slot * NM + m) * (size_t)g.nf[a] + f] = acc[m].value();
}

// Two chunk-wide asynchronous copies of one cell share its sector: allocate in L1.
template <typename T>
__device__ __forceinline__ void cp_async_chunk_ca(Pk<T>* sdst, const T* gsrc) {
#pragma unroll
    for (int i = 0; i < (int)(sizeof(Pk<T>) / 16); ++i) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(reinterpret_cast<char*>(sdst) + 16 * i);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(d),
                     "l"(__cvta_generic_to_global(reinterpret_cast<const char*>(gsrc) + 16 * i))
                     : "memory");
    }
}
// The lanes of a mask of one face's chunk.
template <typename T>
__device__ __forceinline__ void store_lanes(T* dst, int lanes, const Pk<T>& vg, const Pk<T>& vb) {
    T g4[VC], b4[VC];
    vg.get(g4);
    vb.get(b4);
#pragma unroll
    for (int v = 0; v < VC; ++v)
        if ((lanes >> v) & 1) {
            dst[v] = g4[v];
            dst[VC + v] = b4[v];
        }
}
// A cell at the ends `end` (1 low, 2 high) of axis a, on a grid of images
// (Geo::mirror): its face value (plus: of the right face; lanes st, of them zl
// at xi_a = 0) where a ghost beyond the end is its image.
template <typename T>
__device__ __forceinline__ void end_faces(const Geo& g, const Bufs<T>& bf, int a, int plus, int end, int vt, int st, int zl, int ff,
                                          int fs, const Pk<T>& vg, const Pk<T>& vb) {
    const size_t row = (size_t)vt * (size_t)g.nf[a];
    if ((end >> plus) & 1) {
        if (g.bc[a][plus] == BC_PERIODIC) {               // the same face at the other end
            store_lanes(bf.face[a] + (row + (size_t)(ff + (plus ? 1 - g.n[a] : g.n[a]) * fs)) * (2 * VC), st, vg, vb);
        } else {                                          // the ghost's value: this one, mirrored
            T g4[VC], b4[VC];
            vg.get(g4);
            vb.get(b4);
#pragma unroll
            for (int v = 0; v < VC; ++v)
                if ((st >> v) & 1) {
                    const int is = bf.refl[(1 << a) * g.Nvp + vt * VC + v];
                    T* const d = bf.face[a] + ((size_t)(is / VC) * (size_t)g.nf[a] + (size_t)(ff + (plus ? fs : 0))) * (2 * VC)
                                 + (is % VC);
                    d[0] = g4[v];
                    d[VC] = b4[v];
                }
        }
    }
    // lanes at xi_a = 0 (padding too) at a wall's high end, which no mirror image fills
    if (zl && !plus && (end & 2) && g.bc[a][1] == BC_SPECULAR)
        store_lanes(bf.face[a] + (row + (size_t)(ff + fs)) * (2 * VC), zl, vg, vb);
}

// TAB: equilibria from the cell factor tables (lean shapes), else one
// exponential per point (SK: with the Shakhov correction); PRE: phibar+ from the
// pre-pass (acceleration).  What other kernels
// or items wrote is read through coherent copies and loads, so the persistent
// batched step runs the same body.  g and bf lie in the constant bank (single instances) or in shared
// memory (batches) and are read where they are used, which keeps the loop's
// registers for the chunk in flight.
template <typename T, int D, int T0_, int T1_, int T2_, bool TAB, bool NOSRC, bool SK = false, bool MIX = true,
          bool AL = true, bool PRE = false>
__device__ __forceinline__ void usweep_body(const Geo& g, const Bufs<T>& bf, int tile, int grp, unsigned char* smem) {
    using US = USmem<T, D, T0_, T1_, T2_, TAB, SK>;
    using TL = typename US::TL;
    using K = Pk<T>;
    constexpr int NM = 2 + D, BOX = TL::BOX, NT = TL::NT, KH = US::KH, NCV = US::NCV, N8 = 2 * VC, DM = MIX ? mixed_axes(D) : 0;
    constexpr int SX0 = NCV, SPH = NCV + (TAB ? 1 : 0);             // slot kinds: axis-0 factors, staged phi*
    static_assert(NT % 32 == 0, "whole warps");
    static_assert(!SK || (!TAB && NOSRC), "Shakhov equilibria take one exponential and have no b-source");
    K* const P = reinterpret_cast<K*>(smem);                        // [2][2][BOX]
    K* const CC = P + US::nP + threadIdx.x;                         // this thread's slots [NS][1 + KH], NT apart
    unsigned char* const ring = smem + (US::nP + US::nCC) * sizeof(K);
    K* const MO = reinterpret_cast<K*>(ring + US::RING * US::rec_bytes) + threadIdx.x;                 // [DM], NT apart
    Kahan<T>* const MX = reinterpret_cast<Kahan<T>*>(MO - threadIdx.x + mixed_axes(D) * NT) + threadIdx.x;   // [DM][NM]
    auto slot = [&](int kind, int r) -> K& { return CC[(kind * (1 + KH) + r) * NT]; };
    const int t = threadIdx.x;
    int org[3];
    tile_origin<TL, D>(g, tile, org);
    const int j0 = (int)((long long)grp * g.nvis / g.G), j1 = (int)((long long)(grp + 1) * g.nvis / g.G);

    // this thread's cells: its own (slot 0), then the halo cells t, t + NT, ...
    const int la[3] = {t % TL::T0, D >= 2 ? (t / TL::T0) % TL::T1 : 0, D >= 3 ? t / (TL::T0 * TL::T1) : 0};
    const int qa[3] = {org[0] + la[0], org[1] + la[1], org[2] + la[2]};
    bool valid = true;
#pragma unroll
    for (int a = 0; a < D; ++a) valid = valid && qa[a] < g.n[a];
    // per cell: the source cell (-1 none), box index | boundary flags << 16
    constexpr bool CS = D == 3 && !MIX;
    int2 cells[CS ? 1 : 1 + KH];
    int2* const CL = reinterpret_cast<int2*>(ring + US::RING * US::rec_bytes) + threadIdx.x;
    auto cell = [&](int r) -> int2& {
        if constexpr (CS) return CL[r * NT];
        else return cells[r];
    };
    const int k0 = TL::box_of(la[0], la[1], la[2]);
#pragma unroll
    for (int r = 0; r <= KH; ++r) {
        int l[3] = {la[0], la[1], la[2]};
        bool on = true;
        if (r > 0) {
            int h = t + (r - 1) * NT;
            on = h < US::NH;
            if (!on) h = 0;
            int a = 0;
#pragma unroll
            for (int b = 1; b < D; ++b) a += h >= 2 * TL::poff(b) ? 1 : 0;
            h -= 2 * TL::poff(a);
            const int pl = TL::plane(a), side = h / pl, p = h % pl;
            const int end = side ? TL::tdim(a) : -1;
            if (a == 0) { l[0] = end; l[1] = p % TL::T1; l[2] = p / TL::T1; }
            else if (a == 1) { l[0] = p % TL::T0; l[1] = end; l[2] = p / TL::T0; }
            else { l[0] = p % TL::T0; l[1] = p / TL::T0; l[2] = end; }
        }
        int q[3] = {org[0] + l[0], org[1] + l[1], org[2] + l[2]};
        int refl;
        bool dir;
        resolve<D>(g, q, refl, dir);
        const long long c = cell_index(g, q);
        cell(r) = make_int2(on ? (int)c : -1, TL::box_of(l[0], l[1], l[2]) | (refl | (dir ? 8 : 0)) << 16);
    }

    if (j0 >= j1) return;
    // Visit records come to shared memory three visits ahead: issued at visit j,
    // record j + 3 has landed for its copier at the top of visit j + 1 and is
    // visible to all past that visit's barrier; its first reader is fetch() in
    // visit j + 2.  (Eight slots: no reader of the slot's last record is left.)
    auto rec_int = [&](int j) { return reinterpret_cast<const int*>(ring + (size_t)(j & (US::RING - 1)) * US::rec_bytes); };
    auto rec_val = [&](int j) {
        return reinterpret_cast<const K*>(ring + (size_t)(j & (US::RING - 1)) * US::rec_bytes + 4 * kVisitInts);
    };
    auto fetch_rec = [&](int j) {
        constexpr int NQ = (int)(US::rec_bytes / 16);
        static_assert(NQ <= NT, "one 16-byte piece per thread");
        if (t < NQ && j < j1) {
            constexpr int NI = kVisitInts / 4;
            const char* from = t < NI ? reinterpret_cast<const char*>(bf.vint + (size_t)kVisitInts * j) + 16 * t
                                      : reinterpret_cast<const char*>(bf.vrec + (size_t)(kVisitVecs * VC) * j) + 16 * (t - NI);
            cp_async16(ring + (size_t)(j & (US::RING - 1)) * US::rec_bytes + 16 * t, from);
        }
    };
    // The next visit's phi* of this thread's cells, copied asynchronously to its
    // own slots (a mirror image element by element, a Dirichlet ghost needs
    // none; each thread reads back only what it copied), and (TAB) the axis
    // factors of aligned velocity grids: axis 0's are kept while its row stays.
    T x12[TAB ? 1 + KH : 1][2];
    int row0 = -1;
    auto fetch = [&](const int* const ri) {          // the visit's ints
        const int4 vi = *reinterpret_cast<const int4*>(ri);       // chunk, flags, rows of axes 1 and 2
        const int vt = vi.x, r0 = TAB ? ri[4] : 0;
        const unsigned long long nn = (unsigned)g.Nc;
        const T* const phi = PRE ? bf.phibar : bf.phi_in;
        const T* const row = phi + (unsigned)vt * (nn * N8);
        const T *px0 = nullptr, *px1 = nullptr, *px2 = nullptr;
        if constexpr (TAB) {
            px0 = bf.xc + (unsigned)r0 * nn;
            px1 = bf.xc + (unsigned)vi.z * nn;
            px2 = bf.xc + (unsigned)vi.w * nn;
        }
#pragma unroll
        for (int r = 0; r <= KH; ++r) {
            const int2 cl = cell(r);
            if (cl.x < 0) continue;
            const unsigned c = (unsigned)cl.x;
            const int f = cl.y >> 16;
            if (f == 0) {
                cp_async_chunk_ca(&slot(SPH, r), row + (unsigned long long)c * N8);
                cp_async_chunk_ca(&slot(SPH + 1, r), row + (unsigned long long)c * N8 + VC);
                if constexpr (TAB) {
                    if constexpr (AL) {
                        if (r0 != row0) cp_async_chunk_ca(&slot(SX0, r), px0 + (unsigned long long)c * VC);
                        x12[r][0] = __ldg(px1 + c);
                        if constexpr (D == 3) x12[r][1] = __ldg(px2 + c);
                    }
                }
                continue;
            }
            if (!(f & 8)) {
#pragma unroll
                for (int v = 0; v < VC; ++v) {
                    const int is = bf.refl[(f & 7) * g.Nvp + vt * VC + v];
                    const T* p = phi + (size_t)(is / VC) * (nn * N8) + (size_t)c * N8 + (is % VC);
                    cp_async_elem(reinterpret_cast<T*>(&slot(SPH, r)) + v, p);
                    cp_async_elem(reinterpret_cast<T*>(&slot(SPH + 1, r)) + v, p + VC);
                }
            }
            if constexpr (TAB) {
                if constexpr (AL) {
                    const T* X = (f & 8) ? bf.xc0 : bf.xc;
                    if (r0 != row0)
                        cp_async_chunk_ca(&slot(SX0, r), X + (size_t)((f & 1) ? g.nv1[0] - VC - r0 : r0) * nn + (size_t)VC * c);
                    x12[r][0] = __ldg(X + (size_t)((f & 2) ? 2 * g.xrow[1] + g.nv1[1] - 1 - vi.z : vi.z) * nn + c);
                    if constexpr (D == 3)
                        x12[r][1] = __ldg(X + (size_t)((f & 4) ? 2 * g.xrow[2] + g.nv1[2] - 1 - vi.w : vi.w) * nn + c);
                }
            }
        }
        row0 = r0;
    };

    // the first records and visit are in flight while the constants are staged
    {
        fetch_rec(j0);
        fetch_rec(j0 + 1);
        fetch_rec(j0 + 2);
        fetch(bf.vint + (size_t)kVisitInts * j0);
        cp_async_commit();
    }
#pragma unroll
    for (int r = 0; r <= KH; ++r) {
        const int2 cl = cell(r);
        if (cl.x < 0) continue;
        const int refl = cl.y >> 16 & 7;
        const CellC<T>& cs = (cl.y >> 16 & 8) ? bf.cellc0[cl.x] : bf.cellc[cl.x];
        T cst[4 * NCV];
#pragma unroll
        for (int i = 0; i < 4 * NCV; ++i) cst[i] = T(0);
#pragma unroll
        for (int a = 0; a < D; ++a) cst[a] = (refl & (1 << a)) ? -cs.u[a] : cs.u[a];
        if constexpr (!TAB) {
            cst[D + 0] = cs.cexp;
            cst[D + 1] = cs.pref;
        }
        constexpr int o = TAB ? 3 : D + 2;                  // TAB: hu2 at 3 and eb at 4, else eb, then hu2
        cst[TAB ? o : o + 1] = cs.hu2;
        cst[TAB ? o + 1 : o] = cs.eb;
        cst[o + 2] = cs.kp_g;
        cst[o + 3] = cs.kp_b;
        cst[o + 4] = cs.kp_s;
        if constexpr (SK) {
#pragma unroll
            for (int a = 0; a < D; ++a) cst[D + 7 + a] = (refl & (1 << a)) ? -cs.sq[a] : cs.sq[a];
            cst[2 * D + 7] = cs.e2;
        }
#pragma unroll
        for (int i = 0; i < NCV; ++i) {
            const T x[VC] = {cst[4 * i], cst[4 * i + 1], cst[4 * i + 2], cst[4 * i + 3]};
            slot(i, r) = K::of(x);
        }
    }

    // this thread's left faces (the right ones are a stride fstr(a) on), and the
    // domain ends it lies at (bit 2a low, 2a + 1 high)
    int ff[D], ends = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        ff[a] = valid ? (int)face_index(g, a, qa) : 0;
        ends |= (valid && qa[a] == 0 ? 1 : 0) << (2 * a);
        ends |= (valid && qa[a] == g.n[a] - 1 ? 2 : 0) << (2 * a);
    }
    const T hL = SK ? g.consts<T>().ceb : T(0);
    auto fstr = [&](int a) { return a == 0 ? 1 : (a == 1 ? g.fn[1][0] : g.fn[2][0] * g.fn[2][1]); };

    Sums<T, D * NM> acc;
    acc.zero();
    int written = 0;                                 // bit 2a + side: this group's slot holds a value already
    int cls = visit_class(__ldg(bf.vint + (size_t)kVisitInts * j0 + 1)), mixed = 0;
    // a sum x(m) of axis a's side `plus` to (or, if there is one, onto the value in) its slot
    auto put = [&](int a, int plus, auto x) {
        const int wslot = __ldg(bf.slots + (grp * 3 + a) * 2 + plus);
        const bool again = (written >> (2 * a + plus)) & 1;
        const size_t nf = (size_t)g.nf[a];
        double* const dst = bf.wf[a] + (size_t)wslot * NM * nf;
        const int f = ff[a] + (plus ? fstr(a) : 0);
        const bool end = (ends >> (2 * a + plus)) & 1 && g.mirror;
        const bool wall = end && g.bc[a][plus] == BC_SPECULAR;
        const bool dup = end && g.bc[a][plus] == BC_PERIODIC;
        const int f2 = ff[a] + (plus ? 1 - g.n[a] : g.n[a]) * fstr(a);      // the other end's face
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            double v = x(m);
            if (wall) v = m == 1 + a ? 0.0 : dadd(v, v);
            double* p = dst + (size_t)m * nf;
            const double s = again ? dadd(p[f], v) : v;
            p[f] = s;
            if (dup) p[f2] = s;
        }
    };
    auto flush = [&]() {                             // the sums so far to the slots of the main sides of cls
        if (valid)
#pragma unroll
            for (int a = 0; a < D; ++a) put(a, visit_plus(cls, a), [&](int m) { return acc.value(a * NM + m); });
#pragma unroll
        for (int a = 0; a < D; ++a) written |= 1 << (2 * a + visit_plus(cls, a));
        acc.zero();
    };

    cp_async_wait_all();
    __syncthreads();
    int buf = 0;
    for (int j = j0; j < j1; ++j) {
        const int2 vi = *reinterpret_cast<const int2*>(rec_int(j));
        const int vt = vi.x, flags = vi.y;
        const K* const vr = rec_val(j);
        if (visit_class(flags) != cls) {
            flush();
            cls = visit_class(flags);
        }
        if (MIX && (cls & ~mixed & 56)) {            // the first mixed visit along an axis
#pragma unroll
            for (int a = 0; a < DM; ++a)
                if (visit_mixed(cls & ~mixed, a))
#pragma unroll
                    for (int m = 0; m < NM; ++m) MX[(a * NM + m) * NT].zero();
            mixed |= cls & 56;
        }
        K* const Pg = P + (size_t)buf * 2 * BOX;
        K* const Pb = Pg + BOX;
        cp_async_wait_all();
        // ---- phibar+ (eq. phibarplus) of this thread's cells
        {
            K xi[D];
#pragma unroll
            for (int a = 0; a < D; ++a) xi[a] = vr[a];
            const K hx = vr[3];
#pragma unroll
            for (int r = 0; r <= KH; ++r) {
                const int2 cl = cell(r);
                if (cl.x < 0) continue;
                const int fl = cl.y >> 16;
                if (PRE && !(fl & 8)) {              // phibar+ as the pre-pass formed it
                    Pg[cl.y & 0xffff] = slot(SPH, r);
                    Pb[cl.y & 0xffff] = slot(SPH + 1, r);
                    continue;
                }
                T cst[4 * NCV];
#pragma unroll
                for (int i = 0; i < NCV; ++i) {
                    T x[VC];
                    slot(i, r).get(x);
#pragma unroll
                    for (int e = 0; e < 4; ++e) cst[4 * i + e] = x[e];
                }
                constexpr int o = TAB ? 3 : D + 2, oh = TAB ? 3 : D + 3;
                K ge, pb;
                if constexpr (TAB) {
                    if constexpr (AL) {
                        K x = slot(SX0, r);
                        if (fl & 1) {
                            T y[VC];
                            x.get(y);
                            const T z[VC] = {y[3], y[2], y[1], y[0]};
                            x = K::of(z);
                        }
                        ge = x * K::bc(lean_pair<T, D>(x12[r][0], x12[r][1]));
                    } else {
                        // a chunk's lanes lie in at most two velocity rows (the first
                        // lane's and the last one's); a mirror image takes the mirrored ones
                        const int* const ri = rec_int(j);
                        const unsigned long long nn = (unsigned)g.Nc, c = (unsigned)cl.x;
                        const T* const X = (fl & 8) ? bf.xc0 : bf.xc;
                        const int m0 = g.nv1[0] - 1, m1 = 2 * g.xrow[1] + g.nv1[1] - 1, m2 = 2 * g.xrow[2] + g.nv1[2] - 1;
                        auto row = [&](int v) {
                            const int r1 = ri[8 + v], r2 = ri[12 + v];
                            const T x1 = __ldg(X + (unsigned)((fl & 2) ? m1 - r1 : r1) * nn + c);
                            return lean_pair<T, D>(x1, D == 3 ? __ldg(X + (unsigned)((fl & 4) ? m2 - r2 : r2) * nn + c) : T(1));
                        };
                        const int last = ri[7] < 0 ? 0 : 3;      // (padding only follows lanes of one row)
                        const T pa = row(0);
                        T pb = pa;
                        if (ri[8 + last] != ri[8] || ri[12 + last] != ri[12]) pb = row(3);
                        T y[VC];
#pragma unroll
                        for (int v = 0; v < VC; ++v) {
                            const int k = ri[4 + v], k0 = (fl & 1) ? m0 - k : k;
                            const bool in_a = ri[8 + v] == ri[8] && ri[12 + v] == ri[12];
                            y[v] = k < 0 ? T(0) : __ldg(X + ((unsigned)(k0 / VC) * nn + c) * VC + (k0 % VC)) * (in_a ? pa : pb);
                        }
                        ge = K::of(y);
                    }
                } else {
                    eq4<T, D, SK>(cst, xi, hx, hL, ge, pb);
                }
                if constexpr (TAB) pb = (hx + K::bc(cst[o + 1])) * ge;
                K pg = ge;
                if (!PRE && !(fl & 8)) {
                    const K dg = slot(SPH, r) - ge, db = slot(SPH + 1, r) - pb;
                    pg = fma4(K::bc(cst[o + 2]), dg, ge);
                    pb = fma4(K::bc(cst[o + 3]), db, pb);
                    if constexpr (!NOSRC) {
                        K z = K::bc(-cst[oh]);
#pragma unroll
                        for (int a = 0; a < D; ++a) z = fma4(xi[a], K::bc(cst[a]), z);
                        pb = fma4(K::bc(cst[o + 4]) * z, dg, pb);
                    }
                }
                Pg[cl.y & 0xffff] = pg;
                Pb[cl.y & 0xffff] = pb;
            }
        }
        if (j + 1 < j1) {                            // in flight over the rest of this visit
            fetch(rec_int(j + 1));
            fetch_rec(j + 3);
            cp_async_commit();
        }
        __syncthreads();
        // (one barrier per visit: the other buffer is written next, and this one
        // again only after the next barrier, past which every thread has read it)
        if (valid) {
            K vg[D];                                 // g at the main side's faces
            T sm[D * NM];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                if (D == 3) asm volatile("" ::: "memory");     // b's neighbours not before g is done: registers
                const K* const Pf = (f ? Pb : Pg) + k0;
                const K c = Pf[0];
                K base = c, hs[D];
#pragma unroll
                for (int e = 0; e < D; ++e) {
                    const K lo = Pf[-TL::bstride(e)], hi = Pf[TL::bstride(e)];
                    hs[e] = vanleer4(c - lo, hi - c);
                    base = fma4(vr[4 + e], hs[e], base);       // - (2h xi_e / dx_e) of half the slope
                }
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    const int plus = visit_plus(cls, a);
                    const K val = plus ? base + hs[a] : base - hs[a];
                    if (f == 0) {
                        vg[a] = val;
                        if (a < DM && visit_mixed(cls, a)) MO[a * NT] = base - hs[a];
                        continue;
                    }
                    // moments of one side (weights w) and its face values to the face store
                    auto moments = [&](const K& w, const K& g4, const K& b4, T* o) {
                        const K wg = w * g4;
                        o[0] = sum4(wg);
#pragma unroll
                        for (int b = 0; b < D; ++b) o[1 + b] = dot4(vr[b], wg);
                        o[1 + D] = dot4(w, b4);
                    };
                    auto store = [&](int pl, int st, const K& g4, const K& b4) {
                        T* const dst = bf.face[a] + (unsigned)vt * ((unsigned long long)(unsigned)g.nf[a] * N8)
                                       + (unsigned long long)(unsigned)(ff[a] + (pl ? fstr(a) : 0)) * N8;
                        if (st == 15) store_gb(dst, g4, b4);
                        else if (st) store_lanes(dst, st, g4, b4);
                        const int end = (ends >> (2 * a)) & 3;
                        if (end && g.mirror && st)
                            end_faces<T>(g, bf, a, pl, end, vt, st, (rec_int(j)[16] >> (4 * a)) & 15, ff[a], fstr(a), g4, b4);
                    };
                    moments(vr[7 + a], vg[a], val, sm + a * NM);
                    acc.add(sm, a * NM, (a + 1) * NM);
                    store(plus, visit_lanes(flags, a), vg[a], val);
                    if (a < DM && visit_mixed(cls, a)) {
                        const K vo = MO[a * NT], vb = base - hs[a];
                        T so[NM];
                        moments(vr[10 + a], vo, vb, so);
#pragma unroll
                        for (int m = 0; m < NM; ++m) {
                            Kahan<T> k = MX[(a * NM + m) * NT];
                            k.add(so[m]);
                            MX[(a * NM + m) * NT] = k;
                        }
                        store(0, visit_minus_lanes(flags, a), vo, vb);
                    }
                }
            }
        }
        buf ^= 1;
    }
    flush();
    if (MIX && valid && mixed)
#pragma unroll
        for (int a = 0; a < DM; ++a)
            if (visit_mixed(mixed, a)) put(a, 0, [&](int m) { return MX[(a * NM + m) * NT].value(); });
    // what the ghosts beyond the domain's ends add to the end faces
    if (g.mirror) {
        if (valid && ends) {
#pragma unroll
            for (int a = 0; a < D; ++a) {
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    if (!((ends >> (2 * a + side)) & 1) || g.bc[a][side] == BC_PERIODIC) continue;
                    const int wslot = __ldg(bf.slots + (grp * 3 + a) * 2 + (side ? 0 : 1));
                    if (wslot >= 0)                  // in the cell's own slot already
#pragma unroll
                        for (int m = 0; m < NM; ++m)
                            bf.wf[a][((size_t)wslot * NM + m) * (size_t)g.nf[a] + ff[a] + (side ? fstr(a) : 0)] = 0.0;
                }
            }
        }
    } else {
        int tl = tile;
        keep(tl);                                    // (found again here rather than kept over the loop)
        tile_origin<TL, D>(g, tl, org);
        static_assert(NM * sizeof(T) * NT <= US::bytes, "the moments of a round in shared memory");
#pragma unroll 1
        for (int a = 0; a < D; ++a) {
            const int tdim = a == 0 ? TL::T0 : (a == 1 ? TL::T1 : TL::T2), oa = a == 0 ? org[0] : (a == 1 ? org[1] : org[2]);
#pragma unroll 1
            for (int side = 0; side < 2; ++side)
                if (side ? oa + tdim >= g.n[a] : oa == 0)
                    edge_pass<T, D, TL, TAB, NOSRC, SK, PRE>(g, bf, org[0], org[1], org[2], a, side, j0, j1,
                                                        __ldg(bf.slots + (grp * 3 + a) * 2 + (side ? 0 : 1)),
                                                        reinterpret_cast<T*>(smem));
        }
    }
}

// MIX = false: for instances without mixed visits, AL = false (TAB): whose
// velocity rows are not whole chunks.  Each variant's loop holds only what it
// needs: in 3D the registers and the loop's code size are the limit.
template <typename T, int D, int T0_, int T1_, int T2_, bool TAB, bool NOSRC, bool SK = false, bool MIX = true, bool AL = true,
          bool PRE = false>
__global__ void __launch_bounds__(Tile<D, T0_, T1_, T2_>::NT, (UOcc<T, D, T0_, T1_, T2_, TAB, SK>::value))
    k_usweep(const __grid_constant__ Geo g, const __grid_constant__ Bufs<T> bf) {
    extern __shared__ __align__(128) unsigned char smem[];
    pdl_wait();
    usweep_body<T, D, T0_, T1_, T2_, TAB, NOSRC, SK, MIX, AL, PRE>(g, bf, blockIdx.x, blockIdx.y, smem);
}

template <typename T, int D, int T0_, int T1_, int T2_, bool TAB, bool NOSRC, bool SK = false, bool PRE = false>
__global__ void __launch_bounds__(Tile<D, T0_, T1_, T2_>::NT, (UOcc<T, D, T0_, T1_, T2_, TAB, SK>::value))
    k_usweep_batch(const Item* __restrict__ items, const Inst<T>* __restrict__ insts, const int* __restrict__ cur) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(16) unsigned char rec_mem[sizeof(URec<T>)];
    URec<T>& rec = *reinterpret_cast<URec<T>*>(rec_mem);
    pdl_wait();
    const Item it = items[blockIdx.x];
    rec.load(insts[it.inst], cur[it.inst] & 1);
    if (TAB && !rec.g.xal)
        usweep_body<T, D, T0_, T1_, T2_, TAB, NOSRC, SK, true, !TAB>(rec.g, rec.b, it.tile, it.grp, smem);
    else
        usweep_body<T, D, T0_, T1_, T2_, TAB, NOSRC, SK, true, true, PRE>(rec.g, rec.b, it.tile, it.grp, smem);
}

}  // namespace cdg
