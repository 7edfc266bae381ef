// bflux.cuh -- sweep B of the face-store shapes: the face fluxes, their moments
// and phi* of eq. phiupdate, every face formed once per tile.
//
// Per chunk a thread forms the fluxes of its cell's left faces from the stored
// reconstructed values (face equilibrium, the inverse of eq. phibar, xi_a phi:
// eq. flux), a tile's first threads those of the faces on its high sides, and
// the fluxes are exchanged through shared memory: a cell then takes both faces
// of every axis from there.  (Forming a face in both its cells needs no barrier
// but twice the equilibria and inversions; the exchange costs one barrier per
// chunk and 16 bytes in and 32 out of shared memory per face and field.)
// The next chunk's phi* and face values are loaded to registers before the
// barrier (FP32); two CTAs per SM keep enough of them in flight.  Under an
// acceleration the cell's own phi* and force come after the barrier: held over
// the faces' gradients they cost spills (256^2 cells x 32^2 velocities 0.96 -> 0.86 ms).
//
// A face's moments are summed by the thread that forms it as a left face; a
// face at the domain's high end by the thread beyond it, or (a tile that ends
// there) by the thread of the tile's high side, in shared memory.
//
// What bounds it: FP32 the 16 + 8 D B per point at 16 warps per SM; FP64 the FP64
// pipe.  Against forming a face in both its cells, ms per launch: FP32 3D 48^3 cells
// x 24^3 velocities 20.3 -> 13.7 (4.5 TB/s of its 40 B per point), 2D 256^2 x 32^2
// 0.432 -> 0.392 (5.5 TB/s of 32 B), under an acceleration 1.70 -> 0.86; FP64 2D
// 256^2 x 32^2 8.70 -> 6.59, 1D 8192 x 129 0.246 -> 0.173.
#pragma once

#include "usweep.cuh"

namespace cdg {

template <typename T, int D, int T0_, int T1_, int T2_, bool SK, bool XF>
struct BSmem {
    using TL = Tile<D, T0_, T1_, T2_, 1>;
    static constexpr int NT = TL::NT, NX = TL::NPL, NF = D * NT + NX;     // left faces by thread, then the high sides
    static_assert(NX <= NT, "one high-side face per thread");
    static constexpr int NFV = XF ? 2 : EqPack<T, D, SK>::NV, NOV = EqPack<T, D, SK>::NV;
    static constexpr int RING = 8;
    static constexpr size_t rec_bytes = 4 * kChunkInts + kChunkVecs * sizeof(V4<T>);
    static constexpr size_t rs_bytes = (size_t)NX * (2 + D) * sizeof(Kahan<T>);
    static constexpr size_t base = ((size_t)NFV * NF + (size_t)NOV * NT + 1) * sizeof(V4<T>) + (rs_bytes + 15) / 16 * 16 + RING * rec_bytes;
    static constexpr size_t ff = (size_t)2 * NF * sizeof(V4<T>);
    // the exchange is double-buffered (one barrier per chunk) where two CTAs per SM still fit
    static constexpr bool DB = base + 2 * ff <= (size_t)113 * 1024;
    static constexpr size_t bytes = base + (DB ? 2 : 1) * ff;
};
template <typename T, int D, int T0_, int T1_, int T2_, bool SK, bool XF>
struct BOcc {
    static constexpr int NT = T0_ * T1_ * T2_;
    static constexpr int by_smem = (int)((228 * 1024) / (BSmem<T, D, T0_, T1_, T2_, SK, XF>::bytes + 1024));
    static constexpr int by_regs = 65536 / (NT * (sizeof(T) == 8 ? 168 : 128));
    static constexpr int v = by_smem < by_regs ? by_smem : by_regs;
    static constexpr int value = v < 1 ? 1 : (v > 8 ? 8 : v);
};

// ROWS (ACC): the velocity rows are whole chunks.  The other rows' force gradients,
// lane by lane, are in a kernel of their own: beside them the chunk-wide ones lack
// registers (24^3 cells x 12^3 velocities, FP32: sweep B 0.64 -> 0.76 ms).
template <typename T, int D, int T0_, int T1_, int T2_, bool SK, bool NOSRC, bool XF, bool ACC = false, bool PERS = false,
          bool ROWS = true>
__device__ __forceinline__ void bflux_body(const Geo& g, const Bufs<T>& bf, int tile, int grp, unsigned char* smem) {
    using BS = BSmem<T, D, T0_, T1_, T2_, SK, XF>;
    using TL = typename BS::TL;
    using K = Pk<T>;
    constexpr int NM = 2 + D, NT = TL::NT, NF = BS::NF, NX = BS::NX, N8 = 2 * VC, NFV = BS::NFV, NOV = BS::NOV;
    constexpr bool NC = !PERS, PF = sizeof(T) == 4;
    constexpr bool NOZ = SK || NOSRC;
    K* const FC = reinterpret_cast<K*>(smem);               // [NFV][NF] face constants
    K* const OC = FC + (size_t)NFV * NF;                    // [NOV][NT] constants of the own cell
    K* const LC = OC + (size_t)NOV * NT;                    // 1/dx_a, -dt (converted once: conversions use the FP64 pipe)
    K* const FF = LC + 1;                                   // [1 or 2][2][NF] face fluxes
    unsigned char* const tail = reinterpret_cast<unsigned char*>(FF + (BS::DB ? 4 : 2) * NF);
    Kahan<T>* const RS = reinterpret_cast<Kahan<T>*>(tail);  // [NM][NX] moments of the domain's high end
    unsigned char* const ring = tail + (BS::rs_bytes + 15) / 16 * 16;
    const int t = threadIdx.x;
    int org[3] = {0, 0, 0};                                  // (this sweep's own tiling, x fastest)
    {
        const int tx = (g.n[0] + TL::T0 - 1) / TL::T0, ty = D >= 2 ? (g.n[1] + TL::T1 - 1) / TL::T1 : 1;
        org[0] = tile % tx * TL::T0;
        if (D >= 2) org[1] = tile / tx % ty * TL::T1;
        if (D >= 3) org[2] = tile / tx / ty * TL::T2;
    }
    const int j0 = (int)((long long)grp * g.NVT / g.G), j1 = (int)((long long)(grp + 1) * g.NVT / g.G);
    const int la[3] = {t % TL::T0, D >= 2 ? (t / TL::T0) % TL::T1 : 0, D >= 3 ? t / (TL::T0 * TL::T1) : 0};
    const int qa[3] = {org[0] + la[0], org[1] + la[1], org[2] + la[2]};
    bool valid = true;
#pragma unroll
    for (int a = 0; a < D; ++a) valid = valid && qa[a] < g.n[a];

    // the faces this thread forms: bit a its left face of axis a, bit 3 a face of
    // a high side (axis xa; bit 4: of the domain's end, with its moments)
    int mine = 0, ff[D], xa = 0, xf = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        bool ok = qa[a] <= g.n[a];
#pragma unroll
        for (int b = 0; b < D; ++b) ok = ok && (b == a || qa[b] < g.n[b]);
        mine |= (ok ? 1 : 0) << a;
        ff[a] = ok ? (int)face_index(g, a, qa) : 0;
    }
    if (t < NX) {
#pragma unroll
        for (int b = 1; b < D; ++b) xa += t >= TL::poff(b) ? 1 : 0;
        const int p = t - TL::poff(xa);
        int q[3] = {org[0], org[1], org[2]};
        if (xa == 0) { q[0] += TL::T0; q[1] += p % TL::T1; q[2] += p / TL::T1; }
        else if (xa == 1) { q[0] += p % TL::T0; q[1] += TL::T1; q[2] += p / TL::T0; }
        else { q[0] += p % TL::T0; q[1] += p / TL::T0; q[2] += TL::T2; }
        bool ok = true;
#pragma unroll
        for (int b = 0; b < D; ++b) ok = ok && q[b] < g.n[b] + (b == xa ? 1 : 0);
        if (ok) {
            mine |= 8 | (q[xa] == g.n[xa] ? 16 : 0);
            xf = (int)face_index(g, xa, q);
        }
    }
    if (j0 >= j1) return;
    const int cell = valid ? (int)cell_index(g, qa) : 0;
    // chunk records, staged ahead as in sweep A
    auto rec_int = [&](int j) { return reinterpret_cast<const int*>(ring + (size_t)(j & (BS::RING - 1)) * BS::rec_bytes); };
    auto rec_val = [&](int j) {
        return reinterpret_cast<const K*>(ring + (size_t)(j & (BS::RING - 1)) * BS::rec_bytes + 4 * kChunkInts);
    };
    auto fetch_rec = [&](int j) {
        constexpr int NQ = (int)(BS::rec_bytes / 16);
        static_assert(NQ <= NT, "one 16-byte piece per thread");
        if (t < NQ && j < j1) {
            const char* from = t < 4 ? reinterpret_cast<const char*>(bf.cint + (size_t)kChunkInts * j) + 16 * t
                                     : reinterpret_cast<const char*>(bf.crec + (size_t)(kChunkVecs * VC) * j) + 16 * (t - 4);
            cp_async16(ring + (size_t)(j & (BS::RING - 1)) * BS::rec_bytes + 16 * t, from);
        }
        cp_async_commit();
    };
    K fg[D], fb[D], og, ob, xg, xb;
    auto load = [&](int vt) {
        const unsigned long long v = (unsigned)vt;
        if (!ACC && valid) load_gb<NC>(bf.phi_in + (v * (unsigned)g.Nc + (unsigned)cell) * N8, og, ob);
#pragma unroll
        for (int a = 0; a < D; ++a)
            if ((mine >> a) & 1) load_gb<NC>(bf.face[a] + (v * (unsigned)g.nf[a] + (unsigned)ff[a]) * N8, fg[a], fb[a]);
        if (mine & 8) load_gb<NC>(bf.face[xa] + (v * (unsigned)g.nf[xa] + (unsigned)xf) * N8, xg, xb);
    };
    // the first records and chunk are in flight while the constants are staged
    const int vt0 = __ldg(bf.cint + (size_t)kChunkInts * j0);
    for (int i = 0; i < 3; ++i) fetch_rec(j0 + i);
    if (PF) load(vt0);
    auto stage_face = [&](int a, int f, int s) {            // constants of face f of axis a to slot s
        const FaceC<T>& fs = bf.facec[a][f];
        T cst[4 * NFV];
#pragma unroll
        for (int i = 0; i < 4 * NFV; ++i) cst[i] = T(0);
#pragma unroll
        for (int b = 0; b < D; ++b) cst[b] = fs.u[b];
        constexpr int o = XF ? 3 : D + 2;
        if constexpr (!XF) {
            cst[D + 0] = fs.cexp;
            cst[D + 1] = fs.pref;
        }
        cst[XF ? 3 : D + 3] = fs.hu2;
        cst[XF ? 4 : D + 2] = fs.eb;
        cst[o + 2] = fs.al_g;
        cst[o + 3] = fs.al_b;
        cst[o + 4] = fs.gam_b;
        if constexpr (SK) {
#pragma unroll
            for (int b = 0; b < D; ++b) cst[D + 7 + b] = fs.sq[b];
            cst[2 * D + 7] = fs.e2;
        }
#pragma unroll
        for (int i = 0; i < NFV; ++i) {
            const T x[VC] = {cst[4 * i], cst[4 * i + 1], cst[4 * i + 2], cst[4 * i + 3]};
            FC[i * NF + s] = K::of(x);
        }
    };
#pragma unroll
    for (int a = 0; a < D; ++a)
        if ((mine >> a) & 1) stage_face(a, ff[a], a * NT + t);
    if (mine & 8) stage_face(xa, xf, D * NT + t);
    if (valid) {
        // phi* = eq + um (phi - eq) [+ usrc Z (g - g_eq)] - dt dF with phi - eq = fa (phi* - eq)
        const CellC<T>& cs = bf.cellc[cell];
        T cst[4 * NOV];
#pragma unroll
        for (int i = 0; i < 4 * NOV; ++i) cst[i] = T(0);
#pragma unroll
        for (int b = 0; b < D; ++b) cst[b] = cs.u[b];
        cst[D + 0] = cs.cexp;
        cst[D + 1] = cs.pref;
        cst[D + 2] = cs.eb;
        cst[D + 3] = cs.hu2;
        cst[D + 4] = Ar<T>::mul(cs.um_g, cs.fa_g);
        cst[D + 5] = Ar<T>::mul(cs.um_b, cs.fa_b);
        cst[D + 6] = Ar<T>::mul(cs.usrc, cs.fa_g);
        if constexpr (SK) {
#pragma unroll
            for (int b = 0; b < D; ++b) cst[D + 7 + b] = cs.sq[b];
            cst[2 * D + 7] = cs.e2;
        }
#pragma unroll
        for (int i = 0; i < NOV; ++i) {
            const T x[VC] = {cst[4 * i], cst[4 * i + 1], cst[4 * i + 2], cst[4 * i + 3]};
            OC[i * NT + t] = K::of(x);
        }
    }
    if (t < NX)
#pragma unroll
        for (int m = 0; m < NM; ++m) RS[m * NX + t].zero();

    T hL = SK ? g.consts<T>().ceb : T(0);
    if (SK) keep(hL);
    if (t == 0) {
        const T x[VC] = {(T)g.idx[0], (T)g.idx[1], (T)g.idx[2], (T)-g.dt};
        *LC = K::of(x);
    }
    // the acceleration (a specular wall face leaves out its normal component: bit a
    // of `wall` the left face of axis a, bit 3 the high side's), over twice the spacing
    T acc_[ACC ? D : 1], cacc[ACC ? D : 1], hh = T(0);
    int wall = 0;
    if constexpr (ACC) {
        hh = g.consts<T>().hh;
#pragma unroll
        for (int b = 0; b < D; ++b) {
            acc_[b] = (T)g.acc[b];
            cacc[b] = (T)(g.acc[b] / (2.0 * g.dxi[b]));
            wall |= ((qa[b] == 0 && g.bc[b][0] == BC_SPECULAR) || (qa[b] == g.n[b] && g.bc[b][1] == BC_SPECULAR) ? 1 : 0) << b;
        }
        wall |= (mine & 16) && g.bc[xa][1] == BC_SPECULAR ? 8 : 0;
    }
    // -acc . grad_xi of the values of face f (axis a) at chunk j (its own: pg, pb):
    // central differences, zero beyond the velocity grid's ends.  Velocity rows of
    // whole chunks: the neighbours along an axis > 0 are the same lanes of another
    // chunk, along axis 0 the next lanes.
    auto gradient = [&](int a, long long f, int j, bool nowall, const K& pg, const K& pb, K& gg, K& gb) {
        const int* const ri = rec_int(j);
        const T* const base = bf.face[a] + (unsigned long long)(unsigned)f * N8;
        const unsigned long long nf8 = (unsigned long long)(unsigned)g.nf[a] * N8;
        const int vt = ri[0];
        gg = gb = K::bc(T(0));
        if constexpr (ROWS) {
            const int n0c = g.nv1[0] / VC;
#pragma unroll
            for (int b = 0; b < D; ++b) {
                if (g.acc[b] == 0.0 || (b == a && nowall)) continue;
                const int k = b == 0 ? ri[4] : (b == 1 ? ri[8] - g.xrow[1] : ri[12] - g.xrow[2]);
                const int st = b == 0 ? 1 : (b == 1 ? n0c : n0c * g.nv1[1]);
                K ug = K::bc(T(0)), ub = ug, dg = ug, db = ug;               // the chunk above and below
                if (k + (b == 0 ? VC : 1) < g.nv1[b]) load_gb<NC>(base + (unsigned)(vt + st) * nf8, ug, ub);
                if (k >= 1) load_gb<NC>(base + (unsigned)(vt - st) * nf8, dg, db);
                if (b == 0) {
                    auto shift = [](const K& c, K& up, K& dn) {
                        T cv[VC], u[VC], d[VC];
                        c.get(cv);
                        up.get(u);
                        dn.get(d);
                        const T uu[VC] = {cv[1], cv[2], cv[3], u[0]}, dd[VC] = {d[VC - 1], cv[0], cv[1], cv[2]};
                        up = K::of(uu);
                        dn = K::of(dd);
                    };
                    shift(pg, ug, dg);
                    shift(pb, ub, db);
                }
                const K c = K::bc(-cacc[ACC ? b : 0]);
                gg = fma4(c, ug - dg, gg);
                gb = fma4(c, ub - db, gb);
                asm volatile("" ::: "memory");          // one axis's neighbours at a time: registers
            }
        } else {
            // lane by lane: the record holds each lane's node along every axis
            T x[VC], y[VC];
#pragma unroll
            for (int v = 0; v < VC; ++v) {
                x[v] = y[v] = T(0);
                if (ri[4 + v] < 0) continue;                                 // padding
                const int i = vt * VC + v;
#pragma unroll
                for (int b = 0; b < D; ++b) {
                    if (g.acc[b] == 0.0 || (b == a && nowall)) continue;
                    const int k = b == 0 ? ri[4 + v] : (b == 1 ? ri[8 + v] - g.xrow[1] : ri[12 + v] - g.xrow[2]);
                    const int st = b == 0 ? 1 : (b == 1 ? g.nv1[0] : g.nv1[0] * g.nv1[1]);
                    T ug = T(0), ub = T(0), dg = T(0), db = T(0);
                    auto at = [&](int n) { return base + (unsigned)(n / VC) * nf8 + (n % VC); };
                    if (k + 1 < g.nv1[b]) {
                        ug = at(i + st)[0];
                        ub = at(i + st)[VC];
                    }
                    if (k >= 1) {
                        dg = at(i - st)[0];
                        db = at(i - st)[VC];
                    }
                    x[v] = fma(-cacc[ACC ? b : 0], ug - dg, x[v]);
                    y[v] = fma(-cacc[ACC ? b : 0], ub - db, y[v]);
                }
            }
            gg = K::of(x);
            gb = K::of(y);
        }
    };
    // L2 hints: the first thread of each row of the tile asks for the row's data
    // two chunks ahead (its cells, its left faces, on the tile's high sides the
    // right ones); rows are contiguous in every layout
    const int nrow = min(TL::T0, g.n[0] - org[0]);
    const bool lead = la[0] == 0 && nrow > 0;
    auto hint = [&](int vt) {
        constexpr int RB = N8 * (int)sizeof(T);
        const unsigned long long v = (unsigned)vt;
        if (valid) prefetch_l2(bf.phi_in + (v * (unsigned)g.Nc + (unsigned)cell) * N8, nrow * RB);
#pragma unroll
        for (int a = 0; a < D; ++a)
            if ((mine >> a) & 1)
                prefetch_l2(bf.face[a] + (v * (unsigned)g.nf[a] + (unsigned)ff[a]) * N8, (nrow + (a == 0 ? 1 : 0)) * RB);
    };
    Sums<T, D * NM> acc;
    acc.zero();
    // the equilibrium of place `item` of a factor table from the rows of chunk j
    auto table = [&](const T* X, long long n, long long item, int j) {
        const int* const ri = rec_int(j);
        T y[VC];
        const unsigned long long nn = (unsigned)n, it = (unsigned)item;
        if (g.xal) {
            const T* p0 = X + (unsigned)ri[4] * nn + VC * it;
            const T x1 = __ldg(X + (unsigned)ri[2] * nn + it);
            T x2 = T(1);
            if constexpr (D == 3) x2 = __ldg(X + (unsigned)ri[3] * nn + it);
            return ldg4(p0) * K::bc(lean_pair<T, D>(x1, x2));
        }
#pragma unroll
        for (int v = 0; v < VC; ++v) {
            const int r0 = ri[4 + v];
            y[v] = T(0);
            if (r0 < 0) continue;
            T z = __ldg(X + (unsigned)ri[8 + v] * nn + it);
            if constexpr (D == 3) z = lean_pair<T, D>(z, __ldg(X + (unsigned)ri[12 + v] * nn + it));
            y[v] = __ldg(X + ((unsigned)(r0 / VC) * nn + it) * VC + (r0 % VC)) * z;
        }
        return K::of(y);
    };
    cp_async_wait_all();
    __syncthreads();

    int buf = 0;
    for (int j = j0; j < j1; ++j) {
        const int vt = rec_int(j)[0];
        const K* const vr = rec_val(j);
        K* const Fg_ = FF + (size_t)(BS::DB ? buf : 0) * 2 * NF;
        K* const Fb_ = Fg_ + NF;
        if (!PF) load(vt);
        cp_async_wait_all();          // record j + 2, for its copier
        // one face: its flux to the exchange, its moments to sm
        auto face = [&](int a, int s, long long f, const K& pg, const K& pb, T* sm, bool mom) {
            T cst[4 * NFV];
#pragma unroll
            for (int i = 0; i < NFV; ++i) {
                T x[VC];
                FC[i * NF + s].get(x);
#pragma unroll
                for (int e = 0; e < 4; ++e) cst[4 * i + e] = x[e];
            }
            constexpr int oh = XF ? 3 : D + 3, oe = XF ? 4 : D + 2, oa = XF ? 5 : D + 4;
            K ge, be;
            if constexpr (XF) {
                ge = table(bf.xf[a], g.nf[a], f, j);
                be = (vr[3] + K::bc(cst[oe])) * ge;
            } else {
                eq4<T, D, SK>(cst, vr, vr[3], hL, ge, be);
            }
            const K dg = pg - ge;
            K gf = fma4(K::bc(cst[oa]), dg, ge), gg, gb;
            const bool nowall = ACC && ((wall >> (s >= D * NT ? 3 : a)) & 1);
            if constexpr (ACC) {
                gradient(a, f, j, nowall, pg, pb, gg, gb);
                gf = fma4(K::bc(Ar<T>::mul(cst[oa], hh)), gg, gf);
            }
            K bv = fma4(K::bc(cst[oa + 1]), pb - be, be);
            if constexpr (!NOZ) {
                K z = K::bc(-cst[oh]);
#pragma unroll
                for (int b = 0; b < D; ++b) z = fma4(vr[b], K::bc(cst[b]), z);
                bv = fma4(K::bc(cst[oa + 2]) * z, gf - ge, bv);
            }
            if constexpr (ACC) {
                K ax = K::bc(T(0));
#pragma unroll
                for (int b = 0; b < D; ++b)
                    if (!(b == a && nowall)) ax = fma4(K::bc(acc_[b]), vr[b], ax);
                bv = fma4(K::bc(Ar<T>::mul(cst[oa + 1], hh)), fma4(ax, gf, gb), bv);
            }
            const K xi = vr[a], Fg = xi * gf, Fb = xi * bv;
            if (mom) {
                const K w = vr[7], wg = w * Fg;
                sm[0] = sum4(wg);
#pragma unroll
                for (int b = 0; b < D; ++b) sm[1 + b] = dot4(vr[b], wg);
                sm[1 + D] = dot4(w, Fb);
            }
            Fg_[s] = Fg;             // (last: the record's loads above are shared)
            Fb_[s] = Fb;
        };
        T sm[D * NM];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            if ((mine >> a) & 1) {
                face(a, a * NT + t, ff[a], fg[a], fb[a], sm + a * NM, true);
            } else {
#pragma unroll
                for (int m = 0; m < NM; ++m) sm[a * NM + m] = T(0);
            }
            acc.add(sm, a * NM, (a + 1) * NM);
        }
        if (mine & 8) {
            T sx[NM];
            const bool end = (mine & 16) != 0;
            if (D == 1 || xa == 0) face(0, D * NT + t, xf, xg, xb, sx, end);
            else if (D == 2 || xa == 1) face(D >= 2 ? 1 : 0, D * NT + t, xf, xg, xb, sx, end);
            else face(D - 1, D * NT + t, xf, xg, xb, sx, end);
            if (end)
#pragma unroll
                for (int m = 0; m < NM; ++m) {
                    Kahan<T> k = RS[m * NX + t];
                    k.add(sx[m]);
                    RS[m * NX + t] = k;
                }
        }
        K gs, bs;
        if constexpr (!ACC) gs = og, bs = ob;
        if (PF && j + 1 < j1) load(rec_int(j + 1)[0]);      // in flight over the rest of this chunk
        fetch_rec(j + 3);
        __syncthreads();
        if (TL::T0 >= 32 && lead && j + 2 < j1) hint(rec_int(j + 2)[0]);
        if (valid) {
            const unsigned long long own = ((unsigned long long)(unsigned)vt * (unsigned)g.Nc + (unsigned)cell) * N8;
            if constexpr (ACC) load_gb<NC>(bf.phi_in + own, gs, bs);
            K dFg, dFb;
            T lc[VC];
            LC->get(lc);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const int st = a == 0 ? 1 : (a == 1 ? TL::T0 : TL::T0 * TL::T1), s0 = a * NT + t;
                const int s1 = la[a] < TL::tdim(a) - 1 ? s0 + st : D * NT + TL::poff(a) + TL::plane_pos(a, la);
                const K ix = K::bc(lc[a]);
                const K eg = Fg_[s1] - Fg_[s0], eb = Fb_[s1] - Fb_[s0];
                dFg = a == 0 ? ix * eg : fma4(ix, eg, dFg);
                dFb = a == 0 ? ix * eb : fma4(ix, eb, dFb);
            }
            if constexpr (ACC) {     // + dt F^n (eq. phiupdate's source, rectangle rule)
                K fgs, fbs;
                load_gb<NC>(bf.force + own, fgs, fbs);
                dFg = dFg - fgs;
                dFb = dFb - fbs;
            }
            T cst[4 * NOV];
#pragma unroll
            for (int i = 0; i < NOV; ++i) {
                T x[VC];
                OC[i * NT + t].get(x);
#pragma unroll
                for (int e = 0; e < 4; ++e) cst[4 * i + e] = x[e];
            }
            K ge, be;
            if constexpr (XF) {
                ge = table(bf.xc, g.Nc, cell, j);
                be = (vr[3] + K::bc(cst[D + 2])) * ge;
            } else {
                eq4<T, D, SK>(cst, vr, vr[3], hL, ge, be);
            }
            const K dg = gs - ge;
            const K ng = fma4(K::bc(lc[3]), dFg, fma4(K::bc(cst[D + 4]), dg, ge));
            K nb = fma4(K::bc(cst[D + 5]), bs - be, be);
            if constexpr (!NOZ) {
                K z = K::bc(-cst[D + 3]);
#pragma unroll
                for (int b = 0; b < D; ++b) z = fma4(vr[b], K::bc(cst[b]), z);
                nb = fma4(K::bc(cst[D + 6]) * z, dg, nb);
            }
            nb = fma4(K::bc(lc[3]), dFb, nb);
            store_gb(bf.phi_out + ((unsigned long long)(unsigned)vt * (unsigned)g.Nc + (unsigned)cell) * N8, ng, nb);
        }
        if (BS::DB) buf ^= 1;
        else __syncthreads();                               // the fluxes are read
    }
#pragma unroll
    for (int a = 0; a < D; ++a)
        if ((mine >> a) & 1)
#pragma unroll
            for (int m = 0; m < NM; ++m) bf.mf[a][((size_t)grp * NM + m) * (size_t)g.nf[a] + ff[a]] = acc.value(a * NM + m);
    if (mine & 16)
#pragma unroll
        for (int m = 0; m < NM; ++m) bf.mf[xa][((size_t)grp * NM + m) * (size_t)g.nf[xa] + xf] = RS[m * NX + t].value();
}

template <typename T, int D, int T0_, int T1_, int T2_, bool SK, bool NOSRC, bool XF, bool ACC = false, bool ROWS = true>
__global__ void __launch_bounds__(Tile<D, T0_, T1_, T2_>::NT, (BOcc<T, D, T0_, T1_, T2_, SK, XF>::value))
    k_bflux(const __grid_constant__ Geo g, const __grid_constant__ Bufs<T> bf) {
    extern __shared__ __align__(128) unsigned char smem[];
    pdl_wait();
    bflux_body<T, D, T0_, T1_, T2_, SK, NOSRC, XF, ACC, false, ROWS>(g, bf, blockIdx.x, blockIdx.y, smem);
}

template <typename T, int D, int T0_, int T1_, int T2_, bool SK, bool NOSRC, bool XF, bool ACC = false>
__global__ void __launch_bounds__(Tile<D, T0_, T1_, T2_>::NT, (BOcc<T, D, T0_, T1_, T2_, SK, XF>::value))
    k_bflux_batch(const Item* __restrict__ items, const Inst<T>* __restrict__ insts, const int* __restrict__ cur) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(16) unsigned char rec_mem[sizeof(URec<T>)];
    URec<T>& rec = *reinterpret_cast<URec<T>*>(rec_mem);
    pdl_wait();
    const Item it = items[blockIdx.x];
    rec.load(insts[it.inst], cur[it.inst] & 1);
    if (ACC && !rec.g.xal)
        bflux_body<T, D, T0_, T1_, T2_, SK, NOSRC, XF, ACC, false, !ACC>(rec.g, rec.b, it.tile, it.grp, smem);
    else
        bflux_body<T, D, T0_, T1_, T2_, SK, NOSRC, XF, ACC>(rec.g, rec.b, it.tile, it.grp, smem);
}

// The pre-pass of an acceleration along one axis on velocity rows of whole
// chunks (prep_body's results): a thread per cell walks a line of the forced
// axis's nodes, consecutive chunks in sweep B's order, with phi^n of the chunk
// before, this and the next one in registers, so every value is read and every
// equilibrium formed once instead of three times (256^2 x 32^2: the pre-pass
// and sweep A 0.94 -> 0.76 ms).
template <typename T, int D>
__global__ void __launch_bounds__(kPrepCells) k_prep_line(const __grid_constant__ Geo g, const __grid_constant__ Bufs<T> bf,
                                                          int ax, int len) {
    using K = Pk<T>;
    pdl_wait();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.Nc) return;
    constexpr int N8 = 2 * VC;
    const CellC<T> cs = bf.cellc[c];
    const T hh = g.consts<T>().hh, cax = (T)(g.acc[ax] / (2.0 * g.dxi[ax])), aT = (T)g.acc[ax];
    const int j0 = blockIdx.y * len;
    auto vt_of = [&](int j) { return __ldg(bf.cint + (size_t)kChunkInts * j); };
    auto at = [&](int vt) { return ((unsigned long long)(unsigned)vt * (unsigned)g.Nc + (unsigned long long)c) * N8; };
    // g_eq, b_eq, phi* and phi^n of the chunk with record j from its phi* (gs, bs)
    struct Chunk1 {
        K ge, be, gs, bs, g, b;
    };
    auto form = [&](int j, const K& gs, const K& bs) {
        const T* vr = bf.crec + (size_t)(kChunkVecs * VC) * j;
        Chunk1 o;
        K c2;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const K d = ldg4(vr + a * VC) - K::bc(cs.u[a]);
            c2 = a == 0 ? d * d : fma4(d, d, c2);
        }
        o.ge = K::bc(cs.pref) * expo4<T>(K::bc(cs.cexp) * c2);
        o.be = (ldg4(vr + 3 * VC) + K::bc(cs.eb)) * o.ge;
        o.gs = gs;
        o.bs = bs;
        o.g = fma4(K::bc(cs.fa_g), gs, K::bc(cs.fb_g) * o.ge);
        o.b = fma4(K::bc(cs.fa_b), bs, K::bc(cs.fb_b) * o.be);
        return o;
    };
    const K zero = K::bc(T(0));
    K pg = zero, pb = zero, lg, lb;                  // phi^n of the chunk before; the loads in flight
    load_gb<true>(bf.phi_in + at(vt_of(j0)), lg, lb);
    Chunk1 cur = form(j0, lg, lb);
    if (len > 1) load_gb<true>(bf.phi_in + at(vt_of(j0 + 1)), lg, lb);
    for (int k = 0; k < len; ++k) {
        const int j = j0 + k;
        Chunk1 nxt;
        nxt.g = nxt.b = zero;
        if (k + 1 < len) {
            const K gs = lg, bs = lb;
            if (k + 2 < len) load_gb<true>(bf.phi_in + at(vt_of(j + 2)), lg, lb);
            nxt = form(j + 1, gs, bs);
        }
        K ug = nxt.g, ub = nxt.b, dg = pg, db = pb;
        if (ax == 0) {                               // neighbours along axis 0: the next lanes
            auto shift = [](const K& m, K& up, K& dn) {
                T cv[VC], u[VC], d[VC];
                m.get(cv);
                up.get(u);
                dn.get(d);
                const T uu[VC] = {cv[1], cv[2], cv[3], u[0]}, dd[VC] = {d[VC - 1], cv[0], cv[1], cv[2]};
                up = K::of(uu);
                dn = K::of(dd);
            };
            shift(cur.g, ug, dg);
            shift(cur.b, ub, db);
        }
        const K fg = K::bc(-cax) * (ug - dg);
        K fb = K::bc(-cax) * (ub - db);
        const T* vr = bf.crec + (size_t)(kChunkVecs * VC) * j;
        K z = K::bc(-cs.hu2);
#pragma unroll
        for (int a = 0; a < D; ++a) z = fma4(ldg4(vr + a * VC), K::bc(cs.u[a]), z);
        fb = fma4(K::bc(aT) * ldg4(vr + ax * VC), cur.g, fb);
        const K dgq = cur.gs - cur.ge;
        K og = fma4(K::bc(cs.kp_g), dgq, cur.ge);
        K ob = fma4(K::bc(cs.kp_s) * z, dgq, fma4(K::bc(cs.kp_b), cur.bs - cur.be, cur.be));
        og = fma4(K::bc(hh), fg, og);
        ob = fma4(K::bc(hh), fb, ob);
        const unsigned long long ad = at(vt_of(j));
        store_gb(bf.phibar + ad, og, ob);
        store_gb(bf.force + ad, fg, fb);
        pg = cur.g;
        pb = cur.b;
        cur = nxt;
    }
}

}  // namespace cdg
