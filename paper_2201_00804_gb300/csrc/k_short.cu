// Exchange-repulsion (Technical Appendix: S^2/R and S^2/R^2 overlap terms
// over bond-bond, bond-lone pair and lone pair-lone pair pairs), dispersion
// (C6/C8/C10 with damping) and exchange-dispersion.
//
// One lane evaluates everything between two molecules, each pair once: the
// 16 repulsion items and 25 dispersion point pairs share the nine atom
// distances, unit vectors and overlap exponentials, every cosine is one
// product of unit vectors, and the gradients of both molecules' points come
// from the same terms: some 5,500 instructions a pair.  (Item by item from both
// sides, as queues of equal items, a pair took 25,000.)  Of a pair (i, j) of the
// full list one side owns the work, by the parity of i + j, so that every
// molecule owns about half of its neighbours.
//
// A warp walks the lists of a few consecutive molecules, queues the owned
// pairs with anything inside the cutoff and evaluates them 32 at a time,
// across molecules.  The gradients of j's points go to a row of j's inbox, and
// k_short_gather adds up each molecule's rows.  In a box the gradients of i's
// points are summed in shared memory until i is done, and rows are taken by a
// counter; in the gas phase, where molecules have few neighbours, i's go to
// rows as well, and a pair's rows are fixed by its places in the two lists.
//
// Bound in FP32 by the latency of one lane's long chains at two warps a
// quarter of an SM (255 registers, no spill; issue slots 55% busy): with 10,
// 12 and 16 blocks an SM, at 168, 168 and 128 registers with spills, 32,000 waters (rc 9) took
// 914, 912 and 1126 us against 762.  In FP64 bound by the FP64
// pipe (255 registers, 1.9 to 2.1 KB a thread spilled); repulsion and dispersion go to different warps,
// which fills the chip better.
// All launches together, before (item queues) and now: 32,000 waters 1815 and
// 762 us, 4,096 waters 279 and 135, 4,096 clusters of 17 waters 930 and 408, 216 waters in FP64
// 486 and 266, 824 waters in FP64 clusters 592 and 232.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "sibfa_internal.cuh"

namespace sibfa {

namespace {

constexpr int BOX_ROW = 16, GAS_ROW = 24;   // an inbox row: 15 gradients; in the gas phase 3 energies as two parts each
// resident one-warp blocks an SM in FP32
constexpr int SHORT_BLOCKS = 8;

// Points of a molecule and the valence factors 1 - q/N_val of O, H1, H2
template <typename R>
struct Water {
    V3<R> P[5];    // O, H1, H2, LP1, LP2
    R cf[3];
};

// One centre pair (x, y) of a repulsion item: p = u.e and q = v.e of the unit p
// directions u at x and v at y with the unit vector e from x to y; SX, SY are
// the signs of the p orbitals' directions along u and v.  With kinds KX, KY
// the overlap is A + B cx + C cy + D cx cy of the cosines cx = SX p, cy = -SY q.
template <typename R, int KX, int KY, int SX, int SY>
struct Centres {
    R o, dp, dq;   // overlap and its derivatives in p and q
    __device__ __forceinline__ Centres(const Scal<R> &S, R p, R q) {
        const R *c = S.rep_o[KX][KY];
        dq = R(-SY) * c[2] + R(-SX * SY) * c[3] * p;
        dp = R(SX) * c[1] + R(-SX * SY) * c[3] * q;
        o = c[0] + R(SX) * c[1] * p + dq * q;
    }
    // given w1 = dE/dO1 S1, w2 = dE/dO2 S2: adds dE/dp, dE/dq and the rest of dE/d(e r) along e
    __device__ __forceinline__ void back(const KParams &P, R w1, R w2, R p, R q, R ri, R &gp, R &gq, R &gr) const {
        const R w = w1 + w2, a = w * dp, b = w * dq;
        gp += a;
        gq += b;
        gr -= o * (w1 * cval<R>(P.rep_k1[KX][KY]) + w2 * cval<R>(P.rep_k2[KX][KY])) + ri * (a * p + b * q);
    }
};

// E = pref (C1 O1^2 / r + C2 O2^2 / r^2) from ri = 1/r: returns E and dE/dO1,
// dE/dO2 and h = (dE/dr) / r.
template <typename R>
__device__ __forceinline__ R rep_energy(const Scal<R> &S, R pref, R O1, R O2, R ri, R &e1, R &e2, R &h) {
    const R pr = pref * ri, a = pr * S.rep_c1 * O1, b = pr * ri * S.rep_c2 * O2;
    e1 = R(2) * a;
    e2 = R(2) * b;
    const R E1 = a * O1, E2 = b * O2;
    h = -(E1 + R(2) * E2) * ri * ri;
    return E1 + E2;
}

template <typename R>
__device__ __forceinline__ void swap_(R &a, R &b) {
    const R t = a;
    a = b;
    b = t;
}
template <typename R>
__device__ __forceinline__ V3<R> unit(V3<R> v, R &il) {
    il = rsqrt_(dot(v, v));
    return il * v;
}
// gradient of a unit vector n = v / |v| (il = 1 / |v|) to that of v
template <typename R>
__device__ __forceinline__ V3<R> unit_back(V3<R> g, V3<R> n, R il) {
    return il * (g - dot(g, n) * n);
}
template <typename R>
__device__ __forceinline__ void fma3(V3<R> &a, R s, V3<R> v) {
    a.x += s * v.x;
    a.y += s * v.y;
    a.z += s * v.z;
}

// Exchange-repulsion of molecules i (O at the origin, points A) and j (B).
// Items: bond-bond, bond-lone pair, lone pair-bond (lone pairs act as
// pseudo-atoms at their O) and lone pair-lone pair.  Everything about an atom
// pair (unit vector, exponentials) is computed once, the items add to scalar
// sums by atom pair and direction, and these become vectors once.  The rolled
// loops take one bond (lone pair) of i each while the other's data wait.
template <typename R, bool PER>
__device__ __forceinline__ void rep_pair(const KParams &P, const Scal<R> &S, Water<R> &wi, const Water<R> &wj,
                                         V3<R> (&gi)[5], V3<R> (&gj)[5], Acc<R> &Er) {
    const R rc2 = S.rc2;
    const V3<R> z = mk(R(0), R(0), R(0));
    V3<R>(&A)[5] = wi.P;
    const V3<R>(&B)[5] = wj.P;
    auto mask = [&](R r2) { return !PER || r2 < rc2 ? R(1) : R(0); };
    const R cfl = R(1) - S.nlp * S.inv_nval_o;
    const R sgl = sqrt_(S.g_o * cfl), sg0 = sqrt_(S.g_o * wi.cf[0]);
    R sj[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) sj[k] = sqrt_((k ? S.g_h : S.g_o) * wj.cf[k]);
    // directions of j
    R im[2], il[2];
    V3<R> m[2], l[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        m[k] = unit(B[1 + k] - B[0], im[k]);
        l[k] = unit(B[3 + k] - B[0], il[k]);
    }
    // O of i with the atoms of j: e, 1/r, overlap exponentials; dot products with j's directions
    V3<R> e0[3];
    R r0[3], ri0[3], S10[3], S20[3];
#pragma unroll
    for (int y = 0; y < 3; ++y) {
        const V3<R> v = B[y] - A[0];
        const R vv = dot(v, v);
        ri0[y] = rsqrt_(vv);
        r0[y] = vv * ri0[y];
        e0[y] = ri0[y] * v;
        const R M = sg0 * sj[y];
        S10[y] = M * exp_(-mulc(r0[y], P.rep_k1[0][y ? 1 : 0]));
        S20[y] = M * exp_(-mulc(r0[y], P.rep_k2[0][y ? 1 : 0]));
    }
    const R q00[2] = {dot(m[0], e0[0]), dot(m[1], e0[0])}, q0c[2] = {dot(m[0], e0[1]), dot(m[1], e0[2])};
    const R ql0[2] = {dot(l[0], e0[0]), dot(l[1], e0[0])};
    const R sL = sg0 * sgl, L10 = sL * exp_(-mulc(r0[0], P.rep_k1[0][2])), L20 = sL * exp_(-mulc(r0[0], P.rep_k2[0][2]));
    // sums along e0[y] (gr), of m[c] with e0[0] and e0[1 + c] (gq00, gq0c), of l[k] with e0[0] (gl0)
    R gr0[3] = {R(0), R(0), R(0)}, gq00[2] = {R(0), R(0)}, gq0c[2] = {R(0), R(0)}, gl0[2] = {R(0), R(0)};
    V3<R> gm[2] = {z, z}, gl[2] = {z, z};   // gradients of j's directions
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {   // bonds of i
        R in_;
        const V3<R> n = unit(A[1] - A[0], in_);
        const V3<R> mb = R(0.5) * (A[0] + A[1]);
        const R sb = sqrt_(S.g_h * wi.cf[1]);
        V3<R> e[3];
        R ri[3], S1[3], S2[3], p[3], p0[3], rb = R(0);
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const V3<R> v = B[y] - A[1];
            const R vv = dot(v, v);
            ri[y] = rsqrt_(vv);
            const R r = vv * ri[y], M = sb * sj[y];
            e[y] = ri[y] * v;
            S1[y] = M * exp_(-mulc(r, P.rep_k1[1][y ? 1 : 0]));
            S2[y] = M * exp_(-mulc(r, P.rep_k2[1][y ? 1 : 0]));
            p[y] = dot(n, e[y]);
            p0[y] = dot(n, e0[y]);
            if (y == 0) rb = r;
        }
        const R sl = sb * sgl, L1 = sl * exp_(-mulc(rb, P.rep_k1[1][2])), L2 = sl * exp_(-mulc(rb, P.rep_k2[1][2]));
        R gr[3] = {R(0), R(0), R(0)}, gp[3] = {R(0), R(0), R(0)}, gp0[3] = {R(0), R(0), R(0)};
        V3<R> hb = z;   // gradient of the midpoint, halved
        V3<R> F0 = z;   // on B[0] from this bond's H: parts along j's directions
#pragma unroll
        for (int c = 0; c < 2; ++c) {   // bonds of j
            const V3<R> dm = mb - R(0.5) * (B[0] + B[1 + c]);
            const R d2 = dot(dm, dm), irm = rsqrt_(d2);
            const R qb0 = dot(m[c], e[0]), qbc = dot(m[c], e[1 + c]);
            const Centres<R, 0, 0, 1, 1> c00(S, p0[0], q00[c]);
            const Centres<R, 0, 1, 1, -1> c0c(S, p0[1 + c], q0c[c]);
            const Centres<R, 1, 0, -1, 1> cb0(S, p[0], qb0);
            const Centres<R, 1, 1, -1, -1> cbc(S, p[1 + c], qbc);
            const R O1 = c00.o * S10[0] + c0c.o * S10[1 + c] + cb0.o * S1[0] + cbc.o * S1[1 + c];
            const R O2 = c00.o * S20[0] + c0c.o * S20[1 + c] + cb0.o * S2[0] + cbc.o * S2[1 + c];
            R e1, e2, h;
            Er.add(rep_energy(S, mask(d2) * (S.occ * S.occ), O1, O2, irm, e1, e2, h));
            const V3<R> hd = (R(0.5) * h) * dm;
            hb = hb + hd;
            gj[0] = gj[0] - hd;
            gj[1 + c] = gj[1 + c] - hd;
            R gb0 = R(0), gbc = R(0);
            c00.back(P, e1 * S10[0], e2 * S20[0], p0[0], q00[c], ri0[0], gp0[0], gq00[c], gr0[0]);
            c0c.back(P, e1 * S10[1 + c], e2 * S20[1 + c], p0[1 + c], q0c[c], ri0[1 + c], gp0[1 + c], gq0c[c], gr0[1 + c]);
            cb0.back(P, e1 * S1[0], e2 * S2[0], p[0], qb0, ri[0], gp[0], gb0, gr[0]);
            cbc.back(P, e1 * S1[1 + c], e2 * S2[1 + c], p[1 + c], qbc, ri[1 + c], gp[1 + c], gbc, gr[1 + c]);
            fma3(gm[c], gb0, e[0]);
            fma3(gm[c], gbc, e[1 + c]);
            fma3(F0, ri[0] * gb0, m[c]);
            const V3<R> F = (ri[1 + c] * gbc) * m[c];
            gj[1 + c] = gj[1 + c] + F;
            gi[1] = gi[1] - F;
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {   // lone pairs of j
            const V3<R> dm = mb - B[3 + k];
            const R d2 = dot(dm, dm), irm = rsqrt_(d2);
            const R qb = dot(l[k], e[0]);
            const Centres<R, 0, 2, 1, 1> c0(S, p0[0], ql0[k]);
            const Centres<R, 1, 2, -1, 1> cb(S, p[0], qb);
            R e1, e2, h;
            Er.add(rep_energy(S, mask(d2) * (S.occ * S.nlp), c0.o * L10 + cb.o * L1, c0.o * L20 + cb.o * L2, irm, e1, e2, h));
            const V3<R> hd = (R(0.5) * h) * dm;
            hb = hb + hd;
            gj[3 + k] = gj[3 + k] - R(2) * hd;
            R gb = R(0);
            c0.back(P, e1 * L10, e2 * L20, p0[0], ql0[k], ri0[0], gp0[0], gl0[k], gr0[0]);
            cb.back(P, e1 * L1, e2 * L2, p[0], qb, ri[0], gp[0], gb, gr[0]);
            fma3(gl[k], gb, e[0]);
            fma3(F0, ri[0] * gb, l[k]);
        }
        // vectors: the bond's direction and the pairs of its H
        V3<R> gn = z, FO = z;   // FO: on O of i, minus the parts along n
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            fma3(gn, gp[y], e[y]);
            fma3(gn, gp0[y], e0[y]);
            V3<R> F = (ri[y] * gp[y]) * n;
            fma3(F, gr[y], e[y]);
            if (y == 0) F = F + F0;
            gi[1] = gi[1] - F;
            const V3<R> G = (ri0[y] * gp0[y]) * n;
            FO = FO + G;
            gj[y] = gj[y] + F + G;
        }
        const V3<R> t = unit_back(gn, n, in_);
        gi[0] = gi[0] + hb - FO - t;
        gi[1] = gi[1] + hb + t;
        swap_(A[1], A[2]);
        swap_(wi.cf[1], wi.cf[2]);
        swap_(gi[1], gi[2]);
    }
    // lone pairs of i (at its O) with the bonds and lone pairs of j
    R C1[2], C2[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const R s = sgl * sj[1 + c];
        C1[c] = s * exp_(-mulc(r0[1 + c], P.rep_k1[1][2]));
        C2[c] = s * exp_(-mulc(r0[1 + c], P.rep_k2[1][2]));
    }
    const R sO = sgl * sj[0], O10 = sO * exp_(-mulc(r0[0], P.rep_k1[0][2])), O20 = sO * exp_(-mulc(r0[0], P.rep_k2[0][2]));
    const R M = S.g_o * cfl;
    const R T1 = M * exp_(-mulc(r0[0], P.rep_k1[2][2])), T2 = M * exp_(-mulc(r0[0], P.rep_k2[2][2]));
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
        const V3<R> X = A[3];
        R ia;
        const V3<R> a = unit(X - A[0], ia);
        const R p0 = dot(a, e0[0]);
        R gp[3] = {R(0), R(0), R(0)};
        V3<R> gx = z, ga = z, g0 = z;   // gradients of X, of a, of O_i
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const V3<R> dm = X - R(0.5) * (B[0] + B[1 + c]);
            const R d2 = dot(dm, dm), irm = rsqrt_(d2);
            const R pc = dot(a, e0[1 + c]);
            const Centres<R, 2, 0, 1, 1> c0(S, p0, q00[c]);
            const Centres<R, 2, 1, 1, -1> cc(S, pc, q0c[c]);
            R e1, e2, h;
            Er.add(rep_energy(S, mask(d2) * (S.occ * S.nlp), c0.o * O10 + cc.o * C1[c], c0.o * O20 + cc.o * C2[c], irm, e1,
                              e2, h));
            const V3<R> hd = (R(0.5) * h) * dm;
            fma3(gx, R(2), hd);
            gj[0] = gj[0] - hd;
            gj[1 + c] = gj[1 + c] - hd;
            c0.back(P, e1 * O10, e2 * O20, p0, q00[c], ri0[0], gp[0], gq00[c], gr0[0]);
            cc.back(P, e1 * C1[c], e2 * C2[c], pc, q0c[c], ri0[1 + c], gp[1 + c], gq0c[c], gr0[1 + c]);
        }
        // angles toward the other lone pair's position
        R ix[2];
        const V3<R> xb = X - B[0];
        ix[0] = rsqrt_(dot(xb, xb));
        const V3<R> ux = ix[0] * xb;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const V3<R> dIJ = X - B[3 + k], ya = B[3 + k] - A[0];
            const R d2 = dot(dIJ, dIJ), irm = rsqrt_(d2), iy = rsqrt_(dot(ya, ya));
            const V3<R> uy = iy * ya;
            const R ci = dot(a, uy), cj = dot(l[k], ux);
            const R *c = S.rep_o[2][2];
            const R dj = c[2] + c[3] * ci, di = c[1] + c[3] * cj, o = c[0] + c[1] * ci + dj * cj;
            R e1, e2, h;
            Er.add(rep_energy(S, mask(d2) * (S.nlp * S.nlp), o * T1, o * T2, irm, e1, e2, h));
            const R w1 = e1 * T1, w2 = e2 * T2, w = w1 + w2, wi_ = w * di, wj_ = w * dj;
            gr0[0] -= o * (w1 * cval<R>(P.rep_k1[2][2]) + w2 * cval<R>(P.rep_k2[2][2]));
            fma3(ga, wi_, uy);
            fma3(gl[k], wj_, ux);
            const V3<R> gY = (wi_ * iy) * (a - ci * uy), gX = (wj_ * ix[0]) * (l[k] - cj * ux), hd = h * dIJ;
            gx = gx + gX + hd;
            g0 = g0 - gY;
            gj[0] = gj[0] - gX;
            gj[3 + k] = gj[3 + k] + gY - hd;
        }
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            fma3(ga, gp[y], e0[y]);
            const V3<R> G = (ri0[y] * gp[y]) * a;
            g0 = g0 - G;
            gj[y] = gj[y] + G;
        }
        const V3<R> t = unit_back(ga, a, ia);
        gi[0] = gi[0] + g0 - t;
        gi[3] = gi[3] + gx + t;
        swap_(A[3], A[4]);
        swap_(gi[3], gi[4]);
    }
    // the sums of O of i with j's atoms and directions
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        fma3(gm[c], gq00[c], e0[0]);
        fma3(gm[c], gq0c[c], e0[1 + c]);
        fma3(gl[c], gl0[c], e0[0]);
        V3<R> F = (ri0[0] * gq00[c]) * m[c];
        fma3(F, ri0[0] * gl0[c], l[c]);
        const V3<R> G = (ri0[1 + c] * gq0c[c]) * m[c];
        const V3<R> tm = unit_back(gm[c], m[c], im[c]), tl = unit_back(gl[c], l[c], il[c]);
        gi[0] = gi[0] - F - G;
        gj[0] = gj[0] + F - tm - tl;
        gj[1 + c] = gj[1 + c] + G + tm;
        gj[3 + c] = gj[3 + c] + tl;
    }
#pragma unroll
    for (int y = 0; y < 3; ++y) {
        const V3<R> F = gr0[y] * e0[y];
        gi[0] = gi[0] - F;
        gj[y] = gj[y] + F;
    }
}

// Dispersion and exchange-dispersion of molecules i (O at the origin) and j:
// points u of i (rolled: they rotate through place 0) against the five of j.
template <typename R, bool PER>
__device__ __forceinline__ void disp_pair(const KParams &P, const Scal<R> &S, const Water<R> &wi, const Water<R> &wj,
                                          V3<R> (&gi)[5], V3<R> (&gj)[5], Acc<R> &Ed, Acc<R> &Ex) {
    const R rc2 = S.rc2;
    V3<R> U[5] = {wi.P[0], wi.P[1], wi.P[2], wi.P[3], wi.P[4]};
    R cu[5] = {wi.cf[0], wi.cf[1], wi.cf[2], wi.cf[0], wi.cf[0]};
#pragma unroll 1
    for (int u = 0; u < 5; ++u) {
        const int ku = u == 0 ? 0 : (u < 3 ? 1 : 2);
        V3<R> gu = gi[0];
        R ed = R(0), exs = R(0);   // the point's five terms, then one compensated add each
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            const int kv = v == 0 ? 0 : (v < 3 ? 1 : 2);
            const V3<R> dv = U[0] - wj.P[v];
            const R r2 = dot(dv, dv);
            const R in = !PER || r2 < rc2 ? R(1) : R(0);
            const R ri = rsqrt_(r2), r = r2 * ri;
            const R a6 = mulc(ri, P.disp_gS[0][ku][kv]), a8 = mulc(ri, P.disp_gS[1][ku][kv]),
                    a10 = mulc(ri, P.disp_gS[2][ku][kv]);
            const R i2 = ri * ri, i6 = i2 * i2 * (in * i2), i8 = i6 * i2, i10 = i8 * i2;
            const R e6 = S.disp_c[0][ku][kv] * exp_(S.g6 - a6) * i6;
            const R e8 = S.disp_c[1][ku][kv] * exp_(S.g8 - a8) * i8;
            const R e10 = S.disp_c[2][ku][kv] * exp_(S.g10 - a10) * i10;
            const R ex = in * S.xd_c[ku][kv] * (cu[0] * wj.cf[v < 3 ? v : 0]) * exp_(-mulc(r, P.xd_k[ku][kv]));
            ed += e6 + e8 + e10;
            exs += ex;
            const R df = e6 * (a6 - R(6)) + e8 * (a8 - R(8)) + e10 * (a10 - R(10));
            const R c = df * i2 - cval<R>(P.xd_k[ku][kv]) * ex * ri;
            fma3(gu, c, dv);
            fma3(gj[v], -c, dv);
        }
        Ed.add(ed);
        Ex.add(exs);
        // place 0 takes the next point
        const V3<R> t = U[0];
        const R tc = cu[0];
#pragma unroll
        for (int k = 0; k < 4; ++k) U[k] = U[k + 1], cu[k] = cu[k + 1], gi[k] = gi[k + 1];
        U[4] = t;
        cu[4] = tc;
        gi[4] = gu;
    }
}

// Per-molecule data, packed so that a point is one aligned 4-vector: for O,
// H1, H2, LP1, LP2 the offset from O and the valence factor 1 - q/N_val of the
// point's atom (O's for the lone pairs).  Written each evaluation before the
// pair kernel, from the site offsets and the global charges; also clears the
// inbox counters.
template <typename R>
__global__ void k_short_pack(KParams p, DevState<R> d) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= p.M * 5) return;
    const Scal<R> &S = sc<R>(p);
    const int m = t / 5, k = t % 5;
    const int s = k < 3 ? k : k + 2, a = k < 3 ? k : 0;
    const R *o = d.off + (m * NP + s) * 3;
    const R q = d.gmp[(m * NS + a) * GMP];
    R *w = d.spk + (size_t)t * 4;
    w[0] = o[0];
    w[1] = o[1];
    w[2] = o[2];
    w[3] = R(1) - q * (a == 0 ? S.inv_nval_o : S.inv_nval_h);
    if (k == 0) d.inn[m] = 0;
}

template <typename R>
__device__ inline void ld4(const R *w, R &a, R &b, R &c, R &e);
template <>
__device__ inline void ld4<float>(const float *w, float &a, float &b, float &c, float &e) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(w));
    a = v.x, b = v.y, c = v.z, e = v.w;
}
template <>
__device__ inline void ld4<double>(const double *w, double &a, double &b, double &c, double &e) {
    const double2 v0 = __ldg(reinterpret_cast<const double2 *>(w)), v1 = __ldg(reinterpret_cast<const double2 *>(w) + 1);
    a = v0.x, b = v0.y, c = v1.x, e = v1.y;
}
__device__ inline void st4(float *w, float a, float b, float c, float e) {
    *reinterpret_cast<float4 *>(w) = make_float4(a, b, c, e);
}
__device__ inline void st4(double *w, double a, double b, double c, double e) {
    reinterpret_cast<double2 *>(w)[0] = make_double2(a, b);
    reinterpret_cast<double2 *>(w)[1] = make_double2(c, e);
}
template <typename R>
__device__ inline void store_row(R *w, const V3<R> (&g)[5], R last) {
    st4(w, g[0].x, g[0].y, g[0].z, g[1].x);
    st4(w + 4, g[1].y, g[1].z, g[2].x, g[2].y);
    st4(w + 8, g[2].z, g[3].x, g[3].y, g[3].z);
    st4(w + 12, g[4].x, g[4].y, g[4].z, last);
}
// molecule m with its O at o
template <typename R>
__device__ inline void load_water(const DevState<R> &d, int m, V3<R> o, Water<R> &w) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        R a, b, c, cf;
        ld4(d.spk + ((size_t)m * 5 + k) * 4, a, b, c, cf);
        w.P[k] = o + mk(a, b, c);
        if (k < 3) w.cf[k] = cf;
    }
}
// which of two molecules owns their pair
__device__ inline bool owns(int i, int j) { return ((i ^ j) & 1) ? i < j : i > j; }
// place of neighbour j in the list of m, in the gas phase (all of the cluster but m, from lo)
__device__ inline int gas_place(int m, int j, int lo) { return j - lo - (j > m ? 1 : 0); }

template <typename R>
__device__ inline float3 as_f3(V3<R> v) { return make_float3((float)v.x, (float)v.y, (float)v.z); }

// PART: 0 repulsion, 1 dispersion and exchange-dispersion, 2 both, -1 either by blockIdx.y.
template <typename R, bool PER, bool VIR, int PART>
__global__ void __launch_bounds__(32, sizeof(R) == 4 ? SHORT_BLOCKS : 8) k_short(KParams p, DevState<R> d,
                                                                                      int mpw) {
    __shared__ int qi[64], qj[64];
    __shared__ R qd[3][64];   // queued pairs: molecules and displacement
    constexpr int NV = PER ? (VIR ? 24 : 15) : 1;
    __shared__ R buf[NV * 33];   // a box: column sums of molecule cur, by lane
    constexpr bool FOLD = PER && sizeof(R) == 4;   // energies go on in FP64 from molecule to molecule
    __shared__ double es[FOLD ? 3 : 1][32];
    const int lane = threadIdx.x;
    const int part = PART < 0 ? (int)blockIdx.y : PART;
    const Scal<R> &S = sc<R>(p);
    const float rcf = (float)S.rc2 + 0.86f;
    const int first = blockIdx.x * mpw, last = min(p.M, first + mpw);
    Acc<R> Er, Ed, Ex;
    int cur = -1;
    if constexpr (FOLD) es[0][lane] = es[1][lane] = es[2][lane] = 0.0;
    auto store = [&]() {   // points 3, 4 are the lone pairs (point slots 5, 6)
        __syncwarp();
        if (lane < NV) {
            R s0 = R(0), s1 = R(0);
#pragma unroll 8
            for (int k = 0; k < 32; k += 2) s0 += buf[lane * 33 + k], s1 += buf[lane * 33 + k + 1];
            const double s = double(s0 + s1);
            const int pt = lane / 3;
            if (lane < 15) atomicAdd(d.gpt + (cur * NP + (pt < 3 ? pt : pt + 2)) * 3 + lane % 3, s);
            else atomicAdd(d.vir + cur * 9 + lane - 15, s);
        }
        __syncwarp();
    };
    auto clear = [&]() {
#pragma unroll
        for (int k = 0; k < NV; ++k) buf[k * 33 + lane] = R(0);
    };
    auto row_of = [&](int m, int row) -> R * {
        return d.inbox + ((size_t)m * d.in_rows + row) * (PER ? BOX_ROW : GAS_ROW);
    };
    auto round = [&](int n) {   // the first n <= 32 queued pairs
        int mi = 0x7fffffff;
        V3<R> gi[5], gj[5];
        V3<R> dO = mk(R(0), R(0), R(0));
#pragma unroll
        for (int k = 0; k < 5; ++k) gi[k] = gj[k] = dO;
        if (lane < n) {
            mi = qi[lane];
            const int j = qj[lane];
            dO = mk(qd[0][lane], qd[1][lane], qd[2][lane]);
            const int row = PER ? atomicAdd(d.inn + j, 1) : 0;
            if (!PER) Er = Ed = Ex = Acc<R>();
            {
                Water<R> wi, wj;
                load_water(d, mi, mk(R(0), R(0), R(0)), wi);
                load_water(d, j, dO, wj);
                if (part != 1) rep_pair<R, PER>(p, S, wi, wj, gi, gj, Er);
                if (part != 0) disp_pair<R, PER>(p, S, wi, wj, gi, gj, Ed, Ex);
            }
            if (PER) {
                if (row < d.in_rows) {
                    store_row(row_of(j, row), gj, R(0));
                } else {   // the inbox is full
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        double *g = d.gpt + (j * NP + (k < 3 ? k : k + 2)) * 3;
                        atomicAdd(g, double(gj[k].x));
                        atomicAdd(g + 1, double(gj[k].y));
                        atomicAdd(g + 2, double(gj[k].z));
                    }
                }
            } else {
                // (more neighbours than the list holds are an error that is already flagged)
                const int lo = d.cl_start[d.cl_of[mi]], nmax = p.tls / 3, po = PART < 0 ? part * nmax : 0;
                const int ri = gas_place(mi, j, lo), rj = gas_place(j, mi, lo);
                if (rj < nmax) store_row(row_of(j, po + rj), gj, R(0));
                if (ri < nmax) {
                    R *v = row_of(mi, po + ri);
                    store_row(v, gi, Er.hi);
                    st4(v + 16, Er.lo, Ed.hi, Ed.lo, Ex.hi);
                    v[20] = Ex.lo;
                }
            }
        }
        // into the sums of its molecule, one molecule at a time in order
        bool begun = false;
        while (PER) {
            if (cur >= 0 && mi == cur) {
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    buf[(3 * k) * 33 + lane] += gi[k].x;
                    buf[(3 * k + 1) * 33 + lane] += gi[k].y;
                    buf[(3 * k + 2) * 33 + lane] += gi[k].z;
                }
                if constexpr (PER && VIR) {   // by translation invariance: minus the gradient of i's points (x) dO
                    R W[9];
#pragma unroll
                    for (int k = 0; k < 9; ++k) W[k] = buf[(15 + k) * 33 + lane];
                    vir_add(W, gi[0] + gi[1] + gi[2] + gi[3] + gi[4], dO, R(-1));
#pragma unroll
                    for (int k = 0; k < 9; ++k) buf[(15 + k) * 33 + lane] = W[k];
                }
            }
            const int next = __reduce_min_sync(0xffffffffu, mi > cur ? mi : 0x7fffffff);
            if (next == 0x7fffffff) break;
            if (cur >= 0) store();
            clear();
            cur = next;
            begun = true;
        }
        if constexpr (FOLD) {
            if (begun) {   // (each lane its own places)
                es[0][lane] += Er.get();
                es[1][lane] += Ed.get();
                es[2][lane] += Ex.get();
                Er = Ed = Ex = Acc<R>();
            }
        }
    };
    auto total = [&](const Acc<R> &a, int k) {
        if constexpr (FOLD) return warp_sum(es[k][lane] + a.get());
        else return warp_sum_acc(a);
    };
    int nq = 0;
    for (int i = first; i < last; ++i) {
        const int nn = d.nnbr[i];
        const int *nb = d.nbr + (size_t)i * MAXN;
        const R *nd = d.ndo + (size_t)i * MAXN * 3;
        // i's points a as -2 a and |a|^2 for the test below
        float3 a2[5];
        float aa[5];
        if (PER) {
            Water<R> wi;
            load_water(d, i, mk(R(0), R(0), R(0)), wi);
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const float3 a = as_f3(wi.P[u]);
                a2[u] = make_float3(-2.0f * a.x, -2.0f * a.y, -2.0f * a.z);
                aa[u] = a.x * a.x + a.y * a.y + a.z * a.z;
            }
        }
        int jn = i;   // the next 32 entries, read one step ahead
        V3<R> dn = mk(R(0), R(0), R(0));
        auto fetch = [&](int slot) {
            if (slot < nn) {
                jn = nb[slot];
                dn = mk(nd[3 * slot], nd[3 * slot + 1], nd[3 * slot + 2]);
            }
        };
        fetch(lane);
        for (int base = 0; base < nn; base += 32) {
            const int j = jn;
            const V3<R> dj = dn;
            bool take = base + lane < nn && owns(i, j);
            fetch(base + 32 + lane);
            if (PER && take) {
                // Anything inside the cutoff?  A bond midpoint can be nearer than its ends: the squared distance of
                // two midpoints is the mean over the ends less the squared half bonds, which a site extent of
                // 1.3 A (the largest accepted) bounds by 0.85 A^2.
                Water<R> wj;
                load_water(d, j, dj, wj);
                float least = 3.0e38f;
                float3 b[5];
                float bb[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    b[v] = as_f3(wj.P[v]);
                    bb[v] = b[v].x * b[v].x + b[v].y * b[v].y + b[v].z * b[v].z;
                }
#pragma unroll
                for (int u = 0; u < 5; ++u) {
                    float t = 3.0e38f;
#pragma unroll
                    for (int v = 0; v < 5; ++v)
                        t = fminf(t, fmaf(a2[u].x, b[v].x, fmaf(a2[u].y, b[v].y, fmaf(a2[u].z, b[v].z, bb[v]))));
                    least = fminf(least, t + aa[u]);
                }
                take = least < rcf;
            }
            const unsigned b = __ballot_sync(0xffffffffu, take);
            if (take) {
                const int e = nq + __popc(b & ((1u << lane) - 1u));
                qi[e] = i;
                qj[e] = j;
                qd[0][e] = dj.x, qd[1][e] = dj.y, qd[2][e] = dj.z;
            }
            nq += __popc(b);
            __syncwarp();
            if (nq >= 32) {
                round(32);
                __syncwarp();
                nq -= 32;
                if (lane < nq) {
                    qi[lane] = qi[32 + lane];
                    qj[lane] = qj[32 + lane];
#pragma unroll
                    for (int k = 0; k < 3; ++k) qd[k][lane] = qd[k][32 + lane];
                }
                __syncwarp();
            }
        }
    }
    if (nq > 0) round(nq);
    if (PER) {
        if (cur >= 0) store();
        // the energies are summed over all molecules of the box
        const double e0 = total(Er, 0), e1 = total(Ed, 1), e2 = total(Ex, 2);
        if (lane == 0) {
            double *e = d.epart + first * NTERM;
            if (part != 1) atomicAdd(e + T_REP, e0);
            if (part != 0) {
                atomicAdd(e + T_DISP, e1);
                atomicAdd(e + T_XDISP, e2);
            }
        }
    }
}

// Adds up the inbox rows of a molecule, in a box the gradients only.  VIR: also the points' share of the
// virial, sum_p G_p (x) off_p over both sides' terms, and in the gas phase the pairs' -F (x) dO.
template <typename R, bool PER, bool VIR>
__global__ void __launch_bounds__(128) k_short_gather(KParams p, DevState<R> d, int parts) {
    __shared__ double tot[4][16];
    const int wq = threadIdx.x >> 5, lane = threadIdx.x & 31, m = blockIdx.x * 4 + wq;
    if (m >= p.M) return;
    Acc<R> s;
    double g;
    const int pt = lane / 3;
    if (PER) {
        const R *rows = d.inbox + (size_t)m * d.in_rows * BOX_ROW;
        const int half = lane >> 4, c = lane & 15, n = min(d.inn[m], d.in_rows);
        for (int r0 = half; r0 < n; r0 += 8) {
            R v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = c < 15 && r0 + 2 * k < n ? rows[(size_t)(r0 + 2 * k) * BOX_ROW + c] : R(0);
            s.add((v[0] + v[1]) + (v[2] + v[3]));
        }
        g = s.get();
        g += __shfl_xor_sync(0xffffffffu, g, 16);
    } else {
        const R *rows = d.inbox + (size_t)m * d.in_rows * GAS_ROW;
        const int n = d.nnbr[m], lo = d.cl_start[d.cl_of[m]], nmax = p.tls / 3;
        double W = 0;
        for (int r0 = 0; r0 < n; r0 += 32) {
            const int jl = r0 + lane < n ? d.nbr[m * MAXN + r0 + lane] : 0;
            for (int q = 0; q < parts; ++q)
#pragma unroll 4
                for (int r = 0; r < min(32, n - r0); ++r) {
                    const int j = __shfl_sync(0xffffffffu, jl, r);
                    const bool mine = owns(m, j);
                    const R *w = rows + (size_t)(q * nmax + min(gas_place(m, j, lo), nmax - 1)) * GAS_ROW;
                    if (lane < 15 || (mine && lane < 21)) s.add(w[lane]);
                    if (VIR && mine && lane < 9) {
                        const int a = lane / 3;
                        const R F = (w[a] + w[3 + a]) + (w[6 + a] + w[9 + a]) + w[12 + a];
                        W -= double(F * d.ndo[((size_t)m * MAXN + r0 + r) * 3 + lane % 3]);
                    }
                }
        }
        g = s.get();
        const double lo_ = __shfl_down_sync(0xffffffffu, g, 1);
        if (lane == 15) d.epart[m * NTERM + T_REP] += g + lo_;
        if (lane == 17) d.epart[m * NTERM + T_DISP] += g + lo_;
        if (lane == 19) d.epart[m * NTERM + T_XDISP] += g + lo_;
        if (VIR && lane < 9) d.vir[m * 9 + lane] += W;
    }
    double *o = d.gpt + (m * NP + (pt < 3 ? pt : pt + 2)) * 3 + lane % 3;
    if (lane < 15) {
        g += *o;
        *o = g;
    }
    if (VIR) {
        if (lane < 15) tot[wq][lane] = g;
        __syncwarp();
        if (lane < 9) {
            const int a = lane / 3, b = lane % 3;
            double v = 0;
            for (int k = 0; k < 5; ++k) v += tot[wq][3 * k + a] * double(d.spk[((size_t)m * 5 + k) * 4 + b]);
            d.vir[m * 9 + lane] += v;
        }
    }
}

}  // namespace

template <bool PER>
static cudaError_t short_admit() {
    const auto k = k_short<double, PER, false, -1>;
    int dev = 0, most = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
    return e;
}
// Admits any reservation of launch_short, once per context, at creation: the
// limit belongs to the process, so a launch that set its own could be refused
// when another thread's context lowered it in between.
template <typename R>
cudaError_t short_init(const KParams &p) {
    if (sizeof(R) == 4) return cudaSuccess;
    return p.periodic ? short_admit<true>() : short_admit<false>();
}

// FP64: max_per_sm > 0 caps the resident blocks per SM by reserving unused
// dynamic shared memory, which leaves registers on every SM for the kernels of
// the other streams.  FP32 takes no cap (SHORT_BLOCKS an SM by its registers).
template <typename R>
void launch_short(const KParams &p, DevState<R> &d, Launch L, int max_per_sm) {
    int dev = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    constexpr int PART = sizeof(R) == 4 ? 2 : -1;
    constexpr int parts = PART < 0 ? 2 : 1;
    // Molecules a warp: the fewest rounds of 32 pairs in a row over the warps
    // that the chip holds at once.  A molecule has about half its neighbours'
    // pairs (in a box those within rc of any of its points, some 1.4 A more
    // between the O).
    const double rn = p.rc + 1.4, V = p.box[0] * p.box[1] * p.box[2];
    const double nbr = p.periodic ? std::min(p.M - 1.0, p.M / V * 4.18879 * rn * rn * rn) : p.M / (double)p.n_cl - 1.0;
    const double most = p.periodic ? nbr : (double)(p.tls / 3);
    const int mpw = warp_molecules(p.M, 0.5 * nbr, 0.5 * most, parts, sizeof(R) == 4 ? SHORT_BLOCKS : 4,
                                   p.periodic ? 0.0 : 0.25, 64);
    size_t sm = 0;
    k_short_pack<R><<<(p.M * 5 + 255) / 256, 256, 0, L.s>>>(p, d);
    const unsigned ng = (unsigned)((p.M + 3) / 4);
    auto run = [&](auto per, auto vir) {
        auto k = k_short<R, decltype(per)::value, decltype(vir)::value, PART>;
        const int cap = max_per_sm;
        if (sizeof(R) == 8 && cap > 0 && cap < 8 && !p.vir) {   // (registers allow no more than 8)
            cudaFuncAttributes fa;
            cudaFuncGetAttributes(&fa, k);
            // one byte more per block than another block would leave room for
            const long long need = per_sm / (cap + 1) + 1 - (long long)fa.sharedSizeBytes - 1024;
            if (need > 0) sm = (size_t)need;   // (short_init admits it)
        }
        k<<<dim3((unsigned)((p.M + mpw - 1) / mpw), parts), 32, sm, L.s>>>(p, d, mpw);
        k_short_gather<R, decltype(per)::value, decltype(vir)::value><<<ng, 128, 0, L.s>>>(p, d, parts);
    };
    if (p.periodic) p.vir ? run(std::true_type{}, std::true_type{}) : run(std::true_type{}, std::false_type{});
    else p.vir ? run(std::false_type{}, std::true_type{}) : run(std::false_type{}, std::false_type{});
    count(L, 3);
}

template cudaError_t short_init<float>(const KParams &);
template cudaError_t short_init<double>(const KParams &);
template void launch_short<float>(const KParams &, DevState<float> &, Launch, int);
template void launch_short<double>(const KParams &, DevState<double> &, Launch, int);

}  // namespace sibfa
