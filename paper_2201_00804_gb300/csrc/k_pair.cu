// Real-space pair kernels over the full molecular neighbour list.
//
// Every kernel walks the neighbours of one molecule i and accumulates only
// i's quantities (energy halves, gradients of i's points, multipole
// sensitivities of i's sites), so no two threads write the same output and
// no atomics are needed (k_perm_gas: two warps add to a target, once each); the neighbour list is full, each molecule pair is
// visited from both sides.  Pair arithmetic runs in R (float in the mixed
// path, double in the FP64 path); per-lane partial sums are reduced across
// the warp in double.
#include <type_traits>

#include "pair_terms.cuh"

namespace sibfa {


template <typename R>
__device__ inline void symadd(Sym<R> &a, const Sym<R> &b, R s) {
    a.xx += s * b.xx; a.yy += s * b.yy; a.zz += s * b.zz;
    a.xy += s * b.xy; a.xz += s * b.xz; a.yz += s * b.yz;
}
template <typename R>
__device__ __forceinline__ void symacc(Sym<R> &a, const Sym<R> &b) {
    a.xx += b.xx; a.yy += b.yy; a.zz += b.zz;
    a.xy += b.xy; a.xz += b.xz; a.yz += b.yz;
}

// ---------------------------------------------------------------------------
// Work queues.  A warp walks its molecule's neighbour list 32 entries at a
// time, tests each (neighbour, source site) pair against the cutoff and
// appends the pairs inside it to a per-warp ring queue in shared memory
// (source position relative to O_i, neighbour index and site).  Pairs are
// evaluated in rounds of 32 only while the queue holds a full round, so
// lanes stay busy whatever the cutoff rejects; the tail is flushed at the
// end.  Atom and midpoint sources go to separate queues because only atom
// sources carry a valence (penetration), which keeps every round uniform.
//
// The target kernels below run one target site per block of one warp.  They
// are bound by issue and by the latency of each round's source loads, so what
// counts is warps per SM: blocks of one warp take any register count that
// divides the file (96 registers, 21 warps, against 15 in blocks of five),
// and a molecule's heavy targets (atoms) do not hold up its light ones.
// ---------------------------------------------------------------------------
constexpr int QCAP_A = 128;   // >= 31 carried + 3 atom sites x 32 new entries
constexpr int QCAP_M = 96;    // >= 31 carried + 2 midpoints x 32 new entries

template <typename R, int CAP = QCAP_A + QCAP_M>
struct PairQueue {
    int js[CAP];   // j * 8 + s
    R rx[CAP], ry[CAP], rz[CAP];
    __device__ inline void put(int e, int js_, V3<R> r) {
        js[e] = js_;
        rx[e] = r.x;
        ry[e] = r.y;
        rz[e] = r.z;
    }
    __device__ inline V3<R> at(int e) const { return mk(rx[e], ry[e], rz[e]); }
};

// ---------------------------------------------------------------------------
// Permanent electrostatics + penetration (Eq. 2), Thole-damped permanent
// field on the polarizable atoms.
// ---------------------------------------------------------------------------
template <typename R>
struct PermAcc {
    Acc<R> Ue, Up;
    V3<R> gr, gm, ef;
    Sym<R> gt;   // three times the quadrupole sensitivity
    R W[9];      // virial (VIR kernels only)
};

// A warp's target site
template <typename R>
struct PermT {
    Mp<R> m;      // quadrupole / 3
    V3<R> o;      // offset from O_i
    R N, Q;       // valence; charge of molecule i (gas phase)
    int w;        // site
};

// VIR: also accumulate the pair virial 1/2 g (x) x of the target's gradient g
// (both molecules of a pair see it, so each adds half); the lone-pair
// potential's share is taken with the lambda charges in the force pass.
//
// Periodic systems: rv is the source position relative to O_i (O-O
// displacement plus the source's offset).  Gas phase: rv is the O-O
// displacement D = O_j - O_i itself and the pair displacement is formed as
// x = (target offset - source offset) - D.  The energy terms that involve a
// charge are taken as differences from reference points, because over a
// neutral molecule they cancel to the molecular interaction (site-pair
// terms of ~10 kcal/mol for a total of a few) and FP32 would keep only their
// rounding: with a = 1/|x|, b = 1/|y| for a reference vector y and
// d = |y|^2 - |x|^2 computed from the offsets without cancellation,
//   a - b = d a b / (|x| + |y|),  a^3 - b^3 = (a - b)(a^2 + ab + b^2),
//   a^5 - b^5 = (a - b)(a^4 + a^3 b + a^2 b^2 + a b^3 + b^4).
//   charge-charge:        y0 = -D (O_i - O_j):  q_t q_s (a - b0);
//   target charge in the source dipole/quadrupole potential, y1 = O_i - x_s:
//     q_t [mu_s.o_t a^3 + mu_s.y1 (a^3 - b1^3) + (o_t Th_s o_t + 2 y1 Th_s o_t) a^5
//          + y1 Th_s y1 (a^5 - b1^5)]   (x = y1 + o_t);
//   source charge in the target dipole/quadrupole, y2 = x_t - O_j:
//     q_s [mu_t.o_s a^3 - mu_t.y2 (a^3 - b2^3) + (o_s Th_t o_s - 2 y2 Th_t o_s) a^5
//          + y2 Th_t y2 (a^5 - b2^5)]   (x = y2 - o_s).
// The remainders (the reference values times the molecule's total charge,
// zero for neutral molecules) are added once per molecule pair (Q_i Q_j / R),
// per target site and neighbour, and per source site on the O target's warp.
// For gas-phase clusters this brings the FP32 multipole energy some 30x
// closer to FP64 than summing the site-pair energies directly.
//
// What depends on the target site and the source molecule alone (y2, its
// products with the target, y0) is formed once for the molecule's five sources.
//
// ms: source multipole of site s_ (quadrupole / 3).  At a polarizable target
// x, T2 and g1 return the pair's entry of the polarization matrix (field of a
// dipole mu at x: T2 (mu.x) x + g1 mu).
template <typename R>
struct GasRef {
    V3<R> y2, Tty;       // x_t - O_j, (Theta_t / 3) y2
    R b2, r2, mu, yTy;   // 1/|y2|, |y2|, mu_t.y2, y2.Theta_t.y2
    R b0, r0;            // 1/|D|, |D|
    __device__ __forceinline__ GasRef(const PermT<R> &T, V3<R> D) {
        y2 = T.o - D;
        const R yy = dot(y2, y2), DD = dot(D, D);
        b2 = rsqrt_(yy);
        r2 = yy * b2;
        Tty = symv(T.m.th, y2);
        mu = dot(T.m.mu, y2);
        yTy = R(3.0) * dot(y2, Tty);
        b0 = rsqrt_(DD);
        r0 = DD * b0;
    }
    __device__ __forceinline__ GasRef() {}
};

template <typename R, bool PER, bool ATOM_SRC, bool VIR>
__device__ __forceinline__ void perm_pair(const KParams &p, const PermT<R> &T, const GasRef<R> &G, const Mp<R> &ms,
                                          int s_, V3<R> rv, V3<R> osrc, bool energy, PermAcc<R> &acc, R &g1, R &T2,
                                          V3<R> &x) {
    const Scal<R> &S = sc<R>(p);
    const bool atom = T.w < 3;
    const R m1 = R(-1.0), two = R(2.0);
    V3<R> sv;
    if (PER) x = T.o - rv;
    else {
        sv = T.o - osrc;
        x = sv - rv;
    }
    const R r2 = dot(x, x);
    const R rinv = rsqrt_<R>(r2);
    const R r = r2 * rinv, r2i = rinv * rinv;
    R B[6];
    kernel_B<R, PER, 5>(r, rinv, r2i, S.alpha, B);
    const Source<R> s(ms, x);
    const Target<R> t(T.m, x);
    const R pdt = symdd(s.th, t.th);
    Field2<R> F;
    const V3<R> gel = pair_grad(t, s, x, B, pdt, F);
    R U = R(0);
    if (PER) {
        U = t.q * (s.q * B[0] + s.s * B[1] + s.w * B[2]) + dot(t.mu, F.d1) + F.Rr * t.w + two * dot(t.p, F.U) +
            two * B[2] * pdt;
    } else if (energy) {
        const R three = R(3.0);
        const R a = rinv, a3 = a * r2i, a5 = a3 * r2i;
        // charge-charge, reference -D
        U = t.q * s.q * ((two * dot(sv, rv) - dot(sv, sv)) * a * G.b0 / (r + G.r0));
        // target charge, reference O_i - x_s
        const V3<R> y1 = m1 * (rv + osrc);
        const R y1y1 = dot(y1, y1), b1 = rsqrt_<R>(y1y1);
        R D3, D5;
        ref_diff35(m1 * (two * dot(y1, T.o) + dot(T.o, T.o)), a, b1, r, y1y1 * b1, D3, D5);
        const V3<R> Tso = symv(s.th, T.o), Tsy = symv(s.th, y1);
        const R mu_y1 = dot(s.mu, y1), y1Ty1 = three * dot(y1, Tsy);
        U += t.q * (dot(s.mu, T.o) * a3 + mu_y1 * D3 + three * (dot(T.o, Tso) + two * dot(y1, Tso)) * a5 + y1Ty1 * D5);
        if (T.w == 0) {   // sum over the target sites of q_t times the reference value: Q_i phi_s(y1)
            const R b13 = b1 * b1 * b1;
            U += T.Q * (mu_y1 * b13 + y1Ty1 * b13 * b1 * b1);
        }
        // source charge, reference x_t - O_j
        ref_diff35(two * dot(G.y2, osrc) - dot(osrc, osrc), a, G.b2, r, G.r2, D3, D5);
        const V3<R> Tto = symv(t.th, osrc);
        U += s.q * (dot(t.mu, osrc) * a3 - G.mu * D3 + three * (dot(osrc, Tto) - two * dot(osrc, G.Tty)) * a5 +
                    G.yTy * D5);
        // target dipole and quadrupole in the source dipole and quadrupole field
        U += dot(t.mu, s.grad_mp(x, B[1], B[2], B[3])) + (s.s * B[3] + s.w * B[4]) * t.w + two * dot(t.p, F.U) +
             two * B[2] * pdt;
    }
    if (PER) acc.Ue.add(R(0.5) * U);
    else if (energy) acc.Ue.add(U);
    V3<R> g = gel;
    acc.gm = acc.gm + F.d1;
    symacc(acc.gt, F.d2);
    // ---- penetration: charge-charge*, charge-dipole*, charge-quadrupole*
    // Kernels exp(-b r)/r of the source (es) and target (et) valence; the
    // product kernel exp(-(b_s + b_t) r)/r of the N_t N_s term is es0 et0 r.
    if (ATOM_SRC || atom) {
        R pen = R(0.0), gq = R(0.0);   // gq: minus the coefficient of x from the charge terms
        R et[4];
        const R xt = mulc(r, p.pen_b[T.w]);
        if (atom) {
            kernel_exp(xt, rinv, r2i, et);
            const R c2 = s.q * T.N;            // q_s N_t exp(-b_t r)/r
            pen = c2 * et[0];
            gq = c2 * et[1];
        }
        if (ATOM_SRC) {
            const R Ns = zsite<R>(p, s_) - ms.q, xs = mulc(r, p.pen_b[s_]);
            R es[4];
            kernel_exp(xs, rinv, r2i, es);
            const R c1 = t.q * Ns;             // q_t N_s exp(-b_s r)/r
            pen += c1 * es[0];
            gq += c1 * es[1];
            if (atom) {                      // N_t N_s exp(-(b_t + b_s) r)/r
                const R ec = T.N * Ns * es[0] * et[0] * r;
                pen += ec;
                gq += (xt + xs + R(1.0)) * ec * r2i;
            }
            // valence of s in the dipole/quadrupole potential of t, at -x
            const R e2 = Ns * es[2], e1 = Ns * es[1];
            pen += t.w * e2 - t.s * e1;
            const R P = t.s * e2 - t.w * (Ns * es[3]), c = e2 + e2;
            g = g + P * x + c * t.p - e1 * t.mu;
            acc.gm = acc.gm - e1 * x;
            const V3<R> ex = e2 * x;
            acc.gt.xx += ex.x * x.x; acc.gt.yy += ex.y * x.y; acc.gt.zz += ex.z * x.z;
            acc.gt.xy += ex.x * x.y; acc.gt.xz += ex.x * x.z; acc.gt.yz += ex.y * x.z;
        }
        if (atom) {   // valence of t in the dipole/quadrupole potential of s
            const R f1 = T.N * et[1], f2_ = T.N * et[2];
            pen += s.s * f1 + s.w * f2_;
            gq += s.s * f2_ + s.w * (T.N * et[3]);
            const R c = f2_ + f2_;
            g = g + f1 * s.mu + c * s.v;
        }
        g = g - gq * x;
        if (PER) acc.Up.add(R(0.5) * pen);
        else if (energy) acc.Up.add(pen);
    }
    acc.gr = acc.gr + g;
    if (VIR) vir_add(acc.W, g, x, R(0.5));
    // ---- Thole-damped permanent field on the polarizable atom (same base kernel B)
    if (atom) {
        const R u = S.thole * r2 * r * ainv3<R>(p, T.w, s_);
        const R e = exp_(m1 * u), c1 = e, c2 = e + u * e, c3 = c2 + R(0.6) * u * (u * e);
        const R b1 = rinv * r2i, b2 = R(3.0) * b1 * r2i, b3 = R(5.0) * b2 * r2i;
        const R T1 = B[1] - c1 * b1, T3 = B[3] - c3 * b3;
        T2 = B[2] - c2 * b2;
        acc.ef = acc.ef - s.grad(x, T1, T2, T3);
        g1 = m1 * T1;
    }
}

// An entry of the polarization matrix T: the field of a dipole mu at x is
// T2 (mu.x) x + g1 mu = sgn(T2) (mu.y) y + g1 mu with y = sqrt|T2| x: four
// values and the sign in the index's top bit.
template <typename R>
__device__ __forceinline__ void store_tpair(const DevState<R> &d, size_t te, int atom, V3<R> x, R T2, R g1) {
    const R sq = sqrt_(fabs(T2));
    d.tl_j[te] = atom | (T2 < R(0) ? int(0x80000000u) : 0);
    d.tl_x[te] = sq * x.x;
    d.tl_y[te] = sq * x.y;
    d.tl_z[te] = sq * x.z;
    d.tl_g1[te] = g1;
}

// Gas phase: the list entries of consecutive molecules (at most 32) on one
// side of the ownership of pairs, 32 at a time in order.  Molecule i of a
// cluster [lo, hi) owns its pairs with the lower ones of its parity and the
// higher ones of the other; its list holds all of the cluster but itself.  A molecule
// without entries takes one place.
constexpr int GAS_BLOCKS = 16;   // one-warp blocks an SM, FP32
struct GasWalk {
    int first, n_mol, others;   // molecules; 0: the owned entries, 1: the rest
    int nl, ll;                 // lane k's: entries of molecule first + k, and the molecules below it in its cluster
    int m = 0, at = 0;          // next molecule and entry
    int mol, slot;              // this lane's: molecule (-1: idle) and list place (-1: none)
    int n_used;
    template <typename R>
    __device__ GasWalk(const KParams &p, const DevState<R> &d, int mpw, int lane)
        : first(blockIdx.x * mpw), n_mol(min(mpw, p.M - first)), others(blockIdx.z) {
        nl = ll = 0;
        if (lane < n_mol) {
            const int nn = d.nnbr[first + lane];
            ll = min(first + lane - d.cl_start[d.cl_of[first + lane]], nn);   // (a list that overflowed is flagged)
            const int up = nn - ll;
            nl = others ? (ll + 1) / 2 + up / 2 : ll / 2 + (up + 1) / 2;
        }
    }
    __device__ bool next(int lane) {
        mol = slot = -1;
        n_used = 0;
        while (n_used < 32 && m < n_mol) {
            const int n = __shfl_sync(0xffffffffu, nl, m), lo = __shfl_sync(0xffffffffu, ll, m);
            const int places = max(n, 1), take = min(32 - n_used, places - at);
            if (lane >= n_used && lane < n_used + take) {
                mol = first + m;
                if (n > 0) {
                    const int k = at + lane - n_used, below = others ? (lo + 1) / 2 : lo / 2;
                    // below: lo - 1 - others.. downwards by twos; above (places shift by one, i is not listed) upwards
                    slot = k < below ? lo - 2 * (k + 1) + others : lo + 2 * (k - below) + others;
                }
            }
            n_used += take;
            at += take;
            if (at == places) ++m, at = 0;
        }
        return n_used > 0;
    }
    // f(molecule, lanes from, to, whether these hold the molecule's first entry)
    template <typename F>
    __device__ void segments(bool start_new, F f) const {
        int k = 0;
        for (int c = 0; c < n_used; ++k) {
            const int g = __shfl_sync(0xffffffffu, mol, c);
            const int n = __popc(__ballot_sync(0xffffffffu, mol == g));
            f(g, c, c + n, k > 0 || start_new);
            c += n;
        }
    }
};
// sum over columns c0 <= c < c1 of row lane (< nv) of buf (33 a row); FP32: compensated
template <typename R>
__device__ __forceinline__ double segment_sum(const R *buf, int lane, int nv, int c0, int c1) {
    if (lane >= nv) return 0.0;
    Acc<R> a;
    R s = R(0);
    for (int c = c0; c < c1; ++c) {
        if (sizeof(R) == 4) a.add(buf[lane * 33 + c]);
        else s += buf[lane * 33 + c];
    }
    return sizeof(R) == 4 ? a.get() : double(s);
}
// Molecules a warp of k_perm_gas: whole rounds in FP32 (4096 clusters of 17
// waters, at most 2: 1305 us, 4: 1351, 8: 1135, 32: 1050); in FP64, bound by
// the pipe of each quarter of an SM, few, which spreads the work (824 waters, at most 2 or 4: 510 us, 8: 522, 16: 703).
template <typename R>
int gas_mpw(const KParams &p) {
    return warp_molecules(p.M, 0.5 * (p.M / (double)p.n_cl - 1.0), 0.5 * (p.tls / 3), 2 * NS, (sizeof(R) == 4 ? GAS_BLOCKS : 4), 0.25,
                          sizeof(R) == 4 ? 32 : 4);
}

// Boxes.  Blocks per SM, FP32: at least 18 (96 registers, 21 blocks; 32,000 waters
// 1630 us; at 112 registers and 18 blocks 1728, with the five sites in one
// block 1926); FP64 8 (216 waters: 274 us against 416 in one block).
template <typename R, bool VIR>
__global__ void __launch_bounds__(VIR ? 32 * NS : 32,
                                  VIR ? (sizeof(R) == 4 ? 3 : 2) : (sizeof(R) == 4 ? 18 : 8))
    k_real_perm(KParams p, DevState<R> d) {
    constexpr int NW = VIR ? NS : 1;   // warps a block: the virial variant sums the sites' in a fixed order
    __shared__ double s_w[VIR ? NW : 1][9];
    __shared__ PairQueue<R> qs[NW];
    static_assert(sizeof(PairQueue<R>) >= 15 * 33 * sizeof(R), "reduction buffer aliases the queue");
    const int wq = VIR ? threadIdx.x >> 5 : 0, lane = threadIdx.x & 31;
    const int i = VIR ? blockIdx.x : blockIdx.x / NS;
    const int w = VIR ? wq : blockIdx.x % NS;   // target site
    PairQueue<R> &q = qs[wq];
    const Mp<R> mt = load_mp(d.gmp + (i * NS + w) * GMP);
    const PermT<R> T{scaled(mt, R(1.0 / 3.0)), my_pt(d, i, w), zsite<R>(p, w) - mt.q, R(0), w};
    const GasRef<R> none;
    const R rc2 = sc<R>(p).rc2;
    const size_t tbase = (size_t)(i * 3 + (w < 3 ? w : 0)) * p.tls;   // T-pair list of target atom w

    PermAcc<R> acc;
    acc.gr = mk(R(0), R(0), R(0));
    acc.gm = acc.gr;
    acc.ef = acc.gr;
    acc.gt = Sym<R>{};
#pragma unroll
    for (int k = 0; k < 9; ++k) acc.W[k] = R(0);

    auto eval = [&](auto atom_src, int e, size_t te) {
        constexpr bool AT = decltype(atom_src)::value;
        const int js = q.js[e], j = js >> 3, s = js & 7;
        const Mp<R> ms = scaled(load_mp_g(d.gmp + (j * NS + s) * GMP), R(1.0 / 3.0));
        V3<R> x;
        R g1 = R(0), T2 = R(0);
        perm_pair<R, true, AT, VIR>(p, T, none, ms, s, q.at(e), T.o, true, acc, g1, T2, x);
        if (AT && w < 3 && p.tlist) store_tpair(d, te, j * 3 + s, x, T2, g1);
    };

    int ha = 0, ta = 0, hm = 0, tm = 0;   // queue heads and tails (warp-uniform, monotone)
    const int nn = d.nnbr[i];
    for (int base = 0;; base += 32) {
        const bool flush = base >= nn;   // list exhausted: evaluate what is left in the queues
        const int slot = base + lane;
        unsigned bits = 0;
        int j = 0;
        V3<R> rs[NS];
        if (slot < nn) {
            j = d.nbr[i * MAXN + slot];
            const R *dp = d.ndo + ((size_t)i * MAXN + slot) * 3;
            const V3<R> dO = mk(dp[0], dp[1], dp[2]);
            const R *offj = d.off + j * NP * 3;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                rs[s] = dO + mk(__ldg(offj + s * 3), __ldg(offj + s * 3 + 1), __ldg(offj + s * 3 + 2));
                const V3<R> x = T.o - rs[s];
                if (dot(x, x) < rc2) bits |= 1u << s;
            }
        }
        int na, nm;
        int pa = warp_excl_scan(__popc(bits & 7u), lane, na);
        int pm = warp_excl_scan(__popc(bits >> 3), lane, nm);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (!((bits >> s) & 1u)) continue;
            q.put(s < 3 ? (ta + pa++) % QCAP_A : QCAP_A + (tm + pm++) % QCAP_M, j * 8 + s, rs[s]);
        }
        ta += na;
        tm += nm;
        __syncwarp();
        while (ta - ha >= 32 || (flush && ta > ha)) {
            if (lane < ta - ha) eval(std::true_type{}, (ha + lane) % QCAP_A, tbase + ha + lane);
            ha += min(32, ta - ha);
        }
        while (tm - hm >= 32 || (flush && tm > hm)) {
            if (lane < tm - hm) eval(std::false_type{}, QCAP_A + (hm + lane) % QCAP_M, 0);
            hm += min(32, tm - hm);
        }
        __syncwarp();
        if (flush) break;
    }

    if (w < 3 && lane == 0) d.tl_n[i * 3 + w] = ta;
    const double ke = p.ke;
    R *buf = reinterpret_cast<R *>(&q);
    const R vals[15] = {acc.gr.x, acc.gr.y, acc.gr.z, acc.gm.x, acc.gm.y, acc.gm.z, acc.gt.xx, acc.gt.yy, acc.gt.zz,
                        acc.gt.xy, acc.gt.xz, acc.gt.yz, acc.ef.x, acc.ef.y, acc.ef.z};
    const R t = warp_transpose_sum<R, 15>(vals, buf, lane);
    // one destination per lane, so the FP64 update is a single warp instruction
    double *dst = nullptr;
    if (lane < 3) dst = d.gpt + (i * NP + w) * 3 + lane;
    else if (lane < 6) dst = d.gmu + (i * NS + w) * 3 + lane - 3;
    else if (lane < 12) dst = d.gth + (i * NS + w) * 6 + lane - 6;
    else if (lane < 15 && w < 3) dst = d.efield + i * 9 + w * 3 + lane - 12;
    if (dst) *dst += (lane < 6 ? ke : (lane < 12 ? ke * (1.0 / 3.0) : 1.0)) * double(t);
    // per-site energies (summed over the five sites in a fixed order by k_pol_energy)
    const double e0 = warp_sum_acc(acc.Ue), e1 = warp_sum_acc(acc.Up);
    if (lane == 0) {
        d.epw[(i * NS + w) * 2] = ke * e0;
        d.epw[(i * NS + w) * 2 + 1] = ke * e1;
    }
    if (VIR) {   // the site warps' virials in a fixed order
        const R wv = warp_transpose_sum<R, 9>(acc.W, buf, lane);
        if (lane < 9) s_w[wq][lane] = double(wv);
        __syncthreads();
        if (threadIdx.x < 9) {
            double v = 0;
            for (int k = 0; k < NW; ++k) v += s_w[k][threadIdx.x];
            d.vir[i * 9 + threadIdx.x] += ke * v;
        }
    }
}

// Gas phase: no cutoff, so no queue.  The lists of mpw consecutive molecules
// are taken one after another, 32 entries (target molecule, source molecule)
// a round; a lane evaluates the five sources of its entry in turn at target
// site w = blockIdx.y, and the entries of each molecule are then summed.  The
// energy, a quarter of the work here (see perm_pair), is the same from both
// sides of a pair: it is taken from the entries that own their pair (blockIdx.z
// = 0), and the others skip it.  Bound by issue and latency at 16 warps an SM (127
// registers).  4096 clusters of 17 waters 1282 -> 1050 us, 824
// waters in FP64 clusters 600 -> 510 us, against a warp per target site with queues.
template <typename R, bool VIR>
__global__ void __launch_bounds__(32, sizeof(R) == 4 ? GAS_BLOCKS : 8) k_perm_gas(KParams p, DevState<R> d, int mpw) {
    constexpr int NV = 19 + (VIR ? 9 : 0);
    __shared__ R buf[NV * 33];
    const int lane = threadIdx.x, w = blockIdx.y;
    const bool energy = blockIdx.z == 0;
    GasWalk walk(p, d, mpw, lane);
    double carry = 0.0;
    for (bool fresh = true; fresh = walk.at == 0, walk.next(lane);) {
        PermAcc<R> acc;
        acc.gr = mk(R(0), R(0), R(0));
        acc.gm = acc.gr;
        acc.ef = acc.gr;
        acc.gt = Sym<R>{};
#pragma unroll
        for (int k = 0; k < 9; ++k) acc.W[k] = R(0);
        const int i = walk.mol, slot = walk.slot;
        if (i >= 0 && slot >= 0) {
            const int j = d.nbr[i * MAXN + slot];
            const R *dp = d.ndo + ((size_t)i * MAXN + slot) * 3;
            const V3<R> D = mk(dp[0], dp[1], dp[2]);
            const Mp<R> mt = load_mp_g(d.gmp + (i * NS + w) * GMP);
            R Qi = R(0), Qj = R(0);   // molecule charges (remainders, see perm_pair)
            if (w == 0 && energy)
                for (int s = 0; s < NS; ++s) Qi += d.gmp[(i * NS + s) * GMP];
            const PermT<R> T{scaled(mt, R(1.0 / 3.0)), my_pt(d, i, w), zsite<R>(p, w) - mt.q, Qi, w};
            const GasRef<R> G(T, D);
            const size_t te = (size_t)(i * 3 + (w < 3 ? w : 0)) * p.tls + slot * 3;
            auto eval = [&](auto atom_src, int s) {
                constexpr bool AT = decltype(atom_src)::value;
                const Mp<R> m = load_mp_g(d.gmp + (j * NS + s) * GMP);
                Qj += m.q;
                V3<R> x;
                R g1 = R(0), T2 = R(0);
                perm_pair<R, false, AT, VIR>(p, T, G, scaled(m, R(1.0 / 3.0)), s, D, my_pt(d, j, s), energy, acc, g1,
                                              T2, x);
                if (AT && w < 3 && p.tlist) store_tpair(d, te + s, j * 3 + s, x, T2, g1);
            };
#pragma unroll 1
            for (int s = 0; s < 3; ++s) eval(std::true_type{}, s);
#pragma unroll 1
            for (int s = 3; s < NS; ++s) eval(std::false_type{}, s);
            // Q_j times the reference values of the target's terms: the
            // dipole/quadrupole ones and (O target only) the charge-charge one
            if (energy) {
                const R b23 = G.b2 * G.b2 * G.b2;
                R rem = G.yTy * b23 * G.b2 * G.b2 - G.mu * b23;
                if (w == 0) rem += Qi * G.b0;
                acc.Ue.add(Qj * rem);
            }
        }
        const R vals[19] = {acc.gr.x, acc.gr.y, acc.gr.z, acc.gm.x, acc.gm.y, acc.gm.z, acc.gt.xx,
                            acc.gt.yy, acc.gt.zz, acc.gt.xy, acc.gt.xz, acc.gt.yz, acc.ef.x, acc.ef.y,
                            acc.ef.z, acc.Ue.hi, acc.Ue.lo, acc.Up.hi, acc.Up.lo};
#pragma unroll
        for (int k = 0; k < NV; ++k) buf[k * 33 + lane] = k < 19 ? vals[k < 19 ? k : 0] : acc.W[k < 19 ? 0 : k - 19];
        __syncwarp();
        const double ke = p.ke;
        walk.segments(fresh, [&](int m, int c0, int c1, bool first) {
            double t = segment_sum<R>(buf, lane, NV, c0, c1);
            if (!first) t += carry;
            if (c1 == walk.n_used && walk.at != 0) {   // goes on in the next round
                carry = t;
                return;
            }
            double *dst = nullptr;
            if (lane < 3) dst = d.gpt + (m * NP + w) * 3 + lane;
            else if (lane < 6) dst = d.gmu + (m * NS + w) * 3 + lane - 3;
            else if (lane < 12) dst = d.gth + (m * NS + w) * 6 + lane - 6;
            else if (lane < 15 && w < 3) dst = d.efield + m * 9 + w * 3 + lane - 12;
            if (dst) atomicAdd(dst, (lane < 6 ? ke : (lane < 12 ? ke * (1.0 / 3.0) : 1.0)) * t);
            // per-site energies (summed over the five sites in a fixed order by k_pol_energy)
            const double e = ke * (t + __shfl_down_sync(0xffffffffu, t, 1));
            if (energy && (lane == 15 || lane == 17)) d.epw[(m * NS + w) * 2 + (lane == 17)] = e;
            // and the virials of the sites' two sides
            if (VIR && lane >= 19 && lane < NV) d.vir_w[(((size_t)m * NS + w) * 2 + blockIdx.z) * 9 + lane - 19] = ke * t;
            if (energy && w < 3 && lane == 0) d.tl_n[m * 3 + w] = 3 * d.nnbr[m];
        });
        __syncwarp();
    }
}

template <typename R>
void launch_real_perm(const KParams &p, DevState<R> &d, Launch L) {
    if (!p.periodic) {
        const int mpw = gas_mpw<R>(p);
        const dim3 g((unsigned)((p.M + mpw - 1) / mpw), NS, 2);
        if (p.vir) k_perm_gas<R, true><<<g, 32, 0, L.s>>>(p, d, mpw);
        else k_perm_gas<R, false><<<g, 32, 0, L.s>>>(p, d, mpw);
    } else if (p.vir) {
        k_real_perm<R, true><<<p.M, 32 * NS, 0, L.s>>>(p, d);
    } else {
        k_real_perm<R, false><<<p.M * NS, 32, 0, L.s>>>(p, d);
    }
    count(L);
}

// Potential of the permanent multipoles and its gradient at the lone pairs
// (ATOMS = false) or, for the original charge transfer, at O, H1 and H2: the
// five source sites share one queue.  FP32: a warp takes all of a molecule's
// points, which share the list walk, the queue and the source loads (32,000
// waters 270 us, a warp per point 376; 4096 clusters of 17 waters 109 and 155);
// FP64, bound by its pipe: a warp per point, which spreads the work.
constexpr int QCAP_P = 192;   // >= 31 carried + 5 sites x 32 new entries
template <typename R, bool PER, bool ATOMS>
__global__ void __launch_bounds__(128) k_potential(KParams p, DevState<R> d) {
    constexpr int NPT = ATOMS ? 3 : 2;                     // points a molecule
    constexpr int PW = sizeof(R) == 4 ? NPT : 1;           // points a warp
    __shared__ PairQueue<R, QCAP_P> qs[4];
    const int wq = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int a = (blockIdx.x * 4 + wq) * PW, i = a / NPT;   // first point, molecule
    if (i >= p.M) return;
    PairQueue<R, QCAP_P> &q = qs[wq];
    V3<R> ot[PW], gr[PW];
    Acc<R> V[PW];
#pragma unroll
    for (int u = 0; u < PW; ++u) {
        ot[u] = my_pt(d, i, (ATOMS ? 0 : NS) + a % NPT + u);
        gr[u] = mk(R(0), R(0), R(0));
    }
    const R rc2 = sc<R>(p).rc2, alpha = sc<R>(p).alpha;
    int h = 0, t = 0;
    const int nn = d.nnbr[i];
    for (int base = 0;; base += 32) {
        const bool flush = base >= nn;
        const int slot = base + lane;
        unsigned bits = 0;
        int j = 0;
        V3<R> rs[NS];
        if (slot < nn) {
            j = d.nbr[i * MAXN + slot];
            const R *dp = d.ndo + ((size_t)i * MAXN + slot) * 3;
            const V3<R> dO = mk(dp[0], dp[1], dp[2]);
            const R *offj = d.off + j * NP * 3;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                // queued: the source position in a box, the displacement of the molecules in the gas phase
                rs[s] = dO;
                if (!PER) {
                    bits |= 1u << s;
                    continue;
                }
                rs[s] = dO + mk(__ldg(offj + s * 3), __ldg(offj + s * 3 + 1), __ldg(offj + s * 3 + 2));
#pragma unroll
                for (int u = 0; u < PW; ++u) {
                    const V3<R> x = ot[u] - rs[s];
                    if (dot(x, x) < rc2) bits |= 1u << s;
                }
            }
        }
        int n;
        int k = warp_excl_scan(__popc(bits), lane, n);
#pragma unroll
        for (int s = 0; s < NS; ++s)
            if ((bits >> s) & 1u) q.put((t + k++) % QCAP_P, j * 8 + s, rs[s]);
        t += n;
        __syncwarp();
        while (t - h >= 32 || (flush && t > h)) {
            if (lane < t - h) {
                const int e = (h + lane) % QCAP_P, js = q.js[e];
                const Mp<R> ms = scaled(load_mp_g(d.gmp + ((js >> 3) * NS + (js & 7)) * GMP), R(1.0 / 3.0));
                V3<R> os = mk(R(0), R(0), R(0));
                if (!PER) os = my_pt(d, js >> 3, js & 7);
#pragma unroll
                for (int u = 0; u < PW; ++u) {
                    // gas phase: formed as (target - source offset) - D
                    const V3<R> x = PER ? ot[u] - q.at(e) : (ot[u] - os) - q.at(e);
                    const R r2 = dot(x, x);
                    if (PER && PW > 1 && !(r2 < rc2)) continue;   // queued for another point
                    const Source<R> src(ms, x);
                    const R rinv = rsqrt_(r2), r2i = rinv * rinv;
                    R B[4];
                    kernel_B<R, PER, 3>(r2 * rinv, rinv, r2i, alpha, B);
                    V[u].add(src.q * B[0] + src.s * B[1] + src.w * B[2]);
                    gr[u] = gr[u] + src.grad(x, B[1], B[2], B[3]);
                }
            }
            h += min(32, t - h);
        }
        __syncwarp();
        if (flush) break;
    }
    const double ke = p.ke;
    R vals[3 * PW];
#pragma unroll
    for (int u = 0; u < PW; ++u) vals[3 * u] = gr[u].x, vals[3 * u + 1] = gr[u].y, vals[3 * u + 2] = gr[u].z;
    const R g = warp_transpose_sum<R, 3 * PW>(vals, reinterpret_cast<R *>(&q), lane);
    if (lane < 3 * PW) (ATOMS ? d.dva : d.dvlp)[a * 3 + lane] += ke * double(g);
#pragma unroll
    for (int u = 0; u < PW; ++u) {
        const double v = warp_sum_acc(V[u]);
        if (lane == 0) (ATOMS ? d.va : d.vlp)[a + u] += ke * v;
    }
}

template <typename R, bool ATOMS>
void launch_potential(const KParams &p, DevState<R> &d, Launch L) {
    const int warps = p.M * (sizeof(R) == 4 ? 1 : (ATOMS ? 3 : 2));
    const unsigned nb = (unsigned)((warps + 3) / 4);
    if (p.periodic) k_potential<R, true, ATOMS><<<nb, 128, 0, L.s>>>(p, d);
    else k_potential<R, false, ATOMS><<<nb, 128, 0, L.s>>>(p, d);
    count(L);
}

// potential and field of the permanent multipoles at the lone pairs (real
// space); with the original charge transfer also at the atoms O, H1, H2
template <typename R>
void launch_lp_potential(const KParams &p, DevState<R> &d, Launch L) {
    launch_potential<R, false>(p, d, L);
    if (p.ct_orig) launch_potential<R, true>(p, d, L);
}

// ---------------------------------------------------------------------------
// Reduced charge transfer (Eqs. 13-16).  Donors: lone pairs; acceptors: O-H
// bonds of other molecules with carrier-O distance below rc.
// ---------------------------------------------------------------------------
template <typename R>
struct CtOut {
    R E, dV, dVi1, dVi2, dsh;
    V3<R> gc, glp, ga1, ga2;
};

// Vi1, Vi2: the acceptor atoms' potentials in e1, e2 (V_int; the original
// form adds V*); shift: subtracted from the denominator (the original form's
// V(a1)); dsh = dE/dshift.
template <typename R>
__device__ inline CtOut<R> ct_pair(const KParams &p, V3<R> c, V3<R> lp, V3<R> a1, V3<R> a2, R V, R Vi1, R Vi2,
                                   int *flags, R shift = R(0)) {
    CtOut<R> o;
    const Scal<R> &S = sc<R>(p);
    const R cs = S.cs_lp, cp = S.cp_lp, t = S.ct_t, mm = S.ct_m, n = S.nlp;
    const V3<R> v1 = a1 - c, v2 = a2 - c, u = lp - c;
    const R q1 = dot(v1, v1), q2 = dot(v2, v2);
    const R ir1 = rsqrt_(q1), ir2 = rsqrt_(q2), r1 = q1 * ir1, r2 = q2 * ir2;
    V3<R> du1, dv1, du2, dv2;
    const R ca = cosv(u, v1, du1, dv1);
    const R cb = cosv(u, v2, du2, dv2);
    const R E1 = exp_(-mulc(r1, p.ct_k1)), E2 = exp_(-mulc(r2, p.ct_k2));
    const R ek1 = cval<R>(p.ct_k1), ek2 = cval<R>(p.ct_k2);   // eta / (2 sqrt(rv rv))
    const R K1 = cs * t + cp * mm * ca, K2 = cs * t + cp * mm * cb;
    const R e1 = E1 * (Vi1 - V) * K1, e2 = E2 * (Vi2 - V) * K2;
    const R D = e1 - e2;
    const R dE = S.ct_ae + V - S.ct_ah - shift;
    if (!(dE > R(0))) atomicOr(flags, F_CTDEN);
    const R idE = rcp_(dE);
    o.E = -n * D * D * idE;
    const R gD = R(-2) * n * D * idE;
    o.dV = gD * (-E1 * K1 + E2 * K2) + n * D * D * idE * idE;
    o.dVi1 = gD * E1 * K1;
    o.dVi2 = -gD * E2 * K2;
    o.dsh = -n * D * D * idE * idE;
    const R dr1 = gD * (-ek1 * e1), dr2 = gD * (ek2 * e2);
    const R dca = gD * E1 * (Vi1 - V) * cp * mm, dcb = -gD * E2 * (Vi2 - V) * cp * mm;
    const V3<R> n1 = ir1 * v1, n2 = ir2 * v2;
    o.glp = dca * du1 + dcb * du2;
    o.ga1 = dr1 * n1 + dca * dv1;
    o.ga2 = dr2 * n2 + dcb * dv2;
    o.gc = R(-1) * (o.glp + o.ga1 + o.ga2);
    return o;
}

// Bare potential (times ke) of the five multipole sites of molecule m at a
// point y given relative to m's O: the donor's part of an acceptor atom's
// potential in the original charge transfer.
template <typename R>
__device__ inline R mol_phi(const KParams &p, const DevState<R> &d, int m, V3<R> y) {
    R phi = R(0);
#pragma unroll 1
    for (int s = 0; s < NS; ++s) {
        const Mp<R> M = load_mp_g(d.gmp + (m * NS + s) * GMP);
        const V3<R> x = y - my_pt(d, m, s);
        R g[3];
        g_bare<R, 2>(rsqrt_(dot(x, x)), g);
        FieldTerms<R> f;
        source_field<R, 0>(M, x, g, f);
        phi += f.phi;
    }
    return R(p.ke) * phi;
}

// Working-precision per-molecule inputs of the charge transfer, so the pair
// loop reads no FP64: the lone-pair potentials (real space + reciprocal
// chain), V_int of O, H1, H2 and, for the original form, V(a) of O, H1, H2.
constexpr int CT_IN = 8;
template <typename R>
__global__ void k_ct_prep(int M, int orig, DevState<R> d) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    R *o = d.ctin + m * CT_IN;
    o[0] = R(d.vlp[m * 2] + d.vlp_r[m * 2]);
    o[1] = R(d.vlp[m * 2 + 1] + d.vlp_r[m * 2 + 1]);
    for (int a = 0; a < 3; ++a) {
        o[2 + a] = R(d.vint[m * 3 + a]);
        o[5 + a] = orig ? R(d.va[m * 3 + a] + d.va_r[m * 3 + a]) : R(0);
    }
}

// VIR: the virial of the pair terms by translation invariance: with X_p =
// O_i + off_p, sum over a molecule pair of g_p (x) X_p = sum_{p of i} g_p (x)
// off_p + sum_{p of j} g_p (x) off_p - G_{i<-j} (x) dO_ij, where G_{i<-j} is
// the total gradient on i's points and dO_ij = O_j - O_i; each side adds
// its own offsets term and half of the last one.
// One warp per molecule i.  The neighbour list is read 32 slots at a time;
// the slots inside the cutoff (carrier-carrier distance) are queued in
// shared memory and taken in full 32-lane rounds, each lane one molecule
// pair with its 8 donor-acceptor items (i donating to j and j to i).
template <typename R> constexpr int CW = sizeof(R) == 4 ? 4 : 1;   // molecules a block
template <typename R, bool PER, bool VIR>
__global__ void __launch_bounds__(32 * CW<R>) k_ct(KParams p, DevState<R> d) {
    __shared__ R red[CW<R>][23 * 33];
    __shared__ int sq[CW<R>][64];
    const int wq = threadIdx.x >> 5;
    const int i = blockIdx.x * CW<R> + wq;
    const int lane = threadIdx.x & 31;
    if (i >= p.M) return;
    const R rc2 = sc<R>(p).rc2;
    V3<R> P[5];
    for (int k = 0; k < 3; ++k) P[k] = my_pt(d, i, k);
    P[3] = my_pt(d, i, 5);
    P[4] = my_pt(d, i, 6);
    const R *in_i = d.ctin + i * CT_IN;
    const R Vi[2] = {in_i[0], in_i[1]};
    const R Vint_i[3] = {in_i[2], in_i[3], in_i[4]};
    V3<R> G[5];
    for (int k = 0; k < 5; ++k) G[k] = mk(R(0), R(0), R(0));
    R lam[2] = {R(0), R(0)}, kap[3] = {R(0), R(0), R(0)};
    // original form: the acceptor potentials V(a) of i's atoms and dE/dV(a)
    const bool orig = p.ct_orig != 0;
    const R Va_i[3] = {in_i[5], in_i[6], in_i[7]};
    R lama[3] = {R(0), R(0), R(0)};
    R W[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) W[k] = R(0);
    Acc<R> Ect;
    auto pair = [&](int slot) {
        const int j = d.nbr[i * MAXN + slot];
        const R *dp_ = d.ndo + ((size_t)i * MAXN + slot) * 3;
        const V3<R> dO = mk(dp_[0], dp_[1], dp_[2]);
        V3<R> Q[5];
        Q[0] = dO;
        Q[1] = dO + my_pt(d, j, 1);
        Q[2] = dO + my_pt(d, j, 2);
        Q[3] = dO + my_pt(d, j, 5);
        Q[4] = dO + my_pt(d, j, 6);
        const R *in_j = d.ctin + j * CT_IN;
        const R Vj[2] = {in_j[0], in_j[1]};
        // original form: W = V_int + V* in e1, e2 and V(a1) in the denominator,
        // V*(a) = V(a) minus the donor molecule's bare potential at a
        R Wj[3] = {in_j[2], in_j[3], in_j[4]}, Wi[3] = {Vint_i[0], Vint_i[1], Vint_i[2]};
        R sh_j = R(0), sh_i = R(0);
        R cd[3] = {R(0), R(0), R(0)}, ca[3] = {R(0), R(0), R(0)};
        if (orig) {
            for (int a = 0; a < 3; ++a) {
                Wj[a] += in_j[5 + a] - mol_phi(p, d, i, Q[a]);      // i's sites at j's atom a
                Wi[a] += Va_i[a] - mol_phi(p, d, j, P[a] - dO);      // j's sites at i's atom a
            }
            sh_j = in_j[5];
            sh_i = Va_i[0];
        }
        V3<R> Gj = mk(R(0), R(0), R(0));   // gradient on i's points from j (virial)
        for (int l = 0; l < 2; ++l)
            for (int k = 1; k <= 2; ++k) {
                // i donor (lone pair l of i), j acceptor (bond O-H_k of j)
                CtOut<R> o = ct_pair(p, P[0], P[3 + l], Q[0], Q[k], Vi[l], Wj[0], Wj[k], d.flags, sh_j);
                Ect.add(R(0.5) * o.E);
                G[0] = G[0] + o.gc;
                G[3 + l] = G[3 + l] + o.glp;
                lam[l] += o.dV;
                cd[0] += o.dVi1;
                cd[k] += o.dVi2;
                // j donor (lone pair l of j), i acceptor (bond O-H_k of i)
                CtOut<R> q = ct_pair(p, Q[0], Q[3 + l], P[0], P[k], Vj[l], Wi[0], Wi[k], d.flags, sh_i);
                Ect.add(R(0.5) * q.E);
                G[0] = G[0] + q.ga1;
                G[k] = G[k] + q.ga2;
                kap[0] += q.dVi1;
                kap[k] += q.dVi2;
                ca[0] += q.dVi1;
                ca[k] += q.dVi2;
                lama[0] += q.dVi1 + q.dsh;
                lama[k] += q.dVi2;
                if (VIR) Gj = Gj + o.gc + o.glp + q.ga1 + q.ga2;
            }
        if (orig) {
            R *cv = d.cvs + ((size_t)i * MAXN + slot) * 6;
            for (int a = 0; a < 3; ++a) cv[a] = cd[a], cv[3 + a] = ca[a];
        }
        if (VIR) vir_add(W, Gj, dO, R(-0.5));
    };
    int *q = sq[wq];
    int cnt = 0, base = 0;   // queued slots and next list slot (warp-uniform)
    const int nn = d.nnbr[i];
    for (;;) {
        while (cnt < 32 && base < nn) {
            const int slot = base + lane;
            bool in = false;
            if (slot < nn) {
                in = true;
                if (PER) {
                    const R *dp_ = d.ndo + ((size_t)i * MAXN + slot) * 3;
                    const R x = dp_[0], y = dp_[1], z = dp_[2];
                    in = x * x + y * y + z * z < rc2;
                }
                if (!in && orig) {   // no transfer: zero sensitivities for k_ct_vstar
                    R *cv = d.cvs + ((size_t)i * MAXN + slot) * 6;
                    for (int k = 0; k < 6; ++k) cv[k] = R(0);
                }
            }
            const unsigned b = __ballot_sync(0xffffffffu, in);
            if (in) q[cnt + __popc(b & ((1u << lane) - 1u))] = slot;
            cnt += __popc(b);
            base += 32;
            __syncwarp();
        }
        if (cnt == 0) break;
        const int take = cnt < 32 ? cnt : 32;
        if (lane < take) pair(q[lane]);
        __syncwarp();
        if (lane < cnt - take) q[lane] = q[take + lane];
        cnt -= take;
        __syncwarp();
    }
    const R vals[23] = {G[0].x, G[0].y, G[0].z, G[1].x, G[1].y, G[1].z, G[2].x, G[2].y, G[2].z,
                        G[3].x, G[3].y, G[3].z, G[4].x, G[4].y, G[4].z, lam[0], lam[1], kap[0], kap[1], kap[2],
                        lama[0], lama[1], lama[2]};
    const R t = warp_transpose_sum<R, 23>(vals, red[wq], lane);
    const int pt = lane / 3;
    double *dst = nullptr;
    if (lane < 15) dst = d.gpt + (i * NP + (pt < 3 ? pt : pt + 2)) * 3 + lane % 3;
    else if (lane < 17) dst = d.lam + i * 2 + lane - 15;
    else if (lane < 20) dst = d.kap + i * 3 + lane - 17;
    else if (lane < 23 && orig) dst = d.lama + i * 3 + lane - 20;
    if (dst) *dst += double(t);
    if (VIR) vir_points_out(d, i, P, t, W, red[wq], lane);
    const double e = warp_sum_acc(Ect);
    if (lane == 0) d.epart[i * NTERM + T_CT] += e;
}

// Original charge transfer, the dependence through V*(a) = V(a) - phi_D(a)
// (phi_D: the donor molecule's bare potential at the acceptor atom a) and
// through V(a).  With c = dE/dV*(a) per neighbour slot (k_ct: 0-2 at the
// partner's atoms for i donating, 3-5 at i's atoms for the partner
// donating) the energy varies as -sum c phi_D(a).  Warps 0-4: site s of i as
// the donor's source, point charges -c at the partners' atoms acting on its
// multipole (gradient at the site and multipole sensitivities); warps 5-7:
// atom a of i as the acceptor, the gradient of -c phi_j at the atom, plus
// the atom's own share of dE/dV(a) times the gradient of V(a) (the partners'
// share, charges dE/dV(a) on the atoms in the potential of every site, is
// taken in the force pass).
template <typename R>
__global__ void __launch_bounds__(256) k_ct_vstar(KParams p, DevState<R> d) {
    __shared__ R red[8][12 * 33];
    const int i = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nn = d.nnbr[i];
    const R third = R(1) / R(3);
    V3<R> gr = mk(R(0), R(0), R(0)), gm = gr;
    Sym<R> gt{};
    if (w < NS) {
        const Mp<R> mt = load_mp(d.gmp + (i * NS + w) * GMP);
        const V3<R> ot = my_pt(d, i, w);
        for (int slot = lane; slot < nn; slot += 32) {
            const R *c = d.cvs + ((size_t)i * MAXN + slot) * 6;
            if (c[0] == R(0) && c[1] == R(0) && c[2] == R(0)) continue;
            const int j = d.nbr[i * MAXN + slot];
            const R *dp = d.ndo + ((size_t)i * MAXN + slot) * 3;
            const V3<R> dO = mk(dp[0], dp[1], dp[2]);
            for (int a = 0; a < 3; ++a) {
                Mp<R> ms{};
                ms.q = -c[a];
                const V3<R> x = ot - (dO + my_pt(d, j, a));
                R g[6];   // source_field to third derivatives reads g_0..g_5
                g_bare<R, 5>(rsqrt_(dot(x, x)), g);
                FieldTerms<R> f;
                source_field<R, 3>(ms, x, g, f);
                gr = gr + target_grad(mt, ms, x, g, f);
                gm = gm + f.d1;
                symadd(gt, f.d2, third);
            }
        }
    } else {
        const int a = w - NS;
        const V3<R> ot = my_pt(d, i, a);
        for (int slot = lane; slot < nn; slot += 32) {
            const R c = d.cvs[((size_t)i * MAXN + slot) * 6 + 3 + a];
            if (c == R(0)) continue;
            const int j = d.nbr[i * MAXN + slot];
            const R *dp = d.ndo + ((size_t)i * MAXN + slot) * 3;
            const V3<R> dO = mk(dp[0], dp[1], dp[2]);
            for (int s = 0; s < NS; ++s) {
                const Mp<R> ms = load_mp_g(d.gmp + (j * NS + s) * GMP);
                const V3<R> x = ot - (dO + my_pt(d, j, s));
                R g[4];
                g_bare<R, 3>(rsqrt_(dot(x, x)), g);
                FieldTerms<R> f;
                source_field<R, 1>(ms, x, g, f);
                gr = gr - c * f.d1;
            }
        }
    }
    const R vals[12] = {gr.x, gr.y, gr.z, gm.x, gm.y, gm.z, gt.xx, gt.yy, gt.zz, gt.xy, gt.xz, gt.yz};
    const R t = warp_transpose_sum<R, 12>(vals, red[w], lane);
    const double ke = p.ke;
    // warps w < 3 (sites O, H1, H2) and 5 + w (the same atoms) both add to
    // the atom's point gradient: atomically
    if (w < NS) {
        if (lane < 3) atomicAdd(d.gpt + (i * NP + w) * 3 + lane, ke * double(t));
        else if (lane < 6) d.gmu[(i * NS + w) * 3 + lane - 3] += ke * double(t);
        else if (lane < 12) d.gth[(i * NS + w) * 6 + lane - 6] += ke * double(t);
    } else if (lane < 3) {
        const int a = w - NS;
        const double gv = d.dva[(i * 3 + a) * 3 + lane] + d.dva_r[(i * 3 + a) * 3 + lane];
        atomicAdd(d.gpt + (i * NP + a) * 3 + lane, ke * double(t) + d.lama[i * 3 + a] * gv);
    }
}

template <typename R>
void launch_ct(const KParams &p, DevState<R> &d, Launch L) {
    k_ct_prep<R><<<(p.M + 127) / 128, 128, 0, L.s>>>(p.M, p.ct_orig, d);
    count(L);
    const unsigned nb = (p.M + CW<R> - 1) / CW<R>;
    if (p.vir) {
        if (p.periodic) k_ct<R, true, true><<<nb, 32 * CW<R>, 0, L.s>>>(p, d);
        else k_ct<R, false, true><<<nb, 32 * CW<R>, 0, L.s>>>(p, d);
    } else {
        if (p.periodic) k_ct<R, true, false><<<nb, 32 * CW<R>, 0, L.s>>>(p, d);
        else k_ct<R, false, false><<<nb, 32 * CW<R>, 0, L.s>>>(p, d);
    }
    count(L);
    if (p.ct_orig) {
        k_ct_vstar<R><<<p.M, 256, 0, L.s>>>(p, d);
        count(L);
    }
}

// ---------------------------------------------------------------------------
// Polarization matrix-vector product, real-space part: field at each
// polarizable atom from the dipoles vecR of the atoms of other molecules
// within rc (Thole-damped, Ewald-screened in periodic systems), streamed from
// the pair list that the permanent pass recorded.  out += field.  One warp
// per polarizable atom; each lane keeps four entries in flight.
// ---------------------------------------------------------------------------
constexpr int TW = 8;   // warps per block

// entry: partner atom index (the sign of g2 in its top bit), y = sqrt|g2| x, g1
template <typename R>
__device__ inline void tmu_entry(const DevState<R> &d, size_t k, int jraw, V3<R> &ef) {
    const R *mv = d.vecR + (jraw & 0x7fffffff) * 3;
    const V3<R> mu = mk(mv[0], mv[1], mv[2]);
    const V3<R> y = mk(d.tl_x[k], d.tl_y[k], d.tl_z[k]);
    const R my = dot(mu, y);
    ef = ef + (jraw < 0 ? -my : my) * y + d.tl_g1[k] * mu;
}

template <typename R>
__global__ void __launch_bounds__(32 * TW) k_real_tmu(int M, int tls, DevState<R> d, double *out) {
    __shared__ R red[TW][3 * 33];
    if (d.flags[1]) return;   // solver already converged
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * TW + w;
    if (t >= M * 3) return;
    const int n = d.tl_n[t];
    const size_t base = (size_t)t * tls;
    V3<R> ef = mk(R(0), R(0), R(0));
    int e = lane;
    for (; e + 96 < n; e += 128) {
        int jb[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) jb[u] = d.tl_j[base + e + 32 * u];
#pragma unroll
        for (int u = 0; u < 4; ++u) tmu_entry(d, base + e + 32 * u, jb[u], ef);
    }
    for (; e < n; e += 32) tmu_entry(d, base + e, d.tl_j[base + e], ef);
    const R vals[3] = {ef.x, ef.y, ef.z};
    const R s = warp_transpose_sum<R, 3>(vals, red[w], lane);
    if (lane < 3) out[t * 3 + lane] += double(s);
}

template <typename R>
void launch_real_tmu(const KParams &p, DevState<R> &d, double *out, Launch L) {
    k_real_tmu<R><<<(p.M * 3 + TW - 1) / TW, 32 * TW, 0, L.s>>>(p.M, p.tls, d, out);
    count(L);
}

// ---------------------------------------------------------------------------
// Polarization forces, real-space part, at fixed induced dipoles mu and
// charge-transfer sensitivities lambda (point charges on the lone pairs):
//   target site t of i:  d/dr_t and multipole sensitivities of
//       sum_b U(M_t, mu_b)   (Thole-damped)     + sum_l U(M_t, lambda_l) (undamped)
//   target pol atom a of i (a = t < 3): d/dr_a of
//       sum_s U(mu_a, M_s) + sum_b U(mu_a, mu_b)  (Thole-damped)
// One warp per target site; work queues as in the permanent kernel with
// three classes: atom sources (induced dipole and, for a polarizable target,
// permanent multipole, sharing one Thole kernel), midpoint sources
// (permanent multipole, polarizable targets only) and lambda charges.
// ---------------------------------------------------------------------------
constexpr int PQ_A = 128, PQ_M = 96, PQ_L = 96;

template <typename R>
struct PfAcc {
    V3<R> gr, gm;
    Sym<R> gt;   // three times the quadrupole sensitivity
    R W[9];      // virial (VIR kernels only)
};

// VIR: also accumulate the pair virial g (x) x of the target's gradient g:
// half of it for dipole and multipole sources (the partner adds the other
// half), all of it for lambda charges (whose lone-pair side adds none).
//
// Each source is evaluated for what it has: the dipole and charge sources
// carry no quadrupole, and at a polarizable target the source's permanent and
// induced dipoles act on the target's induced dipole through one second
// derivative, contracted as it is formed.  mt: quadrupole / 3.
template <typename R, bool PER, int KIND, bool VIR>   // KIND 0: atom source, 1: midpoint source, 2: lambda charge
__device__ __forceinline__ void polf_pair(const KParams &p, const DevState<R> &d, int w, V3<R> ot, const Mp<R> &mt,
                                          V3<R> mui, int js, V3<R> rs, PfAcc<R> &A) {
    const Scal<R> &S = sc<R>(p);
    const int j = js >> 3, s = js & 7;
    const V3<R> x = ot - rs;
    const R r2 = dot(x, x);
    const R rinv = rsqrt_(r2), r = r2 * rinv, r2i = rinv * rinv;
    // charge source c at the target multipole: gradient and sensitivities
    auto charge = [&](R c, const R *B, const Target<R> &t) {
        const R P = -c * B[1], Q = c * B[2];
        const V3<R> d1 = P * x;
        A.gm = A.gm + d1;
        const V3<R> qx = Q * x;
        A.gt.xx += P + qx.x * x.x; A.gt.yy += P + qx.y * x.y; A.gt.zz += P + qx.z * x.z;
        A.gt.xy += qx.x * x.y; A.gt.xz += qx.x * x.z; A.gt.yz += qx.y * x.z;
        return (t.q * P + t.s * Q - t.w * c * B[3]) * x + P * t.mu + (Q + Q) * t.p;
    };
    if (KIND == 2) {
        R B[4];
        kernel_B<R, PER, 3>(r, rinv, r2i, S.alpha, B);
        const Target<R> t(mt, x);
        const V3<R> gl = charge(d.lamR[j * 2 + s], B, t);
        A.gr = A.gr + gl;
        if (VIR) vir_add(A.W, gl, x, R(1));
        return;
    }
    R B[5], T[5];
    kernel_B<R, PER, 4>(r, rinv, r2i, S.alpha, B);
    {
        const R u = S.thole * r2 * r * ainv3<R>(p, w, s);
        const R e = exp_(-u), ue = u * e, u2e = u * ue;
        const R c2 = e + ue, c3 = c2 + R(0.6) * u2e;
        const R c4 = c2 + R(18.0 / 35.0) * u2e + R(9.0 / 35.0) * u * u2e;
        const R b1 = rinv * r2i, b2 = R(3) * b1 * r2i, b3 = R(5) * b2 * r2i, b4 = R(7) * b3 * r2i;
        T[1] = B[1] - e * b1;
        T[2] = B[2] - c2 * b2;
        T[3] = B[3] - c3 * b3;
        T[4] = B[4] - c4 * b4;
    }
    V3<R> gv = mk(R(0), R(0), R(0));
    V3<R> b = gv;
    if (KIND == 0) {   // induced dipole b of atom s of j at target site w
        const R *mj = d.muR + j * 9 + s * 3;
        b = mk(mj[0], mj[1], mj[2]);
        const Target<R> t(mt, x);
        const R sb = dot(b, x), P = -sb * T[2], Rr = sb * T[3];
        const V3<R> U = (-T[2]) * b, W = T[3] * b;
        const V3<R> d1 = P * x + T[1] * b;
        const Sym<R> d2 = second(x, P, Rr * x + U, U);
        A.gm = A.gm + d1;
        symacc(A.gt, d2);
        const V3<R> pu = symv(t.th, U);
        const R c = R(2) * dot(t.p, W) - t.w * sb * T[4];
        gv = t.q * d1 + symv(d2, t.mu) + (Rr + Rr) * t.p + R(2) * pu + c * x + t.w * W;
        if (p.ct_orig) {   // original charge transfer: dE/dV(a) as a charge on atom s of j, undamped
            const V3<R> gl = charge(d.lamaR[j * 3 + s], B, t);
            A.gr = A.gr + gl;
        }
    }
    if (w < 3) {
        // permanent multipoles (and induced dipole) of site s of j at the
        // induced dipole m of polarizable atom w: d/dx of m . grad phi
        Mp<R> m = load_mp_g(d.gmp + (j * NS + s) * GMP);
        if (KIND == 0) m.mu = m.mu + b;
        const Source<R> q(scaled(m, R(1.0 / 3.0)), x);
        const R P = -(q.q * T[1] + q.s * T[2] + q.w * T[3]);
        const R Rr = q.q * T[2] + q.s * T[3] + q.w * T[4];
        const V3<R> U = (-T[2]) * q.mu + (R(-2) * T[3]) * q.v;
        const R xm = dot(x, mui);
        gv = gv + P * mui + (Rr * xm + dot(U, mui)) * x + xm * U + (T[2] + T[2]) * symv(q.th, mui);
    }
    A.gr = A.gr + gv;
    if (VIR) vir_add(A.W, gv, x, R(0.5));
}

// One target site of one molecule per block of one warp (the virial variant:
// the five sites of a molecule in one block, summed in a fixed order).
template <typename R, bool PER, bool VIR>
__global__ void __launch_bounds__(VIR ? 32 * NS : 32, VIR ? 3 : (sizeof(R) == 4 ? 32 : 8))
    k_real_polforce(KParams p, DevState<R> d) {
    constexpr int NW = VIR ? NS : 1;
    __shared__ double s_w[VIR ? NW : 1][9];
    __shared__ PairQueue<R, PQ_A + PQ_M + PQ_L> qs[NW];
    static_assert(sizeof(PairQueue<R, PQ_A + PQ_M + PQ_L>) >= 12 * 33 * sizeof(R), "reduction buffer");
    const int wq = VIR ? threadIdx.x >> 5 : 0, lane = threadIdx.x & 31;
    const int i = VIR ? blockIdx.x : blockIdx.x / NS;
    const int w = VIR ? wq : blockIdx.x % NS;   // target site
    PairQueue<R, PQ_A + PQ_M + PQ_L> &q = qs[wq];
    const V3<R> ot = my_pt(d, i, w);
    const Mp<R> mt = scaled(load_mp(d.gmp + (i * NS + w) * GMP), R(1.0 / 3.0));
    V3<R> mui = mk(R(0), R(0), R(0));
    if (w < 3) mui = mk(d.muR[i * 9 + w * 3], d.muR[i * 9 + w * 3 + 1], d.muR[i * 9 + w * 3 + 2]);
    const R rc2 = sc<R>(p).rc2;
    PfAcc<R> A;
    A.gr = mk(R(0), R(0), R(0));
    A.gm = A.gr;
    A.gt = Sym<R>{};
#pragma unroll
    for (int k = 0; k < 9; ++k) A.W[k] = R(0);
    int ha = 0, ta = 0, hm = 0, tm = 0, hl = 0, tl = 0;
    const int nn = d.nnbr[i];
    for (int base = 0;; base += 32) {
        const bool flush = base >= nn;
        const int slot = base + lane;
        unsigned bits = 0;   // bits 0-4 sites, 5-6 lone pairs
        int j = 0;
        V3<R> rs[NP];
        if (slot < nn) {
            j = d.nbr[i * MAXN + slot];
            const R *dp = d.ndo + ((size_t)i * MAXN + slot) * 3;
            const V3<R> dO = mk(dp[0], dp[1], dp[2]);
            const R *offj = d.off + j * NP * 3;
#pragma unroll
            for (int s = 0; s < NP; ++s) {
                rs[s] = dO + mk(__ldg(offj + s * 3), __ldg(offj + s * 3 + 1), __ldg(offj + s * 3 + 2));
                const V3<R> x = ot - rs[s];
                const bool in = !PER || dot(x, x) < rc2;
                const bool want = s < 3 || (s < NS ? w < 3 : d.lamR[j * 2 + s - NS] != R(0));
                if (in && want) bits |= 1u << s;
            }
        }
        int na, nm, nl;
        int pa = warp_excl_scan(__popc(bits & 7u), lane, na);
        int pm = warp_excl_scan(__popc((bits >> 3) & 3u), lane, nm);
        int pl = warp_excl_scan(__popc(bits >> 5), lane, nl);
#pragma unroll
        for (int s = 0; s < NP; ++s) {
            if (!((bits >> s) & 1u)) continue;
            if (s < 3) q.put((ta + pa++) % PQ_A, j * 8 + s, rs[s]);
            else if (s < NS) q.put(PQ_A + (tm + pm++) % PQ_M, j * 8 + s, rs[s]);
            else q.put(PQ_A + PQ_M + (tl + pl++) % PQ_L, j * 8 + s - NS, rs[s]);
        }
        ta += na;
        tm += nm;
        tl += nl;
        __syncwarp();
        while (ta - ha >= 32 || (flush && ta > ha)) {
            if (lane < ta - ha) {
                const int e = (ha + lane) % PQ_A;
                polf_pair<R, PER, 0, VIR>(p, d, w, ot, mt, mui, q.js[e], q.at(e), A);
            }
            ha += min(32, ta - ha);
        }
        while (tm - hm >= 32 || (flush && tm > hm)) {
            if (lane < tm - hm) {
                const int e = PQ_A + (hm + lane) % PQ_M;
                polf_pair<R, PER, 1, VIR>(p, d, w, ot, mt, mui, q.js[e], q.at(e), A);
            }
            hm += min(32, tm - hm);
        }
        while (tl - hl >= 32 || (flush && tl > hl)) {
            if (lane < tl - hl) {
                const int e = PQ_A + PQ_M + (hl + lane) % PQ_L;
                polf_pair<R, PER, 2, VIR>(p, d, w, ot, mt, mui, q.js[e], q.at(e), A);
            }
            hl += min(32, tl - hl);
        }
        __syncwarp();
        if (flush) break;
    }
    const double ke = p.ke;
    const R vals[12] = {A.gr.x, A.gr.y, A.gr.z, A.gm.x, A.gm.y, A.gm.z,
                        A.gt.xx, A.gt.yy, A.gt.zz, A.gt.xy, A.gt.xz, A.gt.yz};
    const R s = warp_transpose_sum<R, 12>(vals, reinterpret_cast<R *>(&q), lane);
    double *dst = nullptr;
    if (lane < 3) dst = d.gpt + (i * NP + w) * 3 + lane;
    else if (lane < 6) dst = d.gmu + (i * NS + w) * 3 + lane - 3;
    else if (lane < 12) dst = d.gth + (i * NS + w) * 6 + lane - 6;
    if (dst) *dst += (lane < 6 ? ke : ke * (1.0 / 3.0)) * double(s);
    if (VIR) {   // the warps' virials summed in a fixed order
        const R wv = warp_transpose_sum<R, 9>(A.W, reinterpret_cast<R *>(&q), lane);
        if (lane < 9) s_w[wq][lane] = double(wv);
        __syncthreads();
        if (threadIdx.x < 9) {
            double v = 0;
            for (int k = 0; k < NW; ++k) v += s_w[k][threadIdx.x];
            d.vir[i * 9 + threadIdx.x] += ke * v;
        }
    }
}

template <typename R>
void launch_real_polforce(const KParams &p, DevState<R> &d, Launch L) {
    if (p.vir) {
        if (p.periodic) k_real_polforce<R, true, true><<<p.M, 32 * NS, 0, L.s>>>(p, d);
        else k_real_polforce<R, false, true><<<p.M, 32 * NS, 0, L.s>>>(p, d);
    } else {
        if (p.periodic) k_real_polforce<R, true, false><<<p.M * NS, 32, 0, L.s>>>(p, d);
        else k_real_polforce<R, false, false><<<p.M * NS, 32, 0, L.s>>>(p, d);
    }
    count(L);
}

#define INST(R)                                                                                    \
    template void launch_real_perm<R>(const KParams &, DevState<R> &, Launch);                     \
    template void launch_lp_potential<R>(const KParams &, DevState<R> &, Launch);                  \
    template void launch_ct<R>(const KParams &, DevState<R> &, Launch);                            \
    template void launch_real_tmu<R>(const KParams &, DevState<R> &, double *, Launch);             \
    template void launch_real_polforce<R>(const KParams &, DevState<R> &, Launch);
INST(float)
INST(double)

}  // namespace sibfa
