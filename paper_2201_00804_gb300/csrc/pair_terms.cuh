// Multipole pair terms shared by the pair kernels.  Kernels appear as the positive B_n =
// (-1)^n g_n, quadrupoles as a third of their value (the 1/3 of the multipole
// convention taken once per load), and the products of a multipole with the
// displacement are formed once and reused by the energy, the gradient, the
// penetration and the Thole field.
#pragma once
#include "sibfa_internal.cuh"

namespace sibfa {

template <typename R>
__device__ inline Mp<R> scaled(const Mp<R> &m, R s) {   // quadrupole times s
    return {m.q, m.mu, {s * m.th.xx, s * m.th.yy, s * m.th.zz, s * m.th.xy, s * m.th.xz, s * m.th.yz}};
}

// B_0..B_N of erfc(alpha r)/r or of 1/r
template <typename R, bool PER, int N>
__device__ __forceinline__ void kernel_B(R r, R rinv, R r2i, R alpha, R (&B)[N + 1]) {
    if (PER) {
        const R ar = alpha * r;
        const R ex = exp_(R(-1.0) * ar * ar) * (R(0.56418958354775628695) * rcp_(alpha));
        const R tw = R(2.0) * alpha * alpha;
        R p = tw;
        B[0] = erfc_(ar) * rinv;
#pragma unroll
        for (int n = 1; n <= N; ++n) {
            B[n] = (R(2.0 * n - 1) * B[n - 1] + p * ex) * r2i;
            p = p * tw;
        }
    } else {
        B[0] = rinv;
#pragma unroll
        for (int n = 1; n <= N; ++n) B[n] = R(2.0 * n - 1) * B[n - 1] * r2i;
    }
}
// B_0..B_3 of exp(-b r)/r, x = b r
template <typename R>
__device__ __forceinline__ void kernel_exp(R x, R rinv, R r2i, R (&E)[4]) {
    const R t1 = x + R(1.0), x2 = x * x, t2 = R(3.0) * t1 + x2, t3 = R(5.0) * t2 + x2 * t1;
    R e = exp_(R(-1.0) * x) * rinv;
    E[0] = e;
    e = e * r2i;
    E[1] = t1 * e;
    e = e * r2i;
    E[2] = t2 * e;
    e = e * r2i;
    E[3] = t3 * e;
}

// What a source multipole's field evaluations at x (target minus source) share
template <typename R>
struct Source {
    R q, s, w;      // charge, mu.x, x.(Theta/3).x
    V3<R> mu, v;    // dipole, (Theta/3) x
    Sym<R> th;      // Theta / 3
    __device__ __forceinline__ Source(const Mp<R> &m, V3<R> x)
        : q(m.q), s(dot(m.mu, x)), mu(m.mu), v(symv(m.th, x)), th(m.th) {
        w = dot(x, v);
    }
    // grad phi without the charge: -P x + B1 mu + 2 B2 v
    __device__ __forceinline__ V3<R> grad_mp(V3<R> x, R b1, R b2, R b3) const {
        const R P = R(-1.0) * (s * b2 + w * b3), c = b2 + b2;
        return P * x + b1 * mu + c * v;
    }
    __device__ __forceinline__ V3<R> grad(V3<R> x, R b1, R b2, R b3) const {
        const R P = R(-1.0) * (q * b1 + s * b2 + w * b3), c = b2 + b2;
        return P * x + b1 * mu + c * v;
    }
};

// Second derivatives of the potential and the vectors of the third-order contraction
template <typename R>
struct Field2 {
    R P, Rr;          // coefficients of x in the gradient and of x x in the second derivatives
    V3<R> U, d1;      // vector of the mixed terms x U + U x, gradient
    Sym<R> d2;
};
template <typename R>
__device__ __forceinline__ Sym<R> second(V3<R> x, R P, V3<R> a, V3<R> U) {   // P delta + x a + U x
    return {P + x.x * a.x + U.x * x.x, P + x.y * a.y + U.y * x.y, P + x.z * a.z + U.z * x.z,
            x.x * a.y + U.x * x.y,     x.x * a.z + U.x * x.z,     x.y * a.z + U.y * x.z};
}
template <typename R>
__device__ __forceinline__ Sym<R> plus(const Sym<R> &a, R c, const Sym<R> &b) {
    return {a.xx + c * b.xx, a.yy + c * b.yy, a.zz + c * b.zz, a.xy + c * b.xy, a.xz + c * b.xz, a.yz + c * b.yz};
}

// A target multipole's products with the displacement
template <typename R>
struct Target {
    R q, s, w;      // charge, mu.x, x.(Phi/3).x
    V3<R> mu, p;    // dipole, (Phi/3) x
    Sym<R> th;
    __device__ __forceinline__ Target(const Mp<R> &m, V3<R> x)
        : q(m.q), s(dot(m.mu, x)), mu(m.mu), p(symv(m.th, x)), th(m.th) {
        w = dot(x, p);
    }
};

// Gradient of the target's energy in the source's field (kernels B0..B5),
// with its first and second derivatives left in F.
template <typename R>
__device__ __forceinline__ V3<R> pair_grad(const Target<R> &t, const Source<R> &s, V3<R> x, const R *B, R pdt,
                                           Field2<R> &F) {
    const R m1 = R(-1.0), two = R(2.0);
    const R P = m1 * (s.q * B[1] + s.s * B[2] + s.w * B[3]);
    const R Rr = s.q * B[2] + s.s * B[3] + s.w * B[4];
    const R Sb = s.q * B[3] + s.s * B[4] + s.w * B[5];
    const R c2 = two * B[2], c3 = two * B[3], c4 = two * B[4];
    const R nB2 = m1 * B[2], nc3 = m1 * c3;
    F.U = nB2 * s.mu + nc3 * s.v;
    F.d1 = P * x + B[1] * s.mu + c2 * s.v;
    F.P = P;
    F.Rr = Rr;
    F.d2 = plus(second(x, P, Rr * x + F.U, F.U), c2, s.th);
    const V3<R> W = B[3] * s.mu + c4 * s.v;
    const V3<R> pu = symv(t.th, F.U), tp = symv(s.th, t.p);
    const R c = two * dot(t.p, W) + nc3 * pdt + m1 * t.w * Sb;
    const R rr2 = two * Rr, nc32 = two * nc3;
    return t.q * F.d1 + symv(F.d2, t.mu) + rr2 * t.p + two * pu + c * x + t.w * W + nc32 * tp;
}

}  // namespace sibfa
