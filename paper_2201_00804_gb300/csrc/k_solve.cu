// The polarization solve in one cooperative kernel: initial guess, products
// T u, conjugate-gradient updates and the convergence test, with the vectors
// in shared memory from the first product to the last.
//
// What bounds it: latency.  A product over a few hundred to a few thousand
// waters is a chain of short dependent steps (spread, three transforms,
// convolution, three transforms, gather, two sums), and as separate launches
// each link cost 4 to 15 us whatever its size: 50 us an iteration at 216
// waters, 50 us at 971.  Here the links are phases of one kernel separated
// by a counter in L2 (about 1 us), five per iteration:
//   spread | z and y transforms of whole x-planes | x transforms, convolution
//   and back | y and z transforms back | gather
// The upper half of every block's threads streams the real-space pair list
// meanwhile.  Each block owns a run of molecules: their dipoles, residuals,
// directions, spline weights and intramolecular kernels stay in its shared
// memory, and only the product's vector goes through global memory.
//
// The recurrence is the one-reduction form of conjugate gradients (Chronopoulos
// and Gear 1989): with u = alpha r, w = T u,
//   beta = rz / rz_old, a = rz / (u.w - beta rz / a_old),
//   p = u + beta p, s = w + beta s, mu += a p, r -= a s,
// the same iterates as the usual form; rz and the residual norm travel with
// the barrier after the spread and u.w with the one after the gather.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "pcg_loop.cuh"

namespace sibfa {

namespace {

constexpr int LT = 512;          // threads per block
constexpr int LREC = 256;        // of them on the reciprocal chain (periodic)
constexpr int PGL = 8;           // lanes per atom in the gather

template <typename R> struct Cplx;
template <> struct Cplx<float> { using T = float2; };
template <> struct Cplx<double> { using T = double2; };

template <typename C> __device__ inline C cadd(C a, C b) { return {a.x + b.x, a.y + b.y}; }
template <typename C> __device__ inline C csub(C a, C b) { return {a.x - b.x, a.y - b.y}; }
template <typename C> __device__ inline C cmul(C a, C w) { return {a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x}; }
// sign flips by mask (an FP64 multiplication would hold the narrow pipe)
__device__ inline float flip(float x, unsigned m) { return __uint_as_float(__float_as_uint(x) ^ m); }
__device__ inline double flip(double x, unsigned m) {
    return __hiloint2double(__double2hiint(x) ^ (int)m, __double2loint(x));
}
// a times -i (forward, sg = 0) or +i (inverse, sg = the sign bit)
template <typename C> __device__ inline C rot(C a, unsigned sg) { return {flip(a.y, sg), flip(a.x, ~sg & 0x80000000u)}; }

// r-point transforms in registers.  The direction is a run-time sign: one
// copy of the code serves every axis and both directions, so that an
// iteration's instructions stay in the cache (168 KB with inlined copies of
// each; 216 waters took 25.7 us an iteration with those).
template <int r, typename R, typename C>
__device__ inline void dft(C (&a)[r], unsigned sg) {
    if constexpr (r == 2) {
        const C t = csub(a[0], a[1]);
        a[0] = cadd(a[0], a[1]);
        a[1] = t;
    } else if constexpr (r == 3) {
        const R h = R(0.86602540378443864676);
        const C s = cadd(a[1], a[2]), t = csub(a[1], a[2]);
        const C m = {a[0].x - R(0.5) * s.x, a[0].y - R(0.5) * s.y};
        const C n = rot(C{h * t.x, h * t.y}, sg);
        a[0] = cadd(a[0], s);
        a[1] = cadd(m, n);
        a[2] = csub(m, n);
    } else if constexpr (r == 4) {
        const C s0 = cadd(a[0], a[2]), s1 = csub(a[0], a[2]), s2 = cadd(a[1], a[3]), s3 = rot(csub(a[1], a[3]), sg);
        a[0] = cadd(s0, s2);
        a[2] = csub(s0, s2);
        a[1] = cadd(s1, s3);
        a[3] = csub(s1, s3);
    } else if constexpr (r == 5) {
        const R c1 = R(0.30901699437494742410), c2 = R(-0.80901699437494742410);
        const R s1 = R(0.95105651629515357212), s2 = R(0.58778525229247312917);
        const C p1 = cadd(a[1], a[4]), m1 = csub(a[1], a[4]), p2 = cadd(a[2], a[3]), m2 = csub(a[2], a[3]);
        const C b1 = {a[0].x + c1 * p1.x + c2 * p2.x, a[0].y + c1 * p1.y + c2 * p2.y};
        const C b2 = {a[0].x + c2 * p1.x + c1 * p2.x, a[0].y + c2 * p1.y + c1 * p2.y};
        const C d1 = rot(C{s1 * m1.x + s2 * m2.x, s1 * m1.y + s2 * m2.y}, sg);
        const C d2 = rot(C{s2 * m1.x - s1 * m2.x, s2 * m1.y - s1 * m2.y}, sg);
        a[0] = cadd(a[0], cadd(p1, p2));
        a[1] = cadd(b1, d1);
        a[4] = csub(b1, d1);
        a[2] = cadd(b2, d2);
        a[3] = csub(b2, d2);
    } else {
        static_assert(r == 8, "radix");
        const R h = R(0.70710678118654752440);
        C e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
        dft<4, R>(e, sg);
        dft<4, R>(o, sg);
        const C r1 = rot(o[1], sg), r3 = rot(o[3], sg);
        const C t1 = {h * (o[1].x + r1.x), h * (o[1].y + r1.y)};
        const C t2 = rot(o[2], sg);
        const C t3 = {h * (r3.x - o[3].x), h * (r3.y - o[3].y)};
        a[0] = cadd(e[0], o[0]);
        a[4] = csub(e[0], o[0]);
        a[1] = cadd(e[1], t1);
        a[5] = csub(e[1], t1);
        a[2] = cadd(e[2], t2);
        a[6] = csub(e[2], t2);
        a[3] = cadd(e[3], t3);
        a[7] = csub(e[3], t3);
    }
}

// t / d from the reciprocal m = floor(2^32 / d) + 1: exact for t d < 2^32, d >= 2
__host__ inline unsigned recip(unsigned d) { return 0xffffffffu / d + 1u; }
__device__ inline int quo(int t, unsigned m) { return (int)__umulhi((unsigned)t, m); }

// One radix-r pass (self-sorting, decimation in frequency) over `lines`
// transforms held as [index][line] with `ld` elements per index.
template <int NT, int r, typename R, typename C>
__device__ inline void fft_pass(const C *in, C *out, const FftPass P, int lines, int ld, unsigned div_lines,
                                const C *tw, unsigned sg, int tid) {
    const int sp = P.sp, m = P.m, tasks = lines * sp * m;
#pragma unroll 1
    for (int t = tid; t < tasks; t += NT) {
        const int i = quo(t, div_lines), l = t - i * lines;
        const int q0 = sp > 1 ? quo(i, P.div_sp) : i, q = i - q0 * sp;
        const C *v = in + i * ld + l;   // q + sp q0 = i
        C a[r];
#pragma unroll
        for (int j = 0; j < r; ++j) a[j] = v[j * sp * m * ld];
        dft<r, R>(a, sg);
        C *o = out + (q + sp * r * q0) * ld + l;
        o[0] = a[0];
        if (m == 1) {   // last pass: no twiddles
#pragma unroll
            for (int k = 1; k < r; ++k) o[k * sp * ld] = a[k];
        } else {
#pragma unroll
            for (int k = 1; k < r; ++k) {
                C w = tw[q0 * k * sp];
                w.y = flip(w.y, sg);
                o[k * sp * ld] = cmul(a[k], w);
            }
        }
    }
}

// Named barrier of the NT threads that transform
template <int NT>
__device__ inline void part_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

// dynamic shared memory of the kernel
extern __shared__ __align__(16) unsigned char loop_raw[];

// All passes of one axis on the transform buffers at byte offsets ba and bb of
// the block's shared memory (offsets, so that the accesses stay shared-space
// ones); the data starts in ba, and the offset that holds the result is returned.
template <int NT, typename R>
__device__ __noinline__ int fft_lines(int ba, int bb, const FftAxis &A, int lines, int ld, unsigned div_lines, int tw_at,
                                      unsigned sg, int tid) {
    using C = typename Cplx<R>::T;
    const C *tw = reinterpret_cast<const C *>(loop_raw + tw_at) + A.tw;
#pragma unroll 1
    for (int k = 0; k < A.npass; ++k) {
        const FftPass &P = A.pass[k];
        const C *a = reinterpret_cast<const C *>(loop_raw + ba);
        C *b = reinterpret_cast<C *>(loop_raw + bb);
        if (P.r == 8) fft_pass<NT, 8, R>(a, b, P, lines, ld, div_lines, tw, sg, tid);
        else if (P.r == 4) fft_pass<NT, 4, R>(a, b, P, lines, ld, div_lines, tw, sg, tid);
        else if (P.r == 5) fft_pass<NT, 5, R>(a, b, P, lines, ld, div_lines, tw, sg, tid);
        else if (P.r == 3) fft_pass<NT, 3, R>(a, b, P, lines, ld, div_lines, tw, sg, tid);
        else fft_pass<NT, 2, R>(a, b, P, lines, ld, div_lines, tw, sg, tid);
        part_sync<NT>();
        const int t = ba;
        ba = bb;
        bb = t;
    }
    return ba;
}

// Geometry of the grid and its transforms
template <typename R>
struct GridView {
    using C = typename Cplx<R>::T;
    int K0, K1, K2, nz, L, ldz;        // L: packed line pairs of a plane, ldz their leading size
    int b0, b1, tw;                    // byte offsets of the transform buffers and the twiddles
    R *gs, *gp;                        // spread grid, potential grid
    C *spec;
    const R *infl;
};
template <typename R>
__device__ inline GridView<R> grid_view(const KParams &p, const DevState<R> &d, R *gs, R *gp, int buf, int tw, int nbuf) {
    GridView<R> G;
    G.K0 = p.K[0], G.K1 = p.K[1], G.K2 = p.K[2], G.nz = p.K[2] / 2 + 1;
    G.L = (G.K1 + 1) / 2, G.ldz = G.L | 1;
    G.b0 = buf;
    G.b1 = buf + nbuf * (int)sizeof(typename Cplx<R>::T);
    G.tw = tw;
    G.gs = gs;
    G.gp = gp;
    G.spec = reinterpret_cast<typename Cplx<R>::T *>(d.cgrid);
    G.infl = d.inflR;
    return G;
}
constexpr int GL = 4;   // global loads a thread keeps in flight
template <typename C>
__device__ inline C *at(int off) { return reinterpret_cast<C *>(loop_raw + off); }

// n complex values, rows of `row` of them `pitch` apart in global memory, into
// the buffer at b0, GL of a thread's loads in flight (an L2 access takes some
// 0.4 us); columns past `live` are zero.
template <int NT, typename R>
__device__ inline void load_rows(const typename Cplx<R>::T *g, int n, int row, unsigned div_row, size_t pitch, int live,
                                 int b0, int tid) {
    using C = typename Cplx<R>::T;
    C *b = at<C>(b0);
    for (int t0 = tid; t0 < n; t0 += GL * NT) {
        C v[GL];
#pragma unroll
        for (int u = 0; u < GL; ++u) {
            const int t = t0 + u * NT, x = quo(t, div_row), c = t - x * row;
            v[u] = t < n && c < live ? g[x * pitch + c] : C{R(0), R(0)};
        }
#pragma unroll
        for (int u = 0; u < GL; ++u)
            if (t0 + u * NT < n) b[t0 + u * NT] = v[u];
    }
}

// Forward z and y transforms of plane x: two real lines along z go as the
// real and imaginary part of one complex transform.  CLEAR: the plane is
// cleared for the next spread.
template <int NT, bool CLEAR, typename R>
__device__ void plane_forward(const GridView<R> &G, const LoopPlan &lp, const FftAxis *ax, int x, int tid) {
    using C = typename Cplx<R>::T;
    const int n = G.L * G.K2, K2 = G.K2;
    R *g = G.gs + (size_t)x * G.K1 * K2;
    C *w = at<C>(G.b0);
    for (int t0 = tid; t0 < n; t0 += GL * NT) {
        C v[GL];
#pragma unroll
        for (int u = 0; u < GL; ++u) {
            const int t = t0 + u * NT, l = quo(t, lp.div_k2);
            const R *a = g + t + l * K2;   // line 2 l, point z = t - l K2
            v[u].x = t < n ? a[0] : R(0);
            v[u].y = t < n && 2 * l + 1 < G.K1 ? a[K2] : R(0);
        }
#pragma unroll
        for (int u = 0; u < GL; ++u) {
            const int t = t0 + u * NT, l = quo(t, lp.div_k2);
            if (t < n) w[(t - l * K2) * G.ldz + l] = v[u];
        }
    }
    part_sync<NT>();
    if (CLEAR)
        for (int t = tid; t < G.K1 * K2; t += NT) g[t] = R(0);
    const int ra = fft_lines<NT, R>(G.b0, G.b1, ax[2], G.L, G.ldz, lp.div_l, G.tw, 0u, tid);
    const int rb = ra == G.b0 ? G.b1 : G.b0;
    const C *a = at<C>(ra);
    C *b = at<C>(rb);
    for (int t = tid; t < G.L * G.nz; t += NT) {
        const int k = quo(t, lp.div_l), l = t - k * G.L;
        const C u = a[k * G.ldz + l], v = a[(k ? K2 - k : 0) * G.ldz + l];
        b[2 * l * G.nz + k] = {R(0.5) * (u.x + v.x), R(0.5) * (u.y - v.y)};
        if (2 * l + 1 < G.K1) b[(2 * l + 1) * G.nz + k] = {R(0.5) * (u.y + v.y), R(0.5) * (v.x - u.x)};
    }
    part_sync<NT>();
    b = at<C>(fft_lines<NT, R>(rb, ra, ax[1], G.nz, G.nz, lp.div_nz, G.tw, 0u, tid));
    const int m = G.K1 * G.nz;
    C *out = G.spec + (size_t)x * m;
    for (int t = tid; t < m; t += NT) out[t] = b[t];
    part_sync<NT>();
}

// The way back, into the potential grid.
template <int NT, typename R>
__device__ void plane_inverse(const GridView<R> &G, const LoopPlan &lp, const FftAxis *ax, int x, int tid) {
    using C = typename Cplx<R>::T;
    const int m = G.K1 * G.nz, n = G.L * G.K2;
    load_rows<NT, R>(G.spec + (size_t)x * m, m, G.nz, lp.div_nz, G.nz, G.nz, G.b0, tid);
    part_sync<NT>();
    const int ra = fft_lines<NT, R>(G.b0, G.b1, ax[1], G.nz, G.nz, lp.div_nz, G.tw, 0x80000000u, tid);
    const int rb = ra == G.b0 ? G.b1 : G.b0;
    const C *a = at<C>(ra);
    C *b = at<C>(rb);
    for (int t = tid; t < n; t += NT) {
        const int z = quo(t, lp.div_l), l = t - z * G.L;
        const bool up = z < G.nz;
        const int k = up ? z : G.K2 - z;
        C u = a[2 * l * G.nz + k], v = {R(0), R(0)};
        if (2 * l + 1 < G.K1) v = a[(2 * l + 1) * G.nz + k];
        if (k == 0 || 2 * k == G.K2) u.y = v.y = R(0);   // real coefficients of a real line
        if (!up) u.y = -u.y, v.y = -v.y;
        b[z * G.ldz + l] = {u.x - v.y, u.y + v.x};
    }
    part_sync<NT>();
    b = at<C>(fft_lines<NT, R>(rb, ra, ax[2], G.L, G.ldz, lp.div_l, G.tw, 0x80000000u, tid));
    R *g = G.gp + (size_t)x * G.K1 * G.K2;
    for (int t = tid; t < n; t += NT) {
        const int l = quo(t, lp.div_k2);
        const C v = b[(t - l * G.K2) * G.ldz + l];
        R *o = g + t + l * G.K2;
        o[0] = v.x;
        if (2 * l + 1 < G.K1) o[G.K2] = v.y;
    }
    part_sync<NT>();
}

// x transforms of a tile of columns, the convolution, and back.
template <int NT, typename R>
__device__ void columns(const GridView<R> &G, const LoopPlan &lp, const FftAxis *ax, int tile, int tid) {
    using C = typename Cplx<R>::T;
    const int n = G.K1 * G.nz, xt = lp.xt, c0 = tile * xt, live = min(xt, n - c0), all = G.K0 * xt;
    load_rows<NT, R>(G.spec + c0, all, xt, lp.div_xt, n, live, G.b0, tid);
    part_sync<NT>();
    const int ra = fft_lines<NT, R>(G.b0, G.b1, ax[0], xt, xt, lp.div_xt, G.tw, 0u, tid);
    C *a = at<C>(ra);
    for (int t = tid; t < all; t += NT) {
        const int x = quo(t, lp.div_xt), c = t - x * xt;
        const R f = c < live ? G.infl[(size_t)x * n + c0 + c] : R(0);
        a[t].x *= f;
        a[t].y *= f;
    }
    part_sync<NT>();
    a = at<C>(fft_lines<NT, R>(ra, ra == G.b0 ? G.b1 : G.b0, ax[0], xt, xt, lp.div_xt, G.tw, 0x80000000u, tid));
    for (int t = tid; t < all; t += NT) {
        const int x = quo(t, lp.div_xt), c = t - x * xt;
        if (c < live) G.spec[(size_t)x * n + c0 + c] = a[t];
    }
    part_sync<NT>();
}

// Weights of an atom: x and y axis value (5) and derivative (5) at the grid
// lines base - j; z axis 8 values and 8 derivatives at increasing z from the
// 4-aligned line at or below base - 4, zero outside the five lines, so that a
// row is two aligned 4-wide accesses.
constexpr int AW = 36, AZ = 20;

// c0 w + c1 w' at the five points of a row.  FP32 rows whose length is a
// multiple of 4 take two 4-wide reductions when the points do not wrap.
template <typename R>
__device__ inline void add_row(R *row, int K2, int zb, const R *w, R c0, R c1) {
    const int zlo = zb - (ORDER - 1);
    if constexpr (sizeof(R) == 4) {
        if ((K2 & 3) == 0 && zlo >= 0) {
            float4 *g4 = reinterpret_cast<float4 *>(row + (zlo & ~3));
            const float4 *p = reinterpret_cast<const float4 *>(w);
            const float4 a0 = p[0], a1 = p[1], b0 = p[2], b1 = p[3];
            atomicAdd(g4, make_float4(c0 * a0.x + c1 * b0.x, c0 * a0.y + c1 * b0.y, c0 * a0.z + c1 * b0.z,
                                      c0 * a0.w + c1 * b0.w));
            atomicAdd(g4 + 1, make_float4(c0 * a1.x + c1 * b1.x, c0 * a1.y + c1 * b1.y, c0 * a1.z + c1 * b1.z,
                                          c0 * a1.w + c1 * b1.w));
            return;
        }
    }
    const int r = zlo & 3;
#pragma unroll
    for (int k = 0; k < ORDER; ++k) {
        const int z = zlo + k;
        atomicAdd(row + (z < 0 ? z + K2 : z), c0 * w[r + k] + c1 * w[8 + r + k]);
    }
}
// sums of a row's values with the weights and with their derivatives
template <typename R>
__device__ inline void take_row(const R *row, int K2, int zb, const R *w, R &t0, R &t1) {
    const int zlo = zb - (ORDER - 1);
    t0 = t1 = R(0);
    if constexpr (sizeof(R) == 4) {
        if ((K2 & 3) == 0 && zlo >= 0) {
            const float4 *g4 = reinterpret_cast<const float4 *>(row + (zlo & ~3));
            const float4 *p = reinterpret_cast<const float4 *>(w);
            const float4 u = g4[0], v = g4[1];   // inside the row: zlo + 4 <= K2 - 1, K2 a multiple of 4
            const float4 a0 = p[0], a1 = p[1], b0 = p[2], b1 = p[3];
            t0 = u.x * a0.x + u.y * a0.y + u.z * a0.z + u.w * a0.w + v.x * a1.x + v.y * a1.y + v.z * a1.z + v.w * a1.w;
            t1 = u.x * b0.x + u.y * b0.y + u.z * b0.z + u.w * b0.w + v.x * b1.x + v.y * b1.y + v.z * b1.z + v.w * b1.w;
            return;
        }
    }
    const int r = zlo & 3;
#pragma unroll
    for (int k = 0; k < ORDER; ++k) {
        const int z = zlo + k;
        const R g = row[z < 0 ? z + K2 : z];
        t0 += g * w[r + k];
        t1 += g * w[8 + r + k];
    }
}

// Arrival at and wait for the grid-wide counter, one thread per block.  A
// wait that runs out raises the shared give-up flag, and every block then
// leaves at its next barrier.
__device__ __noinline__ bool counter_wait(unsigned *bar, unsigned target, unsigned polls) {
    __threadfence();
    atomicAdd(bar, 1u);
    unsigned v;
    for (unsigned k = 0; k < polls; ++k) {
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if (v >= target) return true;
        if ((k & 1023u) == 1023u && *(volatile unsigned *)(bar + 1)) return false;
    }
    atomicExch(bar + 1, 1u);
    return false;
}

// sum of the values one per thread in sh[0..n), n a multiple of 32, by one warp
__device__ inline double warp_sum_shared(const double *sh, int n, int lane) {
    double v = 0;
    for (int k = lane; k < n; k += 32) v += sh[k];
    return warp_sum(v);
}
// sum of n block partials in a fixed order, by one warp (every block gets the same bits)
__device__ inline double warp_sum_parts(const double *part, int n, int lane) {
    double v = 0;
    for (int k = lane; k < n; k += 32) v += __ldcg(part + k);
    return warp_sum(v);
}

// Entries of the pair list: partner (sign of g2 in the top bit), sqrt|g2| x, g1
template <typename R>
struct VecR {   // the product's vector, 4 values per atom
    const R *v;
    __device__ inline V3<R> at(int atom) const {
        if constexpr (sizeof(R) == 4) {
            const float4 m = *reinterpret_cast<const float4 *>(v + (size_t)atom * 4);
            return mk(m.x, m.y, m.z);
        } else {
            const double2 m = *reinterpret_cast<const double2 *>(v + (size_t)atom * 4);
            return mk(m.x, m.y, v[(size_t)atom * 4 + 2]);
        }
    }
};
template <typename R>
__device__ inline void entry(int j, V3<R> y, R g1, V3<R> mu, V3<R> &ef) {
    R my = dot(mu, y);
    if (j < 0) my = -my;
    ef = ef + my * y + g1 * mu;
}
template <typename R>
__device__ inline void row_out(V3<R> ef, int lane, double *out) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ef.x += __shfl_xor_sync(0xffffffffu, ef.x, o);
        ef.y += __shfl_xor_sync(0xffffffffu, ef.y, o);
        ef.z += __shfl_xor_sync(0xffffffffu, ef.z, o);
    }
    if (lane < 3) out[lane] = double(lane == 0 ? ef.x : (lane == 1 ? ef.y : ef.z));
}

// real-space field of one atom's list, one warp, straight from global memory
template <typename R>
__device__ inline void row_field(const DevState<R> &d, VecR<R> vec, int t, int tls, int lane, double *out) {
    const int n = d.tl_n[t];
    const size_t base = (size_t)t * tls;
    V3<R> ef = mk(R(0), R(0), R(0));
    for (int e = lane; e < n; e += 64) {
        const size_t k0 = base + e, k1 = base + (e + 32 < n ? e + 32 : e);
        const int j0 = d.tl_j[k0], j1 = d.tl_j[k1];
        const V3<R> y0 = mk(d.tl_x[k0], d.tl_y[k0], d.tl_z[k0]), y1 = mk(d.tl_x[k1], d.tl_y[k1], d.tl_z[k1]);
        const R g0 = d.tl_g1[k0], g1 = d.tl_g1[k1];
        const V3<R> u0 = vec.at(j0 & 0x7fffffff), u1 = vec.at(j1 & 0x7fffffff);
        entry(j0, y0, g0, u0, ef);
        if (e + 32 < n) entry(j1, y1, g1, u1, ef);
    }
    row_out(ef, lane, out);
}

// The same for a warp's rows (first, first + step, ... < rows of the block's
// atoms), the list brought into shared memory CH entries at a time, RS - 1
// chunks ahead: the list's bytes bound this part, and the copies keep
// 60 KB of them in flight per SM at eight warps, where plain loads of the
// same warps kept 20 KB (4096 waters: 66 us a product with loads).
constexpr int RS = 3;
template <typename R> constexpr int CH = sizeof(R) == 4 ? 128 : 64;
template <typename R> constexpr int STAGE = CH<R> * (4 * (int)sizeof(R) + 4);   // bytes

__device__ inline void copy16(void *s, const void *g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g)
                 : "memory");
}

template <typename R>
__device__ void rows_staged(const DevState<R> &d, VecR<R> vec, int t0, int rows, const int *cnt, int first, int step,
                            int tls, unsigned char *buf, int lane, double *out) {
    constexpr int N = CH<R>;
    int pr = first, pc = 0, ps = 0;   // next chunk to ask for: row, entry, stage
    auto ask = [&]() {
        while (pr < rows && pc >= cnt[pr]) pr += step, pc = 0;
        if (pr < rows) {
            const size_t k = (size_t)(t0 + pr) * tls + pc;
            unsigned char *b = buf + ps * STAGE<R>;
            constexpr int per = 16 / (int)sizeof(R);   // values per copy
            if (lane * 4 < N) copy16(b + lane * 16, d.tl_j + k + lane * 4);
            b += N * 4;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const R *src = c == 0 ? d.tl_x : (c == 1 ? d.tl_y : (c == 2 ? d.tl_z : d.tl_g1));
                copy16(b + c * N * sizeof(R) + lane * 16, src + k + lane * per);
            }
            pc += N;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (++ps == RS) ps = 0;
    };
#pragma unroll
    for (int k = 0; k < RS - 1; ++k) ask();
    int cs = 0;
#pragma unroll 1
    for (int r = first; r < rows; r += step) {
        const int n = cnt[r];
        V3<R> ef = mk(R(0), R(0), R(0));
#pragma unroll 1
        for (int c = 0; c < n; c += N) {
            ask();
            asm volatile("cp.async.wait_group %0;" ::"n"(RS - 1) : "memory");
            __syncwarp();
            const unsigned char *b = buf + cs * STAGE<R>;
            const int *js = reinterpret_cast<const int *>(b);
            const R *xs = reinterpret_cast<const R *>(b + N * 4);
            int j[N / 32];
            V3<R> mu[N / 32];
#pragma unroll
            for (int u = 0; u < N / 32; ++u) {
                j[u] = c + lane + 32 * u < n ? js[lane + 32 * u] : 0;
                mu[u] = vec.at(j[u] & 0x7fffffff);
            }
#pragma unroll
            for (int u = 0; u < N / 32; ++u) {
                const int e = lane + 32 * u;
                if (c + e < n) entry(j[u], mk(xs[e], xs[N + e], xs[2 * N + e]), xs[3 * N + e], mu[u], ef);
            }
            __syncwarp();   // the stage is asked for again
            if (++cs == RS) cs = 0;
        }
        row_out(ef, lane, out + r * 3);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

__device__ inline int wrap(int g, int K) { return g < 0 ? g + K : g; }

// Shared-memory layout of a block that owns mper molecules, in bytes: 5 FP64
// vectors of 9 mper (mu, r, p, s, w), the vector in R and the reciprocal
// field in R, list lengths; periodic: spline weights and grid bases,
// intramolecular kernels (5 per atom pair), twiddles, transform buffers;
// then the list's stages of the upper warps.
struct LoopMem {
    size_t weights, bases, own, tw, buf, stage, total;
};
template <typename R>
__host__ __device__ inline LoopMem loop_mem(int mper, int periodic, int ntw, int nbuf, int staged) {
    auto up = [](size_t n) { return (n + 15) & ~(size_t)15; };
    LoopMem m;
    m.weights = up((size_t)mper * 9 * (5 * sizeof(double) + 2 * sizeof(R)) + (size_t)mper * 3 * sizeof(int));
    m.bases = m.weights + (periodic ? (size_t)mper * 3 * AW * sizeof(R) : 0);
    m.own = up(m.bases + (periodic ? (size_t)mper * 9 * sizeof(int) : 0));
    m.tw = up(m.own + (periodic ? (size_t)mper * 15 * sizeof(R) : 0));
    m.buf = up(m.tw + (size_t)ntw * 2 * sizeof(R));
    m.stage = up(m.buf + (size_t)nbuf * 4 * sizeof(R));
    m.total = m.stage + (staged ? (size_t)RS * STAGE<R> * (periodic ? (LT - LREC) / 32 : LT / 32) : 0);
    return m;
}

template <typename R, bool PER>
__global__ void __launch_bounds__(LT, 2)
    k_pcg_loop(KParams p, DevState<R> d, LoopPlan lp, MuGuess guess, int warm, double *push) {
    using C = typename Cplx<R>::T;
    unsigned char *raw = loop_raw;
    __shared__ double red[2][LT];
    __shared__ double s_val[4];
    __shared__ int s_lost, s_end;
    __shared__ FftAxis s_ax[3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * lp.mper, nm = max(0, min(lp.mper, p.M - m0)), n9 = nm * 9, cap9 = lp.mper * 9;
    const LoopMem mem = loop_mem<R>(lp.mper, PER, lp.ntw, lp.nbuf, lp.staged);
    double *smu = reinterpret_cast<double *>(raw), *sr = smu + cap9, *sp = sr + cap9, *ss = sp + cap9, *sw = ss + cap9;
    R *su = reinterpret_cast<R *>(sw + cap9), *sf = su + cap9;
    int *cnt = reinterpret_cast<int *>(sf + cap9);
    R *wt = reinterpret_cast<R *>(raw + mem.weights), *own = reinterpret_cast<R *>(raw + mem.own);
    int *gb = reinterpret_cast<int *>(raw + mem.bases);
    R *gvec = reinterpret_cast<R *>(lp.vec);
    unsigned *bar = reinterpret_cast<unsigned *>(d.scal + 12);
    const unsigned ncta = gridDim.x;
    unsigned target = 0;
    if (tid == 0) s_lost = s_end = 0;

    // grid-wide barrier of whole blocks, and of the reciprocal threads alone
    auto everyone = [&]() {
        __syncthreads();
        target += ncta;
        if (tid == 0 && !counter_wait(bar, target, lp.polls)) s_lost = 1;
        __syncthreads();
    };
    auto chain = [&]() {
        part_sync<LREC>();
        target += ncta;
        if (tid == 0 && !counter_wait(bar, target, lp.polls)) s_lost = 1;
        part_sync<LREC>();
    };

#pragma unroll 1
    for (int t = tid; t < nm * 3; t += LT) cnt[t] = d.tl_n[m0 * 3 + t];
    GridView<R> G{};
    if constexpr (PER) {
        G = grid_view(p, d, d.grid + (size_t)p.K[0] * p.K[1] * p.K[2], d.grid, (int)mem.buf, (int)mem.tw, lp.nbuf);
        C *tw = reinterpret_cast<C *>(raw + mem.tw);
#pragma unroll 1
        for (int t = tid; t < lp.ntw; t += LT) tw[t] = reinterpret_cast<const C *>(lp.tw)[t];
        if (tid < 3) s_ax[tid] = lp.ax[tid];
        // spline weights and grid bases of the owned atoms
#pragma unroll 1
        for (int t = tid; t < n9; t += LT) {
            const int a = t / 3, c = t - a * 3, m = m0 + a / 3, pt = a % 3;
            R w0[ORDER], w1[ORDER], w2[ORDER], w3[ORDER];
            bspline5<R, 1>(d.sfrac[(m * NP + pt) * 3 + c], w0, w1, w2, w3);
            const R scl = sc<R>(p).kl[c];
            const int b = d.sbase[(m * NP + pt) * 3 + c];
            gb[t] = b;
            R *w = wt + a * AW + c * 10;
            if (c < 2) {
#pragma unroll
                for (int j = 0; j < ORDER; ++j) {
                    w[j] = w0[j];
                    w[5 + j] = w1[j] * scl;
                }
            } else {
                const int r = (b - (ORDER - 1)) & 3;
#pragma unroll
                for (int k = 0; k < 16; ++k) w[k] = R(0);
#pragma unroll
                for (int j = 0; j < ORDER; ++j) {
                    w[r + 4 - j] = w0[j];
                    w[8 + r + 4 - j] = w1[j] * scl;
                }
            }
        }
        // erf kernels of the atom pairs (0,1), (1,2), (2,0) of each molecule
#pragma unroll 1
        for (int t = tid; t < nm * 3; t += LT) {
            const int m = m0 + t / 3, a = t % 3, b = (a + 1) % 3;
            const R *o = d.off + (size_t)m * NP * 3;
            const V3<R> x = mk(o[a * 3] - o[b * 3], o[a * 3 + 1] - o[b * 3 + 1], o[a * 3 + 2] - o[b * 3 + 2]);
            R g[4];
            g_erf_s<R, 3>(dot(x, x), sc<R>(p).alpha, g);
            R *q = own + t * 5;
            q[0] = x.x, q[1] = x.y, q[2] = x.z, q[3] = g[1], q[4] = g[2];
        }
    }
#pragma unroll 1
    for (int e = tid; e < n9; e += LT) {
        const int k = m0 * 9 + e;
        if (PER) d.efield[k] += d.efield_r[k];   // the reciprocal chain's part
        double m;
        if (guess.n > 0) {
            m = 0;
            for (int j = 0; j < guess.n; ++j) m += guess.c[j] * guess.h[j][k];
        } else {
            m = warm ? d.mu[k] : p.a_pol[(e / 3) % 3] * d.efield[k];
        }
        smu[e] = m;
        su[e] = R(m);
        gvec[(m0 * 3 + e / 3) * 4 + e % 3] = R(m);
    }
    __syncthreads();

    const int used = min(LT, (n9 + 31) & ~31);   // threads that hold partial sums
    double *partg = lp.part, *partn = lp.part + ncta, *partd = lp.part + 2 * ncta;
    double gam = 0, gam_old = 1, a_old = 1;
    const double tol = d.scal[SC_TOL] / 4.80321, tol2 = tol * tol * (p.M * 3);   // bound of the sum of squares
    int it = 0;
    bool first = true;
    for (;;) {
        // the product's vector is in su and gvec
        if constexpr (PER) {
#pragma unroll 1
            for (int t = tid; t < nm * 75; t += LT) {   // atom x 25 rows of its stencil
                const int a = t / 25, row = t - a * 25, jx = row / 5, jy = row - jx * 5;
                const R *w = wt + a * AW;
                const R u0 = su[a * 3], u1 = su[a * 3 + 1], u2 = su[a * 3 + 2];
                const R x0 = w[jx], x1 = w[5 + jx], y0 = w[10 + jy], y1 = w[15 + jy];
                const int gx = wrap(gb[a * 3] - jx, G.K0), gy = wrap(gb[a * 3 + 1] - jy, G.K1);
                add_row<R>(G.gs + ((size_t)gx * G.K1 + gy) * G.K2, G.K2, gb[a * 3 + 2], w + AZ,
                           u0 * x1 * y0 + u1 * x0 * y1, u2 * x0 * y0);
            }
        }
        everyone();
        if (s_lost) break;
        if (!first) {
            // one thread takes FP64 scalar work (a warp-wide FP64 instruction
            // holds the pipe for some 18 cycles), and none of it on the way
            // that can be done beside the product
            if (warp < 2) {
                const double v = warp_sum_parts(warp ? partn : partg, ncta, lane);
                if (lane == 0) {
                    s_val[warp] = v;
                    if (warp == 1) s_end = v < tol2 ? 1 : (it >= lp.maxit ? 2 : 0);
                }
            }
            __syncthreads();
            gam = s_val[0];
            if (s_end) break;
            if (tid == LT - 1) {
                const double b = it ? gam / gam_old : 0.0;
                s_val[2] = b;
                s_val[3] = it ? b * gam / a_old : 0.0;
            }
        }
        // T u: real space and, beside it, the reciprocal chain
        if (PER && tid < LREC) {
            for (int x = blockIdx.x; x < G.K0; x += ncta) plane_forward<LREC, true>(G, lp, s_ax, x, tid);
            chain();
            if (!s_lost)
                for (int t = blockIdx.x; t * lp.xt < G.K1 * G.nz; t += ncta) columns<LREC>(G, lp, s_ax, t, tid);
            chain();
            if (!s_lost)
                for (int x = blockIdx.x; x < G.K0; x += ncta) plane_inverse<LREC>(G, lp, s_ax, x, tid);
            chain();
            // gather: lanes 0-4 of an atom's group the x-lines of its stencil,
            // lane 5 the self term, lanes 6 and 7 the other two atoms' erf field
            const int sub = tid % PGL;
            for (int a0 = 0; a0 < nm * 3; a0 += LREC / PGL) {
                const int a = a0 + tid / PGL;
                const bool live = a < nm * 3;
                V3<R> E = mk(R(0), R(0), R(0));
                if (live && sub < ORDER) {
                    const R *w = wt + a * AW;
                    const int gx = wrap(gb[a * 3] - sub, G.K0), by = gb[a * 3 + 1], bz = gb[a * 3 + 2];
                    R v1 = R(0), v2 = R(0), v3 = R(0);
#pragma unroll
                    for (int jy = 0; jy < ORDER; ++jy) {
                        R t0, t1;
                        take_row<R>(G.gp + ((size_t)gx * G.K1 + wrap(by - jy, G.K1)) * G.K2, G.K2, bz, w + AZ, t0, t1);
                        v1 += w[10 + jy] * t0;
                        v2 += w[15 + jy] * t0;
                        v3 += w[10 + jy] * t1;
                    }
                    const R ike = sc<R>(p).ike;
                    E = mk(-w[5 + sub] * v1 * ike, -w[sub] * v2 * ike, -w[sub] * v3 * ike);
                } else if (live) {
                    const int b0 = a / 3 * 3, k = a - b0;
                    const R al = sc<R>(p).alpha;
                    if (sub == ORDER) {
                        E = (R(4.0 / 3.0) * al * al * al * R(0.56418958354775628695)) *
                            mk(su[a * 3], su[a * 3 + 1], su[a * 3 + 2]);
                    } else {
                        // pair (k, k + 1) or (k - 1, k) of the molecule; minus the dipole field through the erf kernel
                        const int o = (k + sub - ORDER) % 3, pr = sub - ORDER == 1 ? k : (k + 2) % 3;
                        const R *q = own + (b0 + pr) * 5, *u = su + (b0 + o) * 3;
                        const V3<R> xv = mk(q[0], q[1], q[2]), mu = mk(u[0], u[1], u[2]);
                        E = (-q[4] * dot(mu, xv)) * xv + (-q[3]) * mu;
                    }
                }
#pragma unroll
                for (int o = PGL / 2; o > 0; o >>= 1) {
                    E.x += __shfl_xor_sync(0xffffffffu, E.x, o);
                    E.y += __shfl_xor_sync(0xffffffffu, E.y, o);
                    E.z += __shfl_xor_sync(0xffffffffu, E.z, o);
                }
                if (live && sub < 3) sf[a * 3 + sub] = sub == 0 ? E.x : (sub == 1 ? E.y : E.z);
            }
        } else {
            constexpr int W0 = PER ? LREC / 32 : 0, NW = LT / 32 - W0;
            const VecR<R> vec{gvec};
            if (lp.staged)
                rows_staged(d, vec, m0 * 3, nm * 3, cnt, warp - W0, NW, p.tls,
                            raw + mem.stage + (warp - W0) * RS * STAGE<R>, lane, sw);
            else
                for (int r = warp - W0; r < nm * 3; r += NW) row_field(d, vec, m0 * 3 + r, p.tls, lane, sw + r * 3);
            if (PER) target += 3 * ncta;   // the chain's three barriers
        }
        __syncthreads();
        // w = u / alpha - field, and u.w
        double dl = 0;
#pragma unroll 1
        for (int e = tid; e < n9; e += LT) {
            const int c = (e / 3) % 3;
            const double u = first ? smu[e] : p.a_pol[c] * sr[e];
            const double w = u * p.a_pol_inv[c] - (PER ? sw[e] + double(sf[e]) : sw[e]);
            sw[e] = w;
            dl += u * w;
        }
        if (tid < used) red[0][tid] = dl;
        __syncthreads();
        if (warp == 0) {
            const double v = warp_sum_shared(red[0], used, lane);
            if (lane == 0) partd[blockIdx.x] = v;
        }
        everyone();
        if (s_lost) break;
        double a = 0, beta = 0;
        if (!first) {
            if (warp == 0) {
                const double v = warp_sum_parts(partd, ncta, lane);
                if (lane == 0) s_val[1] = gam / (v - s_val[3]);
            }
            __syncthreads();
            beta = s_val[2];
            a = s_val[1];
            gam_old = gam;
            a_old = a;
            ++it;
        }
        double rz = 0, rr = 0;
#pragma unroll 1
        for (int e = tid; e < n9; e += LT) {
            const int c = (e / 3) % 3;
            const double al = p.a_pol[c];
            double r;
            if (first) {
                r = d.efield[m0 * 9 + e] - sw[e];
                sp[e] = 0;
                ss[e] = 0;
            } else {
                const double q = al * sr[e] + beta * sp[e], s = sw[e] + beta * ss[e];
                sp[e] = q;
                ss[e] = s;
                smu[e] += a * q;
                r = sr[e] - a * s;
            }
            sr[e] = r;
            const double u = al * r;
            su[e] = R(u);
            gvec[(m0 * 3 + e / 3) * 4 + e % 3] = R(u);
            rz += r * u;
            rr += u * u;
        }
        if (tid < used) {
            red[0][tid] = rz;
            red[1][tid] = rr;
        }
        __syncthreads();
        if (warp < 2) {
            const double v = warp_sum_shared(red[warp], used, lane);
            if (lane == 0) (warp ? partn : partg)[blockIdx.x] = v;
        }
        first = false;
    }
#pragma unroll 1
    for (int e = tid; e < n9; e += LT) {
        const int k = m0 * 9 + e;
        d.mu[k] = smu[e];
        if (push) push[k] = smu[e];
    }
    if (blockIdx.x == 0 && tid == 0) {
        const bool done = s_end == 1;
        d.scal[SC_RZ] = gam;
        d.scal[SC_RES] = sqrt(s_val[1] / (p.M * 3)) * 4.80321;
        d.scal[SC_IT] = it;
        d.scal[SC_DONE] = done ? 1.0 : 0.0;
        d.flags[1] = done ? 1 : 0;
        if (!done) atomicOr(d.flags, F_NOCONV);
    }
    if (tid == 0 && s_lost) atomicOr(d.flags, F_TIMEOUT);
}

// ---------------------------------------------------------------------------
// Convolution of ngrid real grids (d.grid) with the influence function in one
// cooperative kernel: the plane and column phases of the solve with all of a
// block's threads.  As library transforms it is seven launches of 4 to 5 us
// each at these sizes (55 us in FP64 at 24^3).
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(LT, 2)
    k_grid_conv(KParams p, DevState<R> d, LoopPlan lp, int ngrid) {
    using C = typename Cplx<R>::T;
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    __shared__ FftAxis s_ax[3];
    const int tid = threadIdx.x;
    C *tw = reinterpret_cast<C *>(loop_raw);
    for (int t = tid; t < lp.ntw; t += LT) tw[t] = reinterpret_cast<const C *>(lp.tw)[t];
    if (tid < 3) s_ax[tid] = lp.ax[tid];
    __syncthreads();
    const size_t ng = (size_t)p.K[0] * p.K[1] * p.K[2];
    GridView<R> G = grid_view(p, d, d.grid, d.grid, (int)((lp.ntw * sizeof(C) + 15) & ~(size_t)15), 0, lp.nbuf);
    const int n = G.K1 * G.nz, tiles = (n + lp.xt - 1) / lp.xt;
    C *spec = G.spec;
    auto pick = [&](int g) {
        G.gs = G.gp = d.grid + g * ng;
        G.spec = spec + (size_t)g * G.K0 * n;
    };
    for (int t = blockIdx.x; t < ngrid * G.K0; t += gridDim.x) {
        pick(t / G.K0);
        plane_forward<LT, false>(G, lp, s_ax, t % G.K0, tid);
    }
    grid.sync();
    for (int t = blockIdx.x; t < ngrid * tiles; t += gridDim.x) {
        pick(t / tiles);
        columns<LT>(G, lp, s_ax, t % tiles, tid);
    }
    grid.sync();
    for (int t = blockIdx.x; t < ngrid * G.K0; t += gridDim.x) {
        pick(t / G.K0);
        plane_inverse<LT>(G, lp, s_ax, t % G.K0, tid);
    }
}

// ---------------------------------------------------------------------------
// Gas phase, FP32 products: one block solves one cluster on its own, with the
// usual conjugate gradients and its own step lengths; it stops when its
// residual is below the tolerance.  The product recomputes the Thole kernels
// from the molecules' displacements in shared memory (about 45 instructions a
// pair) instead of streaming the pair list: on 4096 clusters of 2-32 waters a
// product streamed 260 MB in 81 us, ten of them a solve, and every iteration
// waited for the slowest cluster twice (1430 us a solve).  The vectors stay in
// FP64; their arithmetic is about as long as the products here, on the FP64 pipe
// beside them.
// ---------------------------------------------------------------------------
constexpr int CT = 128;   // threads

// sums of one value per thread, left in out[0..NV): fewer FP64 instructions
// than shuffles in every warp
template <int NV>
__device__ inline void block_totals(const double (&v)[NV], double (*sh)[CT], double *out, int tid) {
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k][tid] = v[k];
    __syncthreads();
    const int w = tid >> 5, l = tid & 31;
    if (w < NV) {
        const double x = warp_sum((sh[w][l] + sh[w][l + 32]) + (sh[w][l + 64] + sh[w][l + 96]));
        if (l == 0) out[w] = x;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(CT, 8)
    k_pcg_cluster(KParams p, DevState<float> d, int maxit, MuGuess guess, int warm, double *push) {
    __shared__ double sh[2][CT];
    __shared__ double s_sum[2], s_val[2];
    __shared__ float s_top;
    const int tid = threadIdx.x;
    const int m0 = d.cl_start[blockIdx.x], n = d.cl_start[blockIdx.x + 1] - m0, n3 = n * 3, n9 = n * 9;
    double *mu = reinterpret_cast<double *>(loop_raw), *r = mu + n9, *pv = r + n9, *ap = pv + n9;
    float4 *u = reinterpret_cast<float4 *>(loop_raw + ((4 * n9 * sizeof(double) + 15) & ~(size_t)15));
    float *off = reinterpret_cast<float *>(u + n3), *ef = off + n9, *D = ef + n9;
    // lanes per row: the largest power of two that fits the block
    int P = 1;
    while (2 * P * n3 <= CT && P < 16) P *= 2;
    const int part = tid & (P - 1);
    // offsets of the atoms, and O_j - O_i of every (i, j != i) in the list's order
    for (int e = tid; e < n9; e += CT) off[e] = d.off[(size_t)(m0 + e / 9) * NP * 3 + e % 9];
    for (int e = tid; e < n * (n - 1) * 3; e += CT) {
        const int i = e / ((n - 1) * 3), k = e - i * (n - 1) * 3;
        D[e] = d.ndo[(size_t)(m0 + i) * MAXN * 3 + k];
    }
    for (int e = tid; e < n9; e += CT) {
        const int k = m0 * 9 + e;
        double m;
        if (guess.n > 0) {
            m = 0;
            for (int j = 0; j < guess.n; ++j) m += guess.c[j] * guess.h[j][k];
        } else {
            m = warm ? d.mu[k] : p.a_pol[(e / 3) % 3] * d.efield[k];
        }
        mu[e] = m;
        reinterpret_cast<float *>(u)[e / 3 * 4 + e % 3] = float(m);
    }
    // field of the dipoles u of the other molecules at every atom
    auto field = [&]() {
        __syncthreads();
        for (int r0 = 0; r0 < n3; r0 += CT / P) {
            const int row = r0 + tid / P;
            float ex = 0.f, ey = 0.f, ez = 0.f;
            if (row < n3) {
                const int i = row / 3, a = row - i * 3;
                const float ox = off[row * 3], oy = off[row * 3 + 1], oz = off[row * 3 + 2];
                const float k0 = p.sf.thole * p.ainv3f[a][0], k1 = p.sf.thole * p.ainv3f[a][1];
                for (int jj = part; jj < n - 1; jj += P) {
                    const int j = jj + (jj >= i);
                    const float *dd = D + (i * (n - 1) + jj) * 3;
                    const float dx = dd[0], dy = dd[1], dz = dd[2];
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        const float *os = off + (j * 3 + b) * 3;
                        const float4 m = u[j * 3 + b];
                        const float x = (ox - os[0]) - dx, y = (oy - os[1]) - dy, z = (oz - os[2]) - dz;
                        const float r2 = x * x + y * y + z * z, ri = rsqrt_(r2), r2i = ri * ri;
                        const float b1 = ri * r2i, t = (b == 0 ? k0 : k1) * r2 * (r2 * ri), e = exp_(-t);
                        const float T1 = b1 - e * b1, b2 = 3.f * b1 * r2i, T2 = b2 - (e + t * e) * b2;
                        const float c = T2 * (m.x * x + m.y * y + m.z * z);
                        ex += c * x - T1 * m.x;
                        ey += c * y - T1 * m.y;
                        ez += c * z - T1 * m.z;
                    }
                }
            }
            for (int o = P >> 1; o > 0; o >>= 1) {
                ex += __shfl_xor_sync(0xffffffffu, ex, o);
                ey += __shfl_xor_sync(0xffffffffu, ey, o);
                ez += __shfl_xor_sync(0xffffffffu, ez, o);
            }
            if (row < n3 && part == 0) ef[row * 3] = ex, ef[row * 3 + 1] = ey, ef[row * 3 + 2] = ez;
        }
        __syncthreads();
    };
    const double tol = d.scal[SC_TOL] / 4.80321, tol2 = tol * tol * n3;   // bound of the sum of squares
    field();
    double v2[2] = {0, 0};
    for (int e = tid; e < n9; e += CT) {
        const int c = (e / 3) % 3;
        const double al = p.a_pol[c], q = d.efield[m0 * 9 + e] - (mu[e] * p.a_pol_inv[c] - double(ef[e])), z = al * q;
        r[e] = q;
        pv[e] = z;
        reinterpret_cast<float *>(u)[e / 3 * 4 + e % 3] = float(z);
        v2[0] += q * z;
        v2[1] += z * z;
    }
    block_totals<2>(v2, sh, s_sum, tid);
    double rz = s_sum[0];
    int it = 0;
    bool done = s_sum[1] < tol2;
    // Thread EST follows the Lanczos matrix of the iteration (diagonal 1/a_k +
    // beta_(k-1)/a_(k-1), beside it sqrt(beta_k)/a_k), whose row sums bound the
    // eigenvalues of 1 - alpha T that the residual has met.
    constexpr int EST = 32;
    float frz = (float)rz, ia = 0.f, below = 0.f, side = 0.f, top = 0.f;
    if (tid == EST) s_top = 1e30f;   // no iteration: nothing known
    while (!done && it < maxit) {
        field();
        double v1[1] = {0};
        for (int e = tid; e < n9; e += CT) {
            const double pe = pv[e], q = pe * p.a_pol_inv[(e / 3) % 3] - double(ef[e]);
            ap[e] = q;
            v1[0] += pe * q;
        }
        block_totals<1>(v1, sh, s_sum, tid);
        if (tid == 0) s_val[0] = rz / s_sum[0];
        if (tid == EST) ia = __fdividef((float)s_sum[0], frz);
        __syncthreads();
        const double a = s_val[0];
        v2[0] = v2[1] = 0;
        for (int e = tid; e < n9; e += CT) {
            mu[e] += a * pv[e];
            const double q = r[e] - a * ap[e], z = p.a_pol[(e / 3) % 3] * q;
            r[e] = q;
            v2[0] += q * z;
            v2[1] += z * z;
        }
        block_totals<2>(v2, sh, s_sum, tid);
        if (tid == 0) s_val[1] = s_sum[0] / rz;
        if (tid == EST) {
            const float f = (float)s_sum[0], b = __fdividef(f, frz), e = b * rsqrtf(fmaxf(b, 1e-30f)) * ia;
            frz = f;
            top = fmaxf(top, ia + below + side + e);
            below = b * ia;
            side = e;
            s_top = top;
        }
        __syncthreads();
        const double beta = s_val[1];
        rz = s_sum[0];
        ++it;
        done = s_sum[1] < tol2;
        for (int e = tid; e < n9; e += CT) {
            const double q = p.a_pol[(e / 3) % 3] * r[e] + beta * pv[e];
            pv[e] = q;
            reinterpret_cast<float *>(u)[e / 3 * 4 + e % 3] = float(q);
        }
    }
    // The last residual is at hand: one more Jacobi step costs no product and
    // leaves the dipoles closer (the batch used to iterate until its slowest
    // cluster was done, which over-converged the others).  It multiplies the
    // residual by alpha T, and so is left out unless the eigenvalues met lie below
    // 2: waters at liquid distances stay below 1.5, but pressed together to O-O
    // distances near 1 A some pass 3, and the step would lead away from the tolerance.
    const bool closer = s_top < 2.f;
    for (int e = tid; e < n9; e += CT) {
        const double m = closer ? mu[e] + p.a_pol[(e / 3) % 3] * r[e] : mu[e];
        d.mu[m0 * 9 + e] = m;
        if (push) push[m0 * 9 + e] = m;
    }
    if (tid == 0) {   // the batch reports its largest iteration count and residual (non-negative doubles order like their bits)
        atomicMax((unsigned long long *)(d.scal + SC_IT), (unsigned long long)__double_as_longlong((double)it));
        atomicMax((unsigned long long *)(d.scal + SC_RES),
                  (unsigned long long)__double_as_longlong(sqrt(s_sum[1] / n3) * 4.80321));
        if (!done) atomicOr(d.flags, F_NOCONV);
    }
}

size_t cluster_smem(int n) {
    return (((size_t)n * 9 * 4 * sizeof(double) + 15) & ~(size_t)15) + (size_t)n * 3 * sizeof(float4) +
           ((size_t)n * 18 + (size_t)n * (n - 1) * 3) * sizeof(float);
}

// Passes of an axis of n points; false when a prime above 5 is left.  FP64
// takes radix 2 for every factor of 2: a pass costs its longest thread's FP64
// instructions times some 73 cycles (a warp-wide one on its quarter of the SM),
// and small radices spread them over more threads.
bool fft_axis(FftAxis &A, int n, int tw, bool fp64) {
    A = FftAxis{};
    A.n = n;
    A.tw = tw;
    int rest = n, two = 0, sp = 1;
    auto take = [&](int r) {
        if (A.npass == FFT_RADICES) return false;
        A.pass[A.npass++] = {r, sp, n / (sp * r), sp > 1 ? recip(sp) : 0u};
        sp *= r;
        return true;
    };
    while (rest % 2 == 0) rest /= 2, ++two;
    while (two > 0) {
        const int b = fp64 ? 1 : (two == 4 ? 2 : (two >= 3 ? 3 : two));   // 16 as 4 x 4
        if (!take(1 << b)) return false;
        two -= b;
    }
    for (int f : {5, 3})
        while (rest % f == 0) {
            rest /= f;
            if (!take(f)) return false;
        }
    return rest == 1;
}

// Transform part of a plan for `blocks` blocks: the axes' passes, buffer size
// and index reciprocals; false for sizes with other primes or above 128.
template <typename R>
bool fft_plan(LoopPlan &L, const int K[3], int blocks) {
    for (int c = 0; c < 3; ++c) {
        if (K[c] > 128 || !fft_axis(L.ax[c], K[c], L.ntw, sizeof(R) == 8)) return false;
        L.ntw += K[c];
    }
    const int nz = K[2] / 2 + 1, n = K[1] * nz, lines = (K[1] + 1) / 2;
    L.xt = std::max(4, (n + blocks - 1) / blocks);
    L.nbuf = std::max(std::max(K[2] * (lines | 1), n), K[0] * L.xt);
    L.div_k2 = recip(K[2]);
    L.div_l = recip(lines);
    L.div_nz = recip(nz);
    L.div_xt = recip(L.xt);
    return true;
}

// whether a block of kernel f with smem bytes of dynamic shared memory fits an SM
bool fits(const void *f, size_t smem) {
    int dev = 0, most = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, f) != cudaSuccess || smem + fa.sharedSizeBytes > (size_t)most) return false;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, LT, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return false;
    }
    return true;
}

}  // namespace

// ncta stays 0 for what the kernel does not take: larger systems (above
// LOOP_MAX_MOL the products are bound by the pair list's bytes and the grid's
// work, which launches of full occupancy stream better) and grid sizes with
// other primes or above 128.
template <typename R>
void loop_plan(LoopPlan &L, int M, int periodic, const int K[3], int tls, int n_sm) {
    L.ncta = 0;
    if (M > LOOP_MAX_MOL || n_sm < 1) return;
    L.mper = (M + n_sm - 1) / n_sm;
    L.nbuf = L.ntw = 0;
    // rows and chunks of the list start on 16-byte boundaries and whole chunks stay inside a row
    L.staged = tls % CH<R> == 0;
    // A box of few waters takes further blocks for the transforms, at least one
    // for every plane: with a block a water only, 30 waters on a 64^3 grid took
    // 1228 us in FP64 (now 894; the separate kernels took 1011) and 268 in the mixed
    // path (now 231).
    int ncta = (M + L.mper - 1) / L.mper;
    if (periodic) ncta = std::max(ncta, std::min(n_sm, K[0]));
    if (periodic && !fft_plan<R>(L, K, ncta)) return;
    L.smem = loop_mem<R>(L.mper, periodic, L.ntw, L.nbuf, L.staged).total;
    const void *f = periodic ? (const void *)k_pcg_loop<R, true> : (const void *)k_pcg_loop<R, false>;
    if (fits(f, L.smem)) L.ncta = ncta;
}

template <typename R>
void conv_plan(LoopPlan &L, const int K[3], int n_sm) {
    L.ncta = 0;
    L.nbuf = L.ntw = 0;
    if (n_sm < 1 || !fft_plan<R>(L, K, n_sm)) return;
    const size_t c = sizeof(typename Cplx<R>::T);
    L.smem = ((L.ntw * c + 15) & ~(size_t)15) + 2 * L.nbuf * c;
    if (fits((const void *)k_grid_conv<R>, L.smem)) L.ncta = n_sm;
}

template <typename R>
cudaError_t launch_grid_conv(const KParams &p, DevState<R> &d, const LoopPlan &lp, int ngrid, Launch L) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)lp.ncta);
    cfg.blockDim = dim3(LT);
    cfg.dynamicSmemBytes = lp.smem;
    cfg.stream = L.s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count(L);
    return cudaLaunchKernelEx(&cfg, k_grid_conv<R>, p, d, lp, ngrid);
}

std::vector<double> loop_twiddles(const int K[3]) {
    std::vector<double> t;
    for (int c = 0; c < 3; ++c)
        for (int k = 0; k < K[c]; ++k) {
            t.push_back(std::cos(2.0 * M_PI * k / K[c]));
            t.push_back(-std::sin(2.0 * M_PI * k / K[c]));
        }
    return t;
}

template <typename R>
cudaError_t launch_pcg_loop(const KParams &p, DevState<R> &d, const LoopPlan &lp, const MuGuess &g, int warm,
                            double *push, Launch L) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)lp.ncta);
    cfg.blockDim = dim3(LT);
    cfg.dynamicSmemBytes = lp.smem;
    cfg.stream = L.s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // the blocks wait on one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count(L);
    return p.periodic ? cudaLaunchKernelEx(&cfg, k_pcg_loop<R, true>, p, d, lp, g, warm, push)
                      : cudaLaunchKernelEx(&cfg, k_pcg_loop<R, false>, p, d, lp, g, warm, push);
}

// The limit belongs to the process: always the largest cluster's, so that no
// context lowers it between another thread's setting and its launch.
cudaError_t cluster_init() {
    return cudaFuncSetAttribute(k_pcg_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cluster_smem(CLUSTER_MAX));
}

cudaError_t launch_pcg_cluster(const KParams &p, DevState<float> &d, int nmax, int maxit, const MuGuess &g, int warm,
                               double *push, Launch L) {
    k_pcg_cluster<<<p.n_cl, CT, cluster_smem(nmax), L.s>>>(p, d, maxit, g, warm, push);
    count(L);
    return cudaGetLastError();
}

#define INST(R)                                                                                              \
    template void loop_plan<R>(LoopPlan &, int, int, const int *, int, int);                                 \
    template void conv_plan<R>(LoopPlan &, const int *, int);                                                \
    template cudaError_t launch_grid_conv<R>(const KParams &, DevState<R> &, const LoopPlan &, int, Launch); \
                                    \
    template cudaError_t launch_pcg_loop<R>(const KParams &, DevState<R> &, const LoopPlan &, const MuGuess &, int, \
                                            double *, Launch);
INST(float)
INST(double)

}  // namespace sibfa
