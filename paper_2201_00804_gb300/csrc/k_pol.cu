// Polarization solve (Technical Appendix: T mu = E, Jacobi-preconditioned
// conjugate gradient with FP64 vectors and dot products), intramolecular
// Ewald corrections, the chain rule from point gradients and multipole
// sensitivities to atom forces, energy totals and the velocity-Verlet kick.
#include <cooperative_groups.h>

#include <algorithm>

#include "sibfa_internal.cuh"
#include "pcg_guess.cuh"

namespace sibfa {

// scal[] layout
enum { S_RZ = 0, S_PAP = 1, S_ALPHA = 2, S_BETA = 3, S_RES = 4, S_RZN = 5, S_IT = 6, S_DONE = 7, S_TOL = 8 };
constexpr int PB = 256;   // threads per block of the vector kernels

__device__ inline double block_sum(double v, double *sh) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double r = 0;
    if (w == 0) {
        r = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
        r = warp_sum(r);
    }
    return r;   // valid in thread 0
}

// Two block partials reduced by the last block to finish, in fixed order.
// Returns true in thread 0 of the last block, with the two totals.
// *is_last (optional) tells every thread of the block whether it is the last one.
__device__ inline bool last_block_sum2(double a, double b, double *partial, unsigned *counter, double &ta,
                                       double &tb, bool *is_last = nullptr) {
    __shared__ double sh[32];
    __shared__ bool s_last;
    a = block_sum(a, sh);
    b = block_sum(b, sh);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
        __threadfence();
        unsigned k = atomicAdd(counter, 1u);
        s_last = (k == gridDim.x - 1);
    }
    __syncthreads();
    if (is_last) *is_last = s_last;
    if (!s_last) return false;
    __threadfence();
    double x = 0, y = 0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        x += __ldcg(&partial[2 * i]);
        y += __ldcg(&partial[2 * i + 1]);
    }
    x = block_sum(x, sh);
    y = block_sum(y, sh);
    if (threadIdx.x == 0) {
        ta = x;
        tb = y;
        *counter = 0;
        return true;
    }
    return false;
}

__device__ inline double apol(const KParams &p, int k) { return p.a_pol[(k / 3) % 3]; }
__device__ inline double apol_inv(const KParams &p, int k) { return p.a_pol_inv[(k / 3) % 3]; }

// Zero the real SPME grid (input of the next spread of the PCG product).
template <typename R>
__device__ inline void zero_grid(const KParams &p, const DevState<R> &d, size_t tid, size_t nth) {
    if (!p.periodic) return;
    const size_t ng = (size_t)p.K[0] * p.K[1] * p.K[2];
    for (size_t k = tid; k < ng; k += nth) d.grid[k] = R(0);
}

template <typename R>
__global__ void k_pcg_init(KParams p, DevState<R> d, int warm, MuGuess g) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    zero_grid(p, d, k, (size_t)gridDim.x * blockDim.x);
    if (p.n_cl > 1 && k < p.n_cl) d.cl_rr[k] = 0.0;
    if (k >= p.M * 9) return;
    if (g.n > 0) {
        double m = 0;
        for (int j = 0; j < g.n; ++j) m += g.c[j] * g.h[j][k];
        d.mu[k] = m;
    } else if (!warm) {
        d.mu[k] = apol(p, k) * d.efield[k];
    }
    d.vecR[k] = R(d.mu[k]);
    d.efp[k] = 0.0;
    d.efp_r[k] = 0.0;
}

// r = E - T mu0, z = alpha r, p = z
template <typename R>
__global__ void k_pcg_first(KParams p, DevState<R> d) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    zero_grid(p, d, k, (size_t)gridDim.x * blockDim.x);
    double rz = 0, rr = 0;
    if (k < p.M * 9) {
        const double a = apol(p, k);
        const double r = d.efield[k] - (d.mu[k] * apol_inv(p, k) - (d.efp[k] + d.efp_r[k]));
        d.res[k] = r;
        d.zv[k] = a * r;
        d.pv[k] = a * r;
        d.vecR[k] = R(a * r);
        d.efp[k] = 0.0;
        d.efp_r[k] = 0.0;
        rz = r * a * r;
        rr = a * r * a * r;
    }
    if (p.n_cl > 1) cluster_rr_add(d, k, k < p.M * 9, rr);
    double trz, trr;
    bool last = false;
    const bool lead = last_block_sum2(rz, rr, d.partial, d.counter, trz, trr, &last);
    double cres = 0;
    if (last && p.n_cl > 1) cres = cluster_res_max(p, d);   // the whole last block
    if (lead) {
        d.scal[S_RZ] = trz;
        const double res = p.n_cl > 1 ? cres : sqrt(trr / (p.M * 3)) * 4.80321;
        d.scal[S_RES] = res;
        d.scal[S_IT] = 0;
        d.scal[S_DONE] = (res < d.scal[S_TOL]) ? 1.0 : 0.0;
        d.flags[1] = res < d.scal[S_TOL];
    }
}

// Cluster batches: the largest per-cluster RMS preconditioned residual (D)
// from the per-cluster sums of squares.  Block-wide (all threads call it);
// every block gets the same value (a maximum does not depend on order).
template <typename R>
__device__ inline double cluster_res_max(const KParams &p, const DevState<R> &d) {
    __shared__ double smx[32];
    double mx = 0;
    for (int c = threadIdx.x; c < p.n_cl; c += blockDim.x) {
        const int n = d.cl_start[c + 1] - d.cl_start[c];
        mx = fmax(mx, __ldcg(d.cl_rr + c) / (3.0 * n));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) smx[threadIdx.x >> 5] = mx;
    __syncthreads();
    double r = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = fmax(r, smx[w]);
    __syncthreads();
    return sqrt(r) * 4.80321;
}

// Cluster batches: add v (element k of the PCG vectors, valid or not) to the
// sum of squares of its cluster.  Warp-collective: a warp whose elements lie
// in one cluster adds its total with one atomic.
template <typename R>
__device__ inline void cluster_rr_add(const DevState<R> &d, int k, bool valid, double v) {
    const int c = valid ? d.cl_of[k / 9] : -1;
    const int c0 = __shfl_sync(0xffffffffu, c, 0);
    if (__all_sync(0xffffffffu, c == c0 || c < 0)) {
        const double s = warp_sum(valid ? v : 0.0);
        if ((threadIdx.x & 31) == 0 && c0 >= 0) atomicAdd(d.cl_rr + c0, s);
    } else if (valid) {
        atomicAdd(d.cl_rr + c, v);
    }
}

// Block sums of two values at once (valid in thread 0): the two FP64 add
// chains interleave, and the second stage runs over the 8 warp totals only.
__device__ inline void block_sum2(double a, double b, double *sh, double &ra, double &rb) {
    static_assert(PB == 256, "8 warps per block");
    a = warp_sum(a);
    b = warp_sum(b);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) {
        sh[w] = a;
        sh[16 + w] = b;
    }
    __syncthreads();
    ra = rb = 0;
    if (w == 0) {
        double x = l < 8 ? sh[l] : 0.0, y = l < 8 ? sh[16 + l] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
        }
        ra = x;
        rb = y;
    }
}

// Sums of nb pairs of block partials (part[2b], part[2b + 1]) in a fixed
// order, both in one pass: every block obtains bit-identical totals.
__device__ inline void sum_partials2(const double *part, int nb, double *sh, double &ta, double &tb) {
    if (threadIdx.x < 32) {
        double a = 0, b = 0;
        for (int k = threadIdx.x; k < nb; k += 32) {
            a += __ldcg(part + 2 * k);
            b += __ldcg(part + 2 * k + 1);
        }
        a = warp_sum(a);
        b = warp_sum(b);
        if (threadIdx.x == 0) {
            sh[0] = a;
            sh[1] = b;
        }
    }
    __syncthreads();
    ta = sh[0];
    tb = sh[1];
    __syncthreads();
}

// Sum of the nb block partials at part[0], part[stride], ... in a fixed
// order (lane l takes l, l+32, ...; then a fixed tree): every block obtains
// the bit-identical total.
__device__ inline double sum_partials(const double *part, int nb, int stride, double *sh) {
    if (threadIdx.x < 32) {
        double v = 0;
        for (int b = threadIdx.x; b < nb; b += 32) v += __ldcg(part + (size_t)b * stride);
        v = warp_sum(v);
        if (threadIdx.x == 0) sh[0] = v;
    }
    __syncthreads();
    const double t = sh[0];
    __syncthreads();
    return t;
}

// One PCG iteration after the product T p (cooperative launch, grid-stride):
//   (a) ap = p / alpha - E(p), alpha_k = rz / p.ap
//   (b) mu += alpha_k p, r -= alpha_k ap, z = alpha r, beta = rz_new / rz,
//       residual check
//   (c) p = z + beta p, working-precision copy of p, clear the field
//       accumulators and the SPME grid for the next product.
// Inside the solver graph (maxit > 0) it also sets the while-node's
// condition: another iteration while not converged and below maxit.
template <typename R>
__global__ void __launch_bounds__(PB) k_pcg_step(KParams p, DevState<R> d, cudaGraphConditionalHandle loop,
                                                 int maxit) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    __shared__ double sh[32];
    if (d.flags[1]) {   // converged before this launch: uniform over the grid
        if (maxit > 0 && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(loop, 0u);
        return;
    }
    const int n = p.M * 9;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const int nb = gridDim.x;
    const double rz_old = d.scal[S_RZ], tol = d.scal[S_TOL];
    double pap = 0;
    unsigned long long *rmax = reinterpret_cast<unsigned long long *>(d.partial + 3 * nb);   // cluster max slot
    if (p.n_cl > 1) {
        for (int c = tid; c < p.n_cl; c += nth) d.cl_rr[c] = 0.0;
        if (tid == 0) *rmax = 0ull;
    }
    for (int k = tid; k < n; k += nth) {
        const double ap = d.pv[k] * apol_inv(p, k) - (d.efp[k] + d.efp_r[k]);
        d.ap[k] = ap;
        pap += d.pv[k] * ap;
    }
    pap = block_sum(pap, sh);
    if (threadIdx.x == 0) d.partial[blockIdx.x] = pap;
    grid.sync();
    const double tpap = sum_partials(d.partial, nb, 1, sh);
    const double al = rz_old / tpap;
    double rz = 0, rr = 0;
    for (int k0 = tid - (threadIdx.x & 31); k0 < n; k0 += nth) {   // warp-uniform trip count
        const int k = k0 + (threadIdx.x & 31);
        double q = 0;
        if (k < n) {
            const double a = apol(p, k);
            d.mu[k] += al * d.pv[k];
            const double r = d.res[k] - al * d.ap[k];
            d.res[k] = r;
            d.zv[k] = a * r;
            rz += r * a * r;
            q = a * r * a * r;
            rr += q;
        }
        if (p.n_cl > 1) cluster_rr_add(d, k, k < n, q);
    }
    double brz, brr;
    block_sum2(rz, rr, sh, brz, brr);
    if (threadIdx.x == 0) {
        d.partial[nb + 2 * blockIdx.x] = brz;
        d.partial[nb + 2 * blockIdx.x + 1] = brr;
    }
    grid.sync();
    double trz, trr;
    sum_partials2(d.partial + nb, nb, sh, trz, trr);
    const double beta = trz / rz_old;
    double res = sqrt(trr / (p.M * 3)) * 4.80321;
    if (p.n_cl > 1) {
        // largest per-cluster mean square: each block a slice, combined by an
        // atomic maximum (non-negative doubles order like their bit patterns)
        double mx = 0;
        for (int c = tid; c < p.n_cl; c += nth)
            mx = fmax(mx, __ldcg(d.cl_rr + c) / (3.0 * (d.cl_start[c + 1] - d.cl_start[c])));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0) atomicMax(rmax, (unsigned long long)__double_as_longlong(mx));
        grid.sync();
        res = sqrt(__longlong_as_double((long long)__ldcg(rmax))) * 4.80321;
    }
    const bool done = res < tol;
    if (tid == 0) {
        d.scal[S_PAP] = tpap;
        d.scal[S_ALPHA] = al;
        d.scal[S_BETA] = beta;
        d.scal[S_RZ] = trz;
        d.scal[S_RES] = res;
        d.scal[S_IT] += 1.0;
        if (done) {
            d.scal[S_DONE] = 1.0;
            d.flags[1] = 1;
        }
        if (maxit > 0) cudaGraphSetConditional(loop, (!done && d.scal[S_IT] < (double)maxit) ? 1u : 0u);
    }
    if (done) return;   // uniform: every block computed the same residual
    for (int k = tid; k < n; k += nth) {
        const double pk = d.zv[k] + beta * d.pv[k];
        d.pv[k] = pk;
        d.vecR[k] = R(pk);
        d.efp[k] = 0.0;
        d.efp_r[k] = 0.0;
    }
    zero_grid(p, d, tid, nth);
}

// The same for one system of at most one element a thread: what a thread owns
// stays in registers from the product to the next direction (z and T p are
// never stored, mu and r are read before the first wait), and the step lengths
// are each one thread's division.  A step is a chain of latencies, two grid
// barriers among them; FP64 quotients and roots in every warp were some 4 us of
// it.  2,028 waters 16.0 -> 13.1 us, 4,096 waters 18.7 -> 13.5.  (With four elements a
// thread, 32,000 waters, 29.1 -> 21.2 alone, but the evaluation stays as long:
// there the other streams' work fills the waits.)
template <typename R>
__global__ void __launch_bounds__(PB, 2) k_pcg_step_regs(KParams p, DevState<R> d, cudaGraphConditionalHandle loop,
                                                         int maxit) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    __shared__ double sh[32];
    __shared__ double s_v[2];
    if (d.flags[1]) {
        if (maxit > 0 && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(loop, 0u);
        return;
    }
    const int n = p.M * 9, k = blockIdx.x * PB + threadIdx.x, nb = gridDim.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double rz_old = d.scal[S_RZ], tol = d.scal[S_TOL];
    double pv = 0, ap = 0, mu = 0, r = 0, pap = 0;
    if (k < n) {
        pv = d.pv[k];
        mu = d.mu[k];
        r = d.res[k];
        ap = pv * apol_inv(p, k) - (d.efp[k] + d.efp_r[k]);
        pap = pv * ap;
    }
    pap = block_sum(pap, sh);
    if (threadIdx.x == 0) d.partial[blockIdx.x] = pap;
    grid.sync();
    if (w == 0) {
        double v = 0;
        for (int b = lane; b < nb; b += 32) v += __ldcg(d.partial + b);
        v = warp_sum(v);
        if (lane == 0) {
            s_v[0] = v;
            s_v[1] = rz_old / v;
        }
    }
    __syncthreads();
    const double tpap = s_v[0], al = s_v[1];
    double rz = 0, rr = 0;
    if (k < n) {
        d.mu[k] = mu + al * pv;
        r -= al * ap;
        d.res[k] = r;
        const double z = apol(p, k) * r;
        rz = r * z;
        rr = z * z;
        r = z;
    }
    double brz, brr;
    block_sum2(rz, rr, sh, brz, brr);
    if (threadIdx.x == 0) {
        d.partial[nb + 2 * blockIdx.x] = brz;
        d.partial[nb + 2 * blockIdx.x + 1] = brr;
    }
    grid.sync();
    __shared__ double s_t[2];
    if (w < 2) {   // warp 0: r.z and the direction's step, warp 1: the residual
        double v = 0;
        for (int b = lane; b < nb; b += 32) v += __ldcg(d.partial + nb + 2 * b + w);
        v = warp_sum(v);
        if (lane == 0) {
            s_t[w] = v;
            s_v[w] = w == 0 ? v / rz_old : sqrt(v / (p.M * 3)) * 4.80321;
        }
    }
    __syncthreads();
    const double beta = s_v[0], res = s_v[1];
    const bool done = res < tol;
    if (k == 0) {
        d.scal[S_PAP] = tpap;
        d.scal[S_ALPHA] = al;
        d.scal[S_BETA] = beta;
        d.scal[S_RZ] = s_t[0];
        d.scal[S_RES] = res;
        d.scal[S_IT] += 1.0;
        if (done) {
            d.scal[S_DONE] = 1.0;
            d.flags[1] = 1;
        }
        if (maxit > 0) cudaGraphSetConditional(loop, (!done && d.scal[S_IT] < (double)maxit) ? 1u : 0u);
    }
    if (done) return;   // uniform: every block computed the same residual
    if (k < n) {
        const double pk = r + beta * pv;
        d.pv[k] = pk;
        d.vecR[k] = R(pk);
        d.efp[k] = 0.0;
        d.efp_r[k] = 0.0;
    }
    zero_grid(p, d, k, (size_t)nb * PB);
}

static inline unsigned nblk(int n) { return (unsigned)((n + PB - 1) / PB); }

// after the solve: record a solve that stopped at the iteration limit
__global__ void k_pcg_check(const double *scal, int *flags) {
    if (scal[S_DONE] == 0.0) atomicOr(flags, F_NOCONV);
}
void launch_pcg_check(const double *scal, int *flags, Launch L) {
    k_pcg_check<<<1, 1, 0, L.s>>>(scal, flags);
    count(L);
}

template <typename R>
void launch_pcg_init(const KParams &p, DevState<R> &d, int warm, Launch L) {
    k_pcg_init<R><<<nblk(p.M * 9), PB, 0, L.s>>>(p, d, warm, MuGuess{});
    count(L);
}
template <typename R>
void launch_pcg_init_guess(const KParams &p, DevState<R> &d, MuGuess g, Launch L) {
    k_pcg_init<R><<<nblk(p.M * 9), PB, 0, L.s>>>(p, d, 1, g);
    count(L);
}
template <typename R>
void launch_pcg_first(const KParams &p, DevState<R> &d, Launch L) {
    k_pcg_first<R><<<nblk(p.M * 9), PB, 0, L.s>>>(p, d);
    count(L);
}
// Cooperative launch of the PCG step: at most two blocks per SM (the grid must
// be co-resident while the short-range kernels occupy part of every SM on
// their own stream) and one per 256 vector entries.
template <typename R>
void launch_pcg_step(const KParams &p, DevState<R> &d, Launch L, cudaGraphConditionalHandle loop, int maxit) {
    decltype(&k_pcg_step<R>) ks[2] = {k_pcg_step<R>, k_pcg_step_regs<R>};
    struct Resident {
        int n_sm = 0, per_sm[2];
    };
    static const Resident res = [&] {   // on first use, whichever thread's it is
        Resident q;
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&q.n_sm, cudaDevAttrMultiProcessorCount, dev);
        for (int v = 0; v < 2; ++v) {
            int b = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, ks[v], PB, 0);
            q.per_sm[v] = std::max(1, std::min(b, 2));
        }
        return q;
    }();
    const int n = p.M * 9, v = p.n_cl == 1 && n <= res.per_sm[1] * res.n_sm * PB;
    const unsigned grid = (unsigned)std::min<long long>(nblk(n), (long long)res.per_sm[v] * res.n_sm);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(PB);
    cfg.stream = L.s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, ks[v], p, d, loop, maxit);
    count(L);
}

// E_pol = -1/2 ke mu . E (value at the solution); working-precision copies
// of mu and of the CT lambdas for the force pass
template <typename R>
__global__ void k_pol_energy(KParams p, DevState<R> d) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= p.M) return;
    double e = 0;
    for (int k = 0; k < 9; ++k) {
        e += d.mu[m * 9 + k] * d.efield[m * 9 + k];
        d.muR[m * 9 + k] = R(d.mu[m * 9 + k]);
    }
    d.lamR[m * 2] = R(d.lam[m * 2]);
    d.lamR[m * 2 + 1] = R(d.lam[m * 2 + 1]);
    if (p.ct_orig)
        for (int a = 0; a < 3; ++a) d.lamaR[m * 3 + a] = R(d.lama[m * 3 + a]);
    d.epart[m * NTERM + T_POL] = -0.5 * p.ke * e;
    // real-space multipole and penetration energies of the five target sites
    double el = 0, pe = 0;
    for (int w = 0; w < NS; ++w) el += d.epw[(m * NS + w) * 2], pe += d.epw[(m * NS + w) * 2 + 1];
    d.epart[m * NTERM + T_ELEC] += el;
    d.epart[m * NTERM + T_PEN] += pe;
    if (p.vir && !p.periodic)   // and in the gas phase the virials of the sites' two sides
        for (int k = 0; k < 9; ++k) {
            double v = 0;
            for (int s = 0; s < 2 * NS; ++s) v += d.vir_w[((size_t)m * 2 * NS + s) * 9 + k];
            d.vir[m * 9 + k] += v;
        }
}
template <typename R>
void launch_pol_energy(const KParams &p, DevState<R> &d, Launch L) {
    k_pol_energy<R><<<(p.M + 127) / 128, 128, 0, L.s>>>(p, d);
    count(L);
}

// ---------------------------------------------------------------------------
// Chain rule to atom forces.  Frame construction: z along zv, x in the
// (z, xv) plane, y = z x x; its vector-Jacobian product maps gradients of the
// axes back to zv and xv.
// ---------------------------------------------------------------------------
template <typename W>
__device__ inline void frame_vjp(V3<W> zv, V3<W> xv, V3<W> gx, V3<W> gy, V3<W> gz, V3<W> &gzv, V3<W> &gxv) {
    const W iz = rsqrt_<W>(dot(zv, zv));
    const V3<W> ez = iz * zv;
    const V3<W> xp = xv - dot(xv, ez) * ez;
    const W ix = rsqrt_<W>(dot(xp, xp));
    const V3<W> ex = ix * xp;
    // y = z x x
    gz = gz + cross(ex, gy);
    gx = gx + cross(gy, ez);
    // x = xp / |xp|
    const V3<W> gxp = ix * (gx - dot(gx, ex) * ex);
    // xp = xv - (xv.z) z
    gxv = gxp - dot(gxp, ez) * ez;
    gz = gz - dot(xv, ez) * gxp - dot(gxp, ez) * xv;
    // z = zv / |zv|
    gzv = iz * (gz - dot(gz, ez) * ez);
}

// Eight molecules a block.  All threads first sum the accumulators of the
// streams in FP64 and bring them and the frames' inputs to shared memory in
// the working precision, coalesced (the sums read by four diverging lanes a
// molecule, as one dependent load after another, took 78 us at 32,000 waters and 21
// at 8); then four lanes of the first warp take each molecule.
// Lane f < 3 carries the multipole sensitivities
// of the sites in frame f (frame 0: O and the lone pairs; frame 1: H1, M1;
// frame 2: H2, M2) back through that frame's construction; lane 3 takes the
// point gradients (lone-pair charge-transfer term, V_int chain rule,
// midpoints, lone-pair carrier).  The four partial atom gradients are summed
// with shuffles.  The chain rule runs in the working precision R, on the same
// frames as the site kernel.
constexpr int FM = 8;   // molecules per block
template <typename R>
struct FinIn {
    R G[FM][NP][3], mu[FM][NS][3], th[FM][NS][6], dv[FM][2][3];   // gradients, sensitivities, d V_lp
    R ml[FM][NS * NMP], off[FM][NP][3], q[FM][NS], lam[FM][2], kap[FM][3];   // kap: times ke
};
// A thread's elements of one array of PER values a molecule (stride apart)
template <int PER, typename T = double>
struct FinLoad {
    static constexpr int N = (FM * PER + 127) / 128;
    T v[N];
    __device__ __forceinline__ FinLoad(const T *a, int m0, int nm, int stride = 1) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int e = k * 128 + threadIdx.x;
            v[k] = e < nm * PER ? a[((size_t)m0 * PER + e) * stride] : T(0);
        }
    }
    __device__ __forceinline__ void add(const FinLoad &o) {
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] += o.v[k];
    }
    __device__ __forceinline__ void scale(T f) {
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] *= f;
    }
    template <typename R> __device__ __forceinline__ void put(R *out, int nm) const {
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k * 128 + (int)threadIdx.x < nm * PER) out[k * 128 + threadIdx.x] = R(v[k]);
    }
};
template <typename R>
__global__ void __launch_bounds__(128) k_finalize(KParams p, DevState<R> d, double *forces) {
    __shared__ FinIn<R> S;
    const int m0 = blockIdx.x * FM, nm = min(FM, p.M - m0);
    // every load first, so that they are all in flight together
    FinLoad<NP * 3> g(d.gpt, m0, nm), gr(d.gpt_r, m0, nm), gs(d.gpt_s, m0, nm);
    FinLoad<NS * 3> u(d.gmu, m0, nm), ur(d.gmu_r, m0, nm);
    FinLoad<NS * 6> h(d.gth, m0, nm), hr(d.gth_r, m0, nm);
    FinLoad<6> dv(d.dvlp, m0, nm), dvr(d.dvlp_r, m0, nm);
    FinLoad<NS * NMP> ml(d.mp_local, m0, nm);
    FinLoad<2> lam(d.lam, m0, nm);
    FinLoad<3> kap(d.kap, m0, nm);
    FinLoad<NP * 3, R> off(d.off, m0, nm);
    FinLoad<NS, R> q(d.gmp, m0, nm, GMP);
    g.add(gr);
    g.add(gs);
    u.add(ur);
    h.add(hr);
    dv.add(dvr);
    kap.scale(p.ke);   // rounded once
    g.put(&S.G[0][0][0], nm);
    u.put(&S.mu[0][0][0], nm);
    h.put(&S.th[0][0][0], nm);
    dv.put(&S.dv[0][0][0], nm);
    ml.put(&S.ml[0][0], nm);
    lam.put(&S.lam[0][0], nm);
    kap.put(&S.kap[0][0], nm);
    off.put(&S.off[0][0][0], nm);
    q.put(&S.q[0][0], nm);
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x >> 2, t = threadIdx.x & 3, m = m0 + l;
    const bool live = l < nm;
    V3<R> gO = mk(R(0), R(0), R(0)), gH1 = gO, gH2 = gO;
    R W[9] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};   // virial (p.vir)
    if (live) {
        V3<R> r1, r2;
        bond_vectors(d.pos + m * 9, r1, r2);
        const R s1 = rsqrt_<R>(dot(r1, r1)), s2 = rsqrt_<R>(dot(r2, r2));
        auto vec = [](const R *a) { return mk(a[0], a[1], a[2]); };
        auto gpt = [&](int k) { return vec(S.G[l][k]); };
        // lone-pair point gradient including the charge-transfer dependence through its potential
        auto glp = [&](int k) { return gpt(5 + k) + S.lam[l][k] * vec(S.dv[l][k]); };
        if (t < 3) {
            const int f = t;
            V3<R> zv, xv, E[3];
            frame_generators(f, r1, r2, s1, s2, zv, xv);
            frame_axes(zv, xv, E[0], E[1], E[2]);
            V3<R> gE[3] = {mk(R(0), R(0), R(0)), mk(R(0), R(0), R(0)), mk(R(0), R(0), R(0))};
            for (int h = 0; h < (f == 0 ? 1 : 2); ++h) {   // the frame's sites: O; H1, M1; H2, M2
                const int s = f + 2 * h;
                const R *ml = S.ml[l] + s * NMP, *g6 = S.th[l][s];
                const V3<R> gmu = vec(S.mu[l][s]);
                const Sym<R> D{g6[0], g6[1], g6[2], g6[3], g6[4], g6[5]};
                const R tl[3][3] = {{ml[4], ml[7], ml[8]}, {ml[7], ml[5], ml[9]}, {ml[8], ml[9], ml[6]}};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const V3<R> acc = tl[k][0] * E[0] + tl[k][1] * E[1] + tl[k][2] * E[2];
                    gE[k] = gE[k] + ml[1 + k] * gmu + R(2) * symv(D, acc);
                }
            }
            if (f == 0)   // lone pairs: X = O + d (-c z_O +/- s y_O)
                for (int k = 0; k < 2; ++k) {
                    const V3<R> G = glp(k);
                    gE[2] = gE[2] + R(-p.d_lp * p.lp_cos) * G;
                    gE[1] = gE[1] + R(k == 0 ? p.d_lp * p.lp_sin : -p.d_lp * p.lp_sin) * G;
                }
            V3<R> gzv, gxv;
            frame_vjp(zv, xv, gE[0], gE[1], gE[2], gzv, gxv);
            if (f == 0) {
                // zv = u1 + u2, u_k = r_k/|r_k|; xv = r1
                const V3<R> u1 = s1 * r1, u2 = s2 * r2;
                const V3<R> gr1 = s1 * (gzv - dot(gzv, u1) * u1) + gxv;
                const V3<R> gr2 = s2 * (gzv - dot(gzv, u2) * u2);
                gH1 = gr1;
                gH2 = gr2;
                gO = -(gr1 + gr2);
            } else if (f == 1) {
                // zv = O - H1, xv = H2 - H1
                gO = gzv;
                gH1 = -(gzv + gxv);
                gH2 = gxv;
            } else {
                // zv = O - H2, xv = H1 - H2
                gO = gzv;
                gH2 = -(gzv + gxv);
                gH1 = gxv;
            }
            if (p.vir) {   // the frame's atoms move affinely: sum_a g_a (x) (x_a - O)
                vir_add(W, gH1, r1, R(1));
                vir_add(W, gH2, r2, R(1));
            }
        } else {
            V3<R> G[NS], X[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                G[k] = gpt(k);
                X[k] = vec(S.off[l][k]);
            }
            // charge-transfer dependence through the intramolecular potentials V_int(O, H1, H2)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const R kk = S.kap[l][a];
                if (kk == R(0)) continue;
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    if (s == a) continue;
                    const V3<R> dd = X[a] - X[s];
                    const R ir = rsqrt_<R>(dot(dd, dd));
                    const R c = kk * S.q[l][s] * ir * ir * ir;
                    G[a] = G[a] - c * dd;
                    G[s] = G[s] + c * dd;
                    if (p.vir) vir_add(W, dd, dd, -c);   // the (a, s) pair's gradient on a is -c dd
                }
            }
            // The pair kernels counted the lone pairs as points moving with
            // the strain; they follow the frame of O instead, which lane 0's
            // chain rule has taken: remove their point share g_lp (x) off_lp.
            if (p.vir)
                for (int k = 0; k < 2; ++k) vir_add(W, glp(k), vec(S.off[l][5 + k]), R(-1));
            // midpoints and the lone pairs' carrier
            gO = G[0] + R(0.5) * (G[3] + G[4]) + glp(0) + glp(1);
            gH1 = G[1] + R(0.5) * G[3];
            gH2 = G[2] + R(0.5) * G[4];
        }
    }
    R v[9] = {gO.x, gO.y, gO.z, gH1.x, gH1.y, gH1.z, gH2.x, gH2.y, gH2.z};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 1, 4);
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 2, 4);
    }
    if (live && t == 0 && forces) {
        double *F = forces + m * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) F[k] = -(double)v[k];
    }
    if (p.vir) {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            W[k] += __shfl_xor_sync(0xffffffffu, W[k], 1, 4);
            W[k] += __shfl_xor_sync(0xffffffffu, W[k], 2, 4);
        }
        if (live && t == 0)
            for (int k = 0; k < 9; ++k) d.vir[m * 9 + k] += (double)W[k];
    }
}

// Virial total: out[3a + b] = -dE/d eps_ab = -(sum over molecules of the
// streams' dE/d eps + the k-space sums of npass convolution passes), summed in
// a fixed order: every block takes a share of both arrays, a thread always the
// same component, and the last block to finish adds the blocks' sums.  (One
// block, with one thread for the k-space sums, was 290 us at 2,028 waters; this is 10.)
constexpr int VT_BLOCKS = 152, VT_ROW = 16;   // partial sums: 9 components, then 7 k-space sums
template <typename R>
__global__ void __launch_bounds__(256) k_virial_total(int M, DevState<R> d, int npass, double *out) {
    __shared__ double sh[2][256];
    __shared__ bool last;
    const int t = threadIdx.x, nb = gridDim.x;
    double v = 0, s = 0;
    if (t < 252)
        for (int e = blockIdx.x * 252 + t; e < M * 9; e += nb * 252) v += d.vir[e] + d.vir_r[e] + d.vir_s[e];
    for (int e = blockIdx.x * 256 + t; e < npass * VK_BLOCKS * 8; e += nb * 256) s += (e & 7) < 7 ? d.virk[e] : 0.0;
    sh[0][t] = v;
    sh[1][t] = s;
    __syncthreads();
    if (t < 9) {
        double a = 0;
        for (int k = t; k < 252; k += 9) a += sh[0][k];
        d.partial[blockIdx.x * VT_ROW + t] = a;
    } else if (t >= 32 && t < 39) {
        double a = 0;
        for (int k = t - 32; k < 256; k += 8) a += sh[1][k];
        d.partial[blockIdx.x * VT_ROW + 9 + t - 32] = a;
    }
    __threadfence();
    __syncthreads();
    if (t == 0) last = atomicAdd(d.counter + 2, 1u) == (unsigned)nb - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double x = 0;
    for (int b = t / VT_ROW; b < nb; b += 256 / VT_ROW) x += __ldcg(d.partial + b * VT_ROW + t % VT_ROW);
    sh[0][t] = x;
    __syncthreads();
    if (t < VT_ROW) {
        double a = 0;
        for (int k = t; k < 256; k += VT_ROW) a += sh[0][k];
        sh[1][t] = a;
    }
    __syncthreads();
    if (t == 0) {
        const double *ks = sh[1] + 9;
        double a[9];
        for (int k = 0; k < 9; ++k) a[k] = sh[1][k];
        // dE/d eps_ab from the k-space sums: -delta_ab sum e + sum e f m_a m_b
        const int ia[6] = {0, 4, 8, 1, 2, 5}, ib[6] = {0, 4, 8, 3, 6, 7};
        for (int k = 0; k < 3; ++k) a[4 * k] -= ks[0];
        for (int k = 0; k < 6; ++k) {
            a[ia[k]] += ks[1 + k];
            if (ib[k] != ia[k]) a[ib[k]] += ks[1 + k];
        }
        for (int k = 0; k < 9; ++k) out[k] = -a[k];
        d.counter[2] = 0;
    }
}

// The partial sums take the solve's array, which is free by now and holds
// 4 ceil(9 M / 256) + 64 values: 16 a block for a block per 128 molecules.
template <typename R>
void launch_virial_total(const KParams &p, DevState<R> &d, double *out, Launch L) {
    const int nb = std::min(VT_BLOCKS, (p.M + 127) / 128);
    k_virial_total<R><<<nb, 256, 0, L.s>>>(p.M, d, p.periodic ? 2 : 0, out);
    count(L);
}

// Join of the reciprocal chain into the permanent field that the
// polarization solve reads (the charge transfer reads both lone-pair
// potential arrays itself).
template <typename R>
__global__ void k_merge_rec(int M, DevState<R> d) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < M * 9) d.efield[k] += d.efield_r[k];
}
template <typename R>
void launch_merge_rec(const KParams &p, DevState<R> &d, Launch L) {
    k_merge_rec<R><<<(p.M * 9 + 255) / 256, 256, 0, L.s>>>(p.M, d);
    count(L);
}

template <typename R>
void launch_finalize(const KParams &p, DevState<R> &d, double *forces_out, Launch L) {
    k_finalize<R><<<(p.M + FM - 1) / FM, 128, 0, L.s>>>(p, d, forces_out);
    count(L);
}

// energy totals: out[k] = sum_m epart[m*NTERM + k], out[NTERM] = total, in a
// fixed order: up to ER_BLOCKS blocks each sum a contiguous slice of molecules
// (threads take independent chains, then a shared-memory tree per term) into
// partials; the last block to finish sums the partials, one warp per term.
constexpr int ER_BLOCKS = 128, ER_THREADS = 256;
__global__ void __launch_bounds__(ER_THREADS) k_energy(int M, const double *epart, const double *epart_r,
                                                      const double *eintra, double *partial, unsigned *counter,
                                                      double *out) {
    __shared__ double sh[ER_THREADS / 32][NTERM];
    __shared__ double tot[NTERM];
    __shared__ bool last;
    const int nb = gridDim.x, per = (M + nb - 1) / nb;
    const int m0 = blockIdx.x * per, m1 = min(M, m0 + per);
    double v[NTERM];
#pragma unroll
    for (int k = 0; k < NTERM; ++k) v[k] = 0.0;
    for (int m = m0 + threadIdx.x; m < m1; m += blockDim.x) {
#pragma unroll
        for (int k = 0; k < NTERM; ++k) v[k] += epart[m * NTERM + k] + epart_r[m * NTERM + k];
        if (eintra) v[T_ELEC] += eintra[m];
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NTERM; ++k) {
        const double x = warp_sum(v[k]);
        if (l == 0) sh[w][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < NTERM) {
        double x = 0.0;
        for (int j = 0; j < ER_THREADS / 32; ++j) x += sh[j][threadIdx.x];
        partial[blockIdx.x * NTERM + threadIdx.x] = x;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == (unsigned)nb - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    static_assert(NTERM <= ER_THREADS / 32, "one warp per term");
    if (w < NTERM) {
        double x = 0.0;
        for (int b = l; b < nb; b += 32) x += __ldcg(partial + b * NTERM + w);
        x = warp_sum(x);
        if (l == 0) {
            out[w] = x;
            tot[w] = x;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double e = 0.0;
        for (int k = 0; k < NTERM; ++k) e += tot[k];
        out[NTERM] = e;
        *counter = 0;
    }
}

void launch_energy_reduce(int M, const double *epart, const double *epart_r, const double *eintra, double *partial,
                          unsigned *counter, double *out, Launch L) {
    const int nb = std::max(1, std::min(ER_BLOCKS, M / ER_THREADS));
    k_energy<<<nb, ER_THREADS, 0, L.s>>>(M, epart, epart_r, eintra, partial, counter, out);
    count(L);
}

// Cluster batches: terms per cluster (one block per cluster, fixed order),
// then their sums over the clusters into out (NTERM terms and the total).
template <typename R>
__global__ void __launch_bounds__(128) k_cluster_energy(KParams p, DevState<R> d) {
    const int c = blockIdx.x * 4 + (threadIdx.x >> 5), l = threadIdx.x & 31;   // one warp a cluster
    if (c >= p.n_cl) return;
    const int m0 = d.cl_start[c], m1 = d.cl_start[c + 1];
    double v[NTERM];
#pragma unroll
    for (int k = 0; k < NTERM; ++k) v[k] = 0.0;
    for (int m = m0 + l; m < m1; m += 32)
#pragma unroll
        for (int k = 0; k < NTERM; ++k) v[k] += d.epart[m * NTERM + k] + d.epart_r[m * NTERM + k];
    double tot = 0;
#pragma unroll
    for (int k = 0; k < NTERM; ++k) {
        v[k] = warp_sum(v[k]);
        tot += v[k];
        if (l == 0) d.cl_energy[c * (NTERM + 1) + k] = v[k];
    }
    if (l == 0) d.cl_energy[c * (NTERM + 1) + NTERM] = tot;
}
// one block per term (and the total)
__global__ void __launch_bounds__(512) k_cluster_total(int n_cl, const double *cl_energy, double *out) {
    __shared__ double sh[32];
    const int k = blockIdx.x;
    double v = 0;
    for (int c = threadIdx.x; c < n_cl; c += blockDim.x) v += cl_energy[c * (NTERM + 1) + k];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) out[k] = v;
}
template <typename R>
void launch_cluster_energy(const KParams &p, DevState<R> &d, double *out, Launch L) {
    k_cluster_energy<R><<<(p.n_cl + 3) / 4, 128, 0, L.s>>>(p, d);
    k_cluster_total<<<NTERM + 1, 512, 0, L.s>>>(p.n_cl, d.cl_energy, out);
    count(L, 2);
}

// velocity-Verlet half kick (and drift): v += dt/2 F/m ; x += dt v
__global__ void k_md_kick(int M, double *pos, double *vel, const double *inv_mass, const double *F, double dt,
                          int drift) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M * 9) return;
    const double conv = 4.184e-4;   // (kcal/mol/A)/amu -> A/fs^2
    double v = vel[k] + 0.5 * dt * F[k] * inv_mass[k / 3] * conv;
    vel[k] = v;
    if (drift) pos[k] += dt * v;
}

// Intramolecular support potential for the MD driver (not part of the
// intermolecular energy): O-H bonds and the H-O-H angle, harmonic or with the
// MM3-style anharmonic factors (anh = 1), and an optional Urey-Bradley H-H
// term; forces added to F in place.
//   bond  E = kb dr^2 (1 - cs dr + (7/12) cs^2 dr^2), cs = 2.55 / A
//   angle E = ka dth^2 (1 - 0.014 D + 5.6e-5 D^2 - 7e-7 D^3 + 9e-10 D^4), D = dth in degrees
//   UB    E = kub (r_HH - rub)^2
__device__ inline double bond_dEdr(double kb, double dr, int anh) {
    if (!anh) return 2.0 * kb * dr;
    const double cs = 2.55, c4 = (7.0 / 12.0) * cs * cs;
    // d/dr [dr^2 - cs dr^3 + c4 dr^4]
    return kb * (2.0 * dr - 3.0 * cs * dr * dr + 4.0 * c4 * dr * dr * dr);
}
__device__ inline double angle_dEdth(double ka, double dth, int anh) {
    if (!anh) return 2.0 * ka * dth;
    const double g = 180.0 / M_PI;   // degrees per radian
    const double D = dth * g;
    const double f = 1.0 - 0.014 * D + 5.6e-5 * D * D - 7.0e-7 * D * D * D + 9.0e-10 * D * D * D * D;
    const double dfdD = -0.014 + 2.0 * 5.6e-5 * D - 3.0 * 7.0e-7 * D * D + 4.0 * 9.0e-10 * D * D * D;
    return ka * (2.0 * dth * f + dth * dth * dfdD * g);
}

__global__ void k_water_intra(int M, const double *pos, double *F, double kb, double r0, double ka, double th0,
                              int anh, double kub, double rub) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const double *x = pos + m * 9;
    const V3<double> O = mk(x[0], x[1], x[2]), H1 = mk(x[3], x[4], x[5]), H2 = mk(x[6], x[7], x[8]);
    const V3<double> a = H1 - O, b = H2 - O;
    const double ra = sqrt(dot(a, a)), rb = sqrt(dot(b, b));
    // bonds
    const V3<double> fa = (-bond_dEdr(kb, ra - r0, anh) / ra) * a;   // force on H1
    const V3<double> fb = (-bond_dEdr(kb, rb - r0, anh) / rb) * b;
    // angle
    const double c = fmax(-1.0, fmin(1.0, dot(a, b) / (ra * rb)));
    const double th = acos(c);
    const double s = fmax(sqrt(1.0 - c * c), 1e-8);
    const double dEdth = angle_dEdth(ka, th - th0, anh);
    // dtheta/da = -(b/(ra rb) - c a/ra^2)/sin
    const V3<double> dca = (1.0 / (ra * rb)) * b - (c / (ra * ra)) * a;
    const V3<double> dcb = (1.0 / (ra * rb)) * a - (c / (rb * rb)) * b;
    const V3<double> ga = (dEdth / s) * dca;     // -dE/da  (dtheta = -dc/sin)
    const V3<double> gb = (dEdth / s) * dcb;
    V3<double> f1 = fa + ga, f2 = fb + gb;
    if (kub > 0.0) {   // Urey-Bradley: force on H1 along H2 -> H1
        const V3<double> hh = H1 - H2;
        const double rhh = sqrt(dot(hh, hh));
        const V3<double> fu = (-2.0 * kub * (rhh - rub) / rhh) * hh;
        f1 = f1 + fu;
        f2 = f2 - fu;
    }
    double *f = F + m * 9;
    f[0] -= f1.x + f2.x; f[1] -= f1.y + f2.y; f[2] -= f1.z + f2.z;
    f[3] += f1.x; f[4] += f1.y; f[5] += f1.z;
    f[6] += f2.x; f[7] += f2.y; f[8] += f2.z;
}

// Capped steepest-descent update used to relax a starting structure:
// x += F * min(gamma, cap / |F|) per atom.
__global__ void k_sd_step(int M, double *pos, const double *F, double gamma, double cap) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= M * 3) return;
    const double fx = F[a * 3], fy = F[a * 3 + 1], fz = F[a * 3 + 2];
    const double f = sqrt(fx * fx + fy * fy + fz * fz);
    const double s = (f * gamma > cap) ? cap / f : gamma;
    pos[a * 3] += s * fx;
    pos[a * 3 + 1] += s * fy;
    pos[a * 3 + 2] += s * fz;
}

void launch_sd_step(int M, double *pos, const double *F, double gamma, double cap, Launch L) {
    k_sd_step<<<(M * 3 + 127) / 128, 128, 0, L.s>>>(M, pos, F, gamma, cap);
    count(L);
}

void launch_water_intra(int M, const double *pos, double *F, double kb, double r0, double ka, double th0, int anh,
                        double kub, double rub, Launch L) {
    k_water_intra<<<(M + 127) / 128, 128, 0, L.s>>>(M, pos, F, kb, r0, ka, th0, anh, kub, rub);
    count(L);
}

// Beeman integrator, first half: x += v dt + (4 a - a_prev) dt^2 / 6,
// v += (5 a - a_prev) dt / 6, then a_prev <- a (stored as forces).
__global__ void k_beeman1(int M, double *pos, double *vel, const double *inv_mass, const double *F, double *Fprev,
                          double dt) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M * 9) return;
    const double conv = 4.184e-4;   // (kcal/mol/A)/amu -> A/fs^2
    const double im = inv_mass[k / 3] * conv;
    const double a = F[k] * im, ap = Fprev[k] * im;
    const double v = vel[k];
    pos[k] += v * dt + (4.0 * a - ap) * dt * dt * (1.0 / 6.0);
    vel[k] = v + (5.0 * a - ap) * dt * (1.0 / 6.0);
    Fprev[k] = F[k];
}
// second half, after the forces at t + dt: v += 2 a(t + dt) dt / 6
__global__ void k_beeman2(int M, double *vel, const double *inv_mass, const double *F, double dt) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M * 9) return;
    vel[k] += 2.0 * F[k] * inv_mass[k / 3] * 4.184e-4 * dt * (1.0 / 6.0);
}
void launch_beeman(int M, double *pos, double *vel, const double *inv_mass, double *F, double *Fprev, double dt,
                   int half, Launch L) {
    if (half == 1) k_beeman1<<<(M * 9 + 255) / 256, 256, 0, L.s>>>(M, pos, vel, inv_mass, F, Fprev, dt);
    else k_beeman2<<<(M * 9 + 255) / 256, 256, 0, L.s>>>(M, vel, inv_mass, F, dt);
    count(L);
}

void launch_md_kick(int M, double *pos, double *vel, const double *inv_mass, const double *forces, double dt,
                    int drift, Launch L) {
    k_md_kick<<<(M * 9 + 255) / 256, 256, 0, L.s>>>(M, pos, vel, inv_mass, forces, dt, drift);
    count(L);
}

#define INST(R)                                                                                        \
    template void launch_pcg_init<R>(const KParams &, DevState<R> &, int, Launch);                     \
    template void launch_pcg_init_guess<R>(const KParams &, DevState<R> &, MuGuess, Launch);           \
    template void launch_pcg_first<R>(const KParams &, DevState<R> &, Launch);                         \
    template void launch_pcg_step<R>(const KParams &, DevState<R> &, Launch, cudaGraphConditionalHandle, int); \
    template void launch_pol_energy<R>(const KParams &, DevState<R> &, Launch);                        \
    template void launch_finalize<R>(const KParams &, DevState<R> &, double *, Launch);                \
    template void launch_merge_rec<R>(const KParams &, DevState<R> &, Launch);                         \
    template void launch_cluster_energy<R>(const KParams &, DevState<R> &, double *, Launch);           \
    template void launch_virial_total<R>(const KParams &, DevState<R> &, double *, Launch);
INST(float)
INST(double)

}  // namespace sibfa
