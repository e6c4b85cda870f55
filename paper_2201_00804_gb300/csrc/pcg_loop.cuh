// The polarization solve as one kernel: what the host lays out for it.
#pragma once
#include <cstdlib>
#include <vector>

#include "pcg_guess.cuh"
#include "sibfa_internal.cuh"

namespace sibfa {

constexpr int FFT_RADICES = 8;   // factors of one axis at most
// Largest system whose solve runs in the one kernel (waters), periodic and gas
// phase.  Measured (dipole solve, us an iteration, one kernel / separate
// kernels): 216 waters 25 / 50, 971 32 / 50, 1690 46 / 57, 4096 54 / 65 alone
// but 68 beside the short-range kernels, whose warps hold up the barriers:
// from about 2000 waters the evaluation is bound by throughput, not latency.
constexpr int LOOP_MAX_MOL = 1700;

// One pass of an axis' transform: its radix, the product sp of the radices
// before it, n / (sp radix), and the reciprocal that divides by sp.
struct FftPass {
    int r, sp, m;
    unsigned div_sp;
};
struct FftAxis {
    int n, npass, tw;   // tw: start of this axis' twiddles in the table
    FftPass pass[FFT_RADICES];
};

// Layout of the solve kernel for one context: blocks and the molecules each
// owns, the passes of the grid axes (radices 2, 3, 4, 5, 8), the twiddles.
struct LoopPlan {
    int ncta = 0;                    // blocks (0: this context's solves take the separate kernels)
    int mper = 0;                    // molecules per block
    int maxit = 200;
    unsigned polls = 1u << 22;       // of the grid counter before a block gives up (seconds; the waits are microseconds)
    FftAxis ax[3] = {};
    int ntw = 0;                     // twiddles of all axes
    int xt = 0;                      // (ky, kz) columns per tile of the x transforms
    int nbuf = 0;                    // complex elements of one transform buffer
    int staged = 0;                  // the pair list goes through shared memory (rows are 16-byte aligned)
    unsigned div_k2 = 0, div_l = 0, div_nz = 0, div_xt = 0;   // reciprocals of the index divisions
    void *tw = nullptr;              // exp(-2 pi i k / K) of every axis, working precision
    void *vec = nullptr;             // the product's vector, 4 values per atom, working precision
    double *part = nullptr;          // 3 x ncta partial sums
    size_t smem = 0;
};

// Fills the plan's sizes for M molecules (grid K when periodic); ncta stays 0
// when the kernel does not take the problem.
template <typename R> void loop_plan(LoopPlan &L, int M, int periodic, const int K[3], int tls, int n_sm);
// Plan of the one-kernel grid convolution (transform fields only); ncta stays
// 0 for grids it does not take, which go through the transform library.
template <typename R> void conv_plan(LoopPlan &L, const int K[3], int n_sm);
template <typename R>
cudaError_t launch_grid_conv(const KParams &p, DevState<R> &d, const LoopPlan &lp, int ngrid, Launch L);
// twiddles of all axes, re/im interleaved
std::vector<double> loop_twiddles(const int K[3]);
template <typename R>
cudaError_t launch_pcg_loop(const KParams &p, DevState<R> &d, const LoopPlan &lp, const MuGuess &g, int warm,
                            double *push, Launch L);

// Largest cluster the per-cluster solve takes (waters): its displacements,
// n (n - 1) of them, stay in shared memory (48 KB at 64 waters).
constexpr int CLUSTER_MAX = 64;
// SIBFA_PCG_HOST_LOOP=1: solves are driven from the host, by separate kernels
inline bool host_loop() {
    const char *e = std::getenv("SIBFA_PCG_HOST_LOOP");
    return e && e[0] == '1';
}
// Whether a context whose largest cluster has n waters solves each on its own,
// and so records no pair list
inline bool own_cluster_solve(int periodic, int precision, int n) {
    return !host_loop() && !periodic && precision == SIBFA_PREC_MIXED && n <= CLUSTER_MAX;
}
// Admits the largest cluster's shared memory; once per context, at creation.
cudaError_t cluster_init();
// Every cluster of a gas-phase batch (mixed path) on its own, one block each; nmax: the largest.
cudaError_t launch_pcg_cluster(const KParams &p, DevState<float> &d, int nmax, int maxit, const MuGuess &g, int warm,
                               double *push, Launch L);

}  // namespace sibfa
