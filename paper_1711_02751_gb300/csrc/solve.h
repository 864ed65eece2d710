// The trace solve of a small or mid-size system as ONE cooperative launch (kernels_solve.inl): the
// choice of the start, every restart cycle of GMRES(m), the true residuals and stop tests, the
// back-transformation and the store of the guess history.
#pragma once

#include "internal.h"

namespace hdgdg {

constexpr int kSolveThreads = 512;
constexpr int kSolveMaxBlocks = 256;
constexpr int kSolveMaxCols = GmresCtl::kM + 1;   // columns of one reduction: 32 basis vectors and a norm

// How a handle's system is laid out over the launch's blocks (plan_solve, fixed at create).
struct SolvePlan {
    bool on = false;        // false: the launch-per-operation path
    int blocks = 0;         // grid: one block an SM, all resident (cooperative)
    int edges = 0;          // consecutive edge rows of each block
    int rows_ld = 0;        // leading dimension of the basis in shared memory, = 8 mod 32 values
    int gather_edges = 0;   // edge rows whose six neighbour traces are gathered at a time
    size_t gather_bytes = 0;   // shared memory of the gathered traces and a product's partial sums
    size_t smem = 0;        // dynamic shared memory, bytes
};

// Clock ticks of the launch's parts, as its first block saw them (kernel-class timers).
struct SolveClocks {
    long long spmv, ortho, residual, guess, precond;
};

// How an edge row (NF rows, 6 NF columns) is shared in an FP64 product: kThreads
// threads, each one row and kLoads columns kSplit apart, kChunk at a time.
template <int NF>
struct SolveTile {
    static constexpr int kSplit = NF <= 9 ? 6 : 9;
    static constexpr int kLoads = 6 * NF / kSplit;
    static constexpr int kThreads = kSplit * NF;
    static constexpr int kChunk = kLoads > 10 ? kLoads / 2 : kLoads;   // loads in flight
    static_assert(kLoads * kSplit == 6 * NF && kThreads <= kSolveThreads - 64, "whole columns, one edge fits");
};
inline int solve_split(int NF) { return NF <= 9 ? 6 : 9; }

struct SolveArgs {
    SolvePlan plan;
    int n_edges, m;
    bool twice;                  // Gram-Schmidt twice (else once, FP32 cycles only)
    const void* St;              // S~ of the cycles (T)
    const double* S64;           // S~ in FP64 (the residual), or
    const float* Slo;            // the FP32 remainder: the residual reads the pair (St, Slo)
    const int* col;
    const double* Minv;          // block-Jacobi inverse, FP64 or (pairs) FP32 pairs in place
    bool minv_pairs;
    const double* g;
    double *xt, *w, *qhat;
    // what crosses blocks, each 32-bit half under the number of its exchange (16-byte aligned, zero at
    // create): two buffers of the vector the next product is taken of (one 8-byte word a value in
    // FP32, two in FP64), x~ (two), and two buffers of kSolveMaxCols x blocks partial sums (two)
    unsigned long long *A, *X, *part;
    unsigned* epoch;             // the last exchange's number, kept between launches
    unsigned* count;             // contributions to exchanges (epoch x blocks, modulo 2^32)
    int* error;                  // set when a bounded wait ran out
    const DevHist* dh;           // guess history (nullptr: none)
    bool start_given;            // x~ = xt, w and sc are already set (the least-squares start)
    double coef[7][6];
    double rtol, inner_rel, stagnation;
    int maxit;
    SolveCtl* sc;
    StepStats* ss;
    SolveClocks* clocks;         // nullptr: not wanted
};

// Shared memory of the basis; the start's and the residuals' sums use the same bytes.
__host__ __device__ inline size_t solve_basis_bytes(int rows_ld, int m, size_t t) {
    size_t b = (size_t)m * rows_ld * t;
    const size_t rows = 2 * (size_t)rows_ld * 8, start = 7 * (size_t)(kSolveThreads + 8) * 8;
    b = b > rows ? b : rows;
    b = b > start ? b : start;
    return (b + 15) / 16 * 16;
}
inline size_t solve_part_bytes(int blocks) { return 2 * (size_t)kSolveMaxCols * blocks * 16; }
// Trace vectors (of the cycle's type) whose bytes A and X need; they take the place of the basis in
// global memory, which the one-launch solve keeps in shared memory.
constexpr int solve_basis_vectors(bool fp32) { return fp32 ? 8 : 6; }
// The layout for a system of n_edges edge rows of degree P - 1, restart length m, FP64 or FP32
// cycles, over at most max_blocks blocks (0: one an SM); on = false where it does not fit their shared
// memory.
SolvePlan plan_solve(int n_edges, int P, int m, bool fp32, int max_blocks = 0);
// Whether the system fits one launch on GB300 (152 SMs, 227 KB of shared memory a block): what a handle has
// room for.  No device call.
bool solve_fits(int n_edges, int P, int m, bool fp32);
cudaError_t launch_solve_f64(int P, const SolveArgs& a, cudaStream_t s);
cudaError_t launch_solve_f32(int P, const SolveArgs& a, cudaStream_t s);

}  // namespace hdgdg
