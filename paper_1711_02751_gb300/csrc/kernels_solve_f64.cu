// The one-launch trace solve with FP64 cycles, and the layout of its launch.
#include <algorithm>

#include "kernels_solve.inl"

namespace hdgdg {

cudaError_t launch_solve_f64(int P, const SolveArgs& a, cudaStream_t s) { return solve_dispatch<double>(P, a, s); }

namespace {

// The layout over at most sms blocks of smem_max bytes of shared memory
SolvePlan lay_out(int n_edges, int P, int m, bool fp32, int sms, int smem_max) {
    SolvePlan p;
    const int NF = 3 * P;
    const size_t t = fp32 ? 4 : 8;
    // at least kMinRows rows a block: below that an exchange grows faster than the work shrinks; FP32
    // blocks begin at a multiple of four rows (the dots' groups of four)
    const int kMinRows = fp32 ? 128 : 32, unit = !fp32 || NF % 4 == 0 ? 1 : NF % 2 == 0 ? 2 : 4;
    p.edges = std::max((n_edges + sms - 1) / sms, (kMinRows + NF - 1) / NF);
    p.edges = (p.edges + unit - 1) / unit * unit;
    p.blocks = (n_edges + p.edges - 1) / p.edges;
    const int rows = p.edges * NF;
    p.rows_ld = (rows + 23) / 32 * 32 + 8;   // >= rows, 8 mod 32
    const size_t fixed = solve_basis_bytes(p.rows_ld, m, t) + 2 * (size_t)p.rows_ld * t + 24 * (size_t)p.edges;
    const size_t limit = ((size_t)smem_max - sizeof(Shared) - 64) & ~(size_t)15;
    // gathered per edge: FP64 cycles its traces and a product's partial sums; FP32 cycles the
    // residual's traces in eight bytes
    const size_t per_edge = (size_t)NF * 8 * (6 + (fp32 ? 0 : solve_split(NF)));
    if (fixed + 2 * per_edge > limit) return p;
    p.gather_edges = (int)std::min<size_t>((limit - fixed) / per_edge, p.edges);
    p.gather_bytes = (p.gather_edges * per_edge + 15) / 16 * 16;
    p.smem = fixed + p.gather_bytes;
    p.on = true;
    return p;
}

}  // namespace

SolvePlan plan_solve(int n_edges, int P, int m, bool fp32, int max_blocks) {
    int dev = 0, sms = 0, coop = 0, smem_max = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return SolvePlan{};
    }
    if (!coop || sms < 1) return SolvePlan{};
    sms = std::min(sms, kSolveMaxBlocks);
    if (max_blocks > 0) sms = std::min(sms, max_blocks);
    return lay_out(n_edges, P, m, fp32, sms, smem_max);
}

bool solve_fits(int n_edges, int P, int m, bool fp32) { return lay_out(n_edges, P, m, fp32, 152, 227 * 1024).on; }

}  // namespace hdgdg
