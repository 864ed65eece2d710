// One launch per trace solve (see solve.h), included by kernels_solve_f64.cu and kernels_solve_f32.cu.
//
// A small trace system leaves the launch-per-operation path nothing but latency: on 8 x 8, k = 2
// (1152 unknowns) an Arnoldi step took 55 us over four launches, of which the product 8 and the
// rest the FP64 reductions of 608 mostly idle blocks and a one-thread Hessenberg update (each FP64
// warp instruction holds an SM partition's pipe for about 60 cycles).  Here each block keeps a fixed
// range of edge rows for the whole solve -- its rows of the basis in shared memory, its rows of S~
// in L1 / L2 -- and an Arnoldi step is
//   product z = S~ v_j of the published v_j, while two warps form the previous step's Hessenberg
//   column, its rotation and the stop test; the dots h1 = V^T z, exchanged between all blocks;
//   w1 = z - V h1; the dots h2 = V^T w1 and ||w1||^2, exchanged; v_{j+1} = (w1 - V h2) / hn, published.
// FP64 cycles delay the second pass: w1 is published and its product corrected to that of v through
// A V = V H (launch_dcgs_fused), which hides the publication behind an exchange.  FP32 cycles keep
// the order of the launch-per-operation path in every FP32 sum that a solution depends on -- products,
// updates, and the dots' groups of four (see contribute): where a solve ends within its tolerance
// depends on their rounding.
// A restart cycle adds two exchanges' worth of waiting (x~ published; the true residual's norm).
// Every block sums all blocks' partial sums itself, in block order, and takes every decision from
// the same numbers.  There is no fenced barrier: every value that crosses blocks -- partial sums,
// the published vectors -- carries the number of its exchange in its upper 32 bits, and its readers
// load it until that number is there (bounded).  A barrier's fence and acquire wait for more trips to
// L2 (a trip within a die takes 555 cycles, across dies 920), and the acquire empties L1 of S~.  A value is
// overwritten only after an exchange to which every block contributed after reading it; the
// published vector has two buffers, since a cycle's last product and the publication of its
// residual have no exchange between them.
// FP32 cycles: sums of four products in FP32, sums of those as FP32 pairs (TwoSum, 48 bits) -- the
// FP64 pipe has no part in them.
//
// Measured (time step, launch-per-operation path -> one launch; GMRES iterations a step in brackets):
//   FP64 form   8^2, k = 2 (80)    4.37 -> 0.90 ms: 55 -> 9.4 us an iteration
//               20^2, k = 8, walls (57)  3.84 -> 1.40 ms: the product 9.7 us of 6.9 us of FP64 FMAs
//   mixed form  32^2, k = 2 (50)   2.51 -> 0.58 ms; 91^2, k = 3 (36)  2.33 -> 0.97 ms;
//               16 x 32^2, k = 3 (48)  4.15 -> 2.83 ms: bound by the 113 MB of S~ a product
// Bounds now: two exchanges an iteration (about 1.4 us each with 128 to 152 blocks) and the chains
// between them at small sizes, S~'s bytes through 448 threads an SM at large ones.
#include <cstdint>

#include "pairsum.h"
#include "solve.h"

namespace hdgdg {
namespace {

constexpr int kNT = kSolveThreads, kNW = kNT / 32;
constexpr int kCtlWarps = 2;                    // warps 0 and 1: Hessenberg column, rotation, stop test
constexpr int kProdThreads = kNT - 32 * kCtlWarps;
constexpr unsigned kMaxSpins = 1u << 22;        // bound of every wait: loads, each a trip to L2 (0.8 s)

// Values that cross blocks: each 32-bit half in an 8-byte word (accessed at once) under the 32-bit
// number of the exchange it belongs to.
using u64 = unsigned long long;
template <typename V>
struct Tagged {   // float: one word
    static constexpr int kWords = 1;
    static __device__ __forceinline__ u64 word(float v, int, unsigned tag) {
        return ((u64)tag << 32) | __float_as_uint(v);
    }
    static __device__ __forceinline__ float value(const u64* w) { return __uint_as_float((unsigned)w[0]); }
};
template <>
struct Tagged<double> {
    static constexpr int kWords = 2;
    static __device__ __forceinline__ u64 word(double v, int k, unsigned tag) {
        return ((u64)tag << 32) | (unsigned)(k ? __double2hiint(v) : __double2loint(v));
    }
    static __device__ __forceinline__ double value(const u64* w) {
        return __hiloint2double((int)(unsigned)w[1], (int)(unsigned)w[0]);
    }
};
template <>
struct Tagged<PairSum> {
    static constexpr int kWords = 2;
    static __device__ __forceinline__ u64 word(PairSum v, int k, unsigned tag) {
        return ((u64)tag << 32) | __float_as_uint(k ? v.lo : v.hi);
    }
    static __device__ __forceinline__ PairSum value(const u64* w) {
        return PairSum{__uint_as_float((unsigned)w[0]), __uint_as_float((unsigned)w[1])};
    }
};
// N words from p (16-byte aligned when N is even), past L1
template <int N>
__device__ __forceinline__ void load_words(const u64* p, u64* w) {
    if constexpr (N % 2 == 0) {
#pragma unroll
        for (int k = 0; k < N; k += 2)
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[k]), "=l"(w[k + 1]) : "l"(p + k));
    } else {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w[0]) : "l"(p));
    }
}
template <int N>
__device__ __forceinline__ bool tags_are(const u64* w, unsigned tag) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < N; ++k) ok = ok && (unsigned)(w[k] >> 32) == tag;
    return ok;
}
template <typename V>
__device__ __forceinline__ void store_tagged(u64* p, V v, unsigned tag) {
    if constexpr (Tagged<V>::kWords == 2)
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(Tagged<V>::word(v, 0, tag)),
                     "l"(Tagged<V>::word(v, 1, tag))
                     : "memory");
    else
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(Tagged<V>::word(v, 0, tag)) : "memory");
}

struct Shared {   // static shared memory of a block
    double sum[kSolveMaxCols];       // the last grid-wide sums
    double h1[kSolveMaxCols], h2[kSolveMaxCols];   // h2[0] = ||w1||^2, h2[1 + k]: the second pass' dots
    double ht[4][kSolveMaxCols];     // h1, h2, c = H h2 and y in the cycle's type, converted once
    PairSum pair[kSolveMaxCols];     // h2 as FP32 pairs (FP32 cycles)
    double Hr[GmresCtl::kM][kSolveMaxCols];    // [column][row], before the rotations
    double Rr[GmresCtl::kM][kSolveMaxCols];    // [column][row], after them
    double Q[kSolveMaxCols][kSolveMaxCols];    // [column][row] of the accumulated rotations
    double inv_r[GmresCtl::kM], s[kSolveMaxCols];
    double inv_hn, inv_beta;
    double bnorm, tol, tol_cycle;
    double seg[kNW][kSolveMaxCols];  // a reduction's segments (8 bytes each, FP64 or FP32 pairs)
    long long clk[5], last;          // spmv, ortho, residual, guess, precond (thread 0 of block 0)
    int done, status, total, cycles, guess, active, go, nonfinite, notconv, gave_up;
};

__device__ __forceinline__ void prod_barrier() {   // the threads that form the product
    asm volatile("bar.sync 1, %0;" ::"n"(kProdThreads) : "memory");
}

// The thread's index, opaque to the compiler: what a phase derives from it is computed in that phase
// again instead of being kept (and spilled) across the whole solve.
__device__ __forceinline__ int thread_index() {
    int t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}

template <int NF, typename T>
struct Solver {
    using S = typename SumOf<T>::S;
    static constexpr bool kF32 = sizeof(T) == 4;
    static constexpr int kGuessLd = kNT + 8;
    // rows a thread holds at a time in the vector updates (FP64: the pipe is full with one)
    static constexpr int kRows = kF32 ? 4 : 1;
    const SolveArgs& a;
    Shared& sh;
    T *V, *z, *ao;       // own rows: basis, product, own part of the published vector
    T *h1t, *h2t, *ct, *yt;
    char* gbuf;          // gathered neighbour traces
    int e0, ne, R, ld;   // first own edge, own edges, own rows, leading dimension
    size_t r0;           // first own row
    unsigned epoch;      // number of the last exchange: the same in every thread of every block
    unsigned abuf;       // which of the two buffers of A holds the vector published last
    int* scol;           // the own edges' six neighbours
    bool timed, quads;   // quads: the vectors' length is a multiple of four

    __device__ Solver(const SolveArgs& args, Shared& s, char* dyn) : a(args), sh(s) {
        ld = a.plan.rows_ld;
        e0 = blockIdx.x * a.plan.edges;
        ne = min(a.plan.edges, a.n_edges - e0);
        R = ne * NF;
        r0 = (size_t)e0 * NF;
        epoch = 0;
        abuf = 0;
        quads = ((size_t)a.n_edges * NF & 3) == 0;
        h1t = reinterpret_cast<T*>(sh.ht[0]);
        h2t = reinterpret_cast<T*>(sh.ht[1]);
        ct = reinterpret_cast<T*>(sh.ht[2]);
        yt = reinterpret_cast<T*>(sh.ht[3]);
        timed = a.clocks && blockIdx.x == 0 && threadIdx.x == 0;
        V = reinterpret_cast<T*>(dyn);
        dyn += solve_basis_bytes(ld, a.m, sizeof(T));
        z = reinterpret_cast<T*>(dyn);
        ao = z + ld;
        gbuf = dyn + 2 * (size_t)ld * sizeof(T);
        scol = reinterpret_cast<int*>(gbuf + a.plan.gather_bytes);
    }

    __device__ __forceinline__ void mark(int cls) {   // the time since the last mark belongs to class cls
        if (!timed) return;
        const long long now = clock64();
        sh.clk[cls] += now - sh.last;
        sh.last = now;
    }

    // Whether to stop waiting after `spins` fruitless loads: the error word is then set, and every later
    // wait of every block ends early.  (A bound that is no constant -- an argument of the launch, a word in
    // memory -- took 0.5 to 1 % of 8^2, k = 2, FP64.)
    __device__ __forceinline__ bool give_up(unsigned spins) {
        if ((spins & 63u) != 63u) return false;
        if (*(volatile int*)&sh.gave_up == 0 && *reinterpret_cast<volatile int*>(a.error) == 0 && spins < kMaxSpins)
            return false;
        atomicExch(a.error, 3);
        *(volatile int*)&sh.gave_up = 1;
        return true;
    }

    __device__ __forceinline__ u64* a_buffer() {
        return a.A + (size_t)abuf * a.n_edges * NF * Tagged<T>::kWords;
    }

    __device__ __forceinline__ u64* part_buffer() {   // the buffer of the exchange `epoch`
        return a.part + (size_t)(epoch & 1u) * kSolveMaxCols * gridDim.x * 2;
    }

    // Begin the next exchange: the block's sums over n rows: with self a first column zz times zz, then
    // nv columns cols + c * ldc (times zz when DOT).  Groups of eight lanes take one column each, the
    // four groups of a warp adjacent columns of the same rows; the rows are cut into segments so that
    // every warp has work.  FP32 dots add the products of four consecutive rows (aligned to four in the
    // whole vector; single products when its length is no multiple of four) in FP32, as a thread's
    // 16-byte lanes in multidot_kernel and axpy_dot_kernel do, and those sums as pairs, in FP64 there.  Up
    // to 466 944 unknowns, where a thread there has one such group (beyond, it chains the next ones in
    // FP32), the coefficients round to the same FP32 values but near ties: 69 of 72 random dots.
    // Starts with a block barrier.
    template <typename U, bool DOT>
    __device__ __forceinline__ void contribute(const U* cols, int ldc, int nv, const U* zz, bool self, int n) {
        using SU = typename SumOf<U>::S;
        const int tid = thread_index(), lane = tid & 31, wid = tid >> 5;
        epoch += 1;
        const int ncols = nv + (self ? 1 : 0), cbs = (ncols + 3) / 4;
        int segs = cbs == 1 ? kNW : cbs == 2 ? kNW / 2 : cbs == 3 ? kNW / 3 : kNW / cbs;
        const int want = (n + 31) >> 5;
        segs = segs < 1 ? 1 : segs > want ? want : segs;
        const int rs = ((n + segs - 1) / segs + 31) & ~31;
        SU* seg = reinterpret_cast<SU*>(&sh.seg[0][0]);
        __syncthreads();
        for (int t = wid; t < cbs * segs; t += kNW) {
            const int cb = t / segs, sg = t - cb * segs, c = 4 * cb + (lane >> 3);
            SU s{};
            if (c < ncols) {
                const U* p = !self ? cols + (size_t)c * ldc : c > 0 ? cols + (size_t)(c - 1) * ldc : zz;
                const int hi = min(n, (sg + 1) * rs);
                if constexpr (DOT && sizeof(U) == 4) {
                    if (quads) {
#pragma unroll 2
                        for (int r = sg * rs + 4 * (lane & 7); r < hi; r += 32) {
                            const float4 v = *reinterpret_cast<const float4*>(p + r);
                            const float4 w = *reinterpret_cast<const float4*>(zz + r);
                            s = add(s, __fmaf_rn(v.w, w.w, __fmaf_rn(v.z, w.z, __fmaf_rn(v.y, w.y, __fmul_rn(v.x, w.x)))));
                        }
                    } else {
#pragma unroll 2
                        for (int r = sg * rs + (lane & 7); r < hi; r += 8) s = add(s, __fmul_rn(p[r], zz[r]));
                    }
                } else {
#pragma unroll 4
                    for (int r = sg * rs + (lane & 7); r < hi; r += 8) {
                        if constexpr (DOT) s += p[r] * zz[r];
                        else s = add(s, p[r]);
                    }
                }
            }
            s = add(s, shfl_xor(s, 4));
            s = add(s, shfl_xor(s, 2));
            s = add(s, shfl_xor(s, 1));
            if ((lane & 7) == 0 && c < ncols) seg[sg * kSolveMaxCols + c] = s;
        }
        __syncthreads();
        if (tid < ncols) {
            SU s = seg[tid];
            for (int k = 1; k < segs; ++k) s = add(s, seg[k * kSolveMaxCols + tid]);
            store_tagged(part_buffer() + 2 * ((size_t)tid * gridDim.x + blockIdx.x), s, epoch);
        }
        if (tid < 32) {
            __syncwarp();
            if (tid == 0) asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(a.count) : "memory");
        }
    }

    // End the exchange: out[c] (outt[c] in the cycle's type, outp[c] as a pair) = the sum of column c
    // over all blocks, in a fixed order.  One thread waits for the count of contributions -- polling
    // the partials themselves costs more the more blocks poll them (152 blocks, 6 columns: 8600
    // cycles an exchange, and 6600 through one owner a column; a counter and its poll 2500) -- and
    // the partials are then read once; their tags, not the count, say that they are there.
    // Ends with a block barrier and reads the flag of a wait that ran out (false: leave).  Every thread has
    // to read the same, so the caller's next wait comes after another block barrier: a thread that went on
    // into it could set the flag, those that saw it would leave and the others wait for them without end.
    template <typename U>
    __device__ __forceinline__ bool collect(int ncols, double* out, T* outt = nullptr, PairSum* outp = nullptr) {
        using SU = typename SumOf<U>::S;
        constexpr int kU = 4;   // loads in flight
        const int tid = thread_index(), G = gridDim.x;
        if (tid == 0) {
            const unsigned all = epoch * (unsigned)G;   // (both count modulo 2^32)
            for (unsigned spins = 0;; ++spins) {
                unsigned v;
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.count));
                if ((int)(v - all) >= 0 || give_up(spins)) break;
            }
        }
        __syncthreads();
        // lanes of one column: FP64 adds share a partition's pipe between its warps, FP32 ones do not
        const int lw = ncols <= (sizeof(U) == 4 ? 16 : 4) ? 5 : ncols <= 8 ? 4 : 3, w = 1 << lw;
        const int c = tid >> lw, l = tid & (w - 1);
        SU s{};
        if (c < ncols) {
            const u64* col = part_buffer() + 2 * (size_t)c * G;
            for (int k0 = l; k0 < G; k0 += kU * w) {
                u64 v[kU][2];
                for (unsigned spins = 0;; ++spins) {
                    bool ok = true;
#pragma unroll
                    for (int u = 0; u < kU; ++u) load_words<2>(col + 2 * min(k0 + u * w, G - 1), v[u]);
#pragma unroll
                    for (int u = 0; u < kU; ++u) ok = ok && tags_are<2>(v[u], epoch);
                    if (ok || give_up(spins)) break;
                }
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (k0 + u * w < G) s = add(s, Tagged<SU>::value(v[u]));
            }
        }
        __syncwarp();
        for (int o = w / 2; o > 0; o >>= 1) s = add(s, shfl_xor(s, o));
        if (c < ncols && l == 0) {
            const double v = value(s);
            out[c] = v;
            if (outt) outt[c] = from_f64<T>(v);
            if constexpr (sizeof(SU) == sizeof(PairSum) && sizeof(U) == 4) {
                if (outp) outp[c] = s;
            }
        }
        __syncthreads();
        return sh.gave_up == 0;
    }

    // The neighbour traces of ng own edge rows from g0 on, of the vector published in `buf` by the
    // exchange `tag`: put(i, value) for i = (edge - g0, slot, component).  Four loads of up to 16 bytes
    // in flight a thread.
    template <typename V, typename F>
    __device__ __forceinline__ void gather(const u64* buf, unsigned tag, int g0, int ng, int t, int nt, F&& put) {
        constexpr int kW = Tagged<V>::kWords, kPer = kW == 1 && NF % 2 == 0 ? 2 : 1;   // values a load
        constexpr int kU = 4, kN = NF / kPer;
        const int* col = scol + g0 * 6;
        const int n = ng * 6 * kN;
        for (int i0 = t; i0 < n; i0 += kU * nt) {
            u64 v[kU][kW * kPer];
            const u64* p[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int i = min(i0 + u * nt, n - 1), slot = i / kN;
                p[u] = buf + ((size_t)col[slot] * NF + (i - slot * kN) * kPer) * kW;
            }
            for (unsigned spins = 0;; ++spins) {
                bool ok = true;
#pragma unroll
                for (int u = 0; u < kU; ++u) load_words<kW * kPer>(p[u], v[u]);
#pragma unroll
                for (int u = 0; u < kU; ++u) ok = ok && tags_are<kW * kPer>(v[u], tag);
                if (ok || give_up(spins)) break;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (i0 + u * nt < n) {
#pragma unroll
                    for (int q = 0; q < kPer; ++q) put((i0 + u * nt) * kPer + q, Tagged<V>::value(v[u] + q * kW));
                }
        }
    }

    // z = x + S~ x on the own rows (own: the own rows of x), by the kProdThreads threads t >= 0 that are
    // not control warps.  FP32: one thread a row, its products added in the order of spmv_pre_kernel
    // (the rounding of an FP32 cycle's products decides where in its tolerance a solve ends), the
    // matrix loaded kAhead blocks ahead.  FP64: Tile::kThreads consecutive threads take an edge row,
    // each every kSplit-th column of its six blocks, since a row's chain of FP64 FMAs is long.  The first
    // entries are loaded before the gathered traces are waited for.
    __device__ __forceinline__ void product(int t, const u64* x, unsigned tag, const T* own) {
        // FP32 needs no room for partial sums: more edges at a time
        const int GE = kF32 ? (int)(a.plan.gather_bytes / (6 * NF * 4)) : a.plan.gather_edges;
        T* sx = reinterpret_cast<T*>(gbuf);
        for (int g0 = 0; g0 < ne; g0 += GE) {
            const int ng = min(GE, ne - g0), nrow = ng * NF;
            const T* __restrict__ S0 = static_cast<const T*>(a.St) + (size_t)(e0 + g0) * 6 * NF * NF;
            if constexpr (kF32) {
                constexpr int kAhead = NF <= 15 ? 2 : 1;
                T m[kAhead + 1][NF];
                const int le0 = t / NF;
                const T* M = S0 + (size_t)le0 * 6 * NF * NF + (t - le0 * NF);
                if (t < nrow) {
#pragma unroll
                    for (int b = 0; b < kAhead; ++b) load_entries<NF, 1>(M + b * NF * NF, m[b]);
                }
                gather<T>(x, tag, g0, ng, t, kProdThreads, [&](int i, T v) { sx[i] = v; });
                prod_barrier();
                for (int rr = t; rr < nrow; rr += kProdThreads) {
                    const int le = rr / NF, next = rr + kProdThreads, ln = next / NF;
                    const T* Mn = S0 + (size_t)ln * 6 * NF * NF + (next - ln * NF);
                    const T* xs = sx + le * 6 * NF;
                    T acc = own[g0 * NF + rr];
#pragma unroll
                    for (int sl = 0; sl < 6; ++sl) {
                        T* into = m[(sl + kAhead) % (kAhead + 1)];
                        if (sl + kAhead < 6) load_entries<NF, 1>(M + (sl + kAhead) * NF * NF, into);
                        else if (next < nrow) load_entries<NF, 1>(Mn + (sl + kAhead - 6) * NF * NF, into);
#pragma unroll
                        for (int jj = 0; jj < NF; ++jj) acc += m[sl % (kAhead + 1)][jj] * xs[sl * NF + jj];
                    }
                    z[g0 * NF + rr] = acc;
                    M = Mn;
                }
                prod_barrier();
            } else {
                using Tl = SolveTile<NF>;
                constexpr int kC = Tl::kChunk, kN = Tl::kLoads / kC, kTPE = Tl::kThreads, kEPP = kProdThreads / kTPE;
                T* ps = sx + GE * 6 * NF;
                const int te = t / kTPE, sub = t - te * kTPE, sp = sub / NF, ii = sub - sp * NF;
                const bool on = te < kEPP;
                const T* M = S0 + (size_t)te * 6 * NF * NF + sp * NF + ii;
                T m[2][kC];
                if (on && te < ng) load_entries<kC, Tl::kSplit>(M, m[0]);
                gather<T>(x, tag, g0, ng, t, kProdThreads, [&](int i, T v) { sx[i] = v; });
                prod_barrier();
                for (int le = te; on && le < ng; le += kEPP) {
                    const T* Mn = M + (size_t)kEPP * 6 * NF * NF;
                    const T* xs = sx + le * 6 * NF + sp;
                    T acc = T(0);
#pragma unroll
                    for (int c = 0; c < kN; ++c) {   // the next chunk is loaded while this one is multiplied
                        if (c + 1 < kN) load_entries<kC, Tl::kSplit>(M + (c + 1) * kC * Tl::kSplit * NF, m[1]);
                        else if (le + kEPP < ng) load_entries<kC, Tl::kSplit>(Mn, m[1]);
#pragma unroll
                        for (int k = 0; k < kC; ++k) acc += m[0][k] * xs[(c * kC + k) * Tl::kSplit];
#pragma unroll
                        for (int k = 0; k < kC; ++k) m[0][k] = m[1][k];
                    }
                    ps[(le * Tl::kSplit + sp) * NF + ii] = acc;
                    M = Mn;
                }
                prod_barrier();
                for (int rr = t; rr < nrow; rr += kProdThreads) {
                    const int le = rr / NF;
                    const T* p = ps + le * (Tl::kSplit - 1) * NF + rr;   // (le kSplit NF + the row of the edge)
                    T v = own[g0 * NF + rr];
#pragma unroll
                    for (int k = 0; k < Tl::kSplit; ++k) v += p[k * NF];
                    z[g0 * NF + rr] = v;
                }
                if (g0 + GE < ne) prod_barrier();
            }
        }
    }

    // kL entries of an edge row's blocks, kSplit columns apart
    template <int kL, int kSplit, typename TM>
    __device__ __forceinline__ void load_entries(const TM* __restrict__ M, TM* m) {
#pragma unroll
        for (int k = 0; k < kL; ++k) m[k] = __ldg(M + k * kSplit * NF);
    }

    // Warps 0 and 1, after the sums of step j's second pass: hn = sqrt(||w1||^2 - ||h2||^2) (the norm
    // of w1 - V h2 for an orthonormal V); warp 0 (FP64 cycles): the Hessenberg column h1 + h2, hn and
    // c = H h2; warp 1: the accumulated rotations applied to the column, the new rotation, the residual
    // estimate and the stop test.  Lane i holds row i.
    __device__ __forceinline__ void control(int j) {
        const int lane = thread_index() & 31, wid = thread_index() >> 5;
        const double h2v = lane <= j ? sh.h2[1 + lane] : 0.0;
        double q = h2v * h2v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        const double s2 = sh.h2[0] - q;
        const double hn = s2 > 0.0 ? sqrt(s2) : 0.0;
        const double hc = lane <= j ? sh.h1[lane] + h2v : 0.0;
        if (wid == 0) {
            if constexpr (!kF32) {   // (FP32 cycles form v before their product)
                sh.Hr[j][lane] = lane == j + 1 ? hn : hc;
                __syncwarp();
                double c = 0.0;
                for (int k = 0; k <= j; ++k) c += sh.Hr[k][lane] * sh.h2[1 + k];
                ct[lane] = from_f64<T>(c);
                if (lane == 0) sh.inv_hn = 1.0 / hn;
            }
        } else {
            double r = 0.0;
            for (int k = 0; k <= j; ++k) r += sh.Q[k][lane] * __shfl_sync(0xffffffffu, hc, k);
            const double p = __shfl_sync(0xffffffffu, r, j);
            const double den = sqrt(p * p + hn * hn);
            const double inv = 1.0 / den;
            const double cs = den > 0.0 ? p * inv : 1.0, sn = den > 0.0 ? hn * inv : 0.0;
            sh.Rr[j][lane] = lane < j ? r : lane == j ? den : 0.0;
            const double qv = lane <= j ? sh.Q[lane][j] : 0.0;
            __syncwarp();
            if (lane <= j) {
                sh.Q[lane][j] = cs * qv;
                sh.Q[lane][j + 1] = -sn * qv;
            } else if (lane == j + 1) {
                sh.Q[lane][j] = sn;
                sh.Q[lane][j + 1] = cs;
            }
            if (lane == 0) {
                const double sj = sh.s[j];
                const double est = fabs(sn * sj);
                sh.s[j] = cs * sj;
                sh.s[j + 1] = -sn * sj;
                sh.inv_r[j] = inv;
                sh.total += 1;
                if (!isfinite(est)) {
                    sh.status = 1;
                    sh.done = 1;
                } else if (est <= sh.tol_cycle || hn == 0.0 || sh.total >= a.maxit || j == a.m - 1) {
                    sh.done = 1;
                }
            }
        }
    }

    // own row r of the vector the next product is taken of
    __device__ __forceinline__ void publish(int r, T v) {
        store_tagged(a_buffer() + (r0 + r) * Tagged<T>::kWords, v, epoch);
    }

    // own row r of the residual w, its square in sq; FP64 cycles begin with the product of w itself
    __device__ __forceinline__ void put_residual(int r, double w, double* sq) {
        a.w[r0 + r] = w;
        if constexpr (!kF32) {
            ao[r] = w;
            publish(r, w);
        }
        sq[r] = w * w;
    }

    // w = g - (x~ + S~ x~) on the own rows (put_residual), and the exchange of ||w||^2 begun.  FP64
    // cycles: the cycles' own product.  FP32 cycles: S~ in FP64, or as the FP32 pair with compensated
    // sums.
    __device__ __forceinline__ void residual() {
        double* sq = reinterpret_cast<double*>(V);
        const int tid = thread_index();
        abuf ^= 1u;
        if constexpr (!kF32) {
            __syncthreads();
            if (tid >= 32 * kCtlWarps) product(tid - 32 * kCtlWarps, a.X, epoch, a.xt + r0);
            __syncthreads();
            for (int r = tid; r < R; r += kNT) put_residual(r, a.g[r0 + r] - z[r], sq);
        } else {
            // one thread a row, in the order of residual_norm_x2_kernel, the pairs of a block ahead
            constexpr int kAhead = NF <= 15 ? 1 : 0;
            const int GE = (int)(a.plan.gather_bytes / (6 * NF * 8));
            double* sx = reinterpret_cast<double*>(gbuf);
            float2* sp2 = reinterpret_cast<float2*>(gbuf);
            __syncthreads();
            for (int g0 = 0; g0 < ne; g0 += GE) {
                const int ng = min(GE, ne - g0), nrow = ng * NF;
                const size_t og = (size_t)(e0 + g0) * 6 * NF * NF;
                const int le0 = tid / NF;
                size_t o = og + (size_t)le0 * 6 * NF * NF + (tid - le0 * NF);
                if (a.Slo) {
                    const float* Sh = static_cast<const float*>(a.St);
                    float mh[kAhead + 1][NF], ml[kAhead + 1][NF];
                    if (kAhead && tid < nrow) {
                        load_entries<NF, 1>(Sh + o, mh[0]);
                        load_entries<NF, 1>(a.Slo + o, ml[0]);
                    }
                    gather<double>(a.X, epoch, g0, ng, tid, kNT,
                                   [&](int i, double v) { hdgdg::split(v, sp2[i].x, sp2[i].y); });
                    __syncthreads();
                    for (int rr = tid; rr < nrow; rr += kNT) {
                        const int r = g0 * NF + rr, next = rr + kNT, ln = next / NF;
                        const float2* xs = sp2 + rr / NF * 6 * NF;
                        const size_t on = og + (size_t)ln * 6 * NF * NF + (next - ln * NF);
                        Dot2 acc;
#pragma unroll
                        for (int sl = 0; sl < 6; ++sl) {
                            const int into = (sl + kAhead) % (kAhead + 1), cur = sl % (kAhead + 1);
                            if (sl + kAhead < 6) {
                                load_entries<NF, 1>(Sh + o + (sl + kAhead) * NF * NF, mh[into]);
                                load_entries<NF, 1>(a.Slo + o + (sl + kAhead) * NF * NF, ml[into]);
                            } else if (next < nrow) {
                                load_entries<NF, 1>(Sh + on, mh[into]);
                                load_entries<NF, 1>(a.Slo + on, ml[into]);
                            }
#pragma unroll
                            for (int jj = 0; jj < NF; ++jj) {
                                const float2 xv = xs[sl * NF + jj];
                                acc.add(mh[cur][jj], ml[cur][jj], xv.x, xv.y);
                            }
                        }
                        put_residual(r, a.g[r0 + r] - (a.xt[r0 + r] + acc.value()), sq);
                        o = on;
                    }
                } else {
                    gather<double>(a.X, epoch, g0, ng, tid, kNT, [&](int i, double v) { sx[i] = v; });
                    __syncthreads();
                    for (int rr = tid; rr < nrow; rr += kNT) {
                        const int r = g0 * NF + rr, le = rr / NF;
                        const double* Sd = a.S64 + og + (size_t)le * 6 * NF * NF + (rr - le * NF);
                        const double* xs = sx + le * 6 * NF;
                        double acc = a.xt[r0 + r];
#pragma unroll 1
                        for (int sl = 0; sl < 6; ++sl) {
                            double m[NF];
                            load_entries<NF, 1>(Sd + sl * NF * NF, m);
#pragma unroll
                            for (int jj = 0; jj < NF; ++jj) acc += m[jj] * xs[sl * NF + jj];
                        }
                        put_residual(r, a.g[r0 + r] - acc, sq);
                    }
                }
                if (g0 + GE < ne) __syncthreads();
            }
        }
        contribute<double, false>(sq, 0, 1, nullptr, false, R);
    }

    // ||g||^2 and the squared residual norms of the start's candidates (the terms of guess_norms_body or, FP32
    // cycles, guess_norms_x2_body; those added as FP32 pairs from the first on): the exchange begun
    __device__ __forceinline__ void candidates(int avail) {
        const int tid = thread_index();
        if (kF32 && avail > 0) {
            PairSum acc[7] = {};
            for (int r = tid; r < R; r += kNT) {
                const double gv = a.g[r0 + r], y0 = a.dh->y[0][r0 + r];
                const float gh = f64_to_f32(gv), e = f64_to_f32(gv - y0);
                float d[6];
#pragma unroll
                for (int j = 1; j < 6; ++j) d[j] = j < avail ? f64_to_f32(y0 - a.dh->y[j][r0 + r]) : 0.f;
                acc[0] = add(acc[0], __fmul_rn(gh, gh));
#pragma unroll
                for (int q = 1; q < 7; ++q) {
                    if (q > avail) break;
                    float v = e;
#pragma unroll
                    for (int j = 1; j < 6; ++j)
                        if (j < q) v = __fmaf_rn(f64_to_f32(a.coef[q][j]), d[j], v);
                    acc[q] = add(acc[q], __fmul_rn(v, v));
                }
            }
            PairSum* buf = reinterpret_cast<PairSum*>(V);
#pragma unroll
            for (int q = 0; q < 7; ++q) buf[q * kGuessLd + tid] = acc[q];
            contribute<PairSum, false>(buf, kGuessLd, avail + 1, nullptr, false, min(R, kNT));
        } else {
            double acc[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
            for (int r = tid; r < R; r += kNT) {
                const double gv = a.g[r0 + r];
                acc[0] += gv * gv;
                if (avail > 0) {
                    double y[6];
#pragma unroll
                    for (int j = 0; j < 6; ++j) y[j] = j < avail ? a.dh->y[j][r0 + r] : 0.0;
#pragma unroll
                    for (int q = 1; q < 7; ++q) {
                        if (q > avail) break;
                        double v = gv;
#pragma unroll
                        for (int j = 0; j < 6; ++j)
                            if (j < q) v -= a.coef[q][j] * y[j];
                        acc[q] += v * v;
                    }
                }
            }
            double* buf = reinterpret_cast<double*>(V);
#pragma unroll
            for (int q = 0; q < 7; ++q) buf[q * kGuessLd + tid] = acc[q];
            contribute<double, false>(buf, kGuessLd, avail + 1, nullptr, false, min(R, kNT));
        }
    }

    // The start: the candidate (zero or an extrapolation order) whose residual is smallest, x~ and
    // its residual w = g - S~ x~ from the stored products; the decisions of solve_begin_kernel.
    __device__ __forceinline__ bool start() {
        const int tid = thread_index();
        double* sq = reinterpret_cast<double*>(V);
        if (a.start_given) {
            if (tid == 0) {
                sh.active = a.sc->active;
                sh.guess = a.sc->guess;
                sh.bnorm = a.sc->bnorm;
                sh.tol = a.sc->tol;
                sh.nonfinite = 0;   // (recorded by the start's own kernels)
            }
            for (int r = tid; r < R; r += kNT) put_residual(r, a.w[r0 + r], sq);
        } else {
            const int avail = a.dh ? min(a.dh->avail, 6) : 0;
            candidates(avail);
            const bool there = kF32 && avail > 0 ? collect<float>(avail + 1, sh.sum) : collect<double>(avail + 1, sh.sum);
            if (!there) return false;
            if (tid == 0) {
                const double bn2 = sh.sum[0];
                sh.active = isfinite(bn2) && bn2 != 0.0 ? 1 : 0;
                sh.nonfinite = isfinite(bn2) ? 0 : 1;
                int guess = 0;
                for (int q = 1; q <= avail; ++q)
                    if (isfinite(sh.sum[q]) && sh.sum[q] < sh.sum[guess]) guess = q;
                sh.guess = sh.active ? guess : 0;
                sh.bnorm = sh.active ? sqrt(bn2) : 0.0;
                sh.tol = a.rtol * sh.bnorm;
            }
            __syncthreads();
            const int q = sh.guess;
            for (int r = tid; r < R; r += kNT) {
                double ax = 0.0, aw = a.g[r0 + r];
                if (q > 0) {
                    const double* c = a.coef[q];
                    ax = a.dh->x[0][r0 + r];
                    const double x0 = ax;
                    ax += (c[0] - 1.0) * x0;
                    aw += (-c[0]) * a.dh->y[0][r0 + r];
                    for (int j = 1; j < q; ++j) {
                        ax += c[j] * a.dh->x[j][r0 + r];
                        aw += (-c[j]) * a.dh->y[j][r0 + r];
                    }
                }
                a.xt[r0 + r] = ax;
                put_residual(r, aw, sq);
            }
        }
        contribute<double, false>(sq, 0, 1, nullptr, false, R);
        return collect<double>(1, sh.sum);
    }

    // x (and y) -= their multiples of the first nv basis vectors, rows rb + u kNT of a thread at a time
    template <bool TWO>
    __device__ __forceinline__ void subtract(int rb, int nv, const T* hx, const T* hy, T* x, T* y) {
        for (int k = 0; k < nv; ++k) {
            const T h = hx[k], c = TWO ? hy[k] : T(0);
            const T* Vk = V + k * ld;
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                const T v = Vk[min(rb + u * kNT, R - 1)];
                x[u] -= h * v;
                if constexpr (TWO) y[u] -= c * v;
            }
        }
    }

    // w1 = z - V h1 into dst, nv basis vectors
    __device__ __forceinline__ void first_pass(int tid, int nv, T* dst, bool pub) {
        for (int rb = tid; rb < R; rb += kRows * kNT) {
            T x[kRows];
#pragma unroll
            for (int u = 0; u < kRows; ++u) x[u] = z[min(rb + u * kNT, R - 1)];
            subtract<false>(rb, nv, h1t, nullptr, x, nullptr);
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                const int r = rb + u * kNT;
                if (r < R) {
                    dst[r] = x[u];
                    if (pub) publish(r, x[u]);
                }
            }
        }
    }

    // the second pass' exchange over nv basis vectors and w1 (once: its norm alone, h2 = 0)
    __device__ __forceinline__ bool second_dots(int nv, const T* w1) {
        contribute<T, true>(V, ld, a.twice ? nv : 0, w1, true, R);
        if (!collect<T>(a.twice ? nv + 1 : 1, sh.h2, h2t, sh.pair)) return false;
        if (!a.twice) {
            const int tid = thread_index();
            if (tid >= 1 && tid <= nv) {
                sh.h2[tid] = 0.0;
                h2t[tid] = T(0);
                sh.pair[tid] = PairSum{0.f, 0.f};
            }
            __syncthreads();
        }
        return true;
    }

    // 1 / sqrt(||w1||^2 - ||h2||^2) rounded to FP32, from the FP32 pairs: one Newton step on the hardware's
    // reciprocal square root with the residual formed exactly (every warp, FP32 pipes alone).  Over 4e6
    // norms in [1e-7, 2], starts two units off: at most 0.50000001 units from exact (FP64 root and
    // quotient rounded once: 0.49999999), the same value in all but one.
    __device__ __forceinline__ float inverse_norm(int lane, int nv) {
        PairSum q{0.f, 0.f};
        if (lane < nv) {
            const PairSum h = sh.pair[1 + lane];
            float p, e;
            two_prod(h.hi, h.hi, p, e);
            q.hi = p;
            q.lo = __fmaf_rn(2.f * h.hi, h.lo, e);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q = add(q, shfl_xor(q, o));
        const PairSum s = add(sh.pair[0], PairSum{-q.hi, -q.lo});
        const float y = rsqrtf(s.hi);
        float p, e, u, d;
        two_prod(y, y, p, e);          // y^2 = p + e
        two_prod(s.hi, p, u, d);       // s y^2 = u + d + s e + lo p
        const float res = __fsub_rn(1.f, u) - (d + __fmaf_rn(s.hi, e, s.lo * p));
        return __fmaf_rn(0.5f * y, res, y);
    }

    // One restart cycle of FP32 Gram-Schmidt in place from the residual w of norm beta; its columns, or
    // -1 when a wait ran out.  The control warps work on step j - 1 while step j's product is formed.
    __device__ __forceinline__ int cycle_in_place(double beta) {
        if (thread_index() == 0) sh.inv_beta = 1.0 / beta;
        __syncthreads();
        abuf ^= 1u;
        for (int r = thread_index(); r < R; r += kNT) {
            const T v = from_f64<T>(a.w[r0 + r] * sh.inv_beta);
            V[r] = v;
            publish(r, v);
        }
        unsigned tag = epoch;
        __syncthreads();
        for (int j = 0;; ++j) {
            const int tid = thread_index();
            if (tid >= 32 * kCtlWarps) product(tid - 32 * kCtlWarps, a_buffer(), tag, V + j * ld);
            else if (j > 0) control(j - 1);
            __syncthreads();
            mark(0);
            if (sh.gave_up) return -1;   // (the next wait follows contribute's barriers)
            if (j > 0 && sh.done) return j;
            contribute<T, true>(V, ld, j + 1, z, false, R);
            if (!collect<T>(j + 1, sh.h1, h1t)) return -1;
            first_pass(tid, j + 1, z, false);
            if (!second_dots(j + 1, z)) return -1;
            mark(1);
            if (j == a.m - 1) {
                if (tid < 32 * kCtlWarps) control(j);
                __syncthreads();
                return a.m;
            }
            const T inv = inverse_norm(tid & 31, j + 1);   // v = (w1 - V h2) / hn
            abuf ^= 1u;
            tag = epoch;
            T* Vn = V + (j + 1) * ld;
            for (int rb = tid; rb < R; rb += kRows * kNT) {
                T x[kRows];
#pragma unroll
                for (int u = 0; u < kRows; ++u) x[u] = z[min(rb + u * kNT, R - 1)];
                subtract<false>(rb, j + 1, h2t + 1, nullptr, x, nullptr);
#pragma unroll
                for (int u = 0; u < kRows; ++u) {
                    const int r = rb + u * kNT;
                    if (r < R) {
                        const T v = x[u] * inv;
                        Vn[r] = v;
                        publish(r, v);
                    }
                }
            }
            __syncthreads();
            mark(1);
        }
    }

    // The same with the second pass delayed (FP64): the products are of the once-projected vectors
    __device__ __forceinline__ int cycle_delayed(double beta) {
        const T bi = from_f64<T>(1.0 / beta);
        unsigned tag = epoch - 1;   // (the residual was published before its norm's exchange began)
        for (int j = 0;; ++j) {
            const int tid = thread_index();
            if (tid >= 32 * kCtlWarps) product(tid - 32 * kCtlWarps, a_buffer(), tag, ao);
            else if (j > 0) control(j - 1);
            __syncthreads();
            mark(0);
            if (sh.gave_up) return -1;   // (the next wait follows contribute's barriers)
            if (j > 0 && sh.done) return j;
            if (j == 0) {
                for (int r = tid; r < R; r += kNT) {
                    V[r] = ao[r] * bi;
                    z[r] *= bi;
                }
            } else {
                const T inv = from_f64<T>(sh.inv_hn), cj = ct[j];
                for (int rb = tid; rb < R; rb += kRows * kNT) {
                    T x[kRows], y[kRows];
#pragma unroll
                    for (int u = 0; u < kRows; ++u) {
                        const int r = min(rb + u * kNT, R - 1);
                        x[u] = ao[r];
                        y[u] = z[r];
                    }
                    subtract<true>(rb, j, h2t + 1, ct, x, y);
#pragma unroll
                    for (int u = 0; u < kRows; ++u) {
                        const int r = rb + u * kNT;
                        x[u] *= inv;
                        if (r < R) {
                            V[j * ld + r] = x[u];
                            z[r] = (y[u] - cj * x[u]) * inv;
                        }
                    }
                }
            }
            contribute<T, true>(V, ld, j + 1, z, false, R);
            if (!collect<T>(j + 1, sh.h1, h1t)) return -1;
            tag = epoch;
            abuf ^= 1u;
            first_pass(tid, j + 1, ao, true);
            const bool there = second_dots(j + 1, ao);
            __syncthreads();   // (the next product waits without another barrier: see collect)
            if (!there) return -1;
            mark(1);
            if (j == a.m - 1) {
                if (tid < 32 * kCtlWarps) control(j);
                __syncthreads();
                return a.m;
            }
        }
    }

    __device__ __forceinline__ int cycle(double beta) {
        if constexpr (kF32) return cycle_in_place(beta);
        else return cycle_delayed(beta);
    }

    // x~ += V y, y = R^{-1} s (back substitution, lane i holding row i); x~ is published
    __device__ __forceinline__ void update(int cols) {
        const int tid = thread_index(), lane = tid & 31;
        if (tid < 32) {
            double s = lane < cols ? sh.s[lane] : 0.0;
            for (int i = cols - 1; i >= 0; --i) {
                const double y = __shfl_sync(0xffffffffu, s, i) * sh.inv_r[i];
                if (lane == 0) yt[i] = from_f64<T>(y);
                if (lane < i) s -= sh.Rr[i][lane] * y;
            }
        }
        __syncthreads();
        for (int r = tid; r < R; r += kNT) {
            T acc = T(0);
            for (int k = 0; k < cols; ++k) acc += yt[k] * V[k * ld + r];
            const double x = a.xt[r0 + r] + to_f64(acc);
            a.xt[r0 + r] = x;
            store_tagged(a.X + (r0 + r) * 2, x, epoch);
        }
    }

    // qhat = M^{-1} x~ on the own edges, and the history's newest entry
    __device__ __forceinline__ void finish() {
        const int tid = thread_index();
        __syncthreads();
        const bool store = a.dh != nullptr && !sh.nonfinite && !sh.notconv;
        for (int r = tid; r < R; r += kNT) {
            const int le = r / NF, ii = r - le * NF;
            const double* x = a.xt + r0 + (size_t)le * NF;
            const double* B = a.Minv + (size_t)(e0 + le) * NF * NF + ii;
            double out;
            if (a.minv_pairs) {
                Dot2 acc;
#pragma unroll 4
                for (int jj = 0; jj < NF; ++jj) {
                    const float2 b = __ldg(reinterpret_cast<const float2*>(B + jj * NF));
                    float xh, xl;
                    hdgdg::split(x[jj], xh, xl);
                    acc.add(b.x, b.y, xh, xl);
                }
                out = acc.value();
            } else {
                double acc = 0.0;
#pragma unroll 4
                for (int jj = 0; jj < NF; ++jj) acc += __ldg(B + jj * NF) * x[jj];
                out = acc;
            }
            a.qhat[r0 + r] = out;
            if (store) {
                a.dh->xw[r0 + r] = x[ii];
                a.dh->yw[r0 + r] = a.g[r0 + r] - a.w[r0 + r];
            }
        }
    }

    __device__ __forceinline__ void run() {
        const int tid = threadIdx.x;
        if (tid == 0) {
            sh.total = 0;
            sh.cycles = 0;
            sh.status = 0;
            sh.notconv = 0;
            sh.nonfinite = 0;
            sh.gave_up = 0;
            for (int k = 0; k < 5; ++k) sh.clk[k] = 0;
            sh.last = clock64();
        }
        for (int i = tid; i < ne * 6; i += kNT) scol[i] = a.col[(size_t)e0 * 6 + i];
        epoch = *a.epoch;   // (rewritten by block 0 only after an exchange to which every block contributed)
        __syncthreads();
        if (!start()) return;
        mark(3);
        double rn = sqrt(sh.sum[0]);
        if (tid == 0) {
            if (sh.active && !isfinite(rn)) sh.nonfinite = 1;
            sh.go = sh.active && isfinite(rn) && rn > sh.tol ? 1 : 0;
        }
        __syncthreads();
        while (sh.go) {
            const bool spent = sh.total >= a.maxit;
            __syncthreads();
            for (int i = tid; i < kSolveMaxCols * kSolveMaxCols; i += kNT) (&sh.Q[0][0])[i] = i == 0 ? 1.0 : 0.0;
            if (tid == 0) {
                sh.s[0] = rn;
                sh.done = 0;
                sh.tol_cycle = fmax(sh.tol, a.inner_rel * rn);
            }
            __syncthreads();
            const int cols = spent ? 0 : cycle(rn);
            if (cols < 0) return;
            update(cols);
            residual();
            if (!collect<double>(1, sh.sum)) return;
            const double prev = rn;
            rn = sqrt(sh.sum[0]);
            if (tid == 0) {   // the tests of cycle_end_kernel, in its order
                sh.cycles += 1;
                if (sh.status != 0 || !isfinite(rn)) {
                    sh.nonfinite = 1;
                    sh.go = 0;
                } else if (rn <= sh.tol) {
                    sh.go = 0;
                } else if (rn <= a.stagnation * sh.bnorm && rn > 0.5 * prev) {
                    sh.go = 0;
                } else if (sh.total >= a.maxit) {
                    sh.notconv = 1;
                    sh.go = 0;
                }
            }
            __syncthreads();
            mark(2);
        }
        finish();
        mark(4);
        if (blockIdx.x == 0 && tid == 0) {
            *a.epoch = epoch;
            StepStats* ss = a.ss;
            const int its = sh.active ? sh.total : 0;
            const double rel = sh.active && sh.bnorm > 0.0 ? rn / sh.bnorm : 0.0;
            ss->its += its;
            ss->last_its = its;
            ss->last_rel = rel;
            if (sh.active) ss->last_guess = sh.guess;
            ss->cycles += sh.cycles;
            if (sh.nonfinite) ss->nonfinite = 1u;
            if (sh.notconv) {
                ss->notconv = 1u;
                ss->notconv_its = sh.total;
                ss->notconv_rel = rel;
            }
            if (a.clocks) *a.clocks = SolveClocks{sh.clk[0], sh.clk[1], sh.clk[2], sh.clk[3], sh.clk[4]};
        }
    }
};

template <int NF, typename T>
__global__ void __launch_bounds__(kNT, 1) solve_kernel(const __grid_constant__ SolveArgs a) {
    extern __shared__ __align__(16) char dyn[];
    __shared__ Shared sh;
    Solver<NF, T> s(a, sh, dyn);
    s.run();
}

template <int NF, typename T>
cudaError_t solve_launch(const SolveArgs& a, cudaStream_t s) {
    const void* f = reinterpret_cast<const void*>(solve_kernel<NF, T>);
    // the kernel's limit is set to the device's, the same in every call: handles of different sizes share
    // it from several threads, between one's setting and its launch (or its graph's instantiation)
    int dev = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)sizeof(Shared) - 64);
    if (e != cudaSuccess) return e;
    SolveArgs arg = a;
    void* params[] = {&arg};
    e = cudaLaunchCooperativeKernel(f, dim3(a.plan.blocks), dim3(kNT), params, a.plan.smem, s);
    if (e != cudaSuccess) return e;
    count_launches(1);
    return cudaGetLastError();
}

template <typename T>
cudaError_t solve_dispatch(int P, const SolveArgs& a, cudaStream_t s) {
    switch (P) {
        case 2: return solve_launch<6, T>(a, s);
        case 3: return solve_launch<9, T>(a, s);
        case 4: return solve_launch<12, T>(a, s);
        case 5: return solve_launch<15, T>(a, s);
        case 6: return solve_launch<18, T>(a, s);
        case 7: return solve_launch<21, T>(a, s);
        case 8: return solve_launch<24, T>(a, s);
        case 9: return solve_launch<27, T>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace hdgdg
