// Two-point 1-Wasserstein distances between the laws of two ensembles on the restriction
// grid: W_{1,2}^v of Eq. (W1_vector) / Algorithm "WassersteinDistance2_vector" (atoms
// (u(x_i), u(x_j)) in R^6) and the component-wise W_{1,2} of Algorithm
// "WassersteinDistance2" (atoms (u_c(x_i), u_c(x_j)) in R^2 for each component c), with
// the Euclidean ground metric, for every point pair i <= j; pairs with i != j count twice
// and the sum is divided by G^2.
//
// Each pair (and component) is one exact optimal-transport problem between two uniform
// empirical measures of M_A and M_B atoms.  Costs are the Euclidean distances of the FP32 atoms
// (taken relative to the atoms' mean) in fixed point (2^40 units for the largest possible cost),
// so that potentials and reduced costs are exact integers and the plan found is optimal for those
// costs; the distance of the problem is then the FP64 cost of that plan, recomputed from the FP64
// atoms.  Two solvers:
//
//  - L = lcm(M_A, M_B) <= 256: repeating every atom of A L / M_A times and every atom of B L / M_B
//    times gives uniform weights 1/L on both sides without changing the optimum, and an optimal
//    plan is then a permutation: one warp solves the L x L assignment problem with the
//    shortest-augmenting-path (Hungarian) method after a column reduction, each lane owning up to
//    eight columns.  Unequal counts whose repetition makes the problem much larger are left to the
//    second solver (match_serves).
//  - otherwise (M_A, M_B <= 1024): one block solves the transportation problem directly, with
//    g = gcd(M_A, M_B), integer supply M_B / g at every atom of A and demand M_A / g at every atom
//    of B (the plan pi = x / (M_A M_B / g)), by successive shortest paths: rows (atoms of A) are
//    inserted one at a time, and each insertion ships the row's supply along shortest paths of
//    reduced costs (Dijkstra over the columns, with the rows that ship to a reached column reached
//    through its flow at no reduced cost), updating the potentials after each path.  Equal sample
//    counts are assignment problems again (supply and demand 1): the matching is kept in shared
//    memory.  Otherwise the integer flows x_ij (at most min(supply, demand) <= 1024, 16 bits) are
//    kept in a column-major matrix in the work buffer, one per block in flight.
#include <math_constants.h>

#include <cmath>
#include <string>

#include "internal.h"

namespace mclbm {

namespace {

constexpr int kPairMaxL = 256;  // largest assignment of the warp kernel (eight columns per lane)
constexpr int kPairWarps = 4;   // warps (problems in flight) per block
constexpr long long kInf = 0x3fffffffffffffffLL;
constexpr double kCostMax = 1.8e19;  // whose square still is a finite FP32 number

struct PairProblem {
    int i, j, c;  // point pair (i <= j) and component (vector problems: c = 0)
};

// Pair k of the row-major upper triangle of G x G: row start s(i) = i (2G - i + 1) / 2.
__device__ __forceinline__ void pair_of(int64_t k, int G, int& i, int& j)
{
    const double b = 2.0 * G + 1.0;
    int r = (int)floor((b - sqrt(b * b - 8.0 * (double)k)) * 0.5);
    auto start = [G](int64_t t) { return t * (2 * (int64_t)G - t + 1) / 2; };
    if (r < 0) r = 0;
    if (r > G - 1) r = G - 1;
    while (r > 0 && start(r) > k) --r;
    while (r < G - 1 && start(r + 1) <= k) ++r;
    i = r;
    j = r + (int)(k - start(r));
}

// Atom of sample m for the problem in FP64: K = 6 (vector) or 2 (component c).
template <int K>
__device__ __forceinline__ void atom64(const double* U, int G, int m, const PairProblem& pb, double (&x)[K])
{
    if constexpr (K == 6) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            x[d] = U[((int64_t)m * G + pb.i) * 3 + d];
            x[3 + d] = U[((int64_t)m * G + pb.j) * 3 + d];
        }
    } else {
        x[0] = U[((int64_t)m * G + pb.i) * 3 + pb.c];
        x[1] = U[((int64_t)m * G + pb.j) * 3 + pb.c];
    }
}

template <int K>
__device__ __forceinline__ double cost64(const double* A, const double* B, int G, int ma, int mb, const PairProblem& pb)
{
    double s = 0.0;
    if constexpr (K == 6) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double e1 = A[((int64_t)ma * G + pb.i) * 3 + d] - B[((int64_t)mb * G + pb.i) * 3 + d];
            const double e2 = A[((int64_t)ma * G + pb.j) * 3 + d] - B[((int64_t)mb * G + pb.j) * 3 + d];
            s += e1 * e1 + e2 * e2;
        }
    } else {
        const double e1 = A[((int64_t)ma * G + pb.i) * 3 + pb.c] - B[((int64_t)mb * G + pb.i) * 3 + pb.c];
        const double e2 = A[((int64_t)ma * G + pb.j) * 3 + pb.c] - B[((int64_t)mb * G + pb.j) * 3 + pb.c];
        s = e1 * e1 + e2 * e2;
    }
    return sqrt(s);
}

template <int K>
__device__ __forceinline__ float dist2(const float (&x)[K], const float (&y)[K])
{
    float s = 0.f;
#pragma unroll
    for (int d = 0; d < K; ++d) {
        const float e = x[d] - y[d];
        s = fmaf(e, e, s);
    }
    return s;
}

template <int K>
__device__ __forceinline__ long long qcost(const float (&x)[K], const float (&y)[K], float scale)
{
    return __float2ll_rn(sqrtf(dist2<K>(x, y)) * scale);
}

// The fixed-point cost as qcost forms it, without the 64-bit conversion (16 results per SM and clock
// at best): the float is split at 2^20 by adding and subtracting 1.5 2^23, which rounds to nearest in
// the low mantissa bits; the high part is exact and even, so the sum rounds as the whole would.
template <int K>
__device__ __forceinline__ long long qcost_split(const float (&x)[K], const float (&y)[K], float scale)
{
    const float c = sqrtf(dist2<K>(x, y)) * scale;
    constexpr float kMagic = 12582912.0f;  // 1.5 2^23
    constexpr int kMagicBits = 0x4B400000;
    const float h = __fmaf_rn(c, 9.5367431640625e-7f, kMagic);
    const float r = __fmaf_rn(__fsub_rn(h, kMagic), -1048576.0f, c);
    const int hi = __float_as_int(h) - kMagicBits;
    const int lo = __float_as_int(__fadd_rn(r, kMagic)) - kMagicBits;
    return (long long)hi * 1048576 + lo;
}

// One assignment problem of L atoms per side per warp, by shortest augmenting paths: rows are
// inserted one at a time along a shortest path of reduced costs (Dijkstra over the columns), then the
// potentials of the scanned columns and their rows are updated.  Lane l owns the columns l + 32 c,
// c < CPL: atom, potential, distance and predecessor row in registers.  Shared memory per warp: the
// rows (atom and potential, one or two 16-byte words), and the matchings and predecessors as 16-bit
// indices.  A scan costs about 45 instructions per column of a lane and two warp-wide minima
// (redux.sync over the halves of the 64-bit distance), with no barrier; the kernel is bound by their
// issue and latency, so problems in flight are what counts: one warp each instead of a block of 256
// threads with five barriers per scan.  On the 8^3 grid (131,328 problems), vector / component-wise,
// against a block per problem: M = 100 487 / 1506 -> 28.5 / 92 ms, M_A, M_B = 100, 50 455 / 1453 ->
// 40.5 / 117 ms, M = 128 715 / 2236 -> 44 / 143 ms; against a warp that updated every potential at
// every scan (L <= 64): M = 64 18.8 / 55 -> 8.4 / 29 ms, M = 4 1.9 / 2.6 -> 1.2 / 1.8 ms.  M = 256 on the
// 4^3 grid 28.4 / 90 -> 5.7 / 12.5 ms: the line to the block kernel is where a lane's columns no longer
// fit its registers.
template <int K>
struct __align__(16) MatchRow {
    float x[K];
    long long u;
};

__host__ __device__ inline int match_smem(int K, int L)  // bytes per warp
{
    const int row = K == 6 ? (int)sizeof(MatchRow<6>) : (int)sizeof(MatchRow<2>);
    return (row * L + 3 * 2 * L + 15) / 16 * 16;
}

template <int K, int CPL>
__global__ void __launch_bounds__(32 * kPairWarps) k_w1_match(const double* __restrict__ A, int MA,
                                                              const double* __restrict__ B, int MB, int G, int L,
                                                              int ncomp, int64_t nprob, double* __restrict__ per)
{
    extern __shared__ __align__(16) unsigned char msm[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    MatchRow<K>* row = reinterpret_cast<MatchRow<K>*>(msm + w * match_smem(K, L));
    short* rowcol = reinterpret_cast<short*>(row + L);  // column of each matched row
    short* pcol = rowcol + L;                           // row of each matched column, else -1
    short* pred = pcol + L;                             // row before a column on its shortest path
    const int ra = L / MA, rb = L / MB;                 // repetitions of each atom
    for (int64_t prob = (int64_t)blockIdx.x * kPairWarps + w; prob < nprob; prob += (int64_t)gridDim.x * kPairWarps) {
        PairProblem pb;
        pair_of(prob / ncomp, G, pb.i, pb.j);
        pb.c = (int)(prob % ncomp);
        // The costs depend on differences only: atoms are taken relative to the mean of both
        // ensembles' atoms (in FP64), so that their FP32 values resolve the spread of the
        // ensembles rather than the magnitude of the velocity.
        double cen[K];
        {
            double ca[K], cb[K];
#pragma unroll
            for (int d = 0; d < K; ++d) ca[d] = cb[d] = 0.0;
            for (int m = lane; m < MA; m += 32) {
                double x[K];
                atom64<K>(A, G, m, pb, x);
#pragma unroll
                for (int d = 0; d < K; ++d) ca[d] += x[d];
            }
            for (int m = lane; m < MB; m += 32) {
                double x[K];
                atom64<K>(B, G, m, pb, x);
#pragma unroll
                for (int d = 0; d < K; ++d) cb[d] += x[d];
            }
            const double ia = 0.5 / MA, ib = 0.5 / MB;
#pragma unroll
            for (int d = 0; d < K; ++d) {
                cen[d] = ca[d] * ia + cb[d] * ib;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) cen[d] += __shfl_xor_sync(0xffffffffu, cen[d], off);
            }
        }
        // rows: atoms of A (row r is sample r / ra); columns: atoms of B (column s is sample s / rb)
        float amax = 0.f;
        for (int r = lane; r < L; r += 32) {
            double x[K];
            atom64<K>(A, G, r / ra, pb, x);
#pragma unroll
            for (int d = 0; d < K; ++d) {
                const float f = (float)(x[d] - cen[d]);
                row[r].x[d] = f;
                amax = fmaxf(amax, fabsf(f));
            }
            row[r].u = 0;
            rowcol[r] = pcol[r] = -1;
        }
        float y[CPL][K];
        long long v[CPL], dist[CPL];
        int from[CPL];
        unsigned mine = 0;  // the lane's columns, as bits
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int col = lane + 32 * c;
#pragma unroll
            for (int d = 0; d < K; ++d) y[c][d] = 0.f;
            if (col < L) {
                mine |= 1u << c;
                double x[K];
                atom64<K>(B, G, col / rb, pb, x);
#pragma unroll
                for (int d = 0; d < K; ++d) {
                    y[c][d] = (float)(x[d] - cen[d]);
                    amax = fmaxf(amax, fabsf(y[c][d]));
                }
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        // fixed-point unit: costs are at most 2 sqrt(K) amax; 2^40 units for that bound leaves
        // room for the potentials (sums of at most L costs) in 64 bits
        const float scale = amax > 0.f ? 1099511627776.0f / (2.0f * sqrtf((float)K) * amax) : 1.0f;
        __syncwarp();
        // Column reduction: v = the column's smallest cost, and a column takes the row of that cost
        // where the row is still free (the lowest column of several).  It halves the scans at K = 6,
        // M = 100 (1104 -> 574 and 100 passes over the rows without a warp-wide minimum).
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            v[c] = kInf;
            from[c] = 0;
        }
        for (int r = 0; r < L; ++r) {
            float x[K];
#pragma unroll
            for (int d = 0; d < K; ++d) x[d] = row[r].x[d];
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const long long q = qcost_split<K>(x, y[c], scale);
                if (q < v[c]) {
                    v[c] = q;
                    from[c] = r;
                }
            }
        }
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int col = lane + 32 * c;
            const bool wants = col < L && rowcol[from[c]] < 0;
            const unsigned same = __match_any_sync(0xffffffffu, wants ? from[c] : -1 - lane);
            if (wants && __ffs(same) - 1 == lane) {
                rowcol[from[c]] = (short)col;
                pcol[col] = (short)from[c];
            }
            __syncwarp();
        }
        bool failed = false;
        for (int r0 = 0; r0 < L && !failed; ++r0) {
            if (rowcol[r0] >= 0) continue;
#pragma unroll
            for (int c = 0; c < CPL; ++c) dist[c] = kInf;
            unsigned open = mine;  // columns not yet scanned
            int i = r0, jstar = -1;
            long long dcur = 0;
            for (int guard = 0; guard <= L; ++guard) {
                float x[K];
#pragma unroll
                for (int d = 0; d < K; ++d) x[d] = row[i].x[d];
                const long long base = dcur - row[i].u;
                long long best = kInf;
                int bc = 0;
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    const long long cand = base + qcost_split<K>(x, y[c], scale) - v[c];
                    const bool is_open = (open >> c) & 1u;
                    if (is_open && cand < dist[c]) {
                        dist[c] = cand;
                        from[c] = i;
                    }
                    if (is_open && dist[c] < best) {
                        best = dist[c];
                        bc = c;
                    }
                }
                // the closest open column: minimum of the high words, then of the low words
                const unsigned hi = (unsigned)(best >> 32), lo = (unsigned)best;
                const unsigned mhi = __reduce_min_sync(0xffffffffu, hi);
                const unsigned mlo = __reduce_min_sync(0xffffffffu, hi == mhi ? lo : 0xffffffffu);
                const int wl = __ffs(__ballot_sync(0xffffffffu, hi == mhi && lo == mlo)) - 1;
                dcur = (long long)(((unsigned long long)mhi << 32) | mlo);
                if (dcur >= kInf) break;  // nothing reachable: NaN below
                const int j = 32 * __shfl_sync(0xffffffffu, bc, wl) + wl;
                i = pcol[j];
                if (i < 0) {
                    jstar = j;
                    break;
                }
                if (lane == wl) open &= ~(1u << bc);
            }
            if (jstar < 0) {
                failed = true;
                break;
            }
            // potentials: scanned columns v -= d* - d, their rows u += d* - d, and the new row u += d*
            const unsigned scanned = mine & ~open;
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int col = lane + 32 * c;
                if ((scanned >> c) & 1u) {
                    const long long delta = dcur - dist[c];
                    v[c] -= delta;
                    row[pcol[col]].u += delta;
                }
                if ((mine >> c) & 1u && ((scanned >> c) & 1u || col == jstar)) pred[col] = (short)from[c];
            }
            __syncwarp();
            if (lane == 0) {  // augment along the path back to r0 (at most L columns)
                row[r0].u += dcur;
                int j = jstar;
                for (int guard = 0; guard <= L; ++guard) {
                    const int ri = pred[j];
                    const int jn = rowcol[ri];
                    pcol[j] = (short)ri;
                    rowcol[ri] = (short)j;
                    if (ri == r0) break;
                    j = jn;
                }
            }
            __syncwarp();
        }
        // W1 of the problem: mean FP64 cost of the matched pairs; NaN if the search failed or if the plan
        // holds a pair whose cost is no finite number in FP32 (qcost_split gives such costs a finite value
        // above any other, so they are in a plan only where it cannot do without)
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int col = lane + 32 * c;
            if (col < L && pcol[col] >= 0) {
                const double d = cost64<K>(A, B, G, pcol[col] / ra, col / rb, pb);
                s += d <= kCostMax ? d : CUDART_NAN;
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) per[prob] = failed ? CUDART_NAN : s / L;
        __syncwarp();
    }
}

// ---- transportation problems beyond the warp kernel (match_serves): one block per problem -----------------
constexpr int kTpMaxM = 1024;          // atoms per side
constexpr int kTpThreads = 256;        // threads per block
constexpr int kTpWarps = kTpThreads / 32;
constexpr int kTpGeneralBlocks = 256;  // blocks in flight for unequal sample counts (one flow matrix each)

// Shared-memory layout of one block: 8-byte arrays first, then 4-byte, then bytes.
struct TpLayout {
    int u, v, dcol, drow;           // long long [MA], [MB], [MB], [MA]: potentials, distances
    int X, Y;                       // float [MA][K], [MB][K]: atoms relative to the mean
    int predc, predr, dem, pcol, newr;  // int [MB], [MA], [MB], [MB], [MA]
    int used, reached;              // unsigned char [MB], [MA]
    int red;                        // scratch: long long [kTpWarps] + int [kTpWarps] + scalars
    int total;
};

__host__ __device__ inline int tp_align(int x) { return (x + 15) & ~15; }

__host__ __device__ inline TpLayout tp_layout(int MA, int MB, int K)
{
    TpLayout L;
    int o = 0;
    L.u = o; o = tp_align(o + 8 * MA);
    L.v = o; o = tp_align(o + 8 * MB);
    L.dcol = o; o = tp_align(o + 8 * MB);
    L.drow = o; o = tp_align(o + 8 * MA);
    L.X = o; o = tp_align(o + 4 * MA * K);
    L.Y = o; o = tp_align(o + 4 * MB * K);
    L.predc = o; o = tp_align(o + 4 * MB);
    L.predr = o; o = tp_align(o + 4 * MA);
    L.dem = o; o = tp_align(o + 4 * MB);
    L.pcol = o; o = tp_align(o + 4 * MB);
    L.newr = o; o = tp_align(o + 4 * MA);
    L.used = o; o = tp_align(o + MB);
    L.reached = o; o = tp_align(o + MA);
    L.red = o; o = tp_align(o + 8 * kTpWarps * (6 + 1) + 4 * kTpWarps + 64);
    L.total = o;
    return L;
}

// Block-wide sum of one double per thread (fixed order: warp trees, then warp 0 over the warps).
__device__ __forceinline__ double tp_block_sum(double x, double* scratch)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    __syncthreads();
    if (lane == 0) scratch[w] = x;
    __syncthreads();
    double t = 0.0;
    for (int k = 0; k < kTpWarps; ++k) t += scratch[k];
    return t;
}

// Block-wide minimum of (value, index) pairs, ties to the smaller index; every thread gets it.
__device__ __forceinline__ void tp_block_argmin(long long& best, int& bj, long long* sv, int* si)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const long long ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, off);
        if (ob < best || (ob == best && oj < bj)) {
            best = ob;
            bj = oj;
        }
    }
    __syncthreads();
    if (lane == 0) {
        sv[w] = best;
        si[w] = bj;
    }
    __syncthreads();
    best = sv[0];
    bj = si[0];
    for (int k = 1; k < kTpWarps; ++k)
        if (sv[k] < best || (sv[k] == best && si[k] < bj)) {
            best = sv[k];
            bj = si[k];
        }
}

// One transportation problem per block (grid-strided over the problems).  MATCH: equal sample
// counts (supply = demand = 1), matching in shared memory; otherwise the block's flow matrix
// flowT [MB][MA] (column-major: the rows shipping to one column are contiguous).  The problem's
// value is NaN if a shortest-path search ends without reaching a column with open demand (with finite
// costs it cannot while the total supply equals the total demand; the check keeps every loop bounded).
template <int K, bool MATCH>
__global__ void __launch_bounds__(kTpThreads, 2) k_w1_transport(const double* __restrict__ A, int MA,
                                                             const double* __restrict__ B, int MB, int G, int ncomp,
                                                             int64_t nprob, int supply, int demand,
                                                             unsigned short* __restrict__ flows,
                                                             double* __restrict__ per)
{
    extern __shared__ __align__(16) unsigned char tsm[];
    const TpLayout Lo = tp_layout(MA, MB, K);
    long long* u = reinterpret_cast<long long*>(tsm + Lo.u);
    long long* v = reinterpret_cast<long long*>(tsm + Lo.v);
    long long* dcol = reinterpret_cast<long long*>(tsm + Lo.dcol);
    long long* drow = reinterpret_cast<long long*>(tsm + Lo.drow);
    float* X = reinterpret_cast<float*>(tsm + Lo.X);
    float* Y = reinterpret_cast<float*>(tsm + Lo.Y);
    int* predc = reinterpret_cast<int*>(tsm + Lo.predc);
    int* predr = reinterpret_cast<int*>(tsm + Lo.predr);
    int* dem = reinterpret_cast<int*>(tsm + Lo.dem);
    int* pcol = reinterpret_cast<int*>(tsm + Lo.pcol);
    int* newr = reinterpret_cast<int*>(tsm + Lo.newr);
    unsigned char* used = tsm + Lo.used;
    unsigned char* reached = tsm + Lo.reached;
    long long* sv = reinterpret_cast<long long*>(tsm + Lo.red);
    double* sd = reinterpret_cast<double*>(sv + kTpWarps);
    int* si = reinterpret_cast<int*>(sd + 6 * kTpWarps);
    int* s_nnew = si + kTpWarps;
    int* s_sup = s_nnew + 1;
    int* s_fail = s_sup + 1;
    const int tid = threadIdx.x;
    // each block's matrix starts on a 16-byte boundary (its zeroing writes whole 16-byte words)
    const size_t fstride = ((size_t)MA * MB + 7) / 8 * 8;
    unsigned short* flowT = MATCH ? nullptr : flows + (size_t)blockIdx.x * fstride;
    const long long total_flow = MATCH ? MA : (long long)MA * supply;

    for (int64_t prob = blockIdx.x; prob < nprob; prob += gridDim.x) {
        PairProblem pb;
        pair_of(prob / ncomp, G, pb.i, pb.j);
        pb.c = (int)(prob % ncomp);
        // atoms relative to the mean of both ensembles' atoms (FP64), as in the warp kernel
        double cen[K];
#pragma unroll
        for (int d = 0; d < K; ++d) cen[d] = 0.0;
        for (int m = tid; m < MA; m += kTpThreads) {
            double x[K];
            atom64<K>(A, G, m, pb, x);
#pragma unroll
            for (int d = 0; d < K; ++d) cen[d] += x[d] / MA;
        }
        for (int m = tid; m < MB; m += kTpThreads) {
            double x[K];
            atom64<K>(B, G, m, pb, x);
#pragma unroll
            for (int d = 0; d < K; ++d) cen[d] += x[d] / MB;
        }
#pragma unroll
        for (int d = 0; d < K; ++d) cen[d] = 0.5 * tp_block_sum(cen[d], sd + d * kTpWarps);
        float amax = 0.f;
        for (int m = tid; m < MA; m += kTpThreads) {
            double x[K];
            atom64<K>(A, G, m, pb, x);
#pragma unroll
            for (int d = 0; d < K; ++d) {
                X[m * K + d] = (float)(x[d] - cen[d]);
                amax = fmaxf(amax, fabsf(X[m * K + d]));
            }
            u[m] = 0;
        }
        for (int m = tid; m < MB; m += kTpThreads) {
            double x[K];
            atom64<K>(B, G, m, pb, x);
#pragma unroll
            for (int d = 0; d < K; ++d) {
                Y[m * K + d] = (float)(x[d] - cen[d]);
                amax = fmaxf(amax, fabsf(Y[m * K + d]));
            }
            v[m] = 0;
            dem[m] = demand;
            pcol[m] = -1;
        }
        if (!MATCH) {
            uint4* f4 = reinterpret_cast<uint4*>(flowT);
            const size_t n4 = fstride / 8;
            for (size_t k = tid; k < n4; k += kTpThreads) f4[k] = make_uint4(0, 0, 0, 0);
        }
        {
            // fixed-point unit: 2^40 for the largest possible cost 2 sqrt(K) amax
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
            __syncthreads();
            if ((tid & 31) == 0) sd[tid >> 5] = amax;
            __syncthreads();
            for (int k = 0; k < kTpWarps; ++k) amax = fmaxf(amax, (float)sd[k]);
        }
        const float scale = amax > 0.f ? 1099511627776.0f / (2.0f * sqrtf((float)K) * amax) : 1.0f;
        if (tid == 0) *s_fail = 0;
        __syncthreads();

        for (int r0 = 0; r0 < MA; ++r0) {
            if (tid == 0) *s_sup = supply;
            __syncthreads();
            // each pass ships at least one unit of the row's supply
            for (int pass = 0; pass < supply && *s_sup > 0; ++pass) {
                for (int j = tid; j < MB; j += kTpThreads) {
                    dcol[j] = kInf;
                    used[j] = 0;
                }
                for (int i = tid; i < MA; i += kTpThreads) reached[i] = 0;
                __syncthreads();
                if (tid == 0) {
                    reached[r0] = 1;
                    drow[r0] = 0;
                    newr[0] = r0;
                    *s_nnew = 1;
                }
                __syncthreads();
                long long dstar = 0;
                int jstar = -1;
                bool found = false;
                for (int it = 0; it <= MB; ++it) {
                    // relax the columns from the rows reached in the last step (ties to the
                    // smaller row, so that the tree does not depend on the order of the list)
                    const int nn = *s_nnew;
                    for (int q = 0; q < nn; ++q) {
                        const int i = newr[q];
                        const long long base = drow[i] - u[i];
                        float xi[K];
#pragma unroll
                        for (int d = 0; d < K; ++d) xi[d] = X[i * K + d];
                        for (int j = tid; j < MB; j += kTpThreads) {
                            if (used[j]) continue;
                            float yj[K];
#pragma unroll
                            for (int d = 0; d < K; ++d) yj[d] = Y[j * K + d];
                            const long long cand = base + qcost<K>(xi, yj, scale) - v[j];
                            if (cand < dcol[j] || (cand == dcol[j] && i < predc[j])) {
                                dcol[j] = cand;
                                predc[j] = i;
                            }
                        }
                    }
                    long long best = kInf;
                    int bj = 0x7fffffff;
                    for (int j = tid; j < MB; j += kTpThreads)
                        if (!used[j] && (dcol[j] < best || (dcol[j] == best && j < bj))) {
                            best = dcol[j];
                            bj = j;
                        }
                    tp_block_argmin(best, bj, sv, si);
                    if (bj >= MB || best >= kInf) break;  // nothing reachable: failure, reported below
                    jstar = bj;
                    dstar = best;
                    if (dem[jstar] > 0) {
                        found = true;
                        break;
                    }
                    __syncthreads();  // every thread has read the search state
                    if (tid == 0) {
                        used[jstar] = 1;
                        *s_nnew = 0;
                    }
                    __syncthreads();
                    // the rows that ship to jstar are reached through their flow at no reduced cost
                    if (MATCH) {
                        if (tid == 0) {
                            const int i = pcol[jstar];
                            if (i >= 0 && !reached[i]) {
                                reached[i] = 1;
                                drow[i] = dstar;
                                predr[i] = jstar;
                                newr[0] = i;
                                *s_nnew = 1;
                            }
                        }
                    } else {
                        const unsigned short* fc = flowT + (size_t)jstar * MA;
                        for (int i = tid; i < MA; i += kTpThreads)
                            if (fc[i] > 0 && !reached[i]) {
                                reached[i] = 1;
                                drow[i] = dstar;
                                predr[i] = jstar;
                                newr[atomicAdd(s_nnew, 1)] = i;
                            }
                    }
                    __syncthreads();
                }
                if (!found) {
                    if (tid == 0) {
                        *s_fail = 1;
                        *s_sup = 0;
                    }
                    __syncthreads();
                    break;
                }
                // potentials: reached rows u += d* - d(row), used columns v -= d* - d(column)
                for (int i = tid; i < MA; i += kTpThreads)
                    if (reached[i]) u[i] += dstar - drow[i];
                for (int j = tid; j < MB; j += kTpThreads)
                    if (used[j]) v[j] -= dstar - dcol[j];
                __syncthreads();
                // augment along the path back to r0 (one thread; at most min(MA, MB) + 1 steps)
                if (tid == 0) {
                    int b = *s_sup < dem[jstar] ? *s_sup : dem[jstar];
                    if (MATCH) {
                        b = 1;
                        int j = jstar;
                        for (int guard = 0; guard <= MB; ++guard) {
                            const int i = predc[j];
                            const int jp = i == r0 ? -1 : predr[i];
                            pcol[j] = i;
                            if (i == r0) break;
                            j = jp;
                        }
                    } else {
                        int j = jstar;
                        for (int guard = 0; guard <= MB; ++guard) {  // bottleneck of the reverse edges
                            const int i = predc[j];
                            if (i == r0) break;
                            const int jp = predr[i];
                            const int f = flowT[(size_t)jp * MA + i];
                            if (f < b) b = f;
                            j = jp;
                        }
                        j = jstar;
                        for (int guard = 0; guard <= MB; ++guard) {
                            const int i = predc[j];
                            flowT[(size_t)j * MA + i] += (unsigned short)b;
                            if (i == r0) break;
                            const int jp = predr[i];
                            flowT[(size_t)jp * MA + i] -= (unsigned short)b;
                            j = jp;
                        }
                    }
                    dem[jstar] -= b;
                    *s_sup -= b;
                }
                __syncthreads();
            }
        }
        // W1 of the problem: the FP64 cost of the plan, sum x_ij c_ij / (total flow)
        double s = 0.0;
        if (MATCH) {
            for (int j = tid; j < MB; j += kTpThreads)
                if (pcol[j] >= 0) s += cost64<K>(A, B, G, pcol[j], j, pb);
        } else {
            const size_t n = (size_t)MA * MB;
            for (size_t k = tid; k < n; k += kTpThreads) {
                const int f = flowT[k];
                if (f > 0) s += f * cost64<K>(A, B, G, (int)(k % MA), (int)(k / MA), pb);
            }
        }
        s = tp_block_sum(s, sd);
        if (tid == 0) per[prob] = *s_fail ? CUDART_NAN : s / (double)total_flow;
        __syncthreads();
    }
}

// Fixed-order total: per-block partial sums of w_k D_k over contiguous chunks, then one thread.
constexpr int kSumThreads = 256;
__global__ void __launch_bounds__(kSumThreads) k_pair_partials(const double* __restrict__ per, int G, int ncomp,
                                                               int64_t nprob, int64_t chunk, double* __restrict__ partial)
{
    __shared__ double sh[kSumThreads];
    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = lo + chunk < nprob ? lo + chunk : nprob;
    double acc = 0.0;
    for (int64_t t = lo + threadIdx.x; t < hi; t += kSumThreads) {
        int i, j;
        pair_of(t / ncomp, G, i, j);
        acc += (i == j ? 1.0 : 2.0) * per[t];
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = kSumThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void k_pair_total(const double* __restrict__ partial, int nparts, double scale, double* __restrict__ out)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int b = 0; b < nparts; ++b) s += partial[b];
        out[0] = s * scale;
    }
}

constexpr int kPairParts = 256;

int gcd_int(int a, int b)
{
    while (b) {
        const int t = a % b;
        a = b;
        b = t;
    }
    return a;
}

// Whether the warp kernel takes the problems (else the block solver).  Unequal counts: the repeated problem has
// c = (L / MA)(L / MB) times the entries of the MA x MB one, and equal atoms lengthen its searches, where
// the block solver repeats nothing; the warp kernel, for its part, solves seven times as many problems at
// once and takes longer for one, the more so the larger L.  Measured warp / block time (vector problems: 1,
// 36, 378, 2080 and 23,436 of them) against c and c L^2: 100, 50 (2; 2e4) 0.41, 0.48, 0.3, 0.1, -; 24, 36 (6;
// 3.1e4) 0.53, 0.74, 0.42, 0.13, 0.09; 200, 100 (2; 8e4) 0.77, 0.86, 0.52, 0.24, 0.15; 256, 128 (2; 1.3e5) 1.02,
// 1.07, 0.5, 0.25, -; 250, 50 (5; 3.1e5) 1.7, 1.7, 0.95, 0.46, 0.27; 100, 40 (10; 4e5) 2.4, 2.6, 1.3, 0.6, 0.4;
// 256, 16 (16; 1.05e6) 2.8, 2.8, 1.4, 0.7, 0.5; 10, 7 (70; 3.4e5) 3.2, 3.4, 2.5, 0.98, 0.73; 12, 11 (132; 2.3e6)
// 8.4, 9.5, 5.5, 3.0, 2.0; 16, 15 (240; 1.4e7) 20, 22, 13, 6.3, -.  Equal counts: below 0.8 throughout.
bool match_serves(int MA, int MB, int64_t L, int64_t nprob)
{
    if (L > kPairMaxL) return false;
    if (L <= 64 || MA == MB) return true;
    const int64_t copies = L / MA * (L / MB), size = copies * L * L;
    if (copies > 20 && copies > nprob / 30) return false;
    return size <= 100000 || (size <= 1200000 && size <= 750 * nprob);
}

}  // namespace

// Work buffer: per-problem values [nprob], partial sums [kPairParts] and the total, then (unequal sample counts beyond the warp kernel) one flow matrix per block in flight.
struct PairWork {
    size_t per, partial, total, flows, bytes;
};

PairWork pair_work(int MA, int MB, int G, int vector)
{
    const int64_t nprob = (int64_t)G * (G + 1) / 2 * (vector ? 1 : 3);
    PairWork w;
    w.per = 0;
    w.partial = (size_t)nprob * sizeof(double);
    w.total = w.partial + kPairParts * sizeof(double);
    w.flows = (w.total + 32 * sizeof(double) + 16 + 255) / 256 * 256;
    const int g = gcd_int(MA, MB);
    const int64_t L = (int64_t)MA / g * MB;
    const bool general = L > 64 && MA != MB;  // whichever solver the number of problems chooses
    const size_t fstride = ((size_t)MA * MB + 7) / 8 * 8;  // elements per block, as in the kernel
    w.bytes = w.flows + (general ? (size_t)kTpGeneralBlocks * fstride * sizeof(unsigned short) : 0);
    return w;
}

}  // namespace mclbm

using namespace mclbm;

extern "C" {

size_t mclbm_w1_2pt_work_bytes(int32_t MA, int32_t MB, int32_t G, int32_t vector)
{
    if (G < 1 || MA < 1 || MB < 1 || MA > kTpMaxM || MB > kTpMaxM) return 0;
    return pair_work(MA, MB, G, vector).bytes;
}

int mclbm_w1_2pt(const double* d_a, int32_t MA, const double* d_b, int32_t MB, int32_t G, int32_t vector, void* d_work,
                 size_t work_bytes, void* cuda_stream, double* W, double* d_per_pair)
{
    if (!d_a || !d_b || !d_work || !W || MA < 1 || MB < 1 || G < 1 || (vector != 0 && vector != 1))
        return set_error(MCLBM_ERR_INVALID_ARG, "bad argument");
    if (MA > kTpMaxM || MB > kTpMaxM)
        return set_error(MCLBM_ERR_SHAPE, "sample counts " + std::to_string(MA) + ", " + std::to_string(MB) +
                                              " exceed " + std::to_string(kTpMaxM) + " per ensemble");
    const int g = gcd_int(MA, MB);
    const int64_t L = (int64_t)MA / g * MB;
    const PairWork pw = pair_work(MA, MB, G, vector);
    if (work_bytes < pw.bytes)
        return set_error(MCLBM_ERR_OOM, "work buffer needs " + std::to_string(pw.bytes) + " bytes");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int ncomp = vector ? 1 : 3;
    const int64_t nprob = (int64_t)G * (G + 1) / 2 * ncomp;
    char* wb = (char*)d_work;
    double* per = d_per_pair ? d_per_pair : (double*)(wb + pw.per);
    double* partial = (double*)(wb + pw.partial);
    double* total = (double*)(wb + pw.total);
    int dev = 0, sms = 0;
    MCLBM_CUDA(cudaGetDevice(&dev));
    MCLBM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (match_serves(MA, MB, L, nprob)) {
        auto launch = [&](auto kernel, int K) -> cudaError_t {
            const int smem = kPairWarps * match_smem(K, (int)L);
            cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            int per_sm = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * kPairWarps, smem);
            if (e != cudaSuccess) return e;
            if (per_sm < 1) return cudaErrorInvalidConfiguration;
            int64_t blocks = (nprob + kPairWarps - 1) / kPairWarps;
            if (blocks > (int64_t)sms * per_sm) blocks = (int64_t)sms * per_sm;
            kernel<<<(unsigned)blocks, 32 * kPairWarps, smem, s>>>(d_a, MA, d_b, MB, G, (int)L, ncomp, nprob, per);
            return cudaGetLastError();
        };
        cudaError_t e;
        if (vector)
            e = L <= 32    ? launch(k_w1_match<6, 1>, 6)
                : L <= 64  ? launch(k_w1_match<6, 2>, 6)
                : L <= 128 ? launch(k_w1_match<6, 4>, 6)
                           : launch(k_w1_match<6, 8>, 6);
        else
            e = L <= 32    ? launch(k_w1_match<2, 1>, 2)
                : L <= 64  ? launch(k_w1_match<2, 2>, 2)
                : L <= 128 ? launch(k_w1_match<2, 4>, 2)
                           : launch(k_w1_match<2, 8>, 2);
        MCLBM_CUDA(e);
    } else {
        const bool match = MA == MB;
        const int K = vector ? 6 : 2;
        const int smem = tp_layout(MA, MB, K).total;
        const int supply = MB / g, demand = MA / g;
        unsigned short* flows = match ? nullptr : (unsigned short*)(wb + pw.flows);
        auto launch = [&](auto kernel) -> cudaError_t {
            cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            int per_sm = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kTpThreads, smem);
            if (e != cudaSuccess) return e;
            if (per_sm < 1) return cudaErrorInvalidConfiguration;
            int64_t blocks = (int64_t)sms * per_sm;
            if (!match && blocks > kTpGeneralBlocks) blocks = kTpGeneralBlocks;
            if (blocks > nprob) blocks = nprob;
            kernel<<<(unsigned)blocks, kTpThreads, smem, s>>>(d_a, MA, d_b, MB, G, ncomp, nprob, supply, demand, flows,
                                                              per);
            return cudaGetLastError();
        };
        cudaError_t e;
        if (vector)
            e = match ? launch(k_w1_transport<6, true>) : launch(k_w1_transport<6, false>);
        else
            e = match ? launch(k_w1_transport<2, true>) : launch(k_w1_transport<2, false>);
        MCLBM_CUDA(e);
    }
    const int64_t chunk = (nprob + kPairParts - 1) / kPairParts;
    k_pair_partials<<<kPairParts, kSumThreads, 0, s>>>(per, G, ncomp, nprob, chunk, partial);
    k_pair_total<<<1, 32, 0, s>>>(partial, kPairParts, 1.0 / ((double)G * G), total);
    MCLBM_CUDA(cudaGetLastError());
    MCLBM_CUDA(cudaMemcpyAsync(W, total, sizeof(double), cudaMemcpyDeviceToHost, s));
    MCLBM_CUDA(cudaStreamSynchronize(s));
    if (!std::isfinite(*W))
        return set_error(MCLBM_ERR_NONFINITE, "a transport problem has no finite value (non-finite atoms?)");
    return MCLBM_OK;
}

}  // extern "C"
