// Léja step for irregular matrices (power-law graphs): every entry gathers a row of W_j from
// somewhere else, and the longest rows hold thousands of entries.
//
// What bounds it is the gathered rows' way from L2 and DRAM and the few instructions that a warp gets
// through while it waits, so the kernel keeps as many rows in flight as the registers allow and does
// nothing else: no staging, no barrier, no tile. A group of G lanes takes a row (16 bytes of it a lane),
// the 32 / G groups of a warp a row each, and a row's entries go twelve at a time, whole batches without a
// test per entry; the entries' lines come to L1 ahead of the warp. Each warp owns a fixed range of rows with
// an equal share of entries and rows (found by a binary search in rowptr[i] + ROW_COST i, which is its own
// prefix sum), so hub rows spread over warps of their own and the sums stay deterministic. (The TMA kernel's
// tiles hold four to six such rows, a gather4 takes about 107 cycles of an SM's TMA unit, and the entries of
// a hub row past its records go through the direct path; the register kernel waits at block barriers for
// its tile's longest row.)
// The per-row arithmetic is that of step_common.cuh in entry order: W and P are the other kernels'
// bit for bit.
// Power-law graph of 2^20 rows and 17 million entries, degree order, FP32-mixed, us a step: 40 columns,
// P-axpy, 1520 on the TMA kernel, 770 here; 80 columns, moments, 2080 and 1380. Eight rows in flight: 1000
// and 1740 (835 and 1570 with the next batch's entries held in registers); sixteen spill (826 and 1500).
// ROW_COST 4: 847 and 1527, 10: 892 and 1604. Rings of rows in shared memory (cp.async, 16 rows ahead
// across row ends) lose L1's hits on the hubs and take more instructions: 1360 and 2350.
#include <algorithm>

#include "common.cuh"
#include "index_range.h"
#include "kernels.cuh"
#include "step_common.cuh"

namespace ll {

namespace {

constexpr int ROWS_THREADS = 256;
constexpr int ROWS_AHEAD = 64;   // entries of a warp's rows on their way to L1
constexpr int ROW_COST = 7;      // a row's own cost (its epilogue and the blocks' rows) in entries

// 16-byte units of a row a lane takes (Q, 1 or 2) hold this many column pairs
template <int PREC> constexpr int rows_np(int Q) { return PREC == LL_PREC_F32_MIXED ? 2 * Q : Q; }

// P's rows: each line is used once
template <typename T>
__device__ __forceinline__ T ld_once(const T* p) {
    const float4 v = __ldcs(reinterpret_cast<const float4*>(p));
    return *reinterpret_cast<const T*>(&v);
}
template <typename T>
__device__ __forceinline__ void st_once(T* p, const T& v) {
    __stcs(reinterpret_cast<float4*>(p), *reinterpret_cast<const float4*>(&v));
}

template <int PREC, int MODE, int Q>
__global__ void __launch_bounds__(ROWS_THREADS, 2) k_leja_rows(const StepParams p) {
    using WP = typename PairT<PREC>::W;
    using PP = typename PairT<PREC>::P;
    using Raw = typename PairT<PREC>::Raw;
    constexpr int NP = rows_np<PREC>(Q);   // column pairs a lane
    constexpr int PU = NP / Q;             // column pairs of a 16-byte unit
    constexpr int MB = base_mode(MODE);
    constexpr int U = 12 / Q;              // operand rows in flight per lane
    struct __align__(16) X { WP w[PU]; };
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = p.tp;                  // lanes per row
    const int groups = 32 / G;           // rows per warp at a time
    const int grp = lane / G;
    const int gl = lane - grp * G;
    const int cp0 = gl * NP;             // the lane's first column pair
    const bool on = grp < groups;
    const int n = p.n;
    const long long ldq = p.ldw >> 1, ldvq = p.ldv >> 1, ldpq = p.ldp >> 1;
    const WP* __restrict__ win = static_cast<const WP*>(p.win);
    WP* wout = static_cast<WP*>(p.wout);
    const Raw* __restrict__ vals = static_cast<const Raw*>(p.vals);
    const WP* vblk = static_cast<const WP*>(p.v);   // (may be eout: moments)
    PP* pblk = static_cast<PP*>(p.p);
    const int* __restrict__ rowptr = p.rowptr;
    const int* __restrict__ colind = p.colind;
    const StepScalars<PREC> S0(p, cp0), S1(p, cp0 + NP - 1);
    TracePart T[NP];
    bool has[Q];   // the lane's units that lie in the row
#pragma unroll
    for (int z = 0; z < Q; ++z) has[z] = on && cp0 + z * PU < ldq;
    int col[Q];   // (a unit past the row's end reads the first, for nothing: no test at each load)
#pragma unroll
    for (int z = 0; z < Q; ++z) col[z] = has[z] ? cp0 + z * PU : 0;
    auto load = [&](X (&x)[Q], const WP* row) {
#pragma unroll
        for (int z = 0; z < Q; ++z) x[z] = *reinterpret_cast<const X*>(row + col[z]);
    };

    const int nnz = rowptr[n];
    const long long total = (long long)nnz + (long long)ROW_COST * n;
    const long long nw = (long long)gridDim.x * (ROWS_THREADS / 32);
    const long long w = (long long)blockIdx.x * (ROWS_THREADS / 32) + warp;
    // (the quotient taken first keeps the products in range)
    const long long quo = total / nw, rem = total - quo * nw;
    const int r0 = rows_start(rowptr, n, ROW_COST, w * quo + min(w, rem));
    const int r1 = w + 1 == nw ? n : rows_start(rowptr, n, ROW_COST, (w + 1) * quo + min(w + 1, rem));

    // (the bounds of the next row and of the one after it are there before they are needed)
    int r = step_to(r0, grp, r1);
    auto bounds = [&](int row, int& a, int& b) {
        a = b = 0;
        if (on && row < r1) {
            a = rowptr[row];
            b = rowptr[row + 1];
        }
    };
    int k0, k1, m0, m1;
    bounds(r, k0, k1);
    bounds(step_to(r, groups, r1), m0, m1);
    while (on && r < r1) {
        int z0, z1;
        bounds(step_to(r, 2 * groups, r1), z0, z1);
        X wr[Q] = {}, vr[Q] = {}, v2r[Q] = {};
        PP po[NP] = {}, pn[NP];
        load(wr, win + (size_t)r * ldq);
        if constexpr (MB == MODE_ACCUM) {
            if (!p.first) {
#pragma unroll
                for (int y = 0; y < NP; ++y)
                    po[y] = ld_once(pblk + (size_t)r * ldpq + col[y / PU] + y % PU);
            }
        }
        if constexpr (mom_mode(MODE)) {
            if (!p.first) load(vr, vblk + (size_t)r * ldvq);
        } else if constexpr (MB == MODE_DOT || MB == MODE_ADJ) {
            load(vr, vblk + (size_t)r * ldvq);
        }
        if constexpr (MB == MODE_ADJ && PREC != LL_PREC_F32_MIXED) {
            if (p.v2) load(v2r, static_cast<const WP*>(p.v2) + (size_t)r * ldq);
        }
        RowAcc A[NP];
        for (int k = k0; k < k1; k = step_to(k, U, k1)) {
            X x[U][Q];
            Raw av[U];
            const int left = k1 - k;
            const bool full = left >= U;
            if (full) {
#pragma unroll
                for (int u = 0; u < U; ++u) av[u] = __ldg(vals + k + u);
#pragma unroll
                for (int u = 0; u < U; ++u) load(x[u], win + (size_t)__ldg(colind + k + u) * ldq);
            } else {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (u < left) {
                        av[u] = __ldg(vals + k + u);
                        load(x[u], win + (size_t)__ldg(colind + k + u) * ldq);
                    }
                }
            }
            const int pf = step_to(k, ROWS_AHEAD, nnz - 1);
            asm volatile("prefetch.global.L1 [%0];" ::"l"(colind + pf));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(vals + pf));
            if (full) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const auto ex = expand(av[u]);
#pragma unroll
                    for (int y = 0; y < NP; ++y) row_mac<PREC>(A[y], ex, x[u][y / PU].w[y % PU]);
                }
            } else {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (u < left) {
                        const auto ex = expand(av[u]);
#pragma unroll
                        for (int y = 0; y < NP; ++y) row_mac<PREC>(A[y], ex, x[u][y / PU].w[y % PU]);
                    }
                }
            }
        }
        X wn[Q], en[Q];
#pragma unroll
        for (int y = 0; y < NP; ++y)
            if (has[y / PU])
                row_epilogue<PREC, MODE>(p, y < NP / 2 || NP == 1 ? S0 : S1, A[y], wr[y / PU].w[y % PU], vr[y / PU].w[y % PU], po[y],
                                         &wn[y / PU].w[y % PU], &pn[y], T[y], v2r[y / PU].w[y % PU], &en[y / PU].w[y % PU]);
#pragma unroll
        for (int z = 0; z < Q; ++z)
            if (has[z]) *reinterpret_cast<X*>(wout + (size_t)r * ldq + cp0 + z * PU) = wn[z];
        if constexpr (mom_mode(MODE)) {
#pragma unroll
            for (int z = 0; z < Q; ++z)
                if (has[z]) *reinterpret_cast<X*>(static_cast<WP*>(p.eout) + (size_t)r * ldq + cp0 + z * PU) = en[z];
        }
        if constexpr (MB == MODE_ACCUM) {
#pragma unroll
            for (int y = 0; y < NP; ++y)
                if (has[y / PU]) st_once(pblk + (size_t)r * ldpq + cp0 + y, pn[y]);
        }
        r = step_to(r, groups, r1);
        k0 = m0;
        k1 = m1;
        m0 = z0;
        m1 = z1;
    }
    if constexpr (MB == MODE_DOT) {
        __syncwarp();
        __shared__ bool s_last;
        // row lane warp * groups + grp, column group gl
        const int slot = on ? (warp * groups + grp) * G + gl : -1;
        trace_reduce<PREC, MODE, NP>(p, T, reinterpret_cast<double*>(smem), G, (ROWS_THREADS / 32) * groups, &s_last, slot);
    }
}

template <int PREC, int MODE, int Q>
cudaError_t rows_typed(const StepLaunch& L, const StepParams& p, bool run, int* per_sm, cudaStream_t s) {
    if (!run) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_leja_rows<PREC, MODE, Q>, ROWS_THREADS, L.smem);
    k_leja_rows<PREC, MODE, Q><<<L.grid, L.threads, L.smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t rows_dispatch(int precision, int mode, int q, const StepLaunch& L, const StepParams& p, bool run, int* per_sm, cudaStream_t s) {
    if (q < 1 || q > 2) return cudaErrorInvalidValue;
    switch ((precision * NUM_MODES + mode) * 2 + q - 1) {
#define RUN(P_, M_)                                                                                           \
    case (P_ * NUM_MODES + M_) * 2: return rows_typed<P_, M_, 1>(L, p, run, per_sm, s);                        \
    case (P_ * NUM_MODES + M_) * 2 + 1: return rows_typed<P_, M_, 2>(L, p, run, per_sm, s);
#define RUN5(P_) RUN(P_, MODE_PLAIN) RUN(P_, MODE_ACCUM) RUN(P_, MODE_DOT) RUN(P_, MODE_DOT_MOM) RUN(P_, MODE_ADJ)
        RUN5(LL_PREC_F64) RUN5(LL_PREC_DF64) RUN5(LL_PREC_F32_MIXED)
#undef RUN5
#undef RUN
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool plan_step_rows(int precision, int mode, int n, int b, StepParams& p, StepLaunch& L, int sm_count) {
    L = StepLaunch{};
    if (n < 1 || b < 1 || stop_mode(mode) || sweep_mode(mode) || grad_mode(mode)) return false;
    const int pu = precision == LL_PREC_F32_MIXED ? 2 : 1;   // column pairs of 16 bytes
    // 16-byte accesses: whole units in every row (FP32: leading dimensions of a multiple of four)
    if (p.ldw % (2 * pu) != 0) return false;
    if (base_mode(mode) == MODE_ACCUM && (p.ldp % 2 != 0 || p.ldp < p.ldw)) return false;
    if ((base_mode(mode) == MODE_DOT || base_mode(mode) == MODE_ADJ) && p.ldv != p.ldw) return false;
    // one unit a lane, or two where that leaves fewer lanes of a warp without work (three rows of nine
    // lanes instead of one of seventeen)
    const int units = (b + 2 * pu - 1) / (2 * pu);
    int best = 0;
    double use = 0.0;
    for (int q = 1; q <= 2; ++q) {
        const int g = (units + q - 1) / q;
        if (g > 32) continue;
        if (base_mode(mode) == MODE_ADJ && pu * q > 2) continue;   // (two sets of per-column coefficients a lane)
        const double u = (double)(32 / g) * units / (32.0 * q);
        if (u > 1.1 * use) {
            use = u;
            best = q;
        }
    }
    if (best == 0) return false;
    const int np = pu * best;
    const int G = (units + best - 1) / best;
    p.tp = G;
    p.rl = (ROWS_THREADS / 32) * (32 / G);
    p.rpt = best;
    p.b = b;
    p.n = n;
    p.num_tiles = 1;
    L.threads = ROWS_THREADS;
    L.smem = base_mode(mode) == MODE_DOT ? (size_t)ROWS_THREADS * 2 * np * sizeof(double) : 0;
    int per_sm = 0;
    if (rows_dispatch(precision, mode, best, L, p, false, &per_sm, nullptr) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return false;
    }
    L.grid = (int)std::min<long long>((long long)per_sm * sm_count, ((long long)n + p.rl - 1) / p.rl);
    return true;
}

cudaError_t launch_step_rows(int precision, int mode, const StepLaunch& L, const StepParams& p, cudaStream_t s) {
    return rows_dispatch(precision, mode, p.rpt, L, p, true, nullptr, s);
}

}  // namespace ll
