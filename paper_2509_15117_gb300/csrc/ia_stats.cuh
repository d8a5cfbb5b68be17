// ia_stats.cuh -- batch statistics of the observables (ensemble step of the method).
//
// The paper turns its trajectory ensembles into complex-formation probabilities (Fig. 3, Fig. 4),
// bounce-count maps (Fig. 1c) and complex lifetime survival curves (Fig. 2). This reduction gives, per
// cell (any grouping of trajectories, e.g. one cell per system), exact integer counts and histograms
// and two floating-point sums, Sigma dE_ion and Sigma dE_ion^2, that are summed in a fixed order so a
// rerun gives the same bits:
//   pass 1: each warp takes a contiguous range of trajectories, 32 at a time. While whole rows of 32
//           belong to one cell (ensembles are laid out cell by cell), every lane keeps its own sums and
//           counts in registers; they are combined (a fixed shuffle tree) when the cell changes. A row of
//           several cells is combined in lane order within each cell (match_any + shuffles). Each warp
//           adds into its own per-cell sums in shared memory, and the block adds its warps in warp order
//           into a per-block partial;
//   pass 2: one warp per cell adds the block partials, lane k those of blocks k, k + 32, ..., then the
//           lanes by the same shuffle tree.
// Counts use integer atomics, which are exact whatever their order.
//
// What bounds it: the reads (44 B per trajectory, 185 MB and 27 us at 2^22). An FP64 instruction takes a
// sub-partition 64-76 cycles on this GPU, so adding the 32 values of a row one after the other (64 FP64
// instructions per row) took 470 us of 659 us, and the global atomics of every trajectory most of the
// rest; lane-wise sums take two FP64 instructions per row, and one atomic per count and cell change:
// 108 us (2^22 trajectories in 250 cells laid out cell by cell), 86.5 us with the rows loaded ahead.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ia_traj.cuh"
#include "../../include/ionatom.h"

namespace ia {

constexpr int STATS_BLOCK = 256;
constexpr int STATS_MAX_CELLS = 1024;
constexpr int STATS_RUN_BINS = IA_STATS_BOUNCE_BINS + IA_STATS_LIFETIME_BINS;

__device__ __forceinline__ int bounce_bin(int nb)
{
    if (nb <= 0) return 0;
    int b = 1 + (31 - __clz(nb));  // 1: one bounce, 2: 2-3, 3: 4-7, ...
    return b < IA_STATS_BOUNCE_BINS ? b : IA_STATS_BOUNCE_BINS - 1;
}

// Complex lifetime t_last - t_first in a.u. of time, two bins per octave from 2^20 a.u. (~25 ps):
// bin = floor(2 (log2 tau - 20)), from the exponent and a comparison of the mantissa with sqrt(2).
__device__ __forceinline__ int lifetime_bin(double tau)
{
    if (!(tau > 0.0)) return 0;
    const long long bits = __double_as_longlong(tau);
    const int e = (int)((bits >> 52) & 0x7ff) - 1023;
    const int half = ((bits & 0xfffffffffffffLL) >= 0x6a09e667f3bcdLL) ? 1 : 0;  // mantissa >= sqrt(2)
    int b = 2 * (e - 20) + half;
    if (b < 0) b = 0;
    if (b >= IA_STATS_LIFETIME_BINS) b = IA_STATS_LIFETIME_BINS - 1;
    return b;
}

// Counts and sums of one cell held by a warp while its rows stay in that cell.
struct CellRun {
    unsigned n, one, cx, ex;     // this lane's trajectories, single bounces, complexes, clean exits
    unsigned long long att;
    double s1, s2;
};

__device__ __forceinline__ double lane_tree(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void add64(int64_t* p, unsigned long long v) { atomicAdd((unsigned long long*)p, v); }

// Adds the run to cell c: counts to the record, sums to the warp's shared sums. h: the warp's bounce and
// lifetime histograms of the run, cleared on return.
__device__ __forceinline__ void flush_run(CellRun& r, int c, int lane, ia_stats* __restrict__ st, double* mine,
                                          unsigned* h)
{
    const unsigned n = __reduce_add_sync(0xffffffffu, r.n);
    const unsigned one = __reduce_add_sync(0xffffffffu, r.one);
    const unsigned cx = __reduce_add_sync(0xffffffffu, r.cx);
    const unsigned ex = __reduce_add_sync(0xffffffffu, r.ex);
    unsigned long long att = r.att;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) att += __shfl_xor_sync(0xffffffffu, att, o);
    const double s1 = lane_tree(r.s1), s2 = lane_tree(r.s2);
    ia_stats* s = st + c;
    __syncwarp();
    if (lane == 0) {
        if (n) add64(&s->n, n);
        if (att) add64(&s->attempts, att);
        if (cx) add64(&s->n_complex, cx);
        if (ex) add64(&s->n_status[IA_STATS_EXIT_SLOT], ex);
        if (one) add64(&s->bounce_hist[1], one);
        mine[2 * c] += s1;
        mine[2 * c + 1] += s2;
    }
    for (int k = lane; k < IA_STATS_BOUNCE_BINS + IA_STATS_LIFETIME_BINS; k += 32) {
        const unsigned v = h[k];
        if (v) {
            add64(k < IA_STATS_BOUNCE_BINS ? &s->bounce_hist[k] : &s->lifetime_hist[k - IA_STATS_BOUNCE_BINS], v);
            h[k] = 0u;
        }
    }
    __syncwarp();
    r.n = r.one = r.cx = r.ex = 0u;
    r.att = 0ull;
    r.s1 = r.s2 = 0.0;
}

// One lane's trajectory of a row.
struct StatsRow {
    int c, nb;
    uint32_t status;
    int steps, rej;
    double dE;
    double t0, t1;  // first and last bounce of a complex
};
__device__ __forceinline__ StatsRow load_row(const ObsPtrs& obs, const int32_t* __restrict__ cell, long long i,
                                             long long hi, int n_cells)
{
    StatsRow r;
    r.c = -1;
    r.nb = r.steps = r.rej = 0;
    r.status = 0u;
    r.dE = r.t0 = r.t1 = 0.0;
    if (i < hi) {
        r.c = cell ? __ldg(cell + i) : 0;
        if (r.c < 0 || r.c >= n_cells) r.c = -1;
        r.status = obs.status[i];
        r.nb = obs.n_bounce[i];
        r.steps = obs.n_steps[i];
        r.rej = obs.n_rej[i];
        r.dE = obs.dE_ion[i];
    }
    return r;
}

__device__ __forceinline__ void load_bounces(const ObsPtrs& obs, long long i, StatsRow& r)
{
    if (r.c >= 0 && r.nb >= 2) {
        r.t0 = obs.t_first[i];
        r.t1 = obs.t_last[i];
    }
}

// chunk: trajectories per warp, a multiple of 32. A warp's rows follow one another: two are loaded ahead of
// the one that is counted, and the bounce times of the next one's complexes.
__global__ void __launch_bounds__(STATS_BLOCK) k_stats_pass1(ObsPtrs obs, long long n, const int32_t* __restrict__ cell,
                                                             int n_cells, ia_stats* __restrict__ st,
                                                             double* __restrict__ partial, long long chunk)
{
    extern __shared__ double sh[];  // [warps][n_cells][2], then [warps][bins] run histograms
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int W = STATS_BLOCK / 32;
    for (int k = threadIdx.x; k < W * n_cells * 2; k += STATS_BLOCK) sh[k] = 0.0;
    unsigned* hist = reinterpret_cast<unsigned*>(sh + (size_t)W * n_cells * 2);
    for (int k = threadIdx.x; k < W * STATS_RUN_BINS; k += STATS_BLOCK) hist[k] = 0u;
    __syncthreads();
    double* mine = sh + (size_t)warp * n_cells * 2;
    unsigned* h = hist + warp * STATS_RUN_BINS;
    const long long lo = ((long long)blockIdx.x * W + warp) * chunk;
    const long long hi = lo + chunk < n ? lo + chunk : n;
    CellRun r;
    r.n = r.one = r.cx = r.ex = 0u;
    r.att = 0ull;
    r.s1 = r.s2 = 0.0;
    int cur = -1;  // cell of the run held in registers
    StatsRow n1 = load_row(obs, cell, lo + lane, hi, n_cells), n2 = load_row(obs, cell, lo + 32 + lane, hi, n_cells);
    load_bounces(obs, lo + lane, n1);
    for (long long base = lo; base < hi; base += 32) {
        const long long i = base + lane;
        const StatsRow row = n1;
        n1 = n2;
        load_bounces(obs, i + 32, n1);
        n2 = load_row(obs, cell, i + 64, hi, n_cells);
        const int c = row.c, nb = row.nb;
        const uint32_t status = row.status;
        const long long att = (long long)row.steps + (long long)row.rej;
        const double dE = row.dE;
        const int c0 = __shfl_sync(0xffffffffu, c, 0);
        const int lt = c >= 0 && nb >= 2 ? lifetime_bin(row.t1 - row.t0) : 0;
        if (__all_sync(0xffffffffu, c == c0)) {
            if (c0 < 0) continue;
            if (c0 != cur) {
                if (cur >= 0) flush_run(r, cur, lane, st, mine, h);
                cur = c0;
            }
            r.n += 1u;
            r.att += (unsigned long long)att;
            r.ex += (status & 0xffu) == 0u ? 1u : 0u;
            if (nb == 1) {
                r.one += 1u;
            } else {
                atomicAdd(h + bounce_bin(nb), 1u);
                if (nb >= 2) {
                    r.cx += 1u;
                    atomicAdd(h + IA_STATS_BOUNCE_BINS + lt, 1u);
                }
            }
            r.s1 += dE;
            r.s2 = fma(dE, dE, r.s2);
        } else {
            if (c >= 0) {
                ia_stats* s = st + c;
                add64(&s->n, 1ull);
                add64(&s->attempts, (unsigned long long)att);
                if (nb >= 2) {
                    add64(&s->n_complex, 1ull);
                    add64(&s->lifetime_hist[lt], 1ull);
                }
                add64(&s->bounce_hist[bounce_bin(nb)], 1ull);
                if ((status & 0xffu) == 0u) add64(&s->n_status[IA_STATS_EXIT_SLOT], 1ull);
            }
            // lanes with the same cell: the lowest lane adds the group's values in lane order
            const unsigned same = __match_any_sync(0xffffffffu, c);
            double s1 = 0.0, s2 = 0.0;
            unsigned m = same;
            while (m) {
                const int src = __ffs(m) - 1;
                const double v = __shfl_sync(same, dE, src);
                s1 += v;
                s2 = fma(v, v, s2);
                m &= m - 1;
            }
            if (c >= 0 && lane == __ffs(same) - 1) {
                mine[2 * c] += s1;
                mine[2 * c + 1] += s2;
            }
            __syncwarp();
        }
        if (c >= 0 && (status & 0x3fu) != 0u) {
            ia_stats* s = st + c;
#pragma unroll
            for (int b = 0; b < 6; ++b)
                if (status & (1u << b)) add64(&s->n_status[b], 1ull);
        }
    }
    if (cur >= 0) flush_run(r, cur, lane, st, mine, h);
    __syncthreads();
    for (int k = threadIdx.x; k < n_cells * 2; k += STATS_BLOCK) {
        double a = 0.0;
        for (int w = 0; w < W; ++w) a += sh[(size_t)w * n_cells * 2 + k];
        partial[(size_t)blockIdx.x * n_cells * 2 + k] = a;
    }
}

__global__ void __launch_bounds__(128) k_stats_pass2(const double* __restrict__ partial, int n_blocks, int n_cells,
                                                     ia_stats* __restrict__ st)
{
    const int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (c >= n_cells) return;
    double a = 0.0, b = 0.0;
    for (int k = lane; k < n_blocks; k += 32) {
        a += partial[(size_t)k * n_cells * 2 + 2 * c];
        b += partial[(size_t)k * n_cells * 2 + 2 * c + 1];
    }
    a = lane_tree(a);
    b = lane_tree(b);
    if (lane == 0) {
        st[c].sum_dE = a;
        st[c].sum_dE2 = b;
    }
}

}  // namespace ia
