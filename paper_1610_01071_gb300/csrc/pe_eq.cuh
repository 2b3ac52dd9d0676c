// Equal-weight loading on a bounded grid (shared by the moment and phase-space loaders):
// the cumulative-mass table of a nodal density profile that is linear inside each of the
// ncell - 1 cells between the walls, the position of the point of quantile (i + 1/2) / n, and
// the storage order of the points.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pe_common.cuh"

namespace pe {

// Scratch of the equal-weight loading: cumulative cell masses and first particle of each
// cell. Layout in the caller's scratch: double C[ncl + 1], int64 first[ncl + 1], double MoN,
// int32 mono.
struct EqTable {
    const double* C;
    const long long* first;
    const double* MoN;
    const int* mono;  // nonzero: positive finite mass, no cell of negative mass (first ascends)
};

constexpr int kEqThreads = 1024;                        // summands of the scan below
constexpr int kEqCluster = 8;                           // ... spread over the blocks of one cluster
constexpr int kEqBlock = kEqThreads / kEqCluster;
static_assert(kEqThreads == 32 * 32, "one warp scans the warps' totals");

// One cluster: cell masses m_c = (n_c f_c + n_{c+1} f_{c+1}) / 2 of the linear profile over
// the ncl = ncell - 1 cells between the walls (f = wall_factor on the wall nodes, 1 inside),
// their cumulative sums C (each thread sums a contiguous run of cells, then an exclusive scan
// of the run totals in a fixed order), M = C[ncl], MoN = M / n and
// first[c] = ceil(C_c n / M - 1/2), the first particle i with (i + 1/2) M / n >= C_c.
// TP: the profile's type (FP32 profiles of the lifting, FP64 ones of the phase-space loader).
// Bound by FP64 issue (64 to 76 cycles per warp instruction on each scheduler): the same 1024
// threads as one block took 36 us at 8192 cells, over eight SMs 11.5 us. The sums and their order
// are those of the one block.
template <typename TP>
__global__ void __cluster_dims__(kEqCluster, 1, 1) __launch_bounds__(kEqBlock)
    k_eq_table(const TP* __restrict__ prof_n, int ncell, float wall_factor, int64_t n, double* C, long long* first,
               double* MoN, int* mono, uint32_t* status)
{
    namespace cg = cooperative_groups;
    __shared__ double part[32];  // totals of all 32 warps of the cluster
    __shared__ double mass;
    __shared__ int rising[kEqCluster];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int ncl = ncell - 1;
    const int per = (ncl + kEqThreads - 1) / kEqThreads;
    const int t = rank * kEqBlock + threadIdx.x;
    const int c0 = t * per, c1 = (c0 + per < ncl) ? c0 + per : ncl;
    auto dens = [&](int j) {
        const double v = (double)prof_n[j];
        return (j == 0 || j == ncell - 1) ? v * (double)wall_factor : v;
    };
    double run = 0.0;
    bool neg = false;
    if (c0 < c1) {
        double d0 = dens(c0);
        for (int c = c0; c < c1; ++c) {
            const double d1 = dens(c + 1), m = 0.5 * (d0 + d1);
            run += m;
            neg |= __double2hiint(m) < 0;
            d0 = d1;
        }
    }
    // exclusive scan of the run totals: within each warp by shuffles, then over the warps' totals
    // (fixed order), which every warp scans itself
    const int lane = t & 31, wid = t >> 5;
    double incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    cluster.sync();  // every block has started
    const double tot = __shfl_sync(0xffffffffu, incl, 31);
    if (lane < kEqCluster) *cluster.map_shared_rank(&part[wid], lane) = tot;
    const int up = __syncthreads_and(!neg);
    if (threadIdx.x == 0) *cluster.map_shared_rank(&rising[rank], 0) = up;
    cluster.sync();
    double ws = part[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, ws, o);
        if (lane >= o) ws += y;
    }
    const double before = __shfl_sync(0xffffffffu, ws, wid > 0 ? wid - 1 : 0);
    const double begin = (wid > 0 ? before : 0.0) + incl - run;
    double acc = begin;
    if (c0 < c1) {
        double d0 = dens(c0);
        for (int c = c0; c < c1; ++c) {
            C[c] = acc;
            const double d1 = dens(c + 1);
            acc += 0.5 * (d0 + d1);
            d0 = d1;
        }
        if (c1 == ncl) {
            C[ncl] = acc;
            for (int r = 0; r < kEqCluster; ++r) *cluster.map_shared_rank(&mass, r) = acc;
        }
    }
    cluster.sync();
    const double M = mass;
    const bool ok = M > 0.0 && isfinite(M);
    if (t == 0) {
        int all = ok ? 1 : 0;
        for (int r = 0; r < kEqCluster; ++r) all &= rising[r];
        *MoN = ok ? M / (double)n : 0.0;
        *mono = all;
        if (!ok) raise_flag(status, PE_FLAG_RANGE);
    }
    const double n_M = (double)n / M;
    for (int c = c0; c < c1; ++c) {
        long long f;
        if (!ok) {
            f = (c == 0) ? 0 : n;  // no mass: every particle in cell 0 with weight 0
        } else {
            const double q = ceil(C[c] * n_M - 0.5);
            f = q < 0.0 ? 0 : (q > (double)n ? n : (long long)q);
        }
        first[c] = f;
    }
    if (c0 < c1 && c1 == ncl) first[ncl] = n;
}

// Cell of particle i: the largest c in [0, ncl) with first[c] <= i (binary search; always
// in range whatever the table holds).
__device__ __forceinline__ int eq_cell_of(const EqTable& tab, int ncell, long long i)
{
    int lo = 0, hi = ncell - 1;  // first[lo] <= i < first[hi] on a valid table
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(tab.first + mid) <= i) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Constants of a cell: the point's share of its cell's mass, r = ((i + 1/2) M/n - C_c) / m_c, is
// a + (i - first_c) s with a = ((first_c + 1/2) M/n - C_c) / m_c and s = (M/n) / m_c, formed in
// FP64 and applied in FP32 (r within ~1e-7 of the FP64 quotient); sig is the relative slope of the
// cell's linear density.
struct EqCell {
    uint32_t first;
    float a, s, sig;
};

template <typename TP>
__device__ __forceinline__ EqCell eq_cell(const EqTable& tab, const TP* __restrict__ prof, float wall_factor,
                                          int ncell, int c)
{
    const double C0 = __ldg(tab.C + c), C1 = __ldg(tab.C + c + 1);
    const double MoN = __ldg(tab.MoN);
    const double mc = C1 - C0;
    const long long i0 = __ldg(tab.first + c);
    EqCell k;
    k.first = (uint32_t)i0;
    if (mc > 0.0) {
        k.a = (float)((((double)i0 + 0.5) * MoN - C0) / mc);
        k.s = (float)(MoN / mc);
    } else {
        k.a = 0.5f;
        k.s = 0.0f;
    }
    float n0 = (float)__ldg(prof + c), n1 = (float)__ldg(prof + c + 1);
    if (c == 0) n0 *= wall_factor;
    if (c + 1 == ncell - 1) n1 *= wall_factor;
    const float sum = n0 + n1;
    k.sig = sum > 0.0f ? (n1 - n0) / sum : 0.0f;
    return k;
}

// Storage order of the equal-weight loading: inside every full aligned block of 2^kEqBlockBits
// slots, slot s holds point i = s with its low kEqBlockBits bits reversed, so that the block's
// points (all within 2^kEqBlockBits mass quantiles of each other) are stored in ascending
// velocity quantile, as a power-of-two cell of pe_quiet_start stores its points: the 128
// slots a warp visits at once then span 1/32 of the velocity range and their co-moving
// targets stay together. The ragged tail keeps i = s. The reversal is its own inverse.
constexpr int kEqBlockBits = 12;
constexpr uint32_t kEqBlockMask = (1u << kEqBlockBits) - 1u;

__device__ __forceinline__ uint32_t eq_point_of_slot(uint32_t s, int64_t n)
{
    return ((int64_t)(s | kEqBlockMask) < n) ? ((s & ~kEqBlockMask) | (__brev(s & kEqBlockMask) >> (32 - kEqBlockBits)))
                                              : s;
}

// Cell at which the walk to the cell of slot i's point pt begins, in the global table; the slots from
// `full` on are the ragged end of a block's chunk. Where the table ascends that is the point's own
// cell. Where it does not (negative densities) several cells hold a point, and which one the walk ends
// in depends on its start: there the start belongs to the smallest point of the slot's group of four.
__device__ __forceinline__ int eq_walk_start(const EqTable& tab, int ncell, int64_t n, int64_t i, int64_t full, uint32_t pt)
{
    if (i < full && !__ldg(tab.mono))
        for (uint32_t k = 0; k < 4u; ++k) pt = min(pt, eq_point_of_slot(((uint32_t)i & ~3u) + k, n));
    return eq_cell_of(tab, ncell, pt);
}

// The cells of a thread block's points, in shared memory: constants once per cell and block (the
// storage order takes a lane back and forth between the cells of 4096 consecutive points, and
// forming the constants at each change, ~40 FP64 instructions of 64 to 76 cycles, took most of
// the loaders' time). At most kEqStageCells cells; a block whose points span more (a near vacuum
// on a large grid), or a table that does not ascend, works from the global table (n = 0).
constexpr int kEqStageCells = 512;

struct EqStage {
    const uint32_t* first;  // [n + 1] first points of the staged cells and of the cell after them
    const float4* cell;     // [n] EqCell
    int c0, n;
};

// Shared memory of a stage of up to `cells` cells (the caller's block starts it 16-byte aligned).
__host__ __device__ constexpr size_t eq_stage_bytes(int cells) { return sizeof(float4) * (size_t)cells + 4 * ((size_t)cells + 1); }
inline int eq_stage_cells(int ncell) { return ncell - 1 < kEqStageCells ? ncell - 1 : kEqStageCells; }

// Stages the cells of the points of slots [begin, end) (all threads of the block; the caller
// synchronises before the first use).
template <typename TP>
__device__ __forceinline__ EqStage eq_stage(void* smem, int cap, const EqTable& tab, const TP* __restrict__ prof,
                                            float wall_factor, int ncell, int64_t n, int64_t begin, int64_t end)
{
    EqStage st{};
    if (begin >= end || !__ldg(tab.mono)) return st;
    // a slot's point lies in its aligned block of 2^kEqBlockBits
    const int64_t last = (end - 1) | (int64_t)kEqBlockMask;
    const int c0 = eq_cell_of(tab, ncell, begin & ~(int64_t)kEqBlockMask);
    const int c1 = eq_cell_of(tab, ncell, last < n ? last : n - 1);
    if (c1 - c0 >= cap) return st;
    float4* cell = static_cast<float4*>(smem);
    uint32_t* first = reinterpret_cast<uint32_t*>(cell + cap);
    st = EqStage{first, cell, c0, c1 - c0 + 1};
    for (int k = threadIdx.x; k <= st.n; k += blockDim.x) {
        first[k] = (uint32_t)__ldg(tab.first + c0 + k);
        if (k < st.n) {
            const EqCell e = eq_cell(tab, prof, wall_factor, ncell, c0 + k);
            cell[k] = make_float4(__uint_as_float(e.first), e.a, e.s, e.sig);
        }
    }
    return st;
}

// A lane's position in the table: the cell last visited and the first point of the next one.
struct EqCursor {
    int c;  // -1 before the first point
    uint32_t next;
    EqCell k;

    __device__ __forceinline__ void reset()
    {
        c = -1;
        next = 0u;
        k = EqCell{1u, 0.0f, 0.0f, 0.0f};
    }
};

// Position of point i: its cell (the last whose first point is not above i: of the stage, or walked
// forward in the global table from c, a cell at or before the point's) into c; returns the offset
// t in [0, 1) at which the cell's linear density (the profile's two nodal values, wall nodes times
// wall_factor) holds the point's share r of the cell mass: t + sig (t^2 - t) = r.
template <typename TP>
__device__ __forceinline__ float eq_position(const EqTable& tab, const EqStage& st, const TP* __restrict__ prof,
                                             float wall_factor, int ncell, uint32_t i, int& c, EqCursor& cur)
{
    if (st.n) {
        if (cur.c < 0 || i < cur.k.first || i >= cur.next) {
            int lo = 0, hi = st.n;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (st.first[mid] <= i) lo = mid;
                else hi = mid;
            }
            const float4 e = st.cell[lo];
            cur.k = EqCell{__float_as_uint(e.x), e.y, e.z, e.w};
            cur.next = st.first[lo + 1];
            cur.c = st.c0 + lo;
        }
        c = cur.c;
    } else {
        while (c < ncell - 2 && __ldg(tab.first + c + 1) <= (long long)i) ++c;
        if (c != cur.c) {
            cur.k = eq_cell(tab, prof, wall_factor, ncell, c);
            cur.c = c;
        }
    }
    float r = fmaf((float)(i - cur.k.first), cur.k.s, cur.k.a);
    r = r < 0.0f ? 0.0f : (r > 1.0f ? 1.0f : r);
    const float sig = cur.k.sig;
    const float om = 1.0f - sig;
    const float den = om + sqrtf(fmaxf(om * om + 4.0f * sig * r, 0.0f));
    const float t = den > 0.0f ? 2.0f * r / den : 0.0f;
    return fminf(fmaxf(t, 0.0f), 0.99999994f);  // stay inside the cell (largest float below 1)
}

}  // namespace pe
