// Field solve: the nonlinear Poisson-Boltzmann equation of Section 3.3 (Eq.
// poisson2rescaled with lambda = n_0 = 1) on the nodes,
//   -(phi_{j+1} - 2 phi_j + phi_{j-1}) / dx^2 + g(phi_j) = n_j,   g = exp or 1 + phi,
// by Newton's method, followed by the centred field E_j = -(phi_{j+1} - phi_{j-1}) / (2 dx).
// Periodic grids wrap; bounded grids (Section 4.2's slab expansion) have walls at nodes 0
// and ncell-1 with phi' = 0 there (mirror ghosts phi_{-1} = phi_1, phi_{ncell} = phi_{ncell-2},
// hence E = 0 on the walls), and a wall node's density is twice its deposit (its CIC
// control volume is the half cell inside the domain).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>
#include <string.h>

#include "pe_common.cuh"
#include "pe_ctx.h"
#include "pe_internal.h"

namespace cg = cooperative_groups;

namespace pe {

// ---------------------------------------------------------------------------------
// Solver: one thread-block cluster of G blocks (G = 1 for small grids, up to 16 for large ones,
// one block per SM); block g owns the B = ncell / G nodes [g B, (g+1) B), one node per thread.
//
// What bounds it: latency. An FP64 instruction (a conversion to or from FP64 among them) holds
// its scheduler's FP64 pipe for 64-76 cycles whatever is independent around it (measured: 76
// cycles per warp instruction with one warp on each of the SM's four schedulers, 152 with two,
// 304 with four), so the time is the number of FP64 instructions per node times the warps per
// scheduler, plus the exchanges between warps and blocks. Hence
//  - FP64 only where the result needs it: the potential, its residual, exp(phi). Conversions
//    between FP32, FP64 and the fixed-point charge are integer operations (bits of the formats);
//    the convergence test runs in FP32;
//  - exp(phi) is evaluated once and then carried multiplicatively, exp(phi + x) = exp(phi) exp(x),
//    with a Taylor polynomial whose degree follows the largest update;
//  - one block barrier and one cluster barrier per linear solve: every warp solves the block's
//    and the cluster's separator systems itself instead of waiting for one warp's result. The
//    second exchange of an iteration (largest update) runs behind the FP64 update.
// One solve of a burst (two updates; the walls' about seven), the mean of 40 cold launches under ncu:
// 8.3 us on 128 nodes (15.2 before these points), 11.0 on 1024 (17.8), 13.8 on 4096 (23.4), 39 on 8192
// with walls (63).
//
// Precision: phi, exp(phi), the Newton residual and the update are FP64; the Jacobian
// correction J d = -F is solved in FP32. This is Newton's method with an inexact linear solve
// (mixed-precision iterative refinement): the FP64 residual drives the iteration, so it converges
// to the FP64 solution of the discrete equation, while the FP32 solve only bounds the final
// contraction rate (~ cond(J) 2^-24 per iteration). Bounded grids with vacuum regions have
// exp(phi) ~ 1e-6 there and cond(J) ~ 1e7: the FP32 solve still contracts, but slowly (7 Newton
// iterations instead of 2 on an 8192-node slab from a warm start); an FP64 elimination needs 3,
// but each costs several times as much.
//
// Linear solve (nested separators, scalar tridiagonal systems only): the last row of every
// warp is a separator, and the last row of every block is a separator of the cluster. Each
// warp solves its other rows (its interior) by parallel cyclic reduction with register
// shuffles, with the couplings to the two separators around it moved to two extra right-hand
// sides (x = y - g S_left - h S_right). Substituting the interiors next to a separator into
// its row leaves a scalar tridiagonal system over the separators: every warp solves the block's
// warp separators in terms of the two block separators around them, and the cyclic system of the
// cluster's block separators, whose rows every block pushes into every other block's shared
// memory before the cluster barrier.
//
// Stopping, besides max |update| < tol: J = L + diag(g'(phi)) has L symmetric with zero row sums
// and non-positive off-diagonals (periodic or mirror-wall rows), so J is an M-matrix with row
// sums g'(phi_j) and ||J^-1||_inf <= 1 / min_j g'(phi_j): the next update is at most max|F| /
// min g' in every component. Before a linear solve |F| is the FP64 residual; after one, the
// residual that the update leaves is bounded in FP32 as |r - J x| + g x^2 (1/2 + |x|) plus the
// rounding of that evaluation, which ends the usual solve after its second update without a
// third residual and reduction only to learn that it has converged. Grids below 32 nodes stop by the
// update alone: their idle lanes count as min g' = 0. One more update costs them little and leaves the
// potential at rounding instead of at the tolerance.

constexpr int kClusterMinCells = 512;   // grids at least this large use the multi-SM solver
constexpr int kClusterMax = 16;
constexpr int kNewtonMaxThreads = 512;  // nodes (threads) per block: 16 blocks cover the largest grid
constexpr int kNewtonMaxWarps = kNewtonMaxThreads / 32;

// Conversions on the integer pipe (their FP64-pipe instructions hold the pipe as long as an FMA).
// FP64 to FP32, round to nearest even; magnitudes below FP32's normal range give 0, those of
// 2^127 and above infinity.
__device__ __forceinline__ float f32_of(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t mag = hi & 0x7FFFFFFFu, sign = hi & 0x80000000u;
    uint32_t b = __funnelshift_l(lo, mag - (896u << 20), 3);
    b += ((lo & 0x1FFFFFFFu) + 0x0FFFFFFFu + (b & 1u)) >> 29;
    if (mag < 0x38100000u) b = 0u;
    if (mag >= 0x47E00000u) b = (mag > 0x7FF00000u || (mag == 0x7FF00000u && lo)) ? 0x7FC00000u : 0x7F800000u;
    return __uint_as_float(b | sign);
}

// FP32 to FP64 (exact); subnormal numbers give 0.
__device__ __forceinline__ double f64_of(float x)
{
    const uint32_t b = __float_as_uint(x), mag = b & 0x7FFFFFFFu, sign = b & 0x80000000u;
    const uint32_t hi = mag >= 0x7F800000u ? 0x7FF00000u | ((mag & 0x007FFFFFu) >> 3) : (mag >> 3) + (896u << 20);
    return mag < 0x00800000u ? 0.0 : __hiloint2double((int)(hi | sign), (int)(mag << 29));
}

// v 2^-shift, round to nearest even: the fixed-point charge as a density.
__device__ __forceinline__ double fixed_to_double(long long v, int shift)
{
    const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)u);
    const unsigned long long m = u << (lz & 63);  // the leading bit at bit 63: 53 bits and 11 below them
    const unsigned long long r = (m >> 11) + (((m & 0x7FFull) + 0x3FFull + ((m >> 11) & 1ull)) >> 11);
    // r holds the implicit bit (and may have carried into the next power of two)
    const unsigned long long bits = ((unsigned long long)(1085 - lz - shift) << 52) + r;
    return u == 0ull ? 0.0 : __longlong_as_double((long long)(bits | ((unsigned long long)v & (1ull << 63))));
}

// exp(x) for |x| <= 2^-5 by its Taylor polynomial to degree 8 (relative error < 1e-18),
// evaluated by Estrin's scheme.
__device__ __forceinline__ double exp_small(double x)
{
    const double x2 = x * x, x4 = x2 * x2;
    const double p01 = 1.0 + x, p23 = fma(x, 1.0 / 6.0, 0.5), p45 = fma(x, 1.0 / 120.0, 1.0 / 24.0),
                 p67 = fma(x, 1.0 / 5040.0, 1.0 / 720.0);
    const double lo = fma(x2, p23, p01), hi = fma(x2, p67, p45);
    return fma(x4, fma(x4, 1.0 / 40320.0, hi), lo);
}

// exp(x) for |x| <= 2^-10 to degree 4 (relative error < 1e-17).
__device__ __forceinline__ double exp_tiny(double x)
{
    const double x2 = x * x;
    return fma(x2, fma(x2, 1.0 / 24.0, fma(x, 1.0 / 6.0, 0.5)), 1.0 + x);
}

// Reciprocal of the elimination: the fast FP32 reciprocal (__fdividef, within 2 ulp for the
// diagonal magnitudes that occur here). The FP32 solve is the inexact linear solve of a Newton
// iteration whose residual is FP64, so this only changes its contraction rate.
__device__ __forceinline__ float recip(float x) { return __fdividef(1.0f, x); }

// Warp maximum / minimum of non-negative floats by their bits (a NaN counts as the largest).
__device__ __forceinline__ float warp_max_bits(uint32_t v)
{
    return __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, v));
}
__device__ __forceinline__ float warp_min_bits(float v)
{
    return __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, __float_as_uint(v)));
}

// Parallel cyclic reduction of a scalar tridiagonal system held by lanes 0 .. n-1 of the
// calling warp (n a power of two, <= 32; all 32 lanes call it; a lane without a row holds the
// identity row). Row k: a x_{k-1} + b x_k + c x_{k+1} = r (three right-hand sides r0, r1,
// r2); the chain ends at 0 and n - 1. Returns x_k for each right-hand side.
__device__ __forceinline__ void warp_chain_pcr(float a, float b, float c, float r0, float r1, float r2, int n, float& x0,
                                               float& x1, float& x2)
{
    const int k = threadIdx.x & 31;
    for (int s = 1; s < n; s <<= 1) {
        const int km = (k - s) & (n - 1), kp = (k + s) & (n - 1);
        const float am = __shfl_sync(0xFFFFFFFFu, a, km), bm = __shfl_sync(0xFFFFFFFFu, b, km);
        const float cm = __shfl_sync(0xFFFFFFFFu, c, km), q0m = __shfl_sync(0xFFFFFFFFu, r0, km);
        const float q1m = __shfl_sync(0xFFFFFFFFu, r1, km), q2m = __shfl_sync(0xFFFFFFFFu, r2, km);
        const float ap = __shfl_sync(0xFFFFFFFFu, a, kp), bp = __shfl_sync(0xFFFFFFFFu, b, kp);
        const float cp = __shfl_sync(0xFFFFFFFFu, c, kp), q0p = __shfl_sync(0xFFFFFFFFu, r0, kp);
        const float q1p = __shfl_sync(0xFFFFFFFFu, r1, kp), q2p = __shfl_sync(0xFFFFFFFFu, r2, kp);
        const float al = (k < n && k >= s) ? a * recip(bm) : 0.0f;
        const float ga = (k + s < n) ? c * recip(bp) : 0.0f;
        a = -al * am;
        c = -ga * cp;
        b = b - al * cm - ga * ap;
        r0 = r0 - al * q0m - ga * q0p;
        r1 = r1 - al * q1m - ga * q1p;
        r2 = r2 - al * q2m - ga * q2p;
    }
    const float rb = recip(b);
    x0 = r0 * rb;
    x1 = r1 * rb;
    x2 = r2 * rb;
}

// The same for a cyclic system (rows couple to (k +- 1) mod n) with one right-hand side, lane k
// holding row k mod n; returns x_{k mod n} on every lane (after the last step the remaining
// couplings reach the row itself and are folded into the diagonal).
__device__ __forceinline__ float warp_cyclic(float a, float b, float c, float r, int n)
{
    const int k = threadIdx.x & 31;
    for (int s = 1; s < n; s <<= 1) {
        const int km = (k - s) & (n - 1), kp = (k + s) & (n - 1);
        const float am = __shfl_sync(0xFFFFFFFFu, a, km), bm = __shfl_sync(0xFFFFFFFFu, b, km);
        const float cm = __shfl_sync(0xFFFFFFFFu, c, km), rm = __shfl_sync(0xFFFFFFFFu, r, km);
        const float ap = __shfl_sync(0xFFFFFFFFu, a, kp), bp = __shfl_sync(0xFFFFFFFFu, b, kp);
        const float cp = __shfl_sync(0xFFFFFFFFu, c, kp), rp = __shfl_sync(0xFFFFFFFFu, r, kp);
        const float al = a * recip(bm), ga = c * recip(bp);
        a = -al * am;
        c = -ga * cp;
        b = b - al * cm - ga * ap;
        r = r - al * rm - ga * rp;
    }
    return r * recip(a + b + c);
}

// Parallel cyclic reduction of the 32 rows held by the calling warp (one per lane; a lane
// without a row holds the identity row). Row i: a x_{i-1} + b x_i + c x_{i+1} = d, with the
// couplings to rows outside the warp already moved to the columns gc (left) and hc (right).
// On return every row is decoupled: x_i = d - gc X_left - hc X_right.
__device__ __forceinline__ void warp_pcr(float a, float b, float c, float& d, float& gc, float& hc)
{
    const int lane = threadIdx.x & 31;
    float rb = recip(b);
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const float am = __shfl_up_sync(0xFFFFFFFFu, a, s), cm = __shfl_up_sync(0xFFFFFFFFu, c, s);
        const float dm = __shfl_up_sync(0xFFFFFFFFu, d, s), gm = __shfl_up_sync(0xFFFFFFFFu, gc, s);
        const float hm = __shfl_up_sync(0xFFFFFFFFu, hc, s), rm = __shfl_up_sync(0xFFFFFFFFu, rb, s);
        const float ap = __shfl_down_sync(0xFFFFFFFFu, a, s), cp = __shfl_down_sync(0xFFFFFFFFu, c, s);
        const float dp = __shfl_down_sync(0xFFFFFFFFu, d, s), gp = __shfl_down_sync(0xFFFFFFFFu, gc, s);
        const float hp = __shfl_down_sync(0xFFFFFFFFu, hc, s), rp = __shfl_down_sync(0xFFFFFFFFu, rb, s);
        const float al = (lane >= s) ? a * rm : 0.0f;
        const float ga = (lane + s < 32) ? c * rp : 0.0f;
        a = -al * am;
        c = -ga * cp;
        b = b - al * cm - ga * ap;
        d = d - al * dm - ga * dp;
        gc = gc - al * gm - ga * gp;
        hc = hc - al * hm - ga * hp;
        rb = recip(b);
    }
    d *= rb;
    gc *= rb;
    hc *= rb;
}

// Parameters of one field solve (one realisation).
struct FieldDesc {
    long long* rho;
    double* phi;
    double* E;
    float* Ef;
    int* diag;
    uint32_t* status;
    double inv_dx2, half_inv_dx;    // 1 / dx^2, 1 / (2 dx)
    float tol;
    int shift;                      // density = rho 2^-shift
    int ncell, mode, maxit, walls;  // walls: 1 for a bounded grid
    // Newton start: phi_prev (may be null) keeps the solution before the current one; with
    // extrap the start is the linear extrapolation 2 phi - phi_prev (solves one fine step apart)
    double* phi_prev;
    int extrap;
    int clear;  // zero rho once read (the push that follows accumulates into it)
    float* Ef0;  // batch: second copy of Ef by the solve that starts a burst (the frozen field), or null
};

// A unit's (a warp's, a block's) rows as its neighbours see them: its first row and its last
// interior row in terms of the separators around it (x = y - g s_left - h s_right) and the row of
// its own separator (a, b, c, d), with its largest |F| and its smallest g'.
struct UnitRow {
    float4 first;  // y, g, h, max |F|
    float4 last;   // y, g, h, min g'
    float4 sep;    // a, b, c, d
};

// Double-buffered by iteration parity: a warp or block may write the next iteration's rows
// while another still reads these (it cannot write the one after that before every warp has
// passed the barrier in between).
struct NewtonShared {
    UnitRow warp[2][kNewtonMaxWarps];                // this block's warps
    UnitRow block[2][kClusterMax];                   // rows pushed by every block of the cluster
    float2 upd[2][kClusterMax * kNewtonMaxWarps];    // every warp's largest |update| and the bound of
                                                     // the residual it leaves
};

// An interior row y - g s_left - h s_right given the separators around it, its operations spelled out: the
// owner of a unit's first row and the left neighbour that keeps it as a halo round alike whatever the
// compiler makes of the code around them, so the halo stays bit-identical to the owner's node.
__device__ __forceinline__ float interior_row(float y, float g, float h, float s_left, float s_right)
{
    return __fmaf_rn(-h, s_right, __fmaf_rn(-g, s_left, y));
}
__device__ __forceinline__ float edge_row(const float4& f, float s_left, float s_right)
{
    return interior_row(f.x, f.y, f.z, s_left, s_right);
}

// Solver body for the realisation of this cluster: B = ncell / G nodes per block, one per thread
// (on grids below 32 nodes the block's one warp has lanes without a node).
__device__ __forceinline__ void newton_body(const FieldDesc& d, cg::cluster_group& cluster)
{
    __shared__ NewtonShared sh;
    const int G = (int)cluster.num_blocks(), g = (int)cluster.block_rank();
    const int ncell = d.ncell, mask = ncell - 1, B = ncell / G;
    const int i = threadIdx.x, lane = i & 31, w = i >> 5;
    const int W = (B + 31) >> 5;  // warps
    const bool act = i < B;
    const int j = g * B + (act ? i : 0);
    const bool walls = d.walls != 0, boltz = d.mode == PE_POISSON_BOLTZMANN;
    const bool wl = walls && j == 0, wr = walls && j == ncell - 1;  // this thread's node is a wall
    const double inv_dx2 = d.inv_dx2, diag0 = 2.0 * inv_dx2;
    const float inv = f32_of(inv_dx2), o = -inv;
    const int sep = (w == W - 1) ? ((B - 1) & 31) : 31;  // this warp's separator lane
    // the couplings of this row: mirror ghosts double a wall row's one coupling
    const float lo = wl ? 0.0f : (wr ? 2.0f * o : o), up = wr ? 0.0f : (wl ? 2.0f * o : o);
    if (G > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    // Newton start: phi, or with extrap the extrapolation 2 phi - phi_prev of the last two
    // solutions. phi and phi_prev are written after the iteration only, so the halo nodes below (the
    // neighbouring warps' edge nodes, on the first and the separator lane) are read unchanged
    // and extrapolated here with the owners' arithmetic; later they are advanced here with the
    // updates their owners apply (values of the reduced systems, known to every warp), so they
    // stay bit-identical to the owners' values.
    const bool hist = d.phi_prev != nullptr, ex = hist && d.extrap;
    auto start = [&](int node) { return ex ? 2.0 * d.phi[node] - d.phi_prev[node] : d.phi[node]; };
    double p = start(j);
    double halo = start(lane == 0 ? ((j - 1) & mask) : ((j + 1) & mask));
    double gj = boltz ? exp(p) : 1.0 + p;
    // the charge is the last push's: everything above overlaps with it in a chain of dependent launches
    grid_wait();
    grid_release();
    const long long q = d.rho[j];
    if (d.clear && act) d.rho[j] = 0;
    // density; a wall node's is twice its deposit
    const double nj = fixed_to_double(q, d.shift - ((wl || wr) ? 1 : 0));
    if (G > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every block has started

    int it = 0;
    bool converged = false;
    for (it = 0; it < d.maxit; ++it) {
        const int par = it & 1;
        // ---- FP64 residual (mirror ghosts at walls)
        double pl = __shfl_up_sync(0xFFFFFFFFu, p, 1), pr = __shfl_down_sync(0xFFFFFFFFu, p, 1);
        if (lane == 0) pl = halo;
        if (lane == sep) pr = halo;
        if (wl) pl = pr;
        if (wr) pr = pl;
        const float r = f32_of(fma(fma(-2.0, p, pl) + pr, inv_dx2, -gj) + nj);  // -F_j
        const float bd = f32_of(diag0 + (boltz ? gj : 1.0));
        const float gf = boltz ? f32_of(gj) : 1.0f;
        const float fw = warp_max_bits(act ? __float_as_uint(fabsf(r)) : 0u);
        const float gw = warp_min_bits(act ? gf : 0.0f);  // below 32 nodes: no bound, see above
        // ---- warp interiors: x = rhs - gc S_left - hc S_right
        float a = 0.0f, b = 1.0f, c = 0.0f, rhs = 0.0f, gc = 0.0f, hc = 0.0f;
        if (act && lane != sep) {  // the separator holds an identity row in the warp's reduction
            b = bd;
            rhs = r;
            // couplings to the separators around the interior become extra right-hand sides
            if (lane == 0) gc = lo;
            else a = lo;
            if (lane == sep - 1) hc = up;
            else c = up;
        }
        warp_pcr(a, b, c, rhs, gc, hc);
        UnitRow* mine = &sh.warp[par][w];
        if (lane == 0) mine->first = make_float4(rhs, gc, hc, fw);
        if (lane == sep - 1) mine->last = make_float4(rhs, gc, hc, gw);
        if (lane == sep) mine->sep = make_float4(lo, bd, up, r);
        __syncthreads();
        // ---- the block's warp separators S_0 .. S_{W-2} in terms of the block separators s_{k-1}
        // (left) and s_k (right): row q = lane < W - 1 lies between warp q's last interior row and
        // warp q + 1's first row
        const UnitRow* wrow = sh.warp[par];
        float la = 0.0f, lb = 1.0f, lc = 0.0f, r0 = 0.0f, r1 = 0.0f, r2 = 0.0f;
        uint32_t fl = 0u;
        float gl = 3.0e38f;
        if (lane < W) {
            fl = __float_as_uint(wrow[lane].first.w);
            gl = wrow[lane].last.w;
        }
        if (lane < W - 1) {
            const float4 ep = wrow[lane].last, sr = wrow[lane].sep, en = wrow[lane + 1].first;
            la = -sr.x * ep.y;
            lb = sr.y - sr.x * ep.z - sr.z * en.y;
            lc = -sr.z * en.z;
            r0 = sr.w - sr.x * ep.x - sr.z * en.x;
            if (lane == 0) {  // S_{-1} = s_{k-1}
                r1 = la;
                la = 0.0f;
            }
            if (lane == W - 2) {  // S_{W-1} = s_k
                r2 = lc;
                lc = 0.0f;
            }
        }
        float Y, Gc, Hc;
        warp_chain_pcr(la, lb, lc, r0, r1, r2, W, Y, Gc, Hc);
        // the block's first row (warp 0) and last interior row (warp W - 1) in terms of s_{k-1}, s_k
        const float4 e0 = wrow[0].first, eL = wrow[W - 1].last;
        UnitRow own;
        own.sep = wrow[W - 1].sep;
        const float fbk = warp_max_bits(fl), gbk = warp_min_bits(gl);  // residual bound of the block
        if (W > 1) {  // first row: x = y - g s_{k-1} - h S_0; last row: x = y - g S_{W-2} - h s_k
            const float Y0 = __shfl_sync(0xFFFFFFFFu, Y, 0), G0 = __shfl_sync(0xFFFFFFFFu, Gc, 0);
            const float H0 = __shfl_sync(0xFFFFFFFFu, Hc, 0), YL = __shfl_sync(0xFFFFFFFFu, Y, W - 2);
            const float GL = __shfl_sync(0xFFFFFFFFu, Gc, W - 2), HL = __shfl_sync(0xFFFFFFFFu, Hc, W - 2);
            own.first = make_float4(e0.x - e0.z * Y0, e0.y - e0.z * G0, -e0.z * H0, fbk);
            own.last = make_float4(eL.x - eL.y * YL, -eL.y * GL, eL.z - eL.y * HL, gbk);
        } else {
            own.first = make_float4(e0.x, e0.y, e0.z, fbk);
            own.last = make_float4(eL.x, eL.y, eL.z, gbk);
        }
        // ---- the cyclic system of the block separators s_0 .. s_{G-1}, and the residual bound
        UnitRow rk = own;
        float4 nf = own.first;  // the next block's first row
        if (G > 1) {
            for (int t = w; t < G; t += W)  // the block's warps share the pushes (they hold the same rows)
                if (lane < 3) {
                    float4* dst = reinterpret_cast<float4*>(cluster.map_shared_rank(&sh.block[par][g], t));
                    dst[lane] = lane == 0 ? own.first : (lane == 1 ? own.last : own.sep);
                }
            cluster.sync();  // every block's pushed rows are visible in every block
            rk = sh.block[par][lane & (G - 1)];
            nf = sh.block[par][(lane + 1) & (G - 1)].first;
        }
        const float fb = warp_max_bits(__float_as_uint(rk.first.w)), gb = warp_min_bits(rk.last.w);
        // the residual bounds the next update below tol: phi is converged (the same decision in
        // every warp: the same pushed values)
        if (it > 0 && fb < d.tol * gb) {
            converged = true;
            break;
        }
        // row of s_k: a x_last(k) + b s_k + c x_first(k+1) = d
        const float sk = warp_cyclic(-rk.sep.x * rk.last.y, rk.sep.y - rk.sep.x * rk.last.z - rk.sep.z * nf.y,
                                     -rk.sep.z * nf.z, rk.sep.w - rk.sep.x * rk.last.x - rk.sep.z * nf.x, G);
        const float Sl = __shfl_sync(0xFFFFFFFFu, sk, (g - 1) & (G - 1)), Sr = __shfl_sync(0xFFFFFFFFu, sk, g);
        const float Sn = __shfl_sync(0xFFFFFFFFu, sk, (g + 1) & (G - 1));  // s_{k-1}, s_k, s_{k+1}
        // ---- back substitution: the warp's separators, then its rows
        const float Sq = lane < W - 1 ? Y - Gc * Sl - Hc * Sr : Sr;  // S_lane
        const float S0 = __shfl_sync(0xFFFFFFFFu, Sq, (w - 1) & 31), Sw_r = __shfl_sync(0xFFFFFFFFu, Sq, w);
        const float S2 = __shfl_sync(0xFFFFFFFFu, Sq, w + 1 < W ? w + 1 : w);
        const float Sw_l = w == 0 ? Sl : S0;
        float x = 0.0f;
        if (act) {
            if (lane == sep) x = Sw_r;
            else if (i == 0) x = edge_row(own.first, Sl, Sr);  // the form the left neighbour uses for its halo
            else x = interior_row(rhs, gc, hc, Sw_l, Sw_r);
        }
        // the updates of the halo nodes: the left neighbour's separator, the right neighbour's first row
        float4 right = wrow[w + 1 < W ? w + 1 : w].first;
        if (w + 1 == W) right = G > 1 ? sh.block[par][(g + 1) & (G - 1)].first : own.first;
        const float x_next = w + 1 < W ? edge_row(right, Sw_r, S2) : edge_row(right, Sr, Sn);
        const float mw = warp_max_bits(__float_as_uint(fabsf(x)));  // the warp's largest |update|
        // ---- exchange of the largest update (damping, convergence) and of the bound of the
        // residual it leaves; the FP64 update runs while the exchange is under way
        float xl = __shfl_up_sync(0xFFFFFFFFu, x, 1), xr = __shfl_down_sync(0xFFFFFFFFu, x, 1);
        if (lane == 0) xl = Sw_l;
        if (lane == sep) xr = x_next;
        if (wl) xl = xr;
        if (wr) xr = xl;
        const float Jx = inv * ((x - xl) + (x - xr)) + gf * x;
        const float ax = fabsf(x), big = fmaxf(ax, fmaxf(fabsf(xl), fabsf(xr)));
        // rounding of r, Jx, g and their difference: a few 2^-24 of the terms
        const float e = fabsf(r - Jx) + 2e-6f * ((4.0f * inv + gf) * big + fabsf(r)) +
                        (boltz ? gf * ax * ax * (0.5f + ax) : 0.0f);
        const float2 v = make_float2(mw, warp_max_bits(act ? __float_as_uint(e) : 0u));
        if (G > 1) {
            if (lane < G) *cluster.map_shared_rank(&sh.upd[par][g * W + w], lane) = v;
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        } else if (lane == 0) {
            sh.upd[par][w] = v;
        }
        // the undamped update, and exp(phi) carried with the small-update polynomial
        const double x1 = f64_of(x), xh = f64_of(lane == 0 ? Sw_l : x_next);
        double pn = p + x1, hn = halo + xh, gn = boltz ? gj * exp_tiny(x1) : 1.0 + pn;
        if (G > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        else __syncthreads();
        uint32_t mb = 0u, rb = 0u;
        for (int k = lane; k < G * W; k += 32) {
            const float2 t = sh.upd[par][k];
            mb = max(mb, __float_as_uint(t.x));
            rb = max(rb, __float_as_uint(t.y));
        }
        const float m = warp_max_bits(mb), rm = warp_max_bits(rb);
        // min g' after the update is at least (1 - m) gb
        const bool done = m < d.tol || (m <= 0.0078125f && rm < 0.99f * d.tol * gb);
        if (!done && !(m <= 0.0009765625f)) {  // 2^-10: the polynomial's degree follows the largest update
            double xs = x1;
            if (m > 2.0f) {  // damped
                const double scale = 2.0 / (double)m;
                xs = __dmul_rn(scale, x1);  // product and sum apart, in the owner and in the halo alike
                pn = __dadd_rn(p, xs);
                hn = __dadd_rn(halo, __dmul_rn(scale, xh));
            }
            if (boltz) gn = (fabs(xs) <= 0.03125) ? gj * exp_small(xs) : exp(pn);
            else gn = 1.0 + pn;
        }
        p = pn;
        halo = hn;
        gj = gn;
        if (done) {
            converged = true;
            ++it;
            break;
        }
    }
    if (d.maxit < 1 && G > 1) cluster.sync();  // no exchange ran: every block has read its halo
    if (d.maxit < 1) __syncthreads();
    double pl = __shfl_up_sync(0xFFFFFFFFu, p, 1), pr = __shfl_down_sync(0xFFFFFFFFu, p, 1);
    if (lane == 0) pl = halo;
    if (lane == sep) pr = halo;
    if (act) {
        const double e = (wl || wr) ? 0.0 : (pl - pr) * d.half_inv_dx;
        if (hist) d.phi_prev[j] = d.phi[j];
        d.phi[j] = p;
        d.E[j] = e;
        d.Ef[j] = f32_of(e);
        if (d.Ef0) d.Ef0[j] = f32_of(e);
    }
    if (g == 0 && i == 0) {
        if (d.diag) {
            d.diag[0] = it;
            d.diag[1] = converged ? 1 : 0;
            d.diag[2] = G;
            d.diag[3] = B;
        }
        if (!converged) raise_flag(d.status, PE_FLAG_NOCONV);
    }
}

__global__ void __launch_bounds__(kNewtonMaxThreads, 1) k_newton_cluster(FieldDesc d)
{
    cg::cluster_group cluster = cg::this_cluster();
    newton_body(d, cluster);
}

// One cluster per realisation: cluster c solves descs[c]; extrap (a solve inside a burst, not the one
// that starts it) applies to every realisation. Two blocks to an SM: the groups of an ensemble's grid
// sizes run side by side, and with one block to an SM (128 registers) 24 realisations of 512 to 8192
// nodes want 169 SMs, which left clusters of 16 waiting for a second wave (20 bytes spill at 64; a
// macro step of those realisations 8.93 ms, 8.65 ms so).
__global__ void __launch_bounds__(kNewtonMaxThreads, 2) k_newton_batch(const FieldDesc* descs, int extrap)
{
    cg::cluster_group cluster = cg::this_cluster();
    FieldDesc d = descs[blockIdx.x / cluster.num_blocks()];
    d.extrap = extrap;
    if (extrap) d.Ef0 = nullptr;
    newton_body(d, cluster);
}

// Largest cluster (<= 16, a power of two) the device accepts for these kernels.
static int cluster_limit()
{
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    if (!cached[dev]) {
        cudaFuncSetAttribute((const void*)k_newton_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaFuncSetAttribute((const void*)k_newton_batch, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kClusterMax;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(kClusterMax);
        cfg.blockDim = dim3(kNewtonMaxThreads);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int size = 0;
        if (cudaOccupancyMaxPotentialClusterSize(&size, (const void*)k_newton_cluster, &cfg) != cudaSuccess) size = 8;
        cudaGetLastError();
        int p = 1;
        while (p * 2 <= size && p * 2 <= kClusterMax) p *= 2;
        cached[dev] = p;
    }
    return cached[dev];
}

// Cluster size of a lone solve: as many blocks as the device clusters, at least 32 nodes each (the
// FP64 work is spread over the SMs), one block for the grids below kClusterMinCells.
static int cluster_size_for(int ncell)
{
    const int gmax = cluster_limit();
    int G = gmax;
    while (G > 1 && ncell / G < 32) G >>= 1;
    if (ncell < kClusterMinCells) G = 1;
    while (ncell / G > kNewtonMaxThreads) G <<= 1;  // at most kNewtonMaxThreads nodes (threads) per block
    return G <= gmax ? G : 0;
}

// Cluster size of a realisation's solve inside a batched launch: as few blocks as hold the grid
// at kNewtonMaxThreads nodes each. A lone solve spreads its nodes over up to 16 SMs to cut the
// latency of the FP64 work; an ensemble fills the GPU with many solves at once, and clusters of
// 16 for small grids left most of them waiting for SMs in later waves.
int newton_batch_cluster_size(int ncell)
{
    const int gmax = cluster_limit();
    int G = 1;
    while (ncell / G > kNewtonMaxThreads) G <<= 1;
    return G <= gmax ? G : 0;
}

// attr[2]: the cluster size, and (chain) the programmatic dependence.
static cudaLaunchConfig_t cluster_config(cudaLaunchAttribute* attr, int G, int nclusters, int B, bool chain,
                                         cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(G * nclusters);
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.blockDim = dim3(B < 32 ? 32 : B);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = chain ? 2 : 1;
    return cfg;
}

static int launch_newton_cluster(int G, const FieldDesc& d, bool chain, cudaStream_t s)
{
    const int B = d.ncell / G;  // one node per thread
    if (B > kNewtonMaxThreads || B < 2) return PE_EINVAL;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(attr, G, 1, B, chain, s);
    if (cudaLaunchKernelEx(&cfg, k_newton_cluster, d) != cudaSuccess) return PE_ECUDA;
    return launch_status();
}

// Batched field solves: descs[R] on the device, every grid of ncell nodes.
int launch_newton_batch(const void* descs, int R, int ncell, bool extrap, cudaStream_t s)
{
    const int G = newton_batch_cluster_size(ncell);
    if (G < 1 || R < 1) return PE_EINVAL;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(attr, G, R, ncell / G, false, s);
    if (cudaLaunchKernelEx(&cfg, k_newton_batch, static_cast<const FieldDesc*>(descs), extrap ? 1 : 0) != cudaSuccess)
        return PE_ECUDA;
    return launch_status();
}

static FieldDesc field_desc(const int64_t* rho, int ncell, double dx, int s_w, int mode, int walls, double tol, int maxit,
                            double* phi, double* E, float* Ef, int32_t* diag, uint32_t* status, double* phi_prev,
                            int extrap, int clear)
{
    float ftol = (float)tol;
    if (tol > 0.0 && ftol < FLT_MIN) ftol = FLT_MIN;  // a positive tolerance stays one: an update of 0 meets it
    return FieldDesc{reinterpret_cast<long long*>(const_cast<int64_t*>(rho)), phi, E, Ef, diag, status, 1.0 / (dx * dx), 0.5 / dx,
                     ftol, s_w + 24, ncell, mode, maxit, walls ? 1 : 0, phi_prev, extrap ? 1 : 0, clear, nullptr};
}

size_t field_desc_size() { return sizeof(FieldDesc); }

void make_field_desc(void* out, const int64_t* rho, int ncell, double dx, int s_w, int mode, int walls, double tol,
                     int maxit, double* phi, double* E, float* Ef, float* Ef0, int32_t* diag, uint32_t* status,
                     double* phi_prev)
{
    FieldDesc d = field_desc(rho, ncell, dx, s_w, mode, walls, tol, maxit, phi, E, Ef, diag, status, phi_prev, 0, 1);
    d.Ef0 = Ef0;
    memcpy(out, &d, sizeof(d));
}

}  // namespace pe

using namespace pe;

namespace pe {
// Field solve with a Newton start from the solution history (context path): phi_prev keeps the
// solution before the current one, extrap selects the extrapolated start.
int field_solve_history(const int64_t* rho_fx, int ncell, double dx, int s_w, int mode, int boundary, double tol,
                        int maxit, double* phi, double* E, float* Ef, int32_t* diag, uint32_t* status,
                        double* phi_prev, int extrap, bool chain, bool clear, cudaStream_t s)
{
    if (!is_pow2(ncell) || ncell < 8 || !rho_fx || !phi || !E || !Ef || !(dx > 0.0) || maxit < 0) return PE_EINVAL;
    if (mode != PE_POISSON_BOLTZMANN && mode != PE_POISSON_LINEARIZED) return PE_EINVAL;
    if (boundary != PE_BOUNDARY_PERIODIC && boundary != PE_BOUNDARY_ABSORBING) return PE_EINVAL;
    if (ncell > kFullGridMax) return PE_EINVAL;
    const int G = cluster_size_for(ncell);
    if (G < 1) return PE_EINVAL;
    const FieldDesc d = field_desc(rho_fx, ncell, dx, s_w, mode, boundary == PE_BOUNDARY_ABSORBING, tol, maxit, phi, E, Ef,
                                   diag, status, phi_prev, extrap, clear ? 1 : 0);
    return launch_newton_cluster(G, d, chain, s);
}
}  // namespace pe

// ---------------------------------------------------------------------------------
// Kinetic electrons (Section 4.1's two-species bursts): periodic Poisson equation for the
// net charge, one block of 256 threads; thread t owns the m = ncell / 256 (at least 1)
// consecutive nodes j0 = t m ... The net charge and then the face fields and potentials live
// in shared memory; every sum runs node by node within a thread, then lane by lane and warp
// by warp, in a fixed order. FP64 throughput of one SM bounds this kernel, so each node costs
// a handful of FP64 operations and the block-wide sums run over 256 partial sums.

constexpr int kPoissonThreads = 256;

// Exclusive prefix sum over the block of one value per thread, and the block total.
// wsum: 32 shared slots. Every thread of the block calls it.
template <typename V>
__device__ __forceinline__ V block_exclusive_scan(V x, V* total, V* wsum)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    V incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const V y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        V s = lane < nw ? wsum[lane] : V(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const V y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        wsum[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    const V base = w > 0 ? wsum[w - 1] : V(0);
    *total = wsum[nw - 1];
    __syncthreads();  // wsum is reused by the next call
    return base + incl - x;
}

// clear: both deposits are zeroed for the pushes that follow, in coalesced stores behind the block's reads
// (a store after each node's reads kept the loads from running ahead: 8192 nodes in 86 us, 72 us so, and
// 69.5 us without the clear).
__global__ void __launch_bounds__(kPoissonThreads)
    k_poisson_periodic(long long* __restrict__ rho_i, long long* __restrict__ rho_e, int clear, int n, double dx,
                       double nscale, double* phi, double* E, float* Ef)
{
    extern __shared__ double psh[];
    double* F = psh;      // [n]: net charge, then the face fields F_{j+1/2}
    double* P = psh + n;  // [n]: potential before its mean is removed
    __shared__ double wd[32];
    grid_wait();
    grid_release();
    const int t = threadIdx.x;
    const int m = n >= (int)blockDim.x ? n / (int)blockDim.x : 1;
    const int nt = n / m;  // threads that own nodes
    const int j0 = t * m;
    const bool act = t < nt;
    // net charge per node (the int64 difference of the deposits is exact), and its sum
    double s = 0.0;
    if (act)
        for (int k = 0; k < m; ++k) {
            const double q = (double)(rho_i[j0 + k] - rho_e[j0 + k]);
            F[j0 + k] = q;
            s += q;
        }
    double tot;
    const double off = block_exclusive_scan(s, &tot, wd);  // past its barriers every deposit has been read
    if (clear)
        for (int j = t; j < n; j += (int)blockDim.x) rho_i[j] = rho_e[j] = 0;
    // face fields before the gauge: F_{j+1/2} - F_{-1/2} = dx nscale (S_j - (j + 1) <S>)
    const double mean = tot / n, c = dx * nscale;
    double fs = 0.0;
    if (act) {
        double acc = off;
        for (int k = 0; k < m; ++k) {
            acc += F[j0 + k];
            const double f = c * (acc - (double)(j0 + k + 1) * mean);
            F[j0 + k] = f;
            fs += f;
        }
    }
    double ftot;
    (void)block_exclusive_scan(fs, &ftot, wd);
    const double gauge = ftot / n;  // the faces of a periodic phi sum to zero
    double ps = 0.0;
    if (act)
        for (int k = 0; k < m; ++k) {
            const double f = F[j0 + k] - gauge;
            F[j0 + k] = f;
            ps += f;
        }
    // phi_0 = 0, phi_{j+1} = phi_j - dx F_{j+1/2}
    double ptot;
    const double poff = block_exclusive_scan(ps, &ptot, wd);
    double psum = 0.0;
    if (act) {
        double p = -dx * poff;
        for (int k = 0; k < m; ++k) {
            P[j0 + k] = p;
            psum += p;
            p -= dx * F[j0 + k];
        }
    }
    double pt;
    (void)block_exclusive_scan(psum, &pt, wd);  // its barriers also publish F to the neighbours
    const double pmean = pt / n;
    if (act)
        for (int k = 0; k < m; ++k) {
            const int j = j0 + k;
            const double e = 0.5 * (F[j] + F[j > 0 ? j - 1 : n - 1]);  // E_j = (F_{j+1/2} + F_{j-1/2}) / 2
            E[j] = e;
            Ef[j] = (float)e;
            phi[j] = P[j] - pmean;
        }
}

__global__ void k_boltzmann_profile(const double* phi, const long long* mom, int n, double vscale, float* nprof,
                                    float* uprof)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) {
        nprof[j] = (float)exp(phi[j]);
        if (uprof) {
            float u = 0.0f;
            if (mom) {  // V_e = V_i: the ions' momentum over their density at the node
                const long long d = mom[j], m = mom[n + j];
                if (d > 0) u = (float)((double)m / (double)d * vscale);
            }
            uprof[j] = u;
        }
    }
}

namespace pe {
int field_solve_kinetic(int64_t* rho_i, int64_t* rho_e, int ncell, double dx, int s_w, double* phi, double* E,
                        float* Ef, bool chain, bool clear, cudaStream_t s)
{
    if (!is_pow2(ncell) || ncell < 8 || ncell > kFullGridMax || !rho_i || !rho_e || !phi || !E || !Ef ||
        !(dx > 0.0))
        return PE_EINVAL;
    const size_t smem = 2 * sizeof(double) * (size_t)ncell;
    if (ensure_smem((const void*)k_poisson_periodic, smem) != PE_OK) return PE_ECUDA;
    long long* ri = reinterpret_cast<long long*>(rho_i);
    long long* re = reinterpret_cast<long long*>(rho_e);
    const double scale = ldexp(1.0, -(s_w + 24));
    if (chain)
        PE_TRY(launch_dependent(k_poisson_periodic, dim3(1), kPoissonThreads, smem, s, ri, re, clear ? 1 : 0, ncell, dx,
                                scale, phi, E, Ef));
    else
        k_poisson_periodic<<<1, kPoissonThreads, smem, s>>>(ri, re, clear ? 1 : 0, ncell, dx, scale, phi, E, Ef);
    return launch_status();
}
}  // namespace pe

extern "C" PE_API int pe_field_kinetic(const int64_t* rho_i, const int64_t* rho_e, int32_t ncell, double dx,
                                       int32_t s_w, double* phi, double* E, float* Ef, void* stream)
{
    return field_solve_kinetic(const_cast<int64_t*>(rho_i), const_cast<int64_t*>(rho_e), ncell, dx, s_w, phi, E, Ef,
                               false, false, (cudaStream_t)stream);
}

extern "C" PE_API int pe_boltzmann_profile(const double* phi, const int64_t* ion_moments, int32_t s_w, int32_t s_p,
                                           int32_t ncell, float* n_prof, float* u_prof, void* stream)
{
    if (!is_pow2(ncell) || ncell < 8 || ncell > kFullGridMax || !phi || !n_prof || (ion_moments && !u_prof))
        return PE_EINVAL;
    k_boltzmann_profile<<<(ncell + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
        phi, reinterpret_cast<const long long*>(ion_moments), ncell, ldexp(1.0, s_w - s_p), n_prof, u_prof);
    return launch_status();
}

extern "C" PE_API int pe_field_ex(const int64_t* rho_fx, int32_t ncell, double dx, int32_t s_w, int32_t mode,
                                  int32_t boundary, double tol, int32_t maxit, double* phi, double* E, float* Ef,
                                  int32_t* diag, uint32_t* status, void* stream)
{
    return field_solve_history(rho_fx, ncell, dx, s_w, mode, boundary, tol, maxit, phi, E, Ef, diag, status, nullptr,
                               0, false, false, (cudaStream_t)stream);
}

extern "C" PE_API int pe_field(const int64_t* rho_fx, int32_t ncell, double dx, int32_t s_w, int32_t mode, double tol,
                               int32_t maxit, double* phi, double* E, float* Ef, int32_t* diag, uint32_t* status,
                               void* stream)
{
    return pe_field_ex(rho_fx, ncell, dx, s_w, mode, PE_BOUNDARY_PERIODIC, tol, maxit, phi, E, Ef, diag, status,
                       stream);
}
