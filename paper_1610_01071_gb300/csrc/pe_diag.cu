// Diagnostics of a particle state (Section 4: the charge, momentum and energy checks of
// the resolved and projective runs; the particle Courant number max|V| dt / dx of the
// fine step, the particle-level counterpart of the macroscopic condition Eq. (CFL)) and the
// coarse-variable error measure of Section 4.1.1.
//
// Two launches: a particle pass (grid-stride, fixed grid for a given n and ncell, so the
// floating-point sums are reproduced bit for bit) writes one partial per block, the nodal energies
// among them; a single block adds the partials in a fixed order.
//
// The FP64 pipe bounds a direct form (seven FP64 instructions per particle at 1.7 lanes per
// cycle and SM: 128 us for 2^23 particles, 16 % of the memory bandwidth). The sums run in FP32
// instead, as unevaluated sums of three floats with error-free additions and products (Knuth's
// and Dekker's two-sum and two-product): about 70 bits, so that a sum is rounded once, at its
// conversion to FP64; FP64 takes only the conversion of the block sums: 42 us for 2^23 particles
// (128 before), and the final pass 6 us (35 with the nodal exponentials in its one block).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "pe_common.cuh"
#include "pe_internal.h"
#include "pepic.h"

namespace pe {
namespace {

constexpr int kDiagThreads = 256;
constexpr int kDiagMaxBlocks = 608;  // four per SM: enough loads in flight to stream the particles
constexpr int kFinalThreads = 1024;

struct DiagScratch {
    long long wq[kDiagMaxBlocks];
    long long invalid[kDiagMaxBlocks];
    double mom[kDiagMaxBlocks];
    double kin[kDiagMaxBlocks];
    double wsum[kDiagMaxBlocks];
    double fe[kDiagMaxBlocks];
    double ee[kDiagMaxBlocks];
    float vmax[kDiagMaxBlocks];
};
static_assert(sizeof(DiagScratch) <= PE_MOMENTS_SCRATCH_BYTES, "scratch size");

__device__ __forceinline__ long long warp_sum_i64(long long v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float warp_maxf(float v)
{
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// a + b = s + e exactly (Knuth).
__device__ __forceinline__ float two_sum(float a, float b, float& e)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// Sum kept as h + l + t; only the additions to t round (2^-72 of the terms).
struct Sum3 {
    float h, l, t;
    __device__ __forceinline__ void reset() { h = l = t = 0.0f; }
    __device__ __forceinline__ void add_low(float x)  // x of the size of an error of h
    {
        float f;
        l = two_sum(l, x, f);
        t = __fadd_rn(t, f);
    }
    __device__ __forceinline__ void add(float x)
    {
        float e;
        h = two_sum(h, x, e);
        add_low(e);
    }
    __device__ __forceinline__ void add(const Sum3& o)
    {
        add(o.h);
        add_low(o.l);
        t = __fadd_rn(t, o.t);
    }
    __device__ __forceinline__ void warp_fold()
    {
        for (int o = 16; o > 0; o >>= 1) {
            Sum3 x;
            x.h = __shfl_xor_sync(0xffffffffu, h, o);
            x.l = __shfl_xor_sync(0xffffffffu, l, o);
            x.t = __shfl_xor_sync(0xffffffffu, t, o);
            add(x);
        }
    }
    __device__ __forceinline__ double value() const { return (double)h + ((double)l + (double)t); }
};

struct MomentSums {
    Sum3 ws, mom, kin;  // sum w, sum w V, sum w V^2
    double ws64, mom64, kin64;  // the same of particles whose products leave FP32's range
    long long wq;
    int bad;
    bool wide;  // the FP64 sums were used
    float vmax;
};

// One particle. Vbar = v + (kick - 1/2) qm dt E(X) is the integer-time velocity; a particle with a
// cell outside [0, ncell), a non-finite offset or velocity, or an offset outside [0, 1] is
// counted as invalid and left out of the sums.
__device__ __forceinline__ void moment_one(MomentSums& S, int c, float th, float vv, float ww,
                                           const float* __restrict__ Ef, int ncell, float hk, float wscale)
{
    if ((unsigned)c >= (unsigned)ncell || !isfinite(vv) || !isfinite(ww) || !(th >= 0.0f && th <= 1.0f)) {
        ++S.bad;
        return;
    }
    const int c1 = (c + 1 == ncell) ? 0 : c + 1;
    const float Ec = __ldg(Ef + c), Ec1 = __ldg(Ef + c1);
    const float vb = fmaf(hk, fmaf(th, Ec1 - Ec, Ec), vv);
    S.wq += (long long)__float2int_rn(ww * wscale);
    S.vmax = fmaxf(S.vmax, fabsf(vb));
    const float p = __fmul_rn(ww, vb), q = __fmul_rn(p, vb), m = fabsf(q);
    // products whose error terms FP32 represents (or a zero factor); others in FP64
    if (fabsf(ww) <= 1.2676506e30f && ((m >= 3.3087225e-24f && m <= 1.2676506e30f) || ww == 0.0f || vb == 0.0f)) {
        S.ws.add(ww);  // 2^-78 <= m <= 2^100
        const float e = fmaf(ww, vb, -p);  // w V = p + e
        S.mom.add(p);
        S.mom.add_low(e);
        const float g = __fmul_rn(e, vb);
        S.kin.add(q);                      // w V^2 = q + (p V - q) + e V
        S.kin.add_low(fmaf(p, vb, -q));
        S.kin.add_low(g);
        S.kin.t = __fadd_rn(S.kin.t, fmaf(e, vb, -g));
    } else {
        const double wd = (double)ww, vd = (double)vb;
        S.wide = true;
        S.ws64 += wd;
        S.mom64 += wd * vd;
        S.kin64 += wd * vd * vd;
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kDiagThreads, 4) k_moments_particles(
    const int32_t* __restrict__ cell, const float* __restrict__ theta, const float* __restrict__ v,
    const float* __restrict__ w, int64_t n, const float* __restrict__ Ef, const double* __restrict__ phi,
    const double* __restrict__ E, int ncell, float hk, float wscale, int mode, DiagScratch* __restrict__ out,
    uint32_t* status)
{
    MomentSums S;
    S.ws.reset();
    S.mom.reset();
    S.kin.reset();
    S.ws64 = S.mom64 = S.kin64 = 0.0;
    S.wq = 0;
    S.bad = 0;
    S.wide = false;
    S.vmax = 0.0f;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // nodal energies, the nodes spread over the blocks (the exponential is FP64 work)
    double fe = 0.0, ee = 0.0;
    for (int64_t j = t0; j < ncell; j += stride) {
        const double e = E ? E[j] : 0.0;
        fe += 0.5 * e * e;
        if (phi) {
            const double p = phi[j];
            ee += (mode == PE_POISSON_BOLTZMANN) ? (p * exp(p) - exp(p) + 1.0) : 0.5 * p * p;
        }
    }
    const bool nodes = (int64_t)blockIdx.x * blockDim.x < ncell;  // this block has some
    const int64_t n4 = VEC ? n >> 2 : 0;
    if (VEC) {
        for (int64_t g = t0; g < n4; g += stride) {
            const int4 c = __ldg(reinterpret_cast<const int4*>(cell) + g);
            const float4 th = __ldg(reinterpret_cast<const float4*>(theta) + g);
            const float4 vv = __ldg(reinterpret_cast<const float4*>(v) + g);
            const float4 ww = __ldg(reinterpret_cast<const float4*>(w) + g);
            moment_one(S, c.x, th.x, vv.x, ww.x, Ef, ncell, hk, wscale);
            moment_one(S, c.y, th.y, vv.y, ww.y, Ef, ncell, hk, wscale);
            moment_one(S, c.z, th.z, vv.z, ww.z, Ef, ncell, hk, wscale);
            moment_one(S, c.w, th.w, vv.w, ww.w, Ef, ncell, hk, wscale);
        }
    }
    for (int64_t i = 4 * n4 + t0; i < n; i += stride)
        moment_one(S, cell[i], theta[i], v[i], w[i], Ef, ncell, hk, wscale);

    constexpr int kW = kDiagThreads / 32;
    __shared__ Sum3 ss[3][kW];
    __shared__ double s64[5][kW];  // FP64 sums of w, w V and w V^2, field and electron energies
    __shared__ long long sq[kW];
    __shared__ int sb[kW];
    __shared__ float sv[kW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    S.ws.warp_fold();
    S.mom.warp_fold();
    S.kin.warp_fold();
    const long long wq = warp_sum_i64(S.wq);
    const int bad = __reduce_add_sync(0xffffffffu, S.bad);
    const float vm = warp_maxf(S.vmax);
    const bool wide = __any_sync(0xffffffffu, S.wide);
    const double w64 = wide ? warp_sum(S.ws64) : 0.0, m64 = wide ? warp_sum(S.mom64) : 0.0;
    const double k64 = wide ? warp_sum(S.kin64) : 0.0;
    if (nodes) {
        fe = warp_sum(fe);
        ee = warp_sum(ee);
    }
    if (lane == 0) {
        ss[0][wid] = S.ws;
        ss[1][wid] = S.mom;
        ss[2][wid] = S.kin;
        s64[0][wid] = w64;
        s64[1][wid] = m64;
        s64[2][wid] = k64;
        s64[3][wid] = fe;
        s64[4][wid] = ee;
        sq[wid] = wq;
        sb[wid] = bad;
        sv[wid] = vm;
    }
    __syncthreads();
    if (wid == 0) {
        if (lane < 3) {
            Sum3 a = ss[lane][0];
            for (int k = 1; k < kW; ++k) a.add(ss[lane][k]);
            double x = a.value();
            for (int k = 0; k < kW; ++k)
                if (s64[lane][k] != 0.0) x += s64[lane][k];
            (lane == 0 ? out->wsum : (lane == 1 ? out->mom : out->kin))[blockIdx.x] = x;
        } else if (lane < 5) {
            double x = s64[lane][0];
            if (nodes)
                for (int k = 1; k < kW; ++k) x += s64[lane][k];
            (lane == 3 ? out->fe : out->ee)[blockIdx.x] = x;
        } else if (lane == 5) {
            long long q = 0, b = 0;
            float m = 0.0f;
            for (int k = 0; k < kW; ++k) {
                q += sq[k];
                b += sb[k];
                m = fmaxf(m, sv[k]);
            }
            out->wq[blockIdx.x] = q;
            out->invalid[blockIdx.x] = b;
            out->vmax[blockIdx.x] = m;
            if (b) raise_flag(status, PE_FLAG_RANGE);
        }
    }
}

template <typename T, typename Op>
__device__ T block_reduce(T x, T* red, Op op)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
    __syncthreads();
    if (lane == 0) red[wid] = x;
    __syncthreads();
    if (wid == 0) {
        x = red[lane];  // 32 warps of 32 threads
        for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
    }
    return x;  // valid in warp 0
}

// Final pass, one quantity per warp (each FP64 addition of a warp holds its scheduler's pipe): the
// block partials in a fixed order.
__global__ void __launch_bounds__(256) k_moments_final(const DiagScratch* __restrict__ part, int nblocks, double dx,
                                                       double dt, double charge_scale, pe_moments* out)
{
    __shared__ double sd[5];
    __shared__ long long si[2];
    __shared__ float sf;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < 5) {
        const double* src = wid == 0 ? part->mom : (wid == 1 ? part->kin : (wid == 2 ? part->wsum : (wid == 3 ? part->fe : part->ee)));
        double x = 0.0;
        for (int b = lane; b < nblocks; b += 32) x += src[b];
        x = warp_sum(x);
        if (lane == 0) sd[wid] = x;
    } else if (wid < 7) {
        const long long* src = wid == 5 ? part->wq : part->invalid;
        long long x = 0;
        for (int b = lane; b < nblocks; b += 32) x += src[b];
        x = warp_sum_i64(x);
        if (lane == 0) si[wid - 5] = x;
    } else {
        float x = 0.0f;
        for (int b = lane; b < nblocks; b += 32) x = fmaxf(x, part->vmax[b]);
        x = warp_maxf(x);
        if (lane == 0) sf = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        pe_moments m;
        m.charge_fx = (long long)((unsigned long long)si[0] << 24);  // modulo 2^64
        m.invalid = si[1];
        m.charge_wq = si[0];
        m.charge_fixed_point = (double)m.charge_fx * charge_scale * dx;
        m.charge = sd[2] * dx;
        m.momentum = sd[0] * dx;
        m.kinetic = 0.5 * sd[1] * dx;
        m.field_energy = sd[3] * dx;
        m.electron_energy = sd[4] * dx;
        m.total_energy = m.kinetic + m.field_energy + m.electron_energy;
        m.max_speed = (double)sf;
        m.cfl = (double)sf * dt / dx;
        *out = m;
    }
}

__global__ void __launch_bounds__(kFinalThreads) k_rel_l2(const double* __restrict__ a, const double* __restrict__ b,
                                                           int64_t n, double* out)
{
    __shared__ double rd[32];
    double num = 0.0, den = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += kFinalThreads) {
        const double x = a[i], y = b[i];
        num += (x - y) * (x - y);
        den += x * x + y * y;
    }
    auto add_d = [](double u, double v) { return u + v; };
    num = block_reduce(num, rd, add_d);
    const double nums = num;
    den = block_reduce(den, rd, add_d);
    if (threadIdx.x == 0) *out = den > 0.0 ? sqrt(nums / den) : 0.0;
}

}  // namespace

// Blocks of the particle pass: 16 particles per thread, and a thread per node, up to kDiagMaxBlocks.
static int moments_blocks(int64_t n, int ncell)
{
    const int64_t per = (int64_t)kDiagThreads * 16;
    int64_t b = std::max((n + per - 1) / per, ((int64_t)ncell + kDiagThreads - 1) / kDiagThreads);
    if (b < 1) b = 1;
    if (b > kDiagMaxBlocks) b = kDiagMaxBlocks;
    return (int)b;
}

}  // namespace pe

using namespace pe;

namespace pe {
namespace {
// Kinetic energy sum w Vbar^2 dx / 2 of one species: FP32 per-thread sums over a fixed
// grid-stride partition, FP64 from the warp sums on (the FP64 pipe is narrow on this part), block
// partials folded in block order by one thread: reproducible.
constexpr int kEnergyBlocks = 1024;

__global__ void __launch_bounds__(kDiagThreads) k_energy_part(const int32_t* __restrict__ cell,
                                                              const float* __restrict__ theta,
                                                              const float* __restrict__ v, const float* __restrict__ w,
                                                              int64_t n, const float* __restrict__ Ef, int ncell,
                                                              float hk, double* __restrict__ part,
                                                              uint32_t* __restrict__ status)
{
    float k = 0.0f;
    bool bad = false;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int c = cell[i];
        if ((unsigned)c >= (unsigned)ncell) {
            bad = true;
            continue;
        }
        const int c1 = (c + 1 == ncell) ? 0 : c + 1;
        const float Ec = __ldg(Ef + c), Ec1 = __ldg(Ef + c1);
        const float vb = fmaf(hk, fmaf(theta[i], Ec1 - Ec, Ec), v[i]);
        k = fmaf(w[i] * vb, vb, k);
    }
    if (bad) raise_flag(status, PE_FLAG_RANGE);
    __shared__ double sk[kDiagThreads / 32];
    const double kw = warp_sum((double)k);
    if ((threadIdx.x & 31) == 0) sk[threadIdx.x >> 5] = kw;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int j = 0; j < kDiagThreads / 32; ++j) t += sk[j];
        part[blockIdx.x] = t;
    }
}

__global__ void k_energy_final(const double* __restrict__ part, int nb, double half_dx, double* __restrict__ out)
{
    if (threadIdx.x != 0) return;
    double t = 0.0;
    for (int b = 0; b < nb; ++b) t += part[b];
    *out = t * half_dx;
}
}  // namespace
}  // namespace pe

extern "C" PE_API int pe_kinetic_energy(const int32_t* cell, const float* theta, const float* v, const float* w,
                                        int64_t n, const float* Ef, int32_t ncell, double dx, float qm_dt, float kick,
                                        double* scratch, double* out, uint32_t* status, void* stream)
{
    if (n < 0 || ncell < 2 || !(dx > 0.0) || !scratch || !out || !status) return PE_EINVAL;
    if (n > 0 && (!cell || !theta || !v || !w || !Ef)) return PE_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (int)std::min<int64_t>(kEnergyBlocks, std::max<int64_t>(1, (n + 4095) / 4096));
    k_energy_part<<<nb, kDiagThreads, 0, s>>>(cell, theta, v, w, n, Ef, ncell, (kick - 0.5f) * qm_dt, scratch,
                                              status);
    k_energy_final<<<1, 32, 0, s>>>(scratch, nb, 0.5 * dx, out);
    return launch_status(2);
}

extern "C" PE_API int pe_compute_moments(const int32_t* cell, const float* theta, const float* v, const float* w, int64_t n,
                                 const float* Ef, const double* phi, const double* E, int32_t ncell, double dx,
                                 double dt, float qm_dt, float kick, int32_t s_w, int32_t mode, void* scratch,
                                 pe_moments* out, uint32_t* status, void* stream)
{
    if (n < 0 || ncell < 2 || !(dx > 0.0) || !(dt >= 0.0) || !scratch || !out) return PE_EINVAL;
    if (n > 0 && (!cell || !theta || !v || !w || !Ef)) return PE_EINVAL;
    if (((uintptr_t)scratch & 15u) || ((uintptr_t)out & 7u)) return PE_EINVAL;
    if (mode != PE_POISSON_BOLTZMANN && mode != PE_POISSON_LINEARIZED) return PE_EINVAL;
    if (s_w < -60 || s_w > 60) return PE_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = moments_blocks(n, ncell);
    DiagScratch* part = (DiagScratch*)scratch;
    const float wscale = ldexpf(1.0f, s_w);
    const float hk = (kick - 0.5f) * qm_dt;
    const bool vec = aligned16(cell) && aligned16(theta) && aligned16(v) && aligned16(w);
    (vec ? k_moments_particles<true> : k_moments_particles<false>)<<<nb, kDiagThreads, 0, s>>>(
        cell, theta, v, w, n, Ef, phi, E, ncell, hk, wscale, mode, part, status);
    k_moments_final<<<1, 256, 0, s>>>(part, nb, dx, dt, ldexp(1.0, -(s_w + 24)), out);
    return launch_status(2);
}

namespace pe {

// Kinetic electrons: the ions' moments (out) absorb the electrons' (e, velocities of the
// electron pass, mass w / |q_e/m_e| per particle): electron_energy = the electrons' kinetic
// energy, momentum of both species, the larger speed and CFL number, total = kinetic of the
// ions + field + electrons.
__global__ void k_moments_kinetic(pe_moments* out, const pe_moments* e, double inv_mass_ratio)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    out->electron_energy = e->kinetic * inv_mass_ratio;
    out->momentum += e->momentum * inv_mass_ratio;
    out->total_energy = out->kinetic + out->field_energy + out->electron_energy;
    out->max_speed = fmax(out->max_speed, e->max_speed);
    out->cfl = fmax(out->cfl, e->cfl);
    out->invalid += e->invalid;
}

int combine_kinetic_moments(pe_moments* out, const pe_moments* electrons, double qm_e, cudaStream_t s)
{
    if (!(qm_e < 0.0)) return PE_EINVAL;
    k_moments_kinetic<<<1, 32, 0, s>>>(out, electrons, 1.0 / -qm_e);
    return launch_status(1);
}

}  // namespace pe

extern "C" PE_API int pe_rel_l2(const double* a, const double* b, int64_t n, double* out, void* stream)
{
    if (n < 0 || !out || (n > 0 && (!a || !b))) return PE_EINVAL;
    k_rel_l2<<<1, kFinalThreads, 0, (cudaStream_t)stream>>>(a, b, n, out);
    return launch_status(1);
}
