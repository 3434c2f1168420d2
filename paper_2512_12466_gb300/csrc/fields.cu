// Per-cell kernels around the march: input validation, the absorber and
// optical-depth field (Sec. 2.6: a_abs = (1 - x) n_H; Eq. 2), the heating
// and deposited-photon reduction after the trace, and the C2-Ray
// time-averaged ionization update of Eq. 3 (Sec. 2.3).
//
// They stream the flat n^3 arrays, but GB300's FP64 pipe (2 lanes a clock and
// SM, 64 cycles of a scheduler per warp instruction) binds them before HBM
// does, so each kernel keeps the FP64 operations its result needs and does the
// rest on the integer pipe: comparisons on the bit patterns, the rounding of
// kappa to float (narrow), sums only where there is something to add. Passes
// over the same arrays are one pass: validation, the sum for the n_th default
// and the copy into the handle; kappa and the clearing of Gamma; heating, the
// deposited photons and the results' way out.
// At 128^3 cells (neutral, FP32) the check takes 16 us, kappa 17 and the heating 14; at 256^3 (half
// ionized) 82, 102 and 176. Before, kappa took 31 and 220 and the heating 35 and 203, beside a validation, a
// mean, the clearing of Gamma and two copies each way. A batch of 48 solves takes 226 and 127 us for kappa and
// heating, one launch each; 48 launches of each took 13 and 18 us apiece.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "rt_internal.h"

namespace nyx {
namespace {

constexpr int kBlock = 256;
constexpr int kUnroll = 4;                        // independent cells in flight per thread
constexpr int kTile = kBlock * kUnroll;           // cells a block takes at a time

int grid_for(int64_t count)
{
    int64_t g = (count + kBlock - 1) / kBlock;
    if (g > 152 * 16) g = 152 * 16;
    return g < 1 ? 1 : (int)g;
}

// Blocks for a tiled pass: one tile each up to eight resident blocks per SM, then grid-stride.
int64_t tiles_for(int64_t ncell)
{
    return std::max<int64_t>(1, std::min<int64_t>((ncell + kTile - 1) / kTile, 152 * 8));
}

__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double part[kBlock / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) part[wid] = v;
    __syncthreads();
    v = 0.0;
    if (wid == 0) {
        v = lane < kBlock / 32 ? part[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;
}

// Order of non-negative doubles by their bit patterns (a NaN counts as larger than everything).
__device__ __forceinline__ long long bits_of(const double v) { return __double_as_longlong(v); }

// n_H finite and not negative, x in [0, 1] (both signs of zero included).
__device__ __forceinline__ bool bad_cell(const double nh, const double x)
{
    const unsigned long long a = (unsigned long long)bits_of(nh), b = (unsigned long long)bits_of(x);
    const bool a_ok = a < 0x7ff0000000000000ull || a == 0x8000000000000000ull;
    const bool b_ok = b <= 0x3ff0000000000000ull || b == 0x8000000000000000ull;
    return !(a_ok && b_ok);
}

// One pass over new fields: invalid values counted, n_H summed (and x, if asked), and both copied
// (nh_out, x_out null: no copy). The last block turns the sum into the default n_th, 0.01 mean(n_H).
__global__ void __launch_bounds__(kBlock) check_fields_kernel(const double* __restrict__ nh,
                                                              const double* __restrict__ x, int64_t ncell,
                                                              double* __restrict__ nh_out, double* __restrict__ x_out,
                                                              bool want_x, FieldCheck* chk)
{
    unsigned bad = 0;
    double sn = 0.0, sx = 0.0;
    for (int64_t t0 = blockIdx.x * (int64_t)kTile; t0 < ncell; t0 += (int64_t)gridDim.x * kTile) {
        double a[kUnroll], b[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t c = t0 + u * kBlock + threadIdx.x;
            a[u] = c < ncell ? nh[c] : 0.0;
            b[u] = c < ncell ? x[c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t c = t0 + u * kBlock + threadIdx.x;
            if (nh_out && c < ncell) {
                nh_out[c] = a[u];
                x_out[c] = b[u];
            }
            bad += bad_cell(a[u], b[u]) ? 1u : 0u;
            sn += a[u];
        }
        if (want_x) {
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) sx += b[u];
        }
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && bad) atomicAdd(&chk->acc_bad, bad);
    sn = block_sum(sn);                       // its barriers also order the counts of bad cells
    if (want_x) sx = block_sum(sx);
    if (threadIdx.x == 0) {
        atomicAdd(&chk->acc_nh, sn);
        if (want_x) atomicAdd(&chk->acc_x, sx);
        __threadfence();
        if (atomicAdd(&chk->blocks_done, 1u) + 1u == gridDim.x) {
            __threadfence();
            const double total = *((volatile double*)&chk->acc_nh);
            chk->sum_nh = total;
            chk->sum_x = *((volatile double*)&chk->acc_x);
            chk->n_th = __dmul_rn(0.01, __ddiv_rn(total, (double)ncell));
            chk->bad = *((volatile unsigned*)&chk->acc_bad);
            chk->acc_nh = chk->acc_x = 0.0;
            chk->acc_bad = chk->blocks_done = 0u;
        }
    }
}

// v rounded to the nearest float, ties to even, on the integer pipe, its sign bit changed by flip (0 or
// 0x80000000): the magnitude's leading 24 bits and the rest, shifted down first where the result is
// subnormal. Negative values pass through the branch of the values that are no normal floats, so that they
// cost the others nothing (both shifts drop the sign bit).
__device__ __forceinline__ float narrow(const double v, unsigned flip)
{
    const unsigned hi = (unsigned)(bits_of(v) >> 32), lo = (unsigned)bits_of(v);
    unsigned u = ((hi - 0x38000000u) << 3) | (lo >> 29), rem = lo << 3;       // rem: in units of 2^-32 of u's last place
    if (hi - 0x38100000u >= 0x47f00000u - 0x38100000u) {                      // negative, or not a normal float (zero among them)
        const unsigned mag = hi & 0x7fffffffu;
        flip ^= hi & 0x80000000u;
        if (mag >= 0x47f00000u)
            return __uint_as_float(flip ^ (mag > 0x7ff00000u || (mag == 0x7ff00000u && lo) ? 0x7fffffffu : 0x7f800000u));
        if (mag < 0x38100000u) {
            const int down = 897 - (int)(mag >> 20);                          // 1 .. 897
            const unsigned long long m = ((unsigned long long)((mag & 0xfffffu) | 0x100000u) << 32) | lo;
            const unsigned long long w = down < 32 ? m >> down : 0ull;        // below 2^-158: nothing
            const bool sticky = down < 32 && (m & ((1ull << down) - 1ull)) != 0ull;
            u = (unsigned)(w >> 29);
            rem = ((unsigned)w << 3) | (sticky ? 1u : 0u);
        }
    }
    u += (rem > 0x80000000u || (rem == 0x80000000u && (u & 1u))) ? 1u : 0u;
    return __uint_as_float(u ^ flip);
}

// n_th for eligible: a NaN of either sign as the positive one, whose bit pattern lies above every density's
// (no cell is eligible then, as none compares >= to it).
inline double ordered_threshold(const double n_th) { return std::isnan(n_th) ? std::fabs(n_th) : n_th; }

// Eqs. 7-8: whether a cell may receive a secondary deposit, n_H >= n_th and n_HI > 0, on the bit patterns.
__device__ __forceinline__ bool eligible(const double nh, const double nhi, const double n_th)
{
    return bits_of(nh) >= bits_of(n_th) && bits_of(nhi) > 0;
}

// k where the cell may receive a secondary deposit, -k elsewhere, for any sign of k (a -0.0 in n_H gives a
// negative zero).
template <class R>
__device__ __forceinline__ R stored_kappa(const double k, const bool elig)
{
    if constexpr (sizeof(R) == 4) return narrow(k, elig ? 0u : 0x80000000u);
    else return __longlong_as_double(bits_of(k) ^ (elig ? 0ll : (long long)0x8000000000000000ull));
}

// kappa = (sigma dx) ((1 - x) n_H), the optical depth per cell length, and Gamma cleared.
// kappa is stored negated (sign bit set) when the cell may not receive a secondary
// deposit under Eqs. 7-8 (n_H < n_th, or n_HI = 0). The decision chain uses
// round-to-nearest intrinsics only; three FP64 operations a cell (a vote that spared neutral gas two of
// them broke the unrolled loop up: 22 against 17 us at 128^3).
template <class R>
__device__ __forceinline__ void prepare_cells(const FieldJob& J, const int64_t first, const int64_t stride)
{
    const double n_th = J.chk ? J.chk->n_th : J.n_th;
    R* const kap = static_cast<R*>(J.kap);
    for (int64_t t0 = first * kTile; t0 < J.ncell; t0 += stride * kTile) {
        double a[kUnroll], b[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t c = t0 + u * kBlock + threadIdx.x;
            a[u] = c < J.ncell ? J.nh[c] : 0.0;
            b[u] = c < J.ncell ? J.x[c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t c = t0 + u * kBlock + threadIdx.x;
            if (c >= J.ncell) break;
            const double nhi = __dmul_rn(__dsub_rn(1.0, b[u]), a[u]);
            const double k = __dmul_rn(J.sdx, nhi);
            kap[c] = stored_kappa<R>(k, eligible(a[u], nhi, n_th));
            J.gamma[c] = 0.0;
        }
    }
}

// heat = e_heat Gamma n_HI; deposited photons = sum Gamma n_HI dx^3; Gamma copied out (gamma_out null:
// not). Most cells of an opaque box have no Gamma: a thread without any in its four reads neither field, a
// warp without any takes no FP64 operation (a test per cell cost more than it saved: 32 against 17 us).
__device__ __forceinline__ void finalize_cells(const FieldJob& J, const int64_t first, const int64_t stride)
{
    double dep = 0.0;
    const double heat0 = J.e_heat * 0.0;          // of a cell without Gamma (n_HI is finite)
    for (int64_t t0 = first * kTile; t0 < J.ncell; t0 += stride * kTile) {
        double g[kUnroll], h[kUnroll];
        bool any = false;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t c = t0 + u * kBlock + threadIdx.x;
            g[u] = c < J.ncell ? J.gamma[c] : 0.0;
            h[u] = heat0;
            any = any || bits_of(g[u]) << 1;
        }
        if (any) {
            double a[kUnroll], b[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int64_t c = t0 + u * kBlock + threadIdx.x;
                a[u] = c < J.ncell ? J.nh[c] : 0.0;
                b[u] = c < J.ncell ? J.x[c] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const double r = g[u] * ((1.0 - b[u]) * a[u]);
                h[u] = J.e_heat * r;
                dep += r;
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t c = t0 + u * kBlock + threadIdx.x;
            if (c >= J.ncell) break;
            if (J.gamma_out) J.gamma_out[c] = g[u];
            if (J.heat) J.heat[c] = h[u];
        }
    }
    if (!__syncthreads_or(bits_of(dep) << 1 != 0)) return;
    dep = block_sum(dep);
    if (threadIdx.x == 0) atomicAdd(&J.st->deposited, dep * J.vol);
}

template <class R>
__global__ void __launch_bounds__(kBlock) prepare_kappa_kernel(const FieldJob J)
{
    if (J.valid && blockIdx.x == 0 && threadIdx.x == 0 && J.valid->bad) atomicAdd(&J.st->bad_input, J.valid->bad);
    prepare_cells<R>(J, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(kBlock) finalize_kernel(const FieldJob J)
{
    // nothing goes to the caller's arrays from inputs found invalid, from a trace that reported an error or
    // from one that is not complete
    if (J.valid && (J.st->bad_input || J.st->err)) return;
    if (J.more && *J.more) return;
    finalize_cells(J, blockIdx.x, gridDim.x);
}

// The same over the solves of a batch in one launch: job j owns the blocks from its block0 up to the
// next job's (jobs[njobs].block0: all of them), so small grids do not each pay a launch and its tail.
__device__ __forceinline__ int job_of_block(const FieldJob* __restrict__ jobs, const int njobs)
{
    int lo = 0, hi = njobs;                       // jobs[lo].block0 <= blockIdx.x < jobs[hi].block0
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (jobs[mid].block0 <= blockIdx.x) lo = mid; else hi = mid;
    }
    return lo;
}

template <class R>
__global__ void __launch_bounds__(kBlock) prepare_many_kernel(const FieldJob* __restrict__ jobs, int njobs)
{
    const int j = job_of_block(jobs, njobs);
    const FieldJob J = jobs[j];
    prepare_cells<R>(J, blockIdx.x - J.block0, jobs[j + 1].block0 - J.block0);
}

__global__ void __launch_bounds__(kBlock) finalize_many_kernel(const FieldJob* __restrict__ jobs,
                                                               const FieldOut* __restrict__ outs,
                                                               const unsigned* err, int njobs)
{
    const unsigned failed = *err;                 // of any solve; requested with the search for the job
    const int j = job_of_block(jobs, njobs);
    FieldJob J = jobs[j];
    J.gamma_out = outs[j].gamma;
    J.heat = outs[j].heat;
    if (failed) return;                           // the run fails and no result is written
    finalize_cells(J, blockIdx.x - J.block0, jobs[j + 1].block0 - J.block0);
}

// One C2-Ray update at fixed Gamma (Eq. 3): with ionization rate
// I = Gamma + n_e C_H and recombination rate R = n_e C alpha_B constant over
// dt, x(dt) = x_eq + (x0 - x_eq) e^{-dt (I+R)} and the time average
// <x> = x_eq + (x0 - x_eq) (1 - e^{-dt (I+R)}) / (dt (I+R)); n_e = <x>_prev n_H (xavg: <x>_prev, the
// average the trace used; xnew: the new one).
__global__ void __launch_bounds__(kBlock) chem_kernel(const double* __restrict__ nh, const double* __restrict__ x0,
                                                      const double* __restrict__ xavg, double* __restrict__ xnew,
                                                      double* __restrict__ xend,
                                                      const double* __restrict__ gamma, int64_t ncell, double dt,
                                                      double alpha_B, double C_H, double clump,
                                                      const unsigned long long* more, DevStats* st)
{
    if (more && *more) return;
    double md = 0.0;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
        const double xp = xavg[c];
        const double ne = xp * nh[c];
        const double ion = gamma[c] + ne * C_H;
        const double tot = ion + ne * clump * alpha_B;
        double xe, xa;
        const double xs = x0[c];
        if (tot > 0.0) {
            const double xeq = ion / tot;
            const double u = dt * tot;
            xe = xeq + (xs - xeq) * exp(-u);
            xa = xeq + (xs - xeq) * (-expm1(-u) / u);
        } else {
            xe = xs;
            xa = xs;
        }
        md = fmax(md, fabs(xa - xp));
        xnew[c] = xa;
        xend[c] = xe;
    }
    for (int o = 16; o > 0; o >>= 1) md = fmax(md, __shfl_down_sync(0xffffffffu, md, o));
    // non-negative doubles order like their bit patterns: an integer max is exact
    if ((threadIdx.x & 31) == 0)
        atomicMax(reinterpret_cast<unsigned long long*>(&st->maxdiff), (unsigned long long)__double_as_longlong(md));
}

}  // namespace

int launch_check_fields(const double* nh, const double* x, int64_t ncell, double* nh_out, double* x_out, bool want_x,
                        FieldCheck* chk, cudaStream_t s)
{
    check_fields_kernel<<<(int)tiles_for(ncell), kBlock, 0, s>>>(nh, x, ncell, nh_out, x_out, want_x, chk);
    return 1;
}

int launch_prepare_kappa(const FieldJob& job, bool fp32, cudaStream_t s)
{
    FieldJob j = job;
    j.n_th = ordered_threshold(j.n_th);
    if (fp32) prepare_kappa_kernel<float><<<(int)tiles_for(j.ncell), kBlock, 0, s>>>(j);
    else prepare_kappa_kernel<double><<<(int)tiles_for(j.ncell), kBlock, 0, s>>>(j);
    return 1;
}

int launch_finalize(const FieldJob& j, cudaStream_t s)
{
    finalize_kernel<<<(int)tiles_for(j.ncell), kBlock, 0, s>>>(j);
    return 1;
}

// Four tiles a block: finding the job costs a block several dependent loads.
uint32_t field_blocks(int64_t ncell) { return (uint32_t)std::max<int64_t>(1, (ncell + 4 * kTile - 1) / (4 * kTile)); }

int launch_prepare_many(const FieldJob* jobs, int njobs, uint32_t blocks, bool fp32, cudaStream_t s)
{
    if (njobs <= 0) return 0;
    if (fp32) prepare_many_kernel<float><<<blocks, kBlock, 0, s>>>(jobs, njobs);
    else prepare_many_kernel<double><<<blocks, kBlock, 0, s>>>(jobs, njobs);
    return 1;
}

int launch_finalize_many(const FieldJob* jobs, const FieldOut* outs, const unsigned* err, int njobs, uint32_t blocks,
                         cudaStream_t s)
{
    if (njobs <= 0) return 0;
    finalize_many_kernel<<<blocks, kBlock, 0, s>>>(jobs, outs, err, njobs);
    return 1;
}

int launch_chem_update(const double* nh, const double* x0, const double* xavg, double* xnew, double* xend,
                       const double* gamma, int64_t ncell, double dt, double alpha_B, double C_H, double clump,
                       const unsigned long long* more, DevStats* st, cudaStream_t s)
{
    chem_kernel<<<grid_for(ncell), kBlock, 0, s>>>(nh, x0, xavg, xnew, xend, gamma, ncell, dt, alpha_B, C_H, clump, more,
                                                   st);
    return 1;
}

__global__ void __launch_bounds__(256) readback_kernel(const ReadbackList r)
{
    for (int k = 0; k < r.n; ++k)
        for (int i = threadIdx.x; i < r.words[k]; i += blockDim.x) r.dst[k][i] = r.src[k][i];
    __threadfence_system();
}

int launch_readback(const ReadbackList& r, cudaStream_t s)
{
    if (r.n == 0) return 0;
    readback_kernel<<<1, 256, 0, s>>>(r);
    return 1;
}

}  // namespace nyx
