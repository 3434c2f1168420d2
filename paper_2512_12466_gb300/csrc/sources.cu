// Source handling before the march (Sec. 2.8): sources that share a cell
// are merged by summing their rates, the catalog is sorted lexicographically
// by (ix, iy, iz), and optionally sources whose ionized bubbles overlap are
// merged (Alg. 3: MAX_RADIUS by shell sampling, union-find over overlapping
// pairs, one source per group at the member nearest the flux-weighted
// centroid). Every per-group sum runs sequentially in member order, so the
// emitted catalog is deterministic.
//
// The stage is bound by launches and by serial chains, not by bytes (32768
// sources are 0.7 MB): a catalog of up to kSmallSources is one launch of one
// block, a larger one a tiled radix sort (one block for all of it took 134 us
// at 32768 keys, the tiles take 33) and prefix sums folded into the kernels that need them. Sizes
// that the device counts (after dedup, of the positive radii, of the groups)
// stay there. The FP64 pipe (64 cycles a warp instruction) is kept for results.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "rt_internal.h"

namespace nyx {
namespace {

constexpr int kBlock = 256;

int blocks_for(int64_t count)
{
    const int64_t g = (count + kBlock - 1) / kBlock;
    return g < 1 ? 1 : (int)g;
}

// Bits per axis of a cell coordinate in [0, n).
int axis_bits(int n)
{
    int b = 0;
    while ((1LL << b) < (long long)n) ++b;
    return b;
}

// Lexicographic (x, y, z) key of a cell, b bits per axis.
__device__ __forceinline__ uint64_t cell_key(int x, int y, int z, int b)
{
    return ((uint64_t)x << (2 * b)) | ((uint64_t)y << b) | (uint64_t)z;
}

// A source that may not be traced: outside the grid, or a rate that is not positive and finite.
__device__ __forceinline__ bool bad_source(int x, int y, int z, double v, int n)
{
    const long long b = __double_as_longlong(v);
    return (unsigned)x >= (unsigned)n || (unsigned)y >= (unsigned)n || (unsigned)z >= (unsigned)n || b <= 0 ||
           b >= 0x7ff0000000000000ll;
}

// a / 12 correctly rounded: a times the rounded reciprocal, then one correction by the exact residual
// (Markstein 1990: with a correctly rounded reciprocal the corrected quotient is the rounded one). Three
// FP64 operations; a division's many, for 32 warps in one block, were a third of the small stage's time.
__device__ __forceinline__ double twelfth(const double a)
{
    const unsigned e = (unsigned)(__double_as_longlong(a) >> 52) & 0x7ffu;
    if (e - 128u > 1790u) return __ddiv_rn(a, 12.0);         // a residual may leave the normal range
    const double y = 1.0 / 12.0, q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-q, 12.0, a), y, q);
}

__device__ __forceinline__ SrcEntry emit_entry(int x, int y, int z, double ndot, double s_over_dx2)
{
    SrcEntry e;
    e.cx = x;
    e.cy = y;
    e.cz = z;
    e.pad = 0;
    e.ph = twelfth(ndot);
    e.gd = __dmul_rn(e.ph, s_over_dx2);
    e.gf = __double2float_rn(e.gd);
    e.pad2 = 0.f;
    return e;
}

// Inclusive prefix sum of one value per thread over a block of whole warps (up to 1024 threads); total:
// the block's sum.
__device__ __forceinline__ int block_scan(int v, int& total)
{
    __shared__ int part[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) part[w] = v;
    __syncthreads();
    if (w == 0) {
        int q = lane < nw ? part[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, q, o);
            if (lane >= o) q += u;
        }
        part[lane] = q;
    }
    __syncthreads();
    v += w > 0 ? part[w - 1] : 0;
    total = part[nw - 1];
    __syncthreads();
    return v;
}

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// The whole stage for up to kSmallSources sources in one block: validation, the stable sort by cell
// (bitonic on (cell key, index), which is unique), the sums over equal cells in index order, and the
// emitted catalog (emit null: only cells and rates). Ten launches and their gaps otherwise.
// The line at 2048 (16 KB of keys): the block's time grows with the catalog (a 64^3 opaque step takes 133 us
// with 1024 sources, 143 with 2048), the tiles' hardly (162 with 2049, 174 with 4096), so beyond it the two meet.
constexpr int kSmallSources = 2048;

__global__ void __launch_bounds__(1024) small_sources_kernel(const int32_t* __restrict__ cells,
                                                             const double* __restrict__ ndot, int m, int np2, int n,
                                                             int b, double s_over_dx2, int32_t* __restrict__ out_cells,
                                                             double* __restrict__ out_ndot, int32_t* count,
                                                             SrcEntry* __restrict__ emit, DevStats* st)
{
    __shared__ uint64_t key[kSmallSources];
    const int t = threadIdx.x, nt = blockDim.x;
    unsigned bad = 0;
    for (int i = t; i < np2; i += nt) {
        uint64_t k = ~0ULL;
        if (i < m) {
            const int x = cells[3 * i], y = cells[3 * i + 1], z = cells[3 * i + 2];
            bad += bad_source(x, y, z, ndot[i], n) ? 1u : 0u;
            k = (cell_key(x, y, z, b) << 32) | (uint64_t)(uint32_t)i;
        }
        key[i] = k;
    }
    if (bad) atomicAdd(&st->bad_input, bad);
    __syncthreads();
    // thread t holds entries t and t + nt (np2 > nt); exchanges within a warp's 32 are shuffles
    const int per = (np2 + nt - 1) / nt;
    for (int size = 2; size <= np2; size <<= 1) {
        int stride = size >> 1;
        for (; stride >= 32; stride >>= 1) {
            for (int q = t; q < np2 / 2; q += nt) {
                const int lo = 2 * q - (q & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint64_t ka = key[lo], kb = key[hi];
                if ((ka > kb) == up) { key[lo] = kb; key[hi] = ka; }
            }
            __syncthreads();
        }
        for (int u = 0; u < per; ++u) {
            const int i = t + u * nt;
            uint64_t k = key[i];
            for (int d = stride; d > 0; d >>= 1) {
                const uint64_t o = __shfl_xor_sync(0xffffffffu, k, d);
                const bool low = (i & d) == 0, up = (i & size) == 0;
                if ((k > o) == (low == up)) k = o;
            }
            key[i] = k;
        }
        __syncthreads();
    }
    double emitted = 0.0;
    int base = 0;
    for (int p0 = 0; p0 < m; p0 += nt) {
        const int p = p0 + t;
        const bool head = p < m && (p == 0 || (key[p] >> 32) != (key[p - 1] >> 32));
        int total;
        const int u = base + block_scan(head ? 1 : 0, total) - 1;
        base += total;
        if (head) {
            const int i = (int)(uint32_t)key[p];
            double s = ndot[i];
            for (int q = p + 1; q < m && (key[q] >> 32) == (key[p] >> 32); ++q)
                s = __dadd_rn(s, ndot[(int)(uint32_t)key[q]]);
            const int x = cells[3 * i], y = cells[3 * i + 1], z = cells[3 * i + 2];
            out_cells[3 * u] = x;
            out_cells[3 * u + 1] = y;
            out_cells[3 * u + 2] = z;
            out_ndot[u] = s;
            if (emit) emit[u] = emit_entry(x, y, z, s, s_over_dx2);
            emitted += s;
        }
    }
    if (t == 0) *count = base;
    if (emit) {
        emitted = warp_sum(emitted);
        if ((t & 31) == 0 && __double_as_longlong(emitted) << 1) atomicAdd(&st->emitted, emitted);
    }
}

// Cell keys of the sources, validated (st null: not). Entries at or beyond *m_dev (where given) get the
// largest key.
__global__ void cell_keys_kernel(const int32_t* __restrict__ cells, const double* __restrict__ ndot, int64_t m,
                                 const int32_t* __restrict__ m_dev, int n, int b, uint64_t* __restrict__ keys,
                                 DevStats* st)
{
    const int64_t have = m_dev ? *m_dev : m;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        if (i >= have) {
            keys[i] = ~0ULL;
            continue;
        }
        const int x = cells[3 * i], y = cells[3 * i + 1], z = cells[3 * i + 2];
        if (st && bad_source(x, y, z, ndot[i], n)) atomicAdd(&st->bad_input, 1u);
        keys[i] = cell_key(x, y, z, b);
    }
}

// Stable sort of keys[0..m) by 8 bits a pass, least significant first: a tile of kSortTile keys a block
// (a warp owns a contiguous chunk of it), two launches a pass. The first counts every tile's digits; the
// second takes each tile's base for a digit from the counts (all smaller digits, and the same digit in
// the tiles before), then each warp places its chunk in sequence order, 32 keys an iteration, a lane after
// the lower lanes that share its digit (8 ballots). 32768 keys of 24 bits: 33 us, one block for all 134.
constexpr int kSortTile = 1024;
constexpr int kSortBlocks = 512;
constexpr int kSortWarps = kBlock / 32;
constexpr int kSortChunk = kSortTile / kSortWarps;

__global__ void __launch_bounds__(kBlock) sort_count_kernel(const uint64_t* __restrict__ keys, int64_t m, int shift,
                                                            int parts, int32_t* __restrict__ hist)
{
    __shared__ int32_t cnt[256];
    const int t = threadIdx.x;
    cnt[t] = 0;
    __syncthreads();
    for (int part = 0; part < parts; ++part) {
        const int64_t i0 = (blockIdx.x * (int64_t)parts + part) * kSortTile;
#pragma unroll
        for (int u = 0; u < kSortTile / kBlock; ++u) {
            const int64_t i = i0 + u * kBlock + t;
            if (i < m) atomicAdd(&cnt[(int)(keys[i] >> shift) & 255], 1);
        }
    }
    __syncthreads();
    hist[blockIdx.x * 256 + t] = cnt[t];
}

__global__ void __launch_bounds__(kBlock) sort_place_kernel(const uint64_t* __restrict__ keys,
                                                            const int32_t* __restrict__ idx, int64_t m, int shift,
                                                            int parts, const int32_t* __restrict__ hist,
                                                            uint64_t* __restrict__ keys_out,
                                                            int32_t* __restrict__ idx_out)
{
    __shared__ int32_t slot[kSortWarps][257];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    // digit t: its count in all tiles and in those before this one
    int all = 0, before = 0;
#pragma unroll 8
    for (int q = 0; q < (int)gridDim.x; ++q) {
        const int v = hist[q * 256 + t];
        all += v;
        before += q < (int)blockIdx.x ? v : 0;
    }
    int total;
    int at = block_scan(all, total) - all + before;
    for (int part = 0; part < parts; ++part) {
        for (int q = t; q < kSortWarps * 257; q += kBlock) (&slot[0][0])[q] = 0;
        __syncthreads();
        const int64_t c0 = (blockIdx.x * (int64_t)parts + part) * kSortTile + w * kSortChunk;
        uint64_t k[kSortChunk / 32];
        int32_t x[kSortChunk / 32];
#pragma unroll
        for (int u = 0; u < kSortChunk / 32; ++u) {
            const int64_t i = c0 + 32 * u + lane;
            k[u] = i < m ? keys[i] : 0ULL;
            x[u] = i < m ? (idx ? idx[i] : (int32_t)i) : 0;
            if (i < m) atomicAdd(&slot[w][(int)(k[u] >> shift) & 255], 1);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kSortWarps; ++q) {
            const int v = slot[q][t];
            slot[q][t] = at;
            at += v;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kSortChunk / 32; ++u) {
            const int64_t i = c0 + 32 * u + lane;
            const bool v = i < m;
            const int d = (int)(k[u] >> shift) & 255;
            unsigned peers = __ballot_sync(0xffffffffu, v);
#pragma unroll
            for (int bit = 0; bit < 8; ++bit) {
                const unsigned bb = __ballot_sync(0xffffffffu, (d >> bit) & 1);
                peers &= ((d >> bit) & 1) ? bb : ~bb;
            }
            if (v) {
                const int32_t dst = slot[w][d] + __popc(peers & ((1u << lane) - 1u));
                keys_out[dst] = k[u];
                idx_out[dst] = x[u];
            }
            __syncwarp();
            if (v && (peers >> lane) == 1u) slot[w][d] += __popc(peers);   // the highest lane of its digit
            __syncwarp();
        }
        __syncthreads();
    }
}

// Runs of equal sorted keys: flag[p] = 1 where entry p < m starts one, and each block's number of runs
// (blocks of kBlock entries). Entries at or beyond *m_dev (where given) start none.
__global__ void __launch_bounds__(kBlock) run_heads_kernel(const uint64_t* __restrict__ sorted, int64_t m,
                                                           const int32_t* __restrict__ m_dev,
                                                           int32_t* __restrict__ flag, int32_t* __restrict__ bsum)
{
    const int64_t have = m_dev ? *m_dev : m;
    const int64_t p = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const bool head = p < have && (p == 0 || sorted[p] != sorted[p - 1]);
    if (p < m) flag[p] = head ? 1 : 0;
    const int c = __syncthreads_count(head);
    if (threadIdx.x == 0) bsum[blockIdx.x] = c;
}

// Exclusive position of this thread's flag among all blocks' (bsum from the kernel that set them); the
// last block's total goes to *total.
__device__ __forceinline__ int flag_position(const int f, const int32_t* __restrict__ bsum, int32_t* total)
{
    int before = 0;
    for (int q = threadIdx.x; q < (int)blockIdx.x; q += kBlock) before += bsum[q];
    int sum_before, mine;
    block_scan(before, sum_before);
    const int pos = sum_before + block_scan(f, mine) - f;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = sum_before + mine;
    return pos;
}

// For each run head: sum the rates of the run in sorted (= input) order.
__global__ void __launch_bounds__(kBlock) dedup_sum_kernel(const int32_t* __restrict__ order,
                                                           const int32_t* __restrict__ flag,
                                                           const int32_t* __restrict__ bsum, int64_t m,
                                                           const int32_t* __restrict__ cells,
                                                           const double* __restrict__ ndot,
                                                           int32_t* __restrict__ out_cells,
                                                           double* __restrict__ out_ndot, int32_t* count)
{
    const int64_t p = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const int f = p < m ? flag[p] : 0;
    const int u = flag_position(f, bsum, count);
    if (!f) return;
    const int32_t i = order[p];
    double s = ndot[i];
    for (int64_t q = p + 1; q < m && !flag[q]; ++q) s = __dadd_rn(s, ndot[order[q]]);
    out_cells[3 * u] = cells[3 * i];
    out_cells[3 * u + 1] = cells[3 * i + 1];
    out_cells[3 * u + 2] = cells[3 * i + 2];
    out_ndot[u] = s;
}

// ---------------------------------------------------------------- Alg. 3

// Minimum-image component of a cell offset on a periodic grid of n cells
// (Sec. 2.8 computes Alg. 3 under minimum-image geometry when periodic).
__device__ __forceinline__ long long minimg(long long d, long long n)
{
    long long r = d % n;
    if (r < 0) r += n;
    return 2 * r > n ? r - n : r;
}

// MAX_RADIUS: one block per source. Shells r = dr, 2 dr, ... <= R_max are
// sampled at the HEALPix directions of the sample level; a sample is the
// cell floor(c + 1/2 + r d), wrapped into the grid when periodic; the shell's
// point set is the distinct in-grid sample cells (bitonic sort in shared
// memory, then run heads).
template <int NP2>
__global__ void __launch_bounds__(kBlock) radius_kernel(const int32_t* __restrict__ cells,
                                                        const int32_t* __restrict__ m_dev, int n,
                                                        const double* __restrict__ x, const int4* __restrict__ dirs,
                                                        int ns, double x_th, double f_req, int n_min, double dr,
                                                        double rmax, int periodic, double* __restrict__ radius)
{
    __shared__ long long key[NP2];
    __shared__ int red[2];
    const int64_t si = blockIdx.x;
    if (si >= *m_dev) return;
    const int c[3] = {cells[3 * si], cells[3 * si + 1], cells[3 * si + 2]};
    const int64_t nn = n;
    const bool in = (unsigned)c[0] < (unsigned)n && (unsigned)c[1] < (unsigned)n && (unsigned)c[2] < (unsigned)n;
    if (!in || x[((int64_t)c[2] * nn + c[1]) * nn + c[0]] < x_th) {
        if (threadIdx.x == 0) radius[si] = 0.0;
        return;
    }
    const double inv = 1.0 / (double)(1 << kDirBits);
    double result = rmax;
    for (double r = dr; r <= rmax; r = __dadd_rn(r, dr)) {
        for (int p = threadIdx.x; p < NP2; p += blockDim.x) {
            long long k = 0x7fffffffffffffffLL;
            if (p < ns) {
                const int4 d = dirs[p];
                const int dd[3] = {d.x, d.y, d.z};
                long long q[3];
                bool inside = true;
                for (int a = 0; a < 3; ++a) {
                    const double pos = __dadd_rn(__dadd_rn((double)c[a], 0.5), __dmul_rn(r, __dmul_rn((double)dd[a], inv)));
                    q[a] = (long long)floor(pos);
                    if (periodic) q[a] = ((q[a] % nn) + nn) % nn;
                    if (q[a] < 0 || q[a] >= nn) inside = false;
                }
                if (inside) k = (q[2] * nn + q[1]) * nn + q[0];
            }
            key[p] = k;
        }
        __syncthreads();
        for (int size = 2; size <= NP2; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int t = threadIdx.x; t < NP2 / 2; t += blockDim.x) {
                    const int lo = 2 * t - (t & (stride - 1));
                    const int hi = lo + stride;
                    const bool up = ((lo & size) == 0);
                    const long long a = key[lo], b = key[hi];
                    if ((a > b) == up) { key[lo] = b; key[hi] = a; }
                }
                __syncthreads();
            }
        }
        if (threadIdx.x < 2) red[threadIdx.x] = 0;
        __syncthreads();
        int ntot = 0, nion = 0;
        for (int p = threadIdx.x; p < NP2; p += blockDim.x) {
            const long long k = key[p];
            if (k != 0x7fffffffffffffffLL && (p == 0 || key[p - 1] != k)) {
                ++ntot;
                if (x[k] >= x_th) ++nion;
            }
        }
        atomicAdd(&red[0], ntot);
        atomicAdd(&red[1], nion);
        __syncthreads();
        ntot = red[0];
        nion = red[1];
        bool fail;
        if (ntot < n_min) fail = nion < ntot;
        else fail = __ddiv_rn((double)nion, (double)ntot) < f_req;
        __syncthreads();
        if (fail) {
            result = __dsub_rn(r, dr);
            break;
        }
    }
    if (threadIdx.x == 0) radius[si] = result;
}

// MAX_RADIUS where every shell's sample positions are exact in FP64 (r a multiple of 2^-10 below 512:
// r times a direction of 21 fraction bits, and the sum with c + 1/2, then keep all their bits): a sample
// cell is c plus floor(1/2 + r d), the same offset for every source. So the distinct offsets of each shell
// are found once (shell_kernel, a block a shell) and a source only looks its cells up, a warp each. With
// periodic boundaries the grid has to be wider than the largest shell, so that no two offsets meet.
// 29815 sources of a 256^3 box: 72 us (13 for the tables), against 376 with radius_kernel (a sort of every
// shell of every source).
constexpr int kMaxShells = 128;
constexpr int kShellBias = 512;

template <int NP2>
__global__ void __launch_bounds__(kBlock) shell_kernel(const int4* __restrict__ dirs, int ns, double dr,
                                                       uint32_t* __restrict__ offs, int32_t* __restrict__ counts)
{
    __shared__ uint32_t key[NP2];
    double r = dr;
    for (int k = 0; k < (int)blockIdx.x; ++k) r = __dadd_rn(r, dr);
    const long long rfx = __double2ll_rn(__dmul_rn(r, 1024.0));
    for (int p = threadIdx.x; p < NP2; p += blockDim.x) {
        uint32_t k = 0xffffffffu;
        if (p < ns) {
            const int4 d = dirs[p];
            const long long half = 1LL << (9 + kDirBits);
            const uint32_t ox = (uint32_t)(((rfx * d.x + half) >> (10 + kDirBits)) + kShellBias);
            const uint32_t oy = (uint32_t)(((rfx * d.y + half) >> (10 + kDirBits)) + kShellBias);
            const uint32_t oz = (uint32_t)(((rfx * d.z + half) >> (10 + kDirBits)) + kShellBias);
            k = (oz << 20) | (oy << 10) | ox;
        }
        key[p] = k;
    }
    __syncthreads();
    for (int size = 2; size <= NP2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < NP2 / 2; t += blockDim.x) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint32_t a = key[lo], b = key[hi];
                if ((a > b) == up) { key[lo] = b; key[hi] = a; }
            }
            __syncthreads();
        }
    int base = 0;
    for (int p0 = 0; p0 < NP2; p0 += kBlock) {
        const int p = p0 + threadIdx.x;
        const bool head = key[p] != 0xffffffffu && (p == 0 || key[p - 1] != key[p]);
        int total;
        const int u = base + block_scan(head ? 1 : 0, total) - 1;
        base += total;
        if (head) offs[blockIdx.x * (int64_t)NP2 + u] = key[p];
    }
    if (threadIdx.x == 0) counts[blockIdx.x] = base;
}

__global__ void __launch_bounds__(kBlock) shell_radius_kernel(const int32_t* __restrict__ cells,
                                                              const int32_t* __restrict__ m_dev, int n,
                                                              const double* __restrict__ x,
                                                              const uint32_t* __restrict__ offs,
                                                              const int32_t* __restrict__ counts, int pitch, int nshell,
                                                              double x_th, double f_req, int n_min, double dr,
                                                              double rmax, int periodic, double* __restrict__ radius)
{
    const int64_t m = *m_dev;
    const int lane = threadIdx.x & 31;
    const long long th = __double_as_longlong(x_th);       // x_th > 0 and x >= 0: ordered by their bits
    const float fq = (float)f_req;
    for (int64_t si = (blockIdx.x * (int64_t)kBlock + threadIdx.x) >> 5; si < m; si += (int64_t)gridDim.x * (kBlock / 32)) {
        const int c0 = cells[3 * si], c1 = cells[3 * si + 1], c2 = cells[3 * si + 2];
        double result = 0.0;
        // (a source outside the grid ends the step with an error; it reads nothing here)
        const bool in = (unsigned)c0 < (unsigned)n && (unsigned)c1 < (unsigned)n && (unsigned)c2 < (unsigned)n;
        if (in && __double_as_longlong(x[((int64_t)c2 * n + c1) * n + c0]) >= th) {
            result = rmax;
            double r = dr;
            for (int k = 0; k < nshell; ++k) {
                int ntot = 0, nion = 0;
                const int cnt = counts[k];
                for (int p = lane; p < cnt; p += 32) {
                    const uint32_t o = offs[k * (int64_t)pitch + p];
                    int q0 = c0 + (int)(o & 1023u) - kShellBias, q1 = c1 + (int)((o >> 10) & 1023u) - kShellBias,
                        q2 = c2 + (int)(o >> 20) - kShellBias;
                    if (periodic) {
                        q0 = q0 < 0 ? q0 + n : (q0 >= n ? q0 - n : q0);
                        q1 = q1 < 0 ? q1 + n : (q1 >= n ? q1 - n : q1);
                        q2 = q2 < 0 ? q2 + n : (q2 >= n ? q2 - n : q2);
                    }
                    if ((unsigned)q0 < (unsigned)n && (unsigned)q1 < (unsigned)n && (unsigned)q2 < (unsigned)n) {
                        ++ntot;
                        nion += __double_as_longlong(x[((int64_t)q2 * n + q1) * n + q0]) >= th ? 1 : 0;
                    }
                }
                ntot = __reduce_add_sync(0xffffffffu, ntot);
                nion = __reduce_add_sync(0xffffffffu, nion);
                bool fail;
                if (ntot < n_min) {
                    fail = nion < ntot;
                } else {
                    // the quotient in float where that settles it, in FP64 next to f_req
                    const float d = __fdividef((float)nion, (float)ntot) - fq;
                    fail = fabsf(d) > 1e-4f ? d < 0.f : __ddiv_rn((double)nion, (double)ntot) < f_req;
                }
                if (fail) {
                    result = __dsub_rn(r, dr);
                    break;
                }
                r = __dadd_rn(r, dr);
            }
        }
        if (lane == 0) radius[si] = result;
    }
}

// Root of a in the union-find forest; parents are read past L1 (they change under concurrent hooks,
// which are atomicCAS on roots, so a stale read only lengthens the walk or fails a CAS that retries).
// A node more than one step below its root is hooked to the root directly (an ancestor it has anyway, and
// it is no root, which alone a CAS changes), so that later walks are short.
__device__ __forceinline__ int uf_find(int* parent, int a)
{
    const int first = a;
    int steps = 0, p = __ldcg(&parent[a]);
    while (p != a) {
        a = p;
        p = __ldcg(&parent[a]);
        ++steps;
    }
    if (steps > 1) __stcg(&parent[first], a);
    return a;
}

// The union-find forest of single sources, flag[i] = 1 where source i has a positive bubble radius (only
// such sources can pair), and each block's number of them.
__global__ void __launch_bounds__(kBlock) positive_radius_kernel(const double* __restrict__ radius, int64_t m,
                                                                 const int32_t* __restrict__ m_dev, int* parent,
                                                                 int32_t* __restrict__ flag, int32_t* __restrict__ bsum)
{
    const int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const bool pos = i < *m_dev && __double_as_longlong(radius[i]) > 0;
    if (i < m) {
        parent[i] = (int)i;
        flag[i] = pos ? 1 : 0;
    }
    const int c = __syncthreads_count(pos);
    if (threadIdx.x == 0) bsum[blockIdx.x] = c;
}

// One source of the pair test: its cell, its radius rounded to float and its index.
struct PairEntry {
    short x, y, z, pad;
    float r;
    int i;
};

// The flagged sources in index order, their number in *np.
__global__ void __launch_bounds__(kBlock) compact_kernel(const int32_t* __restrict__ flag,
                                                         const int32_t* __restrict__ bsum, int64_t m,
                                                         const int32_t* __restrict__ cells,
                                                         const double* __restrict__ radius,
                                                         PairEntry* __restrict__ list, int32_t* np)
{
    const int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const int f = i < m ? flag[i] : 0;
    const int u = flag_position(f, bsum, np);
    if (f)
        list[u] = {(short)cells[3 * i], (short)cells[3 * i + 1], (short)cells[3 * i + 2], 0,
                   __double2float_rn(radius[i]), (int)i};
}

// Pairs of the *np_dev sources of `list` (positive radii, increasing index) whose bubbles
// overlap (d^2 <= (f_ov (r_a + r_b))^2 + eps, d minimum-image when periodic) are united; the
// larger root is hooked under the smaller, so each component's root is its smallest index. A block takes
// a tile of kBlock x kPairTile pairs: a thread one source against the tile's others, in shared memory.
// Almost all pairs are far apart, which integer and float arithmetic settles (the float limit is above
// the FP64 one by more than its rounding); the others take the exact test. 88 us for the ionized
// sources among 29815; 161 with the exact test for every pair.
constexpr int kPairTile = 256;

// minimg of an offset between two cells of the grid, |d| < n
__device__ __forceinline__ int near_image(int d, int n)
{
    d = d < 0 ? d + n : d;
    return 2 * d > n ? d - n : d;
}

__device__ __forceinline__ void unite(const int a, const int b, int* parent, DevStats* st)
{
    int u = a, v = b;
    for (int tries = 0;; ++tries) {
        u = uf_find(parent, u);
        v = uf_find(parent, v);
        if (u == v) break;
        if (u > v) { const int t = u; u = v; v = t; }
        if (atomicCAS(&parent[v], v, u) == v) break;
        if (tries > (1 << 20)) { atomicOr(&st->err, kErrUnionFind); break; }
    }
}

__global__ void __launch_bounds__(kBlock) pair_union_kernel(const double* __restrict__ radius,
                                                            const PairEntry* __restrict__ list,
                                                            const int32_t* __restrict__ np_dev, int n, int periodic,
                                                            double f_ov, double eps, int* parent, DevStats* st)
{
    __shared__ PairEntry tile[kPairTile];
    const long long np = *np_dev;
    const long long rows = (np + kBlock - 1) / kBlock, cols = (np + kPairTile - 1) / kPairTile;
    const float f_f = (float)f_ov, eps_f = fmaxf((float)eps, 0.f) * 1.0001f + 1e-30f;
    for (long long q = blockIdx.x; q < rows * cols; q += gridDim.x) {
        const long long a0 = q / cols * kBlock, b0 = q % cols * kPairTile;
        if (b0 + kPairTile <= a0) continue;                // only pairs ia < ib
        __syncthreads();
        for (int t = threadIdx.x; t < kPairTile; t += kBlock)
            if (b0 + t < np) tile[t] = list[b0 + t];
        __syncthreads();
        const long long ia = a0 + threadIdx.x;
        if (ia >= np) continue;
        const PairEntry A = list[ia];
        const int last = (int)(np - b0 < kPairTile ? np - b0 : kPairTile);
        for (int t = ia + 1 > b0 ? (int)(ia + 1 - b0) : 0; t < last; ++t) {
            const PairEntry B = tile[t];
            int dx = A.x - B.x, dy = A.y - B.y, dz = A.z - B.z;
            if (periodic) {
                dx = near_image(dx, n);
                dy = near_image(dy, n);
                dz = near_image(dz, n);
            }
            const int d2 = dx * dx + dy * dy + dz * dz;
            const float rf = f_f * (A.r + B.r);
            if ((float)d2 > rf * rf * 1.0001f + eps_f) continue;
            const double rs = __dmul_rn(f_ov, __dadd_rn(radius[A.i], radius[B.i]));
            if ((double)d2 <= __dadd_rn(__dmul_rn(rs, rs), eps)) unite(A.i, B.i, parent, st);
        }
    }
}

// Key of source i: its component's root (a stable sort by it keeps members in index order).
// Entries at or beyond *m_dev sort last.
__global__ void label_keys_kernel(int* parent, int64_t m, const int32_t* __restrict__ m_dev,
                                  uint64_t* __restrict__ keys)
{
    const int64_t have = *m_dev;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        keys[i] = i < have ? (uint64_t)(uint32_t)uf_find(parent, (int)i) : ~0ULL;
    }
}

// One merged source per group (members contiguous in `order`, by index):
// summed rate, flux-weighted centroid rounded and clamped into the grid,
// snapped to the nearest member (first in order on ties). Periodic: members
// unwrapped next to the group's first member, centroid wrapped back into the
// grid, snap by minimum-image distance.
__global__ void __launch_bounds__(kBlock) group_kernel(const int32_t* __restrict__ order,
                                                       const int32_t* __restrict__ flag,
                                                       const int32_t* __restrict__ bsum, int64_t m_bound,
                                                       const int32_t* __restrict__ m_dev, int n, int periodic,
                                                       const int32_t* __restrict__ cells,
                                                       const double* __restrict__ ndot,
                                                       int32_t* __restrict__ out_cells, double* __restrict__ out_ndot,
                                                       int32_t* count)
{
    const int64_t m = *m_dev;
    const int64_t p = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const int f = p < m_bound ? flag[p] : 0;
    const int32_t u = flag_position(f, bsum, count);
    if (f) {
        int64_t e = p + 1;
        while (e < m && !flag[e]) ++e;
        const int32_t g = order[p];
        if (e - p == 1) {
            out_cells[3 * u] = cells[3 * g];
            out_cells[3 * u + 1] = cells[3 * g + 1];
            out_cells[3 * u + 2] = cells[3 * g + 2];
            out_ndot[u] = ndot[g];
            return;
        }
        double ftot = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
        for (int64_t q = p; q < e; ++q) {
            const int32_t j = order[q];
            const double v = ndot[j];
            long long w[3] = {cells[3 * j], cells[3 * j + 1], cells[3 * j + 2]};
            if (periodic)
                for (int a = 0; a < 3; ++a) w[a] = cells[3 * g + a] + minimg(w[a] - cells[3 * g + a], n);
            ftot = __dadd_rn(ftot, v);
            sx = __dadd_rn(sx, __dmul_rn(v, (double)w[0]));
            sy = __dadd_rn(sy, __dmul_rn(v, (double)w[1]));
            sz = __dadd_rn(sz, __dmul_rn(v, (double)w[2]));
        }
        long long rc[3];
        const double cs[3] = {sx, sy, sz};
        for (int a = 0; a < 3; ++a) {
            long long v = (long long)floor(__dadd_rn(__ddiv_rn(cs[a], ftot), 0.5));
            if (periodic) v = ((v % n) + n) % n;
            else v = v < 0 ? 0 : (v > n - 1 ? n - 1 : v);
            rc[a] = v;
        }
        int32_t best = -1;
        long long bestd = 0;
        for (int64_t q = p; q < e; ++q) {
            const int32_t j = order[q];
            long long d2 = 0;
            for (int a = 0; a < 3; ++a) {
                long long d = (long long)cells[3 * j + a] - rc[a];
                if (periodic) d = minimg(d, n);
                d2 += d * d;
            }
            if (best < 0 || d2 < bestd) { best = j; bestd = d2; }
        }
        out_cells[3 * u] = cells[3 * best];
        out_cells[3 * u + 1] = cells[3 * best + 1];
        out_cells[3 * u + 2] = cells[3 * best + 2];
        out_ndot[u] = ftot;
    }
}

// The catalog in `order` (null: as it is) and the emitted entries (emit null: none) of its first *count
// sources.
__global__ void __launch_bounds__(kBlock) emit_kernel(const int32_t* __restrict__ order,
                                                      const int32_t* __restrict__ cells,
                                                      const double* __restrict__ ndot,
                                                      const int32_t* __restrict__ count, double s_over_dx2,
                                                      int32_t* __restrict__ out_cells, double* __restrict__ out_ndot,
                                                      SrcEntry* __restrict__ emit, DevStats* st)
{
    const int64_t m = *count;
    double emitted = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)kBlock + threadIdx.x; p < m; p += (int64_t)gridDim.x * kBlock) {
        const int64_t i = order ? order[p] : p;
        const int x = cells[3 * i], y = cells[3 * i + 1], z = cells[3 * i + 2];
        const double v = ndot[i];
        if (order) {
            out_cells[3 * p] = x;
            out_cells[3 * p + 1] = y;
            out_cells[3 * p + 2] = z;
            out_ndot[p] = v;
        }
        if (emit) {
            emit[p] = emit_entry(x, y, z, v, s_over_dx2);
            emitted += v;
        }
    }
    if (!emit) return;
    emitted = warp_sum(emitted);
    if ((threadIdx.x & 31) == 0 && __double_as_longlong(emitted) << 1) atomicAdd(&st->emitted, emitted);
}

// Stable sort of w.keys[0..m) by their low `bits` bits into w.order; returns the sorted keys (w.keys is
// left as it is; w.flag is scratch for the tile counts: m / 4 of its m entries, 256 at least).
const uint64_t* sort_keys(SourceWork& w, int64_t m, int bits, int* launches, cudaStream_t s)
{
    // at most kSortBlocks blocks, of several tiles each if need be: every block reads all blocks' counts
    const int64_t tiles = (m + kSortTile - 1) / kSortTile;
    const int parts = (int)((tiles + kSortBlocks - 1) / kSortBlocks);
    const int blocks = (int)((tiles + parts - 1) / parts);
    const int passes = std::max(1, (bits + 7) / 8);
    const uint64_t* kin = w.keys;
    const int32_t* iin = nullptr;                              // the first pass reads the identity
    uint64_t* kout = w.keys_b;
    int32_t* iout = (passes & 1) ? w.order : w.order_b;        // the last pass writes w.order
    for (int pass = 0; pass < passes; ++pass) {
        sort_count_kernel<<<blocks, kBlock, 0, s>>>(kin, m, 8 * pass, parts, w.flag);
        sort_place_kernel<<<blocks, kBlock, 0, s>>>(kin, iin, m, 8 * pass, parts, w.flag, kout, iout);
        *launches += 2;
        kin = kout;
        kout = kout == w.keys_b ? w.keys_c : w.keys_b;
        iin = iout;
        iout = iout == w.order ? w.order_b : w.order;
    }
    return kin;
}

// Shells of Alg. 3 that shell_kernel can tabulate, 0: none (see there).
int exact_shells(const MergeParams& p, int n, int periodic)
{
    if (!(p.x_th > 0) || !(p.dr > 0) || p.dr * 1024.0 != std::floor(p.dr * 1024.0)) return 0;
    int k = 0;
    double r = p.dr;
    for (; r <= p.rmax; r += p.dr)                             // every r stays a multiple of 2^-10
        if (++k > kMaxShells || r > 500.0) return 0;
    if (periodic && 2 * ((int)std::ceil(r) + 1) + 1 > n) return 0;
    return k;
}

__global__ void __launch_bounds__(kBlock) copy_sources_kernel(const int32_t* __restrict__ cells,
                                                              const double* __restrict__ ndot, int64_t n,
                                                              int32_t* __restrict__ to_cells,
                                                              double* __restrict__ to_ndot)
{
    for (int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x; i < 3 * n; i += (int64_t)gridDim.x * kBlock) {
        to_cells[i] = cells[i];
        if (i < n) to_ndot[i] = ndot[i];
    }
}

}  // namespace

int launch_copy_sources(const int32_t* cells, const double* ndot, int64_t n, int32_t* to_cells, double* to_ndot,
                        cudaStream_t s)
{
    copy_sources_kernel<<<std::min(blocks_for(3 * n), 152 * 8), kBlock, 0, s>>>(cells, ndot, n, to_cells, to_ndot);
    return 1;
}

int launch_sources(SourceWork& w, int64_t nsrc, int n, double s_over_dx2, SrcEntry* emit, DevStats* st, cudaStream_t s)
{
    if (nsrc <= 0) return 0;
    const int ab = axis_bits(n);
    if (nsrc <= kSmallSources) {
        int np2 = 32;
        while (np2 < nsrc) np2 <<= 1;
        const int threads = std::min(1024, np2);
        small_sources_kernel<<<1, threads, 0, s>>>(w.cells_raw, w.ndot_raw, (int)nsrc, np2, n, ab, s_over_dx2, w.cells_a,
                                                   w.ndot_a, w.count, emit, st);
        return 1;
    }
    const int b = blocks_for(nsrc);
    int launches = 3;
    cell_keys_kernel<<<b, kBlock, 0, s>>>(w.cells_raw, w.ndot_raw, nsrc, nullptr, n, ab, w.keys, st);
    const uint64_t* sorted = sort_keys(w, nsrc, 3 * ab, &launches, s);
    run_heads_kernel<<<b, kBlock, 0, s>>>(sorted, nsrc, nullptr, w.flag, w.head_pos);
    dedup_sum_kernel<<<b, kBlock, 0, s>>>(w.order, w.flag, w.head_pos, nsrc, w.cells_raw, w.ndot_raw, w.cells_a, w.ndot_a,
                                          w.count);
    if (emit) launches += launch_emit(w, nsrc, w.count, s_over_dx2, emit, st, s);
    return launches;
}

int launch_emit(const SourceWork& w, int64_t bound, const int32_t* count, double s_over_dx2, SrcEntry* emit,
                DevStats* st, cudaStream_t s)
{
    if (bound <= 0) return 0;
    emit_kernel<<<std::min(blocks_for(bound), 1024), kBlock, 0, s>>>(nullptr, w.cells_a, w.ndot_a, count, s_over_dx2,
                                                                     nullptr, nullptr, emit, st);
    return 1;
}

int launch_merge(SourceWork& w, int64_t bound, int n, int periodic, const double* x, const int4* samp_dirs,
                 int samp_count, const MergeParams& p, double s_over_dx2, SrcEntry* emit, DevStats* st, cudaStream_t s)
{
    if (bound <= 0) return 0;
    const int b = blocks_for(bound);
    const int32_t* const m_dev = w.count;
    int launches = 7;
    const int np2 = samp_count <= 1024 ? 1024 : 4096;
    const int shells = exact_shells(p, n, periodic);
    // the shell tables live where the pair test's sources go later: np2 offsets and a count each
    if (shells > 0 && (int64_t)shells * np2 * 4 <= (int64_t)pair_bytes(w.cap)) {
        uint32_t* const offs = static_cast<uint32_t*>(w.pairs);
        int32_t* const counts = w.order;
        if (np2 == 1024) shell_kernel<1024><<<shells, kBlock, 0, s>>>(samp_dirs, samp_count, p.dr, offs, counts);
        else shell_kernel<4096><<<shells, kBlock, 0, s>>>(samp_dirs, samp_count, p.dr, offs, counts);
        shell_radius_kernel<<<std::min<int64_t>((bound + 7) / 8, 152 * 16), kBlock, 0, s>>>(
            w.cells_a, m_dev, n, x, offs, counts, np2, shells, p.x_th, p.f_req, p.n_min, p.dr, p.rmax, periodic, w.radius);
        launches += 2;
    } else {
        if (np2 == 1024)
            radius_kernel<1024><<<(int)bound, kBlock, 0, s>>>(w.cells_a, m_dev, n, x, samp_dirs, samp_count, p.x_th,
                                                              p.f_req, p.n_min, p.dr, p.rmax, periodic, w.radius);
        else
            radius_kernel<4096><<<(int)bound, kBlock, 0, s>>>(w.cells_a, m_dev, n, x, samp_dirs, samp_count, p.x_th,
                                                              p.f_req, p.n_min, p.dr, p.rmax, periodic, w.radius);
        launches += 1;
    }
    // the sources with a positive radius, compacted (count[1]: how many)
    PairEntry* const list = static_cast<PairEntry*>(w.pairs);
    positive_radius_kernel<<<b, kBlock, 0, s>>>(w.radius, bound, m_dev, w.parent, w.flag, w.head_pos);
    compact_kernel<<<b, kBlock, 0, s>>>(w.flag, w.head_pos, bound, w.cells_a, w.radius, list, w.count + 1);
    pair_union_kernel<<<std::min(b * 64, 152 * 8), kBlock, 0, s>>>(w.radius, list, w.count + 1, n, periodic, p.f_ov,
                                                                    p.eps, w.parent, st);
    // groups: members contiguous under their root, in index order (roots are below `bound`; the tail's
    // keys are larger than any)
    label_keys_kernel<<<b, kBlock, 0, s>>>(w.parent, bound, m_dev, w.keys);
    const uint64_t* sorted = sort_keys(w, bound, axis_bits((int)std::min<int64_t>(bound + 1, 1LL << 30)), &launches, s);
    run_heads_kernel<<<b, kBlock, 0, s>>>(sorted, bound, m_dev, w.flag, w.head_pos);
    group_kernel<<<b, kBlock, 0, s>>>(w.order, w.flag, w.head_pos, bound, m_dev, n, periodic, w.cells_a, w.ndot_a,
                                      w.cells_b, w.ndot_b, w.count + 2);
    // final lexicographic order of the merged catalog, emitted from there
    const int ab = axis_bits(n);
    cell_keys_kernel<<<b, kBlock, 0, s>>>(w.cells_b, nullptr, bound, w.count + 2, n, ab, w.keys, nullptr);
    sort_keys(w, bound, 3 * ab, &launches, s);      // a tail key may tie with the last cell's: it stays behind
    emit_kernel<<<std::min(b, 1024), kBlock, 0, s>>>(w.order, w.cells_b, w.ndot_b, w.count + 2, s_over_dx2, w.cells_a,
                                                     w.ndot_a, emit, st);
    return launches + 1;
}

}  // namespace nyx
