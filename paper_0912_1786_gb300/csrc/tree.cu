// Tree build on the GPU (Sect. 2.2 of the paper): root cube, 63-bit Morton keys, stable sort,
// particle permutation, pre-order octree from the sorted keys, and node moments
// reduced bottom-up.
//
// Node construction does not insert particles one by one.  With keys sorted, the cells of
// level l are the maximal runs of keys sharing their top 3l bits; a cell is a node iff its
// parent cell holds more than `leaf` particles (the root always is).  Writing d_i for the
// number of leading octal digits that keys i-1 and i share, position i begins a level-l cell
// iff d_i < l, so the nodes beginning at i are the levels d_i+1 .. (last level whose parent
// holds > leaf particles).  Counting them per position and scanning gives every node its
// pre-order index directly (pre-order = sorted by (begin, level)); the first child of an
// internal node is the next index and the subtree skip pointer is the first node beginning
// at the node's end.
#include <cuda_runtime.h>
#include <stdint.h>

#include "evol_internal.cuh"

namespace {

constexpr int BB_THREADS = 256;
constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int SC_THREADS = 1024;
constexpr int SC_ITEMS = 4;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;
// The sort's three forms, by size; whole tree builds of a Plummer sphere on one GB300, ms.  Up to RANK_MAX
// each key's position is counted directly, n^2 comparisons in one launch (against fused passes: 4095
// particles 0.146 / 0.196, 8191 0.181 / 0.223, 12000 0.205 / 0.237, 24000 0.275 / 0.241).  Up to FUSED_MAX a
// radix pass is one kernel whose blocks each sum every tile's digit counts, a cost that grows as n^2 (against
// histogram, scan and scatter: 16384 0.237 / 0.258, 131072 0.311 / 0.340, 200000 0.371 / 0.343).
constexpr int RANK_MAX = 12288;
constexpr int FUSED_MAX = EVOL_SORT_FUSED_MAX;
constexpr int SCAN_ONE_MAX = 4 * SC_TILE;    // scans up to this size by one block

// ---------------------------------------------------------------------------------------
// Root cube
// ---------------------------------------------------------------------------------------
// A non-finite position is flagged as EVOL_ENAN (the min/max below ignore NaN, and every later
// phase keeps its loops bounded on such input, so the step completes and reports the error).
__global__ void k_bbox_partial(int n, const float *__restrict__ x, const float *__restrict__ y,
                               const float *__restrict__ z, float *__restrict__ part, int *err)
{
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float v[3] = {x[i], y[i], z[i]};
        if (!(isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]))) evol_flag(err, EVOL_ENAN);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], v[a]);
            hi[a] = fmaxf(hi[a], v[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    }
    __shared__ float s[BB_THREADS / 32][6];
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0)
        for (int a = 0; a < 3; ++a) { s[w][a] = lo[a]; s[w][3 + a] = hi[a]; }
    __syncthreads();
    if (threadIdx.x < 6) {
        float r = s[0][threadIdx.x];
        for (int k = 1; k < BB_THREADS / 32; ++k)
            r = threadIdx.x < 3 ? fminf(r, s[k][threadIdx.x]) : fmaxf(r, s[k][threadIdx.x]);
        part[blockIdx.x * 6 + threadIdx.x] = r;
    }
}

// Minimum (components 0..2) and maximum (3..5) of six values over a block of at most 32 warps; the result
// is on thread 0.
__device__ __forceinline__ void block_bounds(float v[6])
{
    __shared__ float sh[32][6];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
#pragma unroll
    for (int a = 0; a < 6; ++a)
        for (int o = 16; o > 0; o >>= 1) {
            const float t = __shfl_xor_sync(0xffffffffu, v[a], o);
            v[a] = a < 3 ? fminf(v[a], t) : fmaxf(v[a], t);
        }
    if (l == 0)
        for (int a = 0; a < 6; ++a) sh[w][a] = v[a];
    __syncthreads();
    if (w == 0)
#pragma unroll
        for (int a = 0; a < 6; ++a) {
            v[a] = l < nw ? sh[l][a] : (a < 3 ? INFINITY : -INFINITY);
            for (int o = 16; o > 0; o >>= 1) {
                const float t = __shfl_xor_sync(0xffffffffu, v[a], o);
                v[a] = a < 3 ? fminf(v[a], t) : fmaxf(v[a], t);
            }
        }
}

// corner = per-axis minimum; side = smallest power of two >= extent * (1 + 2^-20) (1 if 0)
__device__ __forceinline__ void write_cube(const float v[6], double *cube, float *fcube)
{
    double ext = 0.0;
    for (int a = 0; a < 3; ++a) {
        double e = (double)v[3 + a] - (double)v[a];
        ext = e > ext ? e : ext;
    }
    double target = ext * (1.0 + ldexp(1.0, -20));
    double s = 1.0;
    if (target > 0.0) {
        int ex;
        double fr = frexp(target, &ex);
        s = (fr == 0.5) ? ldexp(1.0, ex - 1) : ldexp(1.0, ex);
    }
    for (int a = 0; a < 3; ++a) {
        cube[a] = (double)v[a];
        fcube[a] = v[a];
    }
    cube[3] = s;
    fcube[3] = (float)s;
}

// One system's cube from the partial bounds, a block wide (one thread going through the 304 partials took
// 28 us), and its offsets.
__global__ void k_bbox_final(int n, int nparts, const float *__restrict__ part, double *cube, float *fcube,
                             int32_t *sys_off)
{
    float v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    for (int b = threadIdx.x; b < nparts; b += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            v[a] = fminf(v[a], part[b * 6 + a]);
            v[3 + a] = fmaxf(v[3 + a], part[b * 6 + 3 + a]);
        }
    block_bounds(v);
    if (threadIdx.x == 0) {
        write_cube(v, cube, fcube);
        sys_off[0] = 0;
        sys_off[1] = n;
    }
}

// ---------------------------------------------------------------------------------------
// Morton keys: q_a = clamp(floor((x_a - corner_a) * 2^21 / side), 0, 2^21 - 1), FP64 (the scale
// is a power of two, so the result is the exact floor of the double difference), interleaved
// with x the most significant bit of each triplet.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t spread3(uint64_t v)
{
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

// 2^21 / side for a power-of-two side (exact, without a double division)
__device__ __forceinline__ double key_scale(double side)
{
    int e;
    frexp(side, &e);                 // side = 2^(e-1)
    return ldexp(1.0, EVOL_MAXLEVEL + 1 - e);
}

// The sum of two floats as a float and what its rounding left out, exactly.
struct Centre {
    float hi, lo;
};

__device__ __forceinline__ Centre two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

// One axis' cell, floor((x - corner) 2^21 / side) of the difference rounded to double, in float arithmetic (FP64
// units made the key kernel ten times as long as its reads and writes: 3.1 M particles 161 -> 60 us).  x - corner
// is d.hi + d.lo exactly and the scale a power of two, so the floor is that of d.hi unless d.hi falls on a
// cell's edge and d.lo lies below it; a d.lo that double would have rounded away is left to double.
__device__ __forceinline__ uint64_t axis_cell(float x, double corner, float scale, double side)
{
    const Centre d = two_sum(x, -(float)corner);
    const float t = d.hi * scale;
    float q = floorf(t);
    const float lim = d.hi * 0x1p-52f;
    const bool edge = q == t && d.lo < 0.f;
    if (edge) q -= 1.f;
    if (scale == 0.f || (edge && !(lim >= 0x1p-126f && -d.lo > lim)))
        q = (float)fmin(fmax(floor(__dmul_rn(__dsub_rn((double)x, corner), key_scale(side))), 0.0), 2097151.0);
    return (uint64_t)fminf(fmaxf(q, 0.f), 2097151.f);
}

__device__ __forceinline__ uint64_t key_of(float x, float y, float z, const double *__restrict__ cb)
{
    // 2^21 / side where it is a normal float, else 0
    const int e = ilogb(cb[3]);
    const float scale = e > -100 && e < 126 ? __int_as_float((127 + EVOL_MAXLEVEL - e) << 23) : 0.f;
    return (spread3(axis_cell(x, cb[0], scale, cb[3])) << 2) | (spread3(axis_cell(y, cb[1], scale, cb[3])) << 1) |
           spread3(axis_cell(z, cb[2], scale, cb[3]));
}

// hist, if given, counts the first digit of the radix sort per tile (zeroed by the caller).
__global__ void k_keys(int n, const float *__restrict__ x, const float *__restrict__ y, const float *__restrict__ z,
                       const double *__restrict__ cube, uint64_t *__restrict__ keys, int32_t *__restrict__ vals,
                       int32_t *__restrict__ hist)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t key = key_of(x[i], y[i], z[i], cube);
    keys[i] = key;
    vals[i] = i;
    if (hist) atomicAdd(&hist[(i / RS_TILE) * 256 + (int)(key & 255u)], 1);
}

__device__ __forceinline__ int sys_of_pos(const int32_t *__restrict__ sys_off, int nsys, int s)
{
    // largest k with sys_off[k] <= s
    int lo = 0, hi = nsys;           // sys_off[0] = 0 <= s < sys_off[nsys]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (sys_off[mid] <= s) lo = mid; else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------------------------------
// Exclusive scan of int32 (reduce / top / down-sweep).  Used for the radix histograms and the
// per-position node counts.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ int32_t block_excl_scan(int32_t v, int32_t *sh, int32_t &total)
{
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int32_t s = lane < nw ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        if (lane < nw) sh[lane] = s;
    }
    __syncthreads();
    int32_t pre = (w > 0 ? sh[w - 1] : 0) + x - v;
    total = sh[nw - 1];
    __syncthreads();
    return pre;
}

__global__ void k_scan_reduce(int n, const int32_t *__restrict__ in, int32_t *__restrict__ part)
{
    __shared__ int32_t sh[32];
    int base = blockIdx.x * SC_TILE;
    int32_t s = 0;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) {
        int i = base + k * SC_THREADS + threadIdx.x;
        if (i < n) s += in[i];
    }
    int32_t tot;
    block_excl_scan(s, sh, tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void k_scan_top(int nparts, int32_t *__restrict__ part)
{
    __shared__ int32_t sh[32];
    int32_t carry = 0;
    for (int b = 0; b < nparts; b += blockDim.x) {
        int i = b + threadIdx.x;
        int32_t v = i < nparts ? part[i] : 0, tot;
        int32_t pre = block_excl_scan(v, sh, tot);
        if (i < nparts) part[i] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) part[nparts] = carry;
}

// out may alias in.  out[n] receives the grand total when write_total is set.
__global__ void k_scan_down(int n, const int32_t *in, int32_t *out, const int32_t *__restrict__ part, int nparts,
                            int write_total)
{
    __shared__ int32_t sh[32];
    int base = blockIdx.x * SC_TILE + threadIdx.x * SC_ITEMS;
    int32_t v[SC_ITEMS], s = 0;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) {
        int i = base + k;
        v[k] = i < n ? in[i] : 0;
        s += v[k];
    }
    int32_t tot;
    int32_t pre = block_excl_scan(s, sh, tot) + part[blockIdx.x];
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) {
        int i = base + k;
        if (i < n) out[i] = pre;
        pre += v[k];
    }
    if (write_total && blockIdx.x == 0 && threadIdx.x == 0) out[n] = part[nparts];
}

// A whole scan by one block.
__global__ void __launch_bounds__(SC_THREADS) k_scan_one(int n, const int32_t *in, int32_t *out, int write_total)
{
    __shared__ int32_t sh[32];
    int32_t carry = 0;
    for (int b = 0; b < n; b += SC_TILE) {
        const int base = b + threadIdx.x * SC_ITEMS;
        int32_t v[SC_ITEMS], s = 0, tot;
#pragma unroll
        for (int k = 0; k < SC_ITEMS; ++k) {
            v[k] = base + k < n ? in[base + k] : 0;
            s += v[k];
        }
        int32_t pre = carry + block_excl_scan(s, sh, tot);
#pragma unroll
        for (int k = 0; k < SC_ITEMS; ++k) {
            if (base + k < n) out[base + k] = pre;
            pre += v[k];
        }
        carry += tot;
    }
    if (write_total && threadIdx.x == 0) out[n] = carry;
}

// ---------------------------------------------------------------------------------------
// Small sets: the sorted position of key i is the number of keys before it in (key, index) order, counted
// directly.  A block ranks 32 keys, one per lane, its eight warps going through eighths of every tile of
// keys; bound by its integer comparisons (1000 particles 5.4 us; 40 launches of a radix sort before).  Several systems: keys of the same system only, from its offset.
// ---------------------------------------------------------------------------------------
template <bool SYS>
__global__ void __launch_bounds__(256) k_rank_sort(int n, const uint64_t *__restrict__ keys,
                                                   const int32_t *__restrict__ sys_off, int nsys,
                                                   uint64_t *__restrict__ kout, int32_t *__restrict__ vout)
{
    constexpr int TILE = 1024;
    __shared__ __align__(16) uint64_t tile[TILE];
    __shared__ int32_t cnt[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, i = i0 + lane;
    const uint64_t key = i < n ? keys[i] : 0ull;
    // this key's system: [b, e)
    int b = 0, e = n;
    if (SYS && i < n) {
        const int sy = sys_of_pos(sys_off, nsys, i);
        b = sys_off[sy];
        e = sys_off[sy + 1];
    }
    int c = 0;
    for (int t0 = 0; t0 < n; t0 += TILE) {
        __syncthreads();
        for (int t = threadIdx.x; t < TILE; t += 256) tile[t] = t0 + t < n ? keys[t0 + t] : ~0ull;
        __syncthreads();
        const int j0 = t0 + w * (TILE / 8);
        if (SYS || (j0 < i0 + 32 && j0 + TILE / 8 > i0)) {
#pragma unroll 4
            for (int t = 0; t < TILE / 8; ++t) {
                const int j = j0 + t;
                const bool before = tile[w * (TILE / 8) + t] < key + (j < i ? 1u : 0u);   // ties by index
                c += before && (!SYS || (j >= b && j < e)) ? 1 : 0;
            }
        } else {
            const uint64_t lim = key + (j0 < i0 ? 1u : 0u);
            const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(tile + w * (TILE / 8));
#pragma unroll 8
            for (int t = 0; t < TILE / 16; ++t) {
                const ulonglong2 k2 = p[t];
                c += k2.x < lim ? 1 : 0;
                c += k2.y < lim ? 1 : 0;
            }
        }
    }
    cnt[w][lane] = c;
    __syncthreads();
    if (w == 0 && i < n) {
        int pos = b;
#pragma unroll
        for (int q = 0; q < 8; ++q) pos += cnt[q][lane];
        kout[pos] = key;
        vout[pos] = i;
    }
}

// ---------------------------------------------------------------------------------------
// Stable LSD radix sort, 8-bit digits, 64-bit keys with int32 values.
// ---------------------------------------------------------------------------------------
__global__ void k_rs_hist(int n, const uint64_t *__restrict__ keys, int shift, int32_t *__restrict__ hist, int nblocks)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    int base = blockIdx.x * RS_TILE;
#pragma unroll 4
    for (int k = 0; k < RS_ITEMS; ++k) {
        int i = base + k * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&h[(unsigned)(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[threadIdx.x * nblocks + blockIdx.x] = (int32_t)h[threadIdx.x];
}

// One pass's scatter of a tile.  A warp owns 32 RS_ITEMS consecutive keys and ranks them 32 at a time (the
// lanes with its digit before it, and the warp's count of that digit so far); the warps' counts are then
// turned into positions.  FUSED: offs holds every tile's histogram, from which the block sums its own
// offsets (at most FUSED_MAX / RS_TILE loads a thread), and the next digit's histogram is counted as the keys
// are written (next), so that a pass is one kernel; else offs is the scanned histogram, digit by digit.
template <bool FUSED>
__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(int n, const uint64_t *__restrict__ kin,
                                                           const int32_t *__restrict__ vin, uint64_t *__restrict__ kout,
                                                           int32_t *__restrict__ vout, int shift,
                                                           const int32_t *__restrict__ offs, int nblocks,
                                                           int32_t *__restrict__ next)
{
    constexpr int NW = RS_THREADS / 32;
    __shared__ uint32_t wcnt[NW][256];
    __shared__ int32_t sh[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
#pragma unroll
    for (int k = 0; k < NW; ++k) wcnt[k][t] = 0;
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    const int base = blockIdx.x * RS_TILE + w * (32 * RS_ITEMS) + lane;
    uint64_t key[RS_ITEMS];
    uint32_t rank[RS_ITEMS];
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) key[r] = base + 32 * r < n ? kin[base + 32 * r] : 0ull;
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const unsigned d = base + 32 * r < n ? ((unsigned)(key[r] >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(peers) - 1;
        uint32_t before = 0;
        if (lane == leader && d < 256u) {
            before = wcnt[w][d];
            wcnt[w][d] = before + __popc(peers);
        }
        rank[r] = __shfl_sync(0xffffffffu, before, leader) + __popc(peers & lt);
        __syncwarp();
    }
    // digit t: where this tile's keys go
    uint32_t run;
    if (FUSED) {
        int32_t mine = 0, all = 0, tot;
#pragma unroll 8
        for (int q = 0; q < nblocks; ++q) {
            const int32_t c = offs[q * 256 + t];
            all += c;
            mine += q < (int)blockIdx.x ? c : 0;
        }
        run = (uint32_t)(block_excl_scan(all, sh, tot) + mine);
    } else {
        run = (uint32_t)offs[t * nblocks + blockIdx.x];
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        const uint32_t c = wcnt[k][t];
        wcnt[k][t] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r)
        if (base + 32 * r < n) {
            const uint32_t pos = wcnt[w][(unsigned)(key[r] >> shift) & 255u] + rank[r];
            kout[pos] = key[r];
            vout[pos] = vin[base + 32 * r];
            if (FUSED && next) atomicAdd(&next[(pos / RS_TILE) * 256 + ((unsigned)(key[r] >> (shift + 8)) & 255u)], 1);
        }
}

// d_i = common leading octal digits of keys i-1 and i; -1 where i starts a system (a forest of
// independent trees, one per system, in one pre-order list).
__device__ __forceinline__ int8_t lcp_of(const uint64_t *__restrict__ keys, int i, bool starts)
{
    if (starts) return -1;
    const uint64_t x = keys[i - 1] ^ keys[i];
    return x == 0 ? (int8_t)EVOL_MAXLEVEL : (int8_t)((__clzll((long long)x) - 1) / 3);
}

// ---------------------------------------------------------------------------------------
// Permutation into sorted order, and each position's system and common digits with its predecessor.
// ---------------------------------------------------------------------------------------
__global__ void k_permute(int n, int n_gas, const int32_t *__restrict__ perm, const float *__restrict__ x,
                          const float *__restrict__ y, const float *__restrict__ z, const float *__restrict__ vx,
                          const float *__restrict__ vy, const float *__restrict__ vz, const float *__restrict__ m,
                          const float *__restrict__ u, const float *__restrict__ h, const float *__restrict__ eps,
                          float4 *__restrict__ pos, float4 *__restrict__ vel, float *__restrict__ lh,
                          float *__restrict__ le, int32_t *__restrict__ orig, int32_t *__restrict__ inv,
                          const float *__restrict__ pred_dt, const float *__restrict__ pred_acc, int64_t stride,
                          const float *__restrict__ pred_tau, const uint64_t *__restrict__ keys,
                          const int32_t *__restrict__ sys_off, int nsys, int8_t *__restrict__ lcp,
                          int32_t *__restrict__ sys_sorted)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    int j = perm[s];
    const int sy = nsys > 1 ? sys_of_pos(sys_off, nsys, s) : 0;
    sys_sorted[s] = sy;
    lcp[s] = lcp_of(keys, s, s == (nsys > 1 ? sys_off[sy] : 0));
    bool gas = j < n_gas;
    pos[s] = make_float4(x[j], y[j], z[j], m[j]);
    float4 v = make_float4(vx ? vx[j] : 0.f, vy ? vy[j] : 0.f, vz ? vz[j] : 0.f, (gas && u) ? u[j] : 0.f);
    if (pred_dt || pred_tau) {
        // integrator: the force step sees the velocity and internal energy predicted to the end of
        // the step, v_n + a_n dt and u_n + (du/dt)_n dt (Sect. 4.1); the caller's arrays hold the
        // half-kicked values, so half a step of the previous accelerations (pred_acc: ax | ay | az |
        // du/dt in the caller's order, `stride` apart) is added -- with individual steps each
        // particle's own time since the middle of its step, pred_tau[j]
        const float hdt = pred_tau ? pred_tau[j] : 0.5f * *pred_dt;
        v.x += hdt * pred_acc[j];
        v.y += hdt * pred_acc[stride + j];
        v.z += hdt * pred_acc[2 * stride + j];
        if (gas && u) v.w += hdt * pred_acc[3 * stride + j];
    }
    vel[s] = v;
    lh[s] = (gas && h) ? h[j] : 0.f;
    le[s] = eps ? eps[j] : 0.f;
    orig[s] = j;
    inv[j] = s;
}

// ---------------------------------------------------------------------------------------
// Node construction.
// ---------------------------------------------------------------------------------------
// Does the level-lam run containing position i hold more than `leaf` particles?
__device__ __forceinline__ bool run_exceeds(int n, const int8_t *__restrict__ lcp, int i, int lam, int leaf)
{
    int c = 1;
    for (int t = i; c <= leaf && t > 0 && lcp[t] >= lam; --t) ++c;
    for (int t = i + 1; c <= leaf && t < n && lcp[t] >= lam; ++t) ++c;
    return c > leaf;
}

__device__ __forceinline__ int nodes_at(int n, const int8_t *__restrict__ lcp, int i, int leaf, int &lo)
{
    lo = lcp[i] + 1;                  // 0 where a system starts (lcp = -1)
    int c = 0;
    for (int l = lo; l <= EVOL_MAXLEVEL; ++l) {
        if (l > 0 && !run_exceeds(n, lcp, i, l - 1, leaf)) break;
        ++c;
    }
    return c;
}

__global__ void k_count(int n, const int8_t *__restrict__ lcp, int leaf, int32_t *__restrict__ cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo;
    cnt[i] = nodes_at(n, lcp, i, leaf, lo);
}

// end of the level-l run beginning at position i; nend = end of i's system
__device__ __forceinline__ int run_end(int nend, const uint64_t *__restrict__ keys, const int8_t *__restrict__ lcp,
                                       int i, int l, int leaf)
{
    int t = i + 1;
    for (int k = 0; k <= leaf && t < nend; ++k, ++t)
        if (lcp[t] < l) return t;
    if (t >= nend) return nend;
    if (l == 0) return nend;
    int sh = 3 * (EVOL_MAXLEVEL - l);
    uint64_t upper = keys[i] | ((1ull << sh) - 1ull);
    // gallop then bisect for the first index with key > upper
    int lo = t - 1, step = 1, hi = t;
    while (hi < nend && keys[hi] <= upper) {
        lo = hi;
        step <<= 1;
        hi = t - 1 + step;
    }
    if (hi > nend) hi = nend;
    while (hi - lo > 1) {
        int mid = lo + ((hi - lo) >> 1);
        if (keys[mid] <= upper) lo = mid; else hi = mid;
    }
    return hi;
}

__global__ void k_fill(int n, const uint64_t *__restrict__ keys, const int8_t *__restrict__ lcp,
                       const int32_t *__restrict__ sys_off, const int32_t *__restrict__ sys_sorted,
                       const int32_t *__restrict__ base, int leaf, int64_t node_cap, int32_t *__restrict__ nbeg,
                       int32_t *__restrict__ nend, int32_t *__restrict__ nlev, int32_t *__restrict__ nnext,
                       int32_t *__restrict__ nnodes, int *err)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int total = base[n];
    if (i == 0) {
        *nnodes = total > node_cap ? (int)node_cap : total;
        if (total > node_cap) evol_flag(err, EVOL_EOVERFLOW);
    }
    if (i >= n) return;
    const int lo = lcp[i] + 1, b = base[i], c = base[i + 1] - b;
    const int send = sys_off[sys_sorted[i] + 1];
    for (int k = 0; k < c; ++k) {
        int id = b + k;
        if (id >= node_cap) return;
        int l = lo + k;
        int e = run_end(send, keys, lcp, i, l, leaf);
        nbeg[id] = i;
        nend[id] = e;
        nlev[id] = l;
        int nx = e < n ? base[e] : total;
        nnext[id] = nx > node_cap ? (int)node_cap : nx;
    }
}

__global__ void k_link(const int32_t *__restrict__ nnodes, int leaf, const int32_t *__restrict__ nbeg,
                       const int32_t *__restrict__ nend, const int32_t *__restrict__ nlev,
                       const int32_t *__restrict__ nnext, int32_t *__restrict__ nparent, int32_t *__restrict__ nnch,
                       int32_t *__restrict__ narrive, int4 *__restrict__ nI, int4 *__restrict__ nK0,
                       int4 *__restrict__ nK1, int nsys, const int32_t *__restrict__ sys_off,
                       const int32_t *__restrict__ base, int32_t *__restrict__ sys_root)
{
    int nn = *nnodes;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nsys; k += gridDim.x * blockDim.x)
        sys_root[k] = base[sys_off[k]];
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < nn; id += gridDim.x * blockDim.x) {
        narrive[id] = 0;
        if (nlev[id] == 0) nparent[id] = -1;     // the root of a system
        int e = nend[id];
        bool internal = (e - nbeg[id] > leaf) && nlev[id] < EVOL_MAXLEVEL;
        int k = 0;
        int ch[8] = {-1, -1, -1, -1, -1, -1, -1, -1};
        if (internal) {
            int c = id + 1;
            while (c < nn && nbeg[c] < e && k < 8) {
                nparent[c] = id;
                ch[k] = c;
                ++k;
                c = nnext[c];
            }
        }
        nK0[id] = make_int4(ch[0], ch[1], ch[2], ch[3]);
        nK1[id] = make_int4(ch[4], ch[5], ch[6], ch[7]);
        nnch[id] = k;
        nI[id] = make_int4(nlev[id] | ((internal ? 0 : 1) << 8), nnext[id], nbeg[id], e);
    }
}

// ---------------------------------------------------------------------------------------
// Moments, leaf-up.  A leaf sums its particles; the last child to finish a parent (atomic
// arrival count) combines the children with the parallel-axis shift of the quadrupole.
//
// FP32 (plain) moments take every position relative to the node's geometric centre (a dyadic point of the
// root cube, see Centre), so the centre of mass and the quadrupole carry rounding on the scale of the
// node, not of the coordinates; a parent combines its children's centre-of-mass offsets shifted by the
// (power-of-two) difference of the two centres, which is exact in float.  The absolute centre of mass
// is formed once, by k_node_geometry.  FP64 (mixed) moments use absolute coordinates.
// ---------------------------------------------------------------------------------------
struct NodeOut {
    float4 *nA, *nB, *nC, *nQ0, *nQ1, *bmin, *bmax, *coff;
    double *M64, *C64, *Q64;
};

// bits 0, 3, 6, ... of v, packed (the inverse of spread3)
__device__ __forceinline__ unsigned compact3(uint64_t v)
{
    v &= 0x1249249249249249ull;
    v = (v | (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v | (v >> 4)) & 0x100f00f00f00f00full;
    v = (v | (v >> 8)) & 0x1f0000ff0000ffull;
    v = (v | (v >> 16)) & 0x1f00000000ffffull;
    return (unsigned)(v | (v >> 32)) & 0x1fffffu;
}

// cell index along axis a (0: x) of the node whose first key is key0 at level lev
__device__ __forceinline__ unsigned cell_index(uint64_t key0, int lev, int a)
{
    return compact3(key0 >> (3 * (EVOL_MAXLEVEL - lev)) >> (2 - a));
}

// A node's geometric centre along one axis, as the sum of two floats.  The cube's corner is a float, and the
// centre's offset from it an odd number of 22 bits times a power of two, so the sum of the two in hi + lo is
// exact, and a float minus the centre is right to the rounding of the result, without double arithmetic.
__device__ __forceinline__ Centre node_centre(float corner, float side, unsigned cell, int lev)
{
    return two_sum(corner, (float)(2u * cell + 1u) * ldexpf(side, -lev - 1));
}

// x minus the centre
__device__ __forceinline__ float from_centre(float x, const Centre &c)
{
    const Centre d = two_sum(x, -c.hi);
    return __fadd_rn(d.hi, __fsub_rn(d.lo, c.lo));
}

// The totals over an octet's eight lanes of eight values each: lane k gets value k's (seven exchanges instead
// of 24).
template <typename T, typename Op>
__device__ __forceinline__ T octet_reduce(T (&v)[8], int sub, Op op)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const bool up = sub & o;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const T give = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
            v[k] = op(keep, __shfl_xor_sync(0xffffffffu, give, o));
        }
    }
    return v[0];
}

// The same of four values: lanes k and k + 4 get value k's.
template <typename T>
__device__ __forceinline__ T octet_sum4(T (&v)[4], int sub)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], 4);
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
        const bool up = sub & o;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const T give = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0];
}

struct Links {
    const int32_t *nnodes, *nparent, *nnch;
    const int4 *nI, *nK0, *nK1;
    int32_t *narrive;
    int *err;
};

// Leaf-up pass over the tree: eight lanes to a node, in a leaf a lane to a particle, above a lane to a child.
// The octet that completes a parent goes on with it, the others end; a warp starts on the leaves among
// its next nodes, four at a time.  leaf(id, I) and node(id, I, child, pre) form and store a node's values
// (id < 0: nothing to do; all 32 lanes call them); pre(child, level) is read ahead of the parent's
// completion, as are all its links: what remains of a level is the chain store, fence, count, load of the
// children's values.  The counts are left at zero for the next pass.
template <typename Leaf, typename Pre, typename Node>
__device__ __forceinline__ void leaf_up(const Links &L, Leaf leaf, Pre pre, Node node)
{
    const int nn = *L.nnodes, lane = threadIdx.x & 31, sub = lane & 7;
    const int warps = gridDim.x * (blockDim.x >> 5), wid = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    // nodes a turn: 32, fewer where that leaves warps without any
    const int per = min(32, (nn / warps + 4) & ~3);
    for (int base = wid * per; base < nn; base += warps * per) {
        unsigned todo = __ballot_sync(0xffffffffu, lane < per && base + lane < nn && L.nnch[base + lane] == 0);
        while (todo) {
            int id = -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if ((lane >> 3) == q && todo) id = base + __ffs(todo) - 1;
                todo &= todo - 1u;
            }
            leaf(id, id >= 0 ? L.nI[id] : make_int4(0, 0, 0, 0));
            for (int climb = 0;; ++climb) {
                if (climb > EVOL_MAXLEVEL + 1) {     // deeper than the tree can be: corrupt parents
                    if (lane == 0) evol_flag(L.err, EVOL_ETIMEOUT);
                    break;
                }
                int p = id >= 0 ? L.nparent[id] : -1;
                if (p >= nn) p = -1;
                int4 I = make_int4(0, 0, 0, 0);
                int nch = 0, c = -1;
                if (p >= 0) {
                    I = L.nI[p];
                    nch = L.nnch[p];
                    c = reinterpret_cast<const int *>(sub < 4 ? L.nK0 : L.nK1)[4 * (size_t)p + (sub & 3)];
                }
                const auto ahead = pre(c, (I.x & 0xff) + 1);
                __threadfence();
                __syncwarp();
                int old = -1;
                if (p >= 0 && sub == 0) old = atomicAdd(&L.narrive[p], 1);
                old = __shfl_sync(0xffffffffu, old, lane & 24);
                const bool last = p >= 0 && old == nch - 1;
                if (last && sub == 0) L.narrive[p] = 0;
                if (!__any_sync(0xffffffffu, last)) break;
                __threadfence();
                __syncwarp();
                id = last ? p : -1;
                node(id, I, last ? c : -1, ahead);
            }
        }
    }
}

// Moments of every node: mass, centre of mass (FP32: its offset from the node's centre), quadrupole about it, and
// the particles' box.  Bound by the chain of dependent steps from the leaves to the root, not by its reads.
// A thread per node, its children one after the other and each in dependent loads, took 54 us with 1000
// particles, 141 with 49 k and 962 with 3.1 M; this and k_node_geometry take 24, 59 and 279 (FP64 of 393 k:
// 389 -> 184), k_node_lengths 12, 32 and 145 (26, 77 and 197).
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 5)
    k_moments(Links L, int n_gas, const float4 *__restrict__ pos, const int32_t *__restrict__ orig,
              const uint64_t *__restrict__ keys, const float *__restrict__ fcube,
              const int32_t *__restrict__ sys_sorted, NodeOut o)
{
    constexpr bool rel = sizeof(T) == sizeof(float);
    const int lane = threadIdx.x & 31, sub = lane & 7, oct = lane & 24;
    // Adds the lanes' masses and masses times positions to the octet's sums.  FP32: one after the other in
    // the order of the particles or children, on every lane, so that a node's opening radius, on which the walk's
    // decisions turn, does not depend on how the lanes split it; FP64: each lane its own, summed by finish.
    auto add = [&](T (&ms)[4], T w, T x, T y, T z) {
#pragma unroll
        for (int k = 0; k < (rel ? 8 : 1); ++k) {
            const T wk = rel ? __shfl_sync(0xffffffffu, w, oct + k) : w;
            ms[0] += wk;
            ms[1] += wk * (rel ? __shfl_sync(0xffffffffu, x, oct + k) : x);
            ms[2] += wk * (rel ? __shfl_sync(0xffffffffu, y, oct + k) : y);
            ms[3] += wk * (rel ? __shfl_sync(0xffffffffu, z, oct + k) : z);
        }
    };
    // an octet's node from its sums and its lanes' shares: box (lo, -hi, -gas), then the quadrupole shares that
    // add_q makes about the centre of mass
    auto finish = [&](int id, int lev, int beg, T (&ms)[4], float (&bx)[8], auto add_q) {
        const T sum = rel ? (sub == 0 ? ms[0] : sub == 1 ? ms[1] : sub == 2 ? ms[2] : ms[3]) : octet_sum4(ms, sub);
        const float bound = octet_reduce(bx, sub, [](float a, float b) { return fminf(a, b); });
        const T M = __shfl_sync(0xffffffffu, sum, oct);
        T c[3];
        const T cv = sum / M;                      // lanes 1 .. 3
#pragma unroll
        for (int a = 0; a < 3; ++a) c[a] = __shfl_sync(0xffffffffu, cv, oct + 1 + a);
        if (__any_sync(0xffffffffu, id >= 0 && !(M > 0))) {
            // no mass: the middle of the box
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float lo = __shfl_sync(0xffffffffu, bound, oct + a), hi = -__shfl_sync(0xffffffffu, bound, oct + 3 + a);
                if (id >= 0 && !(M > 0)) {
                    if (rel) {
                        const float *cb = fcube + 4 * sys_sorted[beg];
                        const Centre cg = node_centre(cb[a], cb[3], cell_index(keys[beg], lev, a), lev);
                        c[a] = (T)(0.5f * (from_centre(lo, cg) + from_centre(hi, cg)));
                    } else {
                        c[a] = (T)0.5 * ((T)lo + (T)hi);
                    }
                }
            }
        }
        T q[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        add_q(c, q);
        const T qv = octet_reduce(q, sub, [](T a, T b) { return a + b; });
        if (id < 0) return;
        float *qf = (float *)(sub >= 3 && sub < 6 ? o.nQ1 : o.nQ0) + 4 * (size_t)id;
        if (sub < 7) qf[sub == 6 ? 3 : sub < 3 ? sub : sub - 3] = sub == 6 ? (float)M : (float)qv;
        float *bf = (float *)(sub == 7 || (sub >= 3 && sub < 6) ? o.bmax : o.bmin) + 4 * (size_t)id;
        bf[sub >= 6 ? 3 : sub < 3 ? sub : sub - 3] = sub == 7 ? 0.f : sub < 3 ? bound : 0.f - bound;
        const T cs = sub == 0 ? c[0] : sub == 1 ? c[1] : sub == 2 ? c[2] : M;
        if (rel) {
            if (sub < 4) reinterpret_cast<float *>(o.coff)[4 * (size_t)id + sub] = (float)cs;
        } else {
            if (sub < 3) o.C64[3 * (size_t)id + sub] = (double)cs;
            if (sub == 3) o.M64[id] = (double)cs;
            if (sub < 6) o.Q64[6 * (size_t)id + sub] = (double)qv;
        }
    };
    auto quad = [](T (&q)[8], T w, T d0, T d1, T d2) {
        const T r2 = d0 * d0 + d1 * d1 + d2 * d2;
        q[0] += w * (3 * d0 * d0 - r2);
        q[1] += w * (3 * d1 * d1 - r2);
        q[2] += w * (3 * d2 * d2 - r2);
        q[3] += w * 3 * d0 * d1;
        q[4] += w * 3 * d0 * d2;
        q[5] += w * 3 * d1 * d2;
    };
    auto box = [](float (&bx)[8]) {
#pragma unroll
        for (int k = 0; k < 6; ++k) bx[k] = INFINITY;
        bx[6] = bx[7] = 0.f;
    };
    leaf_up(
        L,
        [&](int id, const int4 &I) {
            const int lev = I.x & 0xff, b = I.z, e = id >= 0 ? I.w : I.z;
            Centre cg[3] = {};
            if (rel) {
                // axis a's on lane a, then to all
                Centre m = {0.f, 0.f};
                if (id >= 0 && sub < 3) {
                    const float *cb = fcube + 4 * sys_sorted[b];
                    m = node_centre(cb[sub], cb[3], cell_index(keys[b], lev, sub), lev);
                }
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    cg[a] = {__shfl_sync(0xffffffffu, m.hi, oct + a), __shfl_sync(0xffffffffu, m.lo, oct + a)};
            }
            auto coord = [&](float x, int a) -> T { return rel ? (T)from_centre(x, cg[a]) : (T)x; };
            T ms[4] = {0, 0, 0, 0};
            float bx[8];
            box(bx);
            for (int s = b + sub; __any_sync(0xffffffffu, s < e); s += 8) {
                const bool in = s < e;
                const float4 p = in ? pos[s] : make_float4(0.f, 0.f, 0.f, 0.f);
                add(ms, (T)p.w, in ? coord(p.x, 0) : (T)0, in ? coord(p.y, 1) : (T)0, in ? coord(p.z, 2) : (T)0);
                if (!in) continue;
                if (orig[s] < n_gas) bx[6] = -1.f;
                bx[0] = fminf(bx[0], p.x); bx[1] = fminf(bx[1], p.y); bx[2] = fminf(bx[2], p.z);
                bx[3] = fminf(bx[3], -p.x); bx[4] = fminf(bx[4], -p.y); bx[5] = fminf(bx[5], -p.z);
            }
            finish(id, lev, b, ms, bx, [&](const T (&c)[3], T (&q)[8]) {
                for (int s = b + sub; s < e; s += 8) {
                    const float4 p = pos[s];
                    quad(q, (T)p.w, coord(p.x, 0) - c[0], coord(p.y, 1) - c[1], coord(p.z, 2) - c[2]);
                }
            });
        },
        // A child cell is one level below its parent (a cell with one non-empty octant still has that octant
        // as its child), so its centre is the parent's moved by a quarter of the parent's side along each
        // axis, in the direction its octal digit gives: a power of two, exact in float.
        [&](int c, int lev) -> unsigned {
            return rel && c >= 0 ? (unsigned)(keys[L.nI[c].z] >> (3 * (EVOL_MAXLEVEL - lev))) & 7u : 0u;
        },
        [&](int id, const int4 &I, int c, unsigned digit) {
            T ms[4] = {0, 0, 0, 0}, cc[3] = {0, 0, 0}, cq[6] = {0, 0, 0, 0, 0, 0}, M = 0;
            float bx[8];
            box(bx);
            if (c >= 0) {
                const float4 bl = __ldcg(&o.bmin[c]), bh = __ldcg(&o.bmax[c]);
                if (rel) {
                    const float4 co = __ldcg(&o.coff[c]), Q0 = __ldcg(&o.nQ0[c]), Q1 = __ldcg(&o.nQ1[c]);
                    const float q = ldexpf(fcube[4 * sys_sorted[I.z] + 3], -(I.x & 0xff) - 2);
                    M = (T)co.w;
                    cc[0] = (T)co.x + (T)((digit & 4u) ? q : -q);
                    cc[1] = (T)co.y + (T)((digit & 2u) ? q : -q);
                    cc[2] = (T)co.z + (T)((digit & 1u) ? q : -q);
                    cq[0] = (T)Q0.x; cq[1] = (T)Q0.y; cq[2] = (T)Q0.z;
                    cq[3] = (T)Q1.x; cq[4] = (T)Q1.y; cq[5] = (T)Q1.z;
                } else {
                    M = (T)__ldcg(&o.M64[c]);
#pragma unroll
                    for (int a = 0; a < 3; ++a) cc[a] = (T)__ldcg(&o.C64[3 * (size_t)c + a]);
#pragma unroll
                    for (int a = 0; a < 6; ++a) cq[a] = (T)__ldcg(&o.Q64[6 * (size_t)c + a]);
                }
                bx[0] = bl.x; bx[1] = bl.y; bx[2] = bl.z;
                bx[3] = -bh.x; bx[4] = -bh.y; bx[5] = -bh.z;
                bx[6] = -bl.w;
            }
            add(ms, M, cc[0], cc[1], cc[2]);
            finish(id, I.x & 0xff, I.z, ms, bx, [&](const T (&cm)[3], T (&q)[8]) {
                if (c >= 0) {
#pragma unroll
                    for (int a = 0; a < 6; ++a) q[a] = cq[a];
                    quad(q, M, cc[0] - cm[0], cc[1] - cm[1], cc[2] - cm[2]);
                }
            });
        });
}

// What a node's users need beside its moments, one thread per node: the centre of mass and squared opening
// radius, centre and half widths of the box, the distance between the centres of mass and cell.
__global__ void k_node_geometry(const int32_t *__restrict__ nnodes, const int4 *__restrict__ nI,
                                const uint64_t *__restrict__ keys, const double *__restrict__ cube,
                                const float *__restrict__ fcube, const int32_t *__restrict__ sys_sorted, float theta,
                                NodeOut o, int mixed)
{
    const int nn = *nnodes;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < nn; id += gridDim.x * blockDim.x) {
        const int4 I = nI[id];
        const int lev = I.x & 0xff, sys = sys_sorted[I.z];
        const uint64_t key0 = keys[I.z];
        const float4 lo = o.bmin[id], hi = o.bmax[id];
        float com[3], delta;
        if (mixed) {
            double dd = 0.0;
            const double side = ldexp(cube[4 * sys + 3], -lev);
            for (int a = 0; a < 3; ++a) {
                const double c = o.C64[3 * (size_t)id + a];
                const double off = c - (cube[4 * sys + a] + ((double)cell_index(key0, lev, a) + 0.5) * side);
                com[a] = (float)c;
                dd += off * off;
            }
            delta = (float)sqrt(dd);
        } else {
            const float4 co = o.coff[id];
            const float off[3] = {co.x, co.y, co.z};
            float s = 0.f, err = 0.f;              // sum of squares s + err, its error far below FP32's
            for (int a = 0; a < 3; ++a) {
                const Centre cg = node_centre(fcube[4 * sys + a], fcube[4 * sys + 3], cell_index(key0, lev, a), lev);
                const Centre t = two_sum(cg.hi, off[a]);
                com[a] = t.hi + (t.lo + cg.lo);
                const float sq = __fmul_rn(off[a], off[a]);
                const Centre u = two_sum(s, sq);
                s = u.hi;
                err += u.lo + fmaf(off[a], off[a], -sq);
            }
            delta = sqrtf(s);
            if (delta > 0.f && delta < 1e18f) delta += __fdividef(0.5f * (fmaf(-delta, delta, s) + err), delta);
        }
        const float l = ldexpf(fcube[4 * sys + 3], -lev);
        const float ropen = theta > 0.f ? l / theta + delta : INFINITY;
        o.nA[id] = make_float4(com[0], com[1], com[2], ropen * ropen);
        o.nB[id] = make_float4(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z), lo.w != 0.f ? 0.f : -1.f);
        o.nC[id] = make_float4(0.5f * (hi.x - lo.x), 0.5f * (hi.y - lo.y), 0.5f * (hi.z - lo.z), 0.f);
        reinterpret_cast<float *>(o.nQ1)[4 * (size_t)id + 3] = delta;
    }
}

// Node maxima of 2 eps (all particles) and 2 h (gas), leaf-up like the moments.
__global__ void __launch_bounds__(128, 8)
    k_node_lengths(Links L, int n_gas, const int32_t *__restrict__ orig, const float *__restrict__ le,
                   const float *__restrict__ lh, float4 *nB, float4 *nC)
{
    const int sub = threadIdx.x & 7;
    auto finish = [&](int id, float em, float hm) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            em = fmaxf(em, __shfl_xor_sync(0xffffffffu, em, o));
            hm = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, o));
        }
        if (id >= 0 && sub == 0) nC[id].w = em;
        if (id >= 0 && sub == 1) nB[id].w = hm >= 0.f ? hm : -1.f;
    };
    leaf_up(
        L,
        [&](int id, const int4 &I) {
            float em = 0.f, hm = -1.f;
            for (int s = I.z + sub; id >= 0 && s < I.w; s += 8) {
                em = fmaxf(em, 2.f * le[s]);
                if (orig[s] < n_gas) hm = fmaxf(hm, 2.f * lh[s]);
            }
            finish(id, em, hm);
        },
        [](int, int) { return 0; },
        [&](int id, const int4 &, int c, int) {
            finish(id, c >= 0 ? __ldcg(&nC[c].w) : 0.f, c >= 0 ? __ldcg(&nB[c].w) : -1.f);
        });
}

// ---- several independent systems (batched): per-system cube and keys ----------------------
// one block per system: its cube from its own particles
// (also one small system: offsets 0, n are then written here, n > 0)
__global__ void k_bbox_sys(int n, int32_t *__restrict__ sys_off, const float *__restrict__ x,
                           const float *__restrict__ y, const float *__restrict__ z, double *cube, float *fcube,
                           int *err)
{
    const int k = blockIdx.x;
    const int b = n > 0 ? 0 : sys_off[k], e = n > 0 ? n : sys_off[k + 1];
    float v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    bool bad = false;
#pragma unroll 4
    for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
        const float p[3] = {x[i], y[i], z[i]};
        bad |= !(isfinite(p[0]) && isfinite(p[1]) && isfinite(p[2]));
        for (int a = 0; a < 3; ++a) {
            v[a] = fminf(v[a], p[a]);
            v[3 + a] = fmaxf(v[3 + a], p[a]);
        }
    }
    if (bad) evol_flag(err, EVOL_ENAN);
    block_bounds(v);
    if (threadIdx.x == 0) {
        write_cube(v, cube + 4 * k, fcube + 4 * k);
        if (n > 0) {
            sys_off[0] = 0;
            sys_off[1] = n;
        }
    }
}

// keys in the caller's order, each relative to its own system's cube
__global__ void k_keys_sys(int n, const float *__restrict__ x, const float *__restrict__ y,
                           const float *__restrict__ z, const int32_t *__restrict__ sys_off, int nsys,
                           const double *__restrict__ cube, uint64_t *__restrict__ keys, int32_t *__restrict__ vals,
                           int32_t *__restrict__ hist)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int sy = sys_of_pos(sys_off, nsys, i);
    const uint64_t key = key_of(x[i], y[i], z[i], cube + 4 * sy);
    keys[i] = key;
    vals[i] = i;
    if (hist) atomicAdd(&hist[(i / RS_TILE) * 256 + (int)(key & 255u)], 1);
}

// system id of the particle at each position of the current order (digit source of the last passes)
__global__ void k_gather_sys(int n, const int32_t *__restrict__ vals, const int32_t *__restrict__ sys_off, int nsys,
                             uint64_t *__restrict__ skey, int32_t *__restrict__ hist)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int sy = sys_of_pos(sys_off, nsys, vals[i]);
    skey[i] = (uint64_t)sy;
    if (hist) atomicAdd(&hist[(i / RS_TILE) * 256 + (sy & 255)], 1);
}

// Morton keys again, in the final order (the system passes carried only the system digit)
__global__ void k_keys_sorted(int n, const float *__restrict__ x, const float *__restrict__ y,
                              const float *__restrict__ z, const int32_t *__restrict__ vals,
                              const int32_t *__restrict__ sys_off, int nsys, const double *__restrict__ cube,
                              uint64_t *__restrict__ keys, int32_t *__restrict__ vals_out)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int j = vals[s];
    const int sy = sys_of_pos(sys_off, nsys, j);
    keys[s] = key_of(x[j], y[j], z[j], cube + 4 * sy);
    if (vals_out) vals_out[s] = j;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------
int evol_scan_i32(evol_ctx *c, int n, const int32_t *in, int32_t *out, int write_total)
{
    if (n <= SCAN_ONE_MAX) {
        k_scan_one<<<1, SC_THREADS, 0, c->stream>>>(n, in, out, write_total);
        return evol_cuda_ok(cudaGetLastError());
    }
    int nparts = (n + SC_TILE - 1) / SC_TILE;
    if (nparts < 1) nparts = 1;
    k_scan_reduce<<<nparts, SC_THREADS, 0, c->stream>>>(n, in, c->d.scan_part);
    k_scan_top<<<1, SC_THREADS, 0, c->stream>>>(nparts, c->d.scan_part);
    k_scan_down<<<nparts, SC_THREADS, 0, c->stream>>>(n, in, out, c->d.scan_part, nparts, write_total);
    return evol_cuda_ok(cudaGetLastError());
}

namespace {
__global__ void k_active_flags(int n, const int32_t *__restrict__ orig, const int32_t *__restrict__ bact,
                               int32_t *__restrict__ actf)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n) actf[s] = bact[orig[s]];
}

__global__ void k_active_scatter(int n, const int32_t *__restrict__ actf, const int32_t *__restrict__ acts,
                                 int32_t *__restrict__ act)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n && actf[s]) act[acts[s]] = s;
}
}  // namespace

// The active list of an individual-time-step system step: the sorted positions of the flagged
// particles in ascending order (so that consecutive entries stay close in space), and their
// number at d.acts[n].
int evol_launch_active_list(evol_ctx *c, int n)
{
    evol_dev &d = c->d;
    int tb = 256, gb = (n + tb - 1) / tb;
    k_active_flags<<<gb, tb, 0, c->stream>>>(n, d.orig, d.bact, d.actf);
    int rc = evol_scan_i32(c, n, d.actf, d.acts, 1);
    if (rc) return rc;
    k_active_scatter<<<gb, tb, 0, c->stream>>>(n, d.actf, d.acts, d.act);
    return evol_cuda_ok(cudaGetLastError());
}

int evol_launch_build(evol_ctx *c, const evol_particles *p, const evol_params *prm)
{
    evol_dev &d = c->d;
    int n = (int)p->n;
    const int nsys = c->nsys > 0 ? c->nsys : 1;
    int leaf = prm->leaf_size > 0 ? prm->leaf_size : 8;
    cudaStream_t st = c->stream;
    int tb = 256, gb = (n + tb - 1) / tb;
    const int rsb = (n + RS_TILE - 1) / RS_TILE;
    const bool rank = n <= RANK_MAX, fused = !rank && n <= FUSED_MAX;
    // fused passes: a histogram of every tile for each of the passes
    int32_t *hist = (int32_t *)d.hist;
    const size_t hsize = (size_t)256 * rsb;
    int npass = 8;
    for (int shift = 0; nsys > 1 && (1ll << shift) < (long long)nsys; shift += 8) ++npass;
    if (fused && cudaMemsetAsync(hist, 0, npass * hsize * sizeof(int32_t), st) != cudaSuccess) return EVOL_ECUDA;
    int32_t *h0 = fused ? hist : nullptr;
    if (nsys == 1) {
        if (n <= RANK_MAX) {
            k_bbox_sys<<<1, 1024, 0, st>>>(n, d.sys_off, p->x, p->y, p->z, d.cube, d.fcube, d.err);
        } else {
            int nb = (int)c->bbox_blocks;
            k_bbox_partial<<<nb, BB_THREADS, 0, st>>>(n, p->x, p->y, p->z, d.bbox_part, d.err);
            k_bbox_final<<<1, 512, 0, st>>>(n, nb, d.bbox_part, d.cube, d.fcube, d.sys_off);
        }
        k_keys<<<gb, tb, 0, st>>>(n, p->x, p->y, p->z, d.cube, rank ? d.keys_b : d.keys_a, d.vals_a, h0);
    } else {
        // the offsets were copied into d.sys_off by the caller of this launcher
        // wide blocks for large systems, narrow ones where most of a wide block would have no particle (whole
        // builds with 1024 / 256 threads, ms: 16,000 systems of 90 particles 0.800 / 0.704, 1000 of 1450
        // 0.725 / 0.719, 250 of 5800 0.727 / 0.736, 64 of 23,000 0.690 / 0.727, 16 of 93,000 0.784 / 0.930)
        const int bt = n / nsys < 3000 ? BB_THREADS : 1024;
        k_bbox_sys<<<nsys, bt, 0, st>>>(0, d.sys_off, p->x, p->y, p->z, d.cube, d.fcube, d.err);
        k_keys_sys<<<gb, tb, 0, st>>>(n, p->x, p->y, p->z, d.sys_off, nsys, d.cube, rank ? d.keys_b : d.keys_a, d.vals_a,
                                      h0);
    }
    uint64_t *ka = d.keys_a, *kb = d.keys_b;
    int32_t *va = d.vals_a, *vb = d.vals_b;
    int done = 0;
    auto pass = [&](int shift, bool last) -> int {
        if (fused) {
            k_rs_scatter<true><<<rsb, RS_THREADS, 0, st>>>(n, ka, va, kb, vb, shift, hist + done * hsize, rsb,
                                                           last ? nullptr : hist + (done + 1) * hsize);
        } else {
            k_rs_hist<<<rsb, RS_THREADS, 0, st>>>(n, ka, shift, hist, rsb);
            const int rc = evol_scan_i32(c, 256 * rsb, hist, hist, 0);
            if (rc) return rc;
            k_rs_scatter<false><<<rsb, RS_THREADS, 0, st>>>(n, ka, va, kb, vb, shift, hist, rsb, nullptr);
        }
        ++done;
        uint64_t *tk = ka; ka = kb; kb = tk;
        int32_t *tv = va; va = vb; vb = tv;
        return EVOL_OK;
    };
    if (rank) {
        const int blocks = (n + 31) / 32;
        if (nsys == 1) k_rank_sort<false><<<blocks, 256, 0, st>>>(n, d.keys_b, d.sys_off, nsys, d.keys_a, d.vals_a);
        else k_rank_sort<true><<<blocks, 256, 0, st>>>(n, d.keys_b, d.sys_off, nsys, d.keys_a, d.vals_a);
    } else {
        for (int shift = 0; shift < 64; shift += 8)
            if (int rc = pass(shift, shift == 56)) return rc;
        // 8 passes: sorted keys and permutation are back in keys_a / vals_a
        if (nsys > 1) {
            // stable passes on the system id make the order (system, key); then the keys are recomputed
            k_gather_sys<<<gb, tb, 0, st>>>(n, d.vals_a, d.sys_off, nsys, d.keys_b, fused ? hist + 8 * hsize : nullptr);
            ka = d.keys_b; kb = d.keys_a; va = d.vals_a; vb = d.vals_b;
            for (int shift = 0; (1ll << shift) < (long long)nsys; shift += 8)
                if (int rc = pass(shift, (1ll << (shift + 8)) >= (long long)nsys)) return rc;
            // va holds the final permutation; rebuild keys_a / vals_a from it
            k_keys_sorted<<<gb, tb, 0, st>>>(n, p->x, p->y, p->z, va, d.sys_off, nsys, d.cube, d.keys_a,
                                             va == d.vals_a ? nullptr : d.vals_a);
        }
    }
    k_permute<<<gb, tb, 0, st>>>(n, (int)p->n_gas, d.vals_a, p->x, p->y, p->z, p->vx, p->vy, p->vz, p->m, p->u,
                                 p->h, p->eps, d.pos, d.vel, d.len_h, d.len_eps, d.orig, d.inv,
                                 c->pred_dt, c->kdk_acc, c->cap, c->pred_tau, d.keys_a, d.sys_off, nsys, d.lcp,
                                 d.sys_sorted);
    k_count<<<gb, tb, 0, st>>>(n, d.lcp, leaf, d.cnt);
    int rc = evol_scan_i32(c, n, d.cnt, d.base, 1);
    if (rc) return rc;
    k_fill<<<gb, tb, 0, st>>>(n, d.keys_a, d.lcp, d.sys_off, d.sys_sorted, d.base, leaf, c->node_cap, d.nbeg, d.nend,
                              d.nlev, d.nnext, d.nnodes, d.err);
    int ng = c->num_sms * 8;
    k_link<<<ng, 256, 0, st>>>(d.nnodes, leaf, d.nbeg, d.nend, d.nlev, d.nnext, d.nparent, d.nnch, d.narrive, d.nI,
                               d.nK0, d.nK1, nsys, d.sys_off, d.base, d.sys_root);
    NodeOut o{d.nA, d.nB, d.nC, d.nQ0, d.nQ1, d.nBmin, d.nBmax, d.nCoff, d.nM64, d.nC64, d.nQ64};
    const Links L{d.nnodes, d.nparent, d.nnch, d.nI, d.nK0, d.nK1, d.narrive, d.err};
    const bool mixed = prm->precision == EVOL_FP32_MIXED;
    if (mixed) k_moments<double><<<c->num_sms * 5, 128, 0, st>>>(L, (int)p->n_gas, d.pos, d.orig, d.keys_a, d.fcube, d.sys_sorted, o);
    else k_moments<float><<<c->num_sms * 8, 128, 0, st>>>(L, (int)p->n_gas, d.pos, d.orig, d.keys_a, d.fcube, d.sys_sorted, o);
    k_node_geometry<<<ng, 256, 0, st>>>(d.nnodes, d.nI, d.keys_a, d.cube, d.fcube, d.sys_sorted, prm->theta, o, mixed);
    return evol_cuda_ok(cudaGetLastError());
}

int evol_launch_node_lengths(evol_ctx *c, const evol_params *prm, int n_gas)
{
    evol_dev &d = c->d;
    (void)prm;
    const Links L{d.nnodes, d.nparent, d.nnch, d.nI, d.nK0, d.nK1, d.narrive, d.err};
    k_node_lengths<<<c->num_sms * 8, 128, 0, c->stream>>>(L, n_gas, d.orig, d.len_eps, d.len_h, d.nB, d.nC);
    return evol_cuda_ok(cudaGetLastError());
}
