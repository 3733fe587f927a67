// Smoothing and softening lengths (Sect. 2.1 Eqs. rho0, etan, iter; Sect. 3 Eqs. hn, nsum,
// densitySPH, drhodr; Sect. 3.1 "gather" view with an enlarged search radius).
//
// Each particle i needs the particles within its search radius R_i = 2 L_i (1 + 0.1).  A block of
// NW = 4 or 8 warps (see Shape) takes NW SUB consecutive particles in key order, SUB to a warp (set by
// evol_params.length_group, see warp_particles; by default chosen from their number, see group_size).
// The block finds the leaves whose particle box comes within a warp's largest R_i of that warp's
// particle box, from the leaf list of their super-group (k_leaf_lists) or by one walk of the tree
// for all of them, popping up to 32 nodes a warp at a time; the particles of those leaves (the
// candidates) are copied to shared memory, with the box of every 32 of them (a chunk).  Where the
// candidates do not fit, the first of each warp's particles that should fit are taken and the others
// wait for a later round.  A particle then tests the chunks against its own ball and the candidates of
// the chunks that pass; those inside the ball are listed as distances with candidates or masses in
// shared memory.  A particle whose radius grows beyond its warp's waits for a later round too, and one
// whose block's candidates did not fit even for single particles walks the tree on its own.
// On its list a particle solves
//     F(L) = L^3 n(L) - eta^3 = 0,   n(L) = sum_j W(r_ij, L)  (self term included)
// by Newton steps in L^3 kept inside a bisection bracket, gathering again when 2L leaves the gathered
// radius.  F is non-decreasing in L, so the root is unique.  With w(u) = pi L^3 W the sums are
// dimensionless:
//     F = Sw/pi - eta^3,  F' = -Suw/(pi L),  Sw = sum w(u),  Suw = sum u w'(u).
// Four particles are solved together, eight lanes to each (lists of up to SCAP entries); a particle
// whose list does not fit, or that fails to converge there, is solved again by the whole warp with a
// list of up to PCAP entries.  Where most lists would not fit (see whole_warp) every particle is
// solved by the whole warp.
// Outputs (mode 0, gas h):   rho = Smw/(pi h^3), Omega* = -Suw/(3 Sw),
//                           zeta = (3 Smw + Smuw)/(3 Sw)          (Sect. 3, Eq. drhodr)
// Outputs (mode 1, eps):     Upsilon = -Suw/(3 Sw),
//                           X = -(pi eps^2/(3 Sw)) sum_k m_k eps^2 dphi/deps   (Sect. 2.1)
// Mode 2: both, for particle sets that are all gas with the same neighbour number for h and eps, whose
// two root equations are then the same (evol_shared_lengths): one solve instead of two, 4.6 ms instead of
// 9.0 for an ensemble of 64 spheres (1.76 M particles).
// On request, any mode:     div v = 3 sum_j ((v_i - v_j).(r_i - r_j)/r_ij) w'(u) / (L Suw)
//                           (the discretised continuity equation of Sect. 2.1)
// Standard SPH scheme (Sect. 3, mode 0 on request): no root is solved.  Once a gathered ball holds
// at least N + 1 gas particles (the particle itself included), h = (r_(N) + r_(N+1)) / 4 from the
// N-th and (N+1)-th smallest distances, so that exactly N lie inside 2h; then one evaluation with
// Omega* = 1, zeta = 0 (the grad-h terms are dropped) and div v, curl v normalised by n alone.
#include <cuda_runtime.h>
#include <stdint.h>

#include "evol_internal.cuh"

namespace {

constexpr int SCAP = 176;             // neighbour entries of each of four particles solved together
                                      // (SCAP mod 32 = 16 words: their pairwise reads do not conflict)
constexpr int PCAP = 336;             // neighbour entries of a particle solved by the whole warp
constexpr int MAX_ROUNDS = 24;        // rounds of an item after which a particle is left to the whole warp
// Two shapes of block.  Four warps, six blocks per SM, is the faster one as long as the candidates of its
// particles fit (eps of 2^20 Plummer particles: 2.4 ms against 2.6); eight warps with twice the candidates,
// three blocks per SM, where they mostly do not and four warps would go over the leaf list again for parts
// of the particles (eps of 2^21 halo + 2^20 gas: 9.6 ms against 11.5).  The mean number of candidates per
// super-group, which k_leaf_lists counts, decides on the device: 3360 to 3800 of them (Plummer, the gas of
// either, collapsing spheres) want the first, 5370 to 5870 (halo and gas together) the second.  The variants
// with the velocity divergence, whose blocks hold more, and the periodic ones have the first only.
template <int NW, bool FLOW>
struct Shape {
    static constexpr int CC = NW == 8 ? 2400 : 1216;   // candidates staged per block
    static constexpr int NCHUNK = CC / 32;
    static constexpr int LCAP = NW * 4 * SCAP * 3 / 4 - 1;             // leaves listed (in the lists' room)
    static constexpr int MINB = NW == 8 ? 3 : (FLOW ? 5 : 6);          // blocks per SM
};
constexpr unsigned long long WIDE_CANDIDATES = 4600;               // per super-group: the wide shape above this
constexpr int MAX_ITERS = 60;
constexpr int MAX_WALKS = 24;
constexpr float SEARCH_MARGIN = 1.1f;
// Relative step below which one last evaluation is taken: a Newton step that small leaves an
// error of the order of its square (the iteration converges quadratically), far below FP32
// resolution; a bisection step must be smaller, as it halves the error only.
constexpr float NEWTON_TOL = 1e-4f;
constexpr float CONV_TOL = 1e-6f;

// Particles of a solve (gas of an h solve) from which its leaf lists are made; below, the blocks' own walks cost
// less than one more launch (h of 20,000 gas particles among 544 k: 0.29 ms against 0.41 with lists, 60,000
// 0.47 against 0.55; 49,152 of their own 0.38 against 0.41).
constexpr int LISTS_MIN = 65536;
constexpr int LEN_SG = 256;           // list entries per super-group of k_leaf_lists (a multiple of 32 per warp)
constexpr int SG_LEAVES = EVOL_SG_ACAP * LEN_SG / (32 * EVOL_SG_GROUPS);   // leaves of its list at most

enum { ST_DONE = 0, ST_ACTIVE = 1, ST_LAST = 2 };

// Neighbour lists of a warp: four of SCAP entries (distance and candidate), or one of PCAP entries
// (distance, and mass or -- when the velocity divergence is wanted -- the index bits).
union WarpLists {
    struct {
        float r[4 * SCAP];
        unsigned short id[4 * SCAP];
    };
    float2 one[PCAP];
};

template <int NW, bool FLOW>
struct LenSmem {
    static constexpr int CC = Shape<NW, FLOW>::CC, NCHUNK = Shape<NW, FLOW>::NCHUNK;
    union {
        struct {
            float cx[CC], cy[CC], cz[CC], cm[CC];   // candidates: position, mass
        };
        int stk[4 * CC];              // the walk's stack, before they are copied
    };
    union {
        WarpLists nb[NW];
        int2 leaf[Shape<NW, FLOW>::LCAP + 1];          // the walk's leaves: first particle of each, prefix of their counts
    };
    float lo[3][NCHUNK], hi[3][NCHUNK];   // chunk boxes
    float4 gc[NW];              // per warp: centre of its particles' box, squared radius (-1: none)
    float4 gh[NW];              // and half widths
    int2 ws[2][NW];             // per-warp totals of the scans of leaves and candidates
    int sel[NW], nsel[NW], first[NW], listed[NW], item;   // per warp: lowest
                                      // pending system, the round's particles, the first of them, list use
    unsigned lc[NW][5];         // work counts of the warp's current item (kept by lane 0)
    int cj[FLOW ? CC : 1];            // sorted index of each candidate
};

template <bool PER>
__device__ __forceinline__ float image(float d, const evol_kparams &kp, int a)
{
    return PER ? evol_nearest(d, kp.plen[a], kp.pinv[a]) : d;
}

// Minimum and maximum over the warp's lanes (one reduction instruction each).
__device__ __forceinline__ float warp_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// The k-th smallest (k >= 1) of the cnt <= PCAP listed distances: the smallest x with at least k
// distances <= x, by bisection on the bit patterns (non-negative floats order like their bits).
__device__ __forceinline__ float kth_distance(const float2 *nb, int cnt, int k, int lane)
{
    unsigned lo = 0u, hi = 0x7f800000u;
    while (lo < hi) {
        const unsigned mid = lo + ((hi - lo) >> 1);
        int c = 0;
        for (int e = lane; e < cnt; e += 32) c += __float_as_uint(nb[e].x) <= mid ? 1 : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (c >= k) hi = mid;
        else lo = mid + 1u;
    }
    return __uint_as_float(lo);
}

// The candidates of a tree node's particle range: all its particles, or (h solve of a set that is not
// all gas) its gas particles, which d.gpos holds in key order.
template <int MODE>
__device__ __forceinline__ bool gas_lists(const evol_kparams &kp)
{
    return MODE == 0 && kp.n_gas < kp.n;
}

// f over the block's per-warp values.
template <int NW, typename F>
__device__ __forceinline__ int over_warps(const int (&v)[NW], F f)
{
    int r = v[0];
#pragma unroll
    for (int q = 1; q < NW; ++q) r = f(r, v[q]);
    return r;
}

// Does the box (c, hw) come within a warp's radius of that warp's particle box?
template <int NW, bool PER, bool FLOW>
__device__ __forceinline__ bool near_groups(const evol_kparams &kp, const LenSmem<NW, FLOW> &sm, float cx, float cy,
                                            float cz, float hx, float hy, float hz)
{
    bool hit = false;
#pragma unroll
    for (int q = 0; q < NW; ++q) {
        const float4 G = sm.gc[q], H = sm.gh[q];
        const float ex = fmaxf(fabsf(image<PER>(cx - G.x, kp, 0)) - (hx + H.x), 0.f);
        const float ey = fmaxf(fabsf(image<PER>(cy - G.y, kp, 1)) - (hy + H.y), 0.f);
        const float ez = fmaxf(fabsf(image<PER>(cz - G.z, kp, 2)) - (hz + H.z), 0.f);
        hit = hit || ex * ex + ey * ey + ez * ez < G.w;
    }
    return hit;
}

// The deepest node around a round's first particle whose cube holds every warp's box with its radius:
// no particle outside it can be a candidate, so the walk starts there instead of at the root and spends no
// steps (a round trip to L2 each) on the levels above.  The leaf of sorted position s is node
// d.base[s + 1] - 1 (pre-order: the last node that begins at or before s); the climb from it takes one load
// per level.  Boxes that straddle a high-level boundary start at the root.
template <int NW, bool FLOW>
__device__ int start_node(const evol_dev &d, const LenSmem<NW, FLOW> &sm, int sys, int root)
{
    const double *cb = d.cube + 4 * sys;
    const float x = (float)cb[0], y = (float)cb[1], z = (float)cb[2];      // exact: float minima
    const float sc = (float)(1 << EVOL_MAXLEVEL) / (float)cb[3];            // a power of two
    const float top = (float)((1 << EVOL_MAXLEVEL) - 1);
    unsigned diff = 0u;
    int s0 = -1;
    unsigned c0[3] = {0u, 0u, 0u};
#pragma unroll
    for (int q = 0; q < NW; ++q) {
        const float4 G = sm.gc[q], H = sm.gh[q];
        if (G.w < 0.f) continue;
        // outward by 1e-3 of the radius and a part in 2^20 of the coordinates, far above the rounding of both, and
        // by half a finest cell: the offset from the cube's corner is rounded by up to an eighth of one, which is
        // more than the radius of particles far closer to each other than these cells are wide
        const float R = 1.001f * sqrtf(G.w);
        const float o[3] = {x, y, z}, c[3] = {G.x, G.y, G.z}, h[3] = {H.x, H.y, H.z};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float r = R + h[a] + 1e-6f * (fabsf(c[a]) + h[a]);
            const unsigned l = (unsigned)fminf(fmaxf((c[a] - r - o[a]) * sc - 0.5f, 0.f), top);
            const unsigned u = (unsigned)fminf(fmaxf((c[a] + r - o[a]) * sc + 0.5f, 0.f), top);
            if (s0 < 0) c0[a] = l;
            diff |= (l ^ c0[a]) | (u ^ c0[a]);
        }
        if (s0 < 0) s0 = sm.first[q];
    }
    const int lev = EVOL_MAXLEVEL - (32 - __clz((int)diff));       // the cube's level
    if (s0 < 0 || lev < 3) return root;
    int node = d.base[s0 + 1] - 1;
    if (node >= *d.nnodes) return root;               // a node list that overflowed (flagged by the build)
    for (int k = 0; k <= EVOL_MAXLEVEL && node > root; ++k) {
        if (d.nlev[node] <= lev) return node;
        node = d.nparent[node];
    }
    return root;
}

// Block-wide tree walk from `root`: lists the leaves whose particle box comes within a warp's radius of
// that warp's box (sm.gc, sm.gh).  Returns the number of their particles (the candidates), -1 when they,
// the leaves or the stack do not fit, -2 on a corrupt tree (the error word is set).  IDS: the leaves are
// listed by node, and their particles need not fit.  The same on every thread.
template <int NW, int MODE, bool PER, bool FLOW, bool IDS>
__device__ int block_walk(const evol_dev &d, const evol_kparams &kp, LenSmem<NW, FLOW> &sm, int root, long long pop_cap, int &nleaf_out)
{
    constexpr int CC = Shape<NW, FLOW>::CC, LCAP = Shape<NW, FLOW>::LCAP;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int cap = min(4 * CC, 2 * kp.stack_cap);
    int top = 1, nleaf = 0, ncand = 0;
    if (tid == 0) sm.stk[0] = root;
    __syncthreads();
    long long pops = 0;
    while (top > 0) {
        if (++pops > pop_cap) {
            if (tid == 0) {
                evol_flag(d.err, EVOL_ETIMEOUT);
                atomicMax(&d.counters[7], 2ull);
            }
            return -2;
        }
        const int k = min(top, (32 * NW));
        top -= k;
        int nch = 0, c = 0, b = 0, node = 0;
        int ch[8];
        if (tid < k) {
            // every operand of the node at once: one round trip to L2 per step of the walk
            node = sm.stk[top + tid];
            const int4 I = d.nI[node];
            const float4 B = d.nB[node], C = d.nC[node];
            const int4 K0 = d.nK0[node], K1 = d.nK1[node];
            const bool open = (MODE != 0 || B.w >= 0.f) && near_groups<NW, PER, FLOW>(kp, sm, B.x, B.y, B.z, C.x, C.y, C.z);
            if (open) {
                if ((I.x >> 8) & 1) {
                    int e = I.w;
                    b = I.z;
                    if (gas_lists<MODE>(kp)) {
                        b = d.gbase[b];
                        e = d.gbase[e];
                    }
                    c = e - b;
                } else {
                    ch[0] = K0.x; ch[1] = K0.y; ch[2] = K0.z; ch[3] = K0.w;
                    ch[4] = K1.x; ch[5] = K1.y; ch[6] = K1.z; ch[7] = K1.w;
#pragma unroll
                    for (int t = 0; t < 8; ++t) nch += ch[t] >= 0 ? 1 : 0;
                }
            }
        }
        // positions of the children (low half) and leaves (high half), and of the candidates
        int p = nch | (c > 0 ? 1 << 16 : 0), cc = min(c, CC + 1);
        const int p0 = p, cc0 = cc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int tp = __shfl_up_sync(0xffffffffu, p, o), tc = __shfl_up_sync(0xffffffffu, cc, o);
            if (lane >= o) {
                p += tp;
                cc += tc;
            }
        }
        if (lane == 31) sm.ws[0][w] = make_int2(p, cc);
        __syncthreads();
        int pb = 0, cb = 0, pt = 0, ct = 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const int2 v = sm.ws[0][q];
            if (q < w) {
                pb += v.x;
                cb += v.y;
            }
            pt += v.x;
            ct += v.y;
        }
        if (top + (pt & 0xffff) > cap || nleaf + (pt >> 16) > LCAP || (!IDS && ncand + ct > CC)) return -1;
        const int at = pb + p - p0;
        if (nch) {
            const int o = top + (at & 0xffff);
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (t < nch) sm.stk[o + t] = ch[t];
        }
        if (c > 0) sm.leaf[nleaf + (at >> 16)] = make_int2(IDS ? node : b, ncand + cb + cc - cc0);
        top += pt & 0xffff;
        nleaf += pt >> 16;
        ncand += ct;
        __syncthreads();
    }
    nleaf_out = nleaf;
    return ncand;
}

// The leaves of a super-group's list (k_leaf_lists) that the block's own boxes reach, as block_walk lists
// them: a few independent turns over the list instead of a chain of tree levels.  Where they do not fit,
// returns -1 with the number of their candidates in nleaf_out.
template <int NW, int MODE, bool PER, bool FLOW>
__device__ int list_leaves(const evol_dev &d, const evol_kparams &kp, LenSmem<NW, FLOW> &sm, const int *list, int nl,
                           int &nleaf_out)
{
    constexpr int CC = Shape<NW, FLOW>::CC, LCAP = Shape<NW, FLOW>::LCAP;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int nleaf = 0, ncand = 0, buf = 0;
    for (int t0 = 0; t0 < nl; t0 += (32 * NW)) {
        int c = 0, b = 0;
        if (t0 + tid < nl) {
            const int node = list[t0 + tid];
            const int4 I = d.nI[node];
            const float4 B = d.nB[node], C = d.nC[node];
            if (near_groups<NW, PER, FLOW>(kp, sm, B.x, B.y, B.z, C.x, C.y, C.z)) {
                int e = I.w;
                b = I.z;
                if (gas_lists<MODE>(kp)) {
                    b = d.gbase[b];
                    e = d.gbase[e];
                }
                c = e - b;
            }
        }
        const unsigned lm = __ballot_sync(0xffffffffu, c > 0);
        int cc = min(c, CC + 1);
        const int cc0 = cc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int tc = __shfl_up_sync(0xffffffffu, cc, o);
            if (lane >= o) cc += tc;
        }
        if (lane == 31) sm.ws[buf][w] = make_int2(__popc(lm), cc);
        __syncthreads();
        int at = nleaf + __popc(lm & ((1u << lane) - 1u)), cb = ncand;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const int2 v = sm.ws[buf][q];
            if (q < w) {
                at += v.x;
                cb += v.y;
            }
            nleaf += v.x;
            ncand += v.y;
        }
        buf ^= 1;                     // the next turn's totals go to the other row: one barrier a turn
        if (c > 0 && at < LCAP) sm.leaf[at] = make_int2(b, cb + cc - cc0);
    }
    const bool fit = nleaf <= LCAP && ncand <= CC;
    nleaf_out = fit ? nleaf : max(ncand, CC + 1);
    return fit ? ncand : -1;
}

// Copies the candidates to shared memory, a half-warp to a leaf, and forms the chunk boxes.
template <int NW, int MODE, bool FLOW>
__device__ void stage_candidates(const evol_dev &d, const evol_kparams &kp, LenSmem<NW, FLOW> &sm, int nleaf, int ncand)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const float4 *src = gas_lists<MODE>(kp) ? d.gpos : d.pos;
    if (tid == 0) sm.leaf[nleaf] = make_int2(0, ncand);
    __syncthreads();
#pragma unroll 2
    for (int l = tid >> 4; l < nleaf; l += (32 * NW) / 16) {
        const int2 q = sm.leaf[l];
        const int c = sm.leaf[l + 1].y - q.y;
        for (int t = tid & 15; t < c; t += 16) {
            const float4 p = src[q.x + t];
            sm.cx[q.y + t] = p.x;
            sm.cy[q.y + t] = p.y;
            sm.cz[q.y + t] = p.z;
            sm.cm[q.y + t] = p.w;
            if (FLOW) sm.cj[q.y + t] = gas_lists<MODE>(kp) ? d.glist[q.x + t] : q.x + t;
        }
    }
    // the last chunk is filled up with points that no ball holds
    for (int t = ncand + tid; t < ((ncand + 31) & ~31); t += (32 * NW)) sm.cx[t] = sm.cy[t] = sm.cz[t] = INFINITY;
    __syncthreads();
    for (int c = w; c * 32 < ncand; c += NW) {
        const int e = c * 32 + lane;
        const bool in = e < ncand;
        const float x = sm.cx[e], y = sm.cy[e], z = sm.cz[e];
        const float lx = warp_min(in ? x : INFINITY), ly = warp_min(in ? y : INFINITY), lz = warp_min(in ? z : INFINITY);
        const float ux = warp_max(in ? x : -INFINITY), uy = warp_max(in ? y : -INFINITY),
                    uz = warp_max(in ? z : -INFINITY);
        if (lane == 0) {
            sm.lo[0][c] = lx; sm.lo[1][c] = ly; sm.lo[2][c] = lz;
            sm.hi[0][c] = ux; sm.hi[1][c] = uy; sm.hi[2][c] = uz;
        }
    }
    __syncthreads();
}

// A particle's neighbour list from the staged candidates: those within sqrt(R2) of (px, py, pz).  put(k,
// r2, candidate) stores entry k.  Returns their number.
template <int NW, bool PER, bool FLOW, typename Put>
__device__ __forceinline__ int gather_staged(const evol_kparams &kp, const LenSmem<NW, FLOW> &sm, int ncand, int lane,
                                             float px, float py, float pz, float R2, Put put)
{
    const unsigned ltmask = (1u << lane) - 1u;
    const int nchunk = (ncand + 31) >> 5;
    const f32x2 PX = pk2(px, px), PY = pk2(py, py), PZ = pk2(pz, pz);
    int cnt = 0;
    for (int c0 = 0; c0 < nchunk; c0 += 32) {
        const int c = c0 + lane;
        bool hit = false;
        if (c < nchunk) {
            const float lx = sm.lo[0][c], ly = sm.lo[1][c], lz = sm.lo[2][c];
            const float ux = sm.hi[0][c], uy = sm.hi[1][c], uz = sm.hi[2][c];
            float ex, ey, ez;
            if (PER) {
                ex = fabsf(image<true>(0.5f * (lx + ux) - px, kp, 0)) - 0.5f * (ux - lx);
                ey = fabsf(image<true>(0.5f * (ly + uy) - py, kp, 1)) - 0.5f * (uy - ly);
                ez = fabsf(image<true>(0.5f * (lz + uz) - pz, kp, 2)) - 0.5f * (uz - lz);
            } else {
                ex = fmaxf(lx - px, px - ux);
                ey = fmaxf(ly - py, py - uy);
                ez = fmaxf(lz - pz, pz - uz);
            }
            ex = fmaxf(ex, 0.f);
            ey = fmaxf(ey, 0.f);
            ez = fmaxf(ez, 0.f);
            hit = ex * ex + ey * ey + ez * ez < R2;
        }
        unsigned hm = __ballot_sync(0xffffffffu, hit);
        // two chunks a turn, in packed arithmetic
        while (hm) {
            const int ea = (c0 + __ffs(hm) - 1) * 32 + lane;
            hm &= hm - 1u;
            const bool two = hm != 0u;
            const int eb = two ? (c0 + __ffs(hm) - 1) * 32 + lane : ea;
            hm &= hm - 1u;
            f32x2 dx = sub2(PX, pk2(sm.cx[ea], sm.cx[eb])), dy = sub2(PY, pk2(sm.cy[ea], sm.cy[eb])),
                  dz = sub2(PZ, pk2(sm.cz[ea], sm.cz[eb]));
            if (PER) {
                dx = pk2(image<true>(lo2(dx), kp, 0), image<true>(hi2(dx), kp, 0));
                dy = pk2(image<true>(lo2(dy), kp, 1), image<true>(hi2(dy), kp, 1));
                dz = pk2(image<true>(lo2(dz), kp, 2), image<true>(hi2(dz), kp, 2));
            }
            const f32x2 rr = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
            const float ra = lo2(rr), rb = hi2(rr);
            const bool ina = ra < R2, inb = two && rb < R2;
            const unsigned bala = __ballot_sync(0xffffffffu, ina), balb = __ballot_sync(0xffffffffu, inb);
            const int oa = cnt + __popc(bala & ltmask);
            cnt += __popc(bala);
            const int ob = cnt + __popc(balb & ltmask);
            cnt += __popc(balb);
            if (ina) put(oa, ra, ea);
            if (inb) put(ob, rb, eb);
        }
    }
    return cnt;
}

// The same by the particle's own walk from `root`, a warp at a time.  Returns -1 when the walk had to
// stop (corrupt tree or stack overflow; the error word is set).  A list that overflows is of no use, and its
// ball can be the whole set (far outliers of a small sphere), so the walk ends there with a count above cap:
// 9000 particles 3.02 -> 0.82 ms for the solve, 20,000 1.34 -> 0.87 (0.47 and 0.69 with the turns below).
template <int MODE, bool PER, bool FLOW>
__device__ __forceinline__ int gather_ball(const evol_dev &d, const evol_kparams &kp, float2 *nb, int cap, int lane, int *stk, long long pop_cap, int root, float px,
                                        float py, float pz, float R2)
{
    const unsigned ltmask = (1u << lane) - 1u;
    const int stack_cap = 2 * kp.stack_cap;
    if (lane == 0) stk[0] = root;
    int top = 1, cnt = 0;
    __syncwarp();
    long long pops = 0;
    while (top > 0) {
        if (++pops > pop_cap) {
            if (lane == 0) {
                evol_flag(d.err, EVOL_ETIMEOUT);
                atomicMax(&d.counters[7], 2ull);
            }
            return -1;
        }
        const int k = min(top, 32);
        top -= k;
        const int node = lane < k ? stk[top + lane] : -1;
        __syncwarp();
        int nch = 0, b = 0, e = 0;
        int ch[8];
        if (lane < k) {
            const int4 I = d.nI[node];
            const float4 B = d.nB[node], C = d.nC[node];
            const int4 K0 = d.nK0[node], K1 = d.nK1[node];
            bool open = false;
            if (MODE != 0 || B.w >= 0.f) {
                const float ex = fmaxf(fabsf(image<PER>(B.x - px, kp, 0)) - C.x, 0.f);
                const float ey = fmaxf(fabsf(image<PER>(B.y - py, kp, 1)) - C.y, 0.f);
                const float ez = fmaxf(fabsf(image<PER>(B.z - pz, kp, 2)) - C.z, 0.f);
                open = ex * ex + ey * ey + ez * ez < R2;
            }
            if (open) {
                if ((I.x >> 8) & 1) {
                    b = I.z;
                    e = I.w;
                    if (gas_lists<MODE>(kp)) {
                        b = d.gbase[b];
                        e = d.gbase[e];
                    }
                } else {
                    ch[0] = K0.x; ch[1] = K0.y; ch[2] = K0.z; ch[3] = K0.w;
                    ch[4] = K1.x; ch[5] = K1.y; ch[6] = K1.z; ch[7] = K1.w;
#pragma unroll
                    for (int t = 0; t < 8; ++t) nch += ch[t] >= 0 ? 1 : 0;
                }
            }
        }
        // the leaves' particles one after the other, 32 a turn (a leaf a turn took four times as many turns,
        // each a round trip to L2, with leaves of eight)
        int li = e - b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, li, o);
            if (lane >= o) li += t;
        }
        const int lt = __shfl_sync(0xffffffffu, li, 31), l0 = e - li;      // position of entry t: l0 + t
        for (int t0 = 0; t0 < lt && cnt <= cap; t0 += 32) {
            const int t = t0 + lane;
            int q = 0;                          // the leaf of entry t: the first with more entries up to its end
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, li, q + o - 1) <= t) q += o;
            const int j = __shfl_sync(0xffffffffu, l0, q & 31) + t;
            bool in = false;
            float r2 = 0.f, m = 0.f;
            if (t < lt) {
                const float4 p = gas_lists<MODE>(kp) ? d.gpos[j] : d.pos[j];
                const float dx = image<PER>(px - p.x, kp, 0), dy = image<PER>(py - p.y, kp, 1),
                            dz = image<PER>(pz - p.z, kp, 2);
                r2 = dx * dx + dy * dy + dz * dz;
                in = r2 < R2;
                m = p.w;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, in);
            if (in) {
                const int o = cnt + __popc(bal & ltmask);
                if (o < cap)
                    nb[o] = make_float2(sqrtf(r2), FLOW ? __int_as_float(gas_lists<MODE>(kp) ? d.glist[j] : j) : m);
            }
            cnt += __popc(bal);
        }
        if (cnt > cap) return cnt;
        int incl = nch;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        if (top + total > stack_cap) {
            if (lane == 0) evol_flag(d.err, EVOL_EOVERFLOW);
            return -1;
        }
        if (nch) {
            const int pos = top + incl - nch;
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (t < nch) stk[pos + t] = ch[t];
        }
        top += total;
        __syncwarp();
    }
    return cnt;
}

// Kernel sums over a neighbour list, combined over groups of LANES lanes (LANES entries at a time).
struct Sums {
    float w, uw;                      // Sw, Suw
    float mw, muw, mp;                // mass-weighted: w, u w', eps^2 dphi/deps
    float dv, cx, cy, cz;             // velocity divergence and curl
};

template <int LANES>
__device__ __forceinline__ float lanes_sum(float v)
{
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;                         // the same on every lane of the group (each step adds one pair)
}

// Sw and Suw over a list of the whole warp.
__device__ __forceinline__ void newton_sums_one(const float2 *nb, int cnt, int lane, float Linv, float &Sw, float &Suw)
{
    Sw = Suw = 0.f;
    for (int e = lane; e < cnt; e += 32) {
        const float u = nb[e].x * Linv;
        const float aa = fmaxf(2.f - u, 0.f), bb = fmaxf(1.f - u, 0.f);
        const float a2 = aa * aa, b2 = bb * bb;
        Sw += 0.25f * a2 * aa - b2 * bb;                    // w(u)
        Suw += u * (-0.75f * a2 + 3.f * b2);                // u w'(u)
    }
    Sw = lanes_sum<32>(Sw);
    Suw = lanes_sum<32>(Suw);
}

// The same over a list of eight lanes (an even number of distances), two entries a turn in packed
// arithmetic.
__device__ __forceinline__ void newton_sums_four(const float *r, int cnt, int sub, float Linv, float &Sw, float &Suw)
{
    const f32x2 LI = pk2(Linv, Linv), TWO = pk2(2.f, 2.f), ONE = pk2(1.f, 1.f);
    const f32x2 C75 = pk2(-0.75f, -0.75f), C3 = pk2(3.f, 3.f);
    f32x2 sw = 0ull, sb = 0ull, su = 0ull;                  // sum a^3, sum b^3, sum u w'(u)
    for (int e = 2 * sub; e < cnt; e += 16) {
        const float2 rr = *reinterpret_cast<const float2 *>(r + e);
        const f32x2 u = mul2(pk2(rr.x, rr.y), LI);
        const f32x2 ta = sub2(TWO, u), tb = sub2(ONE, u);
        const f32x2 a = pk2(fmaxf(lo2(ta), 0.f), fmaxf(hi2(ta), 0.f));
        const f32x2 b = pk2(fmaxf(lo2(tb), 0.f), fmaxf(hi2(tb), 0.f));
        const f32x2 a2 = mul2(a, a), b2 = mul2(b, b);
        sw = fma2(a2, a, sw);
        sb = fma2(b2, b, sb);
        su = fma2(u, fma2(a2, C75, mul2(b2, C3)), su);
    }
    Sw = lanes_sum<8>(0.25f * (lo2(sw) + hi2(sw)) - (lo2(sb) + hi2(sb)));
    Suw = lanes_sum<8>(lo2(su) + hi2(su));
}

// The last evaluation: entry(e, r, m, p, v) gives entry e's distance and mass and, for the continuity
// equation, its position and velocity.
template <int MODE, bool PER, bool FLOW, int LANES, typename Entry>
__device__ __forceinline__ Sums last_sums(const evol_dev &d, const evol_kparams &kp, int cnt, int sub, float Linv,
                                          float px, float py, float pz, int si, Entry entry)
{
    Sums S = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const bool curl = FLOW && MODE != 1 && kp.want_curl;
    const float4 vi = FLOW && si >= 0 ? d.vel[si] : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int e = sub; e < cnt; e += LANES) {
        float r, m;
        float3 pj = make_float3(0.f, 0.f, 0.f), vj = pj;
        entry(e, r, m, pj, vj);
        const float u = r * Linv;
        float wv, dw;
        evol_w_dw(u, wv, dw);          // zero for u >= 2
        S.w += wv;
        S.uw += u * dw;
        if (MODE != 1) {
            S.mw += m * wv;
            S.muw += m * u * dw;
        }
        if (MODE != 0) S.mp += m * evol_dphideps(u);
        if (FLOW) {
            // (v_i - v_j).(r_i - r_j) / r  w'(u)  (Sect. 2.1, continuity equation); the particle itself has
            // no direction
            const float dx = image<PER>(px - pj.x, kp, 0), dy = image<PER>(py - pj.y, kp, 1),
                        dz = image<PER>(pz - pj.z, kp, 2);
            const float ux = vi.x - vj.x, uy = vi.y - vj.y, uz = vi.z - vj.z;
            const float q = r > 0.f ? dw / r : 0.f;
            S.dv += (ux * dx + uy * dy + uz * dz) * q;
            if (curl) {
                // (v_i - v_j) x (r_i - r_j) / r  w'(u)
                S.cx += (uy * dz - uz * dy) * q;
                S.cy += (uz * dx - ux * dz) * q;
                S.cz += (ux * dy - uy * dx) * q;
            }
        }
    }
    S.w = lanes_sum<LANES>(S.w);
    S.uw = lanes_sum<LANES>(S.uw);
    if (MODE != 1) {
        S.mw = lanes_sum<LANES>(S.mw);
        S.muw = lanes_sum<LANES>(S.muw);
    }
    if (MODE != 0) S.mp = lanes_sum<LANES>(S.mp);
    if (FLOW) {
        S.dv = lanes_sum<LANES>(S.dv);
        if (curl) {
            S.cx = lanes_sum<LANES>(S.cx);
            S.cy = lanes_sum<LANES>(S.cy);
            S.cz = lanes_sum<LANES>(S.cz);
        }
    }
    return S;
}

// Results of the particle at sorted position si with length L (std: standard scheme).
template <int MODE, bool FLOW>
__device__ __forceinline__ void write_result(const evol_dev &d, const evol_kparams &kp, int si, float L, float Linv,
                                             const Sums &S, bool std_)
{
    const float k = 1.f / EVOL_PI_F * Linv * Linv * Linv;
    const float corr = -S.uw / (3.f * S.w);
    if (MODE != 1) {
        d.len_h[si] = L;
        d.nh[si] = S.w * k;
        d.rho[si] = S.mw * k;
        d.omega[si] = std_ ? 1.f : corr;
        d.zeta[si] = std_ ? 0.f : (3.f * S.mw + S.muw) / (3.f * S.w);
    }
    if (MODE != 0) {
        d.len_eps[si] = L;
        d.neps[si] = S.w * k;
        d.ups[si] = corr;
        d.X[si] = -EVOL_PI_F * L * L * S.mp / (3.f * S.w);
    }
    if (FLOW) {
        // div v = -1/(n C) sum_j (v_i - v_j).grad_i W = 3 S5 / (L Suw), C = Upsilon
        // or Omega* = -Suw/(3 Sw), n = Sw/(pi L^3), grad W = r_ij/r w'(u)/(pi L^4)
        // (the standard scheme takes C = 1: div v = -S5 / (L Sw))
        const float dv = std_ ? -S.dv / (L * S.w) : 3.f * S.dv / (L * S.uw);
        if (MODE != 1) d.divv_h[si] = dv;
        if (MODE != 0) d.divv_e[si] = dv;
        // |curl v| = |1/(n C) sum_j (v_i - v_j) x grad_i W| = 3 |S6| / (L |Suw|)
        if (MODE != 1 && kp.want_curl) {
            const float s6 = sqrtf(S.cx * S.cx + S.cy * S.cy + S.cz * S.cz);
            d.curlv_h[si] = std_ ? s6 / (L * S.w) : 3.f * s6 / (L * fabsf(S.uw));
        }
    }
}

// Cube root of the Newton step's factor: near 1, where it sets the converged length, by the binomial
// series (its first omitted term, 22/729 x^5, is below 1e-9 there); elsewhere, where another step follows,
// by the hardware's base-2 logarithm and exponential.
__device__ __forceinline__ float cube_root(float q)
{
    const float x = q - 1.f;
    const float near1 = fmaf(x, fmaf(x, fmaf(x, fmaf(x, -10.f / 243.f, 5.f / 81.f), -1.f / 9.f), 1.f / 3.f), 1.f);
    return fabsf(x) < 0.03f ? near1 : exp2f(__log2f(q) * (1.f / 3.f));
}

// One Newton step from length L with the sums at L: the next length, and whether it has converged.
// lo, hi: the bracket, tightened by the sign of F.
__device__ __forceinline__ bool newton_step(float eta3, float Sw, float Suw, float &L, float &lo, float &hi)
{
    const float F = Sw * (1.f / EVOL_PI_F) - eta3;
    if (F < 0.f) lo = L;
    if (F > 0.f) hi = L;
    float Ln;
    bool newton = false;
    if (F == 0.f) {
        Ln = L;
    } else {
        // Newton step in y = L^3, on which F = n y - eta^3 depends almost linearly
        // (n varies slowly with L): dF/dy = F'/(3 L^2) with F' = -Suw/(pi L), so
        // y' = y (1 + 3 pi F / Suw); bisection where it leaves the bracket
        const float q = 1.f + __fdividef(3.f * EVOL_PI_F * F, Suw);
        newton = Suw < 0.f && q > 0.f;
        Ln = newton ? L * cube_root(q) : (hi < INFINITY ? 0.5f * (lo + hi) : 2.f * L);
        if (newton && fabsf(Ln - L) <= NEWTON_TOL * L) {
            // converged: a step this small goes towards the root (F' > 0), and one
            // below FP32 resolution leaves L on the bracket's end
            if (Ln < lo || Ln > hi) Ln = L;
        } else {
            // below the root with no upper bracket yet, F' counts only the few
            // neighbours inside the kernel and the step can overshoot by orders of
            // magnitude: grow by at most a factor 2 until the root is bracketed
            if (hi == INFINITY && Ln > 2.f * L) {
                Ln = 2.f * L;
                newton = false;
            }
            if (!(Ln > lo && Ln < hi)) {
                Ln = hi < INFINITY ? 0.5f * (lo + hi) : 2.f * L;
                newton = false;
            }
        }
    }
    const bool conv = fabsf(Ln - L) <= (newton ? NEWTON_TOL : CONV_TOL) * L || (hi < INFINITY && hi - lo <= 1e-7f * hi);
    L = Ln;
    return conv;
}

// Particles per warp when the caller leaves it open (length_group = 0): eight, which share the list pass
// and the staging, less for sets too small to give every resident warp four such groups (1000 and 4096
// particles: one, 0.04 and 0.06 ms against 0.08 and 0.19 with eight; 49,152: two, 0.38 against 0.45).
template <int NW>
__device__ __forceinline__ int group_size(int nlist, int blocks)
{
    int sub = 8;
    while (sub > 1 && nlist < 4 * blocks * NW * sub) sub >>= 1;
    return sub;
}

// The caller's starting length of the particle at sorted position s.
template <int MODE>
__device__ __forceinline__ float start_length(const evol_dev &d, const evol_kparams &kp, int s, int sys)
{
    auto valid = [](float L) { return L > 0.f && L < 1e30f; };
    float L = MODE == 1 ? d.len_eps[s] : d.len_h[s];
    if (MODE == 2 && !valid(L)) L = d.len_eps[s];
    return valid(L) ? L : d.fcube[4 * sys + 3] / cbrtf((float)kp.n);
}

// The particle of list entry e of a length solve: its sorted position and starting length; false where
// there is none to solve.
template <int MODE>
__device__ __forceinline__ bool list_particle(const evol_dev &d, const evol_kparams &kp, int e, int nlist, int &s,
                                              int &sys, float &L0)
{
    s = e >= nlist ? 0 : kp.active ? d.act[e] : (gas_lists<MODE>(kp) ? d.glist[e] : e);
    const bool act = e < nlist && (MODE != 0 || !kp.active || d.orig[s] < kp.n_gas);
    sys = act ? d.sys_sorted[s] : 0;
    L0 = act ? start_length<MODE>(d, kp, s, sys) : 0.f;
    return act;
}

// A starting length far above the spacing of m key-consecutive particles (their box taken as a cube of its
// largest side) would gather, and drop, many times the neighbours needed.
__device__ __forceinline__ bool poor_length(float L0, float eta, float side, int m)
{
    const float est = eta * side / cbrtf((float)m);
    return m >= 8 && est > 0.f && L0 > 2.f * est;
}

// The length that the mean density of the smallest cell around the particle at sorted position s with
// more than a leaf's particles would give: a start for particles whose own is poor (the root does not
// depend on it).  The particle's leaf is node d.base[s + 1] - 1 (see start_node); root: side of the root cube.
template <int MODE>
__device__ __forceinline__ float local_length(const evol_dev &d, const evol_kparams &kp, int s, float eta, float root)
{
    const int leaf = d.base[s + 1] - 1;
    if (leaf >= *d.nnodes) return INFINITY;          // a node list that overflowed (flagged by the build)
    const int up = d.nparent[leaf];
    const int node = up >= 0 ? up : leaf;
    int b = d.nbeg[node], e = d.nend[node];
    if (gas_lists<MODE>(kp)) {
        b = d.gbase[b];
        e = d.gbase[e];
    }
    return e - b >= 4 ? eta * ldexpf(root, -d.nlev[node]) / cbrtf((float)(e - b)) : INFINITY;
}

// Leaf lists of super-groups (LEN_SG consecutive entries of the particle list): one block walks the tree
// once for all of them and lists the leaves within reach of the boxes of its four quarters, so that the
// blocks of k_lengths need no walk of their own.  Before, each block's walk (about ten dependent levels)
// took half of its time.  The radius leaves a tenth for lengths that grow.  Super-groups of several systems
// or with too many leaves get no list (-1).
template <int NW, int MODE, bool PER>
__global__ void __launch_bounds__(32 * NW) k_leaf_lists(const __grid_constant__ evol_dev d,
                                                           const __grid_constant__ evol_kparams kp)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LenSmem<NW, false> &sm = *reinterpret_cast<LenSmem<NW, false> *>(smem_raw);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nlist = kp.active ? d.acts[kp.n] : (gas_lists<MODE>(kp) ? kp.n_gas : kp.n);
    const float eta = MODE == 0 ? kp.eta_h : kp.eta_e;
    const long long pop_cap = 2ll * (long long)*d.nnodes + 64;
    const int sg = blockIdx.x;
    if (sg * LEN_SG >= nlist) return;
    float x0 = INFINITY, y0 = INFINITY, z0 = INFINITY, x1 = -INFINITY, y1 = -INFINITY, z1 = -INFINITY, R = -1.f;
    int ms = 0x7fffffff, xs = -1, first = -1;
#pragma unroll
    for (int q = 0; q < LEN_SG / NW; q += 32) {
        int s, sys;
        float L0;
        const bool act = list_particle<MODE>(d, kp, sg * LEN_SG + w * (LEN_SG / NW) + q + lane, nlist, s, sys, L0);
        const float4 p = act ? d.pos[s] : make_float4(0.f, 0.f, 0.f, 0.f);
        const unsigned m = __ballot_sync(0xffffffffu, act);
        const float ax = warp_min(act ? p.x : INFINITY), bx = warp_max(act ? p.x : -INFINITY);
        const float ay = warp_min(act ? p.y : INFINITY), by = warp_max(act ? p.y : -INFINITY);
        const float az = warp_min(act ? p.z : INFINITY), bz = warp_max(act ? p.z : -INFINITY);
        if (act && poor_length(L0, eta, fmaxf(fmaxf(bx - ax, by - ay), bz - az), __popc(m)))
            L0 = fminf(L0, 1.15f * local_length<MODE>(d, kp, s, eta, d.fcube[4 * sys + 3]));
        R = fmaxf(R, warp_max(act ? 2.f * L0 * SEARCH_MARGIN * 1.1f : -1.f));
        x0 = fminf(x0, ax); y0 = fminf(y0, ay); z0 = fminf(z0, az);
        x1 = fmaxf(x1, bx); y1 = fmaxf(y1, by); z1 = fmaxf(z1, bz);
        ms = min(ms, __reduce_min_sync(0xffffffffu, act ? sys : 0x7fffffff));
        xs = max(xs, __reduce_max_sync(0xffffffffu, act ? sys : -1));
        const int s0 = __shfl_sync(0xffffffffu, s, m ? __ffs(m) - 1 : 0);
        if (first < 0 && m) first = s0;
    }
    if (lane == 0) {
        sm.gc[w] = make_float4(0.5f * (x0 + x1), 0.5f * (y0 + y1), 0.5f * (z0 + z1), R >= 0.f ? R * R : -1.f);
        sm.gh[w] = make_float4(0.5f * (x1 - x0), 0.5f * (y1 - y0), 0.5f * (z1 - z0), 0.f);
        sm.first[w] = first;
        sm.sel[w] = ms;
        sm.nsel[w] = xs;
        d.sg_rad[4 * sg + w] = R;
    }
    __syncthreads();
    const int lo = over_warps(sm.sel, [](int a, int b) { return min(a, b); });
    const int hi = over_warps(sm.nsel, [](int a, int b) { return max(a, b); });
    int nleaf = -1, ncand = -1;
    if (lo == hi) {
        const int root = d.sys_root[lo];
        ncand = block_walk<NW, MODE, PER, false, true>(d, kp, sm, PER ? root : start_node<NW, false>(d, sm, lo, root), pop_cap,
                                                       nleaf);
        if (ncand < 0 || nleaf > SG_LEAVES) nleaf = -1;
        for (int l = threadIdx.x; l < nleaf; l += (32 * NW)) d.sg_acc[(size_t)sg * SG_LEAVES + l] = sm.leaf[l].x;
    }
    if (threadIdx.x == 0) {
        d.sg_info[sg] = make_int2(nleaf, 0);
        atomicAdd(&d.sg_stat[0], (unsigned long long)(nleaf < 0 ? 2 * WIDE_CANDIDATES : ncand));
        atomicAdd(&d.sg_stat[1], 1ull);
    }
}

// Variants: PER periodic axes, FLOW the velocity divergence (and |curl v| on request) in the last
// evaluation; each a template parameter, so that the default solve's code carries none of them.
// Bound by latency: a gather is a chain of shared-memory reads, ballots and counts per chunk, so resident
// warps (24 per SM at 80 registers and 37.5 KB of shared memory a block; FLOW 20) decide, and of the warp
// instructions (1630 per particle of the Plummer sphere, 3050 of halo + gas) the gathers take 35 to 40 %, the
// list passes 18 to 27 %, the staging 9 %, the Newton sweeps 8 %, the last evaluation 6 %.  Against one warp
// per group of particles, each particle gathering from L2 and solved by the whole warp: Plummer 2^20 (32
// neighbours) 3.2 -> 2.4 ms, h of the 1.05 M-particle shock tube 3.3 -> 2.1 ms, eps of a 2^18 periodic box
// whose starting lengths come from the mean density 10.9 -> 1.4 ms, eps and h of 2^21 halo + 2^20 gas
// 16.2 -> 12.9 ms.
template <int NW, int MODE, bool PER, bool FLOW>
__global__ void __launch_bounds__(32 * NW, Shape<NW, FLOW>::MINB) k_lengths(const __grid_constant__ evol_dev d,
                                                                               const __grid_constant__ evol_kparams kp,
                                                                               unsigned long long *queue)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int CC = Shape<NW, FLOW>::CC;
    LenSmem<NW, FLOW> &sm = *reinterpret_cast<LenSmem<NW, FLOW> *>(smem_raw);
    // lists: the shape that the candidate counts ask for does the work, the other returns
    if (!FLOW && !PER && kp.lists && (d.sg_stat[0] > WIDE_CANDIDATES * d.sg_stat[1]) != (NW == 8)) return;
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const int wslot = blockIdx.x * NW + w;
    // the warp's stack: node ids, two per int2 slot of the shared traversal-stack buffer
    int *stk = reinterpret_cast<int *>(d.wstack + (size_t)wslot * kp.stack_stride);
    const int n = kp.n;
    const bool subset = gas_lists<MODE>(kp);
    // items of 4 SUB consecutive entries of the particle list: the active list (individual time steps),
    // the gas list, or every particle
    const int nlist = kp.active ? d.acts[n] : (subset ? kp.n_gas : n);
    const int SUB = kp.lsub > 0 ? kp.lsub : group_size<NW>(nlist, gridDim.x);
    const int nitems = (nlist + NW * SUB - 1) / (NW * SUB);
    const float eta = MODE == 0 ? kp.eta_h : kp.eta_e;
    const float nnei = 32.f / 3.f * EVOL_PI_F * eta * eta * eta;
    const float eta3 = eta * eta * eta;
    const long long pop_cap = 2ll * (long long)*d.nnodes + 64;
    WarpLists &nb = sm.nb[w];
    const int slot = lane >> 3, sl = lane & 7;

    for (;;) {
        if (threadIdx.x == 0) sm.item = (int)atomicAdd(queue, 1ull);
        __syncthreads();
        const int g = sm.item;
        if (g >= nitems) break;
        const int e = (g * NW + w) * SUB + lane;      // lanes 0 .. SUB-1 hold the warp's particles
        int s, sys;
        float L0;
        const bool act = list_particle<MODE>(d, kp, lane < SUB ? e : nlist, nlist, s, sys, L0);
        // Newton iterations [4], gathers from the staged candidates [0], by the particle's own walk [1], list overflows [2],
        // walks whose candidates did not fit [3]
        unsigned *lc = sm.lc[w];
        if (lane < 5) lc[lane] = 0u;
        __syncwarp();
        // the super-group's leaf list (number of leaves; -1: none), if the item lies inside one super-group
        // and each warp inside one of its quarters
        const int e0 = g * NW * SUB, sgi = e0 / LEN_SG;
        const bool inside = kp.lists && LEN_SG / 4 % SUB == 0;
        const int lists = inside ? d.sg_info[sgi].x : -1;
        unsigned pending = __ballot_sync(0xffffffffu, act);
        bool broken = false;
        int rounds = 0, limit = 32;
        unsigned grown = 0u;          // particles whose length has grown beyond an earlier round's radius

        // rounds: the block's pending particles of one system; where their candidates do not fit, the
        // lower half of each warp's, and so on
        for (;;) {
            // the lowest system among the block's pending particles
            int ms = (pending >> lane) & 1u ? sys : 0x7fffffff;
            ms = __reduce_min_sync(0xffffffffu, ms);
            if (lane == 0) sm.sel[w] = ms;
            __syncthreads();
            const int cs = over_warps(sm.sel, [](int a, int b) { return min(a, b); });
            if (cs == 0x7fffffff) break;                     // all done (the same on every thread)
            const int root = d.sys_root[cs];
            const float sd = d.fcube[4 * cs + 3];            // side of the system's root cube
            unsigned rm = __ballot_sync(0xffffffffu, ((pending >> lane) & 1u) && sys == cs);
            // no more of them than fitted before in this item (one or two of a later round do no harm)
            if (__popc(rm) > limit + 2)
                while (__popc(rm) > limit) rm &= ~(1u << (31 - __clz(rm)));
            bool local = false;
            int ncand = 0, nleaf = 0;
            float Rg = 0.f;
            ++rounds;
            for (;;) {
                // the warp's box and largest search radius
                const bool in = (rm >> lane) & 1u;
                const float4 pi4 = in ? d.pos[s] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float x0 = warp_min(in ? pi4.x : INFINITY), x1 = warp_max(in ? pi4.x : -INFINITY);
                const float y0 = warp_min(in ? pi4.y : INFINITY), y1 = warp_max(in ? pi4.y : -INFINITY);
                const float z0 = warp_min(in ? pi4.z : INFINITY), z1 = warp_max(in ? pi4.z : -INFINITY);
                const int m = __popc(rm);
                if (rounds == 1 && in && poor_length(L0, eta, fmaxf(fmaxf(x1 - x0, y1 - y0), z1 - z0), m))
                    L0 = fminf(L0, 1.15f * local_length<MODE>(d, kp, s, eta, sd));
                Rg = warp_max(in ? 2.f * L0 * SEARCH_MARGIN : -1.f);
                const int s0 = __shfl_sync(0xffffffffu, s, rm ? __ffs(rm) - 1 : 0);
                if (lane == 0) {
                    sm.gc[w] = make_float4(0.5f * (x0 + x1), 0.5f * (y0 + y1), 0.5f * (z0 + z1), rm ? Rg * Rg : -1.f);
                    sm.gh[w] = make_float4(0.5f * (x1 - x0), 0.5f * (y1 - y0), 0.5f * (z1 - z0), 0.f);
                    sm.nsel[w] = m;
                    sm.first[w] = rm ? s0 : -1;
                    // does the super-group's list hold every leaf within this radius of this warp's box?
                    sm.listed[w] = lists >= 0 && (!rm || Rg <= d.sg_rad[4 * sgi + (e0 + w * SUB) % LEN_SG / (LEN_SG / 4)]);
                }
                __syncthreads();
                const bool listed = over_warps(sm.listed, [](int a, int b) { return a & b; });
                const int mm = over_warps(sm.nsel, [](int a, int b) { return max(a, b); });
                ncand = listed ? list_leaves<NW, MODE, PER, FLOW>(d, kp, sm, d.sg_acc + (size_t)sgi * SG_LEAVES, lists, nleaf)
                               : block_walk<NW, MODE, PER, FLOW, false>(
                                     d, kp, sm, PER ? root : start_node<NW, FLOW>(d, sm, cs, root), pop_cap, nleaf);
                if (ncand != -1) break;
                if (lane == 0) ++lc[3];
                __syncthreads();
                if (mm <= 1 && local) break;                 // not even for single particles: own walks
                if (mm <= 2 && !local) {
                    // a few particles reach too far: their starting lengths are poor
                    local = true;
                    if (((rm & ~grown) >> lane) & 1u) L0 = fminf(L0, 1.15f * local_length<MODE>(d, kp, s, eta, sd));
                } else {
                    // the lowest of each warp's, as many as should fit
                    limit = max(1, listed ? min(mm - 1, (int)((float)mm * 0.9f * (float)CC / (float)nleaf)) : mm / 2);
                    if (limit > 4) limit &= ~3;              // full batches of four
                    while (__popc(rm) > limit) rm &= ~(1u << (31 - __clz(rm)));
                }
            }
            if (ncand == -2) {
                pending &= ~rm;                              // corrupt tree: nothing to solve on
                __syncthreads();
                continue;
            }
            const bool glist = ncand >= 0;
            if (glist) stage_candidates<NW, MODE, FLOW>(d, kp, sm, nleaf, ncand);
            pending &= ~rm;

            // ---- four particles at a time, eight lanes each, from the staged candidates.  A particle whose
            // radius grows beyond the warp's waits for a later round, which walks for its new length.
            unsigned solo = (!glist || rounds > MAX_ROUNDS || kp.whole) ? rm : 0u;
            unsigned fm = rm & ~solo;
            const float *list = nb.r + slot * SCAP;
            while (fm) {
                int t = -1;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (slot == q) t = __ffs(fm) - 1;
                    fm &= fm - 1u;
                }
                const int tl = max(t, 0);
                const int si = __shfl_sync(0xffffffffu, s, tl);
                const float4 pi4 = d.pos[si];
                const float px = pi4.x, py = pi4.y, pz = pi4.z;
                float L = __shfl_sync(0xffffffffu, L0, tl);
                float lo = 0.f, hi = INFINITY, Rc = 0.f;
                int status = t >= 0 ? ST_ACTIVE : ST_DONE, cnt = 0, iters = 0, shrinks = 0;
                bool stale = true, alone = false, later = false;   // left to the whole warp, to a later round
                for (;;) {
                    if (__any_sync(0xffffffffu, status != ST_DONE && stale)) {
                        // a length that has grown is still served where 2 L leaves a margin below the
                        // warp's radius
                        float Rn = 2.f * L * SEARCH_MARGIN;
                        if (Rn > Rg && 2.02f * L < Rg) Rn = Rg;
                        if (status != ST_DONE && stale && !(Rn <= Rg)) {
                            later = true;
                            status = ST_DONE;
                        }
                        unsigned gm = __ballot_sync(0xffffffffu, status != ST_DONE && stale);
                        while (gm) {
                            const int q = (__ffs(gm) - 1) >> 3;
                            gm &= ~(0xffu << (8 * q));
                            if (lane == 0) ++lc[0];
                            const float R = __shfl_sync(0xffffffffu, Rn, 8 * q);
                            float *gr = nb.r + q * SCAP;
                            unsigned short *gi = nb.id + q * SCAP;
                            __syncwarp();
                            const int c = gather_staged<NW, PER, FLOW>(
                                kp, sm, ncand, lane, __shfl_sync(0xffffffffu, px, 8 * q),
                                __shfl_sync(0xffffffffu, py, 8 * q), __shfl_sync(0xffffffffu, pz, 8 * q), R * R,
                                [&](int k, float r2, int e) {
                                    if (k < SCAP) {
                                        gr[k] = r2;
                                        gi[k] = (unsigned short)e;
                                    }
                                });
                            __syncwarp();
                            const int m = min(c, SCAP);
                            for (int k = lane; k < m; k += 32) gr[k] = sqrtf(gr[k]);
                            // an odd list gets a partner outside every kernel
                            if (lane == 0 && (m & 1)) gr[m] = 4.f * R;
                            if (slot == q) cnt = c;
                        }
                        __syncwarp();
                        if (status != ST_DONE && stale) {
                            Rc = Rn;
                            stale = false;
                            if (cnt > SCAP) {
                                // too many: a length for about the wanted number from their count, else
                                // the longer list of the whole warp
                                const float Ln = 0.5f * Rc * cbrtf(nnei / (float)cnt);
                                if (status == ST_ACTIVE && iters == 0 && ++shrinks <= 4 && Ln < L) {
                                    L = Ln;
                                    stale = true;
                                } else {
                                    alone = true;
                                    status = ST_DONE;
                                }
                            }
                        }
                        if (__any_sync(0xffffffffu, status != ST_DONE && stale)) continue;
                    }
                    if (!__any_sync(0xffffffffu, status == ST_ACTIVE)) break;
                    float Sw, Suw;
                    newton_sums_four(list, status == ST_ACTIVE ? cnt : 0, sl, 1.f / L, Sw, Suw);
                    if (status == ST_ACTIVE) {
                        ++iters;
                        if (newton_step(eta3, Sw, Suw, L, lo, hi)) status = ST_LAST;
                        if (2.f * L >= Rc) stale = true;
                        if (iters >= MAX_ITERS || L > 4.f * sd) {
                            alone = true;
                            status = ST_DONE;
                        }
                    }
                }
                const float Linv = 1.f / L;
                const unsigned short *ids = nb.id + slot * SCAP;
                const Sums S = last_sums<MODE, PER, FLOW, 8>(
                    d, kp, status == ST_LAST ? cnt : 0, sl, Linv, px, py, pz, status == ST_LAST ? si : -1,
                    [&](int e, float &r, float &m, float3 &p, float3 &v) {
                        const int k = ids[e];
                        r = list[e];
                        m = sm.cm[k];
                        if (FLOW) {
                            p = make_float3(sm.cx[k], sm.cy[k], sm.cz[k]);
                            const float4 u = d.vel[sm.cj[k]];
                            v = make_float3(u.x, u.y, u.z);
                        }
                    });
                if (status == ST_LAST && sl == 0) write_result<MODE, FLOW>(d, kp, si, L, Linv, S, false);
                __syncwarp();
                // back in the holder lanes: the particles left over
                unsigned om = __ballot_sync(0xffffffffu, (alone || later) && sl == 0);
                while (om) {
                    const int q = __ffs(om) - 1;
                    om &= om - 1u;
                    const int tq = __shfl_sync(0xffffffffu, t, q);
                    const bool lt = __shfl_sync(0xffffffffu, later ? 1 : 0, q) != 0;
                    const float Lq = __shfl_sync(0xffffffffu, L, q);
                    if (lt) {
                        pending |= 1u << tq;
                        grown |= 1u << tq;
                        if (lane == tq) L0 = Lq;
                    } else {
                        solo |= 1u << tq;
                    }
                }
                const int it = __reduce_add_sync(0xffffffffu, sl == 0 ? iters : 0);
                if (lane == 0) lc[4] += (unsigned)it;
            }

            // ---- one particle at a time by the whole warp, with a list of up to PCAP entries
            while (solo && !broken) {
                const int t = __ffs(solo) - 1;
                solo &= solo - 1u;
                const int si = __shfl_sync(0xffffffffu, s, t);
                const float4 pi4 = d.pos[si];
                const float px = pi4.x, py = pi4.y, pz = pi4.z;
                float L = start_length<MODE>(d, kp, si, cs);
                // every lane holds the same solver state for particle t
                float lo = 0.f, hi = INFINITY, Rc = 0.f;
                // after a neighbour-list overflow at search radius Rlim no length with 2 L >= Rlim can
                // be evaluated: the bracket's upper end is kept below Rlim / 2 and every later gather
                // radius below Rlim
                float Rlim = INFINITY;
                int status = ST_ACTIVE;
                bool stale = true;
                int cnt = 0, iters = 0, walks = 0;
                // a particle whose length cannot be found still gets every output written: its length
                // as reached, NaN for the quantities derived from the (missing) root
                auto give_up = [&](int code) {
                    if (lane == 0) {
                        evol_flag(d.err, code);
                        const float qnan = __int_as_float(0x7fc00000);
                        if (MODE != 1) {
                            d.len_h[si] = L;
                            d.nh[si] = qnan; d.rho[si] = qnan; d.omega[si] = qnan; d.zeta[si] = qnan;
                        }
                        if (MODE != 0) {
                            d.len_eps[si] = L;
                            d.neps[si] = qnan; d.ups[si] = qnan; d.X[si] = qnan;
                        }
                    }
                    status = ST_DONE;
                };
                while (status != ST_DONE) {
                    if (stale) {
                        if (walks >= MAX_WALKS) {
                            give_up(EVOL_ENOCONV);
                            break;
                        }
                        ++walks;
                        // gather radius: 2 L (1 + margin), and strictly between 2 L and Rlim
                        Rc = fminf(2.f * L * SEARCH_MARGIN, L + 0.5f * Rlim);
                        __syncwarp();
                        if (glist && Rc <= Rg) {
                            if (lane == 0) ++lc[0];
                            cnt = gather_staged<NW, PER, FLOW>(kp, sm, ncand, lane, px, py, pz, Rc * Rc,
                                                           [&](int k, float r2, int e) {
                                                               if (k < PCAP)
                                                                   nb.one[k] = make_float2(
                                                                       sqrtf(r2), FLOW ? __int_as_float(sm.cj[e]) : sm.cm[e]);
                                                           });
                        } else {
                            if (lane == 0) ++lc[1];
                            cnt = gather_ball<MODE, PER, FLOW>(d, kp, nb.one, PCAP, lane, stk, pop_cap, root, px, py, pz,
                                                               Rc * Rc);
                        }
                        __syncwarp();
                        if (cnt < 0) {
                            broken = true;
                            break;
                        }
                        stale = false;
                        if (cnt > PCAP) {
                            // more neighbours than the list holds: the radius is too large; shrink, gather again
                            if (lane == 0) ++lc[2];
                            Rlim = fminf(Rlim, Rc);
                            hi = fminf(hi, 0.5f * Rlim * (1.f - 1e-6f));
                            float Ln = 0.75f * L;
                            if (Ln <= lo) Ln = 0.5f * (lo + fminf(L, hi));
                            if (!(Ln > lo && Ln < hi)) {          // nothing left to evaluate
                                give_up(EVOL_EOVERFLOW);
                                break;
                            }
                            L = Ln;
                            stale = true;
                            status = ST_ACTIVE;                    // a converged length is solved again
                            continue;
                        }
                    }
                    if (MODE == 0 && kp.standard && status == ST_ACTIVE) {
                        // standard scheme: widen the ball until it holds N + 1 gas particles, then h
                        // from the N-th and (N+1)-th distances (every particle closer than the
                        // (N+1)-th is in the list: the list holds the whole ball)
                        if (cnt < kp.nstd + 1) {
                            if (Rc > 8.f * sd) {                  // fewer gas particles than N + 1
                                give_up(EVOL_ENOCONV);
                                break;
                            }
                            L = Rc;
                            stale = true;
                            continue;
                        }
                        const float rN = kth_distance(nb.one, cnt, kp.nstd, lane);
                        const float rN1 = kth_distance(nb.one, cnt, kp.nstd + 1, lane);
                        L = 0.25f * (rN + rN1);
                        status = ST_LAST;
                    }
                    const float Linv = 1.f / L;
                    if (status == ST_LAST) {
                        const Sums S = last_sums<MODE, PER, FLOW, 32>(
                            d, kp, cnt, lane, Linv, px, py, pz, si, [&](int e, float &r, float &m, float3 &p, float3 &v) {
                                const float2 l = nb.one[e];
                                r = l.x;
                                m = l.y;
                                if (FLOW) {
                                    const int j = __float_as_int(l.y);
                                    const float4 q = d.pos[j], u = d.vel[j];
                                    m = q.w;
                                    p = make_float3(q.x, q.y, q.z);
                                    v = make_float3(u.x, u.y, u.z);
                                }
                            });
                        if (lane == 0) write_result<MODE, FLOW>(d, kp, si, L, Linv, S, MODE == 0 && kp.standard);
                        status = ST_DONE;
                    } else {
                        float Sw, Suw;
                        newton_sums_one(nb.one, cnt, lane, Linv, Sw, Suw);
                        ++iters;
                        if (newton_step(eta3, Sw, Suw, L, lo, hi)) status = ST_LAST;
                        if (iters >= MAX_ITERS) {
                            if (lane == 0) evol_flag(d.err, EVOL_ENOCONV);
                            status = ST_LAST;
                        }
                        if (2.f * L >= Rc) stale = true;
                        if (L > 4.f * sd)                 // no root: fewer neighbours than required
                            give_up(EVOL_ENOCONV);
                        else if (stale && 2.f * L >= Rlim)   // the next gather would overflow again
                            give_up(EVOL_EOVERFLOW);
                    }
                }
                if (lane == 0) lc[4] += (unsigned)iters;
            }
            __syncthreads();                                 // the next round's walk overwrites the lists
        }
        if (lane == 0) {
            atomicAdd(&d.counters[3], (unsigned long long)lc[4]);
            for (int m = 0; m < 2; ++m) {                   // mode 2 counts for both lengths
                if (MODE != 2 && MODE != 1 - m) continue;
                unsigned long long *c4 = d.counters + 16 + 4 * m;
                for (int q = 0; q < 3; ++q) atomicAdd(c4 + q, (unsigned long long)lc[q]);
                if (w == 0) atomicAdd(c4 + 3, (unsigned long long)lc[3]);
                atomicAdd(&d.counters[24 + m], (unsigned long long)lc[4]);
            }
        }
    }
}

// Gas particles in key order (h solve of a set that is not all gas): flags, then their scan gives each
// sorted position the number of gas particles before it; the scatter writes the list and the positions.
__global__ void k_gas_flags(int n, int n_gas, const int32_t *__restrict__ orig, int32_t *__restrict__ flag)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n) flag[s] = orig[s] < n_gas ? 1 : 0;
}

__global__ void k_gas_scatter(int n, int n_gas, const int32_t *__restrict__ orig, const int32_t *__restrict__ gbase,
                              const float4 *__restrict__ pos, int32_t *__restrict__ glist, float4 *__restrict__ gpos)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n || orig[s] >= n_gas) return;
    const int k = gbase[s];
    glist[k] = s;
    gpos[k] = pos[s];
}

template <int NW, int MODE, bool PER, bool FLOW>
int launch_shape(evol_ctx *c, const evol_kparams &kp, unsigned long long *q)
{
    constexpr int smem = (int)sizeof(LenSmem<NW, FLOW>);
    int blocks = 0;
    if (cudaFuncSetAttribute(k_lengths<NW, MODE, PER, FLOW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_lengths<NW, MODE, PER, FLOW>, 32 * NW, smem) !=
            cudaSuccess)
        return EVOL_ECUDA;
    blocks = blocks < 1 ? 1 : (blocks > 32 / NW ? 32 / NW : blocks);      // stack slots exist for 32 warps per SM
    k_lengths<NW, MODE, PER, FLOW><<<c->num_sms * blocks, 32 * NW, smem, c->stream>>>(c->d, kp, q);
    return evol_cuda_ok(cudaGetLastError());
}

template <int MODE, bool PER, bool FLOW>
int launch_lengths(evol_ctx *c, const evol_kparams &kp, unsigned long long *q)
{
    if (kp.lists) {
        constexpr int smem = (int)sizeof(LenSmem<4, false>);
        if (cudaMemsetAsync(c->d.sg_stat, 0, 2 * sizeof(unsigned long long), c->stream) != cudaSuccess ||
            cudaFuncSetAttribute(k_leaf_lists<4, MODE, PER>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
                cudaSuccess)
            return EVOL_ECUDA;
        k_leaf_lists<4, MODE, PER><<<(kp.n + LEN_SG - 1) / LEN_SG, 128, smem, c->stream>>>(c->d, kp);
        if constexpr (!FLOW && !PER) {
            const int rc = launch_shape<8, MODE, PER, false>(c, kp, q);
            if (rc) return rc;
        }
    }
    return launch_shape<4, MODE, PER, FLOW>(c, kp, q);
}

template <int MODE>
int launch_lengths_mode(evol_ctx *c, const evol_kparams &kp, unsigned long long *q, bool per)
{
    if (per) return kp.want_divv ? launch_lengths<MODE, true, true>(c, kp, q) : launch_lengths<MODE, true, false>(c, kp, q);
    return kp.want_divv ? launch_lengths<MODE, false, true>(c, kp, q) : launch_lengths<MODE, false, false>(c, kp, q);
}

}  // namespace

// Particles per warp that a caller's length_group stands for (0: group_size chooses): a power of two, so that an
// item lies inside one quarter of a super-group and can take its leaf list, and at most eight: more of them
// share a list pass, but their candidates seldom fit a block. eps + h of 2^18 halo + 2^17 gas, ms, with 1, 2,
// 4, 8 and 16 per warp: 3.07, 2.22, 1.85, 1.84, 2.21; eps of 2^18 Plummer particles 1.36, 0.95, 0.76, 0.75,
// 0.87. Between, 4 and 8 change places with the set, so 4 is what the sizes up to 15 get (a run of 131 k gas
// particles 9.83 ms with 4, 9.99 with 8) and 8 is what larger ones ask for.
static inline int warp_particles(int group) { return group >= 16 ? 8 : group >= 4 ? 4 : group == 3 ? 2 : group; }

// Neighbour numbers whose balls (gathered SEARCH_MARGIN wide) mostly leave less than 15 % of a short list free:
// particles then go to the whole warp and its longer list at once instead of overflowing the short one first.
// Lengths near their roots, ms, four at a time / whole warp (one warp for each particle and no candidates in
// shared memory: the form before these): eps of 2^20 Plummer particles inside 4 a, 100 neighbours 4.0 / 4.2
// (4.5), 130 5.7 / 4.8 (5.7), 160 9.9 / 5.4 (7.1), 200 11.0 / 6.8 (9.6); eps and h of 2^18 halo + 2^17 gas, 80
// 2.2 / 2.5 (2.6), 110 3.1 / 2.9 (3.3), 130 3.7 / 3.2 (3.9). From poor starting lengths the line lies higher
// (the halo's 110 4.8 / 6.1, 130 5.9 / 6.7, 160 9.7 / 8.2).
static inline bool whole_warp(float n_nei)
{
    return n_nei * SEARCH_MARGIN * SEARCH_MARGIN * SEARCH_MARGIN > 0.85f * SCAP;
}

int evol_launch_lengths(evol_ctx *c, const evol_particles *p, const evol_params *prm, int mode)
{
    evol_kparams kp{};
    kp.n = (int)p->n;
    kp.n_gas = (int)p->n_gas;
    kp.eta_h = 0.5f * cbrtf(3.f * prm->n_nei_sph / (4.f * EVOL_PI_F));
    kp.eta_e = 0.5f * cbrtf(3.f * prm->n_nei_grav / (4.f * EVOL_PI_F));
    kp.periodic_mask = prm->periodic_mask;
    evol_periodic_axes(kp, prm);
    kp.active = c->bins_active;
    kp.want_curl = mode != 1 && evol_needs_curl(prm);
    kp.standard = mode == 0 && prm->sph_scheme == EVOL_SPH_STANDARD;
    kp.nstd = (int)lrintf(prm->n_nei_sph);
    kp.whole = kp.standard || whole_warp(mode == 0 ? prm->n_nei_sph : prm->n_nei_grav);
    kp.want_divv = c->want_divv || kp.want_curl;
    kp.lsub = warp_particles(prm->length_group);
    kp.lists = (mode == 0 ? kp.n_gas : kp.n) >= LISTS_MIN;
    kp.stack_cap = (int)c->wstack_lim;
    kp.stack_stride = (int)c->wstack_cap;
    if (mode == 0 && p->n_gas < p->n) {
        const int n = kp.n, tb = 256, gb = (n + tb - 1) / tb;
        k_gas_flags<<<gb, tb, 0, c->stream>>>(n, kp.n_gas, c->d.orig, c->d.gbase);
        const int rc = evol_scan_i32(c, n, c->d.gbase, c->d.gbase, 1);
        if (rc) return rc;
        k_gas_scatter<<<gb, tb, 0, c->stream>>>(n, kp.n_gas, c->d.orig, c->d.gbase, c->d.pos, c->d.glist, c->d.gpos);
    }
    unsigned long long *q = c->d.counters + (mode == 1 ? 6 : 5);
    cudaMemsetAsync(q, 0, sizeof(unsigned long long), c->stream);
    const bool per = prm->periodic_mask != 0;
    return mode == 0   ? launch_lengths_mode<0>(c, kp, q, per)
           : mode == 1 ? launch_lengths_mode<1>(c, kp, q, per)
                       : launch_lengths_mode<2>(c, kp, q, per);
}

int evol_lengths_list_cap() { return PCAP; }
