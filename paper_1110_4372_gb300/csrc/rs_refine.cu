// rs_refine.cu -- the phase-space FOF hierarchy (Sec. 3.2, Eq. 1).
//
// Members of every refined group are gathered into member slots in group
// order, with positions unwrapped into one periodic image per group (x - box
// for coordinates in the upper half of the box, exact in float32, when the
// group straddles a face).  Nodes own nested slot ranges: a node's children
// occupy the front of its range.
//
// Size classes:
//  * big nodes (> SMALL_N members): processed level by level by tiles of 256
//    members spread over the whole GPU, with per-node accumulators and
//    histograms in global memory.  At the first levels (rs_tuning::kd_levels)
//    their members are put in k-d order (splits at leaf-aligned medians); each
//    node then has a 32-ary box hierarchy over 32-member leaves, searched a
//    leaf a warp for nearest neighbours and friends together (a query a warp
//    for the samples of its bracket).  Children above SMALL_N stay on the big
//    path, smaller children join the small-node queue;
//  * small nodes (<= SMALL_N members): one CTA loads the node into shared
//    memory and builds its whole subtree there (moments, nearest neighbours,
//    exact k-th select, union-find, children, recursion with an explicit
//    stack), as a persistent work queue; a second instance with 128 threads
//    and MID_N-member shared arrays takes the subtrees of at most MID_N
//    members, and a third with one warp those of at most WARP_N, each
//    forwarded by the one before;
//  * tiny nodes (<= TINY_N = 32 members): one warp holds the node in
//    registers, a member per lane, and builds its whole subtree with warp
//    shuffles and votes, eight subtrees per CTA at a time; the one-warp
//    instance forwards them here.
//
// Exactness: means and dispersions come from exact fixed-point integer sums;
// nearest-neighbour and link tests run in float32 against a band of 2^-20
// (relative, on d^2) around the linking length, and everything inside the
// band is re-evaluated in float64.  The linking length itself is the exact
// float64 k-th smallest nearest-neighbour distance: the float32 k-th value
// brackets it, and only the members whose float32 distance lies within twice
// the band of it are re-evaluated in float64 and ranked.
//
// Optionally (subset size s > 0) a big node of more than s members takes its
// linking length from the nearest-neighbour distances of a random s-member
// subset only (Sec. 3.2, the paper's s = 10,000): the subset is found by a
// radix select on per-particle SplitMix64 keys and searched one warp per
// member; the other members skip the nearest-neighbour search.
#include <cmath>
#include <cstring>

#include <cuda_fp16.h>

#include "rs_refine.cuh"

namespace {

constexpr int SMALL_N = 1024;       // largest node handled by one CTA
constexpr int SMALL_THREADS = 256;
constexpr int MID_N = 256;          // largest node of the middle CTA size
constexpr int MID_THREADS = 128;
constexpr int WARP_N = 128;         // largest node of the one-warp CTAs
constexpr int WARP_CTAS = 24;       // of which this many fit an SM (16 and 20 are 15% slower)
constexpr int TINY_N = 32;          // largest node handled in one warp's registers
constexpr int TINY_WARPS = 8;       // warps per block of the tiny-node kernel
constexpr int TINY_STACK = 32;      // pending nodes per warp
constexpr int TQ = 256;             // big-node tile (members per CTA)

// ---------------------------------------------------------------------------
// setup: unwrap decision per group, gather into slots, root nodes
// ---------------------------------------------------------------------------
__device__ __forceinline__ void load3(const float *a, int stride, int64_t i, float &x, float &y, float &z)
{
    const float *p = a + (int64_t)stride * i;
    x = p[0];
    y = p[1];
    z = p[2];
}

// Per group and axis: shift coordinates in the upper half of the box down by
// box if that makes the group's extent smaller than box/2 (bit a of
// shift[g]); minidx of the group.  One block per group.
// float <-> int with the same order (finite values and infinities)
__device__ __forceinline__ int ord_i(float f)
{
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}

__device__ __forceinline__ float ord_f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// start values of the unwrap decision, and the size table of the subtree kernels
__global__ void k_refine_init(int64_t G, int *gred, int *gmin, int nmax, double f, SizeTab *tab)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 12 * G) gred[i] = 0x7f800000;
    if (i < G) gmin[i] = 0x7fffffff;
    if (i <= nmax) {
        long long kk = (long long)ceil(f * (double)i);
        kk = kk < 1 ? 1 : (kk > i ? i : kk);
        tab[i].inv_n = 1.0 / (double)i;
        tab[i].kk = kk;
    }
}

// group of member slot m (off[g] <= base + m < off[g + 1])
__device__ __forceinline__ int64_t group_of(const int64_t *off, int64_t lo, int64_t hi, int64_t at)
{
    // off[lo] <= at < off[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (off[mid] <= at) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Unwrap decision inputs, one member per thread over all groups: per group
// and axis the minima of x and -x, unshifted and with the upper half of the
// box shifted down by the box, and the smallest particle index.  Lanes of
// one group (groups are contiguous runs of slots) combine before their
// atomics, kept on order-preserving integer images of the floats, and an
// atomic that would change nothing is left out.  The positions go to the
// member slots here, so k_gather gathers the velocities only; the group is
// searched for a warp's first and last slot and, where they differ, between
// (134M path: 6.6 -> 5.0 ms, k_gather 2.2 -> 1.3).
__global__ void k_unwrap_tiles(int64_t G, const int64_t *off, const int32_t *perm, int64_t n, int64_t M,
                               const float *pos, int stride, float boxf, int *slot_group, int *gred, int *gmin,
                               float4 *wpos, int *widx, rs_dev_status *st)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t mw = m & ~31ll;
    if (mw >= M) return;
    const bool ok = m < M;
    const int64_t at0 = off[0];
    int64_t g0 = 0, g1 = 0;
    if (lane_id() == 0) g0 = group_of(off, 0, G, at0 + mw);
    g0 = __shfl_sync(0xffffffffu, g0, 0);
    if (lane_id() == 0) g1 = off[g0 + 1] > at0 + min(mw + 31, M - 1) ? g0 : group_of(off, g0, G, at0 + min(mw + 31, M - 1));
    g1 = __shfl_sync(0xffffffffu, g1, 0);
    int g = -1, i = 0x7fffffff;
    float r[12];
    for (int k = 0; k < 12; k++) r[k] = INFINITY;
    if (ok) {
        g = (int)(g0 == g1 ? g0 : group_of(off, g0, g1 + 1, at0 + m));
        slot_group[m] = g;
        i = perm[at0 + m];
        if (i < 0 || i >= n) {
            dev_fail(st, DEV_BADARG, 33, m);
            i = 0x7fffffff;
            wpos[m] = make_float4(0.f, 0.f, 0.f, 0.f);
            widx[m] = 0;
        } else {
            float c[3];
            load3(pos, stride, i, c[0], c[1], c[2]);
            for (int d = 0; d < 3; d++) {
                const float sft = c[d] >= 0.5f * boxf ? c[d] - boxf : c[d];
                r[d] = c[d];
                r[3 + d] = -c[d];
                r[6 + d] = sft;
                r[9 + d] = -sft;
            }
            wpos[m] = make_float4(c[0], c[1], c[2], 0.f);
            widx[m] = i;
        }
    }
    const unsigned grp = __match_any_sync(0xffffffffu, g);
    const int lead = __ffs(grp) - 1;
    int v[12];
    for (int k = 0; k < 12; k++) v[k] = __reduce_min_sync(grp, ord_i(r[k]));
    const int mi = (int)__reduce_min_sync(grp, (unsigned)i);
    if (ok && lane_id() == lead) {
        for (int k = 0; k < 12; k++)
            if (v[k] < __ldcg(&gred[12 * (int64_t)g + k])) atomicMin(&gred[12 * (int64_t)g + k], v[k]);
        if (mi < __ldcg(&gmin[g])) atomicMin(&gmin[g], mi);
    }
}

// per group: which axes wrap (the group spans less than half the box once
// the upper half is shifted down), or an extent error
__global__ void k_unwrap_bits(int64_t G, const int *gred, float boxf, int *shift_bits, rs_dev_status *st)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    const int *r = gred + 12 * g;
    int bits = 0;
    for (int d = 0; d < 3; d++) {
        const float ext = -ord_f(r[3 + d]) - ord_f(r[d]);
        const float exts = -ord_f(r[9 + d]) - ord_f(r[6 + d]);
        if (ext < 0.5f * boxf) {
        } else if (exts < 0.5f * boxf) {
            bits |= 1 << d;
        } else {
            dev_fail(st, DEV_EXTENT, 30, g);
        }
    }
    shift_bits[g] = bits;
}

// the members' velocities to their slots, and their groups' unwrap
__global__ void k_gather(int64_t M, const float *vel, int stride, float boxf, const int *slot_group,
                         const int *shift_bits, float4 *wpos, float4 *wvel, const int *widx)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int bits = shift_bits[slot_group[m]];
    float u, v, w;
    load3(vel, stride, widx[m], u, v, w);
    wvel[m] = make_float4(u, v, w, 0.f);
    if (!bits) return;
    float4 p = wpos[m];
    if ((bits & 1) && p.x >= 0.5f * boxf) p.x = p.x - boxf;
    if ((bits & 2) && p.y >= 0.5f * boxf) p.y = p.y - boxf;
    if ((bits & 4) && p.z >= 0.5f * boxf) p.z = p.z - boxf;
    wpos[m] = p;
}

__global__ void k_check_offsets(int64_t G, const int64_t *off, rs_dev_status *st)
{
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < G && off[g + 1] < off[g]) dev_fail(st, DEV_BADARG, 34, g);
}

__global__ void k_make_roots(int64_t G, const int64_t *off, const int *gmin, const int *shift_bits, int min_n,
                             NodeArrays nd,
                             int *big_list, int *big_len, int *small_list, int *small_len, rs_dev_status *st)
{
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    int64_t cnt = off[g + 1] - off[g];
    if (cnt < min_n) return;
    if (cnt > ((int64_t)8 << 23)) {  // the per-node hierarchy has at most 24 levels
        dev_fail(st, DEV_OVERFLOW, 35, g);
        return;
    }
    int id = atomicAdd(nd.counter, 1);
    if (id >= nd.cap) {
        dev_fail(st, DEV_OVERFLOW, 31, id);
        return;
    }
    nd.parent[id] = -1;
    nd.level[id] = 0;
    nd.first[id] = (int)(off[g] - off[0]);
    nd.count[id] = (int)cnt;
    nd.minidx[id] = gmin[g];
    nd.nchild[id] = 0;
    nd.tie[id] = 0;
    nd.root[id] = id;
    nd.shift[id] = shift_bits[g];
    if (cnt > SMALL_N) big_list[atomicAdd(big_len, 1)] = id;
    else small_list[atomicAdd(small_len, 1)] = id;
}

// pruning slack of the box bounds, and the margin of clique boxes (both explained
// at the boxes, below)
#define RS_PRUNE_SLACK 1.000003814697265625f  // 1 + 2^-18
#define RS_CLIQUE_MARGIN 0.99999237060546875  // 1 - 2^-17

// linking limits of one node: float32 band edges around l^2 (decided in
// float64 inside them), the reporting band for ties, and the pruning radius
struct LinkLim {
    float lo, hi, tlo, thi, part, lim, cl_lim;
    double l2, l;
};

__device__ __forceinline__ LinkLim link_lim(double l2)
{
    LinkLim r;
    r.l2 = l2;
    r.l = sqrt(l2);
    r.lo = (float)(l2 * (1.0 - RS_BAND));
    r.hi = (float)(l2 * (1.0 + RS_BAND));
    r.tlo = (float)(l2 * (1.0 - 3e-6));
    r.thi = (float)(l2 * (1.0 + 3e-6));
    r.part = fmaxf(r.hi, r.thi);
    r.lim = r.part * RS_PRUNE_SLACK;
    r.cl_lim = (float)(l2 * RS_CLIQUE_MARGIN);
    return r;
}

// the float32 edge of the linking and the tie bands: no pair beyond it matters
__device__ __forceinline__ float link_part(double l2)
{
    return fmaxf((float)(l2 * (1.0 + RS_BAND)), (float)(l2 * (1.0 + 3e-6)));
}

// ---------------------------------------------------------------------------
// half-precision points for the matrix units
// ---------------------------------------------------------------------------
// Pairs are screened by m16n8k8 half-precision products.  With points u of
// six coordinates rounded to half, the product of (-2 u_q, 1, 1) and (u_c,
// hi, lo) -- hi + lo the squared norm of the rounded u_c in two halves -- plus
// |u_q|^2 in the float32 accumulator is |u^_q - u^_c|^2 for 16 x 8 pairs.  The
// rounded points differ from the exact ones by at most
//   delta = 1.02 2^-11 (|u_q| + |u_c|) + 3.1e-4
// in all (half's relative 2^-11, the float32 steps before, and subnormal
// halves even if they counted as zero), so the product's square root is
// within delta of the pair's distance, up to float32 accumulation and lo's
// rounding, below 2^-18 (|u_q| + |u_c|)^2 + 1e-4 on the square.  Screens use
// these bounds one-sidedly: what they drop cannot matter, and what they pass
// is evaluated in full.
__device__ __forceinline__ void mma_m16n8k8_f16(float (&d)[4], unsigned a0, unsigned a1, unsigned b0, float c0,
                                                float c1, float c2, float c3)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%8,%9,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

// the eight halves of a point: six coordinates u = (x - c) w, and the squared
// norm s of the rounded coordinates in two halves
__device__ __forceinline__ uint4 half_point(float4 p, float4 v, float4 pc, float4 vc, float wx, float wv, float &s)
{
    const __half2 h0 = __floats2half2_rn((p.x - pc.x) * wx, (p.y - pc.y) * wx),
                  h1 = __floats2half2_rn((p.z - pc.z) * wx, (v.x - vc.x) * wv),
                  h2 = __floats2half2_rn((v.y - vc.y) * wv, (v.z - vc.z) * wv);
    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1), f2 = __half22float2(h2);
    s = f0.x * f0.x + f0.y * f0.y + f1.x * f1.x + f1.y * f1.y + f2.x * f2.x + f2.y * f2.y;
    const __half hi = __float2half_rn(s);
    const __half2 n = __halves2half2(hi, __float2half_rn(s - __half2float(hi)));
    return make_uint4(*(const unsigned *)&h0, *(const unsigned *)&h1, *(const unsigned *)&h2, *(const unsigned *)&n);
}

constexpr unsigned HALF_ONES = 0x3c003c00u;  // (1, 1)
constexpr unsigned HALF_FAR = 0x00007b00u;   // a squared norm of 57344: near nothing (with zero coordinates)

// word t of a query's operand from word t of its point
__device__ __forceinline__ unsigned half_query(unsigned word, int t)
{
    const __half2 h = __hmul2(*(const __half2 *)&word, __float2half2_rn(-2.f));
    return t < 3 ? *(const unsigned *)&h : HALF_ONES;
}

__device__ __forceinline__ float half_norm(unsigned word3)
{
    const float2 f = __half22float2(*(const __half2 *)&word3);
    return f.x + f.y;
}

// bound on the product's value over pairs at most d apart, a point of norm nq
// against points within d of it
__device__ __forceinline__ float half_bound(float d, float nq)
{
    const float rs = 2.f * nq + d;
    const float e = d + 1.02f * 4.8828125e-4f * rs + 3.1e-4f;
    return e * e * 1.00002f + 3.814697265625e-6f * rs * rs + 1.e-4f;
}

// bound on the distance of a point of norm nq from the one whose product with
// it (without a threshold) is m
__device__ __forceinline__ float half_reach(float m, float nq)
{
    const float s = sqrtf(fmaxf(m, 0.f)), rs = 2.f * nq + s;
    const float d = sqrtf(s * s + 4.2e-6f * rs * rs + 2.e-4f);
    return d + 1.05f * 4.8828125e-4f * (2.f * nq + d) + 3.5e-4f;
}

// ---------------------------------------------------------------------------
// small nodes: whole subtree in one CTA
// ---------------------------------------------------------------------------
template <int NMAX, int NT>
struct SmallShared {
    float4 a[NMAX];   // px, py, pz, vx
    float2 b[NMAX];   // vy, vz
    uint4 half[NMAX]; // the node's points (from 0); later, counts of the child partition
    int idx[NMAX];
    float dnn[NMAX];
    int par[NMAX];    // union-find; before it, the band's members
    int csize[2 * NMAX];  // component sizes, then child numbers; before, the band's values (doubles)
    int pairs[NT / 32][64];
    int2 child[NMAX / 2];  // (smallest particle index, first position) of the children
    // pending nodes: pairwise disjoint and larger than the next tier's limit
    // (at least 10, rs_tuning::tiny_max's least)
    static constexpr int STACK_CAP = NMAX / 10 + 2;
    int4 stack[STACK_CAP];
    MomAcc wacc[NT / 32];
    Metric6 met;
    double l2;
    float4 pc, vc;  // the half frame's centre; .w: weights
    float t32;
    int sp, job, umax, nband, below, tie, nchild, next[2];
};

template <class SS>
__device__ __forceinline__ float4 sp4(const SS &S, int i)
{
    const float4 x = S.a[i];
    return make_float4(x.x, x.y, x.z, 0.f);
}
template <class SS>
__device__ __forceinline__ float4 sv4(const SS &S, int i)
{
    const float2 y = S.b[i];
    return make_float4(S.a[i].w, y.x, y.y, 0.f);
}

// One CTA of NT threads per subtree of at most NMAX members; nodes of at most
// `fwd_limit` members (roots or children) go to the next queue, whose kernel
// runs after this one (members are written back in their final order).
//
// A node's n^2 pair loops run on the matrix units, 16 members (a warp's rows)
// against 8 a product.  Nearest neighbours take two passes: the smallest
// product of each row, then the pairs whose product could be the row's
// nearest given it; those are evaluated in float32.  The friends-of-friends
// pass screens the pairs after each member at the linking length.  Passed
// pairs are queued by the warp and evaluated 32 at a time, so results are
// those of the full loops.  The k-th value is found by bisection on its bits
// in one warp, and the children are placed by a stable count instead of a
// sort, so a node costs about 20 block barriers instead of 130.
//
// Issue-bound in the largest instance, by instruction fetch in the one-warp
// one (its warps run at different places of the code, hence one copy of the
// pair loops for both rounds and little unrolling: 2.05 -> 1.52 ms), and
// earlier by the float64 unit, which executes about 2 lanes a clock: what can
// be is taken from tables, done in float32 with the same rounding, or left to
// k_tree_stats.  The one-warp tier spills 108 bytes at its 80 registers, the
// others about 50.  5.0M members in 29,000 groups of 20-600: nodes above 256
// members 6.9 -> 2.0 ms, 129-256 and 33-128 3.9 -> 2.5 ms (as one 128-thread tier 4.1), up
// to 32 1.08 -> 0.67 ms.
template <int NMAX, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    k_small_subtree(const int *queue, const int *queue_len, int *queue_head, float4 *wpos, float4 *wvel, int *widx,
                    int fwd_limit, int *fwd_q, int *fwd_len, NodeArrays nd, const SizeTab *size_tab, double box,
                    int min_n, rs_dev_status *st)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallShared<NMAX, NT> &S = *reinterpret_cast<SmallShared<NMAX, NT> *>(smem_raw);
    constexpr int NW = NT / 32, PER = NMAX / NT;
    static_assert(NW * 32 * PER == NMAX, "");
    const unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = lane_id(), w = warp_id();
    const unsigned below_me = (1u << lane) - 1u;
    const int g = lane >> 2, t4 = lane & 3;  // the product's row and column group of this lane
    int *cmin = S.csize + NMAX;
    for (;;) {
        if (tid == 0) S.job = atomicAdd(queue_head, 1);
        __syncthreads();
        const int job = S.job;
        __syncthreads();
        if (job >= *queue_len) break;
        const int node0 = queue[job];
        const int base = nd.first[node0];
        const int n0 = nd.count[node0];
        if (n0 <= fwd_limit) {  // a subtree for the next, smaller kernel
            if (tid == 0) fwd_q[atomicAdd(fwd_len, 1)] = node0;
            continue;
        }
        for (int i = tid; i < n0; i += NT) {
            float4 p = wpos[base + i], v = wvel[base + i];
            S.a[i] = make_float4(p.x, p.y, p.z, v.x);
            S.b[i] = make_float2(v.y, v.z);
            S.idx[i] = widx[base + i];
        }
        if (tid == 0) {
            S.sp = 1;
            S.stack[0] = make_int4(0, n0, node0, nd.level[node0]);
        }
        __syncthreads();
        for (int guard = 0; guard < 1 << 20; guard++) {
            if (S.sp == 0) break;
            const int4 top = S.stack[S.sp - 1];
            const int lf = top.x, cnt = top.y, node = top.z, lev = top.w;
            // ---- moments (exact) ----
            {
                const MomRef ref = mom_ref(sp4(S, lf), sv4(S, lf));
                MomAcc a;
                mom_zero(a);
                for (int i = lf + tid; i < lf + cnt; i += NT) mom_add(a, sp4(S, i), sv4(S, i), ref);
                mom_warp_reduce(a);
                if (lane == 0) S.wacc[w] = a;
                __syncthreads();
                if (w == 0) {
                    const float4 pr = sp4(S, lf), vr = sv4(S, lf);
                    const MomOutWarp o = mom_finalize_warp(S.wacc, NW, pr, vr, size_tab[cnt].inv_n, box);
                    if (lane < 3) {
                        nd.xbar[3 * node + lane] = o.xbar;
                        nd.vbar[3 * node + lane] = o.vbar;
                    }
                    const Metric6 m = metric_of_warp(o.sigx, o.sigv);
                    if (lane == 0) {
                        nd.sigx[node] = o.sigx;
                        nd.sigv[node] = o.sigv;
                        S.met = m;
                        const float fx = (float)o.sigx, fv = (float)o.sigv;
                        // half frame: units of a quarter dispersion about the mean, so
                        // |u| <= 4 sqrt(2 n) = 181 and subnormal halves stay far below
                        // the distances
                        S.pc = make_float4(o.cx[0], o.cx[1], o.cx[2], fx > 0.f ? 4.f / fx : 0.f);
                        S.vc = make_float4(o.cx[3], o.cx[4], o.cx[5], fv > 0.f ? 4.f / fv : 0.f);
                        S.umax = 0;
                        S.nband = 0;
                        S.below = 0;
                        S.tie = 0;
                        S.nchild = 0;
                        S.next[0] = S.next[1] = 0;
                        S.sp--;
                    }
                }
                __syncthreads();
            }
            const Metric6 met = S.met;
            const int nblk = (cnt + 7) >> 3, ntile = (cnt + 15) >> 4;
            {
                float um = 0.f;
                const float4 pc = S.pc, vc = S.vc;
                for (int i = tid; i < 8 * nblk; i += NT) {
                    uint4 h = make_uint4(0u, 0u, 0u, HALF_FAR);
                    if (i < cnt) {
                        float s;
                        h = half_point(sp4(S, lf + i), sv4(S, lf + i), pc, vc, pc.w, vc.w, s);
                        if (!(s < 5e4f)) {  // outside half's range: every pair will be evaluated
                            s = INFINITY;
                            h = make_uint4(0u, 0u, 0u, 0u);
                        }
                        um = fmaxf(um, s);
                        S.dnn[lf + i] = INFINITY;
                    }
                    S.half[i] = h;
                }
                um = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(um)));
                if (lane == 0) atomicMax(&S.umax, __float_as_int(um));
            }
            __syncthreads();
            const bool in_range = __int_as_float(S.umax) < 5e4f;
            const unsigned *hw = reinterpret_cast<const unsigned *>(S.half);
            int *queue_w = S.pairs[w];
            double l2 = 0.0;
            float lo = 0.f, part = 0.f, lu = 0.f;
            bool screen = in_range;
            int tie = 0;
            // Two rounds over the tiles: nearest neighbours, then (after the
            // linking length) friends.  One copy of the code for both: the
            // one-warp CTAs run at different places of it, and what they wait
            // for most is the instruction cache.
#pragma unroll 1
            for (int round = 0; round < 2; round++) {
                if (round == 1) {
                    __syncthreads();
                    // ---- k-th smallest, float32: bisection on the bits, in one warp ----
                    const int kk = (int)size_tab[cnt].kk;
                    if (w == 0) {
                        unsigned v[NMAX / 32];
                        unsigned x0 = 0xffffffffu, x1 = 0u;
#pragma unroll
                        for (int r = 0; r < NMAX / 32; r++) {
                            const int i = 32 * r + lane;
                            v[r] = i < cnt ? __float_as_uint(S.dnn[lf + i]) : 0xffffffffu;
                            x0 = min(x0, v[r]);
                            if (i < cnt) x1 = max(x1, v[r]);
                        }
                        x0 = __reduce_min_sync(FULL, x0);
                        x1 = __reduce_max_sync(FULL, x1);
                        while (x0 < x1) {  // the smallest x with kk values at most x
                            const unsigned mid = x0 + ((x1 - x0) >> 1);
                            int c = 0;
#pragma unroll
                            for (int r = 0; r < NMAX / 32; r++) c += v[r] <= mid ? 1 : 0;
                            if (__reduce_add_sync(FULL, (unsigned)c) >= (unsigned)kk) x1 = mid;
                            else x0 = mid + 1u;
                        }
                        if (lane == 0) S.t32 = __uint_as_float(x0);
                    }
                    __syncthreads();
                    const float t32 = S.t32;
                    // t32 (1 -+ 2 RS_BAND), rounded once: 2 RS_BAND = 2^-19
                    const float blo = fmaf(t32, (float)(-2.0 * RS_BAND), t32),
                                bhi = fmaf(t32, (float)(2.0 * RS_BAND), t32);
                    // ---- band members: exact float64 nearest-neighbour distances ----
                    // (the whole block over the candidates of one band member after another)
                    unsigned long long *bval = reinterpret_cast<unsigned long long *>(S.csize);
                    int *blist = S.par;
                    for (int i = tid; i < 32 * ((cnt + 31) / 32); i += NT) {
                        const float dq = i < cnt ? S.dnn[lf + i] : INFINITY;
                        const unsigned bm = __ballot_sync(FULL, dq < blo);
                        if (lane == 0 && bm) atomicAdd(&S.below, __popc(bm));
                        if (i < cnt && dq >= blo && dq <= bhi) {
                            const int b = atomicAdd(&S.nband, 1);
                            blist[b] = lf + i;
                            bval[b] = 0x7ff0000000000000ull;  // +infinity
                        }
                    }
                    __syncthreads();
                    const int nb = S.nband;
                    for (int b = 0; b < nb; b++) {
                        const int q = blist[b];
                        const float4 pq = sp4(S, q), vq = sv4(S, q);
                        const float lim = S.dnn[q] * (float)(1.0 + 2.0 * RS_BAND);
#pragma unroll 1
                        for (int c = lf + tid; c < lf + cnt; c += NT) {
                            if (c == q) continue;
                            const float4 pc = sp4(S, c), vc = sv4(S, c);
                            if (d2_32(pq, vq, pc, vc, met) <= lim)
                                atomicMin(&bval[b],
                                          (unsigned long long)__double_as_longlong(d2_64(pq, vq, pc, vc, met)));
                        }
                    }
                    __syncthreads();
                    // rank the band: the exact k-th value is the (k - 1 - below)-th
                    const int want = kk - 1 - S.below;
                    if ((want < 0 || want >= nb) && tid == 0) dev_fail(st, DEV_INTERNAL, 40, node);
                    for (int b = tid; b < nb; b += NT) {
                        int r = 0;
                        const unsigned long long vb = bval[b];
                        for (int c = 0; c < nb; c++) r += (bval[c] < vb || (bval[c] == vb && c < b)) ? 1 : 0;
                        if (r == want) {
                            S.l2 = __longlong_as_double((long long)vb);
                            nd.lnk[node] = S.l2;  // k_tree_stats makes it a length
                        }
                    }
                    __syncthreads();
                    l2 = S.l2;
                    for (int i = lf + tid; i < lf + cnt; i += NT) {
                        S.par[i] = i;
                        S.csize[i] = 0;
                        cmin[i] = 0x7fffffff;
                    }
                    __syncthreads();
                    lo = fminf((float)(l2 * (1.0 - RS_BAND)), (float)(l2 * (1.0 - 3e-6)));
                    part = link_part(l2);
                    // the linking length in the half frame's units (a metric
                    // whose scale float32 cannot hold screens nothing)
                    const float sc = (float)met.scale;
                    lu = 4.f * sqrtf(part / sc) * 1.000001f;
                    screen = in_range && lu < 1e4f && sc > 1e-30f && part > 1e-30f;
                }
                int np = 0;
                auto flush = [&](int k) {
                    np -= k;
                    const int code = lane < k ? queue_w[np + lane] : 0, q = lf + (code >> 10), c = lf + (code & 1023);
                    if (q != c) {
                        const float4 pq = sp4(S, q), vq = sv4(S, q), pc = sp4(S, c), vc = sv4(S, c);
                        const float d2 = d2_32(pq, vq, pc, vc, met);
                        if (round == 0) {
                            atomicMin(reinterpret_cast<int *>(&S.dnn[q]), __float_as_int(d2));
                        } else if (d2 <= part) {
                            // below both bands: a friend, and not a tie-band pair
                            bool link = d2 < lo;
                            if (!link) {
                                const double e = d2_64(pq, vq, pc, vc, met), l = sqrt(l2);
                                link = e <= l2;
                                if (l2 > 0 && e != l2 && fabs(sqrt(e) - l) <= 1e-6 * l) tie++;
                            }
                            if (link) uf_union_s(S.par, q, c, st);
                        }
                    }
                    __syncwarp();
                };
                for (;;) {
                    int tl = 0;
                    if (lane == 0) tl = atomicAdd(&S.next[round], 1);
                    tl = __shfl_sync(FULL, tl, 0);
                    if (tl >= ntile) break;
                    const int r0 = 16 * tl + g, r1 = r0 + 8;  // this lane's two rows
                    const int q0 = min(r0, cnt - 1), q1 = min(r1, cnt - 1);
                    const unsigned a0 = half_query(hw[4 * q0 + t4], t4), a1 = half_query(hw[4 * q1 + t4], t4);
                    const float s0 = half_norm(hw[4 * q0 + 3]), s1 = half_norm(hw[4 * q1 + 3]);
                    bool k0 = r0 < cnt, k1 = r1 < cnt;
                    float d0 = lu, d1 = lu;
                    if (round == 0) {
                        // the smallest product of each row: the nearest is at
                        // most sqrt(m) + delta away, so its own product is at
                        // most the bound for that distance
                        float m0 = INFINITY, m1 = INFINITY;
#pragma unroll 2
                        for (int j = 0; j < nblk; j++) {
                            float d[4];
                            mma_m16n8k8_f16(d, a0, a1, hw[4 * (8 * j + g) + t4], s0, s0, s1, s1);
                            if ((j >> 1) == tl) {  // not itself
                                const int c = 8 * j + 2 * t4;
                                if (c == r0) d[0] = INFINITY;
                                if (c + 1 == r0) d[1] = INFINITY;
                                if (c == r1) d[2] = INFINITY;
                                if (c + 1 == r1) d[3] = INFINITY;
                            }
                            m0 = fminf(m0, fminf(d[0], d[1]));
                            m1 = fminf(m1, fminf(d[2], d[3]));
                        }
#pragma unroll
                        for (int o = 1; o < 4; o <<= 1) {
                            m0 = fminf(m0, __shfl_xor_sync(FULL, m0, o));
                            m1 = fminf(m1, __shfl_xor_sync(FULL, m1, o));
                        }
                        d0 = half_reach(m0, sqrtf(s0));
                        d1 = half_reach(m1, sqrtf(s1));
                    } else {
                        k0 = k0 && S.dnn[lf + q0] <= part;
                        k1 = k1 && S.dnn[lf + q1] <= part;
                        if (!__any_sync(FULL, k0 || k1)) continue;
                    }
                    const float c0 = !k0 ? 60000.f : (screen ? s0 - half_bound(d0, sqrtf(s0)) : -INFINITY);
                    const float c1 = !k1 ? 60000.f : (screen ? s1 - half_bound(d1, sqrtf(s1)) : -INFINITY);
                    for (int jb = round == 0 ? 0 : 2 * tl; jb < nblk; jb += 8) {
                        // the signs of eight blocks' products, oldest at the top
                        unsigned mask = 0;
                        const int je = min(8, nblk - jb);
#pragma unroll 2
                        for (int j = 0; j < je; j++) {
                            float d[4];
                            mma_m16n8k8_f16(d, a0, a1, hw[4 * (8 * (jb + j) + g) + t4], c0, c0, c1, c1);
#pragma unroll
                            for (int i = 0; i < 4; i++) mask = __funnelshift_l(__float_as_uint(d[i]), mask, 1);
                        }
                        mask <<= 32 - 4 * je;
                        while (__any_sync(FULL, mask != 0)) {
                            bool push = false;
                            int q = 0, c = 0;
                            if (mask) {
                                const int e = __clz(mask);
                                mask &= ~(0x80000000u >> e);
                                q = (e & 2) ? r1 : r0;
                                c = 8 * (jb + (e >> 2)) + 2 * t4 + (e & 1);
                                push = c < cnt && (round == 0 ? c != q : c > q);
                            }
                            const unsigned bm = __ballot_sync(FULL, push);
                            if (push) queue_w[np + __popc(bm & below_me)] = (q << 10) | c;
                            np += __popc(bm);
                            __syncwarp();
                            // evaluate when full, and what is left at the end
                            if (np >= 32) flush(32);
                        }
                    }
                }
                if (np > 0) flush(np);
            }
            tie = warp_sum(tie);
            if (lane == 0 && tie) atomicAdd(&S.tie, tie);
            __syncthreads();
            // ---- components (lanes of one component add once) ----
            // each warp takes a run of the members, PER a lane
            const int run = 32 * ((cnt + 32 * NW - 1) / (32 * NW)), i0 = w * run;
#pragma unroll
            for (int r = 0; r < PER; r++) {
                const int i = i0 + 32 * r + lane;
                const bool ok = 32 * r < run && i < cnt;
                const int root = ok ? uf_find_s(S.par, lf + i) : -1;
                const unsigned peers = __match_any_sync(FULL, root);
                const int mi = (int)__reduce_min_sync(peers, ok ? (unsigned)S.idx[lf + i] : 0x7fffffffu);
                if (ok && (peers & below_me) == 0) {
                    atomicAdd(&S.csize[root], __popc(peers));
                    atomicMin(&cmin[root], mi);
                }
            }
            __syncthreads();
            // ---- children, numbered as found; the others are the rest ----
            for (int i = lf + tid; i < lf + cnt; i += NT) {
                if (S.par[i] != i) continue;
                const int sz = S.csize[i];
                if (sz >= min_n && sz < cnt) {
                    const int c = atomicAdd(&S.nchild, 1);
                    S.child[c] = make_int2(cmin[i], sz);
                    cmin[i] = c;
                } else {
                    cmin[i] = -1;
                }
            }
            __syncthreads();
            const int nc = S.nchild;
            if (nc > 0) {
                // their places (by smallest particle index, the rest after
                // them) and their nodes
                unsigned short *wc = reinterpret_cast<unsigned short *>(S.half);  // [NW][nc + 1]
                for (int i = tid; i < NW * (nc + 1); i += NT) wc[i] = 0;
                int *place = reinterpret_cast<int *>(wc + NW * (nc + 1) + ((NW * (nc + 1)) & 1));
                for (int c = tid; c <= nc; c += NT) {
                    const int2 me = c < nc ? S.child[c] : make_int2(0x7fffffff, 0);
                    int at = 0;
                    for (int o = 0; o < nc; o++) {
                        const int2 ch = S.child[o];
                        at += ch.x < me.x ? ch.y : 0;
                    }
                    place[c] = at;
                    if (c == nc) continue;
                    const int id = atomicAdd(nd.counter, 1);
                    if (id >= nd.cap) {
                        dev_fail(st, DEV_OVERFLOW, 41, id);
                        continue;
                    }
                    nd.parent[id] = node;
                    nd.level[id] = lev + 1;
                    nd.first[id] = base + lf + at;
                    nd.count[id] = me.y;
                    nd.minidx[id] = me.x;
                    nd.nchild[id] = 0;
                    nd.tie[id] = 0;
                    nd.root[id] = nd.root[node];
                    nd.shift[id] = nd.shift[node];
                    if (me.y <= fwd_limit) {  // its subtree goes to the next, smaller kernel
                        fwd_q[atomicAdd(fwd_len, 1)] = id;
                        continue;
                    }
                    const int s = atomicAdd(&S.sp, 1);
                    if (s >= SmallShared<NMAX, NT>::STACK_CAP) {
                        dev_fail(st, DEV_OVERFLOW, 42, s);
                        atomicSub(&S.sp, 1);
                    } else {
                        S.stack[s] = make_int4(lf + at, me.y, id, lev + 1);
                    }
                }
                __syncthreads();
                // stable places: the members of one child before this one, in
                // its warp's run and in the runs of the warps before
                int grp[PER], rank[PER];
#pragma unroll
                for (int r = 0; r < PER; r++) {
                    const int i = i0 + 32 * r + lane;
                    const bool ok = 32 * r < run && i < cnt;
                    int c = ok ? cmin[uf_find_s(S.par, lf + i)] : -2;
                    if (c == -1) c = nc;
                    const unsigned peers = __match_any_sync(FULL, c);
                    const unsigned before = ok ? wc[w * (nc + 1) + c] : 0u;
                    __syncwarp();
                    if (ok && (peers & below_me) == 0) wc[w * (nc + 1) + c] = (unsigned short)(before + __popc(peers));
                    __syncwarp();
                    grp[r] = c;
                    rank[r] = (int)before + __popc(peers & below_me);
                }
                __syncthreads();
                for (int c = tid; c <= nc; c += NT) {
                    unsigned tot = 0;
                    for (int u = 0; u < NW; u++) {
                        const unsigned x = wc[u * (nc + 1) + c];
                        wc[u * (nc + 1) + c] = (unsigned short)tot;
                        tot += x;
                    }
                }
                float4 ra[PER];
                float2 rb[PER];
                int ri[PER];
#pragma unroll
                for (int r = 0; r < PER; r++) {
                    const int i = i0 + 32 * r + lane;
                    if (32 * r < run && i < cnt) {
                        ra[r] = S.a[lf + i];
                        rb[r] = S.b[lf + i];
                        ri[r] = S.idx[lf + i];
                    }
                }
                __syncthreads();
#pragma unroll
                for (int r = 0; r < PER; r++) {
                    const int i = i0 + 32 * r + lane;
                    if (32 * r < run && i < cnt) {
                        const int to = lf + place[grp[r]] + wc[w * (nc + 1) + grp[r]] + rank[r];
                        S.a[to] = ra[r];
                        S.b[to] = rb[r];
                        S.idx[to] = ri[r];
                    }
                }
            }
            if (tid == 0) {
                nd.nchild[node] = nc;
                nd.tie[node] = S.tie;
            }
            __syncthreads();
        }
        // members in their final order (the tiny-node kernel reads its nodes here)
        for (int i = tid; i < n0; i += NT) {
            const float4 x = S.a[i];
            const float2 y = S.b[i];
            widx[base + i] = S.idx[i];
            wpos[base + i] = make_float4(x.x, x.y, x.z, 0.f);
            wvel[base + i] = make_float4(x.w, y.x, y.y, 0.f);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// tiny nodes: whole subtree in one warp
// ---------------------------------------------------------------------------
__device__ __forceinline__ float4 shfl_xyz(float4 a, int src)
{
    return make_float4(__shfl_sync(0xffffffffu, a.x, src), __shfl_sync(0xffffffffu, a.y, src),
                       __shfl_sync(0xffffffffu, a.z, src), 0.f);
}

// ascending bitonic sort of one 64-bit key per lane across the warp
__device__ __forceinline__ unsigned long long warp_sort_u64(unsigned long long key)
{
    const int lane = lane_id();
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, key, j);
            const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
            key = keep_min ? (o < key ? o : key) : (o > key ? o : key);
        }
    return key;
}

// One warp per tiny subtree: lane i holds member i of the subtree root's slot
// range, and a node is a contiguous range of lanes.  The steps and their
// arithmetic are those of the one-CTA path: exact moments, float32 nearest
// neighbours, the float32 k-th value and the float64 band around it, the
// float64 k-th value, friends-of-friends with the float64 recheck in the band,
// then children first by smallest particle index and the rest after them.
__global__ void __launch_bounds__(TINY_WARPS * 32)
    k_tiny_subtree(const int *queue, const int *queue_len, int *queue_head, const float4 *wpos, const float4 *wvel,
                   int *widx, NodeArrays nd, const SizeTab *size_tab, double box, int min_n, rs_dev_status *st)
{
    __shared__ MomAcc acc_s[TINY_WARPS];
    __shared__ int par_s[TINY_WARPS][32];
    __shared__ int csz_s[TINY_WARPS][32];
    __shared__ int cmin_s[TINY_WARPS][32];
    __shared__ int4 stk_s[TINY_WARPS][TINY_STACK];
    const unsigned FULL = 0xffffffffu;
    const int w = warp_id(), lane = lane_id();
    int *par = par_s[w], *csz = csz_s[w], *cmn = cmin_s[w];
    int4 *stk = stk_s[w];
    const int qlen = *queue_len;
    for (int guard = 0; guard < (1 << 30); guard++) {
        int job = 0;
        if (lane == 0) job = atomicAdd(queue_head, 1);
        job = __shfl_sync(FULL, job, 0);
        if (job >= qlen) break;
        const int node0 = queue[job];
        const int base = nd.first[node0], n0 = nd.count[node0];
        if (n0 > TINY_N) {
            if (lane == 0) dev_fail(st, DEV_INTERNAL, 44, node0);
            continue;
        }
        float4 p = make_float4(0, 0, 0, 0), v = p;
        int idx = 0x7fffffff;
        if (lane < n0) {
            p = wpos[base + lane];
            v = wvel[base + lane];
            idx = widx[base + lane];
        }
        if (lane == 0) stk[0] = make_int4(0, n0, node0, nd.level[node0]);
        int sp = 1;
        __syncwarp();
        for (int it = 0; sp > 0 && it < 4096; it++) {
            const int4 top = stk[--sp];
            __syncwarp();
            const int off = top.x, cnt = top.y, node = top.z, lev = top.w;
            const bool mine = lane >= off && lane < off + cnt;
            // ---- moments (exact), the node's first member as reference ----
            const float4 pr = shfl_xyz(p, off), vr = shfl_xyz(v, off);
            MomAcc a;
            mom_zero(a);
            if (mine) mom_add(a, p, v, mom_ref(pr, vr));
            mom_warp_reduce(a);
            if (lane == 0) acc_s[w] = a;
            __syncwarp();
            const MomOutWarp o = mom_finalize_warp(&acc_s[w], 1, pr, vr, size_tab[cnt].inv_n, box);
            __syncwarp();
            if (lane < 3) {
                nd.xbar[3 * node + lane] = o.xbar;
                nd.vbar[3 * node + lane] = o.vbar;
            }
            if (lane == 0) {
                nd.sigx[node] = o.sigx;
                nd.sigv[node] = o.sigv;
            }
            const Metric6 met = metric_of_warp(o.sigx, o.sigv);
            // ---- nearest neighbours (float32) ----
            float dnn = INFINITY;
            for (int c = off; c < off + cnt; c++) {
                const float4 pc = shfl_xyz(p, c), vc = shfl_xyz(v, c);
                if (mine && c != lane) dnn = fminf(dnn, d2_32(p, v, pc, vc, met));
            }
            // ---- k-th smallest, float32: the member of rank k - 1 by (value, lane) ----
            const int kk = (int)size_tab[cnt].kk;
            int rank = 0;
            for (int c = off; c < off + cnt; c++) {
                const float dc = __shfl_sync(FULL, dnn, c);
                if (mine && (dc < dnn || (dc == dnn && c < lane))) rank++;
            }
            const unsigned pick = __ballot_sync(FULL, mine && rank == kk - 1);
            const float t32 = __shfl_sync(FULL, dnn, pick ? __ffs(pick) - 1 : off);
            const float blo = fmaf(t32, (float)(-2.0 * RS_BAND), t32), bhi = fmaf(t32, (float)(2.0 * RS_BAND), t32);
            // ---- band members: exact float64 nearest-neighbour distances ----
            const bool inband = mine && dnn >= blo && dnn <= bhi;
            const int below = __popc(__ballot_sync(FULL, mine && dnn < blo));
            double ex = INFINITY;
            if (__any_sync(FULL, inband)) {
                const float lim = dnn * (float)(1.0 + 2.0 * RS_BAND);
                for (int c = off; c < off + cnt; c++) {
                    const float4 pc = shfl_xyz(p, c), vc = shfl_xyz(v, c);
                    if (inband && c != lane && d2_32(p, v, pc, vc, met) <= lim) ex = fmin(ex, d2_64(p, v, pc, vc, met));
                }
            }
            // the exact k-th value is the (k - 1 - below)-th smallest band value
            const int want = (int)(kk - 1) - below;
            const unsigned bmask = __ballot_sync(FULL, inband);
            // (non-negative doubles order as their bits; the float64 unit is
            // what this kernel waits for most)
            const long long eb = __double_as_longlong(ex);
            int brank = 0;
            for (unsigned m = bmask; m; m &= m - 1u) {
                const int c = __ffs(m) - 1;
                const long long ec = __shfl_sync(FULL, eb, c);
                if (inband && (ec < eb || (ec == eb && c < lane))) brank++;
            }
            const unsigned bp = __ballot_sync(FULL, inband && brank == want);
            if (!bp && lane == 0) dev_fail(st, DEV_INTERNAL, 45, node);
            const double l2 = bp ? __shfl_sync(FULL, ex, __ffs(bp) - 1) : 0.0;
            if (lane == 0) nd.lnk[node] = l2;  // k_tree_stats makes it a length
            // ---- friends-of-friends at l (inclusive) ----
            const float lo = fminf((float)(l2 * (1.0 - RS_BAND)), (float)(l2 * (1.0 - 3e-6)));
            const float part = link_part(l2);
            par[lane] = lane;
            __syncwarp();
            int tie = 0;
            const bool act = mine && dnn <= part;
            for (int c = off; c < off + cnt; c++) {
                const float dc = __shfl_sync(FULL, dnn, c);
                const float4 pc = shfl_xyz(p, c), vc = shfl_xyz(v, c);
                if (!act || c <= lane || dc > part) continue;
                const float d2 = d2_32(p, v, pc, vc, met);
                if (d2 > part) continue;
                // below both bands: a friend, and not a tie-band pair
                bool link = d2 < lo;
                if (!link) {
                    const double e = d2_64(p, v, pc, vc, met), l = sqrt(l2);
                    link = e <= l2;
                    if (l2 > 0 && e != l2 && fabs(sqrt(e) - l) <= 1e-6 * l) tie++;
                }
                if (link) uf_union_s(par, lane, c, st);
            }
            tie = warp_sum(tie);
            __syncwarp();
            // ---- components ----
            csz[lane] = 0;
            cmn[lane] = 0x7fffffff;
            __syncwarp();
            int r = lane;
            if (mine) {
                r = uf_find_s(par, lane);
                atomicAdd(&csz[r], 1);
                atomicMin(&cmn[r], idx);
            }
            __syncwarp();
            // ---- children first (by smallest particle index), then the rest ----
            unsigned hiw = 0xffffffffu;
            if (mine) {
                const int sz = csz[r];
                if (sz >= min_n && sz < cnt) hiw = (unsigned)cmn[r];
            }
            const unsigned long long key =
                warp_sort_u64(mine ? (((unsigned long long)hiw << 32) | (unsigned)(lane - off)) : ~0ull);
            // the lane at position q of the node takes the member whose key sorted to q
            const unsigned long long kq = __shfl_sync(FULL, key, mine ? lane - off : lane);
            const int from = mine ? off + (int)(kq & 0xffffffffu) : lane;
            p = shfl_xyz(p, from);
            v = shfl_xyz(v, from);
            idx = __shfl_sync(FULL, idx, from);
            const unsigned khi = mine ? (unsigned)(kq >> 32) : 0xfffffffeu;
            // ---- emit the children ----
            const unsigned same = __match_any_sync(FULL, khi);
            const bool start = mine && khi != 0xffffffffu && (__ffs(same) - 1) == lane;
            const unsigned starts = __ballot_sync(FULL, start);
            const int nch = __popc(starts);
            if (sp + nch > TINY_STACK) {
                if (lane == 0) dev_fail(st, DEV_OVERFLOW, 46, node);
                break;
            }
            int id = -1;
            if (start) {
                id = atomicAdd(nd.counter, 1);
                if (id >= nd.cap) {  // the host retries with a larger capacity
                    dev_fail(st, DEV_OVERFLOW, 47, id);
                    id = -1;
                } else {
                    nd.parent[id] = node;
                    nd.level[id] = lev + 1;
                    nd.first[id] = base + lane;
                    nd.count[id] = __popc(same);
                    nd.minidx[id] = (int)khi;
                    nd.nchild[id] = 0;
                    nd.tie[id] = 0;
                    nd.root[id] = nd.root[node];
                    nd.shift[id] = nd.shift[node];
                }
            }
            const unsigned pushed = __ballot_sync(FULL, id >= 0);
            if (id >= 0) stk[sp + __popc(pushed & ((1u << lane) - 1u))] = make_int4(lane, __popc(same), id, lev + 1);
            sp += __popc(pushed);
            if (lane == 0) {
                nd.nchild[node] = __popc(pushed);
                nd.tie[node] = tie;
            }
            __syncwarp();
        }
        if (lane < n0) widx[base + lane] = idx;
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// big nodes: one level at a time
// ---------------------------------------------------------------------------
struct LevelBufs {
    const int *list;  // node ids, by rank
    int K;
    const int *tile_rank;
    const int *tile_q0;
    const int64_t *seg_off;  // member offset of each rank in the level's member list
    MomAcc *acc;
    Metric6 *met;
    float4 *ref;             // reference pos, vel per rank (2 entries)
    unsigned *hist;          // 2048 per rank
    unsigned *sel_prefix;    // per rank
    int *sel_krem;           // per rank
    int *below;              // per rank
    int *band_len;           // scalar
    int *band_rank;
    int *band_slot;
    double *band_val;
    double *l2;              // per rank
    int *tie;                // per rank
    unsigned *sub_t;         // per rank: subset key threshold, high and low words (2 entries)
    int *sub_cnt;            // per rank: members drawn into the subset
    float2 *lim;             // per rank: below it a friend in float32, beyond it none
    int *need;               // per rank: the link search has to visit the node
    int *ovf;                // per rank: its pair list did not fit
};

// ---- sizes the level's setup needs of the hierarchies and splits below ----
constexpr int BVH_LEAF = 32;
constexpr int BVH_LOG = 5;  // log2 of the leaf size and of the fan-out
constexpr int BVH_MAXH = 8;

__device__ __forceinline__ int bvh_levels(int nl)
{
    int h = 1;
    while (nl > 1) {
        nl = (nl + 31) >> BVH_LOG;
        h++;
    }
    return h;
}

__device__ __forceinline__ int64_t bvh_total(int nl)
{
    int64_t t = nl;
    while (nl > 1) {
        nl = (nl + 31) >> BVH_LOG;
        t += nl;
    }
    return t;
}

__host__ __device__ __forceinline__ int kd_split(int m)
{
    int h = ((m / 2 + 31) / 32) * 32;
    h = h < 32 ? 32 : h;
    return h > m - 1 ? m - 1 : h;
}

// splits until a range of m members is at most `limit`
__host__ __device__ __forceinline__ int kd_rounds(int64_t m, int limit)
{
    int r = 0;
    while (m > limit) {
        m = kd_split((int)m);
        r++;
    }
    return r;
}

constexpr int KD_CTA = 1024;  // ranges of at most this many members finish in one CTA

// Sample size of a node's search bracket: SMP_MAX above
// rs_tuning::bracket_min members (4096 by default), a quarter of it below.  A
// quarter costs up to a quarter of a small node's searches and gives twice as
// wide a bracket, but without one the node takes a search a member and a
// second one a leaf (2M path: the rest of the level's searches 1.3 -> 0.2 ms,
// the whole path 7.2 -> 6.0; 9.6M grouped members 42.0 -> 39.0).
constexpr int SMP_MAX = 1024;
constexpr int SMP_UNIT = SMP_MAX / 4;
__device__ __forceinline__ int smp_units(int n, int bracket_min) { return n > bracket_min ? SMP_MAX / SMP_UNIT : 1; }

// Per-rank offsets of one level (K + 1 entries each, the last the total)
struct LevelOff {
    int64_t *tile;   // tiles of TQ members
    int64_t *seg;    // members
    int64_t *box;    // hierarchy boxes
    int64_t *block;  // blocks of KD_CTA members
    int *smp;        // per SMP_UNIT samples: the rank of their node
    int *smp_at;     // per rank: its first unit of samples, or -1
};

constexpr int KD_MAXR = 16;   // kd_rounds(2^26, KD_CTA) and more
// words of the level's totals, read by the host in one go
enum { LT_K = 0, LT_T, LT_LM, LT_NBX, LT_SMP, LT_SUB, LT_ROUNDS, LT_ROUND0 = 8, LT_WORDS = LT_ROUND0 + 3 * KD_MAXR };

// One block sets a level up: the nodes in descending order of their k-d
// rounds (so the nodes that a round still splits are a prefix of the level's
// tiles, members and blocks), every per-rank offset and the totals, per round
// the prefix's tiles, members and blocks.  One launch and one host read
// instead of a count, a scan and a read for each array and each round.
__global__ void __launch_bounds__(1024) k_lvl_setup(const int *raw, const int *len, int *list, NodeArrays nd,
                                                    LevelOff O, int sub_n, int bracket_min, int64_t *tot)
{
    __shared__ int cls[KD_MAXR + 1], at[KD_MAXR + 1], start[KD_MAXR + 2], nsub;
    const int K = *len, tid = threadIdx.x;
    if (tid <= KD_MAXR) cls[tid] = 0;
    if (tid == 0) nsub = 0;
    __syncthreads();
    for (int i = tid; i < K; i += 1024) atomicAdd(&cls[min(kd_rounds(nd.count[raw[i]], KD_CTA), KD_MAXR)], 1);
    __syncthreads();
    if (tid == 0) {
        int s = 0;
        for (int c = KD_MAXR; c >= 0; c--) {
            start[c] = at[c] = s;  // start[c]: nodes of more than c rounds
            s += cls[c];
        }
    }
    __syncthreads();
    for (int i = tid; i < K; i += 1024) {
        const int node = raw[i];
        list[atomicAdd(&at[min(kd_rounds(nd.count[node], KD_CTA), KD_MAXR)], 1)] = node;
    }
    __syncthreads();
    long long c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0;
    for (int i0 = 0; i0 < K; i0 += 1024) {
        const int i = i0 + tid;
        const bool ok = i < K;
        const int n = ok ? nd.count[list[i]] : 0;
        if (ok && sub_n > 0 && n > sub_n) atomicAdd(&nsub, 1);
        const bool smp = ok && !(sub_n > 0 && n > sub_n);
        const int units = smp ? smp_units(n, bracket_min) : 0;
        long long s0, s1, s2, s3, s4;
        const long long v0 = rs_block_scan<1024, long long>(ceil_div(n, TQ), s0);
        const long long v1 = rs_block_scan<1024, long long>(n, s1);
        const long long v2 = rs_block_scan<1024, long long>(ok ? bvh_total((int)ceil_div(n, BVH_LEAF)) : 0, s2);
        const long long v3 = rs_block_scan<1024, long long>(ceil_div(n, KD_CTA), s3);
        const long long v4 = rs_block_scan<1024, long long>(units, s4);
        if (ok) {
            O.tile[i] = c0 + v0;
            O.seg[i] = c1 + v1;
            O.box[i] = c2 + v2;
            O.block[i] = c3 + v3;
            O.smp_at[i] = smp ? (int)(c4 + v4) : -1;
            for (int u = 0; u < units; u++) O.smp[c4 + v4 + u] = i;
        }
        c0 += s0;
        c1 += s1;
        c2 += s2;
        c3 += s3;
        c4 += s4;
    }
    if (tid == 0) {
        O.tile[K] = c0;
        O.seg[K] = c1;
        O.box[K] = c2;
        O.block[K] = c3;
        tot[LT_K] = K;
        tot[LT_T] = c0;
        tot[LT_LM] = c1;
        tot[LT_NBX] = c2;
        tot[LT_SMP] = c4;
        tot[LT_SUB] = nsub;
        int r = 0;
        while (r < KD_MAXR && start[r] > 0) r++;
        tot[LT_ROUNDS] = r;
    }
    __syncthreads();
    if (tid < KD_MAXR) {
        const int k = start[tid];
        tot[LT_ROUND0 + 3 * tid] = O.tile[k];
        tot[LT_ROUND0 + 3 * tid + 1] = O.seg[k];
        tot[LT_ROUND0 + 3 * tid + 2] = O.block[k];
    }
}

__global__ void k_lvl_tiles(int K, const int64_t *tile_off, int *tile_rank, int *tile_q0)
{
    int k = blockIdx.x;
    if (k >= K) return;
    int64_t a = tile_off[k], b = tile_off[k + 1];
    for (int64_t t = a + threadIdx.x; t < b; t += blockDim.x) {
        tile_rank[t] = k;
        tile_q0[t] = (int)((t - a) * TQ);
    }
}

// Four members a thread before the warp sums (the blocks of every fourth tile
// work): the sums' instructions, not the members' bytes, are what this costs
// (134M path, 7 levels: 5.4 -> 2.2 ms).
__global__ void __launch_bounds__(TQ) k_lvl_moments(LevelBufs L, NodeArrays nd, const float4 *wpos,
                                                    const float4 *wvel)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    if (q0 & (4 * TQ - 1)) return;
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const float4 pref = wpos[first], vref = wvel[first];
    MomRef ref = mom_ref(pref, vref);
    MomAcc a;
    mom_zero(a);
#pragma unroll 1
    for (int q = q0 + threadIdx.x; q < min(n, q0 + 4 * TQ); q += TQ) mom_add(a, wpos[first + q], wvel[first + q], ref);
    mom_warp_reduce(a);
    __shared__ MomAcc w[TQ / 32];
    if (lane_id() == 0) w[warp_id()] = a;
    __syncthreads();
    mom_block_add(&L.acc[k], w, TQ / 32);
    if (threadIdx.x == 0 && q0 == 0) {
        L.ref[2 * k] = pref;
        L.ref[2 * k + 1] = vref;
    }
}

__global__ void k_lvl_finalize(LevelBufs L, NodeArrays nd, double box)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    const int node = L.list[k];
    MomOut o = mom_finalize(L.acc[k], L.ref[2 * k], L.ref[2 * k + 1], nd.count[node], box);
    for (int d = 0; d < 3; d++) {
        nd.xbar[3 * node + d] = o.xbar[d];
        nd.vbar[3 * node + d] = o.vbar[d];
    }
    nd.sigx[node] = o.sigx;
    nd.sigv[node] = o.sigv;
    L.met[k] = metric_of(o.sigx, o.sigv);
    // the k-d order's scales, here and not in its kernels: two float64 divides
    // a member and round were what k_kd_keys spent its time on (134M path:
    // 12.4 -> 4.6 ms)
    L.ref[2 * k].w = o.sigx > 0 ? (float)(1.0 / o.sigx) : 0.f;
    L.ref[2 * k + 1].w = o.sigv > 0 ? (float)(1.0 / o.sigv) : 0.f;
}

// ---- raw-coordinate boxes ----
// A box is (lo, hi) over the six raw float32 coordinates of its members (the
// unwrapped positions and the velocities).  The gap between two boxes along
// an axis is one float32 subtraction of exact input values, so the box
// distance below is within 8 float32 ulps (relative) of the exact minimum
// squared distance between the boxes under the node's metric; a box is
// skipped only when that bound exceeds the current radius by 2^-18 relative,
// which can never skip a member whose float32 distance would change the
// result.

struct Box6 {
    float4 plo, phi, vlo, vhi;
};

// Boxes of one level's hierarchies as three float4 streams (the lows and
// highs of the six coordinates, 48 bytes a box) and one flag byte, so a warp
// reading 32 consecutive boxes uses every byte of every sector it touches.
struct BoxStore {
    float4 *a;         // plo.x, plo.y, plo.z, vlo.x
    float4 *b;         // vlo.y, vlo.z, phi.x, phi.y
    float4 *c;         // phi.z, vhi.x, vhi.y, vhi.z
    unsigned char *cl; // clique flag
};

__device__ __forceinline__ Box6 box_get(const BoxStore &S, int64_t i)
{
    const float4 x = S.a[i], y = S.b[i], z = S.c[i];
    Box6 r;
    r.plo = make_float4(x.x, x.y, x.z, 0.f);
    r.vlo = make_float4(x.w, y.x, y.y, 0.f);
    r.phi = make_float4(y.z, y.w, z.x, 0.f);
    r.vhi = make_float4(z.y, z.z, z.w, 0.f);
    return r;
}

__device__ __forceinline__ void box_put(const BoxStore &S, int64_t i, const Box6 &r)
{
    S.a[i] = make_float4(r.plo.x, r.plo.y, r.plo.z, r.vlo.x);
    S.b[i] = make_float4(r.vlo.y, r.vlo.z, r.phi.x, r.phi.y);
    S.c[i] = make_float4(r.phi.z, r.vhi.x, r.vhi.y, r.vhi.z);
}

__device__ __forceinline__ BoxStore box_shift(const BoxStore &S, int64_t base)
{
    BoxStore r;
    r.a = S.a + base;
    r.b = S.b + base;
    r.c = S.c + base;
    r.cl = S.cl + base;
    return r;
}

// The searched members of one level, packed to the six coordinates (24
// bytes a member, by slot): written while the hierarchy is built.
struct MemberStore {
    float4 *a;  // px, py, pz, vx
    float2 *b;  // vy, vz
};

__device__ __forceinline__ void mem_get(const MemberStore &M, int64_t i, float4 &p, float4 &v)
{
    const float4 x = M.a[i];
    const float2 y = M.b[i];
    p = make_float4(x.x, x.y, x.z, 0.f);
    v = make_float4(x.w, y.x, y.y, 0.f);
}

__device__ __forceinline__ MemberStore mem_shift(const MemberStore &M, int64_t base)
{
    MemberStore r;
    r.a = M.a + base;
    r.b = M.b + base;
    return r;
}

// ---- per-node 32-ary bounding-volume hierarchy over the member range ----
// Leaves hold BVH_LEAF = 32 consecutive members (the range is in k-d order at
// level 0, inherited below); box (h, i) of level h is the union of boxes
// (h-1, 32i .. 32i+31), so it spans members [i 32^(h+1), (i+1) 32^(h+1)).  The fan-out equals the
// warp width: a search gives each lane one child box of the box it opens, or
// one member of the leaf it scans.  Boxes of a node are stored level by
// level from its base offset.
// first member of box (h, i) and the end of its member range
__device__ __forceinline__ int64_t bvh_m0(int h, int i) { return (int64_t)i << (BVH_LOG * (h + 1)); }

__device__ __forceinline__ Box6 box_empty()
{
    Box6 b;
    b.plo = b.vlo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    b.phi = b.vhi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
    return b;
}

// warp min/max votes on order-preserving integer images
__device__ __forceinline__ float wmin_f(float x) { return ord_f(__reduce_min_sync(0xffffffffu, ord_i(x))); }
__device__ __forceinline__ float wmax_f(float x) { return ord_f(__reduce_max_sync(0xffffffffu, ord_i(x))); }

__device__ __forceinline__ float point_box_d2(float4 p, float4 v, const Box6 &b, const Metric6 &m)
{
    float gx = fmaxf(0.f, fmaxf(b.plo.x - p.x, p.x - b.phi.x)), gy = fmaxf(0.f, fmaxf(b.plo.y - p.y, p.y - b.phi.y)),
          gz = fmaxf(0.f, fmaxf(b.plo.z - p.z, p.z - b.phi.z));
    float gu = fmaxf(0.f, fmaxf(b.vlo.x - v.x, v.x - b.vhi.x)), gv = fmaxf(0.f, fmaxf(b.vlo.y - v.y, v.y - b.vhi.y)),
          gw = fmaxf(0.f, fmaxf(b.vlo.z - v.z, v.z - b.vhi.z));
    return (gx * gx + gy * gy + gz * gz) * m.ax + (gu * gu + gv * gv + gw * gw) * m.av;
}

// A node's hierarchy: its boxes and, per level, the first box (off) and the
// box count (cnt).  The two small per-level tables live in shared memory
// the caller provides (2 BVH_MAXH ints): the searches index them by a
// run-time level, which from registers would put them in local memory.
struct BvhView {
    BoxStore S;
    int nl, H;
    const int *off;
    const int *cnt;
};

__device__ __forceinline__ void bvh_fill(int *lv, int nl)
{
    int o = 0, c = nl;
    for (int h = 0; h < BVH_MAXH; h++) {
        lv[h] = o;
        lv[BVH_MAXH + h] = c;
        o += c;
        c = (c + 31) >> BVH_LOG;
    }
}

__device__ __forceinline__ void bvh_set(BvhView &V, const BoxStore &B, int64_t base, int n, const int *lv)
{
    V.S = box_shift(B, base);
    V.nl = (int)ceil_div(n, BVH_LEAF);
    V.H = min(bvh_levels(V.nl), BVH_MAXH);  // n <= 2^26 members per node (checked on the host): H <= 6
    V.off = lv;
    V.cnt = lv + BVH_MAXH;
}

// the view for a whole warp; lv is the warp's own shared table
__device__ __forceinline__ void bvh_view(BvhView &V, const BoxStore &B, int64_t base, int n, int *lv)
{
    if (lane_id() == 0) bvh_fill(lv, (int)ceil_div(n, BVH_LEAF));
    __syncwarp();
    bvh_set(V, B, base, n, lv);
}

// ---- dense boxes at the linking length ----
// A box whose float32 diameter under the node's metric is at most
// l^2 (1 - 2^-17) holds only mutual friends (the float32 diameter is within
// 8 ulps of the exact one), so all its members are joined once and a query
// that reaches the whole box within the same margin joins it with a single
// union.  These pairs lie strictly inside the linking length, never in the
// tie band.  The flag is kept in the box store's flag byte.

__device__ __forceinline__ float box_diam2(const Box6 &b, const Metric6 &m)
{
    float ex = b.phi.x - b.plo.x, ey = b.phi.y - b.plo.y, ez = b.phi.z - b.plo.z;
    float eu = b.vhi.x - b.vlo.x, ev = b.vhi.y - b.vlo.y, ew = b.vhi.z - b.vlo.z;
    return (ex * ex + ey * ey + ez * ez) * m.ax + (eu * eu + ev * ev + ew * ew) * m.av;
}

__device__ __forceinline__ float point_box_far2(float4 p, float4 v, const Box6 &b, const Metric6 &m)
{
    float fx = fmaxf(p.x - b.plo.x, b.phi.x - p.x), fy = fmaxf(p.y - b.plo.y, b.phi.y - p.y),
          fz = fmaxf(p.z - b.plo.z, b.phi.z - p.z);
    float fu = fmaxf(v.x - b.vlo.x, b.vhi.x - v.x), fv = fmaxf(v.y - b.vlo.y, b.vhi.y - v.y),
          fw = fmaxf(v.z - b.vlo.z, b.vhi.z - v.z);
    return (fx * fx + fy * fy + fz * fz) * m.ax + (fu * fu + fv * fv + fw * fw) * m.av;
}

// ---- building the boxes ----
// Three forms.  BOX_ALL, before the searches: boxes over all members, and the
// packed member copy.  BOX_PAIRS, for the nodes of the pair search (below):
// their flags and union-find entries at the bracket's lower edge, the boxes as
// they are.  BOX_LINK, for the nodes of the link search, once the linking
// length is known: the boxes are rebuilt over the members that can have a
// friend (nearest-neighbour value within reach; the others are neither queries
// nor candidates, and their packed x becomes infinite, which no box is within
// reach of), which drops the phase-space outliers that stretch them.  A box
// whose members all can have a friend and whose diameter is within the clique
// margin is flagged, and its members are joined: a leaf's when its members'
// union-find entries are first written, an upper box's by joining the first
// members of its children (a flagged box's children are flagged, their
// diameters being no larger).
enum { BOX_ALL, BOX_PAIRS, BOX_LINK };

// the union of one box per lane, in every lane
__device__ __forceinline__ Box6 warp_box(const Box6 &c)
{
    Box6 b;
    b.plo = make_float4(wmin_f(c.plo.x), wmin_f(c.plo.y), wmin_f(c.plo.z), 0.f);
    b.phi = make_float4(wmax_f(c.phi.x), wmax_f(c.phi.y), wmax_f(c.phi.z), 0.f);
    b.vlo = make_float4(wmin_f(c.vlo.x), wmin_f(c.vlo.y), wmin_f(c.vlo.z), 0.f);
    b.vhi = make_float4(wmax_f(c.vhi.x), wmax_f(c.vhi.y), wmax_f(c.vhi.z), 0.f);
    return b;
}

// whether the form visits node rank k, and the largest diameter of its cliques
template <int MODE>
__device__ __forceinline__ bool box_visits(const LevelBufs &L, int k, const float *R2, const float *STOP, float &clim)
{
    clim = 0.f;
    if (MODE == BOX_PAIRS) {
        clim = (float)((double)STOP[k] * RS_CLIQUE_MARGIN);
        return isfinite(R2[k]);
    }
    if (MODE == BOX_LINK) {
        clim = (float)(L.l2[k] * RS_CLIQUE_MARGIN);
        return L.need[k] != 0;
    }
    return true;
}

// Leaf boxes (one warp a leaf) and the boxes of 32 leaves above them.  A
// block takes the 1024 members of one such box: the tiles' grid, of which the
// blocks of every fourth tile work.  Against one thread a leaf in one block a
// node (the link form before: 3.5 ms of a 16.8M-particle path, its largest
// node alone on one SM), the loads coalesce and a large node spreads over the
// device.
template <int MODE>
__global__ void __launch_bounds__(TQ) k_bvh_leaves(LevelBufs L, NodeArrays nd, int64_t tile0, const int64_t *box_base,
                                                   BoxStore B, MemberStore MS, const float4 *wpos, const float4 *wvel,
                                                   const float *R2, const float *STOP, float *dnn, int *parent,
                                                   int *csize, int *cmin, rs_dev_status *st)
{
    __shared__ float bs[32][12];
    __shared__ unsigned char cs[32];
    const int64_t tile = tile0 + blockIdx.x;
    const int qb = L.tile_q0[tile];
    if (qb & 1023) return;
    const int k = L.tile_rank[tile];
    float clim;
    if (!box_visits<MODE>(L, k, R2, STOP, clim)) return;
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int lane = lane_id();
    const BoxStore bx = box_shift(B, box_base[k]);
    Metric6 met;
    met.ax = L.met[k].ax;
    met.av = L.met[k].av;
    const float part = MODE == BOX_LINK ? link_part(L.l2[k]) : 0.f;
    for (int j = warp_id(); j < 32; j += TQ / 32) {
        const int q0 = qb + 32 * j, m = q0 + lane;
        if (q0 >= n) break;
        const bool ok = m < n;
        bool act = ok;
        Box6 b;
        if (MODE == BOX_PAIRS) {
            b = box_get(bx, q0 / BVH_LEAF);
        } else {
            float4 p = make_float4(0, 0, 0, 0), v = p;
            if (ok) {
                if (MODE == BOX_LINK) {
                    mem_get(mem_shift(MS, first), m, p, v);
                    act = dnn[first + m] <= part;
                    if (!act) MS.a[first + m].x = INFINITY;
                } else {
                    p = wpos[first + m];
                    v = wvel[first + m];
                    MS.a[first + m] = make_float4(p.x, p.y, p.z, v.x);
                    MS.b[first + m] = make_float2(v.y, v.z);
                }
            }
            b = box_empty();
            if (act) {
                b.plo = b.phi = p;
                b.vlo = b.vhi = v;
            }
            b = warp_box(b);
        }
        bool clique = false;
        if (MODE != BOX_ALL) {
            const float diam = box_diam2(b, met);
            clique = __ballot_sync(0xffffffffu, act) == __ballot_sync(0xffffffffu, ok) && diam <= clim;
            // (a lone member has no neighbour in its leaf)
            if (MODE == BOX_PAIRS) clique = clique && q0 + 1 < n;
            if (ok) {
                parent[first + m] = clique ? first + q0 : first + m;
                csize[first + m] = 0;
                cmin[first + m] = 0x7fffffff;
                // a clique's members have a neighbour below the bracket, which
                // is all that matters of its distance
                if (MODE == BOX_PAIRS) dnn[first + m] = clique ? diam : INFINITY;
            }
        }
        if (lane == 0) {
            if (MODE != BOX_PAIRS) box_put(bx, q0 / BVH_LEAF, b);
            if (MODE != BOX_ALL) bx.cl[q0 / BVH_LEAF] = cs[j] = clique ? 1 : 0;
            float *o = bs[j];
            o[0] = b.plo.x; o[1] = b.plo.y; o[2] = b.plo.z; o[3] = b.vlo.x; o[4] = b.vlo.y; o[5] = b.vlo.z;
            o[6] = b.phi.x; o[7] = b.phi.y; o[8] = b.phi.z; o[9] = b.vhi.x; o[10] = b.vhi.y; o[11] = b.vhi.z;
        }
    }
    __syncthreads();
    const int nl = (int)ceil_div(n, BVH_LEAF), i0 = qb / BVH_LEAF;
    if (warp_id() != 0 || nl < 2) return;
    const bool have = i0 + lane < nl;
    Box6 b = box_empty();
    if (have) {
        const float *o = bs[lane];
        b.plo = make_float4(o[0], o[1], o[2], 0.f);
        b.vlo = make_float4(o[3], o[4], o[5], 0.f);
        b.phi = make_float4(o[6], o[7], o[8], 0.f);
        b.vhi = make_float4(o[9], o[10], o[11], 0.f);
    }
    b = warp_box(b);
    const bool clique = MODE != BOX_ALL && !__any_sync(0xffffffffu, have && !cs[lane]) && box_diam2(b, met) <= clim;
    if (lane == 0) {
        if (MODE != BOX_PAIRS) box_put(bx, nl + (qb >> 10), b);
        if (MODE != BOX_ALL) bx.cl[nl + (qb >> 10)] = clique ? 1 : 0;
    }
    if (clique && have && lane > 0) uf_union(parent, first + qb, first + qb + 32 * lane, st);
}

// the levels above, one block a node, one warp a box
template <int MODE>
__global__ void __launch_bounds__(256) k_bvh_build(LevelBufs L, NodeArrays nd, const int64_t *box_base, BoxStore B,
                                                   const float *R2, const float *STOP, int *parent, rs_dev_status *st)
{
    const int k = blockIdx.x;
    float clim;
    if (k >= L.K || !box_visits<MODE>(L, k, R2, STOP, clim)) return;
    const int node = L.list[k], n = nd.count[node], first = nd.first[node];
    const int nl = (int)ceil_div(n, BVH_LEAF);
    const BoxStore bx = box_shift(B, box_base[k]);
    const int H = bvh_levels(nl), lane = lane_id();
    Metric6 met;
    met.ax = L.met[k].ax;
    met.av = L.met[k].av;
    int cprev = (nl + 31) >> BVH_LOG;
    int64_t off_prev = nl, off = nl + cprev;
    for (int h = 2; h < H; h++) {
        const int cnt = (cprev + 31) >> BVH_LOG;
        for (int i = warp_id(); i < cnt; i += 8) {
            const int c = 32 * i + lane;
            const bool have = c < cprev;
            Box6 b = box_empty();
            if (have) b = box_get(bx, off_prev + c);
            b = warp_box(b);
            const bool clique = MODE != BOX_ALL && !__any_sync(0xffffffffu, have && !bx.cl[off_prev + c]) &&
                                box_diam2(b, met) <= clim;
            if (lane == 0) {
                if (MODE != BOX_PAIRS) box_put(bx, off + i, b);
                if (MODE != BOX_ALL) bx.cl[off + i] = clique ? 1 : 0;
            }
            if (clique && have && lane > 0)
                uf_union(parent, first + (int)bvh_m0(h, i), first + (int)bvh_m0(h - 1, c), st);
        }
        __syncthreads();
        off_prev = off;
        off += cnt;
        cprev = cnt;
    }
}

// ---- warp-per-query search over the 32-ary hierarchy ----
// One query at a time per warp.  Opening a box, lane c bounds the query's
// distance to child box c (a float32 point-to-box gap, within 8 ulps of the
// exact one; a box is skipped only when the bound exceeds the radius by
// 2^-18, so no member that could change a float32 result is skipped).
// Scanning a leaf, lane c evaluates member c and the warp minimum (redux on
// the bit patterns, which order like the non-negative floats) updates the
// radius.  The leaves under an opened box are scanned nearest first and
// re-tested as the radius shrinks; needed inner boxes are pushed on a
// shared-memory stack all at once, each with its bound, the nearest on top.
constexpr int W_WARPS = 8;    // warps per block of the search kernels
constexpr int W_STACK = 192;  // stack entries per warp: at most 31 pending per level
constexpr unsigned FULLW = 0xffffffffu;

__device__ __forceinline__ unsigned ford(float x) { return __float_as_uint(x); }

__device__ __forceinline__ float wmin(float x) { return __uint_as_float(__reduce_min_sync(FULLW, ford(x))); }

__device__ __forceinline__ float4 shfl4(float4 a, int src)
{
    return make_float4(__shfl_sync(FULLW, a.x, src), __shfl_sync(FULLW, a.y, src), __shfl_sync(FULLW, a.z, src), 0.f);
}

// Nearest-neighbour distance of member q (coordinates pq, vq) among the
// node's members P, Q (n of them), starting from the radius `best` (the own
// leaf `own` already scanned).  Returns as soon as the radius drops below
// `stop`.  `best` is warp-uniform throughout.
__device__ __forceinline__ float w32_nn(const BvhView &V, const MemberStore &M, int n, int q, float4 pq, float4 vq,
                        const Metric6 &met, float best, float stop, int own, int *si, float *sd, rs_dev_status *st,
                        int node)
{
    const int lane = lane_id();
    if (V.H < 2 || best < stop) return best;
    if (lane == 0) {
        si[0] = (V.H - 1) << 24;
        sd[0] = 0.f;
    }
    int sp = 1;
    __syncwarp();
    for (int it = 0; sp > 0 && it < (1 << 24); it++) {
        sp--;
        const int ent = si[sp];
        const float elb = sd[sp];
        __syncwarp();
        if (elb > best * RS_PRUNE_SLACK) continue;
        const int ch = (ent >> 24) - 1, i = ent & 0xffffff;
        const int c = 32 * i + lane;
        const bool ok = c < V.cnt[ch] && !(ch == 0 && c == own);
        const float lb = ok ? point_box_d2(pq, vq, box_get(V.S, V.off[ch] + c), met) : INFINITY;
        unsigned mask = __ballot_sync(FULLW, ok && lb <= best * RS_PRUNE_SLACK);
        if (ch == 0) {
            // the two nearest needed leaves at a time (their loads overlap)
            while (mask) {
                bool mine = (mask >> lane) & 1u;
                unsigned key = mine ? ford(lb) : 0xffffffffu;
                unsigned mn = __reduce_min_sync(FULLW, key);
                const int s0 = __ffs(__ballot_sync(FULLW, mine && key == mn)) - 1;
                mask &= ~(1u << s0);
                int s1 = -1;
                if (mask) {
                    mine = (mask >> lane) & 1u;
                    key = mine ? ford(lb) : 0xffffffffu;
                    mn = __reduce_min_sync(FULLW, key);
                    s1 = __ffs(__ballot_sync(FULLW, mine && key == mn)) - 1;
                    mask &= ~(1u << s1);
                }
                const int m0 = (32 * i + s0) * BVH_LEAF + lane, m1 = (32 * i + s1) * BVH_LEAF + lane;
                const bool v0 = m0 < n && m0 != q, v1 = s1 >= 0 && m1 < n && m1 != q;
                float4 p0 = make_float4(0, 0, 0, 0), u0 = p0, p1 = p0, u1 = p0;
                if (v0) mem_get(M, m0, p0, u0);
                if (v1) mem_get(M, m1, p1, u1);
                float d = v0 ? d2_32(pq, vq, p0, u0, met) : INFINITY;
                if (v1) d = fminf(d, d2_32(pq, vq, p1, u1, met));
                best = fminf(best, wmin(d));
                if (best < stop) return best;
                mask &= __ballot_sync(FULLW, lb <= best * RS_PRUNE_SLACK);
            }
            continue;
        }
        if (sp + __popc(mask) > W_STACK) {
            if (lane == 0) dev_fail(st, DEV_OVERFLOW, 54, node);
            return best;
        }
        if (mask) {
            const bool mine = (mask >> lane) & 1u;
            const int cntm = __popc(mask);
            if (mine) {
                const int slot = sp + __popc(mask & ((1u << lane) - 1u));
                si[slot] = (ch << 24) | c;
                sd[slot] = lb;
            }
            const unsigned key = mine ? ford(lb) : 0xffffffffu;
            const unsigned mn = __reduce_min_sync(FULLW, key);
            const int src = __ffs(__ballot_sync(FULLW, mine && key == mn)) - 1;
            const int top = sp + cntm - 1, from = sp + __popc(mask & ((1u << src) - 1u));
            __syncwarp();
            if (lane == 0 && from != top) {
                const int e0 = si[from];
                const float d0 = sd[from];
                si[from] = si[top];
                sd[from] = sd[top];
                si[top] = e0;
                sd[top] = d0;
            }
            sp += cntm;
        }
        __syncwarp();
    }
    return best;
}

// nearest-neighbour distances, one warp per job of 32 consecutive members
// (one leaf): the leaf is held in registers, one member per lane, and its 32
// queries are searched one after another.  Blocks are of NN_WARPS warps, so a
// slot frees as soon as its few warps end.
constexpr int NN_WARPS = 4;
template <int MINB>
__global__ void __launch_bounds__(NN_WARPS * 32, MINB * W_WARPS / NN_WARPS)
    k_bvh_nn(LevelBufs L, NodeArrays nd, const int64_t *box_base, BoxStore B, MemberStore MS, const float *R2,
             const float *STOP, int redo_failed, int sub_n, int pairs, float *out, rs_dev_status *st)
{
    __shared__ int si_s[NN_WARPS][W_STACK];
    __shared__ float sd_s[NN_WARPS][W_STACK];
    __shared__ int lv_s[NN_WARPS][2 * BVH_MAXH];
    const int w = warp_id(), lane = lane_id();
    // the grid holds exactly the tiles' warps
    constexpr int bpt = (TQ / 32) / NN_WARPS;
    const int tile = blockIdx.x / bpt;
    const int k = L.tile_rank[tile], q0 = L.tile_q0[tile] + 32 * ((blockIdx.x % bpt) * NN_WARPS + w);
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    // (a node above the subset size searches its subset members one by one)
    if (q0 >= n || (sub_n > 0 && n > sub_n)) return;
    if (pairs && isfinite(R2[k]) && R2[k] >= 0.f) return;  // the pair search took it
    const Metric6 met = L.met[k];
    BvhView V;
    bvh_view(V, B, box_base[k], n, lv_s[w]);
    const MemberStore M = mem_shift(MS, first);
    // start from the node's radius when one is given (just above it, so a
    // result at or above the start means "nothing within the radius"); a
    // query whose radius falls below the stop value is done: its member is
    // certainly below the linking length and its exact value is not needed.
    // With redo_failed, only the nodes whose bracket failed (R2 = -1) are
    // searched again, unbounded.
    float start = INFINITY, stop = 0.f;
    if (redo_failed) {
        if (!(R2[k] < 0.f)) return;
    } else {
        start = R2 ? R2[k] * 1.00000095367431640625f : INFINITY;
        stop = STOP ? STOP[k] : 0.f;
    }
    const int own = q0 / BVH_LEAF;
    const int mo = q0 + lane;
    const bool have = mo < n;
    float4 po = make_float4(0, 0, 0, 0), vo = po;
    if (have) mem_get(M, mo, po, vo);
    const int nq = min(32, n - q0);
    float res = INFINITY;
    for (int j = 0; j < nq; j++) {
        const float4 pq = shfl4(po, j), vq = shfl4(vo, j);
        const float d = (have && lane != j) ? d2_32(pq, vq, po, vo, met) : INFINITY;
        float best = fminf(start, wmin(d));
        best = w32_nn(V, M, n, q0 + j, pq, vq, met, best, stop, own, si_s[w], sd_s[w], st, node);
        if (lane == j) res = best;
    }
    if (have) out[first + mo] = res >= start ? INFINITY : res;
}

// nearest-neighbour distance of single sampled members, one warp each
__global__ void __launch_bounds__(W_WARPS * 32) k_bvh_nn_sample(LevelBufs L, NodeArrays nd, const int64_t *box_base,
                                                                BoxStore B, MemberStore MS, const int *smp,
                                                                const int *smp_at, int bracket_min, float *out,
                                                                rs_dev_status *st)
{
    __shared__ int si_s[W_WARPS][W_STACK];
    __shared__ float sd_s[W_WARPS][W_STACK];
    __shared__ int lv_s[W_WARPS][2 * BVH_MAXH];
    const int w = warp_id(), lane = lane_id();
    const int64_t at = (int64_t)blockIdx.x * W_WARPS + w;  // the grid holds exactly the samples
    const int k = smp[at / SMP_UNIT], s = (int)(at - (int64_t)smp_at[k] * SMP_UNIT);
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int q = (int)(((int64_t)s * n) / (SMP_UNIT * smp_units(n, bracket_min)));
    const Metric6 met = L.met[k];
    BvhView V;
    bvh_view(V, B, box_base[k], n, lv_s[w]);
    const MemberStore M = mem_shift(MS, first);
    float4 pq, vq, pm = make_float4(0, 0, 0, 0), vm = pm;
    mem_get(M, q, pq, vq);
    const int own = q / BVH_LEAF, m = own * BVH_LEAF + lane;
    if (m < n) mem_get(M, m, pm, vm);
    const float d = (m < n && m != q) ? d2_32(pq, vq, pm, vm, met) : INFINITY;
    const float best = w32_nn(V, M, n, q, pq, vq, met, wmin(d), 0.f, own, si_s[w], sd_s[w], st, node);
    if (lane == 0) out[at] = best;
}

// nearest-neighbour distance of listed members (rank, member), one warp
// each, unbounded; the result goes to the member's own slot
__global__ void __launch_bounds__(W_WARPS * 32) k_bvh_nn_list(LevelBufs L, NodeArrays nd, const int64_t *box_base,
                                                              BoxStore B, MemberStore MS, const int2 *qlist,
                                                              const int *qlen, int cap, float *dnn,
                                                              rs_dev_status *st)
{
    __shared__ int si_s[W_WARPS][W_STACK];
    __shared__ float sd_s[W_WARPS][W_STACK];
    __shared__ int lv_s[W_WARPS][2 * BVH_MAXH];
    const int w = warp_id(), lane = lane_id();
    const int64_t s = (int64_t)blockIdx.x * W_WARPS + w;
    if (s >= min(*qlen, cap)) return;
    const int2 e = qlist[s];
    const int k = e.x, q = e.y;
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const Metric6 met = L.met[k];
    BvhView V;
    bvh_view(V, B, box_base[k], n, lv_s[w]);
    const MemberStore M = mem_shift(MS, first);
    float4 pq, vq, pm = make_float4(0, 0, 0, 0), vm = pm;
    mem_get(M, q, pq, vq);
    const int own = q / BVH_LEAF, m = own * BVH_LEAF + lane;
    if (m < n) mem_get(M, m, pm, vm);
    const float d = (m < n && m != q) ? d2_32(pq, vq, pm, vm, met) : INFINITY;
    const float best = w32_nn(V, M, n, q, pq, vq, met, wmin(d), 0.f, own, si_s[w], sd_s[w], st, node);
    if (lane == 0) dnn[first + q] = best;
}

// one candidate pair: bit 0 set when it is within l (decided in float64
// inside the band), bit 1 set for a pair within 1e-6 (relative) of l but not
// at it
// (The float64 metric and l^2 are read from memory on the rare band path
// only, which keeps them out of the search kernel's registers.)
__device__ __forceinline__ int pair_test(const LinkLim &lm, const Metric6 &met, const Metric6 *met64,
                                         const double *l2p, float4 pa, float4 va, float4 pb, float4 vb)
{
    const float d2 = d2_32(pa, va, pb, vb, met);
    if (d2 > lm.part) return 0;
    // below both bands (the linking band and the wider tie band): a friend,
    // and not a tie-band pair
    if (d2 < fminf(lm.lo, lm.tlo)) return 1;
    const Metric6 m = *met64;
    const double l2 = *l2p, l = sqrt(l2);
    const double e64 = d2_64(pa, va, pb, vb, m);
    const int tie = (l2 > 0 && e64 != l2 && fabs(sqrt(e64) - l) <= 1e-6 * l) ? 2 : 0;
    return (e64 <= l2 ? 1 : 0) | tie;
}

// Join a and b; returns the smaller of the two roots it joined (a member of
// the merged set).
__device__ __forceinline__ int uf_union_root(int *parent, int a, int b, rs_dev_status *st)
{
    for (int it = 0; it < RS_SPIN_LIMIT; it++) {
        a = uf_find(parent, a, st);
        b = uf_find(parent, b, st);
        if (a == b) return a;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicCAS(&parent[b], b, a);
        if (old == b) return a;
        b = old;
    }
    dev_fail(st, DEV_TIMEOUT, 2, a);
    return a;
}

// Join the query's set with friend b.  `rq` is a member known to be in the
// query's set (sets only grow, so it stays one): when b's parent is rq the
// two are joined already and the union is skipped.  Dense regions give each
// query many friends whose parent is the set's root, so most unions end at
// this one load.  Returns a member of the merged set, or INT_MAX when skipped.
__device__ __forceinline__ int join_friend(int *parent, int a, int b, int rq, rs_dev_status *st)
{
    if (__ldcg(&parent[b]) == rq) return 0x7fffffff;
    return uf_union_root(parent, a, b, st);
}

// ---- friends-of-friends at l: one warp per leaf, pairs found by the matrix units ----
// A warp takes the 32 members of a leaf together.  It walks the hierarchy
// once for all of them, box against box, for the leaves within reach of its
// own leaf's box; keeps, of each such leaf's 32 members, those within reach of
// the box (a tenth to a seventh of them on the catalogues of synth.py); and
// screens the kept ones, 32 at a time, against its 32 members on the matrix
// units, in units of the linking radius about the leaf box's centre: a pair
// whose product minus T, the bound for pairs within the linking radius (see
// the half-precision points), is positive is no friend.
// T stays below 1.02 for the usual boxes (2.7 linking lengths in radius), so
// the few pairs it lets through (about 20 of 1024) are nearly all friends;
// they are queued and evaluated 32 at a time in full, as float32 differences
// of the members' own coordinates with the float64 recheck in the band.  A
// leaf whose box is too large for half precision (or whose l is 0, or so small
// that float32 cannot hold one over it) queues every kept pair instead.
//
// Bound by instruction issue and the latency of the dependent walk.  Walking
// once a leaf instead of once a query cut the link of the 134M-particle path
// (7 levels) from 240 to 68 ms, of 9.6M members in independent groups from 46
// to 13.8 ms, of a 2M path from 4.3 to 0.85 ms.  32 resident warps (64
// registers, the pair search spilling 40 bytes) against 40 (48 registers and
// 112 bytes: 74 ms) and 48 (81 ms).
constexpr int LK_STACK = 256;   // link stack entries per warp
constexpr int LK_LEAVES = 128;  // pending leaves per warp
constexpr int LK_RING = 128;    // kept candidates per warp (a ring; 32 are consumed at a time)
constexpr float LK_RMAX = 100.f;  // largest box radius, in linking lengths, for the half-precision test

// box-to-box lower bound on the squared distance (each gap is one rounded
// float32 difference of members' coordinates, as in point_box_d2)
__device__ __forceinline__ float box_box_d2(const Box6 &a, const Box6 &b, const Metric6 &m)
{
    const float gx = fmaxf(0.f, fmaxf(b.plo.x - a.phi.x, a.plo.x - b.phi.x)),
                gy = fmaxf(0.f, fmaxf(b.plo.y - a.phi.y, a.plo.y - b.phi.y)),
                gz = fmaxf(0.f, fmaxf(b.plo.z - a.phi.z, a.plo.z - b.phi.z));
    const float gu = fmaxf(0.f, fmaxf(b.vlo.x - a.vhi.x, a.vlo.x - b.vhi.x)),
                gv = fmaxf(0.f, fmaxf(b.vlo.y - a.vhi.y, a.vlo.y - b.vhi.y)),
                gw = fmaxf(0.f, fmaxf(b.vlo.z - a.vhi.z, a.vlo.z - b.vhi.z));
    return (gx * gx + gy * gy + gz * gz) * m.ax + (gu * gu + gv * gv + gw * gw) * m.av;
}

// ---- nearest neighbours and friends in one search: the pair search ----
// A node with a sampled bracket [stop, R2] around its linking length (squared)
// needs one search only.  Walked at R2, leaf against leaf as above, it meets
// every pair that matters: each evaluated pair lowers the nearest-neighbour
// values of both its members; a pair below stop is a friend whatever the
// linking length turns out to be, and is joined at once; the pairs between
// stop and R2 (13 a member at f = 0.7) are listed, and once the linking length
// is known the list is gone through (k_pair_link).  A node whose bracket
// fails, or whose pairs do not fit the list, is searched for friends again
// from scratch.
//
// Against a nearest-neighbour search a member and a link search a leaf: 118 +
// 67 ms of a 134M-particle path became 89 (pairs) + 6 (list), 9.6M members in
// groups 19.5 + 13.7 became 17.1 + 1.2.  The list moves 9 bytes a pair each
// way, a few percent of the search.
//
// The list is in chunks of PAIR_CHUNK pairs of one leaf, with a head (node
// rank, first query, pairs), in PAIR_REGIONS regions with a counter each.  A
// block takes its chunks of one region, and of the following ones once that is
// full: a small level has fewer blocks than regions, and its first leaves list
// twice the mean (a pair is listed with its first member), so without that a
// node of 1100 members ran out of room with two thirds of the chunks unused.
constexpr int PAIR_CHUNK = 64;
constexpr int PAIR_REGIONS = 64;
constexpr int PAIR_PER_MEMBER = 20;                  // room for this many pairs a member
constexpr int64_t PAIR_MAX_BYTES = (int64_t)16 << 30;  // no list beyond this

struct PairList {
    int4 *head;    // (rank, first query, pairs, 0) per chunk
    int2 *pair;    // (query lane << 26 | member, float32 distance) per pair
    int *len;      // chunks taken per region
    int cap;       // chunks per region
    const float *R2, *STOP;
    float *dnn;
};

// a region after a full one with a chunk left, and the chunk (cap when there is
// none), for a whole warp; the pairs of a node that ran out are not needed
static __device__ __noinline__ int2 next_chunk(int *len, int cap, const int *ovf, int full)
{
    int c = cap, r = full;
    if (lane_id() == 0 && !__ldcg(ovf))
        for (int t = 1; t < PAIR_REGIONS && c >= cap; t++) {
            r = (full + t) & (PAIR_REGIONS - 1);
            if (__ldcg(&len[r]) < cap) c = atomicAdd(&len[r], 1);
        }
    return make_int2(__shfl_sync(0xffffffffu, r, 0), __shfl_sync(0xffffffffu, c, 0));
}

template <bool PAIRS>
struct PairStage {
    int2 out[96];  // pairs on their way to the list
    int best[32];  // per query: nearest-neighbour value so far (bits)
};
template <>
struct PairStage<false> {
};

template <bool PAIRS>
struct LinkWarp : PairStage<PAIRS> {
    uint4 cand[32];         // 32 candidates (or, at first, the queries) as eight halves
    float4 qa[32];          // the queries: px, py, pz, vx
    float2 qb[32];          //              vy, vz
    float4 box[4];          // the leaf's box (plo, phi, vlo, vhi)
    float4 pc, vc;          // its centre; .w: the metric's weights over the linking radius
    int ring[LK_RING];      // kept candidates (member of the node)
    int pairs[64];          // (query lane << 26) | member, to be evaluated
    int stack[LK_STACK];
    int leaf[LK_LEAVES];
    int rq[32];             // per query: a member of its set
    int lv[2 * BVH_MAXH];
};

// friends-of-friends at l, one warp per leaf of 32 consecutive members, pairs
// with the candidate after the query in the node's member order; only
// members with a neighbour within reach take part.  A tile's eight warps are
// spread over blocks of LK_WARPS warps: the cost of a leaf varies widely, and
// a small block frees its slot as soon as its own few warps end instead of
// waiting for the slowest of eight.
constexpr int LK_WARPS = 2;
template <int WARPS, bool PAIRS>
__global__ void __launch_bounds__(LK_WARPS * 32, WARPS / LK_WARPS)
    k_bvh_link(LevelBufs L, NodeArrays nd, int64_t tile0, const int64_t *box_base, BoxStore B, MemberStore MS,
               int *parent, PairList P, rs_dev_status *st)
{
    static_assert((TQ / 32) % LK_WARPS == 0, "a tile's warps fill whole blocks");
    __shared__ LinkWarp<PAIRS> sh[LK_WARPS];
    const int w = warp_id(), lane = lane_id();
    LinkWarp<PAIRS> &S = sh[w];
    // the grid holds exactly the tiles' warps: block b takes warps
    // (b % bpt) * LK_WARPS + w of tile b / bpt
    constexpr int bpt = (TQ / 32) / LK_WARPS;
    const int64_t tile = tile0 + blockIdx.x / bpt;
    const int jw = (blockIdx.x % bpt) * LK_WARPS + w;
    const int k = L.tile_rank[tile], q0 = L.tile_q0[tile] + 32 * jw;
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    if (q0 >= n || (PAIRS ? !isfinite(P.R2[k]) : !L.need[k])) return;
    const MemberStore M = mem_shift(MS, first);
    const int mo = q0 + lane;
    float4 po = make_float4(INFINITY, 0, 0, 0), vo = make_float4(0, 0, 0, 0);
    if (mo < n) mem_get(M, mo, po, vo);
    // (in the link search a member without a neighbour within reach has an
    // infinite packed x)
    const bool act = po.x < INFINITY;
    const unsigned actm = __ballot_sync(FULLW, act);
    if (!actm) return;
    Metric6 met;  // float32 factors only; the float64 ones are read where needed
    met.ax = L.met[k].ax;
    met.av = L.met[k].av;
    const Metric6 *met64 = L.met + k;
    const double *l2p = L.l2 + k;
    // search radius: every pair that matters is within it
    LinkLim lm = link_lim(PAIRS ? 0.0 : L.l2[k]);
    const float stop = PAIRS ? P.STOP[k] : 0.f;
    if (PAIRS) {
        lm.part = P.R2[k];
        lm.lim = lm.part * RS_PRUNE_SLACK;
        lm.cl_lim = (float)((double)stop * RS_CLIQUE_MARGIN);
    }
    BvhView V;
    bvh_view(V, B, box_base[k], n, S.lv);
    const int own = q0 / BVH_LEAF;
    S.qa[lane] = make_float4(po.x, po.y, po.z, vo.x);
    S.qb[lane] = make_float2(vo.y, vo.z);
    S.rq[lane] = act ? __ldcg(&parent[first + mo]) : 0;
    if constexpr (PAIRS) S.best[lane] = 0x7f800000;
    const bool own_clique = PAIRS && V.S.cl[own] != 0;  // its own pairs are settled

    // ---- half-precision frame: centre, weights, the queries' fragments ----
    bool brute;
    unsigned a[4];
    float cr[4];
    {
    const Box6 bx = box_get(V.S, own);
    const float4 pc = make_float4(0.5f * bx.plo.x + 0.5f * bx.phi.x, 0.5f * bx.plo.y + 0.5f * bx.phi.y,
                                  0.5f * bx.plo.z + 0.5f * bx.phi.z, 0.f);
    const float4 vc = make_float4(0.5f * bx.vlo.x + 0.5f * bx.vhi.x, 0.5f * bx.vlo.y + 0.5f * bx.vhi.y,
                                  0.5f * bx.vlo.z + 0.5f * bx.vhi.z, 0.f);
    const float wx = sqrtf(met.ax / lm.part), wv = sqrtf(met.av / lm.part);
    const float rb = sqrtf(point_box_far2(pc, vc, bx, met) / lm.part);
    // (weights beyond float32's range would make every product a NaN)
    brute = !(rb <= LK_RMAX && lm.part < 1e30f && lm.part > 1e-30f);
    if (lane == 0) {
        S.box[0] = bx.plo;
        S.box[1] = bx.phi;
        S.box[2] = bx.vlo;
        S.box[3] = bx.vhi;
        S.pc = make_float4(pc.x, pc.y, pc.z, wx);
        S.vc = make_float4(vc.x, vc.y, vc.z, wv);
    }
    const float rsum = 2.f * rb + 1.01f;
    const float dl = 1.02f * 4.8828125e-4f * rsum + 3.1e-4f;
    const float T = (1.f + dl) * (1.f + dl) * 1.00002f + 3.814697265625e-6f * rsum * rsum + 1.e-4f;
        float s;
        const bool in = act && !brute;
        uint4 row = half_point(in ? po : pc, in ? vo : vc, pc, vc, wx, wv, s);
        row.x = half_query(row.x, 0);
        row.y = half_query(row.y, 1);
        row.z = half_query(row.z, 2);
        row.w = HALF_ONES;
        S.cand[lane] = row;
        s = act ? s - T : 60000.f;
        __syncwarp();
        const unsigned *cw = (const unsigned *)S.cand;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            a[i] = cw[4 * (8 * i + (lane >> 2)) + (lane & 3)];
            cr[i] = __shfl_sync(FULLW, s, 8 * i + (lane >> 2));
        }
        __syncwarp();
    }

    int tie = 0, np = 0, no = 0;       // queued pairs, pairs on their way to the list
    int head = 0, nc = 0;              // ring of kept candidates
    const unsigned below = (1u << lane) - 1u;
    // the last cnt staged pairs to a chunk of the list
    auto put_chunk = [&](int cnt) {
        if constexpr (PAIRS) {
            int region = blockIdx.x & (PAIR_REGIONS - 1);
            no -= cnt;
            int c = 0;
            if (lane == 0) c = atomicAdd(&P.len[region], 1);
            c = __shfl_sync(FULLW, c, 0);
            if (c >= P.cap) {
                const int2 next = next_chunk(P.len, P.cap, L.ovf + k, region);
                region = next.x;
                c = next.y;
            }
            if (c < P.cap) {
                const int64_t at = (int64_t)region * P.cap + c;
                for (int i = lane; i < cnt; i += 32) P.pair[at * PAIR_CHUNK + i] = S.out[no + i];
                if (lane == 0) P.head[at] = make_int4(k, q0, cnt, 0);
            } else if (lane == 0) {
                L.ovf[k] = 1;
            }
            __syncwarp();
        }
    };
    // evaluates up to 32 queued pairs, one a lane
    auto flush = [&](int cnt) {
        np -= cnt;
        const int code = lane < cnt ? S.pairs[np + lane] : 0;
        const int r = code >> 26, m = code & 0x3ffffff;
        if constexpr (PAIRS) {
            bool keep = false;
            float d2 = 0.f;
            if (lane < cnt && m > q0 + r) {
                float4 pm, vm;
                mem_get(M, m, pm, vm);
                const float4 x = S.qa[r];
                const float2 y = S.qb[r];
                d2 = d2_32(make_float4(x.x, x.y, x.z, 0.f), make_float4(x.w, y.x, y.y, 0.f), pm, vm, met);
                if (d2 <= lm.part) {
                    const int bits = __float_as_int(d2);
                    int *dm = reinterpret_cast<int *>(P.dnn) + first + m;
                    if (bits < ((volatile int *)S.best)[r]) atomicMin(&S.best[r], bits);
                    if (bits < __ldcg(dm)) atomicMin(dm, bits);
                    keep = !(d2 < stop);
                    if (!keep) {
                        const int root = join_friend(parent, first + q0 + r, first + m, ((volatile int *)S.rq)[r], st);
                        if (root != 0x7fffffff) atomicMin(&S.rq[r], root);
                    }
                }
            }
            const unsigned km = __ballot_sync(FULLW, keep);
            if (keep) S.out[no + __popc(km & below)] = make_int2(code, __float_as_int(d2));
            no += __popc(km);
            __syncwarp();
            if (no >= PAIR_CHUNK) put_chunk(PAIR_CHUNK);
            return;
        }
        if (lane < cnt && m > q0 + r) {
            float4 pm, vm;
            mem_get(M, m, pm, vm);
            const float4 x = S.qa[r];
            const float2 y = S.qb[r];
            const float4 pq = make_float4(x.x, x.y, x.z, 0.f), vq = make_float4(x.w, y.x, y.y, 0.f);
            const int f = pair_test(lm, met, met64, l2p, pq, vq, pm, vm);
            tie += f >> 1;
            if (f & 1) {
                const int root = join_friend(parent, first + q0 + r, first + m, ((volatile int *)S.rq)[r], st);
                if (root != 0x7fffffff) atomicMin(&S.rq[r], root);
            }
        }
        __syncwarp();
    };
    // tests the oldest cnt (at most 32) kept candidates against the queries
    auto test = [&](int cnt) {
        const int m = S.ring[(head + lane) & (LK_RING - 1)];
        unsigned mask = 0;
        if (!brute) {
            uint4 c = make_uint4(0u, 0u, 0u, HALF_FAR);
            if (lane < cnt) {
                float4 pm, vm;
                mem_get(M, m, pm, vm);
                const float4 pc = S.pc, vc = S.vc;
                float s;
                c = half_point(pm, vm, pc, vc, pc.w, vc.w, s);
            }
            S.cand[lane] = c;
            __syncwarp();
            const unsigned *cw = (const unsigned *)S.cand;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const unsigned b = cw[4 * (8 * j + (lane >> 2)) + (lane & 3)];
                float d0[4], d1[4];
                mma_m16n8k8_f16(d0, a[0], a[1], b, cr[0], cr[0], cr[1], cr[1]);
                mma_m16n8k8_f16(d1, a[2], a[3], b, cr[2], cr[2], cr[3], cr[3]);
                // the sign bits, oldest at the top: bit 31 - (8 j + i)
#pragma unroll
                for (int i = 0; i < 4; i++) mask = __funnelshift_l(__float_as_uint(d0[i]), mask, 1);
#pragma unroll
                for (int i = 0; i < 4; i++) mask = __funnelshift_l(__float_as_uint(d1[i]), mask, 1);
            }
            __syncwarp();
        } else {
            for (int e = 0; e < 32; e++) {
                const int row = 16 * ((e >> 2) & 1) + 8 * ((e >> 1) & 1) + (lane >> 2);
                const int col = 8 * (e >> 3) + 2 * (lane & 3) + (e & 1);
                if (((actm >> row) & 1u) && col < cnt) mask |= 0x80000000u >> e;
            }
        }
        for (;;) {
            const unsigned bm = __ballot_sync(FULLW, mask != 0);
            if (!bm) break;
            const int e = mask ? __clz(mask) : 0;
            const int row = 16 * ((e >> 2) & 1) + 8 * ((e >> 1) & 1) + (lane >> 2);
            const int col = 8 * (e >> 3) + 2 * (lane & 3) + (e & 1);
            if (mask) {
                mask &= ~(0x80000000u >> e);
                S.pairs[np + __popc(bm & below)] = (row << 26) | S.ring[(head + col) & (LK_RING - 1)];
            }
            np += __popc(bm);
            __syncwarp();
            if (np >= 32) flush(32);
        }
        head = (head + cnt) & (LK_RING - 1);
        nc -= cnt;
    };
    // whether the child box of this lane of stack entry `ent` has to be
    // searched: it reaches the leaf's own members or later ones, and its box
    // is within reach.  A clique box wholly within l of a query joins it with
    // one union; it is searched only for queries it holds near and far
    // members of.
    auto own_box = [&]() {
        Box6 b;
        b.plo = S.box[0];
        b.phi = S.box[1];
        b.vlo = S.box[2];
        b.vhi = S.box[3];
        return b;
    };
    auto child = [&](int ent) -> bool {
        bool want = false, clique = false;
        Box6 cb = box_empty();
        int c = 0, ch = 0;
        if (ent >= 0) {
            ch = (ent >> 24) - 1;
            c = 32 * (ent & 0xffffff) + lane;
            if (c < V.cnt[ch] && bvh_m0(ch, c + 1) > (int64_t)q0) {
                const int64_t bi = V.off[ch] + c;
                cb = box_get(V.S, bi);
                clique = V.S.cl[bi] != 0;
                want = box_box_d2(own_box(), cb, met) <= lm.lim && !(own_clique && ch == 0 && c == own);
            }
        }
        unsigned cm = __ballot_sync(FULLW, want && clique && !(ch == 0 && c == own));
        while (cm) {
            const int s = __ffs(cm) - 1;
            cm &= cm - 1;
            Box6 b;
            b.plo = shfl4(cb.plo, s);
            b.phi = shfl4(cb.phi, s);
            b.vlo = shfl4(cb.vlo, s);
            b.vhi = shfl4(cb.vhi, s);
            const int m0 = (int)bvh_m0(ch, __shfl_sync(FULLW, c, s));
            const float4 x = S.qa[lane];
            const float2 y = S.qb[lane];
            const float4 po = make_float4(x.x, x.y, x.z, 0.f), vo = make_float4(x.w, y.x, y.y, 0.f);
            const bool near = ((actm >> lane) & 1u) && point_box_d2(po, vo, b, met) <= lm.lim;
            const bool all = near && point_box_far2(po, vo, b, met) <= lm.cl_lim;
            if (all) {
                const int root = join_friend(parent, first + mo, first + m0, S.rq[lane], st);
                if (root != 0x7fffffff) S.rq[lane] = min(S.rq[lane], root);
                // (its members have a neighbour below the bracket already)
                if constexpr (PAIRS)
                    S.best[lane] = min(S.best[lane], __float_as_int(point_box_far2(po, vo, b, met)));
            }
            const bool open = __any_sync(FULLW, near && !all);
            if (lane == s) want = open;
        }
        return want;
    };

    if (lane == 0) S.stack[0] = (V.H - 1) << 24;
    int sp = V.H >= 2 ? 1 : 0, nl = 0;
    if (V.H < 2) {
        if (lane == 0) S.leaf[0] = own;
        nl = 1;
    }
    __syncwarp();
    for (int it = 0; (sp > 0 || nl > 0 || nc > 0) && it < (1 << 24); it++) {
        if (sp > 0 && nl <= LK_LEAVES - 64) {
            const int ea = S.stack[sp - 1];
            const int eb = sp >= 2 ? S.stack[sp - 2] : -1;
            __syncwarp();
            sp -= eb >= 0 ? 2 : 1;
#pragma unroll 1
            for (int u = 0; u < 2; u++) {
                const int ent = u == 0 ? ea : eb;
                if (ent < 0) break;
                const bool want = child(ent);
                const unsigned m = __ballot_sync(FULLW, want);
                const int ch = (ent >> 24) - 1, c = 32 * (ent & 0xffffff) + lane;
                const int slot = __popc(m & below);
                if (ch == 0) {
                    if (want) S.leaf[nl + slot] = c;
                    nl += __popc(m);
                } else {
                    if (sp + __popc(m) > LK_STACK) {
                        if (lane == 0) dev_fail(st, DEV_OVERFLOW, 55, node);
                        return;
                    }
                    if (want) S.stack[sp + slot] = (ch << 24) | c;
                    sp += __popc(m);
                }
            }
            __syncwarp();
            continue;
        }
        // the members of the collected leaves within reach of the own box,
        // two leaves at a time (their loads overlap)
        if (nl > 0) {
            const int m0 = S.leaf[nl - 1] * BVH_LEAF + lane;
            const int m1 = nl >= 2 ? S.leaf[nl - 2] * BVH_LEAF + lane : n;
            nl = max(0, nl - 2);
            float4 p0 = make_float4(INFINITY, 0, 0, 0), u0 = make_float4(0, 0, 0, 0), p1 = p0, u1 = u0;
            if (m0 < n) mem_get(M, m0, p0, u0);
            if (m1 < n) mem_get(M, m1, p1, u1);
            const Box6 bx = own_box();
            const bool k0 = point_box_d2(p0, u0, bx, met) <= lm.lim;
            const bool k1 = point_box_d2(p1, u1, bx, met) <= lm.lim;
            const unsigned b0 = __ballot_sync(FULLW, k0), b1 = __ballot_sync(FULLW, k1);
            if (k0) S.ring[(head + nc + __popc(b0 & below)) & (LK_RING - 1)] = m0;
            nc += __popc(b0);
            if (k1) S.ring[(head + nc + __popc(b1 & below)) & (LK_RING - 1)] = m1;
            nc += __popc(b1);
            __syncwarp();
        }
        const bool last = sp == 0 && nl == 0;
        while (nc >= 32 || (last && nc > 0)) test(min(nc, 32));
    }
    if (np > 0) flush(np);
    if constexpr (PAIRS) {
        if (no > 0) put_chunk(no);
        if (act) atomicMin(reinterpret_cast<int *>(P.dnn) + first + mo, S.best[lane]);
        return;
    }
    tie = warp_sum(tie);
    if (lane == 0 && tie) atomicAdd(&L.tie[k], tie);
}

// the listed pairs at the linking length, a warp a chunk
__global__ void __launch_bounds__(256) k_pair_link(LevelBufs L, NodeArrays nd, MemberStore MS, PairList P, int *parent,
                                                   rs_dev_status *st)
{
    const int lane = lane_id(), gw = (int)((blockIdx.x * 256 + threadIdx.x) >> 5), warps = (int)(gridDim.x * 8);
    const int region = gw & (PAIR_REGIONS - 1), len = min(P.len[region], P.cap);
    for (int c = gw / PAIR_REGIONS; c < len; c += warps / PAIR_REGIONS) {
        const int64_t at = (int64_t)region * P.cap + c;
        const int4 h = P.head[at];
        const int k = h.x;
        if (L.need[k]) continue;
        const float2 lim = L.lim[k];
        const int first = nd.first[L.list[k]];
        int tie = 0;
        for (int i = lane; i < h.z; i += 32) {
            const int2 e = P.pair[at * PAIR_CHUNK + i];
            const float d2 = __int_as_float(e.y);
            if (d2 > lim.y) continue;
            const int q = first + h.y + (e.x >> 26), m = first + (e.x & 0x3ffffff);
            bool link = d2 < lim.x;
            if (!link) {
                float4 pq, vq, pm, vm;
                mem_get(MS, q, pq, vq);
                mem_get(MS, m, pm, vm);
                const double l2 = L.l2[k], l = sqrt(l2), e64 = d2_64(pq, vq, pm, vm, L.met[k]);
                link = e64 <= l2;
                tie += (l2 > 0 && e64 != l2 && fabs(sqrt(e64) - l) <= 1e-6 * l) ? 1 : 0;
            }
            if (link) join_friend(parent, q, m, __ldcg(&parent[q]), st);
        }
        if (__any_sync(FULLW, tie != 0)) {
            tie = warp_sum(tie);
            if (lane == 0) atomicAdd(&L.tie[k], tie);
        }
    }
}

// ---- sampled bracket for the nearest-neighbour search ----
// The exact nearest-neighbour distances of an evenly spread sample of a
// node's members give a radius t_hi that lies above the node's f-quantile
// with overwhelming probability (five binomial standard deviations).  The
// search for every member then starts from t_hi instead of infinity: members
// with a neighbour within t_hi get their exact float32 distance, the others
// stop early with "none within t_hi".  Only values up to the k-th are needed
// for the linking length; if the k-th value is not within t_hi the level
// falls back to the unbounded search, so the result is always exact.
// (nodes that draw a member subset for the linking length are searched without
// one)

// bracket of the search from the sample: the radius R2 is the sample's
// quantile at f + 5 sigma widened by 16 band widths; the stop value is the
// quantile at f - 5 sigma narrowed by 16 band widths (a member with a
// neighbour closer than it is certainly below the linking length)
__global__ void k_smp_thresh(LevelBufs L, NodeArrays nd, const int *smp_at, int bracket_min, const float *sdnn, double f,
                             float *R2, float *STOP)
{
    __shared__ float v[SMP_MAX];
    const int k = blockIdx.x;
    if (k >= L.K) return;
    const int64_t a = (int64_t)smp_at[k] * SMP_UNIT;
    if (a < 0) {  // not sampled: unbounded search, no early stop
        if (threadIdx.x == 0) {
            R2[k] = INFINITY;
            STOP[k] = 0.f;
        }
        return;
    }
    const int S = SMP_UNIT * smp_units(nd.count[L.list[k]], bracket_min);
    for (int i = threadIdx.x; i < S; i += blockDim.x) v[i] = sdnn[a + i];
    __syncthreads();
    for (int kk = 2; kk <= S; kk <<= 1)
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < S / 2; t += blockDim.x) {
                int i = 2 * j * (t / j) + (t % j), l = i + j;
                bool up = (i & kk) == 0;
                float x = v[i], y = v[l];
                if ((x > y) == up) {
                    v[i] = y;
                    v[l] = x;
                }
            }
            __syncthreads();
        }
    if (threadIdx.x == 0) {
        const double sd = 5.0 * sqrt(f * (1.0 - f) / (double)S);
        long long hi = (long long)ceil(fmin(1.0, f + sd) * (double)S) - 1;
        long long lo = (long long)ceil(fmax(0.0, f - sd) * (double)S) - 2;
        hi = hi < 0 ? 0 : (hi >= S ? S - 1 : hi);
        const float th = v[hi];
        R2[k] = isinf(th) ? INFINITY : (float)((double)th * (1.0 + 16.0 * RS_BAND));
        STOP[k] = lo < 0 ? 0.f : (float)((double)v[lo] * (1.0 - 16.0 * RS_BAND));
    }
}

// the level falls back to the full search when the float32 band around a
// node's k-th value is not inside (stop, radius)
// A node whose bracket did not hold gets R2 = -1: the fallback search
// redoes that node only (force_odd, from the injected fault
// RS_FAULT=bracket, fails every node of odd rank that has a bracket).
// need marks the nodes left to the link search: all without a pair search,
// and of those with one the failed ones and those whose list overflowed
// (*again set).
__global__ void k_bracket_check(LevelBufs L, float *R2, const float *STOP, int *fallback, int force_odd, int pairs,
                                const int *smp_at, int *again)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    // the whole float32 band around the k-th value must lie inside the radius,
    // so no member that belongs in the band was cut off by it, and the linking
    // and tie bands (within 5e-6 of t32) between the stop value and the radius,
    // so the pair search joined friends only and listed every pair of the bands
    const float t32 = __uint_as_float(L.sel_prefix[k]);
    const bool bracket = isfinite(R2[k]);
    bool fail = !((double)t32 * (1.0 + 8.0 * RS_BAND) <= (double)R2[k]) ||
                !((double)t32 * (1.0 - 8.0 * RS_BAND) >= (double)STOP[k]);
    if (force_odd && (k & 1) && !isinf(R2[k])) fail = true;
    if (fail) {
        R2[k] = -1.f;
        atomicExch(fallback, 1);
    }
    const bool search = !pairs || !bracket || fail || L.ovf[k];
    L.need[k] = search ? 1 : 0;
    if (search && smp_at[k] >= 0) atomicExch(again, 1);
}

// ---- big-node member order: k-d splits at leaf-aligned medians ----
// A node's member range is split recursively: a range of m > 32 members
// splits at h = m/2 rounded up to a multiple of 32, the h members with the
// smallest coordinate on the round's axis going left, the axes cycling
// through x, vx, y, vy, z, vz.  Every split lands on a leaf boundary, so each
// leaf of 32 consecutive members is one cell of the k-d tree: compact in
// phase space, which is what the leaf boxes of the searches need.  The split
// positions depend only on the node's size, so each round is one stable sort
// of all members by (segment, coordinate), the coordinate of 10 to 16 bits
// relative to the node's reference member in units of its dispersion.
// 16-bit coordinate of a member on an axis (x, vx, y, vy, z, vz), relative to
// the node's reference member in units of its dispersion (.w: one over it)
__device__ __forceinline__ unsigned kd_coord(const float4 *wpos, const float4 *wvel, unsigned slot, int axis,
                                             float4 pref, float4 vref)
{
    const int d = axis >> 1;
    float c, r, inv;
    if ((axis & 1) == 0) {
        const float4 a = wpos[slot];
        c = d == 0 ? a.x : (d == 1 ? a.y : a.z);
        r = d == 0 ? pref.x : (d == 1 ? pref.y : pref.z);
        inv = pref.w;
    } else {
        const float4 a = wvel[slot];
        c = d == 0 ? a.x : (d == 1 ? a.y : a.z);
        r = d == 0 ? vref.x : (d == 1 ? vref.y : vref.z);
        inv = vref.w;
    }
    const float u = ((c - r) * inv + 12.f) * (65536.f / 24.f);
    return (unsigned)fminf(fmaxf(u, 0.f), 65535.f);
}

// One global round over the nodes still being split (a prefix of the level's
// tiles and members): ranges of more than KD_CTA members at this depth are sorted by the
// round's axis; smaller ranges keep their order (value 0).  vcur holds every
// member's slot in the current order.
__global__ void k_kd_keys(LevelBufs L, NodeArrays nd, const int64_t *seg_base, const float4 *wpos, const float4 *wvel,
                          const unsigned *vcur, unsigned long long *kout, unsigned *vout, int round, int drop,
                          int key32, const rs_dev_status *st)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], n = nd.count[node];
    const int p = q0 + threadIdx.x;
    if (p >= n) return;
    const int64_t A = L.seg_off[k] + p;
    const unsigned slot = vcur[A];
    if (dev_is_torn(st)) return;
    int start = 0, size = n;
    for (int i = 0; i < round && size > KD_CTA; i++) {
        const int h = kd_split(size);
        if (p - start < h) {
            size = h;
        } else {
            start += h;
            size -= h;
        }
    }
    unsigned qv = 0;
    if (size > KD_CTA) {
        qv = kd_coord(wpos, wvel, slot, round % 6, L.ref[2 * k], L.ref[2 * k + 1]);
    }
    // Key: (block of KD_CTA members holding the range's start, coordinate).
    // A range still being split has more than KD_CTA members, so it is the
    // only such range whose start lies in its block, and a later range starts
    // in a later block; ranges already final (coordinate 0) that share the
    // block lie before it and keep their places under the stable sort.  So
    // the block number separates what must stay apart, with 5 fewer bits
    // than a leaf number.
    const unsigned long long key = ((unsigned long long)(seg_base[k] + start / KD_CTA) << (16 - drop)) | (qv >> drop);
    if (key32)
        ((unsigned *)kout)[A] = (unsigned)key;
    else
        kout[A] = key;
    if (vout) vout[A] = slot;
}

// the current order before the rounds: every member in its own place
__global__ void k_kd_init(LevelBufs L, NodeArrays nd, unsigned *vcur)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], n = nd.count[node];
    const int p = q0 + threadIdx.x;
    if (p < n) vcur[L.seg_off[k] + p] = (unsigned)(nd.first[node] + p);
}

// Ranges of 33 to KD_CTA members left by the global rounds, one entry per
// range: (rank, start in the node, size, depth).  A thread per 32 members
// descends the splits to its range and lists it if it holds the first ones
// (a thread a node, over all its ranges, took up to 1.5 ms a path of 17M).
__global__ void k_kd_ranges(LevelBufs L, NodeArrays nd, int64_t tiles, int4 *ranges, int *count)
{
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t tile = u / (TQ / 32);
    if (tile >= tiles) return;
    const int k = L.tile_rank[tile], p = L.tile_q0[tile] + 32 * (int)(u % (TQ / 32));
    const int n = nd.count[L.list[k]];
    if (p >= n) return;
    int start = 0, size = n, d = 0;
    for (; size > KD_CTA; d++) {
        const int h = kd_split(size);
        if (p - start < h) {
            size = h;
        } else {
            start += h;
            size -= h;
        }
    }
    if (p == start && size > 32) ranges[atomicAdd(count, 1)] = make_int4(k, start, size, d);
}

// Finish one range in shared memory: the remaining splits.  Round r orders
// every sub-range of more than 32 members (at depth r) along the round's axis,
// which puts its leaf-aligned median split in place, as the global rounds do.
// The members' ranks along each axis the range uses come first, from a
// stable two-pass radix sort of their 16-bit coordinates (ties keep the
// order the range came in); a round then moves member e of sub-range s to s's
// start plus the number of s's members of smaller rank, counted from a
// bitmap of the ranks per sub-range and its prefix popcounts.
constexpr int KDF_ROUNDS = 5;   // kd_rounds(KD_CTA, 32)
constexpr int KDF_SUB = 16;     // sub-ranges ordered in the last round
static_assert(KD_CTA == 8 * 128, "eight warps of 128 positions rank a range");

// stable radix ranking of key[0..m) (16-bit): rk[e] = position of element e
// in the sorted order (8 warps, positions 128 w .. 128 w + 127 per warp)
__device__ __forceinline__ void kdf_rank(int m, const unsigned short *key, unsigned short *rk,
                                         unsigned short (*ord)[KD_CTA], unsigned short (*wcnt)[256],
                                         unsigned *dstart, unsigned *wsum)
{
    const int tid = threadIdx.x, lane = lane_id(), w = warp_id();
    const unsigned lt = (1u << lane) - 1u;
    for (int i = tid; i < m; i += blockDim.x) ord[0][i] = (unsigned short)i;
    int cur = 0;
    for (int sh = 0; sh < 16; sh += 8) {
        for (int i = tid; i < 8 * 256; i += blockDim.x) wcnt[i >> 8][i & 255] = 0;
        __syncthreads();
        unsigned dd[4], rr[4], ee[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int pos = 128 * w + 32 * j + lane;
            const bool ok = pos < m;
            const unsigned e = ok ? ord[cur][pos] : 0u;
            const unsigned d = ok ? ((unsigned)key[e] >> sh) & 255u : 256u;
            const unsigned peers = __match_any_sync(FULLW, d);
            const unsigned before = ok ? wcnt[w][d] : 0u;
            __syncwarp();
            if (ok && (peers & lt) == 0) wcnt[w][d] = (unsigned short)(before + __popc(peers));
            __syncwarp();
            dd[j] = d;
            rr[j] = before + __popc(peers & lt);
            ee[j] = e;
        }
        __syncthreads();
        {
            // thread d: offsets of the warps within digit d, then digit d's start
            const int d = tid;
            unsigned tot = 0;
#pragma unroll
            for (int ww = 0; ww < 8; ww++) {
                const unsigned t = wcnt[ww][d];
                wcnt[ww][d] = (unsigned short)tot;
                tot += t;
            }
            unsigned x = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(FULLW, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) wsum[w] = x;
            __syncthreads();
            unsigned pre = 0;
            for (int ww = 0; ww < w; ww++) pre += wsum[ww];
            dstart[d] = pre + x - tot;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (dd[j] < 256u) ord[cur ^ 1][dstart[dd[j]] + wcnt[w][dd[j]] + rr[j]] = (unsigned short)ee[j];
        __syncthreads();
        cur ^= 1;
    }
    for (int i = tid; i < m; i += blockDim.x) rk[ord[cur][i]] = (unsigned short)i;
    __syncthreads();
}

__global__ void __launch_bounds__(256) k_kd_finish(LevelBufs L, NodeArrays nd, const int4 *ranges, const int *count,
                                                     const float4 *wpos, const float4 *wvel, unsigned *vals,
                                                     const rs_dev_status *st)
{
    if (dev_is_torn(st)) return;
    __shared__ unsigned slot[KD_CTA];
    __shared__ unsigned short rk[KDF_ROUNDS][KD_CTA];
    __shared__ unsigned short key[KD_CTA];
    __shared__ unsigned short pm[2][KD_CTA];  // ranking order, then position -> element
    __shared__ unsigned short wcnt[8][256];
    __shared__ unsigned dstart[256];
    __shared__ unsigned wsum[8];
    __shared__ unsigned bm[KDF_SUB][32];
    __shared__ unsigned short pre[KDF_SUB][32];
    const int tid = threadIdx.x, lane = lane_id(), w = warp_id();
    const int nr = *count;
    for (int ri = blockIdx.x; ri < nr; ri += gridDim.x) {
        const int4 rg = ranges[ri];
        const int k = rg.x, s0 = rg.y, m = rg.z, d0 = rg.w;
        const int64_t P0 = L.seg_off[k] + s0;
        const float4 pref = L.ref[2 * k], vref = L.ref[2 * k + 1];
        const int R = kd_rounds(m, 32);
        for (int i = tid; i < m; i += blockDim.x) slot[i] = vals[P0 + i];
        __syncthreads();
        for (int r = 0; r < R; r++) {
            const int axis = (d0 + r) % 6;
            for (int i = tid; i < m; i += blockDim.x)
                key[i] = (unsigned short)kd_coord(wpos, wvel, slot[i], axis, pref, vref);
            __syncthreads();
            kdf_rank(m, key, rk[r], pm, wcnt, dstart, wsum);
        }
        int cur = 0;
        for (int i = tid; i < m; i += blockDim.x) pm[0][i] = (unsigned short)i;
        for (int r = 0; r < R; r++) {
            for (int i = tid; i < KDF_SUB * 32; i += blockDim.x) bm[i >> 5][i & 31] = 0u;
            __syncthreads();
            for (int j = tid; j < m; j += blockDim.x) {
                int start = 0, size = m, sub = 0;
                for (int i = 0; i < r && size > 32; i++) {
                    const int h = kd_split(size);
                    const int hi = j - start >= h ? 1 : 0;
                    start = hi ? start + h : start;
                    size = hi ? size - h : h;
                    sub = 2 * sub + hi;
                }
                if (size > 32) {
                    const unsigned q = rk[r][pm[cur][j]];
                    atomicOr(&bm[sub][q >> 5], 1u << (q & 31));
                }
            }
            __syncthreads();
            for (int sb = w; sb < (1 << r); sb += 8) {
                const unsigned c = __popc(bm[sb][lane]);
                unsigned x = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(FULLW, x, o);
                    if (lane >= o) x += y;
                }
                pre[sb][lane] = (unsigned short)(x - c);
            }
            __syncthreads();
            for (int j = tid; j < m; j += blockDim.x) {
                int start = 0, size = m, sub = 0;
                for (int i = 0; i < r && size > 32; i++) {
                    const int h = kd_split(size);
                    const int hi = j - start >= h ? 1 : 0;
                    start = hi ? start + h : start;
                    size = hi ? size - h : h;
                    sub = 2 * sub + hi;
                }
                const unsigned short e = pm[cur][j];
                int np = j;
                if (size > 32) {
                    const unsigned q = rk[r][e];
                    np = start + pre[sub][q >> 5] + __popc(bm[sub][q >> 5] & ((1u << (q & 31)) - 1u));
                }
                pm[cur ^ 1][np] = e;
            }
            __syncthreads();
            cur ^= 1;
        }
        for (int j = tid; j < m; j += blockDim.x) vals[P0 + j] = slot[pm[cur][j]];
        __syncthreads();
    }
}

// members into the sorted order of their node's range
__global__ void k_kd_place(LevelBufs L, NodeArrays nd, const unsigned *vals, const float4 *wpos, const float4 *wvel,
                           const int *widx, float4 *wpos2, float4 *wvel2, int *widx2, unsigned *dest,
                           const rs_dev_status *st)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int p = q0 + threadIdx.x;
    if (p >= n) return;
    const int64_t P = L.seg_off[k] + p;
    const unsigned s = vals[P];
    if (dev_is_torn(st)) return;
    const int dd = first + p;
    wpos2[dd] = wpos[s];
    wvel2[dd] = wvel[s];
    widx2[dd] = widx[s];
    dest[P] = (unsigned)dd;
}

// radix select: pass 0 digits bits 31..21, pass 1 bits 20..10, pass 2 bits 9..0
__device__ __forceinline__ void sel_digit(unsigned bits, int pass, unsigned &digit, unsigned &prefix_mask)
{
    if (pass == 0) {
        digit = bits >> 21;
        prefix_mask = 0;
    } else if (pass == 1) {
        digit = (bits >> 10) & 2047u;
        prefix_mask = 0xffe00000u;
    } else {
        digit = bits & 1023u;
        prefix_mask = 0xfffffc00u;
    }
}

// ---- random member subsets for the linking length (Sec. 3.2) ----
// Above sub_n members a node takes its linking length from the nearest-
// neighbour distances of sub_n randomly drawn members (their neighbours are
// still searched among all members).  Each particle carries a 64-bit key from
// the SplitMix64 generator (Steele, Lea & Flood 2014) used counter-based:
// particle i gets the finaliser of seed + (i+1)*gamma.  The finaliser is a
// bijection, so keys are distinct and the subset -- the sub_n members with
// the smallest keys -- is well defined; it is found by a radix select on the
// key's high word, then on its low word among the members that tie on the
// high word.  Members outside the subset get a nearest-neighbour value of -1,
// which the select skips and the link treats as "may have a friend".
__device__ __forceinline__ unsigned long long subset_key(unsigned long long seed, int i)
{
    unsigned long long z = seed + (unsigned long long)(i + 1) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

__global__ void k_sub_init(LevelBufs L, NodeArrays nd, int sub_n)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    const int n = nd.count[L.list[k]];
    L.sel_krem[k] = n > sub_n ? sub_n : 1;
    L.sel_prefix[k] = 0u;
    L.sub_cnt[k] = 0;
}

// one radix-select pass over the keys of the members of nodes above sub_n:
// stage 0 selects on the high word, stage 1 on the low word of the members
// whose high word equals the stage-0 result
__global__ void __launch_bounds__(TQ) k_sub_hist(LevelBufs L, NodeArrays nd, const int *widx,
                                                 unsigned long long seed, int sub_n, int stage, int pass)
{
    __shared__ unsigned h[2048];
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    if (n <= sub_n) return;  // the whole tile belongs to one node
    for (int i = threadIdx.x; i < 2048; i += TQ) h[i] = 0;
    __syncthreads();
    const int q = q0 + threadIdx.x;
    if (q < n) {
        const unsigned long long key = subset_key(seed, widx[first + q]);
        const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
        if (stage == 0 || hi == L.sub_t[2 * k]) {
            const unsigned bits = stage == 0 ? hi : lo;
            unsigned digit, mask;
            sel_digit(bits, pass, digit, mask);
            if ((bits & mask) == (L.sel_prefix[k] & mask)) atomicAdd(&h[digit], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2048; i += TQ)
        if (h[i]) atomicAdd(&L.hist[(int64_t)k * 2048 + i], h[i]);
}

// stores a stage's selected word; the rank still to select carries over
__global__ void k_sub_stage(LevelBufs L, int stage)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    L.sub_t[2 * k + stage] = L.sel_prefix[k];
    L.sel_prefix[k] = 0u;
}

// members of the subset go to the query list (rank, member); the others get
// the "outside the subset" value
__global__ void __launch_bounds__(TQ) k_sub_mark(LevelBufs L, NodeArrays nd, const int *widx,
                                                 unsigned long long seed, int sub_n, float *dnn, int2 *qlist,
                                                 int *qlen, int cap, rs_dev_status *st)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    if (n <= sub_n) return;
    const int q = q0 + threadIdx.x;
    bool in = false;
    if (q < n) {
        const unsigned long long key = subset_key(seed, widx[first + q]);
        const unsigned long long t = ((unsigned long long)L.sub_t[2 * k] << 32) | L.sub_t[2 * k + 1];
        in = key <= t;
        if (!in) dnn[first + q] = -1.0f;
    }
    const unsigned m = __ballot_sync(FULLW, in);
    if (!m) return;
    const int lane = lane_id();
    int base = 0;
    if (lane == __ffs(m) - 1) {
        base = atomicAdd(qlen, __popc(m));
        atomicAdd(&L.sub_cnt[k], __popc(m));
    }
    base = __shfl_sync(FULLW, base, __ffs(m) - 1);
    if (in) {
        const int pos = base + __popc(m & ((1u << lane) - 1u));
        if (pos < cap)
            qlist[pos] = make_int2(k, q);
        else
            dev_fail(st, DEV_OVERFLOW, 58, node);
    }
}

// every node above sub_n drew exactly sub_n members (keys are distinct)
__global__ void k_sub_check(LevelBufs L, NodeArrays nd, int sub_n, rs_dev_status *st)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    const int node = L.list[k], n = nd.count[node];
    if (n > sub_n && L.sub_cnt[k] != sub_n) dev_fail(st, DEV_INTERNAL, 59, node);
}

// number of members whose nearest-neighbour distance sets a node's linking
// length: all of them, or the subset's size above it
__device__ __forceinline__ int n_select(int n, int sub_n) { return (sub_n > 0 && n > sub_n) ? sub_n : n; }

__global__ void k_lvl_initk(LevelBufs L, NodeArrays nd, double f, int sub_n)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    const int n = n_select(nd.count[L.list[k]], sub_n);
    long long kk = (long long)ceil(f * (double)n);
    if (kk < 1) kk = 1;
    if (kk > n) kk = n;
    L.sel_krem[k] = (int)kk;
    L.sel_prefix[k] = 0u;
}

__global__ void __launch_bounds__(TQ) k_lvl_hist(LevelBufs L, NodeArrays nd, const float *dnn, int pass)
{
    __shared__ unsigned h[2048];
    for (int i = threadIdx.x; i < 2048; i += TQ) h[i] = 0;
    __syncthreads();
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int q = q0 + threadIdx.x;
    if (q < n) {
        // a negative value marks a member outside the node's subset
        unsigned bits = __float_as_uint(dnn[first + q]), digit, mask;
        sel_digit(bits, pass, digit, mask);
        if (!(bits >> 31) && (bits & mask) == (L.sel_prefix[k] & mask)) atomicAdd(&h[digit], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2048; i += TQ)
        if (h[i]) atomicAdd(&L.hist[(int64_t)k * 2048 + i], h[i]);
}

// the digit that holds the rank still to select, eight bins a thread (one
// thread over the 2048 bins took 75 us, three times a level); the bins are
// cleared for the next pass
__global__ void __launch_bounds__(256) k_lvl_pick(LevelBufs L, int pass)
{
    const int k = blockIdx.x;
    uint4 *h = reinterpret_cast<uint4 *>(L.hist + (int64_t)k * 2048) + 2 * threadIdx.x;
    const uint4 a = h[0], b = h[1];
    h[0] = h[1] = make_uint4(0u, 0u, 0u, 0u);
    const unsigned c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const unsigned sum = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
    unsigned all;
    unsigned acc = rs_block_scan<256>(sum, all);
    const unsigned krem = (unsigned)L.sel_krem[k];
    const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
    __syncthreads();
    if (krem > all) {  // (fewer values than the rank: the last bin)
        if (threadIdx.x == 0) {
            L.sel_prefix[k] |= (pass == 2 ? 1023u : 2047u) << shift;
            L.sel_krem[k] = (int)(krem - all);
        }
        return;
    }
    if (!(acc < krem && krem <= acc + sum)) return;
    int d = 0;
    while (acc + c[d] < krem) acc += c[d++];
    L.sel_prefix[k] |= (unsigned)(8 * threadIdx.x + d) << shift;
    L.sel_krem[k] = (int)(krem - acc);
}

__global__ void __launch_bounds__(TQ) k_lvl_band(LevelBufs L, NodeArrays nd, const float *dnn)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int q = q0 + threadIdx.x;
    const float t32 = __uint_as_float(L.sel_prefix[k]);
    // t32 (1 -+ 2 RS_BAND), rounded once: 2 RS_BAND = 2^-19
    const float blo = fmaf(t32, (float)(-2.0 * RS_BAND), t32), bhi = fmaf(t32, (float)(2.0 * RS_BAND), t32);
    const float d = q < n ? dnn[first + q] : -1.f;  // (negative: outside the subset)
    const bool in = !(__float_as_uint(d) >> 31);
    const unsigned below = __ballot_sync(FULLW, in && d < blo);
    if (below && lane_id() == 0) atomicAdd(&L.below[k], __popc(below));
    if (in && d >= blo && d <= bhi) {
        int b = atomicAdd(L.band_len, 1);
        L.band_rank[b] = k;
        L.band_slot[b] = first + q;
    }
}

// Exact float64 nearest-neighbour distance of a band member: the minimum
// float64 distance over the members whose float32 distance is within `lim`
// (a bound above the member's float32 value), one warp per band member over
// the node's hierarchy.  A box is skipped only when its float32 bound exceeds
// lim by the pruning slack, so every member that passes the float32 test is
// evaluated.
__global__ void __launch_bounds__(W_WARPS * 32) k_lvl_band_exact(LevelBufs L, NodeArrays nd, const int64_t *box_base,
                                                                 BoxStore B, MemberStore MS, const float *dnn,
                                                                 rs_dev_status *st)
{
    __shared__ int si_s[W_WARPS][W_STACK];
    __shared__ int lv_s[W_WARPS][2 * BVH_MAXH];
    const int w = warp_id(), lane = lane_id();
    const int b = blockIdx.x * W_WARPS + w;
    if (b >= *L.band_len) return;
    const int k = L.band_rank[b], s = L.band_slot[b];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const Metric6 met = L.met[k];
    const MemberStore M = mem_shift(MS, first);
    const int q = s - first;
    float4 pq, vq;
    mem_get(M, q, pq, vq);
    const float lim = dnn[s] * (float)(1.0 + 2.0 * RS_BAND);
    BvhView V;
    bvh_view(V, B, box_base[k], n, lv_s[w]);
    const int own = q / BVH_LEAF;
    double best = INFINITY;
    {
        const int m = own * BVH_LEAF + lane;
        if (m < n && m != q) {
            float4 pc, vc;
            mem_get(M, m, pc, vc);
            if (d2_32(pq, vq, pc, vc, met) <= lim) best = fmin(best, d2_64(pq, vq, pc, vc, met));
        }
    }
    int *si = si_s[w];
    if (V.H >= 2) {
        if (lane == 0) si[0] = (V.H - 1) << 24;
        int sp = 1;
        __syncwarp();
        for (int it = 0; sp > 0 && it < (1 << 24); it++) {
            sp--;
            const int ent = si[sp];
            __syncwarp();
            const int ch = (ent >> 24) - 1, c = 32 * (ent & 0xffffff) + lane;
            const bool ok = c < V.cnt[ch] && !(ch == 0 && c == own) &&
                            point_box_d2(pq, vq, box_get(V.S, V.off[ch] + c), met) <= lim * RS_PRUNE_SLACK;
            unsigned mask = __ballot_sync(FULLW, ok);
            if (ch == 0) {
                while (mask) {
                    const int src = __ffs(mask) - 1;
                    mask &= mask - 1;
                    const int m = (32 * (ent & 0xffffff) + src) * BVH_LEAF + lane;
                    if (m < n && m != q) {
                        float4 pc, vc;
                        mem_get(M, m, pc, vc);
                        if (d2_32(pq, vq, pc, vc, met) <= lim) best = fmin(best, d2_64(pq, vq, pc, vc, met));
                    }
                }
                continue;
            }
            if (sp + __popc(mask) > W_STACK) {
                if (lane == 0) dev_fail(st, DEV_OVERFLOW, 57, node);
                break;
            }
            if (ok) si[sp + __popc(mask & ((1u << lane) - 1u))] = (ch << 24) | c;
            sp += __popc(mask);
            __syncwarp();
        }
    }
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(FULLW, best, o));
    if (lane == 0) L.band_val[b] = best;
}

__global__ void k_lvl_l2(LevelBufs L, NodeArrays nd, double f, int sub_n, rs_dev_status *st)
{
    const int k = blockIdx.x;
    const int node = L.list[k];
    const int n = n_select(nd.count[node], sub_n);
    long long kk = (long long)ceil(f * (double)n);
    if (kk < 1) kk = 1;
    if (kk > n) kk = n;
    const int want = (int)(kk - 1) - L.below[k];
    const int nb = *L.band_len;
    bool found = false;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        if (L.band_rank[b] != k) continue;
        const double v = L.band_val[b];
        int r = 0;
        for (int c = 0; c < nb; c++)
            if (L.band_rank[c] == k && (L.band_val[c] < v || (L.band_val[c] == v && c < b))) r++;
        if (r == want) {
            L.l2[k] = v;
            found = true;
        }
    }
    found = __syncthreads_or(found);
    if (threadIdx.x == 0) {
        if (!found) dev_fail(st, DEV_INTERNAL, 50, node);
        const double l2 = L.l2[k];
        nd.lnk[node] = l2;  // k_tree_stats makes it a length
        L.lim[k] = make_float2(fminf((float)(l2 * (1.0 - RS_BAND)), (float)(l2 * (1.0 - 3e-6))), link_part(l2));
    }
}

__global__ void k_lvl_comp(LevelBufs L, NodeArrays nd, const int *widx, int *parent, int *csize, int *cmin,
                           rs_dev_status *st)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int q = q0 + threadIdx.x;
    const bool ok = q < n;
    const int r = ok ? uf_find(parent, first + q, st) : -1;
    const int mi = ok ? widx[first + q] : 0x7fffffff;
    // lanes of one component add once (consecutive members mostly share a root)
    const unsigned grp = __match_any_sync(0xffffffffu, r);
    const int lead = __ffs(grp) - 1;
    const int gm = (int)__reduce_min_sync(grp, (unsigned)mi);
    if (ok && lane_id() == lead) {
        atomicAdd(&csize[r], __popc(grp));
        atomicMin(&cmin[r], gm);
    }
}

// keys of the child partition: (rank, smallest particle index of the child),
// all ones in the lower cbits for the members outside children.  cbits are what
// a particle index takes, so the sort skips the passes of a 32-bit field's
// empty digits (9.6M grouped members, 6 levels: 34 -> 28 passes, 1.42 -> 1.19 ms)
__global__ void k_lvl_keys(LevelBufs L, NodeArrays nd, int *parent, const int *csize, const int *cmin,
                           unsigned long long *keys, unsigned *vals, int min_n, int cbits, rs_dev_status *st)
{
    const int k = L.tile_rank[blockIdx.x], q0 = L.tile_q0[blockIdx.x];
    const int node = L.list[k], first = nd.first[node], n = nd.count[node];
    const int q = q0 + threadIdx.x;
    if (q >= n) return;
    int r = uf_find(parent, first + q, st);
    int sz = csize[r];
    const unsigned long long comp = (sz >= min_n && sz < n) ? (unsigned)cmin[r] : (1ull << cbits) - 1ull;
    const int64_t p = L.seg_off[k] + q;
    keys[p] = ((unsigned long long)k << cbits) | comp;
    vals[p] = (unsigned)(first + q);
}

__global__ void k_lvl_scatter(LevelBufs L, NodeArrays nd, int64_t LM, const unsigned long long *keys,
                              const unsigned *vals, const float4 *wpos, const float4 *wvel, const int *widx,
                              float4 *wpos2, float4 *wvel2, int *widx2, unsigned *dest, int rank_shift,
                              const rs_dev_status *st)
{
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= LM) return;
    const int k = (int)(keys[p] >> rank_shift);
    if (dev_is_torn(st)) return;
    const int node = L.list[k];
    const int d = nd.first[node] + (int)(p - L.seg_off[k]);
    const unsigned s = vals[p];
    wpos2[d] = wpos[s];
    wvel2[d] = wvel[s];
    widx2[d] = widx[s];
    dest[p] = (unsigned)d;
}

__global__ void k_lvl_copyback(int64_t LM, const unsigned *dest, const float4 *wpos2, const float4 *wvel2,
                               const int *widx2, float4 *wpos, float4 *wvel, int *widx, const rs_dev_status *st)
{
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= LM) return;
    const unsigned d = dest[p];
    if (dev_is_torn(st)) return;
    wpos[d] = wpos2[d];
    wvel[d] = wvel2[d];
    widx[d] = widx2[d];
}

__global__ void k_lvl_children(LevelBufs L, NodeArrays nd, int64_t LM, const unsigned long long *keys,
                               const unsigned *vals, int *parent, const int *csize, int *next_list, int *next_len,
                               int *small_list, int *small_len, int cbits, rs_dev_status *st)
{
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= LM) return;
    const unsigned long long key = keys[p];
    const unsigned long long rest = (1ull << cbits) - 1ull, comp = key & rest;
    if (comp == rest) return;
    if ((p > 0 && keys[p - 1] == key) || dev_is_torn(st)) return;
    const int k = (int)(key >> cbits);
    const int node = L.list[k];
    const int r = uf_find(parent, (int)vals[p], st);
    const int sz = csize[r];
    int id = atomicAdd(nd.counter, 1);
    if (id >= nd.cap) {
        dev_fail(st, DEV_OVERFLOW, 51, id);
        return;
    }
    nd.parent[id] = node;
    nd.level[id] = nd.level[node] + 1;
    nd.first[id] = nd.first[node] + (int)(p - L.seg_off[k]);
    nd.count[id] = sz;
    nd.minidx[id] = (int)comp;
    nd.nchild[id] = 0;
    nd.tie[id] = 0;
    nd.root[id] = nd.root[node];
    nd.shift[id] = nd.shift[node];
    atomicAdd(&nd.nchild[node], 1);
    if (sz > SMALL_N) next_list[atomicAdd(next_len, 1)] = id;
    else small_list[atomicAdd(small_len, 1)] = id;
}

__global__ void k_lvl_store_tie(LevelBufs L, NodeArrays nd)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L.K) return;
    nd.tie[L.list[k]] = L.tie[k];
}

__global__ void k_tree_stats(NodeArrays nd, unsigned long long *out)
{
    // out: [0] nodes, [1] seeds, [2] tie sum, [3] max level, [4] sum of counts
    const int n_nodes = min(*nd.counter, nd.cap);
    if (blockIdx.x == 0 && threadIdx.x == 0) out[0] = (unsigned long long)*nd.counter;
    unsigned long long seeds = 0, tie = 0, sum = 0;
    int maxl = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += gridDim.x * blockDim.x) {
        seeds += nd.nchild[i] == 0;
        tie += (unsigned long long)nd.tie[i];
        sum += (unsigned long long)nd.count[i];
        maxl = max(maxl, nd.level[i]);
        // the node's linking length in units of Eq. 1, from the square in its
        // scaled metric (here, 32 nodes a float64 instruction, and not in the
        // node's own block)
        nd.lnk[i] = sqrt(nd.lnk[i] / metric_of(nd.sigx[i], nd.sigv[i]).scale);
    }
    seeds = warp_sum(seeds);
    tie = warp_sum(tie);
    sum = warp_sum(sum);
    maxl = warp_max(maxl);
    if (lane_id() == 0) {
        atomicAdd(&out[1], seeds);
        atomicAdd(&out[2], tie);
        atomicMax(&out[3], (unsigned long long)maxl);
        atomicAdd(&out[4], sum);
    }
}

template <typename T>
T *carve(char *&p, int64_t count)
{
    T *r = (T *)p;
    size_t b = sizeof(T) * (size_t)(count > 0 ? count : 1);
    p += (b + 255) / 256 * 256;
    return r;
}

size_t tree_bytes(int64_t M, int64_t cap)
{
    size_t s = 0;
    auto add = [&](size_t b) { s += (b + 255) / 256 * 256; };
    for (int i = 0; i < 9; i++) add(sizeof(int) * cap);
    add(sizeof(double) * cap * 3);  // lnk, sigx, sigv
    add(sizeof(double) * cap * 3);
    add(sizeof(double) * cap * 3);
    add(sizeof(double) * cap * 3);
    add(sizeof(double) * cap * 3);
    add(sizeof(int) * 4);
    add(sizeof(int) * (M > 0 ? M : 1));
    return s + 4096;
}

}  // namespace

// the big-node nearest-neighbour search, compiled for 40, 48 or 56 resident
// warps per SM (rs_tuning::nn_blocks_per_sm = 5, 6 or 7, in units of eight)
static rs_status launch_nn(rs_ctx *ctx, const char *name, int64_t T, const LevelBufs &L, const NodeArrays &nd,
                           const int64_t *bo, const BoxStore &boxes, const MemberStore &ms, const float *R2,
                           const float *STOP, int redo_failed, int sub_n, int pairs, float *dnn)
{
    const int64_t g = T * (TQ / 32) / NN_WARPS;
    switch (ctx->tune.nn_blocks_per_sm) {
    case 5:
        RS_LAUNCH(ctx, name, k_bvh_nn<5>, g, NN_WARPS * 32, 0, L, nd, bo, boxes, ms, R2, STOP, redo_failed, sub_n,
                  pairs, dnn, ctx->d_status);
        break;
    case 7:
        RS_LAUNCH(ctx, name, k_bvh_nn<7>, g, NN_WARPS * 32, 0, L, nd, bo, boxes, ms, R2, STOP, redo_failed, sub_n,
                  pairs, dnn, ctx->d_status);
        break;
    default:
        RS_LAUNCH(ctx, name, k_bvh_nn<6>, g, NN_WARPS * 32, 0, L, nd, bo, boxes, ms, R2, STOP, redo_failed, sub_n,
                  pairs, dnn, ctx->d_status);
    }
    return RS_OK;
}

// the pair or the link search over tiles [t0, T): one warp per leaf, LK_WARPS
// to a block, compiled for 24, 32 or 40 resident warps per SM
// (rs_tuning::link_blocks_per_sm = 4, 5 or 6)
template <bool PAIRS>
static rs_status launch_link(rs_ctx *ctx, const char *name, int64_t t0, int64_t T, const LevelBufs &L,
                             const NodeArrays &nd, const int64_t *bo, const BoxStore &boxes, const MemberStore &ms,
                             int *uf, const PairList &pl)
{
    auto k24 = k_bvh_link<24, PAIRS>;
    auto k32 = k_bvh_link<32, PAIRS>;
    auto k40 = k_bvh_link<40, PAIRS>;
    auto k = ctx->tune.link_blocks_per_sm == 4 ? k24 : (ctx->tune.link_blocks_per_sm == 6 ? k40 : k32);
    RS_LAUNCH(ctx, name, k, (T - t0) * (TQ / 32) / LK_WARPS, LK_WARPS * 32, 0, L, nd, t0, bo, boxes, ms, uf, pl,
              ctx->d_status);
    return RS_OK;
}

// ---------------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------------
static rs_status refine_impl(rs_ctx *ctx, const float *pos, const float *vel, int32_t stride, int64_t n, double box,
                             const int32_t *perm, const int64_t *goff, int64_t G, int64_t M, double f, int32_t min_n,
                             int64_t sub_n, uint64_t sub_seed, int64_t node_cap, rs_tree **out)
{
    rs_tree *t = new (std::nothrow) rs_tree();
    if (!t) return RS_ERR_OOM;
    t->n_total = n;
    t->n_members = M;
    t->box = box;
    const int64_t cap = node_cap;
    cudaError_t e = rs_block_alloc(ctx, &t->block, &t->pool, tree_bytes(M, cap));
    if (e != cudaSuccess) {
        delete t;
        cudaGetLastError();
        return rs_fail(ctx, RS_ERR_OOM, "rs_refine6d: tree allocation failed");
    }
    char *p = (char *)t->block;
    NodeArrays &nd = t->nd;
    nd.parent = carve<int>(p, cap);
    nd.level = carve<int>(p, cap);
    nd.first = carve<int>(p, cap);
    nd.count = carve<int>(p, cap);
    nd.minidx = carve<int>(p, cap);
    nd.nchild = carve<int>(p, cap);
    nd.tie = carve<int>(p, cap);
    nd.root = carve<int>(p, cap);
    nd.shift = carve<int>(p, cap);
    nd.lnk = carve<double>(p, cap);
    nd.sigx = carve<double>(p, cap);
    nd.sigv = carve<double>(p, cap);
    nd.xbar = carve<double>(p, 3 * cap);
    nd.vbar = carve<double>(p, 3 * cap);
    nd.counter = carve<int>(p, 4);
    nd.cap = (int)cap;
    t->members = carve<int>(p, M);
    *out = t;

    const float boxf = (float)box;
    RS_CUDA(ctx, cudaMemsetAsync(nd.counter, 0, sizeof(int) * 4, ctx->stream));
    if (M == 0 || G == 0) return RS_OK;

    // working member arrays
    RS_WS(ctx, float4, wpos, WS_RF_POS, M);
    RS_WS(ctx, float4, wvel, WS_RF_VEL, M);
    RS_WS(ctx, float4, wpos2, WS_RF_POS2, M);
    RS_WS(ctx, float4, wvel2, WS_RF_VEL2, M);
    RS_WS(ctx, int, widx2, WS_RF_IDX2, M);
    RS_WS(ctx, float, dnn, WS_RF_DNN, M);
    RS_WS(ctx, int, uf, WS_RF_PARENT, 3 * M);
    int *csize = uf + M, *cmin = uf + 2 * M;
    int *widx = t->members;
    RS_WS(ctx, int, gmisc, WS_RF_MISC0, 14 * G + 2 * M + 8);
    int *shift_bits = gmisc, *gmin = gmisc + G, *slot_group = gmisc + 2 * G, *gred = gmisc + 2 * G + M;
    // node queues: big lists (ping-pong) and the small queue; counters
    // counters first (16 ints = 64 bytes, so everything after stays 8-byte aligned)
    RS_WS(ctx, int, q, WS_RF_NODEQ, 7 * cap + 16);
    int *ctr = q, *big_a = q + 16, *big_b = q + 16 + cap, *small_q = q + 16 + 2 * cap, *tiny_q = q + 16 + 3 * cap,
        *mid_q = q + 16 + 4 * cap, *warp_q = q + 16 + 5 * cap, *big_s = q + 16 + 6 * cap;
    // ctr: [0] big_a len, [1] big_b len, [2] small len, [3] small head, [4] band len,
    // [6] pair-search nodes to link again, [7] bracket fallback flag, [8] tiny len, [9] tiny head, [10] k-d ranges,
    // [11] middle len, [12] middle head, [13] subset query list length,
    // [14] warp-tier len, [15] warp-tier head
    RS_CUDA(ctx, cudaMemsetAsync(ctr, 0, sizeof(int) * 16, ctx->stream));

    RS_WS(ctx, SizeTab, size_tab, WS_RF_SIZES, SMALL_N + 1);
    RS_LAUNCH(ctx, "rf_init", k_refine_init, ceil_div(std::max<int64_t>(12 * G, SMALL_N + 1), 256), 256, 0, G, gred,
              gmin, SMALL_N, f, size_tab);
    RS_LAUNCH(ctx, "rf_group_unwrap", k_unwrap_tiles, ceil_div(M, 256), 256, 0, G, goff, perm, n, M, pos, stride,
              boxf, slot_group, gred, gmin, wpos, widx, ctx->d_status);
    RS_LAUNCH(ctx, "rf_unwrap_bits", k_unwrap_bits, ceil_div(G, 256), 256, 0, G, (const int *)gred, boxf, shift_bits,
              ctx->d_status);
    RS_LAUNCH(ctx, "rf_gather", k_gather, ceil_div(M, 256), 256, 0, M, vel, stride, boxf, (const int *)slot_group,
              (const int *)shift_bits, wpos, wvel, (const int *)widx);
    RS_LAUNCH(ctx, "rf_roots", k_make_roots, ceil_div(G, 256), 256, 0, G, goff, (const int *)gmin,
              (const int *)shift_bits, (int)min_n, nd,
              big_a, ctr + 0, small_q, ctr + 2, ctx->d_status);

    // ---- big levels ----
    int *cur = big_a, *nxt = big_b;
    int *cur_len = ctr + 0, *nxt_len = ctr + 1;
    int64_t sum_level = 0;
    int n_fallback_levels = 0;
    // per-rank offsets: a big node has more than SMALL_N members
    const int64_t kcap = M / SMALL_N + 2;
    RS_WS(ctx, int64_t, lv64, WS_RF_MISC1, 7 * kcap + LT_WORDS + 8);
    LevelOff O;
    O.tile = lv64;
    O.seg = lv64 + kcap;
    O.box = lv64 + 2 * kcap;
    O.block = lv64 + 3 * kcap;
    O.smp = (int *)(lv64 + 4 * kcap);
    O.smp_at = O.smp + (SMP_MAX / SMP_UNIT) * kcap;
    int64_t *dtot = lv64 + 7 * kcap;
    for (int level = 0; level < 4096; level++) {
        RS_LAUNCH(ctx, "rf_lvl_setup", k_lvl_setup, 1, 1024, 0, (const int *)cur, (const int *)cur_len, big_s, nd, O,
                  (int)sub_n, (int)ctx->tune.bracket_min, dtot);
        int64_t tot[LT_WORDS];
        static_assert(LT_WORDS <= 64, "the context's host scratch");
        RS_TRY(rs_read_i64(ctx, dtot, LT_WORDS, tot, "rs_refine6d"));
        const int64_t K = tot[LT_K], T = tot[LT_T], LM = tot[LT_LM], NBX = tot[LT_NBX];
        if (K == 0) break;
        sum_level += LM;
        RS_WS(ctx, int, tl, WS_RF_MISC2, 2 * T + 8);
        LevelBufs L;
        L.list = big_s;
        L.K = (int)K;
        L.tile_rank = tl;
        L.tile_q0 = tl + T;
        L.seg_off = O.seg;
        const int64_t *bo = O.box;
        RS_LAUNCH(ctx, "rf_lvl_tiles", k_lvl_tiles, K, 256, 0, (int)K, (const int64_t *)O.tile, tl, tl + T);
        // per-rank state
        size_t per = sizeof(MomAcc) + sizeof(Metric6) + 2 * sizeof(float4) + 2048 * sizeof(unsigned) +
                     11 * sizeof(int) + sizeof(double) + 64;
        RS_WS(ctx, char, rk, WS_RF_ACC, (int64_t)(per * K + 4096));
        char *rp = rk;
        L.acc = carve<MomAcc>(rp, K);
        L.met = carve<Metric6>(rp, K);
        L.ref = carve<float4>(rp, 2 * K);
        L.l2 = carve<double>(rp, K);
        L.hist = carve<unsigned>(rp, 2048 * K);
        L.sel_prefix = carve<unsigned>(rp, K);
        L.sel_krem = carve<int>(rp, K);
        L.below = carve<int>(rp, K);
        L.tie = carve<int>(rp, K);
        L.sub_t = carve<unsigned>(rp, 2 * K);
        L.sub_cnt = carve<int>(rp, K);
        L.lim = carve<float2>(rp, K);
        L.need = carve<int>(rp, K);
        L.ovf = carve<int>(rp, K);
        RS_CUDA(ctx, cudaMemsetAsync(rk, 0, (size_t)(rp - rk), ctx->stream));
        RS_WS(ctx, char, bandbuf, WS_RF_BAND, (int64_t)(LM * 16 + 64));
        char *bp = bandbuf;
        L.band_len = ctr + 4;
        L.band_rank = carve<int>(bp, LM);
        L.band_slot = carve<int>(bp, LM);
        L.band_val = carve<double>(bp, LM);
        RS_CUDA(ctx, cudaMemsetAsync(ctr + 4, 0, sizeof(int), ctx->stream));

        RS_LAUNCH(ctx, "rf_lvl_moments", k_lvl_moments, T, TQ, 0, L, nd, (const float4 *)wpos, (const float4 *)wvel);
        RS_LAUNCH(ctx, "rf_lvl_finalize", k_lvl_finalize, ceil_div(K, 128), 128, 0, L, nd, box);
        RS_WS(ctx, uint64_t, k0, WS_SORT_K0, LM);
        RS_WS(ctx, uint64_t, k1, WS_SORT_K1, LM);
        RS_WS(ctx, uint32_t, v0, WS_SORT_V0, LM);
        RS_WS(ctx, uint32_t, v1, WS_SORT_V1, LM);
        // bits of the child keys: a particle index, with all ones beyond every index
        int cbits = 1;
        while (((int64_t)1 << cbits) - 1 <= n - 1) cbits++;
        int rbits = 0;
        while (rbits < 32 && ((uint64_t)(K - 1) >> rbits) != 0) rbits++;
        if (level < ctx->tune.kd_levels) {
            // order each big node's members by k-d splits at leaf-aligned
            // medians (levels 0-2 by default, where most of the search work
            // is); deeper levels keep this order through the stable child
            // partition below
            RS_WS(ctx, unsigned, vcur, WS_RF_KDV, LM);
            RS_LAUNCH(ctx, "rf_kd_init", k_kd_init, T, TQ, 0, L, nd, vcur);
            // each round sorts only the members of the nodes still being
            // split, so a node costs the rounds its own size needs, not the
            // largest node's; the range keys shrink with the active blocks
            for (int r = 0; r < (int)tot[LT_ROUNDS]; r++) {
                const int64_t TA = tot[LT_ROUND0 + 3 * r], NA = tot[LT_ROUND0 + 3 * r + 1],
                              NS = tot[LT_ROUND0 + 3 * r + 2];
                int sbits = 0;
                while (sbits < 40 && (NS >> sbits) != 0) sbits++;
                // the coordinate gives up to 6 of its 16 bits where that saves a
                // pass: 9.6M grouped members' sorts 3.38 -> 2.53 ms, the 134M
                // path's 17.1 -> 15.7, their searches unchanged; with 9 bits
                // left the dense cores' members share a coordinate and the
                // 134M path's searches lose more (89.1 -> 90.2 ms), with 8
                // more yet (92.5)
                const int kbits = std::min(16 + sbits, (10 + sbits + 7) / 8 * 8), drop = 16 + sbits - kbits;
                const int key32 = kbits <= 32 ? 1 : 0;  // (half the bytes)
                // the order stays in place, or the sort's last pass writes it there
                const bool odd = rs_sort_alt(NA, kbits);
                unsigned *va = odd ? v0 : vcur, *vb = odd ? vcur : v1;
                RS_LAUNCH(ctx, "rf_kd_keys", k_kd_keys, TA, TQ, 0, L, nd, (const int64_t *)O.block,
                          (const float4 *)wpos, (const float4 *)wvel, (const unsigned *)vcur,
                          (unsigned long long *)k0, odd ? v0 : nullptr, r, drop, key32,
                          (const rs_dev_status *)ctx->d_status);
                bool kalt = false;
                if (key32)
                    RS_TRY(rs_radix_sort_u32(ctx, (uint32_t *)k0, (uint32_t *)k1, va, vb, NA, kbits, &kalt,
                                             "sort_kd"));
                else
                    RS_TRY(rs_radix_sort_u64(ctx, k0, k1, va, vb, NA, kbits, &kalt, "sort_kd"));
                if (kalt != odd) return rs_fail(ctx, RS_ERR_INTERNAL, "rs_refine6d: k-d order");
            }
            // ranges of at most KD_CTA members finish in one CTA each
            const int64_t rcap = ceil_div(LM, 32) + K;
            RS_WS(ctx, int4, kranges, WS_RF_JOBS, rcap + 1);
            int *kcount = ctr + 10;
            RS_CUDA(ctx, cudaMemsetAsync(kcount, 0, sizeof(int), ctx->stream));
            RS_LAUNCH(ctx, "rf_kd_ranges", k_kd_ranges, ceil_div(T * (TQ / 32), 256), 256, 0, L, nd, T, kranges,
                      kcount);
            RS_LAUNCH(ctx, "rf_kd_finish", k_kd_finish, (int64_t)ctx->num_sms * 8, 256, 0, L, nd,
                      (const int4 *)kranges, (const int *)kcount, (const float4 *)wpos, (const float4 *)wvel, vcur,
                      (const rs_dev_status *)ctx->d_status);
            const unsigned *vsorted = vcur;
            {
                unsigned *kdest = v0;
                RS_LAUNCH(ctx, "rf_kd_place", k_kd_place, T, TQ, 0, L, nd, vsorted, (const float4 *)wpos,
                          (const float4 *)wvel, (const int *)widx, wpos2, wvel2, widx2, kdest,
                          (const rs_dev_status *)ctx->d_status);
                RS_LAUNCH(ctx, "rf_lvl_copyback", k_lvl_copyback, ceil_div(LM, 256), 256, 0, LM,
                          (const unsigned *)kdest, (const float4 *)wpos2, (const float4 *)wvel2, (const int *)widx2,
                          wpos, wvel, widx, (const rs_dev_status *)ctx->d_status);
            }
        }
        // bounding-volume hierarchy of every big node
        RS_WS(ctx, char, boxmem, WS_RF_HIST, NBX * 49 + 1024);
        BoxStore boxes;
        {
            char *bp2 = boxmem;
            boxes.a = carve<float4>(bp2, NBX);
            boxes.b = carve<float4>(bp2, NBX);
            boxes.c = carve<float4>(bp2, NBX);
            boxes.cl = carve<unsigned char>(bp2, NBX);
        }
        RS_WS(ctx, char, srch, WS_RF_SRCH, M * 24 + 512);
        MemberStore ms;
        {
            char *sp2 = srch;
            ms.a = carve<float4>(sp2, M);
            ms.b = carve<float2>(sp2, M);
        }
        const float *nof = nullptr;
        int *noi = nullptr;
        RS_LAUNCH(ctx, "rf_bvh_leaves", k_bvh_leaves<BOX_ALL>, T, TQ, 0, L, nd, (int64_t)0, bo, boxes, ms,
                  (const float4 *)wpos, (const float4 *)wvel, nof, nof, (float *)nullptr, noi, noi, noi, ctx->d_status);
        RS_LAUNCH(ctx, "rf_bvh_build", k_bvh_build<BOX_ALL>, K, 256, 0, L, nd, bo, boxes, nof, nof, noi,
                  ctx->d_status);
        // ---- random member subsets of the nodes above sub_n (Sec. 3.2) ----
        int2 *sub_q = nullptr;
        int *sub_len = ctr + 13;
        int64_t QN = 0, qcap = 0;
        if (sub_n > 0) {
            QN = qcap = tot[LT_SUB] * sub_n;  // every node above sub_n draws exactly sub_n members
            RS_WS(ctx, int2, sq, WS_RF_SUBQ, qcap + 1);
            sub_q = sq;
            RS_CUDA(ctx, cudaMemsetAsync(sub_len, 0, sizeof(int), ctx->stream));
            RS_LAUNCH(ctx, "rf_sub_init", k_sub_init, ceil_div(K, 128), 128, 0, L, nd, (int)sub_n);
            for (int stage = 0; stage < 2; stage++) {
                for (int pass = 0; pass < 3; pass++) {
                    RS_LAUNCH(ctx, "rf_sub_hist", k_sub_hist, T, TQ, 0, L, nd, (const int *)widx,
                              (unsigned long long)sub_seed, (int)sub_n, stage, pass);
                    RS_LAUNCH(ctx, "rf_lvl_pick", k_lvl_pick, K, 256, 0, L, pass);
                }
                RS_LAUNCH(ctx, "rf_sub_stage", k_sub_stage, ceil_div(K, 128), 128, 0, L, stage);
            }
            RS_LAUNCH(ctx, "rf_sub_mark", k_sub_mark, T, TQ, 0, L, nd, (const int *)widx,
                      (unsigned long long)sub_seed, (int)sub_n, dnn, sub_q, sub_len, (int)qcap, ctx->d_status);
            RS_LAUNCH(ctx, "rf_sub_check", k_sub_check, ceil_div(K, 128), 128, 0, L, nd, (int)sub_n, ctx->d_status);
        }
        // ---- linking length: sampled bracket, bounded nearest neighbours, exact select ----
        const int64_t SS = tot[LT_SMP] * SMP_UNIT;
        RS_WS(ctx, float, sdnn, WS_RF_SDNN, SS + 32);
        RS_WS(ctx, float, R2, WS_RF_R2, 2 * K + 8);
        float *STOP = R2 + K;
        RS_LAUNCH(ctx, "rf_smp_nn", k_bvh_nn_sample, SS / W_WARPS, W_WARPS * 32, 0, L, nd, bo, boxes, ms,
                  (const int *)O.smp, (const int *)O.smp_at, (int)ctx->tune.bracket_min, sdnn, ctx->d_status);
        RS_LAUNCH(ctx, "rf_smp_thresh", k_smp_thresh, K, 256, 0, L, nd, (const int *)O.smp_at,
                  (int)ctx->tune.bracket_min, (const float *)sdnn, f, R2, STOP);
        int *fallback = ctr + 7;
        RS_CUDA(ctx, cudaMemsetAsync(ctr + 6, 0, 2 * sizeof(int), ctx->stream));
        // every member's nearest-neighbour distance, searched from the radius
        // the nodes with a bracket: nearest neighbours and friends in one
        // search, while the list of pairs stays within bounds
        PairList pl{};
        const int64_t chunks = LM * PAIR_PER_MEMBER / PAIR_CHUNK / PAIR_REGIONS + 4;  // per region
        const int64_t pl_bytes = PAIR_REGIONS * chunks * (int64_t)(sizeof(int4) + PAIR_CHUNK * sizeof(int2));
        int pairs = 0;
        RsStageGuard listed(&ctx->in_pairs);
        if (SS > 0 && pl_bytes <= PAIR_MAX_BYTES) {
            char *pp = (char *)rs_ws_optional(ctx, WS_RF_PAIRS, (size_t)pl_bytes + 1024, "pairs");
            if (pp) {  // (without the room the nodes are searched twice)
                pairs = 1;
                pl.len = carve<int>(pp, PAIR_REGIONS);
                pl.head = carve<int4>(pp, PAIR_REGIONS * chunks);
                pl.pair = carve<int2>(pp, PAIR_REGIONS * chunks * PAIR_CHUNK);
                pl.cap = (int)chunks;
                pl.R2 = R2;
                pl.STOP = STOP;
                pl.dnn = dnn;
            }
        }
        if (pairs) {
            RS_CUDA(ctx, cudaMemsetAsync(pl.len, 0, sizeof(int) * PAIR_REGIONS, ctx->stream));
            RS_LAUNCH(ctx, "rf_pair_leaves", k_bvh_leaves<BOX_PAIRS>, T, TQ, 0, L, nd, (int64_t)0, bo, boxes, ms,
                      (const float4 *)wpos, (const float4 *)wvel, (const float *)R2, (const float *)STOP, dnn, uf, csize,
                      cmin, ctx->d_status);
            RS_LAUNCH(ctx, "rf_pair_build", k_bvh_build<BOX_PAIRS>, K, 256, 0, L, nd, bo, boxes, (const float *)R2,
                      (const float *)STOP, uf, ctx->d_status);
            RS_TRY(launch_link<true>(ctx, "rf_lvl_pairs", 0, T, L, nd, bo, boxes, ms, uf, pl));
        }
        RS_TRY(launch_nn(ctx, "rf_lvl_nn", T, L, nd, bo, boxes, ms, R2, STOP, 0, (int)sub_n, pairs, dnn));
        if (QN > 0)
            RS_LAUNCH(ctx, "rf_sub_nn", k_bvh_nn_list, ceil_div(QN, W_WARPS), W_WARPS * 32, 0, L, nd,
                      bo, boxes, ms, (const int2 *)sub_q, (const int *)sub_len, (int)qcap, dnn,
                      ctx->d_status);
        RS_LAUNCH(ctx, "rf_lvl_initk", k_lvl_initk, ceil_div(K, 128), 128, 0, L, nd, f, (int)sub_n);
        for (int pass = 0; pass < 3; pass++) {
            RS_LAUNCH(ctx, "rf_lvl_hist", k_lvl_hist, T, TQ, 0, L, nd, (const float *)dnn, pass);
            RS_LAUNCH(ctx, "rf_lvl_pick", k_lvl_pick, K, 256, 0, L, pass);
        }
        RS_LAUNCH(ctx, "rf_bracket_check", k_bracket_check, ceil_div(K, 128), 128, 0, L, R2,
                  (const float *)STOP, fallback, rs_fault("bracket") ? 1 : 0, pairs,
                  (const int *)O.smp_at, ctr + 6);
        RS_LAUNCH(ctx, "rf_lvl_band", k_lvl_band, T, TQ, 0, L, nd, (const float *)dnn);
        // ctr[4]: band members; ctr[6]: a node of the pair search needs the link
        // search; ctr[7]: some node's bracket did not hold
        int64_t flags[2];
        RS_TRY(rs_read_i64(ctx, ctr + 4, 2, flags, "rs_refine6d"));
        if ((flags[1] >> 32) != 0) {
            // unbounded search of those nodes (the others keep their values
            // and selection), and the band once more
            RS_TRY(launch_nn(ctx, "rf_lvl_nn_full", T, L, nd, bo, boxes, ms, R2, nullptr, 1, (int)sub_n, 0, dnn));
            RS_LAUNCH(ctx, "rf_lvl_initk", k_lvl_initk, ceil_div(K, 128), 128, 0, L, nd, f, (int)sub_n);
            for (int pass = 0; pass < 3; pass++) {
                RS_LAUNCH(ctx, "rf_lvl_hist", k_lvl_hist, T, TQ, 0, L, nd, (const float *)dnn, pass);
                RS_LAUNCH(ctx, "rf_lvl_pick", k_lvl_pick, K, 256, 0, L, pass);
            }
            RS_CUDA(ctx, cudaMemsetAsync(ctr + 4, 0, sizeof(int), ctx->stream));
            RS_CUDA(ctx, cudaMemsetAsync(L.below, 0, sizeof(int) * (size_t)K, ctx->stream));
            RS_LAUNCH(ctx, "rf_lvl_band", k_lvl_band, T, TQ, 0, L, nd, (const float *)dnn);
            RS_TRY(rs_read_i64(ctx, ctr + 4, 1, flags, "rs_refine6d"));
            n_fallback_levels++;
        }
        const int nbv = (int)(flags[0] & 0xffffffffll);
        RS_LAUNCH(ctx, "rf_lvl_band_exact", k_lvl_band_exact, ceil_div(nbv, W_WARPS), W_WARPS * 32, 0, L, nd,
                  bo, boxes, ms, (const float *)dnn, ctx->d_status);
        RS_LAUNCH(ctx, "rf_lvl_l2", k_lvl_l2, K, 128, 0, L, nd, f, (int)sub_n, ctx->d_status);
        if (pairs)
            RS_LAUNCH(ctx, "rf_pair_link", k_pair_link, (int64_t)ctx->num_sms * 8, 256, 0, L, nd, ms, pl, uf,
                      ctx->d_status);
        ctx->in_pairs = 0;  // (a release waits for the stream)
        // the other nodes; none when every node has a bracket, every bracket
        // held and every list was whole
        const bool again = (flags[1] & 0xffffffffll) != 0;
        const int64_t t0 = pairs && !again && sub_n == 0 ? T : 0;
        RS_LAUNCH(ctx, "rf_link_leaves", k_bvh_leaves<BOX_LINK>, T - t0, TQ, 0, L, nd, t0, bo, boxes, ms,
                  (const float4 *)wpos, (const float4 *)wvel, nof, nof, dnn, uf, csize, cmin, ctx->d_status);
        RS_LAUNCH(ctx, "rf_link_build", k_bvh_build<BOX_LINK>, t0 < T ? K : 0, 256, 0, L, nd, bo, boxes, nof, nof, uf,
                  ctx->d_status);
        RS_TRY(launch_link<false>(ctx, "rf_lvl_link", t0, T, L, nd, bo, boxes, ms, uf, PairList{}));
        RS_LAUNCH(ctx, "rf_lvl_comp", k_lvl_comp, T, TQ, 0, L, nd, (const int *)widx, uf, csize, cmin,
                  ctx->d_status);
        // reorder: children first, by smallest particle index, then the rest
        RS_LAUNCH(ctx, "rf_lvl_keys", k_lvl_keys, T, TQ, 0, L, nd, uf, (const int *)csize, (const int *)cmin,
                  (unsigned long long *)k0, v0, (int)min_n, cbits, ctx->d_status);
        bool alt = false;
        RS_TRY(rs_radix_sort_u64(ctx, k0, k1, v0, v1, LM, cbits + rbits, &alt, "sort_child"));
        const unsigned long long *sk = (const unsigned long long *)(alt ? k1 : k0);
        const unsigned *sv = alt ? v1 : v0;
        unsigned *dest = (unsigned *)(alt ? v0 : v1);
        RS_LAUNCH(ctx, "rf_lvl_children", k_lvl_children, ceil_div(LM, 256), 256, 0, L, nd, LM, sk, sv, uf,
                  (const int *)csize, nxt, nxt_len, small_q, ctr + 2, cbits, ctx->d_status);
        RS_LAUNCH(ctx, "rf_lvl_scatter", k_lvl_scatter, ceil_div(LM, 256), 256, 0, L, nd, LM, sk, sv,
                  (const float4 *)wpos, (const float4 *)wvel, (const int *)widx, wpos2, wvel2, widx2, dest, cbits,
                  (const rs_dev_status *)ctx->d_status);
        RS_LAUNCH(ctx, "rf_lvl_copyback", k_lvl_copyback, ceil_div(LM, 256), 256, 0, LM, (const unsigned *)dest,
                  (const float4 *)wpos2, (const float4 *)wvel2, (const int *)widx2, wpos, wvel, widx,
                  (const rs_dev_status *)ctx->d_status);
        RS_LAUNCH(ctx, "rf_lvl_tie", k_lvl_store_tie, ceil_div(K, 128), 128, 0, L, nd);
        // next level
        RS_CUDA(ctx, cudaMemsetAsync(cur_len, 0, sizeof(int), ctx->stream));
        int *tq = cur;
        cur = nxt;
        nxt = tq;
        int *tl2 = cur_len;
        cur_len = nxt_len;
        nxt_len = tl2;
    }

    // ---- small nodes: whole subtrees ----
    // four size classes, each forwarding its smaller subtrees to the next
    {
        auto kbig = k_small_subtree<SMALL_N, SMALL_THREADS, 3>;
        auto kmid = k_small_subtree<MID_N, MID_THREADS, 8>;
        auto kwarp = k_small_subtree<WARP_N, 32, WARP_CTAS>;
        const size_t sbig = sizeof(SmallShared<SMALL_N, SMALL_THREADS>);
        const size_t smid = sizeof(SmallShared<MID_N, MID_THREADS>);
        const size_t swarp = sizeof(SmallShared<WARP_N, 32>);
        RS_CUDA(ctx, cudaFuncSetAttribute(kbig, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sbig));
        RS_CUDA(ctx, cudaFuncSetAttribute(kmid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smid));
        const rs_tuning &tu = ctx->tune;
        const int mid_max = std::min(tu.mid_max, MID_N), tiny_max = std::min(tu.tiny_max, TINY_N);
        RS_LAUNCH(ctx, "rf_small_subtree", kbig, (int64_t)ctx->num_sms * (tu.small_ctas_per_sm + 1), SMALL_THREADS, sbig,
                  (const int *)small_q, (const int *)(ctr + 2), ctr + 3, wpos, wvel, widx, mid_max, mid_q, ctr + 11,
                  nd, (const SizeTab *)size_tab, box, (int)min_n, ctx->d_status);
        RS_LAUNCH(ctx, "rf_mid_subtree", kmid, (int64_t)ctx->num_sms * tu.mid_ctas_per_sm, MID_THREADS, smid,
                  (const int *)mid_q, (const int *)(ctr + 11), ctr + 12, wpos, wvel, widx,
                  std::min(mid_max, WARP_N), warp_q, ctr + 14, nd, (const SizeTab *)size_tab, box, (int)min_n,
                  ctx->d_status);
        RS_LAUNCH(ctx, "rf_warp_subtree", kwarp, (int64_t)ctx->num_sms * WARP_CTAS * tu.mid_ctas_per_sm / 8, 32, swarp,
                  (const int *)warp_q, (const int *)(ctr + 14), ctr + 15, wpos, wvel, widx, tiny_max, tiny_q, ctr + 8,
                  nd, (const SizeTab *)size_tab, box, (int)min_n, ctx->d_status);
        RS_LAUNCH(ctx, "rf_tiny_subtree", k_tiny_subtree, (int64_t)ctx->num_sms * tu.tiny_ctas_per_sm,
                  TINY_WARPS * 32, 0, (const int *)tiny_q, (const int *)(ctr + 8), ctr + 9, (const float4 *)wpos,
                  (const float4 *)wvel, widx, nd, (const SizeTab *)size_tab, box, (int)min_n, ctx->d_status);
    }

    // ---- summary ----
    RS_WS(ctx, unsigned long long, so, WS_RF_MISC3, 5);
    RS_CUDA(ctx, cudaMemsetAsync(so, 0, 5 * sizeof(unsigned long long), ctx->stream));
    RS_LAUNCH(ctx, "rf_tree_stats", k_tree_stats, std::min<int64_t>(ceil_div(cap, 256), ctx->num_sms * 4), 256, 0, nd,
              so);
    int64_t s5[5];
    RS_TRY(rs_read_i64(ctx, so, 5, s5, "rs_refine6d"));
    const int64_t *s4 = s5 + 1, nn = s5[0];
    if (nn > cap) return rs_fail(ctx, RS_ERR_INTERNAL, "rs_refine6d: node capacity exceeded");
    t->n_nodes = nn;
    t->n_seeds = s4[0];
    t->n_tieband = s4[1];
    t->n_levels = nn > 0 ? (int32_t)s4[2] + 1 : 0;
    t->sum_level_members = s4[3];
    t->sum_big_level_members = sum_level;
    t->n_fallback_levels = n_fallback_levels;
    return RS_OK;
}

// ---------------------------------------------------------------------------
// public tree API
// ---------------------------------------------------------------------------
namespace {

__global__ void k_tree_export(NodeArrays nd, int nn, int32_t *parent, int32_t *level, int64_t *first,
                              int64_t *count, int32_t *minidx, int32_t *nchild, double *lnk, double *xbar,
                              double *vbar, double *sigx, double *sigv, int64_t *tie)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nn; i += gridDim.x * blockDim.x) {
        if (parent) parent[i] = nd.parent[i];
        if (level) level[i] = nd.level[i];
        if (first) first[i] = nd.first[i];
        if (count) count[i] = nd.count[i];
        if (minidx) minidx[i] = nd.minidx[i];
        if (nchild) nchild[i] = nd.nchild[i];
        if (lnk) lnk[i] = nd.lnk[i];
        if (sigx) sigx[i] = nd.sigx[i];
        if (sigv) sigv[i] = nd.sigv[i];
        if (tie) tie[i] = nd.tie[i];
        for (int d = 0; d < 3; d++) {
            if (xbar) xbar[3 * i + d] = nd.xbar[3 * i + d];
            if (vbar) vbar[3 * i + d] = nd.vbar[3 * i + d];
        }
    }
}

// A warp looks at 32 nodes at once; LABEL_SPLIT rows of warps share the nodes,
// and the members of the nodes above 1024 (9.6M members, 8 levels: 1.36
// ms with a warp a node, 0.63 so).
constexpr int LABEL_SPLIT = 16;

__global__ void __launch_bounds__(256) k_level_labels(NodeArrays nd, int nn, int level, const int *members,
                                                      int32_t *labels)
{
    const int lane = lane_id(), y = blockIdx.y;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int i = 32 * w + lane;
    const bool hit = i < nn && nd.level[i] == level;
    const int a0 = hit ? nd.first[i] : 0, c0 = hit ? nd.count[i] : 0, id0 = hit ? nd.minidx[i] : 0;
    unsigned m = __ballot_sync(0xffffffffu, hit && (c0 > 1024 || (lane & (LABEL_SPLIT - 1)) == y));
    while (m) {
        const int s = __ffs(m) - 1;
        m &= m - 1;
        const int a = __shfl_sync(0xffffffffu, a0, s), c = __shfl_sync(0xffffffffu, c0, s),
                  id = __shfl_sync(0xffffffffu, id0, s);
        const int rows = c > 1024 ? LABEL_SPLIT : 1;
        for (int q = 32 * (rows > 1 ? y : 0) + lane; q < c; q += 32 * rows) labels[members[a + q]] = id;
    }
}

__global__ void k_fill_i32(int32_t *p, int64_t n, int32_t v)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

}  // namespace

extern "C" void rs_tree_free(rs_tree *t)
{
    if (!t) return;
    rs_block_give_back(t->block, t->pool);
    delete t;
}

extern "C" rs_status rs_refine6d_sampled(rs_ctx *ctx, const float *pos, const float *vel, int32_t stride, int64_t n,
                                         double box, const int32_t *perm, const int64_t *group_offsets,
                                         int64_t n_groups, double f, int32_t min_n, int64_t subset_n,
                                         uint64_t subset_seed, rs_tree **out)
{
    if (!ctx) return RS_ERR_INVALID_ARG;
    if (!out) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_refine6d: out is NULL");
    *out = nullptr;
    if (n < 0 || n_groups < 0 || (stride != 3 && stride != 4) || !(box > 0) || !(f > 0 && f < 1) || min_n < 2 ||
        !group_offsets || (n > 0 && (!pos || !vel)) || (n_groups > 0 && !perm))
        return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_refine6d: bad argument");
    if (subset_n != 0 && (subset_n < SMALL_N || subset_n >= ((int64_t)1 << 31)))
        return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_refine6d: subset size must be 0 or in [1024, 2^31)");
    if (n >= ((int64_t)1 << 31)) return rs_fail(ctx, RS_ERR_TOO_LARGE, "rs_refine6d: n >= 2^31");
    if ((double)(float)box != box) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_refine6d: box must be a float32 value");
    RsRange range("rs_refine6d");
    // the first and last offset, and the offsets' order, in one host read
    RS_LAUNCH(ctx, "rf_check_offsets", k_check_offsets, ceil_div(n_groups, 256), 256, 0, n_groups, group_offsets,
              ctx->d_status);
    RS_CUDA(ctx, cudaMemcpyAsync(ctx->h_scratch, group_offsets, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    RS_CUDA(ctx, cudaMemcpyAsync(ctx->h_scratch + 1, group_offsets + n_groups, sizeof(int64_t),
                                 cudaMemcpyDeviceToHost, ctx->stream));
    RS_TRY(rs_sync_check(ctx, "rs_refine6d: group offsets must be non-decreasing"));
    const int64_t first = ctx->h_scratch[0], M = ctx->h_scratch[1] - first;
    if (M < 0 || M > n || first < 0)
        return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_refine6d: inconsistent group offsets");
    int64_t cap = M / 4 + 4096;
    for (int attempt = 0; attempt < 4; attempt++) {
        rs_tree *t = nullptr;
        rs_status s = refine_impl(ctx, pos, vel, stride, n, box, perm, group_offsets, n_groups, M, f, min_n,
                                  subset_n, subset_seed, cap, &t);
        if (s == RS_OK) {
            *out = t;
            return RS_OK;
        }
        bool overflow = false;
        if (t) {
            int cnt = 0;
            cudaStreamSynchronize(ctx->stream);
            if (cudaMemcpy(&cnt, t->nd.counter, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess)
                overflow = (int64_t)cnt > cap;
            rs_tree_free(t);
        }
        if (!overflow || cap > ((int64_t)1 << 30)) return s;
        cap *= 4;
    }
    return rs_fail(ctx, RS_ERR_INTERNAL, "rs_refine6d: node capacity");
}

extern "C" rs_status rs_refine6d(rs_ctx *ctx, const float *pos, const float *vel, int32_t stride, int64_t n,
                                 double box, const int32_t *perm, const int64_t *group_offsets, int64_t n_groups,
                                 double f, int32_t min_n, rs_tree **out)
{
    return rs_refine6d_sampled(ctx, pos, vel, stride, n, box, perm, group_offsets, n_groups, f, min_n, 0, 0, out);
}

extern "C" rs_status rs_tree_info(const rs_tree *t, int64_t *n_nodes, int32_t *n_levels, int64_t *n_seeds,
                                  int64_t *n_tieband, int64_t *n_members)
{
    if (!t) return RS_ERR_INVALID_ARG;
    if (n_nodes) *n_nodes = t->n_nodes;
    if (n_levels) *n_levels = t->n_levels;
    if (n_seeds) *n_seeds = t->n_seeds;
    if (n_tieband) *n_tieband = t->n_tieband;
    if (n_members) *n_members = t->n_members;
    return RS_OK;
}

extern "C" rs_status rs_tree_nodes(rs_ctx *ctx, const rs_tree *t, int32_t *parent, int32_t *level, int64_t *first,
                                   int64_t *count, int32_t *minidx, int32_t *nchild, double *lnk, double *xbar,
                                   double *vbar, double *sigx, double *sigv, int64_t *tie)
{
    if (!ctx || !t) return RS_ERR_INVALID_ARG;
    const int nn = (int)t->n_nodes;
    RS_LAUNCH(ctx, "tree_export", k_tree_export, std::min<int64_t>(ceil_div(nn, 256), 4096), 256, 0, t->nd, nn,
              parent, level, first, count, minidx, nchild, lnk, xbar, vbar, sigx, sigv, tie);
    return RS_OK;
}

extern "C" rs_status rs_tree_members(rs_ctx *ctx, const rs_tree *t, int32_t *members)
{
    if (!ctx || !t || (t->n_members > 0 && !members)) return RS_ERR_INVALID_ARG;
    if (t->n_members > 0)
        RS_CUDA(ctx, cudaMemcpyAsync(members, t->members, sizeof(int32_t) * t->n_members, cudaMemcpyDeviceToDevice,
                                     ctx->stream));
    return RS_OK;
}

extern "C" rs_status rs_tree_level_labels(rs_ctx *ctx, const rs_tree *t, int32_t level, int64_t n, int32_t *labels)
{
    if (!ctx || !t || n < 0 || (n > 0 && !labels)) return RS_ERR_INVALID_ARG;
    if (n != t->n_total) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_tree_level_labels: n differs from the tree's");
    if (n == 0) return RS_OK;
    RS_LAUNCH(ctx, "tree_fill", k_fill_i32, std::min<int64_t>(ceil_div(n, 256), 4096), 256, 0, labels, n, -1);
    const int nn = (int)t->n_nodes;
    if (nn > 0) {
        const dim3 grid((unsigned)ceil_div(nn, 256), LABEL_SPLIT);
        const int pr = rs_prof_begin(ctx, "tree_level_labels");
        k_level_labels<<<grid, 256, 0, ctx->stream>>>(t->nd, nn, level, (const int *)t->members, labels);
        ctx->launches++;
        rs_prof_end(ctx, pr);
        RS_CUDA(ctx, cudaGetLastError());
    }
    return RS_OK;
}
