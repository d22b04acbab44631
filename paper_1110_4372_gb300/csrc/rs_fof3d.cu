// rs_fof3d.cu -- periodic 3D friends-of-friends (Sec. 3.1) and the group CSR.
//
// Particles are binned into fine cells of side s <= l / sqrt(3) (with a
// margin that covers the float32 rounding of the cell index), so any two
// particles of one fine cell are friends and a fine cell can stand for all
// of its particles in the union-find.  Fine cells are grouped 4 x 4 x 4 into
// coarse cells; particles are radix-sorted by (coarse cell, fine sub-cell),
// a dense table maps each coarse cell to its first fine cell, and a 64-bit
// mask stored at that first fine cell tells which of the 64 sub-cells are
// occupied.  Every friend of a particle lies within two fine cells per axis,
// which is inside at most 2 x 2 x 2 coarse cells; the fine cells within
// reach of a fine cell follow from the masks by bit operations, and their
// indices by a popcount, with no scan.  Two fine cells are joined as soon as
// one pair between them is within l; pairs already in one set are skipped.
//
// Distances: float32 with the periodic shift applied to the coordinate near
// the top of the box (x - box is exact there), compared against l^2 (1 -+
// 2^-20); pairs inside that band are re-tested in float64 with the same
// separate multiplies and adds as the definition, so the partition is the
// float64 one.
#include <cmath>
#include <utility>

#include "rs_internal.cuh"

namespace {

constexpr int FOF_THREADS = 256;
constexpr int64_t FOF_ONE_PASS = 8192;  // particles linked in one pass (see k_fof_link)
constexpr double BAND_REL = 9.5367431640625e-07;  // 2^-20, relative on d^2

struct FofGeom {
    int32_t Gc;      // coarse cells per side
    int32_t Gf;      // fine cells per side (4 Gc)
    float inv_sf;    // Gf / box (float32)
    float boxf;
    double box;
    double l, l2;
    float lo32, hi32;  // float32 thresholds on d^2 around l^2
};

__device__ __forceinline__ void load_pos(const float *pos, int stride, int64_t i, float &x, float &y, float &z)
{
    const float *p = pos + (int64_t)stride * i;
    x = p[0];
    y = p[1];
    z = p[2];
}

__device__ __forceinline__ int fine_coord(float x, float inv, int Gf)
{
    int f = (int)floorf(x * inv);
    f = f < 0 ? 0 : f;
    f = f >= Gf ? Gf - 1 : f;
    return f;
}

// keys of the particles; the coarse table starts empty
__global__ void k_fof_keys(const float *pos, int stride, int64_t n, FofGeom g, uint64_t *keys, uint32_t *vals,
                           uint32_t *table, int64_t ncoarse, rs_dev_status *st)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t c = i; c < ncoarse; c += (int64_t)gridDim.x * blockDim.x) table[c] = 0xffffffffu;
    if (i >= n) return;
    float x, y, z;
    load_pos(pos, stride, i, x, y, z);
    if (!(x >= 0.f && x < g.boxf && y >= 0.f && y < g.boxf && z >= 0.f && z < g.boxf))
        dev_fail(st, DEV_BADARG, 10, i);
    int fx = fine_coord(x, g.inv_sf, g.Gf), fy = fine_coord(y, g.inv_sf, g.Gf), fz = fine_coord(z, g.inv_sf, g.Gf);
    uint64_t c = ((uint64_t)(fz >> 2) * (uint64_t)g.Gc + (uint64_t)(fy >> 2)) * (uint64_t)g.Gc + (uint64_t)(fx >> 2);
    uint32_t sub = (uint32_t)(((fz & 3) << 4) | ((fy & 3) << 2) | (fx & 3));
    keys[i] = (c << 6) | sub;
    vals[i] = (uint32_t)i;
}

// One pass over the sorted keys: sorted positions as float4, the fine cells
// numbered (runs of equal keys, by a scan with look-back: a warp takes rows of
// 32 keys and counts run starts by votes), and every per-cell array started
// where its cell is.  One launch instead of a gather, a copy, a scan of three
// launches, the numbering and three fills over n.
constexpr int CELL_ROWS = 8;  // rows of 32 particles per warp
constexpr int64_t CELL_TILE = (int64_t)CELL_ROWS * FOF_THREADS;

__global__ void __launch_bounds__(FOF_THREADS) k_fof_cells(const float *pos, int stride, int64_t n, const uint64_t *keys,
                                                           const uint32_t *idx, float4 *spos, uint32_t *cell_of,
                                                           uint32_t *cell_start, uint64_t *cell_key, uint32_t *table,
                                                           uint64_t *occ, int *parent, int *root_min,
                                                           uint32_t *n_cells, RsLookback lb, rs_dev_status *st)
{
    const unsigned FULL = 0xffffffffu;
    // (for the whole block: other blocks' look-backs may run out meanwhile)
    if (__syncthreads_or(*(volatile int32_t *)&st->torn)) return;
    const int64_t tile = rs_next_tile(lb);
    const int lane = lane_id();
    const int64_t base = tile * CELL_TILE + (int64_t)warp_id() * 32 * CELL_ROWS;
    uint64_t key[CELL_ROWS];
    unsigned starts[CELL_ROWS], coarse[CELL_ROWS];
    int count = 0;
#pragma unroll
    for (int j = 0; j < CELL_ROWS; j++) {
        const int64_t q = base + 32 * j + lane;
        key[j] = q < n ? keys[q] : 0;
        uint64_t prev = __shfl_up_sync(FULL, key[j], 1);
        if (lane == 0 && q > 0 && q < n) prev = keys[q - 1];
        starts[j] = __ballot_sync(FULL, q < n && (q == 0 || key[j] != prev));
        coarse[j] = __ballot_sync(FULL, q < n && (q == 0 || (key[j] >> 6) != (prev >> 6)));
        count += __popc(starts[j]);
    }
    uint32_t tot;
    uint32_t c0 = rs_block_scan<FOF_THREADS>(lane == 0 ? (uint32_t)count : 0u, tot);
    c0 = __shfl_sync(FULL, c0, 0) + (uint32_t)rs_lookback(lb, tile, tot, st);
    const unsigned upto = (2u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < CELL_ROWS; j++) {
        const int64_t q = base + 32 * j + lane;
        const uint32_t c = c0 + (uint32_t)__popc(starts[j] & upto) - 1u;
        c0 += (uint32_t)__popc(starts[j]);
        if (q >= n || c >= n) continue;  // (after a look-back that ran out of time: see dev_torn)
        float x, y, z;
        load_pos(pos, stride, idx[q], x, y, z);
        spos[q] = make_float4(x, y, z, 0.f);
        cell_of[q] = c;
        if ((starts[j] >> lane) & 1u) {
            cell_start[c] = (uint32_t)q;
            cell_key[c] = key[j];
            occ[c] = 0;
            parent[c] = (int)c;
            root_min[c] = 0x7fffffff;
            if ((coarse[j] >> lane) & 1u) table[key[j] >> 6] = c;
        }
        if (q == n - 1) {
            *n_cells = c + 1u;
            cell_start[c + 1u] = (uint32_t)n;
        }
    }
}

// occupancy mask of each coarse cell, kept at its first fine cell.  After a
// torn sort or scan there are no cells: the kernels that go over them then do
// nothing.
__global__ void k_fof_occ(uint32_t *n_cells_p, const uint64_t *cell_key, const uint32_t *table, uint64_t *occ,
                          const rs_dev_status *st)
{
    if (dev_is_torn(st)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *n_cells_p = 0u;
        return;
    }
    const int64_t M = *n_cells_p;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < M; c += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = cell_key[c];
        atomicOr((unsigned long long *)&occ[table[k >> 6]], 1ull << (k & 63));
    }
}

// sub-cells (4 per axis, bit (z << 4) | (y << 2) | x) of the coarse cell at
// coarse offset d (per axis) whose fine offset from sub-cell u of the query's
// coarse cell is at most R on every axis
__device__ __forceinline__ unsigned axis_range(int u, int d, int R)
{
    const int lo = max(u - R - 4 * d, 0), hi = min(u + R - 4 * d, 3);
    return lo > hi ? 0u : ((2u << hi) - 1u) & ~((1u << lo) - 1u);
}

__device__ __forceinline__ uint64_t reach_mask(int ux, int uy, int uz, int dx, int dy, int dz, int R)
{
    const unsigned mx = axis_range(ux, dx, R), my = axis_range(uy, dy, R), mz = axis_range(uz, dz, R);
    unsigned m16 = 0;
    for (int y = 0; y < 4; y++)
        if ((my >> y) & 1u) m16 |= mx << (4 * y);
    uint64_t m = 0;
    for (int z = 0; z < 4; z++)
        if ((mz >> z) & 1u) m |= (uint64_t)m16 << (16 * z);
    return m;
}

// Tables that combine four bits per axis into a coarse cell's 64 sub-cells,
// filled by the whole block
struct ReachTab {
    uint64_t axis[3][16];
    __device__ __forceinline__ void fill()
    {
        if (threadIdx.x < 16) {
            const unsigned m = threadIdx.x;
            uint64_t x = 0, y = 0, z = 0;
            for (int b = 0; b < 64; b++) {
                x |= (uint64_t)((m >> (b & 3)) & 1u) << b;
                y |= (uint64_t)((m >> ((b >> 2) & 3)) & 1u) << b;
                z |= (uint64_t)((m >> (b >> 4)) & 1u) << b;
            }
            axis[0][m] = x;
            axis[1][m] = y;
            axis[2][m] = z;
        }
        __syncthreads();
    }
    __device__ __forceinline__ uint64_t mask(unsigned mx, unsigned my, unsigned mz) const
    {
        return axis[0][mx] & axis[1][my] & axis[2][mz];
    }
};

__device__ __forceinline__ void coarse_coords(uint64_t c, int Gc, int &cx, int &cy, int &cz)
{
    const uint32_t cc = (uint32_t)c, G = (uint32_t)Gc;  // fewer than 2^32 coarse cells
    const uint32_t r = cc / G;
    cx = (int)(cc - r * G);
    cz = (int)(r / G);
    cy = (int)(r - (uint32_t)cz * G);
}

// wrapped fine-cell offset b - a in [-Gf/2, Gf/2); shift tells which point
// sits on the far side of the periodic face (+1: b near the top, -1: a)
__device__ __forceinline__ int fine_offset(int a, int b, int Gf, int &shift)
{
    int d = b - a;
    shift = 0;
    if (d > Gf / 2) {
        d -= Gf;
        shift = 1;
    } else if (d < -(Gf / 2)) {
        d += Gf;
        shift = -1;
    }
    return d;
}

__device__ __forceinline__ float sdiff(float a, float b, int shift, float box)
{
    // b - a with the periodic image chosen by shift; x - box is exact for x >= box/2
    if (shift > 0) return (b - box) - a;
    if (shift < 0) return b - (a - box);
    return b - a;
}

__device__ __forceinline__ double ddiff(float a, float b, int shift, double box)
{
    if (shift > 0) return f64_sub(f64_sub((double)b, box), (double)a);
    if (shift < 0) return f64_sub((double)b, f64_sub((double)a, box));
    return f64_sub((double)b, (double)a);
}

// 0 = not friends, 1 = friends
__device__ __forceinline__ int pair_link(const float4 &pa, const float4 &pb, int sx, int sy, int sz,
                                         const FofGeom &g)
{
    float dx = sdiff(pa.x, pb.x, sx, g.boxf), dy = sdiff(pa.y, pb.y, sy, g.boxf), dz = sdiff(pa.z, pb.z, sz, g.boxf);
    float d2 = dx * dx + dy * dy + dz * dz;
    if (d2 <= g.lo32) return 1;
    if (d2 > g.hi32) return 0;
    double ex = ddiff(pa.x, pb.x, sx, g.box), ey = ddiff(pa.y, pb.y, sy, g.box), ez = ddiff(pa.z, pb.z, sz, g.box);
    double e2 = f64_add(f64_add(f64_mul(ex, ex), f64_mul(ey, ey)), f64_mul(ez, ez));
    return e2 <= g.l2 ? 1 : 0;
}

// Join fine cell A with every fine cell of larger index within two fine cells
// per axis that has a friend pair with it.  Pass 0 takes the 26 adjacent
// cells (offsets of at most 1 per axis), where pairs are friends almost at
// once in dense regions; pass 1 takes the cells two apart on some axis, by
// which time dense regions are mostly one set: a coarse cell whose fine cells
// all had one root after pass 0 (uroot at its first fine cell, else -1) is
// skipped whole when that root is A's, and the same-set check skips the
// rest.  Coarse cells numbered below A's hold only fine cells of smaller
// index and are not visited.
//
// Pass 2 takes all cells at once, for boxes so small that the passes' chains
// of dependent loads cost more than their pairs (32,768 particles: 166 us in
// one pass, 76 in two, so up to 8192 only).  Where the rows of 32 cells do not
// fill the device a warp takes only 8 / split of the eight coarse cells, so
// that more warps share the chain, and the root kernels between the passes are
// left out (32,768 particles: 117 -> 76 us).
//
// A warp takes 32 consecutive fine cells, a lane each.  Its reach per axis and
// neighbouring coarse cell is formed once (four bits an axis, combined per
// coarse cell through tables), and a coarse cell is looked up only when the
// reach touches it.  Candidate pairs go to the warp's queue, the lanes' lowest
// bits at a time, and are tested 32 at a time whatever their spread over the
// cells.  Bound by instruction issue and the loads of the tests.  Numbering
// the candidates by a prefix sum and finding each lane's by its rank (with
// __fns), and looking up all eight coarse cells, took 6.7 ms for 33M
// particles; this takes 4.6.
__global__ void __launch_bounds__(FOF_THREADS, 6) k_fof_link(const uint32_t *n_cells_p, const uint64_t *cell_key,
                                                            const uint32_t *cell_start, const uint32_t *table,
                                                            const uint64_t *occ, const float4 *spos, int *parent,
                                                            const int *uroot, FofGeom g, int pass, int split,
                                                            rs_dev_status *st)
{
    const unsigned FULL = 0xffffffffu;
    __shared__ ReachTab tab;
    __shared__ int qa_s[FOF_THREADS / 32][64], qb_s[FOF_THREADS / 32][64];
    __shared__ unsigned char qs_s[FOF_THREADS / 32][64];  // periodic shifts, two bits an axis (0: none, 1: +, 2: -)
    tab.fill();
    const int64_t M = *n_cells_p;
    const int lane = lane_id(), w = warp_id();
    int *qa = qa_s[w], *qb = qb_s[w];
    unsigned char *qs = qs_s[w];
    int np = 0;
    // tests up to 32 queued pairs, one a lane
    auto flush = [&](int cnt) {
        np -= cnt;
        if (lane < cnt) {
            const int A = qa[np + lane], B = qb[np + lane], s = qs[np + lane];
            if (uf_find(parent, A, st) != uf_find(parent, B, st)) {
                const int sx = (s & 1) - ((s >> 1) & 1), sy = ((s >> 2) & 1) - ((s >> 3) & 1),
                          sz = ((s >> 4) & 1) - ((s >> 5) & 1);
                const uint32_t a0 = cell_start[A], a1 = cell_start[A + 1], b0 = cell_start[B], b1 = cell_start[B + 1];
                bool linked = false;
                for (uint32_t i = a0; i < a1 && !linked; i++) {
                    const float4 pa = spos[i];
                    for (uint32_t q = b0; q < b1; q++)
                        if (pair_link(pa, spos[q], sx, sy, sz, g)) {
                            linked = true;
                            break;
                        }
                }
                if (linked) uf_union(parent, A, B, st);
            }
        }
        __syncwarp();
    };
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t warps = (int64_t)gridDim.x * blockDim.x >> 5;
    for (int64_t u = warp0; u < (M + 31) / 32 * split; u += warps) {
        const int64_t A = u / split * 32 + lane;
        const int s0 = (int)(u % split) * (8 / split), s1 = s0 + 8 / split;
        const bool va = A < M;
        uint64_t ca = 0;
        int sa = 0, ccx = 0, ccy = 0, ccz = 0;
        if (va) {
            const uint64_t ka = cell_key[A];
            ca = ka >> 6;
            sa = (int)(ka & 63);
            coarse_coords(ca, g.Gc, ccx, ccy, ccz);
        }
        // per axis, for the lower and the upper of the two coarse cells in
        // reach: the sub-cells at most 1 away (bits 0-3) and at most 2 (4-7)
        const int ux = sa & 3, uy = (sa >> 2) & 3, uz = sa >> 4;
        const int lox = ux < 2 ? -1 : 0, loy = uy < 2 ? -1 : 0, loz = uz < 2 ? -1 : 0;
        auto ranges = [](int c, int d) { return axis_range(c, d, 1) | axis_range(c, d, 2) << 4; };
        const unsigned rx = ranges(ux, lox) | ranges(ux, lox + 1) << 8, ry = ranges(uy, loy) | ranges(uy, loy + 1) << 8,
                       rz = ranges(uz, loz) | ranges(uz, loz + 1) << 8;
        // a root of A's set (sets only grow, so a coarse cell whose common
        // root equals it is in A's set for the rest of the pass)
        const int ra = (va && uroot) ? uf_find(parent, (int)A, st) : -1;
        for (int s8 = s0; s8 < s1; s8++) {
            const unsigned mx = rx >> (8 * (s8 & 1)), my = ry >> (8 * ((s8 >> 1) & 1)), mz = rz >> (8 * (s8 >> 2));
            const uint64_t near = tab.mask(mx & 15u, my & 15u, mz & 15u);
            uint64_t cand = near;
            if (pass > 0) {
                cand = tab.mask((mx >> 4) & 15u, (my >> 4) & 15u, (mz >> 4) & 15u);
                if (pass == 1) cand &= ~near;
            }
            uint64_t om = 0;
            uint32_t b0c = 0xffffffffu;
            unsigned shift = 0;
            if (va && cand) {
                int cx = ccx + lox + (s8 & 1), cy = ccy + loy + ((s8 >> 1) & 1), cz = ccz + loz + (s8 >> 2);
                // (a cell reached across the lower face lies near the top)
                shift = (cx < 0 ? 1u : (cx >= g.Gc ? 2u : 0u)) | (cy < 0 ? 4u : (cy >= g.Gc ? 8u : 0u)) |
                        (cz < 0 ? 16u : (cz >= g.Gc ? 32u : 0u));
                cx = cx < 0 ? cx + g.Gc : (cx >= g.Gc ? cx - g.Gc : cx);
                cy = cy < 0 ? cy + g.Gc : (cy >= g.Gc ? cy - g.Gc : cy);
                cz = cz < 0 ? cz + g.Gc : (cz >= g.Gc ? cz - g.Gc : cz);
                const uint64_t cc = ((uint64_t)cz * g.Gc + cy) * g.Gc + cx;
                if (cc == ca) cand &= ~((2ull << sa) - 1ull);  // sub-cells after A's
                // (coarse cells below A's hold only fine cells of smaller index)
                if (cc >= ca && cand) b0c = table[cc];
                if (b0c != 0xffffffffu && !(ra >= 0 && uroot[b0c] == ra)) om = occ[b0c];
            }
            cand &= om;
            for (;;) {
                const unsigned bm = __ballot_sync(FULL, cand != 0);
                if (!bm) break;
                if (cand) {
                    const int sb = __ffsll((long long)cand) - 1;
                    cand &= cand - 1ull;
                    const int at = np + __popc(bm & ((1u << lane) - 1u));
                    qa[at] = (int)A;
                    qb[at] = (int)(b0c + (uint32_t)__popcll(om & ((1ull << sb) - 1ull)));
                    qs[at] = (unsigned char)shift;
                }
                np += __popc(bm);
                __syncwarp();
                if (np >= 32) flush(32);
            }
        }
    }
    if (np > 0) flush(np);
}

// the root of every coarse cell's first fine cell, kept at that cell
__global__ void k_fof_uroot_first(const uint32_t *n_cells_p, const uint64_t *cell_key, const uint32_t *table,
                                  int *parent, int *uroot, rs_dev_status *st)
{
    const int64_t M = *n_cells_p;
    for (int64_t A = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; A < M; A += (int64_t)gridDim.x * blockDim.x)
        if (table[cell_key[A] >> 6] == (uint32_t)A) uroot[A] = uf_find(parent, (int)A, st);
}

// -1 at the first fine cell of every coarse cell whose fine cells do not all
// share that root (no unions run meanwhile, so roots are fixed)
__global__ void k_fof_uroot_check(const uint32_t *n_cells_p, const uint64_t *cell_key, const uint32_t *table,
                                  int *parent, int *uroot, rs_dev_status *st)
{
    const int64_t M = *n_cells_p;
    for (int64_t A = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; A < M; A += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t b0 = table[cell_key[A] >> 6];
        if (b0 != (uint32_t)A && uf_find(parent, (int)A, st) != uroot[b0]) uroot[b0] = -1;
    }
}

// (find_limit bounds each find; it is RS_SPIN_LIMIT except under the
// injected fault RS_FAULT=timeout1, where it is 1)
__global__ void k_fof_rootmin(const uint32_t *n_cells_p, const uint32_t *cell_start, const uint32_t *idx,
                              int *parent, int *root_min, int find_limit, rs_dev_status *st)
{
    const int64_t M = *n_cells_p;
    for (int64_t A = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; A < M; A += (int64_t)gridDim.x * blockDim.x) {
        // (a cell's particles are in index order; reading them all, and adding
        // to roots that already hold less, took 0.63 ms for 33M particles,
        // this 0.1)
        const int m = (int)idx[cell_start[A]];
        // No path halving here: a cell's parent is written by its own thread
        // alone, so that it is the root when the labels read it (a late
        // halving write of another thread would put back an ancestor).
        int r = (int)A, it = 0;
        for (; it < find_limit; it++) {
            const int p = __ldcg(&parent[r]);
            if (p == r) break;
            r = p;
        }
        if (it >= find_limit) dev_fail(st, DEV_TIMEOUT, 1, r);
        if (r != (int)A) parent[A] = r;
        if (m < __ldcg(&root_min[r])) atomicMin(&root_min[r], m);
    }
}

// (every cell's parent is its root by now)
__global__ void k_fof_labels(int64_t n, const uint32_t *idx, const uint32_t *cell_of, const int *parent,
                             const int *root_min, int32_t *labels, const rs_dev_status *st)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const uint32_t i = idx[q], c = cell_of[q];
    if (dev_is_torn(st)) return;
    labels[i] = root_min[parent[c]];
}

__global__ void k_fof_count_roots(const uint32_t *n_cells_p, const int *parent, unsigned long long *count)
{
    const int64_t M = *n_cells_p;
    unsigned long long c = 0;
    for (int64_t A = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; A < M; A += (int64_t)gridDim.x * blockDim.x)
        c += parent[A] == (int)A ? 1ull : 0ull;
    c = warp_sum(c);
    if (lane_id() == 0 && c) atomicAdd(count, c);
}

// Tie-band census: every pair (i < j in sorted order) within the fine-cell
// reach whose float64 distance satisfies |d - l| <= 1e-6 l.
__global__ void __launch_bounds__(FOF_THREADS) k_fof_tieband(const uint32_t *n_cells_p, const uint64_t *cell_key,
                                                               const uint32_t *cell_start, const uint32_t *table,
                                                               const uint64_t *occ, const float4 *spos, FofGeom g,
                                                               unsigned long long *count)
{
    const int64_t M = *n_cells_p;
    const float flo = (float)(g.l2 * (1.0 - 4e-6)), fhi = (float)(g.l2 * (1.0 + 4e-6));
    unsigned long long c = 0;
    for (int64_t A = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; A < M; A += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t ka = cell_key[A], ca = ka >> 6;
        const int sa = (int)(ka & 63), ux = sa & 3, uy = (sa >> 2) & 3, uz = sa >> 4;
        int ccx, ccy, ccz;
        coarse_coords(ca, g.Gc, ccx, ccy, ccz);
        const int ax = 4 * ccx + ux, ay = 4 * ccy + uy, az = 4 * ccz + uz;
        const uint32_t a0 = cell_start[A], a1 = cell_start[A + 1];
        const int lox = ux < 2 ? -1 : 0, loy = uy < 2 ? -1 : 0, loz = uz < 2 ? -1 : 0;
        for (int dz = loz; dz <= loz + 1; dz++)
            for (int dy = loy; dy <= loy + 1; dy++)
                for (int dx = lox; dx <= lox + 1; dx++) {
                    int cx = ccx + dx, cy = ccy + dy, cz = ccz + dz;
                    cx = cx < 0 ? cx + g.Gc : (cx >= g.Gc ? cx - g.Gc : cx);
                    cy = cy < 0 ? cy + g.Gc : (cy >= g.Gc ? cy - g.Gc : cy);
                    cz = cz < 0 ? cz + g.Gc : (cz >= g.Gc ? cz - g.Gc : cz);
                    const uint64_t cc = ((uint64_t)cz * g.Gc + cy) * g.Gc + cx;
                    if (cc < ca) continue;
                    const uint32_t b0c = table[cc];
                    if (b0c == 0xffffffffu) continue;
                    const uint64_t om = occ[b0c];
                    uint64_t cand = om & reach_mask(ux, uy, uz, dx, dy, dz, 2);
                    if (cc == ca) cand &= ~((1ull << sa) - 1ull);  // A itself and the sub-cells after it
                    while (cand) {
                        const int sb = __ffsll((long long)cand) - 1;
                        cand &= cand - 1ull;
                        const int64_t B = (int64_t)b0c + __popcll(om & ((1ull << sb) - 1ull));
                        const int bx = 4 * cx + (sb & 3), by = 4 * cy + ((sb >> 2) & 3), bz = 4 * cz + (sb >> 4);
                        int sx, sy, sz;
                        fine_offset(ax, bx, g.Gf, sx);
                        fine_offset(ay, by, g.Gf, sy);
                        fine_offset(az, bz, g.Gf, sz);
                        for (uint32_t i = a0; i < a1; i++) {
                            const float4 pa = spos[i];
                            for (uint32_t j = (B == A ? i + 1 : cell_start[B]); j < cell_start[B + 1]; j++) {
                                const float4 pb = spos[j];
                                float ddx = sdiff(pa.x, pb.x, sx, g.boxf), ddy = sdiff(pa.y, pb.y, sy, g.boxf),
                                      ddz = sdiff(pa.z, pb.z, sz, g.boxf);
                                float d2 = ddx * ddx + ddy * ddy + ddz * ddz;
                                if (d2 < flo || d2 > fhi) continue;
                                double ex = ddiff(pa.x, pb.x, sx, g.box), ey = ddiff(pa.y, pb.y, sy, g.box),
                                       ez = ddiff(pa.z, pb.z, sz, g.box);
                                double d = sqrt(f64_add(f64_add(f64_mul(ex, ex), f64_mul(ey, ey)), f64_mul(ez, ez)));
                                if (fabs(d - g.l) <= 1e-6 * g.l) c++;
                            }
                        }
                    }
                }
    }
    c = warp_sum(c);
    if (lane_id() == 0 && c) atomicAdd(count, c);
}

// ---- accelerated variant (Sec. 3.1) ----
// The paper's faster FOF visits particles one by one: a particle with more
// than dense_n neighbours within l joins every particle within 2l, and its
// neighbours skip their own search.  Taking the visit order to be the
// particle index, the groups have a closed form that needs no order: call a
// dense particle a centre when no centre of smaller index lies within l (the
// index-greedy maximal independent set of the dense particles); the groups
// are the components of the plain FOF graph plus an edge from every centre
// to every particle within 2l of it (a skipped particle lies within l of a
// centre, so its own FOF edges end within 2l of that centre).  So the plain
// FOF runs first, then: neighbour counts up to dense_n + 1; rounds that
// decide the centres (a dense particle becomes a centre once every dense
// neighbour of smaller index is decided and none is a centre, and drops out
// once one is a centre); and the 2l joins of the centres' fine cells.
//
// The rounds work on fine cells, not on particles.  A cell's particles are
// mutual neighbours in index order, so only its first undecided particle (its
// head) can be decided, and a centre settles the whole cell.  A cell's state
// is one 64-bit word, (head, centre + 1), written and read whole.  A round has
// two kernels: one decides the heads of the unsettled cells, a warp a cell,
// seeing a neighbouring cell through its word and its particles from its head
// up to the own index; one lets each new centre mark the particles within l
// as out, once per centre.  Bound by the dependent loads of the cell walks.
// Before, a round went over every particle and scanned all neighbours of the
// undecided ones: 14 rounds of 1.16 ms at 2M particles, now 8 of 0.16 ms (a
// thread walking a cell's heads one after another in one launch instead took
// 100 ms: the cores' cells hold thousands).  The whole call takes 4.0 ms
// instead of 18 to 21 at 2M particles, 201 instead of 1128 at 134M.
// Calls f(B, b0, b1, sx, sy, sz) for every occupied fine cell B within R fine
// cells per axis of the fine cell at fine coordinates (ax, ay, az) (coarse
// cell (ccx, ccy, ccz), sub-cell (ux, uy, uz)), with B's particle range and
// the periodic shifts; stops when f returns true.  Visits the 27 coarse
// cells around the query's, which hold every fine cell within R <= 4.
template <typename F>
__device__ __forceinline__ void acc_cells(int ccx, int ccy, int ccz, int ux, int uy, int uz, int R,
                                          const uint32_t *cell_start, const uint32_t *table, const uint64_t *occ,
                                          const FofGeom &g, F f)
{
    const int ax = 4 * ccx + ux, ay = 4 * ccy + uy, az = 4 * ccz + uz;
    for (int dz = -1; dz <= 1; dz++)
        for (int dy = -1; dy <= 1; dy++)
            for (int dx = -1; dx <= 1; dx++) {
                uint64_t cand = reach_mask(ux, uy, uz, dx, dy, dz, R);
                if (!cand) continue;
                int cx = ccx + dx, cy = ccy + dy, cz = ccz + dz;
                cx = cx < 0 ? cx + g.Gc : (cx >= g.Gc ? cx - g.Gc : cx);
                cy = cy < 0 ? cy + g.Gc : (cy >= g.Gc ? cy - g.Gc : cy);
                cz = cz < 0 ? cz + g.Gc : (cz >= g.Gc ? cz - g.Gc : cz);
                const uint64_t cc = ((uint64_t)cz * g.Gc + cy) * g.Gc + cx;
                const uint32_t b0c = table[cc];
                if (b0c == 0xffffffffu) continue;
                const uint64_t om = occ[b0c];
                cand &= om;
                while (cand) {
                    const int sb = __ffsll((long long)cand) - 1;
                    cand &= cand - 1ull;
                    const uint32_t B = b0c + (uint32_t)__popcll(om & ((1ull << sb) - 1ull));
                    const int bx = 4 * cx + (sb & 3), by = 4 * cy + ((sb >> 2) & 3), bz = 4 * cz + (sb >> 4);
                    int sx, sy, sz;
                    fine_offset(ax, bx, g.Gf, sx);
                    fine_offset(ay, by, g.Gf, sy);
                    fine_offset(az, bz, g.Gf, sz);
                    if (f(B, cell_start[B], cell_start[B + 1], sx, sy, sz)) return;
                }
            }
}

__device__ __forceinline__ void acc_where(const uint64_t *cell_key, uint32_t A, const FofGeom &g, int &ccx, int &ccy,
                                          int &ccz, int &ux, int &uy, int &uz)
{
    const uint64_t k = cell_key[A];
    const int sa = (int)(k & 63);
    ux = sa & 3;
    uy = (sa >> 2) & 3;
    uz = sa >> 4;
    coarse_coords(k >> 6, g.Gc, ccx, ccy, ccz);
}

// dense flag of every particle (sorted slot q): more than dense_n others
// within l.  The own fine cell is a clique; other cells are tested pair by
// pair until the count is exceeded.
__global__ void __launch_bounds__(FOF_THREADS) k_acc_count(int64_t n, const uint32_t *cell_of, const uint64_t *cell_key,
                                                           const uint32_t *cell_start, const uint32_t *table,
                                                           const uint64_t *occ, const float4 *spos, FofGeom g,
                                                           int dense_n, uint8_t *dense, const rs_dev_status *st)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n || dev_is_torn(st)) return;
    const uint32_t A = cell_of[q];
    int cnt = (int)(cell_start[A + 1] - cell_start[A]) - 1;
    if (cnt <= dense_n) {
        int ccx, ccy, ccz, ux, uy, uz;
        acc_where(cell_key, A, g, ccx, ccy, ccz, ux, uy, uz);
        const float4 p = spos[q];
        acc_cells(ccx, ccy, ccz, ux, uy, uz, 2, cell_start, table, occ, g,
                  [&](uint32_t B, uint32_t b0, uint32_t b1, int sx, int sy, int sz) {
                      if (B == A) return false;
                      for (uint32_t r = b0; r < b1; r++)
                          if (pair_link(p, spos[r], sx, sy, sz, g) && ++cnt > dense_n) return true;
                      return false;
                  });
    }
    dense[q] = cnt > dense_n ? 1 : 0;
}

__device__ __forceinline__ uint64_t acc_word(uint32_t head, uint32_t centre1) { return (uint64_t)head << 32 | centre1; }

__device__ __forceinline__ uint32_t acc_next(const uint8_t *dense, uint32_t q, uint32_t end)
{
    while (q < end && !dense[q]) q++;
    return q;
}

// every cell's first dense particle; the cells that have one are unsettled
__global__ void k_acc_init(const uint32_t *n_cells_p, const uint32_t *cell_start, const uint8_t *dense, uint64_t *word,
                           uint32_t *list, unsigned *len)
{
    const int64_t M = *n_cells_p;
    for (int64_t wb = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); wb < M;
         wb += (int64_t)gridDim.x * blockDim.x) {
        const int64_t A = wb + lane_id();
        bool open = false;
        if (A < M) {
            const uint32_t end = cell_start[A + 1], h = acc_next(dense, cell_start[A], end);
            word[A] = acc_word(h, 0u);
            open = h < end;
        }
        const unsigned m = __ballot_sync(0xffffffffu, open);
        unsigned base = 0;
        if (lane_id() == 0 && m) base = atomicAdd(len, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (open) list[base + __popc(m & ((1u << lane_id()) - 1u))] = (uint32_t)A;
    }
}

// One round of the centre choice: the head of every listed cell waits (its
// cell goes to the next list) while an undecided dense particle of smaller
// index lies within l, or one that became a centre in this very round, and is
// a centre otherwise.  A warp a cell, a lane two of a coarse cell's sub-cells.
__global__ void __launch_bounds__(FOF_THREADS) k_acc_round(const uint32_t *list, const unsigned *len,
                                                           const uint64_t *cell_key, const uint32_t *cell_start,
                                                           const uint32_t *table, const uint64_t *occ,
                                                           const float4 *spos, const uint32_t *idx, FofGeom g,
                                                           const uint8_t *dense, uint64_t *word, uint32_t *list2,
                                                           unsigned *len2, uint32_t *clist, unsigned *clen)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned n = *len;
    const int lane = lane_id();
    for (unsigned k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += gridDim.x * blockDim.x >> 5) {
        const uint32_t A = list[k], end = cell_start[A + 1];
        uint32_t h = (uint32_t)(__ldcg(&word[A]) >> 32);
        unsigned f = 0;
        while (h < end && !(f = __ballot_sync(FULL, h + lane < end && dense[h + lane] != 0))) h += 32;
        h = f ? h + (uint32_t)__ffs(f) - 1u : end;
        if (lane == 0) __stcg(&word[A], acc_word(h, 0u));
        if (h >= end) continue;  // every particle is out
        int ccx, ccy, ccz, ux, uy, uz;
        acc_where(cell_key, A, g, ccx, ccy, ccz, ux, uy, uz);
        const int ax = 4 * ccx + ux, ay = 4 * ccy + uy, az = 4 * ccz + uz;
        const uint32_t me = idx[h];
        const float4 p = spos[h];
        bool blocked = false;
        for (int c8 = 0; c8 < 8 && !blocked; c8++) {
            const int dx = (ux < 2 ? -1 : 0) + (c8 & 1), dy = (uy < 2 ? -1 : 0) + ((c8 >> 1) & 1),
                      dz = (uz < 2 ? -1 : 0) + (c8 >> 2);
            int cx = ccx + dx, cy = ccy + dy, cz = ccz + dz;
            cx = cx < 0 ? cx + g.Gc : (cx >= g.Gc ? cx - g.Gc : cx);
            cy = cy < 0 ? cy + g.Gc : (cy >= g.Gc ? cy - g.Gc : cy);
            cz = cz < 0 ? cz + g.Gc : (cz >= g.Gc ? cz - g.Gc : cz);
            const uint32_t b0c = table[((uint64_t)cz * g.Gc + cy) * g.Gc + cx];
            if (b0c == 0xffffffffu) continue;
            const uint64_t om = occ[b0c], cand = om & reach_mask(ux, uy, uz, dx, dy, dz, 2);
            bool mine = false;
            for (int sb = lane; sb < 64; sb += 32) {
                if (!((cand >> sb) & 1ull)) continue;
                const uint32_t B = b0c + (uint32_t)__popcll(om & ((1ull << sb) - 1ull));
                if (B == A) continue;
                const uint64_t w = __ldcg(&word[B]);
                const uint32_t c1 = (uint32_t)w, b1 = c1 ? c1 : cell_start[B + 1];
                int sx, sy, sz;
                fine_offset(ax, 4 * cx + (sb & 3), g.Gf, sx);
                fine_offset(ay, 4 * cy + ((sb >> 2) & 3), g.Gf, sy);
                fine_offset(az, 4 * cz + (sb >> 4), g.Gf, sz);
                for (uint32_t r = c1 ? c1 - 1u : (uint32_t)(w >> 32); !mine && r < b1 && idx[r] < me; r++)
                    mine = dense[r] && pair_link(p, spos[r], sx, sy, sz, g);
            }
            blocked = __any_sync(FULL, mine);
        }
        if (lane == 0) {
            if (blocked) {
                list2[atomicAdd(len2, 1u)] = A;
            } else {
                __stcg(&word[A], acc_word(end, h + 1u));
                clist[atomicAdd(clen, 1u)] = A;
            }
        }
    }
}

// the particles within l of the round's centres are out (a centre's own cell
// is settled by its word); a warp a centre, the lanes over a cell's particles
__global__ void __launch_bounds__(FOF_THREADS) k_acc_mark(const uint32_t *clist, const unsigned *clen,
                                                          const uint64_t *cell_key, const uint32_t *cell_start,
                                                          const uint32_t *table, const uint64_t *occ,
                                                          const float4 *spos, FofGeom g, const uint64_t *word,
                                                          uint8_t *dense)
{
    const unsigned n = *clen;
    for (unsigned k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += gridDim.x * blockDim.x >> 5) {
        const uint32_t A = clist[k];
        int ccx, ccy, ccz, ux, uy, uz;
        acc_where(cell_key, A, g, ccx, ccy, ccz, ux, uy, uz);
        const float4 p = spos[(uint32_t)word[A] - 1u];
        acc_cells(ccx, ccy, ccz, ux, uy, uz, 2, cell_start, table, occ, g,
                  [&](uint32_t B, uint32_t, uint32_t b1, int sx, int sy, int sz) {
                      if (B == A) return false;
                      for (uint32_t r = (uint32_t)(word[B] >> 32) + lane_id(); r < b1; r += 32)
                          if (dense[r] && pair_link(p, spos[r], sx, sy, sz, g)) dense[r] = 0;
                      return false;
                  });
    }
}

// every centre joins the fine cells that hold a particle within 2l of it
// (a fine cell is one set already, so one such particle joins it); g2 is the
// geometry with the thresholds of 2l.  A warp takes a centre, a lane two of a
// coarse cell's 64 sub-cells.
__global__ void __launch_bounds__(FOF_THREADS) k_acc_join(const uint32_t *n_cells_p, const uint64_t *cell_key,
                                                          const uint32_t *cell_start, const uint32_t *table,
                                                          const uint64_t *occ, const float4 *spos, FofGeom g2,
                                                          const uint64_t *word, int *parent,
                                                          unsigned long long *centres, rs_dev_status *st)
{
    const unsigned FULL = 0xffffffffu;
    const int64_t M = *n_cells_p;
    const int lane = lane_id();
    for (int64_t wb = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); wb < M;
         wb += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t mine = wb + lane < M ? (uint32_t)word[wb + lane] : 0u;
        unsigned m = __ballot_sync(FULL, mine != 0u);
        if (lane == 0 && m) atomicAdd(centres, (unsigned long long)__popc(m));
        while (m) {
            const int s = __ffs(m) - 1;
            m &= m - 1u;
            const uint32_t A = (uint32_t)(wb + s);
            const float4 p = spos[__shfl_sync(FULL, mine, s) - 1u];
            int ccx, ccy, ccz, ux, uy, uz;
            acc_where(cell_key, A, g2, ccx, ccy, ccz, ux, uy, uz);
            const int ax = 4 * ccx + ux, ay = 4 * ccy + uy, az = 4 * ccz + uz;
            for (int c27 = 0; c27 < 27; c27++) {
                const int dz = c27 / 9 - 1, dy = c27 / 3 % 3 - 1, dx = c27 % 3 - 1;
                int cx = ccx + dx, cy = ccy + dy, cz = ccz + dz;
                cx = cx < 0 ? cx + g2.Gc : (cx >= g2.Gc ? cx - g2.Gc : cx);
                cy = cy < 0 ? cy + g2.Gc : (cy >= g2.Gc ? cy - g2.Gc : cy);
                cz = cz < 0 ? cz + g2.Gc : (cz >= g2.Gc ? cz - g2.Gc : cz);
                const uint32_t b0c = table[((uint64_t)cz * g2.Gc + cy) * g2.Gc + cx];
                if (b0c == 0xffffffffu) continue;
                const uint64_t om = occ[b0c], cand = om & reach_mask(ux, uy, uz, dx, dy, dz, 4);
                for (int sb = lane; sb < 64; sb += 32) {
                    if (!((cand >> sb) & 1ull)) continue;
                    const uint32_t B = b0c + (uint32_t)__popcll(om & ((1ull << sb) - 1ull));
                    if (uf_find(parent, (int)A, st) == uf_find(parent, (int)B, st)) continue;
                    int sx, sy, sz;
                    fine_offset(ax, 4 * cx + (sb & 3), g2.Gf, sx);
                    fine_offset(ay, 4 * cy + ((sb >> 2) & 3), g2.Gf, sy);
                    fine_offset(az, 4 * cz + (sb >> 4), g2.Gf, sz);
                    for (uint32_t r = cell_start[B]; r < cell_start[B + 1]; r++)
                        if (pair_link(p, spos[r], sx, sy, sz, g2)) {
                            uf_union(parent, (int)A, (int)B, st);
                            break;
                        }
                }
                __syncwarp();
            }
        }
    }
}

rs_status fof_geometry(rs_ctx *ctx, int64_t n, double box, double b, FofGeom *g)
{
    // fine side s with sqrt(3) s (1 + 2 err) < l, err = float32 error of the
    // fine-cell coordinate in cell units (2.0001 u Gf)
    const FofGridSize gs = fof_grid_size(n, box, b);
    const double l = gs.l, gf_est = gs.gf_est, err = gs.err, gc = gs.gc;
    if (!(l > 0)) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_fof3d: linking length must be positive");
    if (gc < 3) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_fof3d: box narrower than about seven linking lengths");
    if (gc * gc * gc >= 4294967295.0) return rs_fail(ctx, RS_ERR_TOO_LARGE, "rs_fof3d: more than 2^32 coarse cells");
    g->Gc = (int32_t)gc;
    g->Gf = 4 * g->Gc;
    if (g->Gf > gf_est) return rs_fail(ctx, RS_ERR_INTERNAL, "rs_fof3d: grid estimate");
    // the link kernels look two fine cells per axis around a cell: two
    // friends' fine indices differ by less than 1 + l/s + 2 err, so l/s must
    // not exceed 2 - 2 err.  With s rounded down to box / (4 Gc) this fails
    // only in narrow windows of box/l below 14 (e.g. 6.9-8, 11.55-12).
    if (l * (double)g->Gf / box > 2.0 - 2.0 * err)
        return rs_fail(ctx, RS_ERR_INVALID_ARG,
                       "rs_fof3d: no cell grid fits this box and linking length (cells of side between l/2 and "
                       "l/sqrt(3) that divide the box 4k times); use a box of at least 14 linking lengths");
    g->inv_sf = (float)((double)g->Gf / box);
    g->boxf = (float)box;
    g->box = box;
    g->l = l;
    g->l2 = l * l;
    g->lo32 = (float)(g->l2 * (1.0 - BAND_REL));
    g->hi32 = (float)(g->l2 * (1.0 + BAND_REL));
    if ((double)g->boxf != box) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_fof3d: box must be a float32 value");
    return RS_OK;
}

int key_bits(const FofGeom &g)
{
    uint64_t maxkey = (((uint64_t)g.Gc * g.Gc * g.Gc) << 6);
    int bits = 0;
    while (bits < 64 && (maxkey >> bits) != 0) bits++;
    return bits;
}

}  // namespace

namespace {

constexpr int ACC_MAX_ROUNDS = 1 << 16;  // bound on the centre-choice rounds
constexpr int ACC_BATCH = 4;             // rounds between two looks at how many cells are left

// plain FOF (dense_n < 0) or the accelerated variant (dense_n >= 0)
rs_status fof_run(rs_ctx *ctx, const float *pos, int32_t stride, int64_t n, double box, double b, int32_t dense_n,
                  int32_t *labels, int64_t *n_groups, int64_t *n_tieband, int64_t *n_centres)
{
    if (!ctx) return RS_ERR_INVALID_ARG;
    if (n < 0 || (n > 0 && (!pos || !labels)) || (stride != 3 && stride != 4) || !(box > 0) || !(b > 0))
        return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_fof3d: bad argument");
    if (n >= ((int64_t)1 << 31)) return rs_fail(ctx, RS_ERR_TOO_LARGE, "rs_fof3d: n >= 2^31");
    if (n == 0) {
        if (n_groups) *n_groups = 0;
        if (n_tieband) *n_tieband = 0;
        if (n_centres) *n_centres = 0;
        return RS_OK;
    }
    RsStageGuard running(&ctx->in_fof);
    RsRange range(dense_n >= 0 ? "rs_fof3d_accel" : "rs_fof3d");
    FofGeom g;
    RS_TRY(fof_geometry(ctx, n, box, b, &g));
    const int64_t T = FOF_THREADS;
    const int64_t nb = ceil_div(n, T);
    const int64_t ncoarse = (int64_t)g.Gc * g.Gc * g.Gc;

    RS_WS(ctx, uint64_t, k0, WS_SORT_K0, n);
    RS_WS(ctx, uint64_t, k1, WS_SORT_K1, n);
    RS_WS(ctx, uint32_t, v0, WS_SORT_V0, n);
    RS_WS(ctx, uint32_t, v1, WS_SORT_V1, n);
    RS_WS(ctx, uint32_t, table, WS_FOF_TABLE, ncoarse);
    RS_LAUNCH(ctx, "fof_keys", k_fof_keys, nb, T, 0, pos, stride, n, g, k0, v0, table, ncoarse, ctx->d_status);
    bool alt = false;
    RS_TRY(rs_radix_sort_u64(ctx, k0, k1, v0, v1, n, key_bits(g), &alt, "sort_fof"));
    uint64_t *keys = alt ? k1 : k0;
    uint32_t *idx = alt ? v1 : v0;

    RS_WS(ctx, float4, spos, WS_FOF_POS4, n);
    RS_WS(ctx, uint32_t, misc, WS_FOF_MISC, n + 8);
    uint32_t *n_cells = misc;                                     // device scalar
    unsigned long long *cnt = (unsigned long long *)(misc + 2);  // groups, tie-band pairs
    int *uroot = (int *)(misc + 8);  // common root of each coarse cell between the link passes
    RS_WS(ctx, uint32_t, cell_of, WS_FOF_CELLOF, n);
    RS_WS(ctx, uint32_t, cell_start, WS_FOF_CELLSTART, n + 1);
    RS_WS(ctx, uint64_t, cell_key, WS_FOF_CELLKEY, n);
    RS_WS(ctx, uint64_t, occ, WS_FOF_OCC, n);
    RS_WS(ctx, int, parent, WS_FOF_PARENT, n);
    RS_WS(ctx, int, root_min, WS_FOF_ROOTMIN, n);
    const int64_t ctiles = ceil_div(n, CELL_TILE);
    RsLookback lb;
    RS_TRY(rs_lookback_init(ctx, ctiles, &lb, "fof_cells"));
    RS_LAUNCH(ctx, "fof_cells", k_fof_cells, ctiles, T, 0, pos, stride, n, (const uint64_t *)keys,
              (const uint32_t *)idx, spos, cell_of, cell_start, cell_key, table, occ, parent, root_min, n_cells, lb,
              ctx->d_status);
    const int64_t grid = std::min<int64_t>(nb, (int64_t)ctx->num_sms * ctx->tune.fof_link_ctas_per_sm);
    RS_LAUNCH(ctx, "fof_occ", k_fof_occ, grid, T, 0, n_cells, (const uint64_t *)cell_key, (const uint32_t *)table, occ,
              (const rs_dev_status *)ctx->d_status);
    const int64_t rows = ceil_div(n, 32), warps = (int64_t)ctx->num_sms * 48;
    const bool small = n <= FOF_ONE_PASS;
    int split = 1;
    while (split < 8 && rows * split * 2 <= 2 * warps) split *= 2;
    const int64_t lgrid = split > 1 ? ceil_div(rows * split, T / 32) : grid;
    const bool roots = split == 1;  // the root kernels pay where most warps run more than one row
    for (int pass = small ? 2 : 0; pass < (small ? 3 : 2); pass++) {
        if (pass == 1 && roots) {
            RS_LAUNCH(ctx, "fof_uroot_first", k_fof_uroot_first, grid, T, 0, (const uint32_t *)n_cells,
                      (const uint64_t *)cell_key, (const uint32_t *)table, parent, uroot, ctx->d_status);
            RS_LAUNCH(ctx, "fof_uroot_check", k_fof_uroot_check, grid, T, 0, (const uint32_t *)n_cells,
                      (const uint64_t *)cell_key, (const uint32_t *)table, parent, uroot, ctx->d_status);
        }
        RS_LAUNCH(ctx, "fof_link", k_fof_link, lgrid, T, 0, (const uint32_t *)n_cells, (const uint64_t *)cell_key,
                  (const uint32_t *)cell_start, (const uint32_t *)table, (const uint64_t *)occ, (const float4 *)spos,
                  parent, pass == 1 && roots ? (const int *)uroot : nullptr, g, pass, split, ctx->d_status);
    }
    if (dense_n >= 0) {
        // accelerated variant: dense flags, centre rounds, 2l joins
        const int64_t acc8 = n + ceil_div(3 * n, 2) + ceil_div(n, 8);
        RS_WS(ctx, uint64_t, word, WS_FOF_ACC, acc8 + 20);
        uint32_t *la = (uint32_t *)(word + n), *lb = la + n, *clist = lb + n;
        uint8_t *dense = (uint8_t *)(clist + n);
        // list lengths before and after each of a batch's rounds, each
        // round's new centres, then the number of centres
        unsigned *len = (unsigned *)(word + acc8 + 2), *clen = len + 8;
        unsigned long long *acnt = (unsigned long long *)len + 8;
        RS_LAUNCH(ctx, "fof_acc_count", k_acc_count, nb, T, 0, n, (const uint32_t *)cell_of,
                  (const uint64_t *)cell_key, (const uint32_t *)cell_start, (const uint32_t *)table,
                  (const uint64_t *)occ, (const float4 *)spos, g, (int)dense_n, dense, (const rs_dev_status *)ctx->d_status);
        RS_CUDA(ctx, cudaMemsetAsync(len, 0, 4, ctx->stream));
        RS_LAUNCH(ctx, "fof_acc_init", k_acc_init, grid, T, 0, (const uint32_t *)n_cells,
                  (const uint32_t *)cell_start, (const uint8_t *)dense, word, la, len);
        // the host looks at the length after every ACC_BATCH rounds (a round
        // over an empty list ends at once)
        for (int round = 0;; round += ACC_BATCH) {
            if (round >= ACC_MAX_ROUNDS)
                return rs_fail(ctx, RS_ERR_INTERNAL, "rs_fof3d_accel: the centre choice did not settle");
            RS_CUDA(ctx, cudaMemsetAsync(len + 1, 0, 4 * 15, ctx->stream));
            for (int r = 0; r < ACC_BATCH; r++) {
                RS_LAUNCH(ctx, "fof_acc_round", k_acc_round, std::min<int64_t>(nb, (int64_t)ctx->num_sms * 8), T, 0,
                          (const uint32_t *)la, (const unsigned *)len + r, (const uint64_t *)cell_key,
                          (const uint32_t *)cell_start, (const uint32_t *)table, (const uint64_t *)occ,
                          (const float4 *)spos, (const uint32_t *)idx, g, (const uint8_t *)dense, word, lb,
                          len + r + 1, clist, clen + r);
                RS_LAUNCH(ctx, "fof_acc_mark", k_acc_mark, std::min<int64_t>(nb, (int64_t)ctx->num_sms * 8), T, 0,
                          (const uint32_t *)clist, (const unsigned *)clen + r, (const uint64_t *)cell_key,
                          (const uint32_t *)cell_start, (const uint32_t *)table, (const uint64_t *)occ,
                          (const float4 *)spos, g, (const uint64_t *)word, dense);
                std::swap(la, lb);
            }
            int64_t left = 0;
            RS_TRY(rs_read_i64(ctx, len + ACC_BATCH, 1, &left, "rs_fof3d_accel"));
            if ((left & 0xffffffffll) == 0) break;
            RS_CUDA(ctx, cudaMemcpyAsync(len, len + ACC_BATCH, 4, cudaMemcpyDeviceToDevice, ctx->stream));
        }
        // the same tests at 2l: every threshold scales by exactly 2 or 4
        FofGeom g2 = g;
        g2.l = 2.0 * g.l;
        g2.l2 = 4.0 * g.l2;
        g2.lo32 = 4.0f * g.lo32;
        g2.hi32 = 4.0f * g.hi32;
        RS_CUDA(ctx, cudaMemsetAsync(acnt, 0, sizeof(unsigned long long), ctx->stream));
        RS_LAUNCH(ctx, "fof_acc_join", k_acc_join, grid, T, 0, (const uint32_t *)n_cells, (const uint64_t *)cell_key,
                  (const uint32_t *)cell_start, (const uint32_t *)table, (const uint64_t *)occ, (const float4 *)spos,
                  g2, (const uint64_t *)word, parent, acnt, ctx->d_status);
        if (n_centres) RS_TRY(rs_read_i64(ctx, acnt, 1, n_centres, "rs_fof3d_accel"));
    }
    RS_LAUNCH(ctx, "fof_rootmin", k_fof_rootmin, grid, T, 0, (const uint32_t *)n_cells,
              (const uint32_t *)cell_start, (const uint32_t *)idx, parent, root_min,
              rs_fault("timeout1") ? 1 : RS_SPIN_LIMIT, ctx->d_status);
    RS_LAUNCH(ctx, "fof_labels", k_fof_labels, nb, T, 0, n, (const uint32_t *)idx, (const uint32_t *)cell_of,
              (const int *)parent, (const int *)root_min, labels, (const rs_dev_status *)ctx->d_status);
    if (n_groups || n_tieband) {
        RS_CUDA(ctx, cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), ctx->stream));
        if (n_groups)
            RS_LAUNCH(ctx, "fof_count_roots", k_fof_count_roots, grid, T, 0, (const uint32_t *)n_cells,
                      (const int *)parent, cnt);
        if (n_tieband)
            RS_LAUNCH(ctx, "fof_tieband", k_fof_tieband, grid, T, 0, (const uint32_t *)n_cells,
                      (const uint64_t *)cell_key, (const uint32_t *)cell_start, (const uint32_t *)table,
                      (const uint64_t *)occ, (const float4 *)spos, g, cnt + 1);
        int64_t h[2];
        RS_TRY(rs_read_i64(ctx, cnt, 2, h, "rs_fof3d"));
        if (n_groups) *n_groups = h[0];
        if (n_tieband) *n_tieband = h[1];
    }
    return RS_OK;
}

}  // namespace

extern "C" rs_status rs_fof3d(rs_ctx *ctx, const float *pos, int32_t stride, int64_t n, double box, double b,
                              int32_t *labels, int64_t *n_groups, int64_t *n_tieband)
{
    return fof_run(ctx, pos, stride, n, box, b, -1, labels, n_groups, n_tieband, nullptr);
}

extern "C" rs_status rs_fof3d_accel(rs_ctx *ctx, const float *pos, int32_t stride, int64_t n, double box, double b,
                                    int32_t dense_n, int32_t *labels, int64_t *n_groups, int64_t *n_centres)
{
    if (ctx && dense_n < 0) return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_fof3d_accel: dense_n must be >= 0");
    return fof_run(ctx, pos, stride, n, box, b, dense_n, labels, n_groups, nullptr, n_centres);
}

// ---------------------------------------------------------------------------
// group CSR (App. A work units)
// ---------------------------------------------------------------------------
namespace {

// Members per label besides the label's own particle (which alone makes most
// of a catalogue's groups and needs no count).  A block counts GS_TILE
// particles in a shared hash table before it adds to memory: the members of a
// large group, spread over the catalogue, would otherwise queue on its one
// counter (33M particles: 2.02 -> 0.24 ms).
constexpr int GS_THREADS = 256;
constexpr int GS_TILE = 16384;

__global__ void __launch_bounds__(GS_THREADS) k_gs_count(int64_t n, const int32_t *labels, uint32_t *count,
                                                         rs_dev_status *st)
{
    __shared__ RsBlockCount<uint32_t, 12> C;
    C.clear();
    const int64_t i0 = (int64_t)blockIdx.x * GS_TILE;
    for (int64_t i = i0 + threadIdx.x; i < min(n, i0 + GS_TILE); i += GS_THREADS) {
        const int32_t l = labels[i];
        if (l < 0 || l > i) {
            dev_fail(st, DEV_BADARG, 20, i);
            continue;
        }
        if (l != i) C.add(l, count);
    }
    C.flush(count);
}

// One pass with look-back: the members of groups of >= min_n members, in
// index order, and the groups (numbered by their label, the root's index)
// with their sizes.  The scanned sum packs groups << 31 | members.
constexpr int GS_ROWS = 8;
constexpr int64_t GS_SCAN_TILE = (int64_t)GS_ROWS * GS_THREADS;

__global__ void __launch_bounds__(GS_THREADS) k_gs_select(int64_t n, const int32_t *labels, const uint32_t *count,
                                                          int32_t min_n, uint32_t *members, uint32_t *group,
                                                          int64_t *sizes, int64_t cap, uint32_t *tot, RsLookback lb,
                                                          rs_dev_status *st)
{
    const unsigned FULL = 0xffffffffu;
    const int64_t tile = rs_next_tile(lb);
    const int lane = lane_id();
    const int64_t base = tile * GS_SCAN_TILE + (int64_t)warp_id() * 32 * GS_ROWS;
    unsigned mem[GS_ROWS], root[GS_ROWS];
    uint32_t size[GS_ROWS];
    unsigned long long sum = 0;
#pragma unroll
    for (int j = 0; j < GS_ROWS; j++) {
        const int64_t i = base + 32 * j + lane;
        const int32_t l = i < n ? labels[i] : -1;
        size[j] = l >= 0 && l <= i ? count[l] + 1u : 0u;
        const bool in = size[j] >= (uint32_t)min_n && size[j] > 0u;
        mem[j] = __ballot_sync(FULL, in);
        root[j] = __ballot_sync(FULL, in && l == i);
        sum += (unsigned long long)__popc(root[j]) << 31 | (unsigned)__popc(mem[j]);
    }
    unsigned long long all;
    unsigned long long at = rs_block_scan<GS_THREADS>(lane == 0 ? sum : 0ull, all);
    at = __shfl_sync(FULL, at, 0) + rs_lookback(lb, tile, all, st);
    uint32_t m0 = (uint32_t)(at & 0x7fffffffull), g0 = (uint32_t)(at >> 31);
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < GS_ROWS; j++) {
        const int64_t i = base + 32 * j + lane;
        const uint32_t m = m0 + (uint32_t)__popc(mem[j] & below), g = g0 + (uint32_t)__popc(root[j] & below);
        if (((mem[j] >> lane) & 1u) && m < n) members[m] = (uint32_t)i;
        if ((root[j] >> lane) & 1u) {
            group[i] = g;
            if (g < cap) sizes[g] = size[j];
        }
        m0 += (uint32_t)__popc(mem[j]);
        g0 += (uint32_t)__popc(root[j]);
    }
    if ((tile + 1) * GS_SCAN_TILE >= n && threadIdx.x == GS_THREADS - 1) {
        tot[0] = g0;
        tot[1] = m0;
    }
}

// the members' group numbers
__global__ void k_gs_keys(int64_t m, const uint32_t *members, const int32_t *labels, const uint32_t *group,
                          uint32_t *keys)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < m) keys[p] = group[labels[members[p]]];
}

}  // namespace

extern "C" rs_status rs_group_sort(rs_ctx *ctx, const int32_t *labels, int64_t n, int32_t min_n, int32_t *perm,
                                   int64_t *offsets, int64_t offsets_cap, int64_t *n_groups, int64_t *n_members)
{
    if (!ctx) return RS_ERR_INVALID_ARG;
    if (n < 0 || !n_groups || !n_members || min_n < 1 || offsets_cap < 1 || !offsets ||
        (n > 0 && (!labels || !perm)))
        return rs_fail(ctx, RS_ERR_INVALID_ARG, "rs_group_sort: bad argument");
    if (n >= ((int64_t)1 << 31)) return rs_fail(ctx, RS_ERR_TOO_LARGE, "rs_group_sort: n >= 2^31");
    if (n == 0) {
        *n_groups = 0;
        *n_members = 0;
        RS_CUDA(ctx, cudaMemsetAsync(offsets, 0, sizeof(int64_t), ctx->stream));
        return RS_OK;
    }
    RsStageGuard running(&ctx->in_gs);
    RsRange range("rs_group_sort");
    RS_WS(ctx, uint32_t, count, WS_GS_COUNT, n);
    RS_WS(ctx, uint32_t, fl, WS_GS_FLAG, n + 8);
    uint32_t *tot = fl, *group = fl + 8;  // tot: groups, members
    RS_CUDA(ctx, cudaMemsetAsync(count, 0, sizeof(uint32_t) * n, ctx->stream));
    RS_LAUNCH(ctx, "gs_count", k_gs_count, ceil_div(n, GS_TILE), GS_THREADS, 0, n, labels, count, ctx->d_status);
    const int64_t tiles = ceil_div(n, GS_SCAN_TILE);
    RsLookback lb;
    RS_TRY(rs_lookback_init(ctx, tiles, &lb, "gs_select"));
    RS_LAUNCH(ctx, "gs_select", k_gs_select, tiles, GS_THREADS, 0, n, labels, (const uint32_t *)count, min_n,
              (uint32_t *)perm, group, offsets, offsets_cap, tot, lb, ctx->d_status);
    uint32_t h2[2];
    RS_CUDA(ctx, cudaMemcpyAsync(ctx->h_scratch, tot, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, ctx->stream));
    RS_TRY(rs_sync_check(ctx, "rs_group_sort"));
    memcpy(h2, ctx->h_scratch, sizeof h2);
    const int64_t G = h2[0], Mm = h2[1];
    *n_groups = G;
    *n_members = Mm;
    if (offsets_cap < G + 1) return rs_fail(ctx, RS_ERR_INTERNAL, "rs_group_sort: offsets capacity too small");
    RS_WS(ctx, uint64_t, kbuf, WS_SORT_K0, 2 * Mm);  // reused as two u32 key arrays
    uint32_t *k0 = (uint32_t *)kbuf, *k1 = (uint32_t *)kbuf + Mm;
    RS_WS(ctx, uint32_t, vtmp, WS_SORT_V1, Mm);
    uint32_t *v0 = (uint32_t *)perm;
    RS_LAUNCH(ctx, "gs_keys", k_gs_keys, ceil_div(Mm, 256), 256, 0, Mm, (const uint32_t *)v0, labels,
              (const uint32_t *)group, k0);
    int bits = 0;
    while (bits < 32 && ((uint64_t)(G > 0 ? G - 1 : 0) >> bits) != 0) bits++;
    bool alt = false;
    RS_TRY(rs_radix_sort_u32(ctx, k0, k1, v0, vtmp, Mm, bits, &alt, "sort_gs"));
    if (alt)
        RS_CUDA(ctx, cudaMemcpyAsync(perm, vtmp, sizeof(uint32_t) * Mm, cudaMemcpyDeviceToDevice, ctx->stream));
    RS_CUDA(ctx, cudaMemsetAsync(offsets + G, 0, sizeof(int64_t), ctx->stream));
    RS_TRY(rs_scan_i64(ctx, offsets, G + 1, nullptr, "scan_gs"));
    return rs_sync_check(ctx, "rs_group_sort");
}
