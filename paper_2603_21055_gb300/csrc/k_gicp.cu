// Geometric tracking (Sec. 3.3, Eq. 2): geometry Gaussians of a depth map, a spatial hash
// grid of the global set, point-to-surface correspondences, the GICP Gauss-Newton system
// and its solve, and the map update. The operations, readings and layouts are stated in
// include/sgad_gicp.h.
//
// Where floating point decides an integer (neighbour ranks, correspondences, overlaps)
// the kernels use explicitly rounded FP32 operations (__fmul_rn, __fadd_rn, ...) in a
// fixed order, so the decision does not depend on the compiler's contraction choices.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstring>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "sgad_gicp.h"
#include "sgad_launch.cuh"

namespace sgad {
sgad_status report_error(sgad_status code, const char *msg);
}

namespace {

using sgad::report_error;

constexpr int kSys = 29;                 // H upper triangle (21), g (6), cost, count
constexpr int kSelBlock = 1024;          // cells per selection block (4 per thread)
constexpr int kMaxSelBlocks = 16384;     // selection grids of up to 16.7 M cells
constexpr int kRowPts = 16;              // source points of one row of partial sums
constexpr int kStepThreads = 32 * kRowPts;   // correspondence step: one warp per point of a row
constexpr int kMaxRows = 4 * 152;        // rows of partial sums; more points share the rows
constexpr int kInsThreads = 256;         // map-update kernels
constexpr int kInsPts = 64;              // source points per block of the overlap test
constexpr int kKMatchMax = 8;

struct GicpState {
    double pose[12];
    float posef[12];
    double cost, step;
    int32_t iters, done, converged, n, status, max_iters;
    float tol;
    int32_t map_old, ins_total;
    int32_t blocks_done;     // step blocks finished in the current iteration
    uint32_t sync;           // grid-wide steps completed (the tracking kernel waits on it)
    int32_t gave_up;         // 1: a wait of the last track ended without the others. A word of its own,
                             // which the next frame does not clear: a caller may read the state of a
                             // track while the next frame is selected
    int32_t level;           // cell size of the map's index (see kLevels); the next build starts with it
};

struct GLayout {
    size_t state, sel_counts, hash_head, hash_pts, knn_head, knn_pts, partial, ins_flags, ins_counts, total;
    int32_t table, knn_table, max_blocks, rows;
};

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

int32_t table_for(int32_t cap)
{
    int32_t t = 1024;
    while (t < 2 * cap && t < (1 << 24)) t <<= 1;
    return t;
}

// Every call computes the same layout from the parameters (capacities included).
GLayout glayout(const sgad_gicp_params &p)
{
    GLayout L;
    L.table = table_for(p.map_capacity);
    L.knn_table = table_for(p.src_capacity);
    L.max_blocks = (p.src_capacity + kInsThreads - 1) / kInsThreads;
    // rows of 16 points each; points beyond kMaxRows rows are added to the rows in turn (the
    // solve sums one partial row per 16 points)
    L.rows = std::min((p.src_capacity + kRowPts - 1) / kRowPts, kMaxRows);
    size_t o = 0;
    const auto take = [&o](size_t bytes) {
        const size_t at = o;
        o = a256(o + bytes);
        return at;
    };
    L.state = take(sizeof(GicpState));
    L.sel_counts = take((size_t)kMaxSelBlocks * sizeof(int32_t));
    L.hash_head = take(((size_t)L.table + 1) * sizeof(int32_t));      // and the occupied buckets
    L.hash_pts = take((size_t)p.map_capacity * sizeof(float4));
    L.knn_head = take((size_t)L.knn_table * sizeof(int32_t));
    L.knn_pts = take((size_t)p.src_capacity * sizeof(float4));
    L.partial = take((size_t)L.rows * 32 * sizeof(float));
    L.ins_flags = take((size_t)p.src_capacity * sizeof(int32_t));
    L.ins_counts = take(((size_t)p.src_capacity / kInsPts + 2) * sizeof(int32_t));
    L.total = o;
    return L;
}

// ------------------------------------------------------------------ device helpers
struct Pose12 {
    float p[12];
};
struct PoseD {
    double p[12];
};

__device__ __forceinline__ float3 transform(const float *P, float4 a)
{
    float3 x;
    x.x = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[0], a.x), __fmul_rn(P[1], a.y)), __fmul_rn(P[2], a.z)), P[3]);
    x.y = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[4], a.x), __fmul_rn(P[5], a.y)), __fmul_rn(P[6], a.z)), P[7]);
    x.z = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[8], a.x), __fmul_rn(P[9], a.y)), __fmul_rn(P[10], a.z)), P[11]);
    return x;
}

// ((dx dx + dy dy) + dz dz), d = b - a, explicitly rounded
__device__ __forceinline__ float sqdist(float bx, float by, float bz, float ax, float ay, float az)
{
    const float dx = __fsub_rn(bx, ax), dy = __fsub_rn(by, ay), dz = __fsub_rn(bz, az);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

__device__ __forceinline__ int cell_of(float x, float inv_cell) { return (int)floorf(__fmul_rn(x, inv_cell)); }

// Spatial hash of a cell (Teschner et al. 2003: XOR of the coordinates times three
// large primes), masked to the power-of-two table.
__device__ __forceinline__ uint32_t cell_hash(int ix, int iy, int iz, uint32_t mask)
{
    return (((uint32_t)ix * 73856093u) ^ ((uint32_t)iy * 19349663u) ^ ((uint32_t)iz * 83492791u)) & mask;
}

// Symmetric 3x3 eigen-decomposition by cyclic Jacobi rotations (the symmetric Schur
// method, Golub & Van Loan Sec. 8.5): A (row-major, symmetric) -> eigenvalues w
// ascending, eigenvectors as the columns of V.
__device__ __forceinline__ void eig3(float A[3][3], float w[3], float V[3][3])
{
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) V[r][c] = r == c ? 1.f : 0.f;
#pragma unroll 1
    for (int sweep = 0; sweep < 8; ++sweep) {
        const float off = fabsf(A[0][1]) + fabsf(A[0][2]) + fabsf(A[1][2]);
        const float scale = fabsf(A[0][0]) + fabsf(A[1][1]) + fabsf(A[2][2]);
        if (off <= 1e-9f * scale || off == 0.f) break;
#pragma unroll
        for (int pq = 0; pq < 3; ++pq) {
            const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2;
            const float apq = A[p][q];
            if (apq == 0.f) continue;
            const float theta = (A[q][q] - A[p][p]) / (2.f * apq);
            const float t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
            const float c = rsqrtf(t * t + 1.f), s = t * c;
            // A <- J^T A J with J the rotation in the (p, q) plane
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float akp = A[k][p], akq = A[k][q];
                A[k][p] = c * akp - s * akq;
                A[k][q] = s * akp + c * akq;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float apk = A[p][k], aqk = A[q][k];
                A[p][k] = c * apk - s * aqk;
                A[q][k] = s * apk + c * aqk;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float vkp = V[k][p], vkq = V[k][q];
                V[k][p] = c * vkp - s * vkq;
                V[k][q] = s * vkp + c * vkq;
            }
        }
    }
    w[0] = A[0][0];
    w[1] = A[1][1];
    w[2] = A[2][2];
    // sort ascending with the vectors
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2 - a; ++b)
            if (w[b] > w[b + 1]) {
                const float tw = w[b];
                w[b] = w[b + 1];
                w[b + 1] = tw;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float tv = V[k][b];
                    V[k][b] = V[k][b + 1];
                    V[k][b + 1] = tv;
                }
            }
}

// Inverse of a symmetric 3x3 (xx, xy, xz, yy, yz, zz) by its adjugate.
__device__ __forceinline__ void inv_sym3(const float S[6], float M[6])
{
    const float a = S[0], b = S[1], c = S[2], d = S[3], e = S[4], f = S[5];
    const float A = d * f - e * e, B = c * e - b * f, C = b * e - c * d;
    const float det = a * A + b * B + c * C;
    const float r = 1.f / det;
    M[0] = A * r;
    M[1] = B * r;
    M[2] = C * r;
    M[3] = (a * f - c * c) * r;
    M[4] = (b * c - a * e) * r;
    M[5] = (a * d - b * b) * r;
}

// Exclusive prefix of per-block counts [0, upto) summed by the whole block.
__device__ int block_prefix(const int32_t *counts, int upto, int *red)
{
    int s = 0;
    for (int k = threadIdx.x; k < upto; k += blockDim.x) s += counts[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    int tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    __syncthreads();
    return tot;
}

// Exclusive scan of one int per thread across the block; returns the block total in *total.
__device__ int block_exclusive_scan(int v, int *red, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) red[warp] = x;
    __syncthreads();
    int base = 0, tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        if (w < warp) base += red[w];
        tot += red[w];
    }
    __syncthreads();
    *total = tot;
    return base + x - v;
}

}  // namespace

namespace {

// ------------------------------------------------------------------ selection
struct SelArgs {
    const float *depth;
    int32_t W, H, R, ncx, ncells;
    float fx, fy, cx, cy;
    float4 *pos;
    int32_t *pix;
    int32_t *count;
    int32_t capacity;
    int32_t *blk;
    int32_t *cell_point;     // [ncells] point of a cell or -1, or null
    int32_t *point_cell;     // [capacity] cell of a point (with cell_point)
    GicpState *state;
};

__device__ __forceinline__ bool cell_valid(const SelArgs &a, int c, int *u, int *v, float *d)
{
    if (c >= a.ncells) return false;
    const int cy = c / a.ncx, cx = c - cy * a.ncx;
    *u = cx * a.R;
    *v = cy * a.R;
    *d = a.depth[(size_t)(*v) * a.W + *u];
    return *d > 0.f;
}

__global__ void __launch_bounds__(256) k_select_count(const __grid_constant__ SelArgs a)
{
    sgad::dependency_wait();
    __shared__ int red[8];
    if (blockIdx.x == 0 && threadIdx.x == 0) a.state->status = 0;   // a new frame: fresh flags
    int n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int u, v;
        float d;
        n += cell_valid(a, blockIdx.x * kSelBlock + threadIdx.x * 4 + k, &u, &v, &d) ? 1 : 0;
    }
    int total;
    block_exclusive_scan(n, red, &total);
    if (threadIdx.x == 0) a.blk[blockIdx.x] = total;
}

__global__ void __launch_bounds__(256) k_select_write(const __grid_constant__ SelArgs a)
{
    sgad::dependency_wait();
    __shared__ int red[8];
    const int prefix = block_prefix(a.blk, blockIdx.x, red);
    int u[4], v[4];
    float d[4];
    bool ok[4];
    int n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        ok[k] = cell_valid(a, blockIdx.x * kSelBlock + threadIdx.x * 4 + k, &u[k], &v[k], &d[k]);
        n += ok[k] ? 1 : 0;
    }
    int total;
    int o = prefix + block_exclusive_scan(n, red, &total);
    bool over = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = blockIdx.x * kSelBlock + threadIdx.x * 4 + k;
        if (a.cell_point && c < a.ncells) a.cell_point[c] = ok[k] && o < a.capacity ? o : -1;
        if (!ok[k]) continue;
        if (o < a.capacity) {
            // p = d ((u - cx) / fx, (v - cy) / fy, 1), each step rounded as written
            const float x = __fmul_rn(d[k], __fdiv_rn(__fsub_rn((float)u[k], a.cx), a.fx));
            const float y = __fmul_rn(d[k], __fdiv_rn(__fsub_rn((float)v[k], a.cy), a.fy));
            a.pos[o] = make_float4(x, y, d[k], 0.f);
            if (a.pix) a.pix[o] = v[k] * a.W + u[k];
            if (a.cell_point) a.point_cell[o] = c;
        } else {
            over = true;
        }
        ++o;
    }
    if (over) atomicOr(&a.state->status, 1);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *a.count = min(prefix + total, a.capacity);
}

// ------------------------------------------------------------------ neighbour search
// A search runs one query per warp. Its result is the list of the nearest points as 64-bit
// keys (bits of the squared distance << 32 | index), ascending over the lanes: lane k holds
// the (k + 1)-th nearest, ~0 past the last found, so the order is by distance, then index.
// A search is a chain of dependent loads, so a warp's 32 lanes load as many cells at once
// as they can; with 8 lanes per query and the cells of a ring in turn the first step of a
// track took 103 us at 8,160 points, half of it a tail of a few slow queries.
constexpr unsigned kFull = 0xffffffffu;
constexpr uint64_t kNone = ~0ull;
constexpr int kRings = 6;                // rings searched before the exhaustive pass

// Cell sizes of the map's index: half to a sixth of the larger search radius R, so that as many
// rings of cells as kDivisor prove a search of that radius. Half of it where a cell holds few
// points (cells of a third took 343 to reach as far, most of them empty at the 2-8 cm spacing of
// most maps' points). A chain is walked by one lane, so of a dense map, whose searches end in
// the first ring, smaller cells are linked (k_hash_relink). 640x480 frames at R = 0.1 m, a
// sequence's time per frame with cells of R / 2 alone and with these: stride 1 (307,200 points,
// 190 in a cell of R / 2) 64 and 24 ms, stride 2 at R = 0.3 23.6 and 4.7, stride 3 at 0.3 3.5 and
// 1.6, stride 5 at 0.6 1.20 and 0.50, stride 10 0.28 and 0.27.
constexpr int kLevels = 4;
__device__ constexpr int kDivisor[kLevels] = {2, 3, 4, 6};
constexpr int kMaxRings = 6;

struct Grid {
    const int32_t *head;      // [table] first point of a bucket's chain + 1, 0: empty
    const float4 *pts;        // [cap] x, y, z, next point of the chain + 1 (bits)
    float inv_cell, cell;
    uint32_t mask;
    int32_t cap;
    int32_t divisor;          // of the map's index
};

// The map's index as the last build left it: level 0's grid and the cells of every level.
struct MapGrid {
    Grid g;
    float cell[kLevels], inv_cell[kLevels];
};

__device__ __forceinline__ int valid_level(int l) { return l >= 0 && l < kLevels ? l : 0; }

__device__ __forceinline__ Grid grid_at(const MapGrid &m, int level)
{
    Grid g = m.g;
#pragma unroll
    for (int l = 1; l < kLevels; ++l)
        if (level == l) {
            g.cell = m.cell[l];
            g.inv_cell = m.inv_cell[l];
            g.divisor = kDivisor[l];
        }
    return g;
}

__device__ __forceinline__ uint64_t pack_key(float d, int j)
{
    return ((uint64_t)__float_as_uint(d) << 32) | (uint32_t)j;
}
__device__ __forceinline__ float key_dist(uint64_t k) { return __uint_as_float((uint32_t)(k >> 32)); }

// Compare-exchange with the lane `o` away: the lane keeps the smaller key if `low`.
__device__ __forceinline__ uint64_t exchange(uint64_t k, int o, bool low)
{
    const uint64_t y = __shfl_xor_sync(kFull, k, o);
    return (k < y) == low ? k : y;
}

// Takes the lanes' new keys c (kNone: none) into the sorted list `best`, of which the
// `keep` smallest are wanted. Keys are unique (every point is seen once). A few keys are
// shifted in one by one (~100 cycles each); more are sorted across the lanes (a bitonic
// network, 15 exchanges) and merged (the smaller of the list and the reversed keys is
// bitonic and holds the 32 smallest: 5 exchanges).
__device__ __forceinline__ void warp_insert(uint64_t &best, uint64_t c, int keep)
{
    const int lane = threadIdx.x & 31;
    const uint64_t worst = __shfl_sync(kFull, best, keep - 1);
    unsigned m = __ballot_sync(kFull, c < worst);
    if (__popc(m) > 8) {
#pragma unroll
        for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
            for (int o = size >> 1; o > 0; o >>= 1) c = exchange(c, o, ((lane & size) == 0) == ((lane & o) == 0));
        const uint64_t r = __shfl_xor_sync(kFull, c, 31);
        best = r < best ? r : best;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = exchange(best, o, (lane & o) == 0);
        return;
    }
    while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const uint64_t v = __shfl_sync(kFull, c, src);
        const int p = __popc(__ballot_sync(kFull, best < v));
        const uint64_t up = __shfl_up_sync(kFull, best, 1);
        best = lane < p ? best : (lane == p ? v : up);
    }
}

// Walks the chains of the lanes' buckets (first point + 1 = e) in step and calls
// f(point, index), index -1 for a lane whose point is none or lies in another cell than
// (cx, cy, cz), with the whole warp. Indexes are checked and the steps bounded by the
// capacity.
template <typename F>
__device__ __forceinline__ void walk_chain(const Grid &g, int e, float4 q, int cx, int cy, int cz, F &&f)
{
    for (int t = 0; t <= g.cap && __any_sync(kFull, e > 0); ++t) {
        int i = -1, next = 0;
        if (e > 0) {
            if (cell_of(q.x, g.inv_cell) == cx && cell_of(q.y, g.inv_cell) == cy && cell_of(q.z, g.inv_cell) == cz)
                i = e - 1;
            next = __float_as_int(q.w);
        }
        next = next > 0 && next <= g.cap ? next : 0;
        float4 qn = q;
        if (next) qn = g.pts[next - 1];                        // on its way during f
        f(q, i);
        e = next;
        q = qn;
    }
}

// The cells at Chebyshev distance R around x's cell (BALL: at most R), 32 at a time; four
// of a lane's bucket heads are loaded together, then their first points. f(point, index, -1
// for a lane without one) is called by the whole warp.
template <int R, bool BALL, typename F>
__device__ __forceinline__ void ring_walk(const Grid &g, float3 x, F &&f)
{
    constexpr int side = 2 * R + 1, ncube = side * side * side;
    constexpr int kAhead = ncube > 32 ? 4 : 1;
    const int lane = threadIdx.x & 31;
    const int ix = cell_of(x.x, g.inv_cell), iy = cell_of(x.y, g.inv_cell), iz = cell_of(x.z, g.inv_cell);
#pragma unroll 1
    for (int c0 = 0; c0 < ncube; c0 += 32 * kAhead) {
        int e[kAhead];
        float4 q[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int c = c0 + 32 * u + lane;
            const int dx = c % side - R, dy = (c / side) % side - R, dz = c / (side * side) - R;
            const bool on = c < ncube && (BALL || max(abs(dx), max(abs(dy), abs(dz))) == R);
            const int h = on ? g.head[cell_hash(ix + dx, iy + dy, iz + dz, g.mask)] : 0;
            e[u] = h > 0 && h <= g.cap ? h : 0;
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) q[u] = e[u] ? g.pts[e[u] - 1] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int c = c0 + 32 * u + lane;
            const int dx = c % side - R, dy = (c / side) % side - R, dz = c / (side * side) - R;
            walk_chain(g, e[u], q[u], ix + dx, iy + dy, iz + dz, f);
        }
    }
}

template <int R, bool BALL, typename F>
__device__ __forceinline__ void ring_cells(const Grid &g, float3 x, F &&f)
{
    ring_walk<R, BALL>(g, x, [&](float4 q, int i) {
        if (i >= 0) f(q);
    });
}

// Ring r (r = 1: with the cell itself) into the sorted list. The points found are gathered
// in `buf` (64 keys of shared memory of the warp) and taken 32 at a time: a step along the
// chains finds a few points, and taking them in step by step was most of the search.
__device__ __forceinline__ void search_ring(const Grid &g, float3 x, int r, int keep, uint64_t &best, uint64_t *buf)
{
    const int lane = threadIdx.x & 31;
    uint64_t worst = __shfl_sync(kFull, best, keep - 1);
    int cnt = 0;
    const auto take = [&](float4 q, int i) {
        uint64_t c = kNone;
        if (i >= 0) {
            const float d = sqdist(q.x, q.y, q.z, x.x, x.y, x.z);
            if (d <= FLT_MAX) c = pack_key(d, i);
        }
        const unsigned m = __ballot_sync(kFull, c < worst);
        if (m == 0u) return;
        if (c < worst) buf[cnt + __popc(m & ((1u << lane) - 1u))] = c;
        cnt += __popc(m);
        if (cnt >= 32) {
            __syncwarp();
            const uint64_t k = buf[lane], rest = buf[32 + lane];
            __syncwarp();
            cnt -= 32;
            if (lane < cnt) buf[lane] = rest;
            warp_insert(best, k, keep);
            worst = __shfl_sync(kFull, best, keep - 1);
        }
    };
    switch (r) {
    case 1: ring_walk<1, true>(g, x, take); break;
    case 2: ring_walk<2, false>(g, x, take); break;
    case 3: ring_walk<3, false>(g, x, take); break;
    case 4: ring_walk<4, false>(g, x, take); break;
    case 5: ring_walk<5, false>(g, x, take); break;
    default: ring_walk<6, false>(g, x, take); break;
    }
    __syncwarp();
    const uint64_t k = lane < cnt ? buf[lane] : kNone;
    __syncwarp();
    warp_insert(best, k, keep);
}

// ------------------------------------------------------------------ shapes
// One warp per selected point: its K_c nearest selected points (FP32 squared distance,
// ties by index) and their covariance, kShapeRounds points in turn; then the block's first
// warp, a point per lane, takes the eigen-decompositions and writes the normalised shapes
// (a decomposition is ~1,400 dependent instructions, the same for a warp of one point or
// of 32).
constexpr int kShapeRounds = 2;
constexpr int kShapeThreads = 512;
constexpr int kShapePts = kShapeThreads / 32 * kShapeRounds;
static_assert(kShapePts == 32, "one point per lane of the block's first warp");

// The selection grid: cell (cu, cv) is the pixel (cu R, cv R), whose ray is
// (x0 + cu step_x, y0 + cv step_y, 1).
struct Window {
    const int32_t *point_cell, *cell_point;
    int32_t ncx, ncy;
    float step_x, step_y, x0, y0;
};

struct ShapeArgs {
    const float4 *pos;
    const int32_t *count;
    float4 *cov, *normal;
    int32_t *knn_out;
    int32_t K;
    float eps;
    Window w;
    Grid g;
};

// Distance from the point at depth d on the ray slope r to the nearest ray with a slope
// between r + a and r + b (both on one side of r): a point of such a ray lies in the plane
// through the centre with its slope s, at d |s - r| / sqrt(1 + s^2), which has no minimum
// inside the interval (it rises while 1 + r s > 0 and falls after).
__device__ __forceinline__ float slope_gap(float d, float r, float a, float b)
{
    return d * fminf(fabsf(a) * rsqrtf(1.f + (r + a) * (r + a)), fabsf(b) * rsqrtf(1.f + (r + b) * (r + b)));
}

// Every point.
__device__ __forceinline__ uint64_t all_nearest(const ShapeArgs &a, float4 me, int n, int K)
{
    const int lane = threadIdx.x & 31;
    uint64_t best = kNone;
    float4 next = lane < n ? a.pos[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int j = lane; j - lane < n; j += 32) {
        const float4 q = next;
        if (j + 32 < n) next = a.pos[j + 32];
        uint64_t k = kNone;
        if (j < n) {
            const float d = sqdist(q.x, q.y, q.z, me.x, me.y, me.z);
            if (d <= FLT_MAX) k = pack_key(d, j);
        }
        warp_insert(best, k, K);
    }
    return best;
}

// K nearest points by windows of the selection grid around the point's cell: the points
// outside the window lie on rays at least one window edge away, so the search ends once the
// K-th distance is below the smallest distance to such a ray. No hash grid is built (its
// build was 6 launches) and a window's 25 cells are one step of the warp. A window that has grown
// to twice as many cells as there are points gives way to a pass over the points, and where the
// cells are so sparsely filled that it would (K points take K ncells / n cells of an even spread,
// and two to three times as many to prove it) the pass is taken at once. 1 % of 640x480 pixels at
// stride 1 valid, K = 10: 135 us (443 by windows alone, 728 by the hash grid of all points), 0.1 %
// with K = 32: 42 (16,850 and 416); 10 % of 1200x680: 2.8 ms (4.2, 5.4; giving way at as many
// cells as points 1.9, but at 3 % of 640x480 280 us instead of 183).
constexpr float kSparse = 4.f;
constexpr int kWindowMost = 2;
__device__ __forceinline__ uint64_t window_nearest(const ShapeArgs &a, int i, float4 me, int n, int K)
{
    const Window &w = a.w;
    const int lane = threadIdx.x & 31;
    const int c = w.point_cell[i], cv = c / w.ncx, cu = c - cv * w.ncx;
    const float rx = w.x0 + (float)cu * w.step_x, ry = w.y0 + (float)cv * w.step_y;
    // the points' FP32 coordinates are off their rays by a few units in the last place
    const float off_ray = 1e-6f * me.z * (1.f + fabsf(rx) + fabsf(ry));
    uint64_t best = kNone;
    const auto take = [&](int u, int v, bool on) {
        uint64_t k = kNone;
        if (on && u >= 0 && u < w.ncx && v >= 0 && v < w.ncy) {
            const int j = w.cell_point[(size_t)v * w.ncx + u];
            if (j >= 0) {
                const float4 q = a.pos[j];
                const float d = sqdist(q.x, q.y, q.z, me.x, me.y, me.z);
                if (d <= FLT_MAX) k = pack_key(d, j);
            }
        }
        warp_insert(best, k, K);
    };
    take(cu - 2 + lane % 5, cv - 2 + lane / 5, lane < 25);
#pragma unroll 1
    for (int m = 2;; ++m) {
        const bool l = cu - m > 0, r = cu + m < w.ncx - 1, t = cv - m > 0, b = cv + m < w.ncy - 1;
        if (!(l || r || t || b)) break;                          // every cell was seen
        float gap = FLT_MAX;
        const float mx = (float)(m + 1) * w.step_x, my = (float)(m + 1) * w.step_y;
        if (l) gap = fminf(gap, slope_gap(me.z, rx, -mx, -(float)cu * w.step_x));
        if (r) gap = fminf(gap, slope_gap(me.z, rx, mx, (float)(w.ncx - 1 - cu) * w.step_x));
        if (t) gap = fminf(gap, slope_gap(me.z, ry, -my, -(float)cv * w.step_y));
        if (b) gap = fminf(gap, slope_gap(me.z, ry, my, (float)(w.ncy - 1 - cv) * w.step_y));
        const uint64_t kth = __shfl_sync(kFull, best, K - 1);
        gap = gap * (1.f - 1e-4f) - off_ray;
        if (gap > 0.f && kth != kNone && key_dist(kth) < gap * gap) break;
        if ((2 * m + 1) * (2 * m + 1) >= kWindowMost * n) return all_nearest(a, me, n, K);
        // the next frame of cells: 8 (m + 1) of them, side by side
        const int m1 = m + 1, edge = 2 * m1;
#pragma unroll 1
        for (int c0 = 0; c0 < 4 * edge; c0 += 32) {
            const int k = c0 + lane, s = k / edge, o = k - s * edge;
            const int du = s == 0 ? o - m1 : (s == 1 ? m1 : (s == 2 ? m1 - o : -m1));
            const int dv = s == 0 ? -m1 : (s == 1 ? o - m1 : (s == 2 ? m1 : m1 - o));
            take(cu + du, cv + dv, k < 4 * edge);
        }
    }
    return best;
}

// The same from the points' hash grid: rings of cells until the K-th distance is below the
// searched radius, else every point.
__device__ __forceinline__ uint64_t hash_nearest(const ShapeArgs &a, float4 me, int n, int K, uint64_t *buf)
{
    const float3 x = make_float3(me.x, me.y, me.z);
    uint64_t best = kNone;
#pragma unroll 1
    for (int r = 1; r <= kRings; ++r) {
        search_ring(a.g, x, r, K, best, buf);
        const float reach = (float)r * a.g.cell * (1.f - 1e-4f);
        const uint64_t kth = __shfl_sync(kFull, best, K - 1);
        if (kth != kNone && key_dist(kth) < reach * reach) return best;
    }
    return all_nearest(a, me, n, K);
}

template <bool WINDOW>
__global__ void __launch_bounds__(kShapeThreads) k_shape(const __grid_constant__ ShapeArgs a)
{
    sgad::dependency_wait();
    __shared__ float s_cov[kShapePts][7];
    __shared__ uint64_t s_buf[WINDOW ? 1 : kShapeThreads / 32][64];
    const int n = *a.count;
    const int i0 = blockIdx.x * kShapePts;
    if (i0 >= n) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = min(a.K, n);                                // fewer points than K_c: all of them
    const bool sparse = WINDOW && (float)n * (float)n < kSparse * (float)K * (float)a.w.ncx * (float)a.w.ncy;
#pragma unroll 1
    for (int t = 0; t < kShapeRounds; ++t) {
        const int slot = t * (kShapeThreads / 32) + warp, i = i0 + slot;
        if (i >= n) break;
        const float4 me = a.pos[i];
        const uint64_t best = sparse   ? all_nearest(a, me, n, K)
                              : WINDOW ? window_nearest(a, i, me, n, K)
                                       : hash_nearest(a, me, n, K, s_buf[WINDOW ? 0 : warp]);
        const int nb = best != kNone ? (int)(uint32_t)best : -1;
        if (a.knn_out && lane < a.K) a.knn_out[(size_t)i * a.K + lane] = lane < K ? nb : -1;
        const float4 q = lane < K && nb >= 0 ? a.pos[nb] : me;
        // covariance of the K neighbours (FP32), nearest first: mean, then centred second
        // moments
        float mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll 1
        for (int k = 0; k < K; ++k) {
            mx += __shfl_sync(kFull, q.x, k);
            my += __shfl_sync(kFull, q.y, k);
            mz += __shfl_sync(kFull, q.z, k);
        }
        const float invk = 1.f / (float)K;
        mx = __fmul_rn(mx, invk);
        my = __fmul_rn(my, invk);
        mz = __fmul_rn(mz, invk);
        const float qx = q.x - mx, qy = q.y - my, qz = q.z - mz;
        float A[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int k = 0; k < K; ++k) {
            const float dx = __shfl_sync(kFull, qx, k), dy = __shfl_sync(kFull, qy, k), dz = __shfl_sync(kFull, qz, k);
            A[0] += dx * dx;
            A[1] += dx * dy;
            A[2] += dx * dz;
            A[3] += dy * dy;
            A[4] += dy * dz;
            A[5] += dz * dz;
        }
        if (lane == 0) {
#pragma unroll
            for (int e = 0; e < 6; ++e) s_cov[slot][e] = A[e] * invk;
        }
    }
    __syncthreads();
    const int i = i0 + lane;
    if (warp != 0 || i >= n) return;
    float A[3][3];
    A[0][0] = s_cov[lane][0];
    A[0][1] = A[1][0] = s_cov[lane][1];
    A[0][2] = A[2][0] = s_cov[lane][2];
    A[1][1] = s_cov[lane][3];
    A[1][2] = A[2][1] = s_cov[lane][4];
    A[2][2] = s_cov[lane][5];
    float w[3], V[3][3];
    eig3(A, w, V);
    float sc[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) sc[k] = sqrtf(fmaxf(w[k], 0.f));
    const float smax = sc[2];
    const float floor_s = sqrtf(a.eps);
#pragma unroll
    for (int k = 0; k < 3; ++k) sc[k] = fmaxf(smax > 0.f ? sc[k] / smax : 1.f, floor_s);
    float C[6];
    const int rr[6] = {0, 0, 0, 1, 1, 2}, cc[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) acc += V[rr[e]][k] * (sc[k] * sc[k]) * V[cc[e]][k];
        C[e] = acc;
    }
    a.cov[2 * i] = make_float4(C[0], C[1], C[2], C[3]);
    a.cov[2 * i + 1] = make_float4(C[4], C[5], 0.f, 0.f);
    a.normal[i] = make_float4(V[0][0], V[1][0], V[2][0], 0.f);
}

// ------------------------------------------------------------------ hash grid
// Links points into their buckets' chains (any order: a search's result does not depend on it).
// The chains replace a counting sort of the buckets (a count, three scans and a fill). Returns
// how many buckets the thread was the first of.
__device__ __forceinline__ int link_points(const float4 *pos, int n, const Grid &g, int32_t *head, float4 *pts, int first,
                                           int step)
{
    int fresh = 0;
    for (int i = first; i < n; i += step) {
        const float4 p = pos[i];
        const uint32_t h = cell_hash(cell_of(p.x, g.inv_cell), cell_of(p.y, g.inv_cell), cell_of(p.z, g.inv_cell), g.mask);
        const int next = atomicExch(&head[h], i + 1);
        pts[i] = make_float4(p.x, p.y, p.z, __int_as_float(next));
        fresh += next == 0 ? 1 : 0;
    }
    return fresh;
}

// state: the points are the map, linked at the level of its last build, and the occupied buckets
// are counted after the last head; commit: the map after an update, whose count becomes
// min(old + inserted, capacity).
__global__ void __launch_bounds__(256) k_hash_link(const float4 *pos, int32_t *count, int32_t cap,
                                                   const __grid_constant__ MapGrid m, int32_t *head, float4 *pts,
                                                   const GicpState *state, int commit)
{
    sgad::dependency_wait();
    const int n = min(commit ? state->map_old + state->ins_total : *count, cap);
    if (commit && blockIdx.x == 0 && threadIdx.x == 0) *count = n;
    const Grid g = grid_at(m, state ? valid_level(state->level) : 0);
    const int fresh = __reduce_add_sync(
        kFull, link_points(pos, n, g, head, pts, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x));
    if (state && fresh && (threadIdx.x & 31) == 0) atomicAdd(&head[g.mask + 1u], fresh);
}

// Links the map again where its density does not suit the level: longer chains than kLongChain
// points, or shorter than kShortChain at a small cell. One cluster, which has nothing to do
// otherwise (a surface's points per cell go with the square of the cell's size, so a new level's
// chains lie between the two and it stays).
constexpr int kLongChain = 24, kShortChain = 4;
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(1024)
    k_hash_relink(const float4 *pos, const int32_t *count, int32_t cap, const __grid_constant__ MapGrid m, int32_t *head,
                  float4 *pts, GicpState *state)
{
    sgad::dependency_wait();
    const int n = min(*count, cap), level = valid_level(state->level);
    const float chain = (float)n / (float)max(head[m.g.mask + 1u], 1);
    if (!(chain > (float)kLongChain && level < kLevels - 1) && !(chain < (float)kShortChain && level > 0)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) state->level = level;
        return;
    }
    const float d = 0.5f * (float)kDivisor[level], coarse = chain * d * d;    // points per cell of half the radius
    const int want = coarse < 16.f ? 0 : (coarse < 32.f ? 1 : (coarse < 64.f ? 2 : 3));
    const int first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    cluster.sync();                                            // every block has read the level and the counts
    if (first == 0) state->level = want;
    for (uint32_t i = first; i <= m.g.mask; i += step) head[i] = 0;
    __threadfence();
    cluster.sync();
    link_points(pos, n, grid_at(m, want), head, pts, first, step);
}

// ------------------------------------------------------------------ Gauss-Newton step
struct StepArgs {
    const float4 *spos, *scov;
    const int32_t *scount;
    const float4 *mpos, *mcov, *mnorm;
    const int32_t *mcount;
    MapGrid grid;
    float r_max;
    int32_t kmatch;
    int32_t system;          // accumulate the Gauss-Newton system
    int32_t rows;            // rows of partial sums
    GicpState *state;
    Pose12 pose;             // of a single step (tracking takes the state's)
    int32_t *idx_out;
    float *partial;          // [rows][32]
};

// Rows of partial sums that hold points: row v sums points 16 (v + k rows) .. + 15. Every such
// row has points (the barriers between zeroing its terms and summing them are in the loop over
// them); an empty set has no row, and its sums are zero.
__device__ __forceinline__ int rows_used(int n, int rows) { return min(rows, (n + kRowPts - 1) / kRowPts); }

// The contribution of one correspondence to the Gauss-Newton system (H upper triangle,
// g = J^T M e, cost, count) in FP32.
__device__ __forceinline__ void gn_terms(const float *P, float3 x, float4 b, float4 cb0, float4 cb1, float4 ca0,
                                         float4 ca1, float *acc)
{
    const float Ca[3][3] = {{ca0.x, ca0.y, ca0.z}, {ca0.y, ca0.w, ca1.x}, {ca0.z, ca1.x, ca1.y}};
    const float R[3][3] = {{P[0], P[1], P[2]}, {P[4], P[5], P[6]}, {P[8], P[9], P[10]}};
    float RC[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) RC[r][c] = R[r][0] * Ca[0][c] + R[r][1] * Ca[1][c] + R[r][2] * Ca[2][c];
    float S[6];
    const int rr[6] = {0, 0, 0, 1, 1, 2}, cc[6] = {0, 1, 2, 1, 2, 2};
    const float cb[6] = {cb0.x, cb0.y, cb0.z, cb0.w, cb1.x, cb1.y};
#pragma unroll
    for (int e = 0; e < 6; ++e)
        S[e] = cb[e] + RC[rr[e]][0] * R[cc[e]][0] + RC[rr[e]][1] * R[cc[e]][1] + RC[rr[e]][2] * R[cc[e]][2];
    float Mi[6];
    inv_sym3(S, Mi);
    const float M[3][3] = {{Mi[0], Mi[1], Mi[2]}, {Mi[1], Mi[3], Mi[4]}, {Mi[2], Mi[4], Mi[5]}};
    const float e3[3] = {b.x - x.x, b.y - x.y, b.z - x.z};
    // J = [[x]_x, -I]
    const float J[3][6] = {{0.f, -x.z, x.y, -1.f, 0.f, 0.f}, {x.z, 0.f, -x.x, 0.f, -1.f, 0.f},
                           {-x.y, x.x, 0.f, 0.f, 0.f, -1.f}};
    float MJ[3][6];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 6; ++c) MJ[r][c] = M[r][0] * J[0][c] + M[r][1] * J[1][c] + M[r][2] * J[2][c];
    int t = 0;
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int c = r; c < 6; ++c) acc[t++] += J[0][r] * MJ[0][c] + J[1][r] * MJ[1][c] + J[2][r] * MJ[2][c];
    float Me[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) Me[r] = M[r][0] * e3[0] + M[r][1] * e3[1] + M[r][2] * e3[2];
#pragma unroll
    for (int c = 0; c < 6; ++c) acc[21 + c] += J[0][c] * Me[0] + J[1][c] * Me[1] + J[2][c] * Me[2];
    acc[27] += e3[0] * Me[0] + e3[1] * Me[1] + e3[2] * Me[2];
    acc[28] += 1.f;
}


// A tracked point's candidates, kept between the iterations of one track in shared memory:
// the 32 nearest map points of x0 with their normals, and a radius rho: every map point
// nearer than rho to x0 is among them. So at x, with delta = |x - x0|, every map point
// nearer than rho - delta is, and the k_match nearest within r_max are exact as long as
// they lie inside that radius (a margin covers the rounding of the distances). As the pose
// converges delta shrinks, and an iteration reads 32 kept points instead of searching the
// grid.
struct Kept {
    float4 src;               // the source point
    float4 x0;                // x0, rho (0: no candidates)
    float4 pos[32];           // x, y, z, index (-1: none)
    float nx[32], ny[32], nz[32];
};
constexpr int kKeptPts = 4;               // points per warp with candidates; further ones search each time
constexpr size_t kTrackSmem = (size_t)kKeptPts * kRowPts * sizeof(Kept);
constexpr int kBatchRows = 2;             // rows whose points' terms are taken together
constexpr float kMargin = 1.f - 1e-4f;

// Correspondence of x, or -1; whole warp. kept: the point's candidates (null: none kept).
// first: the first step of a track, which moves the points most: its search ends as soon as
// its result is proven and keeps nothing; a later one goes on until the candidates allow a
// move of `slack` (0.3 of a cell, 1.5 cm at the default radius: with half of that, single
// points outran theirs in each of the next ten iterations, and one search delays the
// iteration of all by 10-15 us).
__device__ __forceinline__ int match_point(const StepArgs &a, const Grid &grid, float3 x, Kept *kept, bool first,
                                           uint64_t *buf)
{
    const int lane = threadIdx.x & 31;
    const int K = a.kmatch;
    const float r2 = a.r_max * a.r_max;
    bool member = false;
    float d = FLT_MAX, nx = 0.f, ny = 0.f, nz = 0.f;
    int j = INT_MAX;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    bool ok = false;
    if (kept && !first && kept->x0.w > 0.f) {
        const float4 h = kept->x0;
        q = kept->pos[lane];
        nx = kept->nx[lane];
        ny = kept->ny[lane];
        nz = kept->nz[lane];
        j = __float_as_int(q.w);
        const float s2 = sqdist(h.x, h.y, h.z, x.x, x.y, x.z);
        const float delta = s2 > 0.f ? s2 * rsqrtf(s2) : 0.f;
        const float lim = h.w * kMargin - delta * (2.f - kMargin);
        d = sqdist(q.x, q.y, q.z, x.x, x.y, x.z);
        member = j >= 0 && d <= r2;
        // the K nearest are known if K lie inside the radius, or all within r_max do
        ok = lim > 0.f && (__popc(__ballot_sync(kFull, member && d < lim * lim)) >= K || a.r_max < lim);
        // the first K were the nearest to x0: the farthest of them bounds the K-th distance
        const unsigned far = __reduce_max_sync(kFull, lane >= K ? 0u : (member ? __float_as_uint(d) : 0xffffffffu));
        member = member && __float_as_uint(d) <= far;
    }
    if (!ok) {
        const bool keep = kept && !first;
        const float slack = 0.3f * a.grid.cell[0];
        uint64_t best = kNone;
        float rho = 0.f;
        // as many rings as the cells' divisor prove any result
#pragma unroll 1
        for (int r = 1; r <= min(grid.divisor + 1, kMaxRings); ++r) {
            search_ring(grid, x, r, keep ? 32 : K, best, buf);
            const float reach = (float)r * grid.cell * (1.f - 1e-4f);
            const uint64_t kth = __shfl_sync(kFull, best, K - 1), end = __shfl_sync(kFull, best, 31);
            const bool have = kth != kNone && key_dist(kth) <= r2;
            const bool proven = reach >= a.r_max || (kth != kNone && key_dist(kth) < reach * reach);
            const bool full = end != kNone && sqrtf(key_dist(end)) < reach;
            rho = full ? sqrtf(key_dist(end)) : reach;
            const float need = have ? sqrtf(key_dist(kth)) : a.r_max;
            if (proven && (!keep || full || rho - need >= slack)) break;
        }
        d = best != kNone ? key_dist(best) : FLT_MAX;
        j = best != kNone ? (int)(uint32_t)best : -1;
        member = lane < K && j >= 0 && d <= r2;
        if (keep ? j >= 0 : member) {
            q = grid.pts[j];
            const float4 nr = a.mnorm[j];
            nx = nr.x;
            ny = nr.y;
            nz = nr.z;
        }
        if (keep) {
            q.w = __int_as_float(j);
            kept->pos[lane] = q;
            kept->nx[lane] = nx;
            kept->ny[lane] = ny;
            kept->nz[lane] = nz;
            if (lane == 0) kept->x0 = make_float4(x.x, x.y, x.z, rho);
            __syncwarp();
        }
    }
    // The smallest point-to-surface distance among the K nearest members (ties by distance,
    // index): the members in the order of that distance, until one is among the K nearest.
    unsigned bm = 0xffffffffu;
    if (member) {
        const float dx = __fsub_rn(q.x, x.x), dy = __fsub_rn(q.y, x.y), dz = __fsub_rn(q.z, x.z);
        bm = __float_as_uint(fabsf(__fadd_rn(__fadd_rn(__fmul_rn(nx, dx), __fmul_rn(ny, dy)), __fmul_rn(nz, dz))));
    }
    const uint64_t key = pack_key(d, j);
#pragma unroll 1
    for (;;) {
        const unsigned m1 = __reduce_min_sync(kFull, bm);
        if (m1 == 0xffffffffu) return -1;
        const unsigned eq = __ballot_sync(kFull, bm == m1);
        uint64_t k = __shfl_sync(kFull, key, __ffs(eq) - 1);
        if (eq & (eq - 1)) {                                     // equal distances to the surface
            for (unsigned rest = eq & (eq - 1); rest; rest &= rest - 1) {
                const uint64_t o = __shfl_sync(kFull, key, __ffs(rest) - 1);
                k = o < k ? o : k;
            }
        }
        if (__popc(__ballot_sync(kFull, member && key < k)) < K) return (int)(uint32_t)k;
        if (bm == m1) bm = 0xffffffffu;
    }
}

__device__ void sum_partials(const float *partial, int nrows, double *sys);
__device__ bool solve_state(GicpState *st, const double *sys, double &step2);

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A wait on the other blocks gives up after about a second, and later where a block's searches
// may take longer: after four times as many tries more as a warp's searches may visit points (a
// point of a chain takes 0.3 us, about a try). 16 points in a map of 4.2 M points in one cell take
// 1.3 s an iteration.
constexpr uint32_t kSyncSpins = 1u << 22;
__device__ __forceinline__ uint32_t spin_limit(int n, int map, int blocks)
{
    const unsigned long long per_warp = ((unsigned)n + (unsigned)(blocks * kRowPts) - 1u) / (unsigned)(blocks * kRowPts);
    return kSyncSpins + (uint32_t)min(4ull * per_warp * (unsigned)max(map, 0), 1ull << 31);
}

// Correspondences and partial sums of the Gauss-Newton system. A block takes rows of 16
// points, one warp per point. TRACK: the whole of a track in one cooperative launch: after
// each iteration the last block to finish sums the rows, solves and updates the pose, and
// the others wait for it. One launch per iteration, with a search for every point, took
// 100-200 us each (8,160-12,288 points, 15-25 iterations); here the first two iterations,
// which search, take 45-65 us and the others 13-16 us: 3-5 us for the kept candidates, 1 for
// the terms, 3 for the sum, 4.5 for the solve (dependent FP64 operations) and 2-3 for the
// blocks to meet. A track of 25 iterations of 8,160 points: 0.41 ms, one of 15 iterations of
// 12,288: 0.32 ms.
template <bool TRACK>
__global__ void __launch_bounds__(kStepThreads, 2) k_gicp_step(const __grid_constant__ StepArgs a)
{
    extern __shared__ float4 track_smem[];                     // TRACK: Kept [kKeptPts][16 warps]
    Kept *const cache = reinterpret_cast<Kept *>(track_smem);
    __shared__ float s_acc[kBatchRows][kRowPts][33];
    __shared__ int s_match[kBatchRows][kRowPts];
    __shared__ uint64_t s_buf[kRowPts][64];
    __shared__ float s_pose[12];
    __shared__ double s_sys[kSys];
    __shared__ int s_last, s_done;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = *a.scount;
    const int used = rows_used(n, a.rows);
    const uint32_t epoch = TRACK && threadIdx.x == 0 ? ld_acquire(&a.state->sync) : 0u;
    const Grid grid = grid_at(a.grid, valid_level(a.state->level));
#pragma unroll 1
    for (uint32_t it = 0;; ++it) {
        if (threadIdx.x < 12) s_pose[threadIdx.x] = TRACK ? __ldcg(&a.state->posef[threadIdx.x]) : a.pose.p[threadIdx.x];
        __syncthreads();
        int slot = 0;
#pragma unroll 1
        for (int v0 = blockIdx.x; v0 < used; v0 += kBatchRows * gridDim.x) {
#pragma unroll
            for (int b = 0; b < kBatchRows; ++b) s_acc[b][warp][lane] = 0.f;
#pragma unroll 1
            for (int base = 0; base + v0 * kRowPts < n; base += a.rows * kRowPts) {
#pragma unroll 1
                for (int b = 0; b < kBatchRows; ++b, ++slot) {
                    const int v = v0 + b * (int)gridDim.x, i = base + v * kRowPts + warp;
                    int j = -1;
                    if (v < used && i < n) {                   // whole warp
                        Kept *kept = TRACK && slot < kKeptPts ? cache + slot * kRowPts + warp : nullptr;
                        float4 src;
                        if (kept && it > 0) {
                            src = kept->src;
                        } else {
                            src = a.spos[i];
                            if (kept && lane == 0) {
                                kept->src = src;
                                kept->x0 = make_float4(0.f, 0.f, 0.f, 0.f);
                            }
                        }
                        j = match_point(a, grid, transform(s_pose, src), kept, it == 0, s_buf[warp]);
                        if (!TRACK && a.idx_out && lane == 0) a.idx_out[i] = j;
                    }
                    if (lane == 0) s_match[b][warp] = j;
                }
                if (!a.system) continue;
                __syncthreads();
                // the terms of the batch's points, one per thread (a point's ~300 operations
                // are one dependent chain, paid once for the batch)
                if (threadIdx.x < kBatchRows * kRowPts) {
                    const int b = threadIdx.x / kRowPts, w = threadIdx.x % kRowPts, j = s_match[b][w];
                    const int i = base + (v0 + b * (int)gridDim.x) * kRowPts + w;
                    if (j >= 0)
                        gn_terms(s_pose, transform(s_pose, a.spos[i]), a.mpos[j], a.mcov[2 * j], a.mcov[2 * j + 1],
                                 a.scov[2 * i], a.scov[2 * i + 1], s_acc[b][w]);
                }
                __syncthreads();
            }
            if (!a.system) continue;
            if (threadIdx.x < kBatchRows * 32 && lane < kSys) {
                // the 16 points in a fixed order: pairs two apart, then neighbours, then fours
                const int b = threadIdx.x >> 5, v = v0 + b * (int)gridDim.x;
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < kRowPts; w += 4) {
                    const float(*r)[33] = &s_acc[b][w];
                    s += (r[0][lane] + r[2][lane]) + (r[1][lane] + r[3][lane]);
                }
                if (v < used) a.partial[v * 32 + lane] = s;
            }
            __syncthreads();
        }
        if (!TRACK) return;
        // (the barrier and thread 0's fence order every thread's rows before the count)
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(&a.state->blocks_done, 1) == (int)gridDim.x - 1;
            __threadfence();
        }
        __syncthreads();
        if (s_last) {
            sum_partials(a.partial, used, s_sys);
            if (warp == 0) {
                double step2 = 0.0;
                const bool done = solve_state(a.state, s_sys, step2);
                if (lane == 0) {
                    a.state->blocks_done = 0;
                    s_done = done;
                    __threadfence();
                    st_release(&a.state->sync, epoch + it + 1u);
                    // (stored before this block is counted in the next iteration)
                    if (step2 >= 0.0) a.state->step = sqrt(step2);
                }
            }
        } else if (threadIdx.x == 0) {
            const uint32_t limit = spin_limit(n, *a.mcount, (int)gridDim.x);
            uint32_t t = 0;
            while (ld_acquire(&a.state->sync) != epoch + it + 1u && ++t < limit) {
            }
            if (t >= limit) {                             // recorded; the block ends
                a.state->gave_up = 1;
                s_done = 1;
            } else {
                s_done = __ldcg(&a.state->done);
            }
        }
        __syncthreads();
        if (s_done) return;
    }
}

// Sum of the rows of partials in a fixed order: warp w takes rows w, w + nw, ..., one
// column per lane, and adds them without a rounding that matters: with sigma a power of two
// above the sum of their magnitudes, (v + sigma) - sigma is v's part in multiples of
// sigma's last place, whose sum is exact (Rump, Ogita and Oishi 2008); the rests are split
// and added the same way once more, which leaves 2^-34 of the largest row to a plain sum.
// The warps' three parts are then added in FP64 in warp order. FP64 adds and conversions
// run at 2 lanes per cycle and SM on this chip: adding 510 rows in FP64 took one block
// about 9 us, this 2-3 us. Partials are read through L2 (written by other blocks of the
// same grid).
__device__ void sum_partials(const float *partial, int nrows, double *sys)
{
    constexpr int kWarps = kStepThreads / 32, kPer = (kMaxRows + kWarps - 1) / kWarps;
    __shared__ double part[kWarps][kSys];
    const int w = threadIdx.x >> 5, k = threadIdx.x & 31;
    if (k < kSys) {
        float v[kPer], top = 0.f;
#pragma unroll
        for (int u = 0; u < kPer; ++u)
            v[u] = w + u * kWarps < nrows ? __ldcg(partial + (w + u * kWarps) * 32 + k) : 0.f;
#pragma unroll
        for (int u = 0; u < kPer; ++u) top = fmaxf(top, fabsf(v[u]));
        // the power of two above 64 times the largest (kPer < 64 rows)
        const int e = (int)(__float_as_uint(top) >> 23) + 7;
        double total = 0.0;
        if (e < 254 && e > 32) {
            const float s1 = __uint_as_float((uint32_t)e << 23), s2 = __uint_as_float((uint32_t)(e - 17) << 23);
            float a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const float h = __fsub_rn(__fadd_rn(v[u], s1), s1), r = __fsub_rn(v[u], h);
                const float m = __fsub_rn(__fadd_rn(r, s2), s2);
                a1 = __fadd_rn(a1, h);
                a2 = __fadd_rn(a2, m);
                a3 = __fadd_rn(a3, __fsub_rn(r, m));
            }
            total = ((double)a1 + (double)a2) + (double)a3;
        } else {                                                // infinities, NaN, subnormals
            for (int u = 0; u < kPer; ++u) total += (double)v[u];
        }
        part[w][k] = total;
    }
    __syncthreads();
    if (threadIdx.x < kSys) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int q = 0; q < kStepThreads / 32; ++q) s[q & 3] += part[q][threadIdx.x];
        sys[threadIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kStepThreads) k_gicp_sum(const float *partial, const int32_t *count, int rows,
                                                           double *out)
{
    __shared__ double sys[kSys];
    sum_partials(partial, rows_used(*count, rows), sys);
    if (threadIdx.x < kSys) out[threadIdx.x] = sys[threadIdx.x];
}

// One warp: from the summed system, an L D L^T solve of H xi = -g in FP64 and the pose
// update (R, t) <- (Exp(omega) R, Exp(omega) t + v); returns whether the track is over, and
// |xi|^2 (-1: no step) in step2.
// Lane r < 6 holds row r of H and lane 6 the row -g, whose factor is the forward
// substitution; FP64 operations are slow and dependent here, so the rows go side by side,
// with one rounded reciprocal per column instead of square roots and a division per element
// (one thread with a Cholesky factor took ~20 us, this ~3 us).
__device__ bool solve_state(GicpState *st, const double *sys, double &step2)
{
    const int lane = threadIdx.x & 31;
    double old[3] = {0.0, 0.0, 0.0};                           // the column of the old pose that a lane needs
    if (lane < 12) {
#pragma unroll
        for (int m = 0; m < 3; ++m) old[m] = st->pose[4 * m + (lane & 3)];
    }
    const int iters = st->iters + 1, max_iters = st->max_iters;
    const double tol = (double)st->tol;
    if (lane == 0) {
        st->n = (int)sys[28];
        st->cost = sys[27];
    }
    bool good = sys[28] >= 6.0;
    const int row = min(lane, 6);
    double A[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const int lo = min(row, c), hi = max(row, c);          // upper triangle, row by row
        A[c] = row < 6 ? sys[lo * 6 - lo * (lo - 1) / 2 + hi - lo] : -sys[21 + c];
    }
    // column by column; A becomes the rows of L (unit diagonal), of lane 6 D^-1 L^-1 (-g)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const double d = __shfl_sync(kFull, A[j], j);
        good = good && d > 0.0;
        const double u = A[j];
        A[j] = u * __drcp_rn(d);
#pragma unroll
        for (int c = j + 1; c < 6; ++c) A[c] -= A[j] * __shfl_sync(kFull, u, c);
    }
    if (!good) {                                               // uniform: too few points, or not positive definite
        if (lane == 0) {
            st->status |= 2;
            st->done = 1;
        }
        step2 = -1.0;
        return true;
    }
    // back substitution
    double xi[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) xi[c] = __shfl_sync(kFull, A[c], 6);
#pragma unroll
    for (int i = 5; i >= 1; --i)
#pragma unroll
        for (int c = 0; c < i; ++c) xi[c] -= __shfl_sync(kFull, A[c], i) * xi[i];
    // Exp(omega) = I + a K + b K^2 with a = sin(th) / th, b = (1 - cos(th)) / th^2: their
    // Taylor series for a small angle (the terms after the last are below 1e-17 of the sum)
    const double t2 = xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2];
    double ea, eb;
    if (t2 < 0.01) {
        ea = 1.0 + t2 * (-1.0 / 6 + t2 * (1.0 / 120 + t2 * (-1.0 / 5040 + t2 * (1.0 / 362880 - t2 * (1.0 / 39916800)))));
        eb = 0.5 + t2 * (-1.0 / 24 + t2 * (1.0 / 720 + t2 * (-1.0 / 40320 + t2 * (1.0 / 3628800 - t2 * (1.0 / 479001600)))));
    } else {
        const double th = sqrt(t2);
        ea = sin(th) / th;
        eb = (1.0 - cos(th)) / t2;
    }
    // lane e < 12: element (e / 4, e % 4) of the new pose. K^2 = w w^T - th^2 I
    if (lane < 12) {
        const int r = lane >> 2, c = lane & 3;
        const double w[3] = {xi[0], xi[1], xi[2]};
        const double wr = r == 0 ? w[0] : (r == 1 ? w[1] : w[2]);
        const double K[3] = {r == 0 ? 0.0 : (r == 1 ? w[2] : -w[1]), r == 0 ? -w[2] : (r == 1 ? 0.0 : w[0]),
                             r == 0 ? w[1] : (r == 1 ? -w[0] : 0.0)};
        double v = c == 3 ? (r == 0 ? xi[3] : (r == 1 ? xi[4] : xi[5])) : 0.0;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const double E = (r == m ? 1.0 - eb * t2 : 0.0) + ea * K[m] + eb * (wr * w[m]);
            v += E * old[m];
        }
        st->pose[lane] = v;
        st->posef[lane] = (float)v;
    }
    step2 = (t2 + xi[3] * xi[3]) + (xi[4] * xi[4] + xi[5] * xi[5]);
    const bool conv = step2 < tol * tol;                       // |xi| < tol
    const bool done = conv || iters >= max_iters;
    if (lane == 0) {
        st->iters = iters;
        if (conv) st->converged = 1;
        if (done) st->done = 1;
    }
    __syncwarp();
    return done;
}

__global__ void k_gicp_init(GicpState *st, PoseD p0, int keep_pose, int max_iters, float tol, int done)
{
    sgad::dependency_wait();
    if (!keep_pose)
        for (int k = 0; k < 12; ++k) st->pose[k] = p0.p[k];
    for (int k = 0; k < 12; ++k) st->posef[k] = (float)st->pose[k];
    st->iters = 0;
    st->done = done;
    st->converged = 0;
    st->n = 0;
    st->cost = 0.0;
    st->step = 0.0;
    st->max_iters = max_iters;
    st->tol = tol;
    st->status &= 1;                 // keep the source's overflow flag, clear the rest
    st->gave_up = 0;
    st->blocks_done = 0;
}

// ------------------------------------------------------------------ map update
struct InsArgs {
    const float4 *spos, *scov, *snorm;
    const int32_t *scount;
    float4 *mpos, *mcov, *mnorm;
    int32_t *mcount;
    int32_t mcap;
    MapGrid grid;
    float d_ov;
    GicpState *state;
    int32_t *flags;
    int32_t *blk;
};

// Whether an indexed point lies within d_ov of x; whole warp.
__device__ __forceinline__ bool overlaps(float3 x, const Grid &g, float d_ov)
{
    const float d2ov = d_ov * d_ov;
    bool hit = false;
    const auto near = [&](float4 b) {
        if (sqdist(b.x, b.y, b.z, x.x, x.y, x.z) <= d2ov) hit = true;
    };
    // (as many rings as the cells' divisor reach d_ov)
#pragma unroll 1
    for (int r = 1; r <= kMaxRings; ++r) {
        switch (r) {
        case 1: ring_cells<1, true>(g, x, near); break;
        case 2: ring_cells<2, false>(g, x, near); break;
        case 3: ring_cells<3, false>(g, x, near); break;
        case 4: ring_cells<4, false>(g, x, near); break;
        case 5: ring_cells<5, false>(g, x, near); break;
        default: ring_cells<6, false>(g, x, near); break;
        }
        if (__any_sync(kFull, hit)) return true;
        if ((float)r * g.cell * (1.f - 1e-4f) >= d_ov) break;
    }
    return false;
}

// One warp per source point, kInsPts points per block: the search is a chain of dependent
// loads, so it takes a warp's lanes for the 27 nearest cells at once.
__global__ void __launch_bounds__(1024) k_insert_flag(const __grid_constant__ InsArgs a)
{
    sgad::dependency_wait();
    __shared__ int s_keep[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = *a.scount;
    if ((int)blockIdx.x * kInsPts >= n) {
        if (threadIdx.x == 0) a.blk[blockIdx.x] = 0;
        return;
    }
    const bool empty = *a.mcount == 0;
    const Grid grid = grid_at(a.grid, valid_level(a.state->level));
    int kept = 0;
#pragma unroll 1
    for (int k = 0; k < kInsPts / 32; ++k) {
        const int i = blockIdx.x * kInsPts + k * 32 + warp;
        if (i >= n) break;
        const bool keep = empty || !overlaps(transform(a.state->posef, a.spos[i]), grid, a.d_ov);
        if (lane == 0) a.flags[i] = keep ? 1 : 0;
        kept += keep ? 1 : 0;
    }
    if (lane == 0) s_keep[warp] = kept;
    __syncthreads();
    if (warp == 0) {
        const int tot = __reduce_add_sync(kFull, s_keep[lane]);
        if (lane == 0) a.blk[blockIdx.x] = tot;
    }
}

__global__ void __launch_bounds__(256) k_insert_write(const __grid_constant__ InsArgs a)
{
    sgad::dependency_wait();
    __shared__ int red[8];
    const int prefix = block_prefix(a.blk, blockIdx.x * (256 / kInsPts), red);
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int n = *a.scount;
    const bool keep = i < n && a.flags[i] != 0;
    int total;
    const int local = block_exclusive_scan(keep ? 1 : 0, red, &total);
    const int old = *a.mcount;
    if (keep) {
        const int o = old + prefix + local;
        if (o < a.mcap) {
            const float *P = a.state->posef;
            const float3 x = transform(P, a.spos[i]);
            const float R[3][3] = {{P[0], P[1], P[2]}, {P[4], P[5], P[6]}, {P[8], P[9], P[10]}};
            const float4 c0 = a.scov[2 * i], c1 = a.scov[2 * i + 1], nr = a.snorm[i];
            const float C[3][3] = {{c0.x, c0.y, c0.z}, {c0.y, c0.w, c1.x}, {c0.z, c1.x, c1.y}};
            float RC[3][3], W[3][3];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c) RC[r][c] = R[r][0] * C[0][c] + R[r][1] * C[1][c] + R[r][2] * C[2][c];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c) W[r][c] = RC[r][0] * R[c][0] + RC[r][1] * R[c][1] + RC[r][2] * R[c][2];
            a.mpos[o] = make_float4(x.x, x.y, x.z, 0.f);
            a.mcov[2 * o] = make_float4(W[0][0], W[0][1], W[0][2], W[1][1]);
            a.mcov[2 * o + 1] = make_float4(W[1][2], W[2][2], 0.f, 0.f);
            a.mnorm[o] = make_float4(R[0][0] * nr.x + R[0][1] * nr.y + R[0][2] * nr.z,
                                     R[1][0] * nr.x + R[1][1] * nr.y + R[1][2] * nr.z,
                                     R[2][0] * nr.x + R[2][1] * nr.y + R[2][2] * nr.z, 0.f);
        } else {
            atomicOr(&a.state->status, 1);
        }
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        a.state->map_old = old;
        a.state->ins_total = prefix + total;
    }
}

}  // namespace

// ====================================================================== host entry points
namespace {

sgad_status fail(const char *msg) { return report_error(SGAD_ERR_INVALID_ARG, msg); }

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

sgad_status check_params(const sgad_gicp_params *p)
{
    if (!p) return fail("sgad_gicp: NULL params");
    if (p->stride < 1 || p->k_cov < 3 || p->k_cov > 32 || p->k_match < 1 || p->k_match > kKMatchMax ||
        p->max_iters < 1 || p->max_iters > 100 || !(p->r_max > 0.f) || !(p->d_overlap >= 0.f) || !(p->tol >= 0.f) ||
        !(p->eps > 0.f && p->eps <= 1.f) || !std::isfinite(p->r_max) || !std::isfinite(p->d_overlap) ||
        p->src_capacity < 1 || p->map_capacity < 1 || p->src_capacity > (1 << 24) || p->map_capacity > (1 << 24))
        return fail("sgad_gicp: parameter out of range");
    return SGAD_OK;
}

sgad_status check_set(const sgad_gaussian_set *s, int32_t max_capacity, const char *what)
{
    if (!s || !s->pos || !s->cov || !s->normal || !s->count || s->capacity < 1 || s->capacity > max_capacity)
        return fail(what);
    if (!aligned(s->pos, 16) || !aligned(s->cov, 16) || !aligned(s->normal, 16) || !aligned(s->count, 4))
        return fail(what);
    return SGAD_OK;
}

sgad_status check_ws(void *ws, size_t bytes, size_t need)
{
    if (!ws || !aligned(ws, 256)) return fail("sgad_gicp: workspace NULL or not 256-byte aligned");
    if (bytes < need) return report_error(SGAD_ERR_WORKSPACE_TOO_SMALL, "sgad_gicp: workspace too small");
    return SGAD_OK;
}

template <typename T>
T *at(void *ws, size_t off) { return reinterpret_cast<T *>(static_cast<char *>(ws) + off); }

MapGrid grid_of(const sgad_gicp_params *p, void *ws, const GLayout &L)
{
    MapGrid m;
    m.g.head = at<int32_t>(ws, L.hash_head);
    m.g.pts = at<float4>(ws, L.hash_pts);
    m.g.cap = p->map_capacity;
    m.g.mask = (uint32_t)L.table - 1u;
    m.g.divisor = 2;
    const int divisor[kLevels] = {2, 3, 4, 6};
    for (int l = 0; l < kLevels; ++l) {
        m.cell[l] = fmaxf(p->r_max, p->d_overlap) * (1.001f / (float)divisor[l]);
        m.inv_cell[l] = 1.f / m.cell[l];
    }
    m.g.cell = m.cell[0];
    m.g.inv_cell = m.inv_cell[0];
    return m;
}

sgad_status launched(const char *what)
{
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SGAD_OK : report_error(SGAD_ERR_CUDA, what);
}

// Index of a set: empty chains, then every point linked into its cell's chain. state, commit:
// the map's (see k_hash_link).
sgad_status hash_build(const float4 *pos, int32_t *count, int32_t capacity, const MapGrid &m, int32_t *head,
                       float4 *pts, GicpState *state, int commit, cudaStream_t st)
{
    if (cudaMemsetAsync(head, 0, ((size_t)m.g.mask + (state ? 2 : 1)) * sizeof(int32_t), st) != cudaSuccess)
        return report_error(SGAD_ERR_CUDA, "sgad_gicp: memset failed");
    const int blocks = std::min((capacity + 255) / 256, 4 * 152);
    sgad::launch_after(k_hash_link, blocks, 256, 0, st, pos, count, capacity, m, head, pts, state, commit);
    if (state) sgad::launch_after(k_hash_relink, 8, 1024, 0, st, pos, count, capacity, m, head, pts, state);
    return launched("sgad_gicp: index launch failed");
}

sgad_status build_index(const sgad_gicp_params *p, const sgad_gaussian_set *map, void *ws, const GLayout &L,
                        int commit, cudaStream_t st)
{
    return hash_build(reinterpret_cast<const float4 *>(map->pos), map->count, map->capacity, grid_of(p, ws, L),
                      at<int32_t>(ws, L.hash_head), at<float4>(ws, L.hash_pts), at<GicpState>(ws, L.state), commit, st);
}

StepArgs step_args(const sgad_gicp_params *p, const sgad_gaussian_set *src, const sgad_gaussian_set *map, void *ws,
                   const GLayout &L)
{
    StepArgs a;
    std::memset(&a, 0, sizeof(a));
    a.spos = reinterpret_cast<const float4 *>(src->pos);
    a.scov = reinterpret_cast<const float4 *>(src->cov);
    a.scount = src->count;
    a.mpos = reinterpret_cast<const float4 *>(map->pos);
    a.mcov = reinterpret_cast<const float4 *>(map->cov);
    a.mnorm = reinterpret_cast<const float4 *>(map->normal);
    a.mcount = map->count;
    a.grid = grid_of(p, ws, L);
    a.r_max = p->r_max;
    a.kmatch = p->k_match;
    a.state = at<GicpState>(ws, L.state);
    a.partial = at<float>(ws, L.partial);
    a.rows = L.rows;
    return a;
}

}  // namespace

extern "C" sgad_status sgad_gicp_default_params(sgad_gicp_params *out)
{
    if (!out) return fail("sgad_gicp_default_params: NULL");
    out->stride = 10;
    out->k_cov = 10;
    out->k_match = 5;
    out->max_iters = 30;
    out->r_max = 0.1f;
    out->d_overlap = 0.02f;
    out->tol = 1e-6f;
    out->eps = 1e-3f;
    out->src_capacity = 1 << 16;
    out->map_capacity = 1 << 20;
    return SGAD_OK;
}

extern "C" sgad_status sgad_gicp_workspace_size(const sgad_gicp_params *p, size_t *bytes)
{
    sgad_status s = check_params(p);
    if (s) return s;
    if (!bytes) return fail("sgad_gicp_workspace_size: NULL");
    *bytes = glayout(*p).total;
    return SGAD_OK;
}

extern "C" sgad_status sgad_gicp_frame(const sgad_gicp_params *p, const sgad_camera *cam, const float *depth,
                                       const sgad_gaussian_set *out, int32_t *pix_out, int32_t *knn_out,
                                       void *workspace, size_t ws_bytes, void *stream)
{
    sgad_status s = check_params(p);
    if (s) return s;
    if ((s = check_set(out, p->src_capacity, "sgad_gicp_frame: bad output set"))) return s;
    if (!cam || !depth || cam->width < 1 || cam->height < 1 || !(cam->fx > 0.f) || !(cam->fy > 0.f))
        return fail("sgad_gicp_frame: bad camera or depth");
    const GLayout L = glayout(*p);
    if ((s = check_ws(workspace, ws_bytes, L.total))) return s;
    SelArgs a;
    a.depth = depth;
    a.W = cam->width;
    a.H = cam->height;
    a.R = p->stride;
    a.ncx = (cam->width + p->stride - 1) / p->stride;
    const long long ncells = (long long)a.ncx * ((cam->height + p->stride - 1) / p->stride);
    if (ncells > (long long)kMaxSelBlocks * kSelBlock) return fail("sgad_gicp_frame: too many selection cells");
    a.ncells = (int32_t)ncells;
    a.fx = cam->fx;
    a.fy = cam->fy;
    a.cx = cam->cx;
    a.cy = cam->cy;
    a.pos = reinterpret_cast<float4 *>(out->pos);
    a.pix = pix_out;
    a.count = out->count;
    a.capacity = out->capacity;
    a.blk = at<int32_t>(workspace, L.sel_counts);
    a.state = at<GicpState>(workspace, L.state);
    // The neighbour search scans the selection grid around a point's cell, which needs the
    // maps between cells and points (in the room of the hash grid's points, four words per
    // point). A set of far fewer points than cells takes the hash grid instead.
    const bool window = ncells <= 3ll * p->src_capacity;
    a.point_cell = at<int32_t>(workspace, L.knn_pts);
    a.cell_point = window ? a.point_cell + p->src_capacity : nullptr;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nb = (int)((ncells + kSelBlock - 1) / kSelBlock);
    sgad::launch_after(k_select_count, nb, 256, 0, st, a);
    sgad::launch_after(k_select_write, nb, 256, 0, st, a);
    ShapeArgs sa;
    std::memset(&sa, 0, sizeof(sa));
    sa.pos = reinterpret_cast<const float4 *>(out->pos);
    sa.count = out->count;
    sa.K = p->k_cov;
    sa.eps = p->eps;
    sa.cov = reinterpret_cast<float4 *>(out->cov);
    sa.normal = reinterpret_cast<float4 *>(out->normal);
    sa.knn_out = knn_out;
    const int sb = (out->capacity + kShapePts - 1) / kShapePts;
    if (window) {
        sa.w.point_cell = a.point_cell;
        sa.w.cell_point = a.cell_point;
        sa.w.ncx = a.ncx;
        sa.w.ncy = (cam->height + p->stride - 1) / p->stride;
        sa.w.step_x = (float)p->stride / cam->fx;
        sa.w.step_y = (float)p->stride / cam->fy;
        sa.w.x0 = -cam->cx / cam->fx;
        sa.w.y0 = -cam->cy / cam->fy;
        sgad::launch_after(k_shape<true>, sb, kShapeThreads, 0, st, sa);
    } else {
        // cells of about twice the selection spacing at 2 m (a performance choice only: the
        // search proves its result)
        Grid &g = sa.g;
        g.head = at<int32_t>(workspace, L.knn_head);
        g.pts = at<float4>(workspace, L.knn_pts);
        g.cell = fmaxf(5e-3f, 2.f * (float)p->stride * 2.f / cam->fx);
        g.inv_cell = 1.f / g.cell;
        g.mask = (uint32_t)L.knn_table - 1u;
        g.cap = p->src_capacity;
        MapGrid m = {};
        m.g = g;
        if ((s = hash_build(sa.pos, out->count, out->capacity, m, at<int32_t>(workspace, L.knn_head),
                            at<float4>(workspace, L.knn_pts), nullptr, 0, st)))
            return s;
        sgad::launch_after(k_shape<false>, sb, kShapeThreads, 0, st, sa);
    }
    return launched("sgad_gicp_frame: launch failed");
}

extern "C" sgad_status sgad_gicp_index(const sgad_gicp_params *p, const sgad_gaussian_set *map, void *workspace,
                                       size_t ws_bytes, void *stream)
{
    sgad_status s = check_params(p);
    if (s) return s;
    if ((s = check_set(map, p->map_capacity, "sgad_gicp_index: bad map set"))) return s;
    const GLayout L = glayout(*p);
    if ((s = check_ws(workspace, ws_bytes, L.total))) return s;
    return build_index(p, map, workspace, L, 0, static_cast<cudaStream_t>(stream));
}

namespace {
sgad_status pair_checks(const sgad_gicp_params *p, const sgad_gaussian_set *src, const sgad_gaussian_set *map,
                        void *ws, size_t bytes, GLayout *L)
{
    sgad_status s = check_params(p);
    if (s) return s;
    if ((s = check_set(src, p->src_capacity, "sgad_gicp: bad source set"))) return s;
    if ((s = check_set(map, p->map_capacity, "sgad_gicp: bad map set"))) return s;
    *L = glayout(*p);
    return check_ws(ws, bytes, L->total);
}

bool finite_pose(const float *P)
{
    for (int k = 0; k < 12; ++k)
        if (!std::isfinite(P[k])) return false;
    return true;
}
}  // namespace

extern "C" sgad_status sgad_gicp_correspond(const sgad_gicp_params *p, const sgad_gaussian_set *src,
                                            const sgad_gaussian_set *map, const float pose[12], int32_t *idx_out,
                                            void *workspace, size_t ws_bytes, void *stream)
{
    GLayout L;
    sgad_status s = pair_checks(p, src, map, workspace, ws_bytes, &L);
    if (s) return s;
    if (!pose || !idx_out || !finite_pose(pose)) return fail("sgad_gicp_correspond: bad pose or output");
    StepArgs a = step_args(p, src, map, workspace, L);
    std::memcpy(a.pose.p, pose, sizeof(a.pose.p));
    a.idx_out = idx_out;
    k_gicp_step<false><<<L.rows, kStepThreads, 0, static_cast<cudaStream_t>(stream)>>>(a);
    return launched("sgad_gicp_correspond: launch failed");
}

extern "C" sgad_status sgad_gicp_linearize(const sgad_gicp_params *p, const sgad_gaussian_set *src,
                                           const sgad_gaussian_set *map, const float pose[12], double *system_out,
                                           void *workspace, size_t ws_bytes, void *stream)
{
    GLayout L;
    sgad_status s = pair_checks(p, src, map, workspace, ws_bytes, &L);
    if (s) return s;
    if (!pose || !system_out || !finite_pose(pose)) return fail("sgad_gicp_linearize: bad pose or output");
    StepArgs a = step_args(p, src, map, workspace, L);
    std::memcpy(a.pose.p, pose, sizeof(a.pose.p));
    a.system = 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_gicp_step<false><<<L.rows, kStepThreads, 0, st>>>(a);
    k_gicp_sum<<<1, kStepThreads, 0, st>>>(a.partial, a.scount, L.rows, system_out);
    return launched("sgad_gicp_linearize: launch failed");
}

extern "C" sgad_status sgad_gicp_set_pose(const double pose[12], void *workspace, size_t ws_bytes, void *stream)
{
    if (!pose) return fail("sgad_gicp_set_pose: NULL pose");
    for (int k = 0; k < 12; ++k)
        if (!std::isfinite(pose[k])) return fail("sgad_gicp_set_pose: non-finite pose");
    sgad_status s = check_ws(workspace, ws_bytes, sizeof(GicpState));
    if (s) return s;
    PoseD p0;
    std::memcpy(p0.p, pose, sizeof(p0.p));
    sgad::launch_after(k_gicp_init, 1, 1, 0, static_cast<cudaStream_t>(stream), at<GicpState>(workspace, 0), p0, 0, 0,
                       0.f, 1);
    return launched("sgad_gicp_set_pose: launch failed");
}

extern "C" sgad_status sgad_gicp_track(const sgad_gicp_params *p, const sgad_gaussian_set *src,
                                       const sgad_gaussian_set *map, const double pose0[12], void *workspace,
                                       size_t ws_bytes, void *stream)
{
    GLayout L;
    sgad_status s = pair_checks(p, src, map, workspace, ws_bytes, &L);
    if (s) return s;
    PoseD p0;
    std::memset(&p0, 0, sizeof(p0));
    if (pose0) {                              // else: start from the workspace's pose
        for (int k = 0; k < 12; ++k)
            if (!std::isfinite(pose0[k])) return fail("sgad_gicp_track: non-finite pose");
        std::memcpy(p0.p, pose0, sizeof(p0.p));
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StepArgs a = step_args(p, src, map, workspace, L);
    a.system = 1;
    // every block of the tracking kernel waits for the others once an iteration, so its grid
    // is what the device holds at once (a cooperative launch), at most a block per row
    static int resident[64] = {};
    constexpr size_t smem = kTrackSmem;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    int blocks = e == cudaSuccess && dev >= 0 && dev < 64 ? resident[dev] : 0;
    if (e == cudaSuccess && blocks == 0) {
        int per_sm = 0, sms = 0;
        e = cudaFuncSetAttribute(k_gicp_step<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gicp_step<true>, kStepThreads, smem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        blocks = per_sm * sms;
        if (e == cudaSuccess && dev >= 0 && dev < 64) resident[dev] = blocks;
    }
    if (e != cudaSuccess || blocks < 1) return report_error(SGAD_ERR_CUDA, "sgad_gicp_track: no resident blocks");
    sgad::launch_after(k_gicp_init, 1, 1, 0, st, a.state, p0, pose0 ? 0 : 1, p->max_iters, p->tol, 0);
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel((const void *)k_gicp_step<true>, dim3(std::min(blocks, L.rows)),
                                    dim3(kStepThreads), args, smem, st);
    if (e != cudaSuccess) return report_error(SGAD_ERR_CUDA, "sgad_gicp_track: cooperative launch failed");
    return launched("sgad_gicp_track: launch failed");
}

extern "C" sgad_status sgad_gicp_insert(const sgad_gicp_params *p, const sgad_gaussian_set *src,
                                        const sgad_gaussian_set *map, void *workspace, size_t ws_bytes, void *stream)
{
    GLayout L;
    sgad_status s = pair_checks(p, src, map, workspace, ws_bytes, &L);
    if (s) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    InsArgs a;
    a.spos = reinterpret_cast<const float4 *>(src->pos);
    a.scov = reinterpret_cast<const float4 *>(src->cov);
    a.snorm = reinterpret_cast<const float4 *>(src->normal);
    a.scount = src->count;
    a.mpos = reinterpret_cast<float4 *>(map->pos);
    a.mcov = reinterpret_cast<float4 *>(map->cov);
    a.mnorm = reinterpret_cast<float4 *>(map->normal);
    a.mcount = map->count;
    a.mcap = map->capacity;
    a.grid = grid_of(p, workspace, L);
    a.d_ov = p->d_overlap;
    a.state = at<GicpState>(workspace, L.state);
    a.flags = at<int32_t>(workspace, L.ins_flags);
    a.blk = at<int32_t>(workspace, L.ins_counts);
    sgad::launch_after(k_insert_flag, (p->src_capacity + kInsPts - 1) / kInsPts, 1024, 0, st, a);
    sgad::launch_after(k_insert_write, L.max_blocks, 256, 0, st, a);
    if ((s = launched("sgad_gicp_insert: launch failed"))) return s;
    return build_index(p, map, workspace, L, 1, st);
}

extern "C" sgad_status sgad_gicp_result(void *workspace, size_t ws_bytes, double pose[12], sgad_gicp_stats *stats,
                                        void *stream)
{
    sgad_status s = check_ws(workspace, ws_bytes, sizeof(GicpState));
    if (s) return s;
    // on the caller's stream alone: a plain copy would wait for the work of the default stream
    // too
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    GicpState h;
    if (cudaMemcpyAsync(&h, workspace, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return report_error(SGAD_ERR_CUDA, "sgad_gicp_result: copy failed");
    if (cudaStreamSynchronize(st) != cudaSuccess)
        return report_error(SGAD_ERR_CUDA, "sgad_gicp_result: stream failed");
    if (pose) std::memcpy(pose, h.pose, sizeof(h.pose));
    if (stats) {
        stats->iterations = h.iters;
        stats->converged = h.converged;
        stats->n_matches = h.n;
        stats->status = (h.status & 3) | (h.gave_up == 1 ? 4 : 0);
        stats->cost = h.cost;
        stats->step = h.step;
    }
    return SGAD_OK;
}
