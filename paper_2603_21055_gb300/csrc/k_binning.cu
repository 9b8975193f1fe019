// Projection and tile binning (forward steps a1-a4).
//
//   k_project_count : per Gaussian, the world centre mu = R_i (|D + delta| r) + t_i
//                     (Sec. 3.2), opacity sigmoid(logit), the view-independent record,
//                     and for every view the tile rectangle of its 3-sigma square;
//                     per-tile counts with warp-aggregated atomics.
//   k_scan_tiles    : exclusive scan of the per-tile counts -> list offsets; flags a
//                     key overflow.
//   k_emit          : per Gaussian and view, one 8-byte entry (f32 depth bits << 32 |
//                     Gaussian index) per tile of the rectangle the count kernel left in
//                     the workspace (8 bytes per Gaussian and view), written into the
//                     tile's bucket. The depth is evaluated in double-float so the key is
//                     the exactly-rounded f32 of the view depth. For the warp-local passes
//                     the index takes 24 bits and the low 8 say which of the tile's 8x4
//                     pixel blocks the Gaussian's alpha >= 1/255 box may touch (the sort
//                     keeps its order and separates the two).
#include "sgad_device.cuh"
#include "sgad_launch.cuh"

namespace sgad {

constexpr int kOrderClasses = 128;
// Tiles of a lane whose cursor updates are under way together: two measure 263 us on the room
// workload (8 x 640x480 keyframes into 8 views), one and four 278. (Runs of neighbouring
// lanes with the same tile in place of the match cost the count 12 us more.)
constexpr int kEmitAhead = 2;

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// TRIM: the rectangles carry the block trims that the packed emission forms masks from (the
// projection is at hand here). The trims are those of the Gaussian's own alpha >= 1/255 box:
// with the bound sqrt(2 ln 255) sqrt(lambda_max) of its extents for any opacity, which needs
// no logarithm, this kernel is 6 us faster on the room workload and the forward 56 us slower.
template <bool TRIM>
__global__ void __launch_bounds__(256) k_project_count(const __grid_constant__ Scene sc, World *__restrict__ world,
                                                       uint32_t *__restrict__ tile_cnt, uint2 *__restrict__ rects)
{
    dependency_wait();
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = g < sc.n_gauss;
    float4 w0 = make_float4(0.f, 0.f, 0.f, 0.f);
    float reach = 0.f;               // 2 ln(255 o), as in stage()
    if (valid) {
        const KfDev &k = sc.kf[find_kf(sc, g)];
        const uint32_t j = g - k.gbase;
        const int u = (int)(j % (uint32_t)k.W), v = (int)(j / (uint32_t)k.W);
        const size_t hw = (size_t)k.W * k.H;
        const float D = k.depth[j], delta = k.offset[j];
        const float d = fabsf(__fadd_rn(D, delta));
        const float rx = __fdiv_rn(__fsub_rn((float)u, k.cx), k.fx);
        const float ry = __fdiv_rn(__fsub_rn((float)v, k.cy), k.fy);
        const float qx = __fmul_rn(d, rx), qy = __fmul_rn(d, ry);
        w0.x = __fmaf_rn(k.R[0], qx, __fmaf_rn(k.R[1], qy, __fmaf_rn(k.R[2], d, k.t[0])));
        w0.y = __fmaf_rn(k.R[3], qx, __fmaf_rn(k.R[4], qy, __fmaf_rn(k.R[5], d, k.t[1])));
        w0.z = __fmaf_rn(k.R[6], qx, __fmaf_rn(k.R[7], qy, __fmaf_rn(k.R[8], d, k.t[2])));
        if (k.xform) {          // device transform of the centres: mu <- R mu + t
            const float *X = k.xform;
            const float mx = w0.x, my = w0.y, mz = w0.z;
            w0.x = __fmaf_rn(X[0], mx, __fmaf_rn(X[1], my, __fmaf_rn(X[2], mz, X[3])));
            w0.y = __fmaf_rn(X[4], mx, __fmaf_rn(X[5], my, __fmaf_rn(X[6], mz, X[7])));
            w0.z = __fmaf_rn(X[8], mx, __fmaf_rn(X[9], my, __fmaf_rn(X[10], mz, X[11])));
        }
        w0.w = k.scale[j];
        const float o = 1.0f / (1.0f + expf(-k.logit[j]));
        World w;
        w.w0 = w0;
        w.w1 = make_float4(o, k.rgb[j], k.rgb[hw + j], k.rgb[2 * hw + j]);
        world[g] = w;
        if (TRIM) reach = 2.0f * (__logf(255.0f * o) + 2e-6f) * 1.0001f;
    }
    const unsigned full = 0xffffffffu;
    for (int vi = 0; vi < sc.n_views; ++vi) {
        const ViewDev &v = sc.view[vi];
        Rect r;
        int n = 0;
        if (valid) {
            const Proj p = project(w0, v);
            n = bin_rect(p, v, sc.tw_log2, sc.th_log2, r);
            if (rects) {
                Trim tx = {0, 0}, ty = {0, 0};
                if (TRIM && n > 0) {
                    // stage()'s box with a wider pad; a Gaussian below the alpha floor
                    // everywhere is trimmed from both ends
                    if (reach > 0.0f) {
                        const float ex = reach * p.cxx, ey = reach * p.cyy;
                        const int cl = sc.tw_log2 - 3, rl = sc.th_log2 - 2;
                        tx = block_trim(p.px, ex * rsqrtf(ex) + 0.03f, 0.125f, r.tx0 << cl, r.nx << cl);
                        ty = block_trim(p.py, ey * rsqrtf(ey) + 0.03f, 0.25f, r.ty0 << rl, r.ny << rl);
                    } else {
                        tx = ty = {15, 15};
                    }
                }
                rects[(size_t)vi * sc.n_gauss + g] = pack_rect(r, n, tx, ty);
            }
        }
        const int maxn = __reduce_max_sync(full, n);
        uint32_t row = (uint32_t)(v.tile_base + r.ty0 * v.tiles_x + r.tx0);   // first tile of the current rectangle row
        int col = 0;
        for (int i = 0; i < maxn; ++i) {
            uint32_t tile = kInvalidTile;
            if (i < n) {
                tile = row + (uint32_t)col;
                if (++col == r.nx) {
                    col = 0;
                    row += (uint32_t)v.tiles_x;
                }
            }
            const uint32_t peers = __match_any_sync(full, tile);
            if (tile != kInvalidTile && (threadIdx.x & 31) == __ffs(peers) - 1)
                atomicAdd(&tile_cnt[tile], (uint32_t)__popc(peers));
        }
    }
}

// Position of a tile with `len` list entries in the heavy-first order: 128 classes, four
// per power of two of the length, longest first (lengths 0 and 1 share the last class).
__device__ __forceinline__ int order_class(uint32_t len)
{
    if (len <= 1) return kOrderClasses - 1;
    const int e = 31 - __clz(len);
    const int sub = e >= 2 ? (int)((len >> (e - 2)) & 3u) : (int)((len << (2 - e)) & 3u);
    return kOrderClasses - 1 - (4 * e + sub);
}

// Single-CTA exclusive scan of the per-tile counts (1024 threads, 4 tiles per thread per
// round). Also resets the counts to serve as emission cursors and, when `order` is
// given, writes the tiles in heavy-first order (by list-length class; the order within a
// class is unspecified) for the persistent compositing schedule.
__global__ void __launch_bounds__(1024) k_scan_tiles(uint32_t *__restrict__ cnt, uint32_t *__restrict__ off, int n_tiles,
                                                     uint64_t key_cap, WsHeader *hdr, uint32_t *__restrict__ order)
{
    dependency_wait();
    __shared__ uint32_t warp_sums[32];
    __shared__ uint64_t carry_s;
    __shared__ uint32_t cls_cnt[kOrderClasses];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int base = 0; base < n_tiles; base += 4096) {
        uint32_t c[4];
        uint32_t sum = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = base + threadIdx.x * 4 + q;
            c[q] = i < n_tiles ? cnt[i] : 0u;
            sum += c[q];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sums[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            uint32_t ws = warp_sums[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, ws, o);
                if (lane >= o) ws += y;
            }
            warp_sums[lane] = ws;       // inclusive over warps
        }
        __syncthreads();
        const uint64_t carry = carry_s;
        uint64_t run = carry + (wid > 0 ? warp_sums[wid - 1] : 0u) + (incl - sum);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = base + threadIdx.x * 4 + q;
            if (i < n_tiles) {
                off[i] = (uint32_t)(run < 0xffffffffull ? run : 0xffffffffull);
                cnt[i] = 0u;
            }
            run += c[q];
        }
        __syncthreads();
        if (threadIdx.x == 0) carry_s = carry + warp_sums[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const uint64_t total = carry_s;
        off[n_tiles] = (uint32_t)(total < 0xffffffffull ? total : 0xffffffffull);
        hdr->n_keys = (uint32_t)(total < 0xffffffffull ? total : 0xffffffffull);
        hdr->needed = (uint32_t)(total < 0xffffffffull ? total : 0xffffffffull);
        hdr->overflow = total > key_cap ? 1u : 0u;
        if (total > key_cap) {
            record_error(hdr, SGAD_ERR_KEY_OVERFLOW);
            atomicMax(&hdr->sticky_needed, (uint32_t)(total < 0xffffffffull ? total : 0xffffffffull));
        }
    }
    if (!order) return;
    // heavy-first order: class histogram, exclusive scan of the classes, scatter
    for (int i = threadIdx.x; i < kOrderClasses; i += blockDim.x) cls_cnt[i] = 0u;
    __syncthreads();     // also makes this block's writes of off[] visible to all its threads
    for (int i = threadIdx.x; i < n_tiles; i += blockDim.x) atomicAdd(&cls_cnt[order_class(off[i + 1] - off[i])], 1u);
    __syncthreads();
    if (threadIdx.x < 32) {
        constexpr int kPer = kOrderClasses / 32;
        uint32_t c[kPer], sum = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            c[q] = cls_cnt[threadIdx.x * kPer + q];
            sum += c[q];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t run = incl - sum;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            cls_cnt[threadIdx.x * kPer + q] = run;
            run += c[q];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_tiles; i += blockDim.x)
        order[atomicAdd(&cls_cnt[order_class(off[i + 1] - off[i])], 1u)] = (uint32_t)i;
}

// Bits lo .. hi (<= 31); zero when empty.
__device__ __forceinline__ uint32_t bit_range(int lo, int hi) { return lo <= hi ? (2u << hi) - (1u << lo) : 0u; }

// Row bits of a tile's block mask at the stride of its columns (1 << cl of them).
__device__ __forceinline__ uint32_t spread_rows(uint32_t r, int cl)
{
    if (cl == 1) {                                      // four rows to every second bit
        r = (r | (r << 2)) & 0x33u;
        r = (r | (r << 1)) & 0x55u;
    } else if (cl == 2) {                               // two rows to bits 0 and 4
        r = (r & 1u) | ((r & 2u) << 3);
    }
    return r;
}

template <bool PACK>
__global__ void __launch_bounds__(256) k_emit(const __grid_constant__ Scene sc, const uint2 *__restrict__ rects,
                                              const uint32_t *__restrict__ off, uint32_t *__restrict__ cursor,
                                              uint64_t *__restrict__ entries, WsHeader *hdr)
{
    dependency_wait(rects, off);
    if (hdr->overflow) return;
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = g < sc.n_gauss;
    dvec3 m = {};
    if (valid) {
        const KfDev &k = sc.kf[find_kf(sc, g)];
        const uint32_t j = g - k.gbase;
        m = df_world_point(k, (int)(j % (uint32_t)k.W), (int)(j / (uint32_t)k.W), k.depth[j], k.offset[j]);
        if (k.xform) m = df_transform(m, k.xform);
    }
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int cl = sc.tw_log2 - 3, rl = sc.th_log2 - 2;       // log2 of a tile's block columns and rows
    for (int vi = 0; vi < sc.n_views; ++vi) {
        const ViewDev &v = sc.view[vi];
        Rect r;
        int n = 0;
        uint2 q = make_uint2(0u, 0u);
        if (valid) {
            q = rects[(size_t)vi * sc.n_gauss + g];           // the count kernel's rectangle
            n = unpack_rect(q, r);
        }
        const int maxn = __reduce_max_sync(full, n);
        if (maxn == 0) continue;
        uint64_t key = 0;
        // The untrimmed block columns and rows of the rectangle as bits, shifted along with the
        // walk over its tiles (all blocks of a rectangle of more than 32 either way).
        uint32_t cols0 = ~0u, cols = ~0u, rows = ~0u, spread = 0xffu;
        bool big = true;
        if (n > 0) {
            key = ((uint64_t)__float_as_uint(df_view_depth(m, v)) << 32) | (PACK ? g << 8 : g);
            if (PACK) {
                big = (r.nx << cl) > 32 || (r.ny << rl) > 32;
                const Trim tx = unpack_trim(q.x), ty = unpack_trim(q.y);
                cols0 = cols = bit_range(tx.lo, (r.nx << cl) - 1 - tx.hi);
                rows = bit_range(ty.lo, (r.ny << rl) - 1 - ty.hi);
                spread = spread_rows(rows & ((1u << (1 << rl)) - 1u), cl);
            }
        }
        uint32_t row = (uint32_t)(v.tile_base + r.ty0 * v.tiles_x + r.tx0);
        int col = 0;
        // kEmitAhead tiles of every lane at a time
        for (int i0 = 0; i0 < maxn; i0 += kEmitAhead) {
            uint32_t tile[kEmitAhead], blocks[kEmitAhead], peers[kEmitAhead], base[kEmitAhead];
#pragma unroll
            for (int k = 0; k < kEmitAhead; ++k) {
                tile[k] = kInvalidTile;
                blocks[k] = 0u;
                if (i0 + k < n) {
                    tile[k] = row + (uint32_t)col;
                    if (PACK) {
                        blocks[k] = big ? 0xffu : spread * (cols & ((1u << (1 << cl)) - 1u));
                        cols >>= 1 << cl;
                    }
                    if (++col == r.nx) {
                        col = 0;
                        row += (uint32_t)v.tiles_x;
                        if (PACK) {
                            cols = cols0;
                            rows >>= 1 << rl;
                            spread = spread_rows(rows & ((1u << (1 << rl)) - 1u), cl);
                        }
                    }
                }
                base[k] = peers[k] = 0u;
                if (i0 + k < maxn) {
                    peers[k] = __match_any_sync(full, tile[k]);
                    if (tile[k] != kInvalidTile && lane == __ffs(peers[k]) - 1)
                        base[k] = atomicAdd(&cursor[tile[k]], (uint32_t)__popc(peers[k]));
                }
            }
#pragma unroll
            for (int k = 0; k < kEmitAhead; ++k) {
                if (i0 + k >= maxn) continue;
                const uint32_t first = __shfl_sync(full, base[k], __ffs(peers[k]) - 1);
                if (tile[k] != kInvalidTile) {
                    const uint32_t slot = off[tile[k]] + first + __popc(peers[k] & lanemask_lt());
                    if (slot < off[tile[k] + 1]) {
                        entries[slot] = key | blocks[k];
                    } else {
                        atomicExch(&hdr->emit_overrun, 1u);
                        atomicExch(&hdr->sticky_overrun, 1u);
                    }
                }
            }
        }
    }
}

void launch_project_count(const Scene &sc, World *world, uint32_t *tile_cnt, uint2 *rects, bool trim, cudaStream_t st)
{
    const unsigned blocks = (sc.n_gauss + 255) / 256;
    if (!blocks) return;
    if (trim)
        launch_after(k_project_count<true>, blocks, 256, 0, st, sc, world, tile_cnt, rects);
    else
        launch_after(k_project_count<false>, blocks, 256, 0, st, sc, world, tile_cnt, rects);
}

void launch_scan_tiles(uint32_t *cnt, uint32_t *off, int n_tiles, uint64_t key_cap, WsHeader *hdr, uint32_t *order,
                       cudaStream_t st)
{
    launch_after(k_scan_tiles, 1, 1024, 0, st, cnt, off, n_tiles, key_cap, hdr, order);
}

// pack: entries with block masks (n_gauss <= 2^24, rectangles with trims).
void launch_emit(const Scene &sc, const uint2 *rects, const uint32_t *off, uint32_t *cursor, uint64_t *entries,
                 WsHeader *hdr, bool pack, cudaStream_t st)
{
    const unsigned blocks = (sc.n_gauss + 255) / 256;
    if (!blocks) return;
    if (pack)
        launch_after(k_emit<true>, blocks, 256, 0, st, sc, rects, off, cursor, entries, hdr);
    else
        launch_after(k_emit<false>, blocks, 256, 0, st, sc, rects, off, cursor, entries, hdr);
}

}  // namespace sgad
