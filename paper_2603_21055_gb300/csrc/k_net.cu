// Learned proposal net (workload extension; the paper initialises offsets at zero):
// 3x3 convolutions as implicit GEMMs on the tcgen05 tensor cores, bf16 operands, f32
// accumulation in tensor memory.
//
// Activations are bf16 with 16 or 32 channels (the 4-channel input and 2-channel output
// are zero-padded), stored chunk-planar: 16-byte units of 8 channels, [frame][row][channel
// chunk][pixel], so the units of one chunk of one image row are contiguous (a TMA box of a
// chunk over a row reads whole sectors).
//
// Forward and input gradient (conv_block): a tile is 128 consecutive output pixels of
// one image row (the MMA's M), all output channels and K = 9 taps x C_in. The input rows
// arrive by TMA, 130 pixels of a (row, chunk), which in shared memory is the K-major
// canonical layout; the tap column dx is a descriptor start offset of dx units, so no im2col
// copy is made, and one MMA covers the taps of a column: the output rows above, at and below
// the input row side by side as N. Weights are staged once per block in the B layout [dx]
// [channel chunk][dy = 2, 1, 0][c_out]. A producer lane, an MMA lane and four epilogue warps
// overlap loads, MMAs (a ring of TMEM accumulators) and the epilogue (bias + ReLU + bf16; or
// the ReLU-masked input gradient; or the two f32 outputs).
//
// Weight gradient (wgrad_block): dW[t][i][o] = sum_p x[p + d_t][i] dy[p][o] is a
// GEMM with the pixels as K; the same TMA boxes, read with the channels as M (x) or N
// (dy), are the MN-major canonical layout, so three taps share one M = 128 MMA (below)
// and no shared-memory transpose is needed; the accumulators stay in tensor memory for
// a chain of K blocks, then in registers, and are added to the output with one 16-byte atomic
// per (row, 4 columns) at the end of the block.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "sgad_launch.cuh"
#include "sgad_net_device.cuh"
#include "tc5.cuh"

namespace sgad {
namespace net {

constexpr uint32_t kSpinLimit = 1u << 22;   // bounded mbarrier waits (each try_wait may suspend)
constexpr int kTileM = 128;                  // output pixels per conv tile
constexpr int kRowUnits = kTileM + 2;        // staged pixels per input row (1-pixel halo)

__device__ __forceinline__ void set_status(uint32_t *status, uint32_t code)
{
    atomicCAS(status, 0u, code);
}

// Unit index of (pixel p = (frame * H + row) * W + x, channel chunk c) in a chunk-planar
// tensor with kc chunks per pixel.
__device__ __forceinline__ size_t planar_unit(size_t p, int c, int kc, int w)
{
    const size_t row = p / (size_t)w;
    return (row * kc + c) * (size_t)w + (p - row * (size_t)w);
}

// ------------------------------------------------------------------ small kernels

// (N,3,H,W) colour + (N,H,W) depth (f32) -> chunk-planar bf16, 16 channels (R, G, B, D, 0 ...).
__global__ void k_pack_input(const float *__restrict__ rgb, const float *__restrict__ depth, uint4 *__restrict__ x0,
                             int n, int h, int w)
{
    dependency_wait(rgb, depth);
    const size_t hw = (size_t)h * w, total = (size_t)n * hw;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < total; p += (size_t)gridDim.x * blockDim.x) {
        const size_t f = p / hw, q = p - f * hw;
        const float *c = rgb + f * 3 * hw + q;
        __nv_bfloat162 rg = __floats2bfloat162_rn(c[0], c[hw]);
        __nv_bfloat162 bd = __floats2bfloat162_rn(c[2 * hw], depth[p]);
        uint4 v0;
        v0.x = *reinterpret_cast<uint32_t *>(&rg);
        v0.y = *reinterpret_cast<uint32_t *>(&bd);
        v0.z = 0u;
        v0.w = 0u;
        x0[planar_unit(p, 0, 2, w)] = v0;
        x0[planar_unit(p, 1, 2, w)] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// f32 master weights W[9][ci_p][co_p] (tap 3 dy + dx) -> forward B units [dx][ci_p/8][dy =
// 2, 1, 0][co_p] (unit = 8 consecutive input channels of one output channel) and, when bwd
// != nullptr, the input-gradient B units [dx][co_p/8][dy = 2, 1, 0][ci_p] of the flipped
// taps (unit = 8 consecutive output channels of one input channel). blockIdx.y: layer.
__global__ void k_prep_weights(const PrepArgs a)
{
    dependency_wait();
    const float *w = a.w[blockIdx.y];
    uint4 *fwd = a.fwd[blockIdx.y], *bwd = a.bwd[blockIdx.y];
    const int ci_p = a.ci_p[blockIdx.y], co_p = a.co_p[blockIdx.y];
    const int n = 9 * ci_p * co_p / 8;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    {
        const int co = i % co_p, dy = 2 - i / co_p % 3, kc = i / (3 * co_p) % (ci_p / 8);
        const int t = 3 * dy + i / (3 * co_p * (ci_p / 8));
        uint32_t u[4];
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat162 v = __floats2bfloat162_rn(w[((size_t)t * ci_p + 8 * kc + 2 * j) * co_p + co],
                                                     w[((size_t)t * ci_p + 8 * kc + 2 * j + 1) * co_p + co]);
            u[j] = *reinterpret_cast<uint32_t *>(&v);
        }
        fwd[i] = make_uint4(u[0], u[1], u[2], u[3]);
    }
    if (bwd) {
        const int ci = i % ci_p, dy = 2 - i / ci_p % 3, kc = i / (3 * ci_p) % (co_p / 8);
        const int t = 3 * dy + i / (3 * ci_p * (co_p / 8));
        const int tf = 8 - t;     // (ky, kx) -> (2 - ky, 2 - kx)
        uint32_t u[4];
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat162 v = __floats2bfloat162_rn(w[((size_t)tf * ci_p + ci) * co_p + 8 * kc + 2 * j],
                                                     w[((size_t)tf * ci_p + ci) * co_p + 8 * kc + 2 * j + 1]);
            u[j] = *reinterpret_cast<uint32_t *>(&v);
        }
        bwd[i] = make_uint4(u[0], u[1], u[2], u[3]);
    }
}

// Zeroes the parameter gradients of all layers. blockIdx.y: layer.
__global__ void k_zero_grads(const ZeroArgs a)
{
    dependency_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.n_w[blockIdx.y]) a.dw[blockIdx.y][i] = 0.f;
    if (i < a.n_b[blockIdx.y]) a.db[blockIdx.y][i] = 0.f;
}

// Training loss mean_p (y0 - delta_t / 0.01)^2 + lw (y1 - logit_t)^2 and its gradient,
// written as the 16-channel bf16 output gradient (channels 0, 1; the rest zero).
__global__ void k_loss(const float2 *__restrict__ y4, const float *__restrict__ td, const float *__restrict__ tl,
                       float lw, uint4 *__restrict__ dy4, float *loss, size_t total, int w)
{
    dependency_wait(y4, td, tl);
    const float inv = 1.0f / (float)total;
    float acc = 0.f;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < total; p += (size_t)gridDim.x * blockDim.x) {
        const float2 y = y4[p];
        const float e0 = y.x - td[p] * 100.0f, e1 = y.y - tl[p];
        acc += e0 * e0 + lw * e1 * e1;
        __nv_bfloat162 g = __floats2bfloat162_rn(2.0f * e0 * inv, 2.0f * lw * e1 * inv);
        uint4 v = make_uint4(*reinterpret_cast<uint32_t *>(&g), 0u, 0u, 0u);
        dy4[planar_unit(p, 0, 2, w)] = v;
        dy4[planar_unit(p, 1, 2, w)] = make_uint4(0u, 0u, 0u, 0u);
    }
    // one addition per block: one per warp (7000 on one address at 3 x 315x237) took 9 of the
    // kernel's 12 us
    __shared__ float part[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (loss && threadIdx.x < 32) {
        acc = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.f;
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) atomicAdd(loss, acc * inv);
    }
}

// ------------------------------------------------------------------ conv (forward / input gradient)

__device__ __forceinline__ bool bf16_positive(uint32_t half_bits) { return (half_bits & 0x8000u) == 0 && (half_bits & 0x7FFFu) != 0; }

// Epilogue of output pixel x of image row `row` (frame * H + y) from its accumulator row r
// (CO f32 values); bias: this layer's, in shared memory.
template <int CO, int MODE>
__device__ __forceinline__ void conv_epilogue(const ConvArgs &a, const float *bias, size_t row, int x,
                                              const uint32_t (&r)[32])
{
    if (MODE == kModeOut) {
        const size_t p = row * (size_t)a.W + x;
        const float y0 = __uint_as_float(r[0]) + bias[0], y1 = __uint_as_float(r[1]) + bias[1];
        a.y4[p] = make_float2(y0, y1);
        if (a.delta) a.delta[p] = 0.01f * y0;
        if (a.logit) a.logit[p] = y1;
    } else {
        const size_t unit = row * (CO / 8) * (size_t)a.W + x;      // of chunk 0
        uint32_t packed[CO / 2];
        if (MODE == kModeRelu) {
#pragma unroll
            for (int c = 0; c < CO; c += 4) {
                const float4 bb = *reinterpret_cast<const float4 *>(bias + c);
                __nv_bfloat162 h0 = __floats2bfloat162_rn(fmaxf(__uint_as_float(r[c]) + bb.x, 0.0f),
                                                          fmaxf(__uint_as_float(r[c + 1]) + bb.y, 0.0f));
                __nv_bfloat162 h1 = __floats2bfloat162_rn(fmaxf(__uint_as_float(r[c + 2]) + bb.z, 0.0f),
                                                          fmaxf(__uint_as_float(r[c + 3]) + bb.w, 0.0f));
                packed[c / 2] = *reinterpret_cast<uint32_t *>(&h0);
                packed[c / 2 + 1] = *reinterpret_cast<uint32_t *>(&h1);
            }
        } else {     // kModeMask: input gradient times [activation > 0]
#pragma unroll
            for (int u = 0; u < CO / 8; ++u) {
                const uint4 mm = __ldg(&a.mask[unit + (size_t)u * a.W]);
                const uint32_t mw[4] = {mm.x, mm.y, mm.z, mm.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 8 * u + 2 * j;
                    const float v0 = bf16_positive(mw[j] & 0xFFFFu) ? __uint_as_float(r[c]) : 0.0f;
                    const float v1 = bf16_positive(mw[j] >> 16) ? __uint_as_float(r[c + 1]) : 0.0f;
                    __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
                    packed[c / 2] = *reinterpret_cast<uint32_t *>(&h);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < CO / 8; ++u)
            a.out[unit + (size_t)u * a.W] = make_uint4(packed[4 * u], packed[4 * u + 1], packed[4 * u + 2],
                                                       packed[4 * u + 3]);
    }
}

// ------------------------------------------------------------------ conv, TMA-fed pipeline
//
// A block owns a run of output tiles that follow one another down the image columns of 128
// pixels (tile order: frame, column, row with the rows fastest; the runs of two blocks
// differ by one tile at most) and streams the input rows of the run, each loaded once (and
// one above and one below every column part). Input row r takes part in the output rows
// r - 1, r and r + 1, whose accumulators lie side by side in tensor memory: one MMA of N =
// 3 C_out columns (the taps dy = 2, 1, 0 of one dx) adds to all three, so the 128 pixels are
// read from shared memory once per (dx, 16 input channels) and not once per tap. The
// accumulators are a ring of kAcc; where three of them cross its end the MMA is two.
//   warp 0 (one lane)  TMA producer: an input row arrives as CI/8 slabs [pixel][8 channels],
//                      each two boxes of consecutive 16-byte units (128, and the 2 of the
//                      halo), zero-filled outside the image, in one of kRing slots; an
//                      mbarrier per slot counts the bytes;
//   warp 1 (one lane)  MMA issuer: waits for the row and for the accumulator of the output
//                      row that starts with it, issues the MMAs (the new accumulator's
//                      first one by itself: it overwrites), and commits to the slot's
//                      "empty" barrier and the finished accumulator's "full" barrier;
//   warps 2-5          epilogue: wait for a full accumulator, read their 32 rows (warp
//                      w reads lanes 32 (w % 4) ...), release the accumulator, store.
// Every wait is bounded; a wait that gives up records a status and ends the block's loop.
//
// Bound by memory and the latency of a row's steps. 8 x 640x480: 32 -> 32 channels (315 MB
// in and out) 59 us, 16 -> 32 43, 32 -> 16 43. With every tap an MMA of its own on a row
// window of the ring: 69, 46 and 59 (48 cycles per MMA, 2/3 of them spent re-reading the
// pixels); with three rows loaded per tile as rows of 16 bytes: 129, 112 and 76. Fewer slots
// and more blocks per SM win: 2 slots 65 us, 3: 59, 4: 61, 6: 63; 8 accumulators (2 blocks) 98.
constexpr int kRing = 3;               // input row slots
constexpr int kAcc = 4;                // accumulators (C_out tensor memory columns each): three in
                                       // work, one in the epilogue
static_assert(kAcc >= 4 && (kAcc & (kAcc - 1)) == 0 && kRing >= 2, "ring sizes");
constexpr int kSlabUnits = 136;        // 16-byte units per staged (row, chunk) slab: 130 used, 128-byte aligned

template <int CI, int CO>
struct TmaConvSmem {
    static constexpr int kB = 9 * (CI / 8) * CO * 16;                 // weights (bytes)
    static constexpr int kRow = (CI / 8) * kSlabUnits * 16;           // one slot
    static constexpr uint32_t kRowTx = (CI / 8) * kRowUnits * 16;     // bytes the TMA boxes deliver
    static constexpr size_t bytes = (size_t)kB + (size_t)kRing * kRow + 1024;   // + alignment slack
};

// The units x0 - 1 .. x0 + 128 of chunk slabs of image row y into consecutive slabs at dst.
template <int KC>
__device__ __forceinline__ void load_row(uint32_t dst, const CUtensorMap &wide, const CUtensorMap &halo, int x0, int y,
                                         int n, uint64_t *bar)
{
#pragma unroll
    for (int kc = 0; kc < KC; ++kc) {
        const uint32_t d = dst + (uint32_t)(kc * kSlabUnits * 16);
        tc::tma_load_4d(d, &wide, 2 * (x0 - 1), kc, y, n, bar);
        tc::tma_load_4d(d + kTileM * 16, &halo, 2 * (x0 - 1 + kTileM), kc, y, n, bar);
    }
}

// Walks a block's run of tiles, one column part (output rows y0 .. y1 of one column of 128
// pixels of one frame) at a time.
struct TileRun {
    int y0, y1, xs, n, left;     // left: tiles of the run from y0 on
    int H, segs;
    __device__ __forceinline__ TileRun(const ConvArgs &a, int block, int blocks)
    {
        H = a.H;
        segs = (a.W + kTileM - 1) / kTileM;
        const long long total = (long long)a.N * segs * a.H;
        const long long t0 = total * block / blocks, t1 = total * (block + 1) / blocks;
        left = (int)(t1 - t0);
        const long long col = t0 / a.H;
        y0 = (int)(t0 - col * a.H);
        n = (int)(col / segs);
        xs = (int)(col - (long long)n * segs);
        y1 = min(H - 1, y0 + left - 1);
    }
    __device__ __forceinline__ void next()
    {
        left -= y1 - y0 + 1;
        y0 = 0;
        y1 = min(H - 1, left - 1);
        if (++xs == segs) xs = 0, ++n;
    }
};

// Block `block` of `blocks` of a convolution; 192 threads.
template <int CI, int CO, int MODE>
__device__ __forceinline__ void conv_block(const CUtensorMap &wide, const CUtensorMap &halo, const ConvArgs &a, int block,
                                           int blocks)
{
    static_assert(CI % 16 == 0 && (CO == 16 || CO == 32), "channel counts");
    using S = TmaConvSmem<CI, CO>;
    constexpr int kcn = CI / 8;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint4 *sB = reinterpret_cast<uint4 *>(base);
    uint8_t *sA = base + S::kB;
    __shared__ uint64_t full[kRing], empty[kRing], tfull[kAcc], tempty[kAcc], drain;
    __shared__ uint32_t taddr_s;
    __shared__ __align__(16) float bias[CO];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == 0) tc::tmem_alloc(&taddr_s, kAcc * CO);
    if (threadIdx.x == 32) {
        tc::mbar_init(&drain, 1);
        for (int i = 0; i < kRing; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < kAcc; ++i) {
            tc::mbar_init(&tfull[i], 1);
            tc::mbar_init(&tempty[i], 4);
        }
    }
    dependency_wait();
    if (MODE != kModeMask && threadIdx.x >= 64 && threadIdx.x < 64 + CO)
        bias[threadIdx.x - 64] = a.bias[threadIdx.x - 64];
#pragma unroll 6
    for (int i = threadIdx.x; i < S::kB / 16; i += 192) sB[i] = a.wB[i];
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = taddr_s;

    if (warp == 0) {
        if (lane == 0) {                                       // TMA producer
            uint32_t slot = 0, turn = 0, loads = 0;
            const uint32_t s0 = tc::smem_u32(sA);
            bool ok = true;
            for (TileRun t(a, block, blocks); t.left > 0 && ok; t.next())
                for (int r = t.y0 - 1; r <= t.y1 + 1; ++r) {
                    // (the slot's previous row landed before the MMAs that freed it ran)
                    if (!tc::mbar_wait_bounded(&empty[slot], (turn & 1) ^ 1, kSpinLimit)) {
                        ok = false;
                        break;
                    }
                    tc::mbar_arrive_expect_tx(&full[slot], S::kRowTx);
                    load_row<kcn>(s0 + slot * (uint32_t)S::kRow, wide, halo, t.xs * kTileM, r, t.n, &full[slot]);
                    ++loads;
                    if (++slot == kRing) slot = 0, ++turn;
                }
            // drain: the last rows have landed before the block may exit
            for (uint32_t q = loads < (uint32_t)kRing ? 0u : loads - kRing; q < loads; ++q)
                if (!tc::mbar_wait_bounded(&full[q % kRing], (q / kRing) & 1, kSpinLimit)) ok = false;
            if (!ok) set_status(a.status, 3u);
        }
    } else if (warp == 1) {
        if (lane == 0) {                                       // MMA issuer
            const uint64_t a0 = tc::sdesc(tc::smem_u32(sA), kSlabUnits * 16, 128);
            const uint64_t b0 = tc::sdesc(tc::smem_u32(sB), 3 * CO * 16, 128);
            uint32_t slot = 0, turn = 0;
            int k = 0;                                         // tiles before this column part
            bool ok = true;
            for (TileRun t(a, block, blocks); t.left > 0 && ok; k += t.y1 - t.y0 + 1, t.next())
                for (int r = t.y0 - 1; r <= t.y1 + 1; ++r) {
                    const int lo = max(r - 1, t.y0), hi = min(r + 1, t.y1);     // output rows
                    const int k_lo = k + lo - t.y0, k_hi = k + hi - t.y0;
                    const bool fresh = hi == r + 1;            // row hi starts
                    if (!tc::mbar_wait_bounded(&full[slot], turn & 1, kSpinLimit) ||
                        (fresh && !tc::mbar_wait_bounded(&tempty[k_hi % kAcc], ((k_hi / kAcc) & 1) ^ 1, kSpinLimit))) {
                        set_status(a.status, 3u);
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    // rows lo .. lo + n0 - 1 in accumulators up to the ring's end, then n1 from its start
                    const int rows = hi - lo + 1, n0 = min(rows, kAcc - k_lo % kAcc), n1 = rows - n0;
                    const uint32_t d0 = tmem + (uint32_t)(k_lo % kAcc * CO), d1 = tmem;
                    const uint64_t ad = a0 + (uint64_t)(slot * (uint32_t)(S::kRow / 16));
                    // taps dy = 2, 1, 0 for the output rows r - 1, r, r + 1
                    const uint64_t bd = b0 + (uint64_t)((lo - (r - 1)) * CO);
                    const uint32_t i0 = tc::idesc_bf16(kTileM, 0) + ((uint32_t)(n0 * CO / 8) << 17);
                    const uint32_t i1 = tc::idesc_bf16(kTileM, 0) + ((uint32_t)(n1 * CO / 8) << 17);
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int sk = 0; sk < CI / 16; ++sk) {
                            const uint64_t aa = ad + (uint64_t)(2 * sk * kSlabUnits + dx);
                            const uint64_t bb = bd + (uint64_t)((dx * kcn + 2 * sk) * 3 * CO);
                            if ((dx | sk) == 0 && fresh) {
                                // the new row's accumulator is overwritten, the others added to
                                constexpr uint32_t one = tc::idesc_bf16(kTileM, CO);
                                const uint32_t dn = tmem + (uint32_t)(k_hi % kAcc * CO);
                                const int m0 = min(rows - 1, n0), m1 = rows - 1 - m0;
                                if (m0) tc::mma_bf16(d0, aa, bb, i0 - ((uint32_t)((n0 - m0) * CO / 8) << 17), true);
                                if (m1) tc::mma_bf16(d1, aa, bb + (uint64_t)(m0 * CO),
                                                     i1 - ((uint32_t)((n1 - m1) * CO / 8) << 17), true);
                                tc::mma_bf16(dn, aa, bb + (uint64_t)((rows - 1) * CO), one, false);
                            } else {
                                tc::mma_bf16(d0, aa, bb, i0, true);
                                if (n1) tc::mma_bf16(d1, aa, bb + (uint64_t)(n0 * CO), i1, true);
                            }
                        }
                    tc::mma_commit(&empty[slot]);
                    if (r > t.y0) tc::mma_commit(&tfull[(k + r - 1 - t.y0) % kAcc]);    // row r - 1 is done
                    if (++slot == kRing) slot = 0, ++turn;
                }
            // drain: the last committed MMAs finish before the accumulators are freed (an
            // output row's last MMAs are the last ones of a run)
            if (ok) {
                if (k > 0) tc::mbar_wait_bounded(&tfull[(k - 1) % kAcc], ((k - 1) / kAcc) & 1, kSpinLimit);
            } else {
                tc::mma_commit(&drain);
                tc::mbar_wait_bounded(&drain, 0, kSpinLimit);
            }
        }
    } else {                                                   // epilogue warps 2..5
        const int quarter = warp & 3;
        int k = 0;
        bool ok = true;
        for (TileRun t(a, block, blocks); t.left > 0 && ok; t.next())
        for (int y = t.y0; y <= t.y1; ++y, ++k) {
            const int acc = k % kAcc;
            if (!tc::mbar_wait_bounded(&tfull[acc], (k / kAcc) & 1, kSpinLimit)) {
                if (lane == 0) set_status(a.status, 3u);
                ok = false;
                break;
            }
            tc::fence_after_sync();
            const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * CO);
            uint32_t r[32];
            {
                uint32_t q[16];
                tc::tmem_ld16(trow, q);
#pragma unroll
                for (int c = 0; c < 16; ++c) r[c] = q[c];
                if (CO == 32) {
                    tc::tmem_ld16(trow + 16, q);
#pragma unroll
                    for (int c = 0; c < 16; ++c) r[16 + c] = q[c];
                }
            }
            tc::tmem_wait_ld();
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&tempty[acc]);
            const int x = t.xs * kTileM + quarter * 32 + lane;
            if (x < a.W) conv_epilogue<CO, MODE>(a, bias, (size_t)t.n * a.H + y, x, r);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kAcc * CO);
}

template <int CI, int CO, int MODE>
__global__ void __launch_bounds__(192, 4) k_conv3x3_tma(const __grid_constant__ CUtensorMap wide,
                                                        const __grid_constant__ CUtensorMap halo, const ConvArgs a)
{
    conv_block<CI, CO, MODE>(wide, halo, a, (int)blockIdx.x, (int)gridDim.x);
}

// ------------------------------------------------------------------ weight gradient, TMA-fed
//
// The same sums, with the operands read in the layout the TMA boxes land in, so that no
// shared-memory transpose is needed. A K block is 128 consecutive pixels q of one image row
// y: the input's rows y - 1, y, y + 1 at q (one box of 3 x CI/8 slabs [pixel][8 channels] of
// 128 units) and the output gradient's row y at x0 - 1 .. x0 + 128 (CO/8 slabs of kSlabUnits
// units, two boxes each: only this operand needs the halo, which makes 9 copies per K block
// of 32 -> 32 channels instead of 28). Read with the pixels as K and the channels as M (x)
// or N (dy), a slab is the MN-major canonical layout: a core matrix is 8 pixels x 8
// channels, 128 contiguous bytes; the next 8 channels are one slab further, the next 8
// pixels 128 bytes further. The (dy, channel group) rows of the three input rows form one
// uniformly strided M dimension of 3 CI rows; tap dx pairs the input pixel q with the
// gradient pixel q + 1 - dx, a start offset of 2 - dx units, so one M = 128 MMA per (dx,
// 16-pixel K step) covers the three taps (dy, dx). The M rows after 3 CI read a slab of ones
// (row 3 CI: the bias gradient, taken from dx = 1) and then whatever follows it in the
// stage, rows whose products are not used. Accumulators: three TMEM blocks of CO columns
// (one per dx), added to dW at the end with 16-byte atomics. One thread of warp 0 issues the
// TMA loads into kWgStages stages, one thread of warp 1 the MMAs (its descriptors precomputed:
// an offset adds to the address field); warps 2 to 5 sum and add. Every wait is bounded.
//
// The final additions of all blocks meet on the same 3 CI CO addresses, so a small problem
// takes fewer blocks: kWgTiles K blocks each, at least one block per SM (4: 55 us
// for two 32 -> 32 layers of 3 x 315x237 in launches of their own, 8: 50, 32: 57).
// 3 x 315x237, 32 -> 32 channels (28 MB in) in a launch of its own: 24 us, of which the
// additions 8 and the launch, setup and drain 8; 94 us with single-float atomics from every
// resident block (4.2 M onto 9216 addresses) and 28 copies of 16-byte rows per K block.
constexpr int kWgTiles = 8;                // K blocks per block of a small problem
constexpr int kWgPix = 128;                // pixels per K block
constexpr int kWgGroups = 16;              // M groups read by an M = 128 MMA
constexpr int kWgStages = 3;               // shared-memory stages of the load pipeline

template <int CI, int CO, int STAGES = kWgStages>
struct WgradTmaSmem {
    static constexpr int kXBytes = (3 * (CI / 8) + 1) * kWgPix * 16;       // slabs of x, then the ones slab
    static constexpr int kYBytes = (CO / 8) * kSlabUnits * 16;             // slabs of dy
    // an M = 128 MMA reads kWgGroups slabs from the x base: past the ones slab it reads
    // the dy slabs (or padding), rows whose products are not used
    static constexpr int kStage = kXBytes + kYBytes > kWgGroups * kWgPix * 16 ? kXBytes + kYBytes
                                                                             : kWgGroups * kWgPix * 16;
    static constexpr uint32_t kTx = (uint32_t)(3 * (CI / 8) * kWgPix * 16 + (CO / 8) * kRowUnits * 16);
    static constexpr size_t bytes = (size_t)STAGES * kStage + 1024;   // + alignment slack
    static constexpr int kCols = 3 * CO <= 32 ? 32 : (3 * CO <= 64 ? 64 : 128);
    static_assert(3 * (CI / 8) + 1 <= kWgGroups, "the three rows and the ones slab fit one M = 128 MMA");
};

// Instruction descriptor of kind::f16, bf16 A and B both MN-major (transposed), f32
// accumulator, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N)
{
    return tc::idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// Descriptor of an MN-major operand without swizzle: the leading byte offset is the
// distance between core matrices adjacent in K (here 8 pixels, 128 bytes), the stride byte
// offset the distance between core matrices adjacent in M or N (8 channels, one slab).
// (The weight-gradient parity tests fail with the two offsets exchanged.)
__device__ __forceinline__ uint64_t sdesc_mn(uint32_t saddr, uint32_t mn_stride, uint32_t k_stride)
{
    return tc::sdesc(saddr, k_stride, mn_stride);
}

// A bounded wait of warps with nothing else to do, off the issue slots between tries.
__device__ __forceinline__ bool wait_idle(uint64_t *bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (tc::mbar_try_wait(bar, parity)) return true;
        __nanosleep(200);
    }
    return false;
}

// Block `block` of `blocks` of a weight gradient; 192 threads. The tensor core's FP32
// accumulation loses up to a last place of the sum per step, so a sum in tensor memory ends
// after a.chain K blocks, and warps 2-5 add it to FP32 registers, rounded to nearest. With one
// sum per block of twelve K blocks the last layer's gradient of 3 x 315x237 was 1.7 times as
// far from FP64 as with 304 blocks of seven; now every layer is as far as those or nearer.
// The sums cost the backward 15 us of 105 at 3 x 315x237; added to the output with atomics
// instead of kept in registers, 29.
template <int CI, int CO, int STAGES>
__device__ __forceinline__ void wgrad_block(const CUtensorMap &xmap, const CUtensorMap &ywide, const CUtensorMap &yhalo,
                                            const WgradArgs &a, int block, int blocks)
{
    static_assert(CI % 16 == 0 && (CO == 16 || CO == 32), "channel counts");
    using S = WgradTmaSmem<CI, CO, STAGES>;
    constexpr int kcx = CI / 8, kcy = CO / 8;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[STAGES], empty[STAGES], sum_full, sum_empty;
    __shared__ uint32_t taddr_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int segs = (a.W + kWgPix - 1) / kWgPix;
    const int n_kb = a.N * a.H * segs;          // < 2^31 (checked by the launcher)

    if (warp == 0) tc::tmem_alloc(&taddr_s, S::kCols);
    if (threadIdx.x == 32) {
        for (int i = 0; i < STAGES; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        tc::mbar_init(&sum_full, 1);
        tc::mbar_init(&sum_empty, 4);
    }
    // the slab after the three input rows: ones (first element of each unit)
    for (int st = 0; st < STAGES; ++st) {
        uint4 *x = reinterpret_cast<uint4 *>(base + (size_t)st * S::kStage) + 3 * kcx * kWgPix;
        for (int i = threadIdx.x; i < kWgPix; i += blockDim.x) x[i] = make_uint4(0x3F80u, 0u, 0u, 0u);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    dependency_wait();
    const uint32_t tmem = taddr_s;
    constexpr uint32_t idesc = idesc_bf16_mn(128, CO);

    if (threadIdx.x == 0) {                                    // TMA producer
        int k = 0;
        bool ok = true;
        for (int kb = block; kb < n_kb; kb += blocks, ++k) {
            const int st = k % STAGES;
            if (!tc::mbar_wait_bounded(&empty[st], (uint32_t)(((k / STAGES) & 1) ^ 1), kSpinLimit)) {
                ok = false;
                break;
            }
            const int xs = kb % segs, ry = kb / segs;
            const int y = ry % a.H, n = ry / a.H;
            const uint32_t xb = tc::smem_u32(base + (size_t)st * S::kStage), yb = xb + (uint32_t)S::kXBytes;
            tc::mbar_arrive_expect_tx(&full[st], S::kTx);
            tc::tma_load_4d(xb, &xmap, 2 * xs * kWgPix, 0, y - 1, n, &full[st]);
            load_row<kcy>(yb, ywide, yhalo, xs * kWgPix, y, n, &full[st]);
        }
        // drain: the last boxes have landed before the block may exit
        if (k > 0 && !tc::mbar_wait_bounded(&full[(k - 1) % STAGES], (uint32_t)(((k - 1) / STAGES) & 1), kSpinLimit))
            ok = false;
        if (!ok) set_status(a.status, 3u);
    } else if (threadIdx.x == 32) {                           // MMA issuer
        // descriptors of stage 0 at offset 0; an offset of o bytes adds o / 16
        const uint32_t x0 = tc::smem_u32(base), y0 = x0 + (uint32_t)S::kXBytes;
        const uint64_t ad0 = sdesc_mn(x0, kWgPix * 16, 128), bd0 = sdesc_mn(y0, kSlabUnits * 16, 128);
        int k = 0, in_sum = 0;                                 // K blocks in the current sum
        uint32_t sums = 0;
        bool ok = true;
        for (int kb = block; kb < n_kb; kb += blocks, ++k) {
            const int st = k % STAGES;
            if (!tc::mbar_wait_bounded(&full[st], (uint32_t)((k / STAGES) & 1), kSpinLimit) ||
                (in_sum == 0 && !tc::mbar_wait_bounded(&sum_empty, (sums & 1) ^ 1, kSpinLimit))) {
                ok = false;
                break;
            }
            tc::fence_after_sync();
            const uint64_t so = (uint64_t)(st * S::kStage / 16);
#pragma unroll
            for (int s = 0; s < kWgPix / 16; ++s)
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
                    tc::mma_bf16(tmem + (uint32_t)(dx * CO), ad0 + so + (uint64_t)(s * 16),
                                 bd0 + so + (uint64_t)(2 - dx + s * 16), idesc, (in_sum | s) != 0);
            tc::mma_commit(&empty[st]);
            if (++in_sum == a.chain || kb + blocks >= n_kb) {
                tc::mma_commit(&sum_full);
                in_sum = 0;
                ++sums;
            }
        }
        // drain: the last MMAs have completed before the accumulators are freed
        if (k > 0 && !tc::mbar_wait_bounded(&empty[(k - 1) % STAGES], (uint32_t)(((k - 1) / STAGES) & 1), kSpinLimit))
            ok = false;
        if (!ok) set_status(a.status, 2u);
    } else if (warp >= 2 && warp < 6) {                       // sums
        constexpr int kParts = 3 * (CO / 16);                  // of 16 columns
        const int quarter = warp & 3, row = 32 * quarter + lane;
        const int n_k = block < n_kb ? (n_kb - block + blocks - 1) / blocks : 0, n_sums = (n_k + a.chain - 1) / a.chain;
        float acc[kParts][16];
#pragma unroll
        for (int p = 0; p < kParts; ++p)
#pragma unroll
            for (int c = 0; c < 16; ++c) acc[p][c] = 0.f;
        bool ok = n_k > 0;
        for (int i = 0; i < n_sums; ++i) {
            if (!wait_idle(&sum_full, (uint32_t)(i & 1))) {
                if (lane == 0) set_status(a.status, 2u);
                ok = false;
                break;
            }
            tc::fence_after_sync();
#pragma unroll
            for (int p = 0; p < kParts; ++p) {
                uint32_t q[16];
                tc::tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(p * 16), q);
                tc::tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 16; ++c) acc[p][c] += __uint_as_float(q[c]);
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sum_empty);
        }
        const auto add = [&](int p) {
            const int dx = p / (CO / 16), c0 = p % (CO / 16) * 16;
            if (row < 3 * CI) {
                const int tap = 3 * (row / CI) + dx, ci = row % CI;
                float *dst = a.dw + ((size_t)tap * CI + ci) * CO + c0;
                if (a.vec) {
#pragma unroll
                    for (int c = 0; c < 16; c += 4)
                        atomicAdd(reinterpret_cast<float4 *>(dst + c),
                                  make_float4(acc[p][c], acc[p][c + 1], acc[p][c + 2], acc[p][c + 3]));
                } else {
#pragma unroll
                    for (int c = 0; c < 16; ++c) atomicAdd(dst + c, acc[p][c]);
                }
            } else if (row == 3 * CI && dx == 1) {
#pragma unroll
                for (int c = 0; c < 16; ++c) atomicAdd(a.db + c0 + c, acc[p][c]);
            }
        };
        // neighbouring blocks start at opposite ends
        if (ok && (block & 1)) {
#pragma unroll
            for (int p = kParts - 1; p >= 0; --p) add(p);
        } else if (ok) {
#pragma unroll
            for (int p = 0; p < kParts; ++p) add(p);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, S::kCols);
}

template <int CI, int CO>
__global__ void __launch_bounds__(192, 2) k_conv3x3_wgrad_tma(const __grid_constant__ CUtensorMap xmap,
                                                           const __grid_constant__ CUtensorMap ywide,
                                                           const __grid_constant__ CUtensorMap yhalo,
                                                           const WgradArgs a)
{
    wgrad_block<CI, CO, kWgStages>(xmap, ywide, yhalo, a, (int)blockIdx.x, (int)gridDim.x);
}

// Both gradients of a layer (CI channels in, CO out) side by side: the first n_conv blocks the
// input gradient, the others the weight gradient. Each is a chain of latencies at small sizes
// and leaves bandwidth at large ones: the net's backward of 1 x 315x237 takes 71 us against 76
// with a launch each, of 3 x 315x237 106 against 131, of 2 x 640x480 162 against 183, of 4 x
// 640x480 284 against 309, of 8 x 640x480 533 against 545, of 8 x 1200x680 1455 against 1445. At
// most half of the blocks for the weight gradient (three eighths 314 us at 4 x 640x480 and 588 at
// 8, five eighths 291 and 542), and one per 8 K blocks (one per 12: 81 us at 1 x 315x237).
constexpr int kPairStages = 2;             // load stages of the weight gradient: three blocks fit an SM
constexpr int kPairBlocks = 3;
template <int CI, int CO>
__global__ void __launch_bounds__(192, kPairBlocks) k_conv3x3_grads(const __grid_constant__ CUtensorMap xmap,
                                                                    const __grid_constant__ CUtensorMap ywide,
                                                                    const __grid_constant__ CUtensorMap yhalo,
                                                                    const ConvArgs c, const WgradArgs w, int n_conv)
{
    const int b = (int)blockIdx.x;
    if (b < n_conv)
        conv_block<CO, CI, kModeMask>(ywide, yhalo, c, b, n_conv);
    else
        wgrad_block<CI, CO, kPairStages>(xmap, ywide, yhalo, w, b - n_conv, (int)gridDim.x - n_conv);
}

// ------------------------------------------------------------------ launchers

namespace {

// Blocks of a persistent grid: resident blocks per SM (from the kernel's registers and
// shared memory and the SM's limits) times SMs, at most `work`.
int resident_grid(const void *fn, size_t smem, long long work, int threads = 128)
{
    int dev = 0, sms = 1, smem_sm = 0, regs_sm = 65536, reserved = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    cudaFuncAttributes fa;
    int per_sm = 1;
    if (cudaFuncGetAttributes(&fa, fn) == cudaSuccess) {
        const size_t block_smem = smem + fa.sharedSizeBytes + (size_t)reserved;
        const int by_smem = block_smem ? (int)((size_t)smem_sm / block_smem) : 16;
        const int regs = fa.numRegs > 0 ? fa.numRegs : 64;
        const int warps = (threads + 31) / 32;
        const int by_regs = regs_sm / (((regs * 32 + 255) / 256) * 256 * warps);
        per_sm = by_smem < by_regs ? by_smem : by_regs;
        if (per_sm > 2048 / (warps * 32)) per_sm = 2048 / (warps * 32);         // 2048 threads per SM
        if (per_sm < 1) per_sm = 1;
    }
    long long g = (long long)per_sm * sms;
    if (g > work) g = work;
    return (int)(g > 0 ? g : 1);
}

template <class F>
cudaError_t set_smem(F *fn, size_t bytes)
{
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    return e;
}

}  // namespace

// cuTensorMapEncodeTiled from the driver, fetched once through the runtime.
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

cudaError_t encode_tiled(EncodeTiledFn *out)
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !p) return cudaErrorNotSupported;
        fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    *out = fn;
    return cudaSuccess;
}

// Tensor map of a chunk-planar bf16 activation with ci channels, with the W 16-byte units
// (8 channels of a pixel) of a chunk of an image row as 2 W 8-byte elements in a row: dims
// (2 W, ci/8, H, N), boxes of box_px consecutive units of box_kc chunks of box_rows rows, zero
// fill outside. (With the 8
// channels as the inner dimension a box is box_px rows of 16 bytes, and the copy engine's
// rate in rows bounded every convolution: 129 us for 32 -> 32 channels at 8 x 640x480.)
cudaError_t input_map(const void *base, int ci, int n, int h, int w, CUtensorMap *m, int box_px, int box_kc = 1,
                      int box_rows = 1)
{
    EncodeTiledFn fn = nullptr;
    cudaError_t e = encode_tiled(&fn);
    if (e != cudaSuccess) return e;
    const cuuint64_t kc = (cuuint64_t)(ci / 8);
    const cuuint64_t dims[4] = {2 * (cuuint64_t)w, kc, (cuuint64_t)h, (cuuint64_t)n};
    const cuuint64_t strides[3] = {(cuuint64_t)w * 16, kc * w * 16, (cuuint64_t)h * kc * w * 16};
    const cuuint32_t box[4] = {2 * (cuuint32_t)box_px, (cuuint32_t)box_kc, (cuuint32_t)box_rows, 1};
    const cuuint32_t elem[4] = {1, 1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_INT64, 4, const_cast<void *>(base), dims, strides, box, elem,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int CI, int CO, int MODE>
cudaError_t launch_conv(const ConvArgs &a, cudaStream_t st)
{
    const size_t smem = TmaConvSmem<CI, CO>::bytes;
    cudaError_t e = set_smem(k_conv3x3_tma<CI, CO, MODE>, smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)a.N * a.H * ((a.W + kTileM - 1) / kTileM);
    if (tiles <= 0) return cudaSuccess;
    CUtensorMap wide, halo;
    e = input_map(a.in, CI, a.N, a.H, a.W, &wide, kTileM);
    if (e == cudaSuccess) e = input_map(a.in, CI, a.N, a.H, a.W, &halo, 2);
    if (e != cudaSuccess) return e;
    int grid = resident_grid((const void *)k_conv3x3_tma<CI, CO, MODE>, smem, tiles, 192);
    // tensor memory: 512 columns per SM
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (grid > sms * (512 / (kAcc * CO))) grid = sms * (512 / (kAcc * CO));
    return launch_after(k_conv3x3_tma<CI, CO, MODE>, grid, 192, smem, st, wide, halo, a);
}

// K blocks of one sum in tensor memory: what a block would take if there were two per SM.
int sum_chain(long long k_blocks, int sms) { return (int)std::max<long long>(1, k_blocks / (2 * sms)); }

template <int CI, int CO>
cudaError_t launch_wgrad(WgradArgs a, cudaStream_t st)
{
    using S = WgradTmaSmem<CI, CO>;
    cudaError_t e = set_smem(k_conv3x3_wgrad_tma<CI, CO>, S::bytes);
    if (e != cudaSuccess) return e;
    const long long blocks = (long long)a.N * a.H * ((a.W + kWgPix - 1) / kWgPix);
    if (blocks <= 0) return cudaSuccess;
    if (blocks >= (1ll << 31)) return cudaErrorInvalidValue;
    CUtensorMap xm, wide, halo;
    e = input_map(a.x, CI, a.N, a.H, a.W, &xm, kWgPix, CI / 8, 3);
    if (e == cudaSuccess) e = input_map(a.dy, CO, a.N, a.H, a.W, &wide, kTileM);
    if (e == cudaSuccess) e = input_map(a.dy, CO, a.N, a.H, a.W, &halo, 2);
    if (e != cudaSuccess) return e;
    // keep (resident blocks x TMEM columns) within the 512 columns of an SM
    int grid = resident_grid((const void *)k_conv3x3_wgrad_tma<CI, CO>, S::bytes, blocks, 192);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long cap = (long long)sms * (512 / S::kCols);
    if (grid > cap) grid = (int)cap;
    const long long by_work = blocks / kWgTiles;
    if (grid > by_work) grid = (int)(by_work > sms ? by_work : (grid < sms ? grid : sms));
    a.chain = sum_chain(blocks, sms);
    return launch_after(k_conv3x3_wgrad_tma<CI, CO>, grid, 192, S::bytes, st, xm, wide, halo, a);
}

template <int CI, int CO>
cudaError_t launch_grads(const ConvArgs &c, WgradArgs w, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (long long)c.N * c.H * ((c.W + kTileM - 1) / kTileM);
    constexpr size_t smem = WgradTmaSmem<CI, CO, kPairStages>::bytes > TmaConvSmem<CO, CI>::bytes
                                ? WgradTmaSmem<CI, CO, kPairStages>::bytes
                                : TmaConvSmem<CO, CI>::bytes;
    cudaError_t e = set_smem(k_conv3x3_grads<CI, CO>, smem);
    if (e != cudaSuccess || tiles <= 0) return e;
    CUtensorMap xm, wide, halo;
    e = input_map(w.x, CI, w.N, w.H, w.W, &xm, kWgPix, CI / 8, 3);
    if (e == cudaSuccess) e = input_map(w.dy, CO, w.N, w.H, w.W, &wide, kTileM);
    if (e == cudaSuccess) e = input_map(w.dy, CO, w.N, w.H, w.W, &halo, 2);
    if (e != cudaSuccess) return e;
    // (tiles and K blocks are the same in number)
    const int room = kPairBlocks * sms;
    const int n_wgrad = (int)std::min<long long>(std::max<long long>(1, tiles / kWgTiles), room / 2);
    const int n_conv = (int)std::min<long long>(tiles, room - n_wgrad);
    w.chain = sum_chain(tiles, sms);
    return launch_after(k_conv3x3_grads<CI, CO>, n_conv + n_wgrad, 192, smem, st, xm, wide, halo, c, w, n_conv);
}

template cudaError_t launch_conv<16, 32, kModeRelu>(const ConvArgs &, cudaStream_t);
template cudaError_t launch_conv<32, 32, kModeRelu>(const ConvArgs &, cudaStream_t);
template cudaError_t launch_conv<32, 16, kModeOut>(const ConvArgs &, cudaStream_t);
template cudaError_t launch_wgrad<16, 32>(WgradArgs, cudaStream_t);
template cudaError_t launch_grads<32, 32>(const ConvArgs &, WgradArgs, cudaStream_t);
template cudaError_t launch_grads<32, 16>(const ConvArgs &, WgradArgs, cudaStream_t);

cudaError_t launch_pack_input(const float *rgb, const float *depth, uint4 *x0, int n, int h, int w, cudaStream_t st)
{
    const size_t total = (size_t)n * h * w;
    if (!total) return cudaSuccess;
    const int grid = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
    return launch_after(k_pack_input, grid, 256, 0, st, rgb, depth, x0, n, h, w);
}

cudaError_t launch_prep_weights(const PrepArgs &a, cudaStream_t st)
{
    int n = 0;
    for (int l = 0; l < kLayers; ++l) n = max(n, 9 * a.ci_p[l] * a.co_p[l] / 8);
    return launch_after(k_prep_weights, dim3((n + 127) / 128, kLayers), 128, 0, st, a);
}

cudaError_t launch_zero_grads(const ZeroArgs &a, cudaStream_t st)
{
    int n = 0;
    for (int l = 0; l < kLayers; ++l) n = max(n, max(a.n_w[l], a.n_b[l]));
    return launch_after(k_zero_grads, dim3((n + 255) / 256, kLayers), 256, 0, st, a);
}

cudaError_t launch_loss(const float2 *y4, const float *td, const float *tl, float lw, uint4 *dy4, float *loss,
                        size_t total, int w, cudaStream_t st)
{
    if (!total) return cudaSuccess;
    const int grid = (int)((total + 255) / 256 < 2048 ? (total + 255) / 256 : 2048);
    return launch_after(k_loss, grid, 256, 0, st, y4, td, tl, lw, dy4, loss, total, w);
}

}  // namespace net
}  // namespace sgad
