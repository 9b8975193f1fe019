// Per-Gaussian and per-pixel elementwise kernels:
//   k_finalize   : last link of the adjoint (a10): d |D + delta| -> d delta,
//                  d opacity -> d logit, written into the caller's gradient planes of
//                  learnable keyframes.
//   k_l1_grad    : L1 terms of Eq. 1 and their image gradients (a8).
//   k_adam       : bias-corrected Adam step (a11).
#include "sgad_device.cuh"
#include "sgad_launch.cuh"

namespace sgad {

// Zeroes all ranges of a list: one launch where one memset each (and its gap) cost about 2 us.
__global__ void __launch_bounds__(256) k_clear(const __grid_constant__ ClearList c)
{
    dependency_wait();
    const size_t first = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    for (int r = 0; r < c.n; ++r) {
        uint32_t *const p = c.at[r];
        const size_t n = c.words[r];
        const size_t vec = (reinterpret_cast<uintptr_t>(p) & 15) == 0 ? n / 4 : 0;
        for (size_t i = first; i < vec; i += step) reinterpret_cast<uint4 *>(p)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (size_t i = 4 * vec + first; i < n; i += step) p[i] = 0u;
    }
}

cudaError_t launch_clear(const ClearList &c, cudaStream_t st)
{
    size_t most = 0;
    for (int r = 0; r < c.n; ++r) most = most > c.words[r] ? most : c.words[r];
    if (!most) return cudaSuccess;
    const size_t blocks = (most + 1023) / 1024;
    return launch_after(k_clear, (unsigned)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, st, c);
}

__global__ void __launch_bounds__(256) k_finalize(const __grid_constant__ Scene sc, const float4 *__restrict__ gacc)
{
    dependency_wait(gacc);
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= sc.n_gauss) return;
    const KfDev &k = sc.kf[find_kf(sc, g)];
    if (!k.learnable) return;
    const uint32_t j = g - k.gbase;
    const size_t hw = (size_t)k.W * k.H;
    // (d |D + delta|, d s, d o, d r), (d g, d b)
    const float4 a = gacc[2 * (size_t)g];
    const float2 b = *reinterpret_cast<const float2 *>(&gacc[2 * (size_t)g + 1]);
    const float sum = k.depth[j] + k.offset[j];
    const float sgn = sum > 0.0f ? 1.0f : (sum < 0.0f ? -1.0f : 0.0f);
    // the opacity as the projection computed it (same expression: bit-identical), from the
    // 4-byte logit instead of the 32-byte world record
    const float o = 1.0f / (1.0f + expf(-k.logit[j]));
    k.d_offset[j] = sc.freeze_offset ? 0.0f : sgn * a.x;
    k.d_scale[j] = a.y;
    k.d_logit[j] = a.z * o * (1.0f - o);
    k.d_rgb[j] = a.w;
    k.d_rgb[hw + j] = b.x;
    k.d_rgb[2 * hw + j] = b.y;
}

void launch_finalize(const Scene &sc, const float4 *gacc, cudaStream_t st)
{
    const unsigned blocks = (sc.n_gauss + 255) / 256;
    if (blocks) launch_after(k_finalize, blocks, 256, 0, st, sc, gacc);
}

__device__ __forceinline__ float sgnf(float x) { return x > 0.0f ? 1.0f : (x < 0.0f ? -1.0f : 0.0f); }

__device__ __forceinline__ float block_sum(float x, float *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    __syncthreads();
    return t;
}

// All views of one loss call; every view owns a contiguous range of CTAs of `chunk` pixels:
// 4096, or 1024 (one access of four pixels per thread) when CTAs of 4096 would leave SMs
// without one: 2 views of 160x120 took 24 us on ten CTAs and take 5 on 38; one of 1200x680 (200
// of 4096) takes 10.0 us with depth and 5.8 without in the large chunk, 10.9 and 6.7 in the small.
// The CTAs of a cluster add their parts of the loss through distributed shared memory, one
// FP32 addition to the loss per cluster: an eighth (with the small chunk half) of the
// additions, and of their rounding and order dependence, that one per 4096 pixels made.
constexpr uint32_t kLossChunk = 4096, kLossChunkSmall = 1024;
constexpr int kLossCluster = 8;

struct LossView {
    const float *rgb, *depth, *alpha, *trgb, *tdep;   // alpha: null unless masking
    float *drgb, *ddep;
    uint32_t *nvalid;
    uint32_t hw;
    uint32_t block0;
    int32_t vec;                    // hw % 4 == 0 and every plane 16-byte aligned
};

struct LossBatch {
    int32_t n;
    uint32_t chunk;                 // pixels per CTA
    float wrgb, wdep, min_alpha;
    LossView v[SGAD_MAX_VIEWS];
};

__device__ __forceinline__ int loss_view(const LossBatch &B)
{
    int k = 0;
    for (int i = 1; i < B.n; ++i)
        if (B.v[i].block0 <= blockIdx.x) k = i;
    return k;
}

__global__ void __launch_bounds__(256) k_count_valid(const __grid_constant__ LossBatch B)
{
    dependency_wait();
    __shared__ float red[32];
    const LossView &v = B.v[loss_view(B)];
    const size_t base = (size_t)(blockIdx.x - v.block0) * B.chunk;
    const size_t end = base + B.chunk < v.hw ? base + B.chunk : v.hw;
    float c = 0.f;
    for (size_t i = base + threadIdx.x; i < end; i += blockDim.x) c += v.tdep[i] > 0.0f ? 1.0f : 0.0f;
    const float t = block_sum(c, red);
    if (threadIdx.x == 0 && t > 0.f) atomicAdd(v.nvalid, (uint32_t)t);
}

// ALL_VEC: every view's planes take 16-byte accesses (the other loop's registers would cost
// this one its occupancy: 34 us against 23 at 8 x 640x480).
template <bool ALL_VEC>
__global__ void __cluster_dims__(kLossCluster, 1, 1) __launch_bounds__(256)
    k_l1_grad(const __grid_constant__ LossBatch B, float *loss)
{
    cluster_begin();
    dependency_wait();
    __shared__ float red[32], part[kLossCluster];
    const LossView &v = B.v[loss_view(B)];
    const size_t hw = v.hw;
    // (a CTA past the last has no pixels: its base is past the end)
    const size_t base = (size_t)(blockIdx.x - v.block0) * B.chunk;
    const size_t end = base + B.chunk < hw ? base + B.chunk : hw;
    const float inv_rgb = B.wrgb / (3.0f * (float)hw);
    const uint32_t nv = v.nvalid ? *v.nvalid : 0u;
    const float inv_dep = nv > 0 ? B.wdep / (float)nv : 0.0f;
    float l = 0.f;
    if (ALL_VEC || v.vec) {          // four pixels per thread and access
        for (size_t i = base + 4 * threadIdx.x; i < end; i += 4 * blockDim.x) {
            const float4 al = v.alpha ? *reinterpret_cast<const float4 *>(v.alpha + i) : make_float4(1.f, 1.f, 1.f, 1.f);
            const bool keep[4] = {!v.alpha || al.x > B.min_alpha, !v.alpha || al.y > B.min_alpha,
                                  !v.alpha || al.z > B.min_alpha, !v.alpha || al.w > B.min_alpha};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float4 r = *reinterpret_cast<const float4 *>(v.rgb + c * hw + i);
                const float4 t = *reinterpret_cast<const float4 *>(v.trgb + c * hw + i);
                const float d[4] = {r.x - t.x, r.y - t.y, r.z - t.z, r.w - t.w};
                float gq[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (keep[q]) l += fabsf(d[q]) * inv_rgb;
                    gq[q] = keep[q] ? sgnf(d[q]) * inv_rgb : 0.0f;
                }
                *reinterpret_cast<float4 *>(v.drgb + c * hw + i) = make_float4(gq[0], gq[1], gq[2], gq[3]);
            }
            if (v.ddep) {
                float gd[4] = {0.f, 0.f, 0.f, 0.f};
                if (v.tdep && inv_dep > 0.0f) {
                    const float4 dp = *reinterpret_cast<const float4 *>(v.depth + i);
                    const float4 td = *reinterpret_cast<const float4 *>(v.tdep + i);
                    const float dv[4] = {dp.x, dp.y, dp.z, dp.w}, tv[4] = {td.x, td.y, td.z, td.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (keep[q] && tv[q] > 0.0f) {
                            const float d = dv[q] - tv[q];
                            l += fabsf(d) * inv_dep;
                            gd[q] = sgnf(d) * inv_dep;
                        }
                }
                *reinterpret_cast<float4 *>(v.ddep + i) = make_float4(gd[0], gd[1], gd[2], gd[3]);
            }
        }
    } else if constexpr (!ALL_VEC) {
        // four pixels, 256 apart, per pass; all loads before the stores, which the compiler may
        // not move loads across
        const bool use_depth = v.tdep && inv_dep > 0.0f;
        for (size_t i = base + threadIdx.x; i < end; i += 4 * 256) {
            float r[4][3], t[4][3], dp[4], td[4];
            bool keep[4];                    // silhouette mask
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t p = i + 256 * q;
                keep[q] = p < end && (!v.alpha || v.alpha[p] > B.min_alpha);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    r[q][c] = p < end ? v.rgb[c * hw + p] : 0.f;
                    t[q][c] = p < end ? v.trgb[c * hw + p] : 0.f;
                }
                dp[q] = use_depth && p < end ? v.depth[p] : 0.f;
                td[q] = use_depth && p < end ? v.tdep[p] : 0.f;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t p = i + 256 * q;
                if (p >= end) break;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float d = r[q][c] - t[q][c];
                    if (keep[q]) l += fabsf(d) * inv_rgb;
                    v.drgb[c * hw + p] = keep[q] ? sgnf(d) * inv_rgb : 0.0f;
                }
                if (v.ddep) {
                    float gd = 0.f;
                    if (use_depth && keep[q] && td[q] > 0.0f) {
                        const float d = dp[q] - td[q];
                        l += fabsf(d) * inv_dep;
                        gd = sgnf(d) * inv_dep;
                    }
                    v.ddep[p] = gd;
                }
            }
        }
    }
    if (loss) {
        const float t = block_sum(l, red);
        cluster_add(loss, t, part);
    }
}

// views: per view (rgb, depth, target rgb, target depth or NULL, d_rgb, d_depth or NULL,
// valid counter or NULL, pixel count).
void launch_l1_batch(int n, const float *const *rgb, const float *const *depth, const float *const *alpha,
                     const float *const *trgb, const float *const *tdep, float *const *drgb, float *const *ddep,
                     uint32_t *nvalid, const uint32_t *hw, float wrgb, float wdep, float min_alpha, float *loss,
                     cudaStream_t st)
{
    LossBatch B;
    B.n = n;
    B.wrgb = wrgb;
    B.wdep = wdep;
    B.min_alpha = min_alpha;
    uint32_t blocks = 0;
    size_t full = 0;
    for (int i = 0; i < n; ++i) full += (hw[i] + kLossChunk - 1) / kLossChunk;
    B.chunk = full < 152 ? kLossChunkSmall : kLossChunk;
    const bool use_depth = wdep != 0.0f && tdep && ddep && nvalid;
    for (int i = 0; i < n; ++i) {
        LossView &v = B.v[i];
        v.rgb = rgb[i];
        v.depth = depth ? depth[i] : nullptr;
        v.alpha = alpha ? alpha[i] : nullptr;
        v.trgb = trgb[i];
        v.tdep = use_depth ? tdep[i] : nullptr;
        v.drgb = drgb[i];
        v.ddep = ddep ? ddep[i] : nullptr;
        v.nvalid = use_depth ? nvalid + i : nullptr;
        v.hw = hw[i];
        uintptr_t al = reinterpret_cast<uintptr_t>(v.rgb) | reinterpret_cast<uintptr_t>(v.trgb) |
                       reinterpret_cast<uintptr_t>(v.drgb) | reinterpret_cast<uintptr_t>(v.alpha) |
                       reinterpret_cast<uintptr_t>(v.ddep);
        if (v.tdep) al |= reinterpret_cast<uintptr_t>(v.depth) | reinterpret_cast<uintptr_t>(v.tdep);
        v.vec = (hw[i] % 4 == 0 && (al & 15u) == 0) ? 1 : 0;
        v.block0 = blocks;
        blocks += (hw[i] + B.chunk - 1) / B.chunk;
    }
    if (use_depth) launch_after(k_count_valid, blocks, 256, 0, st, B);
    const unsigned grid = (blocks + kLossCluster - 1) / kLossCluster * kLossCluster;
    bool all_vec = true;
    for (int i = 0; i < n; ++i) all_vec = all_vec && B.v[i].vec != 0;
    if (all_vec)
        launch_after(k_l1_grad<true>, grid, 256, 0, st, B, loss);
    else
        launch_after(k_l1_grad<false>, grid, 256, 0, st, B, loss);
}

template <bool kLog>
__global__ void k_adam(int64_t n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2)
{
    dependency_wait(g);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float pi = p[i];
        const float gi = kLog ? g[i] * pi : g[i];     // d/d(log s) = s d/ds
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float step = lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = kLog ? expf(logf(pi) - step) : pi - step;
    }
}

// ---------------------------------------------------------- multi-tensor Adam

constexpr int kAdamChunk = 4096;    // elements per CTA

struct AdamDesc {
    float *p;
    const float *g;
    float *m, *v;
    int64_t n;
    float lr;
    int32_t mode;
    int32_t vec;                    // n % 4 == 0 and all four arrays 16-byte aligned
    int64_t block0;                 // first CTA of this tensor
};

struct AdamBatch {
    int32_t n;
    float b1, b2, eps;
    AdamDesc t[SGAD_ADAM_MAX_TENSORS];
};

// One Adam update of element (p, g, m, v) with the bias corrections' reciprocals.
__device__ __forceinline__ void adam_one(float &p, float g, float &m, float &v, float b1, float b2, float eps, float lr,
                                         float ic1, float ic2, bool log_mode)
{
    const float gi = log_mode ? g * p : g;
    m = b1 * m + (1.0f - b1) * gi;
    v = b2 * v + (1.0f - b2) * gi * gi;
    const float stp = lr * (m * ic1) / (sqrtf(v * ic2) + eps);
    p = log_mode ? p * expf(-stp) : p - stp;
}

__global__ void __launch_bounds__(256) k_adam_multi(const __grid_constant__ AdamBatch B, const int32_t *step)
{
    dependency_wait();
    int lo = 0, hi = B.n - 1;
    while (lo < hi) {                 // last tensor whose first CTA <= blockIdx.x
        const int mid = (lo + hi + 1) >> 1;
        if (B.t[mid].block0 <= (int64_t)blockIdx.x)
            lo = mid;
        else
            hi = mid - 1;
    }
    const AdamDesc &d = B.t[lo];
    const float s = (float)(*step + 1);
    const float ic1 = 1.0f / (1.0f - powf(B.b1, s)), ic2 = 1.0f / (1.0f - powf(B.b2, s));
    const bool log_mode = d.mode == SGAD_ADAM_LOG;
    const int64_t base = ((int64_t)blockIdx.x - d.block0) * kAdamChunk;
    const int64_t end = base + kAdamChunk < d.n ? base + kAdamChunk : d.n;
    if (d.vec) {                      // four elements per thread and access
        for (int64_t i = base + 4 * (int64_t)threadIdx.x; i < end; i += 4 * (int64_t)blockDim.x) {
            float4 p = *reinterpret_cast<const float4 *>(d.p + i);
            const float4 g = *reinterpret_cast<const float4 *>(d.g + i);
            float4 m = *reinterpret_cast<const float4 *>(d.m + i);
            float4 v = *reinterpret_cast<const float4 *>(d.v + i);
            adam_one(p.x, g.x, m.x, v.x, B.b1, B.b2, B.eps, d.lr, ic1, ic2, log_mode);
            adam_one(p.y, g.y, m.y, v.y, B.b1, B.b2, B.eps, d.lr, ic1, ic2, log_mode);
            adam_one(p.z, g.z, m.z, v.z, B.b1, B.b2, B.eps, d.lr, ic1, ic2, log_mode);
            adam_one(p.w, g.w, m.w, v.w, B.b1, B.b2, B.eps, d.lr, ic1, ic2, log_mode);
            *reinterpret_cast<float4 *>(d.m + i) = m;
            *reinterpret_cast<float4 *>(d.v + i) = v;
            *reinterpret_cast<float4 *>(d.p + i) = p;
        }
        return;
    }
    for (int64_t i = base + threadIdx.x; i < end; i += blockDim.x) {
        float p = d.p[i], m = d.m[i], v = d.v[i];
        adam_one(p, d.g[i], m, v, B.b1, B.b2, B.eps, d.lr, ic1, ic2, log_mode);
        d.m[i] = m;
        d.v[i] = v;
        d.p[i] = p;
    }
}

__global__ void k_increment(int32_t *c)
{
    dependency_wait();
    *c += 1;
}

cudaError_t launch_adam_multi(int n_t, const sgad_adam_tensor *t, float b1, float b2, float eps, int32_t *step,
                              cudaStream_t st)
{
    AdamBatch B;
    B.n = n_t;
    B.b1 = b1;
    B.b2 = b2;
    B.eps = eps;
    int64_t blocks = 0;
    for (int i = 0; i < n_t; ++i) {
        AdamDesc &d = B.t[i];
        d.p = t[i].param;
        d.g = t[i].grad;
        d.m = t[i].m;
        d.v = t[i].v;
        d.n = t[i].n;
        d.lr = t[i].lr;
        d.mode = t[i].mode;
        const uintptr_t al = reinterpret_cast<uintptr_t>(d.p) | reinterpret_cast<uintptr_t>(d.g) |
                             reinterpret_cast<uintptr_t>(d.m) | reinterpret_cast<uintptr_t>(d.v);
        d.vec = (d.n % 4 == 0 && (al & 15u) == 0) ? 1 : 0;
        d.block0 = blocks;
        blocks += (t[i].n + kAdamChunk - 1) / kAdamChunk;
    }
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    if (blocks > 0) launch_after(k_adam_multi, (unsigned)blocks, 256, 0, st, B, step);
    launch_after(k_increment, 1, 1, 0, st, step);
    return cudaGetLastError();
}

void launch_adam(int64_t n, float *p, const float *g, float *m, float *v, float lr, float b1, float b2, float eps,
                 float c1, float c2, bool log_mode, cudaStream_t st)
{
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (blocks <= 0) return;
    if (log_mode)
        launch_after(k_adam<true>, (unsigned)blocks, 256, 0, st, n, p, g, m, v, lr, b1, b2, eps, c1, c2);
    else
        launch_after(k_adam<false>, (unsigned)blocks, 256, 0, st, n, p, g, m, v, lr, b1, b2, eps, c1, c2);
}

// ------------------------------------------------- rendering-based camera initialisation
//
// One warp, an element or a power per lane: the FP64 chain on one thread (twelve powers, three
// 3x4 products) took 28 us, this 11.
// State layout (device floats): E [0, 12), M = W0^-1 E W0 [12, 24), Adam m [24, 30) and
// v [30, 36), step count [36], current pose E W0 [37, 49). 3x4 row-major [R | t].
struct PoseArgs {
    double W0[12];
    double lr[6];
    double b1, b2, eps;
};

// Element (r, c) of A B (as 4x4).
__device__ __forceinline__ double mat34_elem(const double *A, const double *B, int r, int c)
{
    double s = c == 3 ? A[4 * r + 3] : 0.0;
    for (int k = 0; k < 3; ++k) s += A[4 * r + k] * B[4 * k + c];
    return s;
}

__global__ void __launch_bounds__(32) k_pose_adam_step(const float *__restrict__ d_pose, float *__restrict__ st,
                                                       const PoseArgs a)
{
    dependency_wait(d_pose);
    __shared__ double G[12], E[12], M[9], xi[6], X[12], En[12], Wi[12], EW[12];
    const int lane = threadIdx.x;
    const double *W = a.W0;
    const float n0 = st[36];
    const double n = (double)n0 + 1.0;
    double m0 = 0.0, v0 = 0.0;
    if (lane < 6) {
        m0 = (double)st[24 + lane];
        v0 = (double)st[30 + lane];
    }
    const int r = lane >> 2, k = lane & 3;                 // element (r, k) of a 3x4 matrix
    if (lane < 12) {
        G[lane] = d_pose[lane];
        E[lane] = st[lane];
        // W0^-1 = [R0^T | -R0^T t0]
        Wi[lane] = k < 3 ? W[4 * k + r] : -(W[r] * W[3] + W[4 + r] * W[7] + W[8 + r] * W[11]);
    }
    __syncwarp();
    if (lane == 0) st[36] = (float)n;
    // one power per lane: b1^n and b2^n
    const double pw = lane < 2 ? pow(lane == 0 ? a.b1 : a.b2, n) : 0.0;
    const double c1 = 1.0 - __shfl_sync(0xffffffffu, pw, 0), c2 = 1.0 - __shfl_sync(0xffffffffu, pw, 1);
    // M = R0 G^T; d/d omega = vee(M - M^T) + t0 x c; d/d v = c
    if (lane < 9) {
        const int mr = lane / 3, mk = lane - 3 * mr;
        double s = 0.0;
        for (int q = 0; q < 3; ++q) s += W[4 * mr + q] * G[4 * mk + q];
        M[lane] = s;
    }
    __syncwarp();
    if (lane < 6) {
        const int i = lane, p = (i + 1) % 3, q = (i + 2) % 3;
        const double g = i < 3 ? M[3 * p + q] - M[3 * q + p] + (W[4 * p + 3] * G[4 * q + 3] - W[4 * q + 3] * G[4 * p + 3])
                               : G[4 * (i - 3) + 3];
        const double m = a.b1 * m0 + (1.0 - a.b1) * g;
        const double v = a.b2 * v0 + (1.0 - a.b2) * g * g;
        st[24 + i] = (float)m;
        st[30 + i] = (float)v;
        xi[i] = -a.lr[i] * (m / c1) / (sqrt(v / c2) + a.eps);
    }
    __syncwarp();
    // exp(xi) = [Rodrigues(omega) | v]
    const double th = sqrt(xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2]);
    double sn, cs;
    sincos(th, &sn, &cs);
    const double sa = th < 1e-12 ? 1.0 : sn / th, sb = th < 1e-12 ? 0.0 : (1.0 - cs) / (th * th);
    if (lane < 12) {
        const double K[9] = {0.0, -xi[2], xi[1], xi[2], 0.0, -xi[0], -xi[1], xi[0], 0.0};
        double kk = 0.0, k1 = 0.0;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            if (j / 3 != r || j % 3 != k) continue;
            k1 = K[j];
#pragma unroll
            for (int q = 0; q < 3; ++q) kk += K[3 * (j / 3) + q] * K[3 * q + j % 3];
        }
        X[lane] = k == 3 ? xi[3 + r] : (r == k ? 1.0 : 0.0) + sa * k1 + sb * kk;
    }
    __syncwarp();
    if (lane < 12) En[lane] = mat34_elem(X, E, r, k);
    __syncwarp();
    if (lane < 12) EW[lane] = mat34_elem(En, W, r, k);      // pose = E W0
    __syncwarp();
    if (lane < 12) {
        st[lane] = (float)En[lane];
        st[12 + lane] = (float)mat34_elem(Wi, EW, r, k);    // M = W0^-1 E W0
        st[37 + lane] = (float)EW[lane];
    }
}

cudaError_t launch_pose_adam_step(const float *d_pose, const float *W0, float *state, float lr_rot, float lr_trans,
                                  float b1, float b2, float eps, cudaStream_t st)
{
    PoseArgs a;
    for (int i = 0; i < 12; ++i) a.W0[i] = W0[i];
    for (int i = 0; i < 3; ++i) {
        a.lr[i] = lr_rot;
        a.lr[3 + i] = lr_trans;
    }
    a.b1 = b1;
    a.b2 = b2;
    a.eps = eps;
    launch_after(k_pose_adam_step, 1, 32, 0, st, d_pose, state, a);
    return cudaGetLastError();
}

}  // namespace sgad
