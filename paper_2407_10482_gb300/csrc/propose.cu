// propose.cu -- learned per-ray proposal: a small MLP on (o / in_scale, d) that
// predicts the interval [t_near, t_far] holding the ray's significant weights and
// its opacity A^.  Not in the paper (Sec. 2 calls adaptive sampling orthogonal to
// NGP-RT); the renderer marches only inside the interval, and a fallback pass
// re-marches rays whose interval missed more than 1% of the predicted opacity.
//   h1 = relu(W0 e + b0), h2 = relu(W1 h1 + b1), z = W2 h2 + b2,
//   t_near = t_scale sigmoid(z0), t_far = t_scale sigmoid(z1), A^ = sigmoid(z2)
// Parameters, flat float: W0 [32][6], b0 [32], W1 [32][32], b1 [32], W2 [3][32], b2 [3].
#include <cooperative_groups.h>

#include "march.cuh"

namespace ngprt {
namespace {

constexpr int kPW = 32;
constexpr int kPIn = 6;
constexpr int kPParams = kPW * kPIn + kPW + kPW * kPW + kPW + 3 * kPW + 3;

struct PropParams {
    MarchParams m;  // ray source only
    const float* w;
    const __half* w16;  // propose with FP16 weights (widened to FP32 in shared memory)
    float in_scale, t_scale, margin_near, margin_far, a_min;
    float* interval;
    float* a_hat;
    const float* targets;
    float* g_w;
    float* loss;
};

__device__ __forceinline__ float psig(float x) { return 1.0f / (1.0f + expf(-x)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// e = (o / in_scale, d / |d|) of this thread's ray; false when the lane has none.
__device__ __forceinline__ bool prop_input(const PropParams& p, int64_t& ray, float e[kPIn], int64_t tile = -1) {
    float o[3], d[3];
    df dd[3];
    if (!thread_ray(p.m, ray, o, dd, tile)) return false;
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = df_float(dd[a]);
    const float n = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        e[a] = o[a] / p.in_scale;
        e[3 + a] = d[a] / n;
    }
    return true;
}

// Offsets of the layers in the flat parameters (all rows of W1 and W2 are 16-byte
// aligned, those of W0 8-byte).
constexpr int kOffB0 = kPW * kPIn, kOffW1 = kOffB0 + kPW, kOffB1 = kOffW1 + kPW * kPW, kOffW2 = kOffB1 + kPW,
              kOffB2 = kOffW2 + 3 * kPW;

// First layer of NR rays: a1 = W0 e + b0.
template <int NR>
__device__ __forceinline__ void prop_layer0(const float* w, const float (&e)[NR][kPIn], float (&a1)[NR][kPW]) {
#pragma unroll
    for (int o = 0; o < kPW; ++o) {
        const float2* row = reinterpret_cast<const float2*>(w + o * kPIn);
        const float2 w0 = row[0], w1 = row[1], w2 = row[2];
        const float b = w[kOffB0 + o];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            float a = fmaf(w0.x, e[r][0], b);
            a = fmaf(w0.y, e[r][1], a);
            a = fmaf(w1.x, e[r][2], a);
            a = fmaf(w1.y, e[r][3], a);
            a = fmaf(w2.x, e[r][4], a);
            a1[r][o] = fmaf(w2.y, e[r][5], a);
        }
    }
}

// Output o of the second layer for NR rays from the rectified first layer.
template <int NR>
__device__ __forceinline__ void prop_layer1(const float* w, int o, const float (&h1)[NR][kPW], float (&a2)[NR]) {
    const float4* row = reinterpret_cast<const float4*>(w + kOffW1 + o * kPW);
    const float b = w[kOffB1 + o];
#pragma unroll
    for (int r = 0; r < NR; ++r) a2[r] = b;
#pragma unroll
    for (int k = 0; k < kPW / 4; ++k) {
        const float4 q = row[k];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            a2[r] = fmaf(q.x, h1[r][4 * k], a2[r]);
            a2[r] = fmaf(q.y, h1[r][4 * k + 1], a2[r]);
            a2[r] = fmaf(q.z, h1[r][4 * k + 2], a2[r]);
            a2[r] = fmaf(q.w, h1[r][4 * k + 3], a2[r]);
        }
    }
}

// Two runs of 32 rays per warp: a broadcast 16-byte load of four weights from shared
// memory occupies its pipe for about two cycles, as long as the four multiply-adds it
// feeds for one ray, so each load serves two rays (FP32 sums in the order of the
// weights).  1920 x 1080 rays: 286 -> 150 us (one ray per thread, scalar loads
// before); the 1312 multiply-adds a ray take 68 us at the FP32 rate.
constexpr int kPropRays = 2;
__global__ void __launch_bounds__(128) propose_kernel(const __grid_constant__ PropParams p) {
    __shared__ __align__(16) float ws[kPParams];
    for (int i = threadIdx.x; i < kPParams; i += blockDim.x) ws[i] = p.w16 ? __half2float(p.w16[i]) : p.w[i];
    __syncthreads();
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t ray[kPropRays];
    bool has[kPropRays];
    float e[kPropRays][kPIn], h[kPropRays][kPW], z[kPropRays][3];
#pragma unroll
    for (int r = 0; r < kPropRays; ++r) {
        has[r] = prop_input(p, ray[r], e[r], kPropRays * warp + r);
        if (!has[r])
            for (int k = 0; k < kPIn; ++k) e[r][k] = 0.0f;
    }
    prop_layer0<kPropRays>(ws, e, h);
#pragma unroll
    for (int r = 0; r < kPropRays; ++r) {
#pragma unroll
        for (int o = 0; o < kPW; ++o) h[r][o] = fmaxf(h[r][o], 0.0f);
#pragma unroll
        for (int k = 0; k < 3; ++k) z[r][k] = ws[kOffB2 + k];
    }
#pragma unroll 4
    for (int o = 0; o < kPW; ++o) {
        float a2[kPropRays];
        prop_layer1<kPropRays>(ws, o, h, a2);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float w2 = ws[kOffW2 + k * kPW + o];
#pragma unroll
            for (int r = 0; r < kPropRays; ++r) z[r][k] = fmaf(w2, fmaxf(a2[r], 0.0f), z[r][k]);
        }
    }
#pragma unroll
    for (int r = 0; r < kPropRays; ++r) {
        if (!has[r]) continue;
        const float tn = p.t_scale * psig(z[r][0]), tf = p.t_scale * psig(z[r][1]), ah = psig(z[r][2]);
        float lo, hi;
        if (ah < p.a_min) {
            lo = INFINITY;   // predicted empty: march nothing
            hi = -INFINITY;
        } else if (!(tf > tn)) {
            lo = -INFINITY;  // no usable interval: march the whole ray
            hi = INFINITY;
        } else {
            lo = tn - p.margin_near;
            hi = tf + p.margin_far;  // +inf: no far clip (termination ends the ray)
        }
        p.interval[2 * ray[r]] = lo;
        p.interval[2 * ray[r] + 1] = hi;
        if (p.a_hat) p.a_hat[ray[r]] = ah;
    }
}

__device__ __forceinline__ float sl1_grad(float x, float beta) {
    const float ax = fabsf(x);
    return ax < beta ? x / beta : (x > 0.0f ? 1.0f : -1.0f);
}

__device__ __forceinline__ float sl1(float x, float beta) {
    const float ax = fabsf(x);
    return ax < beta ? 0.5f * x * x / beta : ax - 0.5f * beta;
}

// Shared memory of the reverse pass: the weights, then channel by channel over the
// tile's rays (rows of kRS floats: 16-byte aligned, and rows of neighbouring channels
// fall on different banks) e (6), h1, h2, the gradients of both hidden layers'
// pre-activations and of the three outputs.
constexpr int kTileRays = 64, kBwdThreads = 256, kBwdCluster = 8;
constexpr int kRS = kTileRays + 4;
constexpr int kPWs = (kPParams + 3) / 4 * 4;
constexpr int kPropBwdSmem = (int)sizeof(float) * (kPWs + (kPIn + 4 * kPW + 3) * kRS);
static_assert(kPropBwdSmem <= 48 * 1024, "within the default limit");

// Loss and gradient, mean over n rays.  A block takes 64 rays and runs each layer as a
// small matrix product from shared memory, 4 rays x 2 channels per thread (2 x 2 outputs
// of the W1 gradient over the tile's rays); the eight blocks of a cluster add their
// weight sums up before they go to g_w.  2^15 rays, each step measured: a shuffle
// reduction per weight and warp with a shared atomic each 226 us; one ray per thread, which
// leaves fewer than two warps a scheduler to wait on shared memory, 50 us; four threads
// per ray 47 us; 512 blocks' atomics on the same 1379 addresses cut to 64 by the clusters
// 32 us; 16-byte loads in place of 4-byte ones 29 us.
__global__ void __cluster_dims__(kBwdCluster, 1, 1) __launch_bounds__(kBwdThreads)
    propose_backward_kernel(const __grid_constant__ PropParams p) {
    extern __shared__ __align__(16) float sm[];
    float* ws = sm;
    float* E = ws + kPWs;
    float* H1 = E + kPIn * kRS;
    float* H2 = H1 + kPW * kRS;
    float* G1 = H2 + kPW * kRS;
    float* G2 = G1 + kPW * kRS;
    float* GZ = G2 + kPW * kRS;  // the outputs z first, then their gradients
    auto at4 = [](float* m, int row, int col) { return reinterpret_cast<float4*>(m + row * kRS + col); };
    const int t = threadIdx.x;
    for (int i = t; i < kPParams; i += kBwdThreads) ws[i] = __ldg(p.w + i);
    int64_t ray = 0;
    bool active = false;
    if (t < kTileRays) {
        float e[kPIn];
        active = prop_input(p, ray, e, (int64_t)blockIdx.x * (kTileRays / 32) + (t >> 5));
#pragma unroll
        for (int k = 0; k < kPIn; ++k) E[k * kRS + t] = active ? e[k] : 0.0f;
    }
    __syncthreads();
    // this thread's rays r0 .. r0 + 3 and channels c0, c0 + 1 of the hidden layers
    const int r0 = (t & 15) * 4, c0 = (t >> 4) * 2;
    float4 acc[2];
    auto fma4 = [](float w, const float4& x, float4& a) {
        a.x = fmaf(w, x.x, a.x);
        a.y = fmaf(w, x.y, a.y);
        a.z = fmaf(w, x.z, a.z);
        a.w = fmaf(w, x.w, a.w);
    };
    auto relu4 = [](const float4& a) {
        return make_float4(fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f), fmaxf(a.z, 0.0f), fmaxf(a.w, 0.0f));
    };
    auto where4 = [](const float4& h, const float4& a) {
        return make_float4(h.x > 0.0f ? a.x : 0.0f, h.y > 0.0f ? a.y : 0.0f, h.z > 0.0f ? a.z : 0.0f,
                           h.w > 0.0f ? a.w : 0.0f);
    };
    auto all4 = [](float v) { return make_float4(v, v, v, v); };
    // h1 = relu(W0 e + b0)
    acc[0] = all4(ws[kOffB0 + c0]);
    acc[1] = all4(ws[kOffB0 + c0 + 1]);
#pragma unroll
    for (int k = 0; k < kPIn; ++k) {
        const float4 x = *at4(E, k, r0);
        fma4(ws[c0 * kPIn + k], x, acc[0]);
        fma4(ws[(c0 + 1) * kPIn + k], x, acc[1]);
    }
    *at4(H1, c0, r0) = relu4(acc[0]);
    *at4(H1, c0 + 1, r0) = relu4(acc[1]);
    __syncthreads();
    // h2 = relu(W1 h1 + b1)
    acc[0] = all4(ws[kOffB1 + c0]);
    acc[1] = all4(ws[kOffB1 + c0 + 1]);
#pragma unroll 4
    for (int k = 0; k < kPW; k += 4) {
        const float4 q0 = *reinterpret_cast<const float4*>(ws + kOffW1 + c0 * kPW + k);
        const float4 q1 = *reinterpret_cast<const float4*>(ws + kOffW1 + (c0 + 1) * kPW + k);
        const float w0[4] = {q0.x, q0.y, q0.z, q0.w}, w1[4] = {q1.x, q1.y, q1.z, q1.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 x = *at4(H1, k + j, r0);
            fma4(w0[j], x, acc[0]);
            fma4(w1[j], x, acc[1]);
        }
    }
    *at4(H2, c0, r0) = relu4(acc[0]);
    *at4(H2, c0 + 1, r0) = relu4(acc[1]);
    __syncthreads();
    // z = W2 h2 + b2: one output of one ray per thread
    if (t < 3 * kTileRays) {
        const int r = t & (kTileRays - 1), k = t / kTileRays;
        float z = ws[kOffB2 + k];
#pragma unroll 8
        for (int o = 0; o < kPW; ++o) z = fmaf(ws[kOffW2 + k * kPW + o], H2[o * kRS + r], z);
        GZ[k * kRS + r] = z;
    }
    __syncthreads();
    if (t < kTileRays) {
        const float inv_n = 1.0f / (float)p.m.n_rays;
        const float beta = 0.01f;
        float gz[3] = {0.0f, 0.0f, 0.0f}, L = 0.0f;
        if (active) {
            const float t0 = p.targets[3 * ray], t1 = p.targets[3 * ray + 1], A = p.targets[3 * ray + 2];
            const float s0 = psig(GZ[t]), s1 = psig(GZ[kRS + t]), s2 = psig(GZ[2 * kRS + t]);
            const float x0 = (p.t_scale * s0 - t0) / p.t_scale, x1 = (p.t_scale * s1 - t1) / p.t_scale;
            // conservative intervals: a late t_near or an early t_far costs 4x
            const float a0 = x0 > 0.0f ? 4.0f : 1.0f, a1 = x1 < 0.0f ? 4.0f : 1.0f;
            L = inv_n * (A * (a0 * sl1(x0, beta) + a1 * sl1(x1, beta)) + (s2 - A) * (s2 - A));
            gz[0] = inv_n * A * a0 * sl1_grad(x0, beta) * s0 * (1.0f - s0);
            gz[1] = inv_n * A * a1 * sl1_grad(x1, beta) * s1 * (1.0f - s1);
            gz[2] = inv_n * 2.0f * (s2 - A) * s2 * (1.0f - s2);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) GZ[k * kRS + t] = gz[k];
        const float ls = warp_sum(L);
        if ((t & 31) == 0 && p.loss) atomicAdd(p.loss, ls);
    }
    __syncthreads();
    // g2 = (W2^T gz) where h2 > 0
    acc[0] = acc[1] = all4(0.0f);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float4 g = *at4(GZ, k, r0);
        fma4(ws[kOffW2 + k * kPW + c0], g, acc[0]);
        fma4(ws[kOffW2 + k * kPW + c0 + 1], g, acc[1]);
    }
    *at4(G2, c0, r0) = where4(*at4(H2, c0, r0), acc[0]);
    *at4(G2, c0 + 1, r0) = where4(*at4(H2, c0 + 1, r0), acc[1]);
    __syncthreads();
    // g1 = (W1^T g2) where h1 > 0
    acc[0] = acc[1] = all4(0.0f);
#pragma unroll 8
    for (int o = 0; o < kPW; ++o) {
        const float2 w = *reinterpret_cast<const float2*>(ws + kOffW1 + o * kPW + c0);
        const float4 g = *at4(G2, o, r0);
        fma4(w.x, g, acc[0]);
        fma4(w.y, g, acc[1]);
    }
    *at4(G1, c0, r0) = where4(*at4(H1, c0, r0), acc[0]);
    *at4(G1, c0 + 1, r0) = where4(*at4(H1, c0 + 1, r0), acc[1]);
    __syncthreads();
    // the weights have been read for the last time: the block's sums take their place
    auto dot4 = [](const float4& a, const float4& b, float s) {
        return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
    };
    // W1: outputs (o, o + 16) x (k, k + 16)
    {
        const int o = t >> 4, k = t & 15;
        float s[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll 4
        for (int r = 0; r < kTileRays; r += 4) {
            const float4 g0 = *at4(G2, o, r), g1 = *at4(G2, o + 16, r);
            const float4 h0 = *at4(H1, k, r), h1 = *at4(H1, k + 16, r);
            s[0][0] = dot4(g0, h0, s[0][0]);
            s[0][1] = dot4(g0, h1, s[0][1]);
            s[1][0] = dot4(g1, h0, s[1][0]);
            s[1][1] = dot4(g1, h1, s[1][1]);
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) ws[kOffW1 + (o + 16 * a) * kPW + k + 16 * b] = s[a][b];
    }
    // W0, b0 and b1, W2 and b2: one or two outputs a thread
    {
        const int o = t & 31, k = t >> 5;  // k < 6: W0[o][k]; 6: b0; 7: b1
        float s = 0.0f;
#pragma unroll 4
        for (int r = 0; r < kTileRays; r += 4) {
            const float4 x = k < kPIn ? *at4(E, k, r) : all4(1.0f);
            s = dot4(*at4(k == 7 ? G2 : G1, o, r), x, s);
        }
        ws[k < kPIn ? o * kPIn + k : (k == 6 ? kOffB0 : kOffB1) + o] = s;
        if (k < 3 || (k == 3 && o < 3)) {  // W2[k][o]; then b2[o]
            float s2 = 0.0f;
#pragma unroll 4
            for (int r = 0; r < kTileRays; r += 4)
                s2 = dot4(*at4(GZ, k < 3 ? k : o, r), k < 3 ? *at4(H2, o, r) : all4(1.0f), s2);
            ws[k < 3 ? kOffW2 + k * kPW + o : kOffB2 + o] = s2;
        }
    }
    // the cluster's sums: each block adds up an eighth of the weights over the blocks'
    // shared memory, and adds them to g_w
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    const int part = (kPParams + kBwdCluster - 1) / kBwdCluster, first = (int)cluster.block_rank() * part;
    for (int i = first + t; i < min(first + part, kPParams); i += kBwdThreads) {
        float s = 0.0f;
#pragma unroll
        for (int b = 0; b < kBwdCluster; ++b) s += cluster.map_shared_rank(ws, b)[i];
        if (s != 0.0f) atomicAdd(p.g_w + i, s);
    }
    cluster.sync();  // no block leaves while its sums are read
}

// Blocks of `threads` threads for the runs of 32 rays (camera tiles) that setup_rays laid
// out as 4 per 128-thread block, `per_warp` runs to a warp.
unsigned prop_blocks(const MarchParams& m, int threads, int per_warp) {
    const int64_t runs = m.mode == 0 ? (int64_t)m.tiles_per_view * m.n_cams : (m.n_rays + 31) / 32;
    const int64_t per_block = (int64_t)(threads / 32) * per_warp;
    return (unsigned)((runs + per_block - 1) / per_block);
}

}  // namespace

int32_t setup_rays(MarchParams& p, const ngprt_camera* cams, int32_t n_cams, const int32_t* pixel_ids,
                   const float* rays_o, const float* rays_d, int64_t n_rays, dim3& grid, const char* fn);

}  // namespace ngprt

using namespace ngprt;

extern "C" int32_t ngprt_proposal_param_count(void) { return kPParams; }

extern "C" int32_t ngprt_propose(const void* prop_w, int32_t prop_dtype, const ngprt_camera* cams, int32_t n_cams,
                                 const int32_t* pixel_ids, const float* rays_o, const float* rays_d, int64_t n_rays,
                                 float in_scale, float t_scale, float margin_near, float margin_far, float a_min,
                                 float* t_interval_out, float* a_hat_out, void* stream) {
    const char* fn = "ngprt_propose";
    PropParams p;
    memset(&p, 0, sizeof p);
    NGPRT_REQUIRE(prop_w != nullptr, "%s: prop_w is NULL", fn);
    NGPRT_REQUIRE(prop_dtype == NGPRT_F32 || prop_dtype == NGPRT_F16, "%s: prop_dtype=%d (F32 or F16)", fn,
                  prop_dtype);
    NGPRT_REQUIRE(n_rays >= 0 && in_scale > 0.0f && t_scale > 0.0f && margin_near >= 0.0f && margin_far >= 0.0f,
                  "%s: bad scalar argument", fn);
    dim3 grid;
    int32_t rc;
    if ((rc = setup_rays(p.m, cams, n_cams, pixel_ids, rays_o, rays_d, n_rays, grid, fn)) != NGPRT_OK) return rc;
    if (n_rays == 0) return NGPRT_OK;
    NGPRT_REQUIRE(t_interval_out != nullptr, "%s: t_interval_out is NULL", fn);
    p.w = prop_dtype == NGPRT_F32 ? static_cast<const float*>(prop_w) : nullptr;
    p.w16 = prop_dtype == NGPRT_F16 ? static_cast<const __half*>(prop_w) : nullptr;
    p.in_scale = in_scale;
    p.t_scale = t_scale;
    p.margin_near = margin_near;
    p.margin_far = margin_far;
    p.a_min = a_min;
    p.interval = t_interval_out;
    p.a_hat = a_hat_out;
    propose_kernel<<<prop_blocks(p.m, 128, kPropRays), 128, 0, static_cast<cudaStream_t>(stream)>>>(p);
    return cuda_status(fn);
}

extern "C" int32_t ngprt_propose_backward(const float* prop_w, const ngprt_camera* cams, int32_t n_cams,
                                          const int32_t* pixel_ids, const float* rays_o, const float* rays_d,
                                          int64_t n_rays, float in_scale, float t_scale, const float* targets,
                                          float* g_prop_w, float* loss, void* stream) {
    const char* fn = "ngprt_propose_backward";
    PropParams p;
    memset(&p, 0, sizeof p);
    NGPRT_REQUIRE(prop_w != nullptr && g_prop_w != nullptr, "%s: NULL weights or gradient", fn);
    NGPRT_REQUIRE(n_rays >= 0 && in_scale > 0.0f && t_scale > 0.0f, "%s: bad scalar argument", fn);
    dim3 grid;
    int32_t rc;
    if ((rc = setup_rays(p.m, cams, n_cams, pixel_ids, rays_o, rays_d, n_rays, grid, fn)) != NGPRT_OK) return rc;
    if (n_rays == 0) return NGPRT_OK;
    NGPRT_REQUIRE(targets != nullptr, "%s: targets is NULL", fn);
    p.w = prop_w;
    p.in_scale = in_scale;
    p.t_scale = t_scale;
    p.targets = targets;
    p.g_w = g_prop_w;
    p.loss = loss;
    const unsigned blocks = (prop_blocks(p.m, kTileRays, 1) + kBwdCluster - 1) / kBwdCluster * kBwdCluster;
    propose_backward_kernel<<<blocks, kBwdThreads, kPropBwdSmem,
                              static_cast<cudaStream_t>(stream)>>>(p);
    return cuda_status(fn);
}
