// distortion.cuh -- the distortion regulariser's forward kernel (Eq. S2), templated
// on the aggregation form: distortion.cu builds Eq. 8, distortion_agg.cu the other
// forms of Table 3 (whose reverse pass is the reverse march in distortion mode).
#pragma once
#include "records.cuh"

namespace ngprt {

struct DistParams {
    MarchParams m;
    float* dist_state;       // forward: [n][4] = (L_dist, W, S, 0) out; backward: in
    float scale;             // forward: loss += scale L_dist; backward: dL_total/dL_dist per ray
    float* loss;
    float* g_tables;
    float* g_coarse;
    const int2* list;        // backward: only these rays, from these samples on (NULL: all)
    const int32_t* n_list;
};

template <class Weights>
struct DistSampler {
    Weights fw;
    float W, S, Lp, Ls;
    __device__ __forceinline__ bool sample(const float u[3], float t, float delta) {
        const bool stop = fw.sample(u, t, delta);
        const float w = fw.w_last;
        const float m = fmaf(0.5f, delta, t);
        Lp = fmaf(2.0f * w, fmaf(m, W, -S), Lp);
        Ls = fmaf(w * w, delta * (1.0f / 3.0f), Ls);
        // rounded by itself, as in the reverse pass: that pass subtracts running sums from
        // these totals
        W = fadd(W, w);
        S = fmaf(w, m, S);
        return stop;
    }
};

template <bool kSnap, class Weights>
__device__ __forceinline__ void distortion_ray(const DistParams& p, const Weights& weights, int64_t tile = -1) {
    int64_t ray = 0;
    Ray ry;
    bool hit = false;
    const bool has_ray = ray_setup(p.m, ray, ry, hit, tile);
    float Ld = 0.0f;
    if (has_ray) {
        DistSampler<Weights> smp{weights, 0.0f, 0.0f, 0.0f, 0.0f};
        int n_march = 0, n_samp = 0;
        if (hit) march_loop<kSnap>(p.m, ry, smp, n_march, n_samp);
        Ld = smp.Lp + smp.Ls;
        reinterpret_cast<float4*>(p.dist_state)[ray] = make_float4(Ld, smp.W, smp.S, 0.0f);
    }
    if (p.loss) {
        __syncwarp();
        float v = Ld;
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
        if ((threadIdx.x & 31) == 0 && v != 0.0f) atomicAdd(p.loss, p.scale * v);
    }
}

// Blocks per SM where the compiler's own choice of registers is slow (0: its choice).  Shared
// gates of 16 levels: 3 (168 registers; with its 96 it spills, 16384 rays 667 us against
// 568).  Eq. 8 of up to 2 levels: 7 (72 registers; 2 levels, paper shape, 4096 free rays 605
// us, 842 as it comes, 750 at 8 blocks); of 8 levels: 5 (96 registers; 2^18 pixels 2261 us,
// 2521 as it comes).
template <int L, int AGG>
constexpr int distortion_blocks() {
    if (AGG == NGPRT_AGG_SHARED_V) return L == 16 ? 3 : 0;
    return AGG != NGPRT_AGG_SEPARATE_V ? 0 : L <= 2 ? 7 : L == 8 ? 5 : 0;
}

template <int L, int AGG>
__global__ void __launch_bounds__(128, distortion_blocks<L, AGG>())
    distortion_kernel(const __grid_constant__ DistParams p) {
    extern __shared__ float gate_smem[];
    using Weights = ForwardSampler<L, NGPRT_F32, AGG, kGatesUpFront>;
    distortion_ray<true>(p, Weights(p.m.g, p.m.opts.attn_mode, p.m.opts.t_term, gate_smem + threadIdx.x));
}

// The same from the density channel alone (p.m.plane), tiles handed out at run time.
template <int L>
__global__ void __launch_bounds__(128, kWeightMinBlocks) distortion_plane_kernel(const __grid_constant__ DistParams p) {
    for (int64_t tile; (tile = next_tile(p.m)) >= 0;) {
        distortion_ray<false>(p, WeightSampler<L>(p.m.g, p.m.plane, p.m.opts.attn_mode, p.m.opts.t_term), tile);
        __syncwarp();
    }
}

// The forms of Table 3 other than Eq. 8 (distortion_agg.cu): L = 2, 4, 16.
void launch_dist_fwd_agg(int L, int agg, const DistParams& p, dim3 grid, cudaStream_t st);
void launch_dist_bwd_agg(int L, int agg, const MarchBwdParams& p, dim3 grid, cudaStream_t st);

}  // namespace ngprt
