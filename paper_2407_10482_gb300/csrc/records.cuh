// records.cuh -- the reverse passes in two kernels: a march that writes one record per
// sample, and a scatter that sums the records of a ray before it touches the gradient
// grids.  For Eq. 8 scenes (SEPARATE_V): the render's reverse pass (kDist = false) and
// the distortion regulariser's (kDist = true, the density path alone).
//
// What bounds the one-kernel form (march_backward_kernel): every sample adds to 8 corner
// rows of 16 levels and of the coarse grid, 336 16-byte reductions, and the L2 takes
// about 180 G a second of them whether they hit or miss; reductions to the few hot rows
// of the coarse grid and the dense levels serialise on top, the more so the closer the
// rays of a warp are, so the march could not run in pixel-tile order, where its gathers
// cost half.
//
// Consecutive samples of a ray lie in the same cell of every level whose cells are wide
// against the step (hd: 39 steps to a cell at N = 16, 8.5 at 70, 1.2 at 512).  The colour
// channels of a level's gradient are one sum per corner times the ray's cotangents,
//     d entry[1..7] = (sum_i cw_i beta_i w_i) gq,   d entry[0] = sum_i cw_i omega_i gs_i,
// so a thread that walks a ray's records at one level needs 16 sums, and adds them to the
// 8 rows when the cell changes or the records end.
//
// Kernel 1 (record_kernel): warps take runs of 32 rays (large lists of camera pixels in
// pixel-tile order: the rays are binned by 32 x 32 pixel tile first) and march them together; each
// step of the warp is one slot of a chunk of kSlots steps x 32 lanes, taken from a
// counter when the previous chunk is full.  Record fields are lane-contiguous:
//     u (3), gs, w, then omega, beta, sigma^l, q^l per level   (kDist: u, gs, omega, sigma^l)
// Kernel 2 (scatter_levels_kernel, scatter_logits_kernel): one warp per (job, chunk), a
// job being a level, the coarse feature channels or a group of coarse logits; job-major,
// so that one level's gradient rows (16.7 MB for a hashed hd level) stay in L2 while all
// chunks add to them.
// Marches on a lattice (lattice_snap) keep the one-kernel forms.
// Rays whose records find no chunk left go to a list (with their first unrecorded
// sample) that the one-kernel form finishes.
//
// hd scene, 2^18 camera pixels of 8 views: march 3.3 ms (4 blocks per SM; 3.8 at 5, where
// it spills) + scatter 4.4 ms in place of 21.0 ms in one kernel.  The scatter was 7.0 ms
// with 8 steps a chunk and each lane adding its rows by itself, 6.4 with 16 steps, 4.8 with
// the lanes in pairs; levels and logits in kernels of their own, each with the blocks its
// registers allow, gave the rest.  The march is bound by the same 180 G sectors a second
// that its gathers take from L2.
//
// The regulariser takes records up to kDistRecordRays rays: 2^16 camera pixels of the hd
// scene, forward and reverse pass, 2.6 ms in place of 10.3; 8 levels 1.41 in place of 3.14.
// Beyond, its reverse pass stays in one kernel.  The gradients of a row are many small
// terms of both signs there, and what a float accumulator keeps of them depends on how
// they are grouped: at 2^18 rays the one-kernel form is 4e-5 of the coarse gradient away
// from sums in 64 bits and the run sums 3e-6, so that the two forms differ by up to 4e-5,
// more than FP32 results of one call are to move here; at 2^16 by 8e-6.  (2^18 rays took
// 6.5 ms by run sums in place of 36; 10.6 with the dense levels added sample by sample in
// the given ray order, which left 2.2e-5 on 8 levels.)
#pragma once
#include <string.h>

#include "backward_march.cuh"

namespace ngprt {

constexpr int kSlots = 16;      // steps per chunk
constexpr int kRunChunks = 8;   // chunks provided per run of 32 rays, at most
constexpr size_t kRecordBytes = (size_t)3 << 30;  // and of all runs, at most
constexpr int64_t kRecordRays = 1 << 18;   // rays per pass (records of more are processed in turn)
constexpr int64_t kRecordMinRays = 4096;   // fewer rays take the one-kernel form
// Render's records are taken in pixel-tile order from so many rays on.  Below, neighbours
// add to the same rows at the same time and wait for one another (us without records, in
// tile order and in the given order: 2 levels, 16384 random pixels 503, 806 and 555; 16
// levels, 32768 2890, 2122 and 1963); above, their gathers meet in L1 (16 levels, 2^17
// 10622, 4559 and 5301).  Tables of fewer than 2^16 rows, all of them hot whatever the
// order, from half as many on (bounded 4 levels of 2^12 rows, 50001 pixels on a full grid
// 1171, 956 and 1279).  The regulariser's records never are: 16 levels, 2^16 1892 and 1681;
// 2 levels, 16384 747 and 473, without records 516.
constexpr int64_t kBinRays = 1 << 16;
inline bool tile_order_pays(const MarchParams& m, int L) {
    return m.n_rays >= (((int64_t)m.g.T_mask + 1) * L < 1 << 16 ? kBinRays / 2 : kBinRays);
}
// Pixel lists of 2 and 4 levels take the one-kernel form up to so many rays: it adds whole
// rows of their coarse grid at a time, and its latency hides what records save (16384
// pixels: 2 levels 503 us against 555, 4 levels 603 against 669, bounded 488 against 523;
// 65536: 1266 against 863).
constexpr int64_t kFewLevelRays = 1 << 15;
//
// A coarse grid as fine as the steps (the paper shape's 512^3) leaves the coarse rows no run
// of samples to sum: there records start above 2^15 rays whatever their source, and with up
// to 2 levels they serve pixel lists above 2^17 alone (paper shape, ms without records and
// with: 4 levels, 16384 free rays 0.99 and 1.31, 65536 4.08 and 3.53; 2 levels, 2^18 free
// rays 9.0 and 10.7, pixels 6.2 and 5.7, 65536 pixels 2.05 and 2.41).
inline bool records_pay(int L, const MarchParams& m) {
    const float cell = (m.g.bounded ? 2.0f : 4.0f) / (float)(m.g.R_C - 1);
    const bool fine = cell < 4.0f * m.opts.step_base * m.opts.step_gamma;
    if (fine && L <= 2) return m.mode == 1 && m.n_rays > 4 * kFewLevelRays;
    return (!fine && (m.mode != 1 || (L != 2 && L != 4))) || m.n_rays > kFewLevelRays;
}
constexpr int64_t kDistRecordRays = 1 << 16;  // more rays of the regulariser take the one-kernel form
constexpr int kMaxBins = 1 << 16;

template <int L, bool kDist>
__host__ __device__ constexpr int record_floats() {
    return kDist ? 4 + 2 * L : 5 + 4 * L;
}
inline int record_floats_of(int L, bool dist) { return dist ? 4 + 2 * L : 5 + 4 * L; }

struct RecParams {
    MarchParams m;
    const int32_t* perm;      // ray order, or NULL (the given one)
    int64_t ray0, n_rays;     // the pass's range of that order
    const float* cot;         // render: cotangent records
    const float* dist_state;  // distortion: per ray (L_dist, W, S, 0)
    float dist_scale;
    float* g_tables;
    float* g_coarse;
    float* g_plane;           // distortion: the density channel's gradient, one float per row
    float* rec;               // [max_chunks][kSlots][fields][32]
    int32_t* chunk_ray;       // [max_chunks][32] ray of each lane
    int32_t* chunk_n;         // [max_chunks][32] records of each lane
    uint32_t max_chunks;
    uint32_t* n_chunks;       // chunks asked for (may pass max_chunks)
    unsigned long long* run_counter;
    int2* list;               // rays left to the one-kernel form: (ray, first sample)
    int32_t* n_list;
};

template <int L, bool kDist>
__global__ void __launch_bounds__(128, kDist ? 6 : 4) record_kernel(const __grid_constant__ RecParams p) {
    // levels whose gates are interpolated at a time: with 4, 50001 rays of 8 levels, forward
    // and reverse pass, take 4% less than one by one; 2^18 of 16 levels 12.65 and 12.58 ms
    constexpr int RG = L % 4 == 0 ? 4 : L % 2 == 0 ? 2 : 1;
    constexpr int F = record_floats<L, kDist>();
    const int lane = threadIdx.x & 31;
    const int64_t runs = (p.n_rays + 31) / 32;
    for (;;) {
        unsigned long long run = 0;
        if (lane == 0) run = atomicAdd(p.run_counter, 1ull);
        run = __shfl_sync(0xffffffffu, run, 0);
        if (run >= (unsigned long long)runs) break;
        const int64_t at = (int64_t)run * 32 + lane;
        bool live = at < p.n_rays;
        int32_t ray = 0;
        Ray ry;
        MarchState st;
        if (live) {
            ray = p.perm ? p.perm[p.ray0 + at] : (int32_t)(p.ray0 + at);
            live = ray_setup_at(p.m, ray, ry);
            if (live) st = march_state(ry);
        }
        // per-ray running sums: T; colour: the prefix of sum w q against the total;
        // distortion: W, S, G against their totals
        float T = 1.0f, s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, tot0 = 0.0f, tot1 = 0.0f, tot2 = 0.0f;
        float gq[7] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, gA = 0.0f, gD = 0.0f;
        if (live) {
            if constexpr (kDist) {
                const float4 ds = reinterpret_cast<const float4*>(p.dist_state)[ray];
                tot0 = ds.y;
                tot1 = ds.z;
                tot2 = 2.0f * ds.x;
            } else {
                const float4* c4 = reinterpret_cast<const float4*>(p.cot + (int64_t)ray * kCotFloats);
                const float4 q0 = c4[0], q1 = c4[1], q2 = c4[2];
                gq[0] = q0.x; gq[1] = q0.y; gq[2] = q0.z; gq[3] = q0.w;
                gq[4] = q1.x; gq[5] = q1.y; gq[6] = q1.z;
                gA = q1.w;
                gD = q2.x;
                tot0 = q2.y;
            }
        }
        uint32_t chunk = 0;
        int slot = kSlots;
        for (;;) {
            float u[3], delta, dt;
            if (live) live = march_advance<false>(p.m, ry, st, u, delta, dt);
            if (!__any_sync(0xffffffffu, live)) break;
            if (slot == kSlots) {
                uint32_t c = 0;
                if (lane == 0) c = atomicAdd(p.n_chunks, 1u);
                c = __shfl_sync(0xffffffffu, c, 0);
                if (c >= p.max_chunks) {
                    if (live) p.list[atomicAdd(p.n_list, 1)] = make_int2(ray, st.n_samp);
                    break;
                }
                chunk = c;
                slot = 0;
                p.chunk_ray[(size_t)chunk * 32 + lane] = ray;
                p.chunk_n[(size_t)chunk * 32 + lane] = 0;
            }
            if (live) {
                float* r = p.rec + ((size_t)chunk * kSlots + slot) * (F * 32) + lane;
                r[0] = u[0];
                r[32] = u[1];
                r[64] = u[2];
                float f[8];
                if constexpr (kDist) f[0] = sample_density<L, true>(p.m.g, p.m.plane, u, p.m.opts.attn_mode, r + 4 * 32);
                else sample_features<L, NGPRT_F32, NGPRT_AGG_SEPARATE_V, false, true, RG>(
                    p.m.g, u, p.m.opts.attn_mode, f, r + 5 * 32, 32, gq);
                const float t = df_float(st.t);
                const float sigma = expf(f[0]);
                const float trans = expf(-sigma * delta);
                const float w = fmul(T, fsub(1.0f, trans));
                const float T_next = T * trans;
                float gs;
                if constexpr (kDist) {
                    const float m = fmaf(0.5f, delta, t);
                    const float W_lt = s0, S_lt = s1;
                    s0 += w;
                    s1 = fmaf(w, m, s1);
                    const float gw = 2.0f * (fmaf(m, W_lt, -S_lt) + (tot1 - s1) - m * (tot0 - s0)) +
                                     (2.0f / 3.0f) * w * delta;
                    s2 = fmaf(w, gw, s2);
                    gs = p.dist_scale * (delta * (T_next * gw - (tot2 - s2))) * expf(fminf(f[0], 15.0f));
                } else {
                    float qg = fmaf(gD, t, gA);
#pragma unroll
                    for (int k = 0; k < 7; ++k) qg = fmaf(gq[k], f[1 + k], qg);
                    s0 = fmaf(w, qg, s0);
                    gs = delta * (T_next * qg - (tot0 - s0)) * expf(fminf(f[0], 15.0f));
                    r[4 * 32] = w;
                }
                r[3 * 32] = gs;
                p.chunk_n[(size_t)chunk * 32 + lane] = slot + 1;
                T = T_next;
                if (T < p.m.opts.t_term) live = false;
                else march_after_sample<false>(p.m, st, dt);
            }
            ++slot;
        }
        __syncwarp();
    }
}

// NV consecutive floats added at p (4-byte, 8-byte or 16-byte reductions by the row's
// alignment kAlign, in floats).
template <int NV, int kAlign>
__device__ __forceinline__ void add_row(float* p, const float* v) {
    if constexpr (kAlign % 4 == 0 && NV % 4 == 0) {
#pragma unroll
        for (int k = 0; k < NV; k += 4) atomic_add4(p + k, v[k], v[k + 1], v[k + 2], v[k + 3]);
    } else {
        static_assert(kAlign % 2 == 0 && NV % 2 == 0, "rows are pairs");
#pragma unroll
        for (int k = 0; k < NV; k += 2) atomicAdd(reinterpret_cast<float2*>(p + k), make_float2(v[k], v[k + 1]));
    }
}

// Adds the halves of 8-float rows with the two lanes of a pair side by side: a row is one
// sector, and the pair adds the two halves of one lane's row in the same instruction, then
// of the other's, so that L2 gets one request per row and not one per half.  row: this
// lane's (kNoRow: none); mine, theirs: the half (even lanes the first, odd lanes the
// second) of this lane's row and of its neighbour's.
constexpr uint32_t kNoRow = 0xFFFFFFFFu;
template <int kAlign>
__device__ __forceinline__ void add_pair(float* grid, uint32_t row, size_t row_floats, const float* mine,
                                         const float* theirs) {
    const bool odd = threadIdx.x & 1;
    const uint32_t other = __shfl_xor_sync(0xffffffffu, row, 1);
    float* half = grid + (odd ? 4 : 0);
    const uint32_t r1 = odd ? other : row, r2 = odd ? row : other;
    if (r1 != kNoRow) add_row<4, kAlign>(half + r1 * row_floats, odd ? theirs : mine);
    if (r2 != kNoRow) add_row<4, kAlign>(half + r2 * row_floats, odd ? mine : theirs);
}

__device__ __forceinline__ uint32_t vertex_row(const int b[3], int c, uint32_t N) {
    return (uint32_t)(b[0] + (c & 1)) + N * ((uint32_t)(b[1] + ((c >> 1) & 1)) + N * (uint32_t)(b[2] + ((c >> 2) & 1)));
}

// Scatter of the levels and of the coarse feature channels (job L: omega = beta = 1).  One
// warp per (job, chunk), a lane per ray.  The next record is loaded while the present one
// is added; 6 blocks per SM (2^18 pixels of the hd scene, forward and reverse pass: 12.62 ms
// against 12.66 at 7, 12.87 at 8 and 14.5 at 10, where it spills).
// kDist adds to a plane of the density gradient (hd: 25 MB, all of it in L2): the rows of
// two x neighbours are one 8-byte reduction there where they are an aligned pair (every
// hashed cell with an even x, and every other dense one).
template <int L, bool kDist>
__global__ void __launch_bounds__(128, kDist ? 8 : 6) scatter_levels_kernel(const __grid_constant__ RecParams p) {
    constexpr int F = record_floats<L, kDist>();
    constexpr int NC = kNFeat + 2 * L;
    constexpr int kLf = kDist ? 4 : 5, kPer = kDist ? 2 : 4;  // first level field, fields a level
    const Grid& g = p.m.g;
    const int lane = threadIdx.x & 31;
    const uint32_t n_chunks = min(*p.n_chunks, p.max_chunks);
    const uint64_t items = (uint64_t)(L + 1) * n_chunks;
    const uint64_t n_warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t it = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += n_warps) {
        const int job = (int)(it / n_chunks);
        const uint32_t chunk = (uint32_t)(it - (uint64_t)job * n_chunks);
        const int n = p.chunk_n[(size_t)chunk * 32 + lane];
        const int n_max = __reduce_max_sync(0xffffffffu, n);
        const float* rec = p.rec + (size_t)chunk * (kSlots * F * 32) + lane;
        const bool coarse = job == L;
        const int N = coarse ? g.R_C : g.N[job];
        float* const grid = coarse ? p.g_coarse : kDist ? p.g_plane : p.g_tables + (size_t)g.level_off[job] * 8;
        // cotangents of the row half that this lane adds (even lanes channels 0-3, odd
        // lanes 4-7): of its own ray and of its neighbour's
        float own[4] = {0.0f, 0.0f, 0.0f, 0.0f}, nbr[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if constexpr (!kDist) {
            const float* c = p.cot + (int64_t)p.chunk_ray[(size_t)chunk * 32 + lane] * kCotFloats;
            const float* cn = p.cot + (int64_t)p.chunk_ray[(size_t)chunk * 32 + (lane ^ 1)] * kCotFloats;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // floats 0-6 of the record are the cotangents of channels 1-7
                if (lane & 1) {
                    own[k] = c[3 + k];
                    nbr[k] = cn[3 + k];
                } else if (k > 0) {
                    own[k] = c[k - 1];
                    nbr[k] = cn[k - 1];
                }
            }
        }
        float sa[8], sb[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) sa[c] = sb[c] = 0.0f;
        int pb[3] = {-1, -1, -1};
        // adds the sums of the lanes with `go` to their 8 rows
        auto flush = [&](bool go) {
            if (!__any_sync(0xffffffffu, go)) return;
            auto row_of = [&](int c) {
                return coarse ? vertex_row(pb, c, (uint32_t)N)
                              : level_index(g, job, (uint32_t)(pb[0] + (c & 1)), (uint32_t)(pb[1] + ((c >> 1) & 1)),
                                            (uint32_t)(pb[2] + ((c >> 2) & 1)));
            };
            if constexpr (kDist) {
                if (!go) return;
#pragma unroll
                for (int c = 0; c < 8; c += 2) {
                    if (coarse) {
                        atomicAdd(grid + (size_t)row_of(c) * NC, sa[c]);
                        atomicAdd(grid + (size_t)row_of(c + 1) * NC, sa[c + 1]);
                        continue;
                    }
                    const uint32_t r0 = g.level_off[job] + row_of(c), r1 = g.level_off[job] + row_of(c + 1);
                    if ((r0 ^ r1) == 1u) {
                        const bool swap = r0 & 1u;
                        atomicAdd(reinterpret_cast<float2*>(grid + (r0 & ~1u)),
                                  make_float2(swap ? sa[c + 1] : sa[c], swap ? sa[c] : sa[c + 1]));
                    } else {
                        atomicAdd(grid + r0, sa[c]);
                        atomicAdd(grid + r1, sa[c + 1]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) sa[c] = 0.0f;
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint32_t row = go ? row_of(c) : kNoRow;
                    const float an = __shfl_xor_sync(0xffffffffu, sa[c], 1), bn = __shfl_xor_sync(0xffffffffu, sb[c], 1);
                    const bool odd = lane & 1;
                    const float v[4] = {odd ? sb[c] * own[0] : sa[c], sb[c] * own[1], sb[c] * own[2], sb[c] * own[3]};
                    const float vn[4] = {odd ? bn * nbr[0] : an, bn * nbr[1], bn * nbr[2], bn * nbr[3]};
                    if (coarse) add_pair<NC>(grid, row, NC, v, vn);
                    else add_pair<8>(grid, row, 8, v, vn);
                    if (go) sa[c] = sb[c] = 0.0f;
                }
            }
        };
        // u, gs and w times the level's omega and beta of record k
        float u[3] = {0.0f, 0.0f, 0.0f}, x[4] = {0.0f, 0.0f, 1.0f, 1.0f};
        auto load = [&](int k) {
            if (k >= n) return;
            const float* r = rec + k * (F * 32);
            u[0] = r[0];
            u[1] = r[32];
            u[2] = r[64];
            x[0] = r[96];
            if constexpr (!kDist) x[1] = r[128];
            if (!coarse) {
                x[2] = r[(kLf + kPer * job) * 32];
                if constexpr (!kDist) x[3] = r[(kLf + kPer * job + 1) * 32];
            }
        };
        load(0);
#pragma unroll 1
        for (int k = 0; k < n_max; ++k) {
            const bool on = k < n;
            int b[3];
            float w[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) grid_cell(u[d], N, b[d], w[d]);
            const float a = x[0] * x[2], bw = x[1] * x[3];
            load(k + 1);
            const bool moved = on && (b[0] != pb[0] || b[1] != pb[1] || b[2] != pb[2]);
            flush(moved && k > 0);
            if (on) {
                pb[0] = b[0]; pb[1] = b[1]; pb[2] = b[2];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float cw = corner_w(w, c);
                    sa[c] = fmaf(cw, a, sa[c]);
                    if constexpr (!kDist) sb[c] = fmaf(cw, bw, sb[c]);
                }
            }
        }
        flush(n > 0);
    }
}

// Scatter of the coarse logits, kGroup levels at a time: 8 channels' sums at 8 corners.
template <int L, bool kDist>
__global__ void __launch_bounds__(128, 4) scatter_logits_kernel(const __grid_constant__ RecParams p) {
    constexpr int F = record_floats<L, kDist>();
    constexpr int NC = kNFeat + 2 * L;
    constexpr int kGroup = kDist ? 8 : 4;
    constexpr int kLf = kDist ? 4 : 5, kPer = kDist ? 2 : 4;
    constexpr int NV = 8;
    const Grid& g = p.m.g;
    const int lane = threadIdx.x & 31, mode = p.m.opts.attn_mode, R = g.R_C;
    const uint32_t n_chunks = min(*p.n_chunks, p.max_chunks);
    const uint64_t items = (uint64_t)((L + kGroup - 1) / kGroup) * n_chunks;
    const uint64_t n_warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t it = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += n_warps) {
        const int l0 = (int)(it / n_chunks) * kGroup;
        const uint32_t chunk = (uint32_t)(it % n_chunks);
        const int n = p.chunk_n[(size_t)chunk * 32 + lane];
        const int n_max = __reduce_max_sync(0xffffffffu, n);
        const float* rec = p.rec + (size_t)chunk * (kSlots * F * 32) + lane;
        float* const grid = p.g_coarse + kNFeat + 2 * l0;
        float s[8][NV];
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int v = 0; v < NV; ++v) s[c][v] = 0.0f;
        int pb[3] = {-1, -1, -1};
        auto flush = [&](bool go) {
            if (!__any_sync(0xffffffffu, go)) return;
            const bool odd = lane & 1;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t row = go ? vertex_row(pb, c, (uint32_t)R) : kNoRow;
                if constexpr (!kDist && L % 4 == 0) {
                    float mine[4], theirs[4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        mine[v] = odd ? s[c][4 + v] : s[c][v];
                        theirs[v] = __shfl_xor_sync(0xffffffffu, odd ? s[c][v] : s[c][4 + v], 1);
                    }
                    add_pair<NC>(grid, row, NC, mine, theirs);
                } else if constexpr (kDist && L % 8 == 0) {
                    // the omega logits are every other channel; a zero added to the beta
                    // logit between two of them costs less than a second request
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float* q = s[c] + 4 * h;
                        const float mine[4] = {odd ? q[2] : q[0], 0.0f, odd ? q[3] : q[1], 0.0f};
                        const float theirs[4] = {__shfl_xor_sync(0xffffffffu, odd ? q[0] : q[2], 1), 0.0f,
                                                 __shfl_xor_sync(0xffffffffu, odd ? q[1] : q[3], 1), 0.0f};
                        add_pair<NC>(grid + 8 * h, row, NC, mine, theirs);
                    }
                } else if (go) {
                    float* gp = grid + (size_t)row * NC;
                    if constexpr (kDist) {
#pragma unroll
                        for (int v = 0; v < NV; ++v)
                            if (v < L && l0 + v < L) atomicAdd(gp + 2 * v, s[c][v]);
                    } else {
#pragma unroll
                        for (int v = 0; v < NV; v += 2)
                            if (v / 2 < L && l0 + v / 2 < L)
                                atomicAdd(reinterpret_cast<float2*>(gp + v), make_float2(s[c][v], s[c][v + 1]));
                    }
                }
                if (go) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) s[c][v] = 0.0f;
                }
            }
        };
#pragma unroll 1
        for (int k = 0; k < n_max; ++k) {
            const bool on = k < n;
            int b[3] = {pb[0], pb[1], pb[2]};
            float w[3] = {0.0f, 0.0f, 0.0f}, val[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) val[v] = 0.0f;
            if (on) {
                const float* r = rec + k * (F * 32);
                const float u[3] = {r[0], r[32], r[64]};
                const float gs = r[96];
                const float w_ = kDist ? 0.0f : r[128];
#pragma unroll
                for (int j = 0; j < kGroup; ++j) {
                    if (j >= L || l0 + j >= L) continue;
                    const float* q = r + (kLf + kPer * (l0 + j)) * 32;
                    if constexpr (kDist) {
                        const float om = q[0], sh = q[32];
                        val[j] = gs * sh * om * (1.0f - om);
                    } else {
                        const float om = q[0], be = q[32], sh = q[64], qd = q[96];
                        if (mode == 0) {
                            val[2 * j] = sh * gs * om * (1.0f - om);
                            val[2 * j + 1] = w_ * qd * be * (1.0f - be);
                        } else {
                            val[2 * j] = (sh * gs + w_ * qd) * om * (1.0f - om);
                        }
                    }
                }
#pragma unroll
                for (int d = 0; d < 3; ++d) grid_cell(u[d], R, b[d], w[d]);
            }
            const bool moved = b[0] != pb[0] || b[1] != pb[1] || b[2] != pb[2];
            flush(moved && k > 0);
            if (on) {
                pb[0] = b[0]; pb[1] = b[1]; pb[2] = b[2];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float cw = corner_w(w, c);
#pragma unroll
                    for (int v = 0; v < NV; ++v) s[c][v] = fmaf(cw, val[v], s[c][v]);
                }
            }
        }
        flush(n > 0);
    }
}

// ------------------------------------------------------- pixel-tile order of a ray list

struct BinParams {
    const int32_t* pixel_ids;
    int64_t n;
    int32_t n_cams, W, H, tile, tx, ty;
    uint32_t* bins;  // [n_cams ty tx] counts, then first positions
    int32_t* perm;
};

__device__ __forceinline__ uint32_t bin_of(const BinParams& p, int64_t i) {
    int64_t id = p.pixel_ids[i];
    if (id < 0) id = 0;
    const int64_t wh = (int64_t)p.W * p.H;
    int64_t view = id / wh;
    const int rem = (int)(id - view * wh);
    if (view >= p.n_cams) view = p.n_cams - 1;
    const int row = rem / p.W, col = rem - row * p.W;
    return ((uint32_t)view * p.ty + (uint32_t)(row / p.tile)) * p.tx + (uint32_t)(col / p.tile);
}

// Scratch of a records pass, laid out from a 256-byte aligned start.
struct RecLayout {
    size_t counters, perm, bins, list, chunk_ray, chunk_n, rec, bytes;
    uint32_t max_chunks;
    bool order;  // room for the pixel-tile order
};

inline RecLayout record_layout(int L, bool dist, int64_t n_rays) {
    RecLayout a;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const int64_t pass = n_rays < kRecordRays ? n_rays : kRecordRays;
    const size_t chunk_bytes = (size_t)kSlots * record_floats_of(L, dist) * 32 * sizeof(float);
    const int64_t want = (pass + 31) / 32 * kRunChunks, room = (int64_t)(kRecordBytes / chunk_bytes);
    a.max_chunks = (uint32_t)(want < room ? want : room);
    size_t at = 0;
    a.counters = at; at += 256;
    a.order = !dist && n_rays >= kBinRays / 2;
    a.perm = at; at += a.order ? up((size_t)n_rays * sizeof(int32_t)) : 0;
    a.bins = at; at += a.order ? up((size_t)kMaxBins * sizeof(uint32_t)) : 0;
    a.list = at; at += up((size_t)pass * sizeof(int2));
    a.chunk_ray = at; at += up((size_t)a.max_chunks * 32 * sizeof(int32_t));
    a.chunk_n = at; at += up((size_t)a.max_chunks * 32 * sizeof(int32_t));
    a.rec = at; at += (size_t)a.max_chunks * chunk_bytes;
    a.bytes = at + 256;  // slack to align the start
    return a;
}

// Scratch of the passes on the density channel: its plane, with `grad` a plane of its
// gradient, then the pixel-tile order of the rays (n_rays = 0: none).
struct PlaneLayout {
    size_t counter, plane, grad, bins, perm, bytes;
};

inline PlaneLayout plane_layout(int64_t entries, int64_t n_rays, bool grad = false) {
    PlaneLayout a;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    a.counter = 0;  // tiles handed out at run time
    a.plane = 256;
    a.grad = a.plane + up((size_t)entries * sizeof(float));
    a.bins = a.grad + (grad ? up((size_t)entries * sizeof(float)) : 0);
    const bool order = n_rays >= kRecordMinRays && n_rays <= 0x7FFFFFFF;
    a.perm = a.bins + (order ? (size_t)kMaxBins * sizeof(uint32_t) : 0);
    a.bytes = a.perm + (order ? up((size_t)n_rays * sizeof(int32_t)) : 0) + 256;
    return a;
}

// Fills the plane (backward.cu) and, with order, the rays' order and the tile counter into
// p; scratch of
// plane_layout(entries, order ? p.n_rays : 0).
void density_scratch(MarchParams& p, int64_t entries, bool order, void* scratch, cudaStream_t st);

// The gradient plane of plane_layout(entries, 0, true), zeroed; and its values added to
// channel 0 of the table gradient.
float* gradient_plane(int64_t entries, void* scratch, cudaStream_t st);
void add_gradient_plane(const float* plane, int64_t entries, float* g_tables, cudaStream_t st);

// The Eq. 8 scenes on FP32 tables with at least this many rows (a level stack that L1 and
// L2 hold whole gains nothing from a copy): the passes on the density channel take its
// plane.
constexpr int64_t kPlaneMinEntries = 1 << 18;
inline bool plane_serves(const ngprt_scene* s) {
    return s && s->aggregation == NGPRT_AGG_SEPARATE_V && s->table_dtype == NGPRT_F32 &&
           ngprt_table_entries(s) >= kPlaneMinEntries;
}

// Whether the plane's copy (hd, 6.1 M rows: 45 us; 42 M rows: 250 us) pays for a forward
// pass over rays: from 4096 rays on, and a ray for every 2000 rows, for shorter stacks, whose
// samples gain less, for every 700 (8 levels) or 140.  us without and with the plane,
// visibility pass: hd, 1 ray 97 and 152, 1000 random pixels 1072 and 1038, 4096 1323 and
// 889; 42 M rows, 1 ray 97 and 352, 6912 pixels of an image 1183 and 1332, 65536 1668 and
// 1399; 8 levels, 52 M rows, 32768 pixels 805 and 1089; 4 levels, 17 M rows, 16384 1005 and
// 1253, 2^18 3436 and 1724.  (Where every ray ends after some 14 samples the copy does not
// pay back at 4096 rays: 174 and 219.)  Up to 3 levels of 2^20 rows or more gain by the
// pixel-tile order alone (8 M rows, 2^18 pixels 2892 and 1378, free rays 3965 and 5053).
inline bool plane_pays(const ngprt_scene* s, int64_t n_rays) {
    if (!plane_serves(s)) return false;
    const int64_t rows = ngprt_table_entries(s);
    return n_rays >= kRecordMinRays && n_rays >= rows / (s->L <= 2 ? 67 : s->L <= 4 ? 140 : s->L <= 8 ? 700 : 2000);
}
inline bool plane_pays(const ngprt_scene* s, const MarchParams& m) {
    return plane_pays(s, m.n_rays) && (s->L > 3 || m.mode == 1 || ngprt_table_entries(s) < 1 << 20);
}

// The same for the regulariser's records, which take a second plane, of the gradient: us
// without and with, 4 levels, 17 M rows, 16384 free rays 1097 and 1401, 65536 5587 and 3457;
// 16 levels, 80 M rows, 4096 pixels 1777 and 1710, 16384 2338 and 2000.
inline bool plane_pays_records(const ngprt_scene* s, int64_t n_rays) {
    if (!plane_serves(s)) return false;
    const int64_t rows = ngprt_table_entries(s);
    return n_rays >= rows / (s->L <= 3 ? 200 : s->L <= 4 ? 400 : 16000);
}

// The same for a density at R^3 voxels: a voxel for every 32 rows, and enough work for
// another launch.  hd: 32^3 32 and 56 us, 64^3 122 and 81, 128^3 698 and 263; 42 M rows:
// 64^3 234 and 290, 128^3 1487 and 493; 2 levels: 64^3 17 and 19, 128^3 82 and 54.
inline bool plane_pays_voxels(const ngprt_scene* s, int32_t R) {
    const int64_t n = (int64_t)R * R * R;
    return plane_serves(s) && n >= ngprt_table_entries(s) / 32 && n * s->L > 1 << 20;
}

// Bytes that the records of a reverse pass take (0: the pass keeps none).
inline size_t record_scratch_bytes(int L, bool dist, int64_t n_rays) {
    if (n_rays < kRecordMinRays || n_rays > (dist ? kDistRecordRays : 0x7FFFFFFF)) return 0;
    return record_layout(L, dist, n_rays).bytes;
}

// The bins' kernels and launch (backward.cu): perm of the camera pixels in pixel-tile
// order, or NULL where the rays stay in the given order.
const int32_t* bin_rays(const MarchParams& m, uint32_t* bins, int32_t* perm, cudaStream_t st);

// Records and scatter of all rays of p.m; rest(p) finishes the rays of p.list.
template <int L, bool kDist, class Rest>
void launch_records(RecParams p, void* scratch, cudaStream_t st, Rest rest) {
    const int64_t n = p.m.n_rays;
    const RecLayout a = record_layout(L, kDist, n);
    char* base = reinterpret_cast<char*>(((uintptr_t)scratch + 255) & ~(uintptr_t)255);
    p.n_chunks = reinterpret_cast<uint32_t*>(base + a.counters);
    p.n_list = reinterpret_cast<int32_t*>(base + a.counters + 8);
    p.run_counter = reinterpret_cast<unsigned long long*>(base + a.counters + 16);
    p.list = reinterpret_cast<int2*>(base + a.list);
    p.chunk_ray = reinterpret_cast<int32_t*>(base + a.chunk_ray);
    p.chunk_n = reinterpret_cast<int32_t*>(base + a.chunk_n);
    p.rec = reinterpret_cast<float*>(base + a.rec);
    p.max_chunks = a.max_chunks;
    p.perm = nullptr;
    if (a.order && tile_order_pays(p.m, L))
        p.perm = bin_rays(p.m, reinterpret_cast<uint32_t*>(base + a.bins), reinterpret_cast<int32_t*>(base + a.perm), st);
    static int cache1[16] = {0}, cache2[16] = {0}, cache3[16] = {0};
    const unsigned g1 = resident_grid(record_kernel<L, kDist>, cache1),
                   g2 = resident_grid(scatter_levels_kernel<L, kDist>, cache2),
                   g3 = resident_grid(scatter_logits_kernel<L, kDist>, cache3);
    for (int64_t r0 = 0; r0 < n; r0 += kRecordRays) {
        p.ray0 = r0;
        p.n_rays = n - r0 < kRecordRays ? n - r0 : kRecordRays;
        cudaMemsetAsync(base + a.counters, 0, 256, st);
        const unsigned blocks = (unsigned)((p.n_rays + 127) / 128);
        record_kernel<L, kDist><<<blocks < g1 ? blocks : g1, 128, 0, st>>>(p);
        scatter_levels_kernel<L, kDist><<<g2, 128, 0, st>>>(p);
        if (p.m.opts.attn_mode != 1) scatter_logits_kernel<L, kDist><<<g3, 128, 0, st>>>(p);
        rest(p, blocks);
    }
}

}  // namespace ngprt
