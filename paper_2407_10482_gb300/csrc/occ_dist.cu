// occ_dist.cu -- occupancy pyramid and occupancy distance grid G (Sec. 3.3, Eq. 9;
// Sec. S2.5).  Integer work, bit-exact.
//
// G(p) = min(255, floor(sqrt(D2(p)))), D2(p) = min over occupied q of
// sum_a max(|p_a - q_a| - 1, 0)^2: the squared distance between voxel boxes.
// The sum is separable, so D2 is three exact 1-D minimisations.  G saturates at 255, so
// every partial sum may saturate at 255^2 (which already gives G = 255) and fits 16 bits:
// the x gaps come straight from the bits of a row, the y pass runs on their squares in
// shared memory, and one 16-bit grid goes to the z pass.
//
// The y and z passes minimise f(q) + gap(i, q)^2 along a line.  With E(j) = min_q f(q) +
// (j - q)^2 the box gap's minimum is min(E(i - 1), E(i), E(i + 1)): a q below i has its
// gap i - 1 - q in E(i - 1), one above in E(i + 1), and no term of the three is below its
// box gap's.  E's leftmost minimiser does not decrease with j, so after 4 seeds searched
// over the whole line each round of midpoints searches only between its neighbours'
// minimisers: about 4 R + R log2(R / 4) steps a line of R in place of R^2 (R = 256: 12 a
// voxel).  An outward search that stopped when the gap alone passed the best sum was no
// faster than R^2 steps where voxels are far from anything (512^3 grid, G at 256^3: 1.8 and
// 1.0 ms for the two passes; these take 0.19 and 0.16, bound by instruction issue).
#include <algorithm>

#include "common.cuh"

namespace ngprt {
namespace {

// Level 0 of the pyramid: one thread packs 32 consecutive voxels into a word, from two
// 16-byte loads where the grid allows it (kWide: occ 16-byte aligned, whole words).
// 512^3: 23 us, 112 with byte loads.
template <bool kWide>
__global__ void pack_bits_kernel(const uint8_t* __restrict__ occ, size_t n_vox, uint32_t* __restrict__ bits,
                                 size_t n_words) {
    size_t w = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n_words) return;
    uint32_t v = 0;
    if constexpr (kWide) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(occ) + 2 * w + h);
            const uint32_t x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // 0/1 per byte, then the four bytes' bits side by side in the top byte
                const uint32_t t = __vsetgtu4(x[k], 0u);
                v |= (((t * 0x01020408u) >> 24) & 0xFu) << (16 * h + 4 * k);
            }
        }
    } else {
        for (int b = 0; b < 32; ++b) {
            size_t i = w * 32 + b;
            if (i < n_vox && occ[i]) v |= 1u << b;
        }
    }
    bits[w] = v;
}

// The even bits of x, packed into its lower half.
__device__ __forceinline__ uint32_t even_bits(uint32_t x) {
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0x0000FFFFu;
}

// Word w of level k+1 (rc >= 32 per axis) from level k: OR of the 2 x 2 fine rows of two
// neighbouring words, their bit pairs folded.
__device__ __forceinline__ uint32_t coarse_word(const uint32_t* fine, int rc, size_t w) {
    const int rf = 2 * rc;
    const int wpr = rc >> 5;  // coarse words per row; fine rows have twice as many
    const int wx = (int)(w % wpr);
    const size_t row = w / wpr;
    const size_t y = row % rc, z = row / rc;
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t* f = fine + ((2 * y + (c & 1)) + (size_t)rf * (2 * z + (c >> 1))) * (2 * wpr) + 2 * wx;
        lo |= f[0];
        hi |= f[1];
    }
    return even_bits(lo | (lo >> 1)) | (even_bits(hi | (hi >> 1)) << 16);
}

__global__ void downsample_kernel(const uint32_t* __restrict__ fine, uint32_t* __restrict__ coarse, int rc,
                                  size_t n_words) {
    const size_t w = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w < n_words) coarse[w] = coarse_word(fine, rc, w);
}

// The rest of the pyramid, from a level of rf <= kTailRes per axis down to n_left more
// levels, in one block: each level is a few thousand words at most and a launch of its
// own would cost more than its work.
constexpr int kTailRes = 64;
__global__ void __launch_bounds__(1024) downsample_tail_kernel(uint32_t* fine, int rf, int n_left) {
    for (int k = 0; k < n_left; ++k) {
        const int rc = rf >> 1;
        const size_t wf = ((size_t)rf * rf * rf + 31) / 32, wc = ((size_t)rc * rc * rc + 31) / 32;
        uint32_t* coarse = fine + wf;
        if (rc >= 32) {
            for (size_t w = threadIdx.x; w < wc; w += blockDim.x) coarse[w] = coarse_word(fine, rc, w);
        } else {
            // one voxel per thread, a warp's votes make the word
            const int n_vox = rc * rc * rc;
            for (int i = threadIdx.x; i < (int)wc * 32; i += blockDim.x) {
                uint32_t any = 0;
                if (i < n_vox) {
                    const int x = i % rc, y = (i / rc) % rc, z = i / (rc * rc);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int fi = 2 * x + rf * ((2 * y + (c & 1)) + rf * (2 * z + (c >> 1)));
                        any |= (fine[fi >> 5] >> (fi & 31)) & 3u;
                    }
                }
                const uint32_t word = __ballot_sync(0xffffffffu, any != 0);
                if ((threadIdx.x & 31) == 0) coarse[i >> 5] = word;
            }
        }
        __syncthreads();  // the block's writes are visible to it after the barrier
        fine = coarse;
        rf = rc;
    }
}

// x gap of voxel x in its row of R bits (min(255, distance to the nearest set bit - 1),
// 0 on a set bit and its neighbours; 255 without one).
__device__ __forceinline__ int row_gap(const uint32_t* __restrict__ bits, size_t row_bit0, int R, int x) {
    int best = 256;  // distance, saturated
    if (R >= 32) {
        const uint32_t* row = bits + (row_bit0 >> 5);
        const int wx = x >> 5, b = x & 31, nw = R >> 5;
        const uint32_t w = __ldg(row + wx);
        uint32_t m = w & (0xFFFFFFFFu >> (31 - b));  // bits 0..b
        if (m) best = b - (31 - __clz(m));
        else
            for (int k = wx - 1; k >= 0 && k >= wx - 8; --k) {
                m = __ldg(row + k);
                if (m) {
                    best = min(best, x - (32 * k + 31 - __clz(m)));
                    break;
                }
            }
        m = w & (0xFFFFFFFFu << b);  // bits b..31
        if (m) best = min(best, (__ffs(m) - 1) - b);
        else
            for (int k = wx + 1; k < nw && k <= wx + 8; ++k) {
                m = __ldg(row + k);
                if (m) {
                    best = min(best, 32 * k + __ffs(m) - 1 - x);
                    break;
                }
            }
    } else {
        for (int q = 0; q < R; ++q) {
            const size_t i = row_bit0 + q;
            if ((__ldg(bits + (i >> 5)) >> (i & 31)) & 1u) best = min(best, q < x ? x - q : q - x);
        }
    }
    return min(max(best - 1, 0), 255);
}

constexpr int kSat = 255 * 255;

// E of every entry of the TX columns f [R][TX] in shared memory (saturated at kSat; arg:
// scratch for the minimisers).  All threads of the block.  Bound by the search's
// instructions: the sums, at most 255^2 + 1023^2 < 2^21, carry their position in 10 low
// bits, so that one minimum keeps both (and the leftmost of equal ones): load, two
// multiply-adds, add and minimum a step.
template <int TX>
__device__ __forceinline__ void line_minima(const uint16_t* f, uint16_t* E, uint16_t* arg, int R) {
    auto search = [&](int j, int x, int lo, int hi) {
        const uint16_t* p = f + lo * TX + x;
        uint32_t best = 0xFFFFFFFFu;
        int d = j - lo, n = hi - lo + 1, q = lo;
        auto key = [&](int i) {
            const int e = d - i;
            return ((uint32_t)p[i * TX] + (uint32_t)(e * e)) * 1024u + (uint32_t)i;
        };
        for (; n >= 8; n -= 8, p += 8 * TX, d -= 8, q += 8) {
            const uint32_t a = min(min(key(0), key(1)), min(key(2), key(3)));
            const uint32_t b = min(min(key(4), key(5)), min(key(6), key(7)));
            best = min(best, min(a, b) + (uint32_t)q);
        }
        for (; n > 0; --n, p += TX, --d, ++q) best = min(best, key(0) + (uint32_t)q);
        E[j * TX + x] = (uint16_t)min(best >> 10, (uint32_t)kSat);
        arg[j * TX + x] = (uint16_t)(best & 1023u);
    };
    int s = R >= 4 ? R >> 2 : 1;
    for (int i = threadIdx.x; i < (R / s) * TX; i += blockDim.x) search((i / TX) * s, i & (TX - 1), 0, R - 1);
    for (; s > 1; s >>= 1) {
        __syncthreads();
        const int h = s >> 1;  // the midpoints h, h + s, h + 2 s, ...
        for (int i = threadIdx.x; i < (R / s) * TX; i += blockDim.x) {
            const int j = (i / TX) * s + h, x = i & (TX - 1);
            search(j, x, arg[(j - h) * TX + x], j + h < R ? arg[(j + h) * TX + x] : R - 1);
        }
    }
    __syncthreads();
}

// The box gap's minimum of entry i (see above).
template <int TX>
__device__ __forceinline__ int line_value(const uint16_t* E, int i, int x, int R) {
    int v = E[i * TX + x];
    if (i > 0) v = min(v, (int)E[(i - 1) * TX + x]);
    if (i + 1 < R) v = min(v, (int)E[(i + 1) * TX + x]);
    return v;
}

// x and y passes.  Block = TX neighbouring x over all y of one z (lanes along x: a warp
// reads whole rows).
template <int TX>
__global__ void __launch_bounds__(256) edt_xy_kernel(const uint32_t* __restrict__ bits, uint16_t* __restrict__ out,
                                                     int R) {
    extern __shared__ uint16_t lines[];
    const int n = R * TX;
    uint16_t *f = lines, *E = f + n, *arg = E + n;
    const int x0 = blockIdx.x * TX, z = blockIdx.y;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int g = row_gap(bits, (size_t)R * ((size_t)(i / TX) + (size_t)R * z), R, x0 + (i & (TX - 1)));
        f[i] = (uint16_t)(g * g);
    }
    __syncthreads();
    line_minima<TX>(f, E, arg, R);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int x = i & (TX - 1), y = i / TX;
        out[(size_t)(x0 + x) + (size_t)R * ((size_t)y + (size_t)R * z)] = (uint16_t)line_value<TX>(E, y, x, R);
    }
}

// z pass and the root.  Block = TX neighbouring x over all z of one y.
template <int TX>
__global__ void __launch_bounds__(256) edt_z_kernel(const uint16_t* __restrict__ in, uint8_t* __restrict__ dist, int R) {
    extern __shared__ uint16_t lines[];
    const int n = R * TX;
    uint16_t *f = lines, *E = f + n, *arg = E + n;
    const int x0 = blockIdx.x * TX, y = blockIdx.y;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        f[i] = in[(size_t)(x0 + (i & (TX - 1))) + (size_t)R * ((size_t)y + (size_t)R * (i / TX))];
    __syncthreads();
    line_minima<TX>(f, E, arg, R);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int x = i & (TX - 1), z = i / TX;
        // exact floor: sqrtf is correctly rounded, and the root of a non-square below
        // 2^16 is at least 1/512 away from an integer
        dist[(size_t)(x0 + x) + (size_t)R * ((size_t)y + (size_t)R * z)] =
            (uint8_t)(int)sqrtf((float)line_value<TX>(E, z, x, R));
    }
}

template <int TX>
void launch_edt(const uint32_t* bits, uint16_t* sums, uint8_t* dist, int R, cudaStream_t st) {
    const dim3 grid((unsigned)(R / TX), (unsigned)R);
    const size_t shm = 3 * (size_t)R * TX * sizeof(uint16_t);
    edt_xy_kernel<TX><<<grid, 256, shm, st>>>(bits, sums, R);
    edt_z_kernel<TX><<<grid, 256, shm, st>>>(sums, dist, R);
}

size_t words(size_t bits) { return (bits + 31) / 32; }

}  // namespace
}  // namespace ngprt

using namespace ngprt;

extern "C" size_t ngprt_occ_bits_words(int32_t R, int32_t n_levels) {
    if (R <= 0 || n_levels <= 0) return 0;
    size_t total = 0;
    for (int k = 0; k < n_levels; ++k) {
        size_t r = (size_t)(R >> k);
        total += words(r * r * r);
    }
    return total;
}

extern "C" size_t ngprt_build_occ_dist_workspace_bytes(int32_t R) {
    if (R <= 0) return 0;
    size_t n = (size_t)R * R * R;
    return 2 * ((n * sizeof(int32_t) + 255) / 256 * 256);
}

extern "C" int32_t ngprt_build_occ_dist(const uint8_t* occ, int32_t R, int32_t n_levels, int32_t dist_level,
                                        uint32_t* occ_bits_out, uint8_t* dist_out, void* workspace, size_t ws_bytes,
                                        void* stream) {
    NGPRT_REQUIRE(occ != nullptr, "ngprt_build_occ_dist: occ is NULL");
    NGPRT_REQUIRE(occ_bits_out != nullptr, "ngprt_build_occ_dist: occ_bits_out is NULL");
    NGPRT_REQUIRE(R >= 2 && R <= 1024 && (R & (R - 1)) == 0, "ngprt_build_occ_dist: R=%d must be a power of two in [2, 1024]", R);
    NGPRT_REQUIRE(n_levels >= 1 && n_levels <= kMaxOccLevels && (R >> (n_levels - 1)) >= 1,
                  "ngprt_build_occ_dist: n_levels=%d invalid for R=%d", n_levels, R);
    NGPRT_REQUIRE(dist_level >= 0 && dist_level < n_levels, "ngprt_build_occ_dist: dist_level=%d not in [0, %d)",
                  dist_level, n_levels);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t n = (size_t)R * R * R;
    // pyramid
    size_t w0 = words(n);
    const unsigned pb = (unsigned)((w0 + 255) / 256);
    if (((uintptr_t)occ & 15) == 0 && n % 32 == 0) pack_bits_kernel<true><<<pb, 256, 0, st>>>(occ, n, occ_bits_out, w0);
    else pack_bits_kernel<false><<<pb, 256, 0, st>>>(occ, n, occ_bits_out, w0);
    size_t off_prev = 0, off = w0, dist_off = 0;
    int k = 1;
    for (; k < n_levels && (R >> (k - 1)) > kTailRes; ++k) {
        const int rc = R >> k;
        const size_t wk = words((size_t)rc * rc * rc);
        downsample_kernel<<<(unsigned)((wk + 127) / 128), 128, 0, st>>>(occ_bits_out + off_prev, occ_bits_out + off, rc,
                                                                        wk);
        off_prev = off;
        off += wk;
    }
    if (k < n_levels)
        downsample_tail_kernel<<<1, 1024, 0, st>>>(occ_bits_out + off_prev, R >> (k - 1), n_levels - k);
    for (int j = 0; j < dist_level; ++j) dist_off += words((size_t)(R >> j) * (R >> j) * (R >> j));
    if (dist_out) {
        size_t need = ngprt_build_occ_dist_workspace_bytes(R);
        if (workspace == nullptr || ws_bytes < need) {
            set_error("ngprt_build_occ_dist: workspace %zu bytes < %zu needed", ws_bytes, need);
            return NGPRT_ERR_WORKSPACE;
        }
        NGPRT_REQUIRE(((uintptr_t)workspace & 255) == 0, "ngprt_build_occ_dist: workspace not 256-byte aligned");
        // G on level dist_level, from its bits
        const int Rg = R >> dist_level;
        uint16_t* sums = static_cast<uint16_t*>(workspace);
        // 32 columns a block (fewer where the grid has fewer, or where three 16-bit
        // arrays of R x TX would pass 48 KB of shared memory)
        const uint32_t* bits = occ_bits_out + dist_off;
        switch (Rg) {
            case 1: launch_edt<1>(bits, sums, dist_out, Rg, st); break;
            case 2: launch_edt<2>(bits, sums, dist_out, Rg, st); break;
            case 4: launch_edt<4>(bits, sums, dist_out, Rg, st); break;
            case 8: launch_edt<8>(bits, sums, dist_out, Rg, st); break;
            case 16: case 512: launch_edt<16>(bits, sums, dist_out, Rg, st); break;
            case 1024: launch_edt<8>(bits, sums, dist_out, Rg, st); break;
            default: launch_edt<32>(bits, sums, dist_out, Rg, st); break;
        }
    }
    return cuda_status("ngprt_build_occ_dist");
}
