// render_l8.cu -- the fused march of Eq. 8 scenes with 8 levels, every table type (one
// translation unit per level count, so that the build compiles them in parallel).
#include "march.cuh"

namespace ngprt {

void launch_march_l8(int dt, const MarchParams& p, dim3 grid, cudaStream_t st) {
    launch_march_kernel<8, NGPRT_AGG_SEPARATE_V>(dt, p, grid, st);
}

}  // namespace ngprt
