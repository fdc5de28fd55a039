// render_l1.cu -- the fused march of Eq. 8 scenes with 1 level, every table type (one
// translation unit per level count, so that the build compiles them in parallel).
#include "march.cuh"

namespace ngprt {

void launch_march_l1(int dt, const MarchParams& p, dim3 grid, cudaStream_t st) {
    launch_march_kernel<1, NGPRT_AGG_SEPARATE_V>(dt, p, grid, st);
}

}  // namespace ngprt
