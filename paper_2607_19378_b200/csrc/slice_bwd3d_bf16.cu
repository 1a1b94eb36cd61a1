// Instances of the slice-fused backward for 3-D grids of bf16 tensors.
#include "slice_bwd.cuh"
#define HN_SLICE_T bf16

namespace hn {

int launch_slice_bwd_3d_bf16(const SliceBwdArgs &a, cudaStream_t st)
{
    HN_SLICE_3D(HN_SLICE_BWD_CASE)
    return -1;
}

}  // namespace hn
