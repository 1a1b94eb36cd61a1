// Instances of the slice-fused forward for 3-D grids of bf16 tensors.
#include "slice_fwd.cuh"
#define HN_SLICE_T bf16
#define HN_SLICE_MIX false

namespace hn {

int launch_slice_3d_bf16(const SliceArgs &a, cudaStream_t st)
{
    HN_SLICE_3D(HN_SLICE_CASE)
    return -1;
}

}  // namespace hn
