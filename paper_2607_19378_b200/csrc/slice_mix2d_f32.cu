// Instances of the slice-fused forward inside Eq. 2 for 2-D grids of fp32 tensors.
#include "slice_fwd.cuh"
#define HN_SLICE_T float
#define HN_SLICE_MIX true

namespace hn {

int launch_slice_mix_2d_f32(const SliceArgs &a, cudaStream_t st)
{
    HN_SLICE_2D(HN_SLICE_CASE)
    return -1;
}

}  // namespace hn
