// Instances of the slice-fused forward inside Eq. 2 for 1-D grids of bf16 tensors.
#include "slice_fwd.cuh"
#define HN_SLICE_T bf16
#define HN_SLICE_MIX true

namespace hn {

int launch_slice_mix_1d_bf16(const SliceArgs &a, cudaStream_t st)
{
    HN_SLICE_1D(HN_SLICE_CASE)
    return -1;
}

}  // namespace hn
