// Slice-fused path: the whole operator for one (b,c) slice in one group of threads, spectra in shared memory only.
#pragma once
#include "common.cuh"

namespace hn {

// How a slice's grid sits on the padded grid of the slice engine: n0 x n1 x n2 complex points, n2 = P2 / 2.
struct SliceGeo {
    int l0, l1, l2;           // log2 of n0, n1, n2
    int L[3];                 // grid extents
    int K[3];                 // tap extents
    int shift[3];             // padded position x holds tap (x + shift) mod P (0: causal, circular)
    int full;                 // 1: circular mode (nothing padded)
    long long vol, kvol;
};

// Chooses the padded grid for extents L (internal 3-axis form); false where the engine has no instance for it.
bool slice_geo(SliceGeo *g, const int *L, int mode_causal, int mode_circular);

struct SliceArgs {
    const void *q, *k, *v, *h;
    void *y;
    long long s0, s1;         // slices [s0, s1) of the tensors q, k, v, y (h: the same slices, or slice c when shared)
    int C;                    // channels, for a filter shared over the batch; 0: one filter per slice
    int nb;                   // batch entries per unit of work (shared filter)
    int h_bf16;               // element type of the taps
    // Eq. 2 around the convolution (nullptr: none): k, v, q are the operator's q, k, v, y is fp32
    const float *token_scale; // [B][grid]
    const float *g_in;        // [mix_C]
    int mix_C;
    SliceGeo g;
    const float2 *gtw;
    int gtw_n;
};

int launch_slice(const SliceArgs &a, int dtype, cudaStream_t st);

// Gradients of `slices` slices (backward pass).
struct SliceBwdArgs {
    const void *q, *k, *v, *h, *dy;
    void *dq, *dk, *dv;
    void *dh;                 // one set of taps per slice
    int dh_f32;               // taps leave in fp32 (they are summed over the batch afterwards), else in the tensors' type
    long long slices;
    int C;                    // channels, for a filter shared over the batch (slices start at a batch entry); 0: one per slice
    SliceGeo g;
    const float2 *gtw;
    int gtw_n;
};
int launch_slice_bwd(const SliceBwdArgs &a, int dtype, cudaStream_t st);

// resident CTAs of a kernel on the current device (cached in `cache`, one entry per device); sets its shared-memory limit
int slice_resident(int (&cache)[64], const void *fn, int threads, size_t smem);

}  // namespace hn
