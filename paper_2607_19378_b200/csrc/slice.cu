// Slice-fused path: which grids it takes and how they are padded.
#include "slice_bwd.cuh"

namespace hn {

bool slice_geo(SliceGeo *g, const int *L, int causal, int circular)
{
    const bool one_d = L[0] == 1 && L[1] == 1;
    int l[3];
    for (int a = 0; a < 3; ++a) {
        const int need = circular ? L[a] : 2 * L[a] - 1;
        int b = 0;
        while ((1 << b) < need) ++b;
        if (circular && (1 << b) != L[a]) return false;
        // zero-padded axes may be padded further, to the smallest instance; an axis of one point is no axis
        if (!circular && a < 2 && L[a] > 1 && b < 4) b = 4;
        if (!circular && a == 2 && b < (one_d ? 7 : 5)) b = one_d ? 7 : 5;
        l[a] = b;
    }
    g->l0 = l[0]; g->l1 = l[1]; g->l2 = l[2] - 1;
    bool known = false;
#define HN_SLICE_KNOWN(A, B, C) known = known || (g->l0 == A && g->l1 == B && g->l2 == C);
    HN_SLICE_1D(HN_SLICE_KNOWN) HN_SLICE_2D(HN_SLICE_KNOWN) HN_SLICE_3D(HN_SLICE_KNOWN)
#undef HN_SLICE_KNOWN
    if (!known) return false;
    g->vol = g->kvol = 1;
    g->full = circular;
    for (int a = 0; a < 3; ++a) {
        g->L[a] = L[a];
        g->K[a] = (causal || circular) ? L[a] : 2 * L[a] - 1;
        g->shift[a] = (causal || circular) ? 0 : L[a] - 1;
        g->vol *= g->L[a]; g->kvol *= g->K[a];
    }
    return true;
}

int slice_resident(int (&cache)[64], const void *fn, int threads, size_t smem)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (!cache[dev]) {
        int sms = 0, per = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem) != cudaSuccess) return -1;
        cache[dev] = sms * per;
    }
    return cache[dev];
}

int launch_slice_bwd(const SliceBwdArgs &a, int dtype, cudaStream_t st)
{
    if (a.g.l0 > 0) return dtype == 0 ? launch_slice_bwd_3d_f32(a, st) : launch_slice_bwd_3d_bf16(a, st);
    if (a.g.l1 > 0) return dtype == 0 ? launch_slice_bwd_2d_f32(a, st) : launch_slice_bwd_2d_bf16(a, st);
    return dtype == 0 ? launch_slice_bwd_1d_f32(a, st) : launch_slice_bwd_1d_bf16(a, st);
}

static int launch_range(const SliceArgs &a, int dtype, cudaStream_t st)
{
    const bool f = dtype == 0, m = a.token_scale != nullptr;
    if (a.g.l0 > 0) return m ? (f ? launch_slice_mix_3d_f32(a, st) : launch_slice_mix_3d_bf16(a, st)) : (f ? launch_slice_3d_f32(a, st) : launch_slice_3d_bf16(a, st));
    if (a.g.l1 > 0) return m ? (f ? launch_slice_mix_2d_f32(a, st) : launch_slice_mix_2d_bf16(a, st)) : (f ? launch_slice_2d_f32(a, st) : launch_slice_2d_bf16(a, st));
    return m ? (f ? launch_slice_mix_1d_f32(a, st) : launch_slice_mix_1d_bf16(a, st)) : (f ? launch_slice_1d_f32(a, st) : launch_slice_1d_bf16(a, st));
}

// The kernel's units of a shared filter are channels by groups of whole batch entries.  A range that starts or ends inside an
// entry (hyenand_forward_host above 64 MB) would leave it units without a slice, whose filter it transforms with no barrier
// before the next unit writes the same buffer.  The partial entries run as slices with a filter each, the channel's own (tested
// in the kernel instead, a batch of short sequences takes 147.6 us for 146.8).
int launch_slice(const SliceArgs &a, int dtype, cudaStream_t st)
{
    if (a.C <= 0) return launch_range(a, dtype, st);
    const long long C = a.C, first = (a.s0 + C - 1) / C * C, last = a.s1 / C * C;          // whole entries: [first, last)
    int launches = 0;
    auto run = [&](long long s0, long long s1, bool shared) {
        if (launches < 0 || s0 >= s1) return;
        SliceArgs r = a;
        r.s0 = s0; r.s1 = s1;
        if (!shared) {                                       // slice s of entry s0 / C takes filter s - s0 / C * C
            r.C = 0;
            r.h = (const char *)a.h - s0 / C * C * a.g.kvol * (a.h_bf16 ? 2 : 4);
        }
        const int n = launch_range(r, dtype, st);
        launches = n < 0 ? n : launches + n;
    };
    run(a.s0, first < a.s1 ? first : a.s1, false);
    run(first, last, true);
    if (last >= first) run(last, a.s1, false);
    return launches;
}

}  // namespace hn
