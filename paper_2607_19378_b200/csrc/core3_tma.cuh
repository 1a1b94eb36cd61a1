// Spectral core of the backward pass with TMA tile copies (core3_tma.cu): interface used by the scheduler.
#pragma once
#include <cuda_runtime.h>
#include "common.cuh"

namespace hn {

// Lines (o, c), element a at base[o * outer + a * nc + c]: u and g with L rows, h and the tap gradients with K rows.
struct Core3Args {
    float2 *u, *g;            // spectra of k v and of dy q; replaced by those of h conv u and of h' conv g, h'[d] = h[-d]
    const float2 *h;          // filter spectra
    float2 *dh;               // spectra of the taps' gradients (may be the filter's own buffer)
    long long n_outer;        // slices
    long long u_outer, h_outer;
    int nc, L, K;
    int h_shift;              // tap row (pos + h_shift) mod P sits at position pos
    int log2p;
    int full;                 // 1: periodic axis, L == K == P
    long long h_mod, h_off;   // filter outer index = h_mod ? (o + h_off) % h_mod : o
    float scale;
    const float2 *gtw;
    int gtw_n;
};

// Tensor maps of the four buffers, for at most max_outer slices (and h_count filters).
struct Core3Maps {
    alignas(64) unsigned char u[128];
    alignas(64) unsigned char g[128];
    alignas(64) unsigned char h[128];
    alignas(64) unsigned char dh[128];
    bool valid;
};

bool core3_tma_supported(int log2p, int full, int nc);
bool core3_tma_make(Core3Maps *m, const Core3Args &a, long long max_outer, long long h_count);
// -1 if the axis length has no kernel (nothing launched); *status: as launch_core_tma
int launch_core3_tma(const Core3Args &a, const Core3Maps &m, int *status, cudaStream_t st);

}  // namespace hn
