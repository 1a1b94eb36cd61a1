// Pointwise stages of the full HyenaND operator, Eq. 2 of the paper (Section 3.2):
//
//     y = RMSNorm( Sigmoid(v) * ( K conv RMSNorm( l2(q) * SiLU(k) ) ) )
//
// Both normalisations and the l2 norm act per token across the C channels, which lie L elements apart in the [B][C][L]
// layout.  A CTA takes a tile of neighbouring tokens; its warps share the channels and walk them with the loads of several
// channels in flight (whole 64- or 128-byte segments each), the partial sums meet in shared memory.  (One thread per token
// walking all channels left 64 CTAs on the GPU for 4 x 64 x 64 tokens and one load in flight per thread: 245 us for the
// inner stage, 64 for the outer one at C = 384, bf16; now 14 and 16.)
//
//   token_scale   one number per token: both inner norms together.  Where the convolution is one kernel it evaluates
//                 q scale g_in SiLU(k) and Sigmoid(v) itself as it reads its tensors; elsewhere they are written out in
//                 fp32 by the same kernel.
//   mixer_post    the outer RMSNorm.
// All arithmetic is fp32; nothing is rounded to bf16 before the final store of y.
#include "common.cuh"
#include "mix.cuh"
#include "mixer.cuh"
#include <type_traits>

namespace hn {

constexpr int kMixThreads = 256;
constexpr float kL2Floor = 1e-12f;

// VEC neighbouring tokens of one channel
template <typename T, int VEC> struct MixVec;
template <typename T> struct MixVec<T, 1> {
    static __device__ __forceinline__ void ld(const T *p, float (&f)[1]) { f[0] = IO<T>::ld(p, 0); }
    static __device__ __forceinline__ void st(T *p, const float (&f)[1]) { IO<T>::st(p, 0, f[0]); }
};
template <> struct MixVec<float, 2> {
    static __device__ __forceinline__ void ld(const float *p, float (&f)[2]) { HN_G(p, 8); const float2 v = __ldg(reinterpret_cast<const float2 *>(p)); f[0] = v.x; f[1] = v.y; }
    static __device__ __forceinline__ void st(float *p, const float (&f)[2]) { HN_G(p, 8); *reinterpret_cast<float2 *>(p) = make_float2(f[0], f[1]); }
};
template <> struct MixVec<bf16, 2> {
    static __device__ __forceinline__ void ld(const bf16 *p, float (&f)[2])
    {
        HN_G(p, 4);
        const unsigned v = __ldg(reinterpret_cast<const unsigned *>(p));
        f[0] = __uint_as_float(v << 16); f[1] = __uint_as_float(v & 0xffff0000u);
    }
    static __device__ __forceinline__ void st(bf16 *p, const float (&f)[2]) { HN_G(p, 4); *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(f[0], f[1]); }
};
template <> struct MixVec<float, 4> {
    static __device__ __forceinline__ void ld(const float *p, float (&f)[4])
    {
        HN_G(p, 16);
        const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
    }
    static __device__ __forceinline__ void st(float *p, const float (&f)[4]) { HN_G(p, 16); *reinterpret_cast<float4 *>(p) = make_float4(f[0], f[1], f[2], f[3]); }
};
template <> struct MixVec<bf16, 4> {
    static __device__ __forceinline__ void ld(const bf16 *p, float (&f)[4])
    {
        HN_G(p, 8);
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
        f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xffff0000u);
        f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xffff0000u);
    }
    static __device__ __forceinline__ void st(bf16 *p, const float (&f)[4])
    {
        HN_G(p, 8);
        __nv_bfloat162 h[2] = {__floats2bfloat162_rn(f[0], f[1]), __floats2bfloat162_rn(f[2], f[3])};
        *reinterpret_cast<uint2 *>(p) = *reinterpret_cast<const uint2 *>(h);
    }
};

// Dependent launches: as pdl_join, but tiles of 32 warps that hold most of the SMs and not all of them keep their successor out.  The
// CTAs of a kernel that comes in under them crowd onto the SMs left over (Eq. 2 on 100 to 132 such tiles 0.93 to 1.00 of its speed
// with a plain launch; below 74 tiles 1.00 to 1.4).
template <int NW> __device__ __forceinline__ void mix_join()
{
    pdl_wait();
    if (NW < 32 || gridDim.x * gridDim.y < kSms / 2) pdl_trigger();
}

// a token's scale from sum_c q^2 and sum_c (q SiLU(k))^2: mean_c (l2(q) SiLU(k))^2 = s2 / (C ||q||^2)
__device__ __forceinline__ float token_factor(float s1, float s2, int C, float eps)
{
    const float inv = 1.f / fmaxf(sqrtf(s1), kL2Floor);
    return inv * rsqrtf(s2 * inv * inv / (float)C + eps);
}

// 32 * VEC tokens per CTA of NW warps; channels c = warp, warp + NW, ... in rounds of U.
// GATES: the kernel also writes qz = Sigmoid(v) and the gated signal, kz = q scale g_in with vz = SiLU(k), or the product of
// both as kz where vz is nullptr; q and k are read once more (from the caches) where a thread's channels need several rounds.
template <typename T, int VEC, int NW, bool GATES>
__global__ void __launch_bounds__(NW * 32) token_scale_kernel(const T *q, const T *k, const T *v, const float *g_in, float eps, int C, long long L,
                                                              float *scale, float *qz, float *kz, float *vz)
{
    constexpr int U = 8;
    __shared__ float red[2][NW][32 * VEC];
    mix_join<NW>();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long i = ((long long)blockIdx.x * 32 + lane) * VEC, b = blockIdx.y, base = b * C * L + i;
    const bool live = i < L;                                 // (VEC > 1 only where it divides L)
    float s1[VEC] = {}, s2[VEC] = {};                        // sum q^2, sum (q SiLU(k))^2
    float qv[U][VEC], kv[U][VEC];
    for (int c0 = w; c0 < C; c0 += NW * U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + u * NW;
#pragma unroll
            for (int e = 0; e < VEC; ++e) qv[u][e] = kv[u][e] = 0.f;
            if (live && c < C) { MixVec<T, VEC>::ld(q + base + c * L, qv[u]); MixVec<T, VEC>::ld(k + base + c * L, kv[u]); }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const float qs = qv[u][e] * (kv[u][e] * mix_sigmoid(kv[u][e]));
                s1[e] = fmaf(qv[u][e], qv[u][e], s1[e]);
                s2[e] = fmaf(qs, qs, s2[e]);
            }
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) { red[0][w][lane * VEC + e] = s1[e]; red[1][w][lane * VEC + e] = s2[e]; }
    __syncthreads();
    for (int t = threadIdx.x; t < 32 * VEC; t += NW * 32) {
        float a = 0.f, d = 0.f;
#pragma unroll
        for (int j = 0; j < NW; ++j) { a += red[0][j][t]; d += red[1][j][t]; }       // (red[0][0][t] is this thread's alone to replace)
        const long long tok = (long long)blockIdx.x * 32 * VEC + t;
        const float sc = token_factor(a, d, C, eps);
        if constexpr (GATES) red[0][0][t] = sc;
        else if (tok < L) { HN_G(scale + b * L + tok, 4); scale[b * L + tok] = sc; }
    }
    if constexpr (GATES) {
        __syncthreads();
        float sc[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) sc[e] = red[0][0][lane * VEC + e];
        auto gates = [&](int c, float (&a)[VEC], float (&x)[VEC], float (&z)[VEC]) {
            HN_G(g_in + c, 4);
            const float g = __ldg(g_in + c);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                a[e] *= sc[e] * g;
                x[e] *= mix_sigmoid(x[e]);
                z[e] = mix_sigmoid(z[e]);
                if (!vz) a[e] *= x[e];
            }
            MixVec<float, VEC>::st(kz + base + c * L, a);
            if (vz) MixVec<float, VEC>::st(vz + base + c * L, x);
            MixVec<float, VEC>::st(qz + base + c * L, z);
        };
        if (C <= NW * U) {                                   // the one round's q and k are still in registers
            float z[U][VEC];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (live && w + u * NW < C) MixVec<T, VEC>::ld(v + base + (w + u * NW) * L, z[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (live && w + u * NW < C) gates(w + u * NW, qv[u], kv[u], z[u]);
            return;
        }
        constexpr int UG = 4;
        for (int c0 = w; c0 < C; c0 += NW * UG) {
            float x[3][UG][VEC];
#pragma unroll
            for (int u = 0; u < UG; ++u) {
                const int c = c0 + u * NW;
                if (live && c < C) {
                    MixVec<T, VEC>::ld(q + base + c * L, x[0][u]); MixVec<T, VEC>::ld(k + base + c * L, x[1][u]); MixVec<T, VEC>::ld(v + base + c * L, x[2][u]);
                }
            }
#pragma unroll
            for (int u = 0; u < UG; ++u)
                if (live && c0 + u * NW < C) gates(c0 + u * NW, x[0][u], x[1][u], x[2][u]);
        }
    }
}

// KEEP > 0: a thread's channels (at most KEEP) stay in registers between the sum and the result; 0: read twice
template <typename T, int VEC, int NW, int KEEP>
__global__ void __launch_bounds__(NW * 32) mixer_post_kernel(const float *o, const float *g_out, float eps, int C, long long L, T *y)
{
    constexpr int U = KEEP ? KEEP : 8;
    __shared__ float red[NW][32 * VEC];
    __shared__ float scl[32 * VEC];
    mix_join<NW>();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long i = ((long long)blockIdx.x * 32 + lane) * VEC, base = (long long)blockIdx.y * C * L + i;
    const bool live = i < L;
    float s[VEC] = {}, x[U][VEC];
    for (int c0 = w; c0 < C; c0 += NW * U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + u * NW;
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[u][e] = 0.f;
            if (live && c < C) MixVec<float, VEC>::ld(o + base + c * L, x[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int e = 0; e < VEC; ++e) s[e] = fmaf(x[u][e], x[u][e], s[e]);
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) red[w][lane * VEC + e] = s[e];
    __syncthreads();
    for (int t = threadIdx.x; t < 32 * VEC; t += NW * 32) {
        float a = 0.f;
#pragma unroll
        for (int j = 0; j < NW; ++j) a += red[j][t];
        scl[t] = rsqrtf(a / (float)C + eps);
    }
    __syncthreads();
    float sc[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) sc[e] = scl[lane * VEC + e];
    for (int c0 = w; c0 < C; c0 += NW * U) {
        if (!KEEP) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + u * NW;
                if (live && c < C) MixVec<float, VEC>::ld(o + base + c * L, x[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + u * NW;
            if (live && c < C) {
                HN_G(g_out + c, 4);
                const float g = __ldg(g_out + c);
                float r[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) r[e] = x[u][e] * sc[e] * g;
                MixVec<T, VEC>::st(y + base + c * L, r);
            }
        }
    }
}

// Few channels and many tokens: a thread owns VEC tokens and walks their channels, four at a time and the rest one by one; no
// shared memory, no barrier.  (A tile of four warps has less than a channel per warp and loop slot there and is gone before it has
// paid for its start: operator on 16 x 512 x 512 tokens of 2 channels, fp32, 1066 us with tiles, here 881.)
template <typename T, int VEC, bool GATES>
__global__ void __launch_bounds__(kMixThreads) token_solo_kernel(const T *q, const T *k, const T *v, const float *g_in, float eps, int C, long long L,
                                                                 float *scale, float *qz, float *kz, float *vz)
{
    constexpr int U = 4;
    const long long i = ((long long)blockIdx.x * kMixThreads + threadIdx.x) * VEC, b = blockIdx.y, base = b * C * L + i;
    pdl_join();
    if (i >= L) return;                                      // (VEC > 1 only where it divides L)
    float s1[VEC] = {}, s2[VEC] = {}, sc[VEC];
    auto sums = [&](int c, auto n) {
        constexpr int N = decltype(n)::value;
        float x[N][VEC], y[N][VEC];
#pragma unroll
        for (int u = 0; u < N; ++u) { MixVec<T, VEC>::ld(q + base + (c + u) * L, x[u]); MixVec<T, VEC>::ld(k + base + (c + u) * L, y[u]); }
#pragma unroll
        for (int u = 0; u < N; ++u)
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const float qs = x[u][e] * (y[u][e] * mix_sigmoid(y[u][e]));
                s1[e] = fmaf(x[u][e], x[u][e], s1[e]);
                s2[e] = fmaf(qs, qs, s2[e]);
            }
    };
    auto write = [&](int c, auto n) {
        constexpr int N = decltype(n)::value;
        float a[N][VEC], x[N][VEC], z[N][VEC];
#pragma unroll
        for (int u = 0; u < N; ++u) {
            MixVec<T, VEC>::ld(q + base + (c + u) * L, a[u]); MixVec<T, VEC>::ld(k + base + (c + u) * L, x[u]); MixVec<T, VEC>::ld(v + base + (c + u) * L, z[u]);
        }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            HN_G(g_in + c + u, 4);
            const float g = __ldg(g_in + c + u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                a[u][e] *= sc[e] * g;
                x[u][e] *= mix_sigmoid(x[u][e]);
                z[u][e] = mix_sigmoid(z[u][e]);
                if (!vz) a[u][e] *= x[u][e];
            }
            MixVec<float, VEC>::st(kz + base + (c + u) * L, a[u]);
            if (vz) MixVec<float, VEC>::st(vz + base + (c + u) * L, x[u]);
            MixVec<float, VEC>::st(qz + base + (c + u) * L, z[u]);
        }
    };
    const std::integral_constant<int, U> several{};
    const std::integral_constant<int, 1> one{};
    int c = 0;
    for (; c + U <= C; c += U) sums(c, several);
    for (; c < C; ++c) sums(c, one);
#pragma unroll
    for (int e = 0; e < VEC; ++e) sc[e] = token_factor(s1[e], s2[e], C, eps);
    if constexpr (GATES) {
        for (c = 0; c + U <= C; c += U) write(c, several);
        for (; c < C; ++c) write(c, one);
    } else {
        MixVec<float, VEC>::st(scale + b * L + i, sc);
    }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(kMixThreads) post_solo_kernel(const float *o, const float *g_out, float eps, int C, long long L, T *y)
{
    constexpr int U = 4;
    const long long i = ((long long)blockIdx.x * kMixThreads + threadIdx.x) * VEC, base = (long long)blockIdx.y * C * L + i;
    pdl_join();
    if (i >= L) return;
    float s[VEC] = {};
    auto sums = [&](int c, auto n) {
        constexpr int N = decltype(n)::value;
        float x[N][VEC];
#pragma unroll
        for (int u = 0; u < N; ++u) MixVec<float, VEC>::ld(o + base + (c + u) * L, x[u]);
#pragma unroll
        for (int u = 0; u < N; ++u)
#pragma unroll
            for (int e = 0; e < VEC; ++e) s[e] = fmaf(x[u][e], x[u][e], s[e]);
    };
    auto write = [&](int c, auto n) {
        constexpr int N = decltype(n)::value;
        float x[N][VEC];
#pragma unroll
        for (int u = 0; u < N; ++u) MixVec<float, VEC>::ld(o + base + (c + u) * L, x[u]);
#pragma unroll
        for (int u = 0; u < N; ++u) {
            HN_G(g_out + c + u, 4);
            const float g = __ldg(g_out + c + u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[u][e] *= s[e] * g;
            MixVec<T, VEC>::st(y + base + (c + u) * L, x[u]);
        }
    };
    const std::integral_constant<int, U> several{};
    const std::integral_constant<int, 1> one{};
    int c = 0;
    for (; c + U <= C; c += U) sums(c, several);
    for (; c < C; ++c) sums(c, one);
#pragma unroll
    for (int e = 0; e < VEC; ++e) s[e] = rsqrtf(s[e] / (float)C + eps);
    for (c = 0; c + U <= C; c += U) write(c, several);
    for (; c < C; ++c) write(c, one);
}

template <typename T> __global__ void widen_kernel(const T *src, long long n, float *dst)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        { HN_G(dst + i, 4); dst[i] = IO<T>::ld(src, i); }
}

static int mix_grid(long long items)
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 148;
    }
    const long long want = (items + kMixThreads - 1) / kMixThreads, cap = (long long)sms * 8;
    return (int)(want < cap ? want : cap);
}

// Tiles of 32 tokens, or of 64 or 128 (two or four per lane) where rows divide that way and 1024 such tiles exist; the fewest
// warps per tile that make 4096 warps in all, but no more than one per 8 channels or so.  Measured (bf16, scale + outer norm,
// us): 512 tiles of 384 channels 29 with 8 warps, 34 with 16, 41 with 32; 42 tiles of 1170 channels 51, 31, 22.
// A thread per token (token_solo_kernel) takes few channels of many tokens, and rows that no vector of tokens divides, whose
// tiles of 32 tokens start anywhere (operators, us, tiles -> solo: 8 x 511 x 511 tokens of 12 channels bf16 1292 -> 1106, of 48
// 3995 -> 3490; fp32 of 24 2096 -> 1959, but 365 x 365 of 96 574 -> 604: few tokens or many fp32 channels stay with the tiles).
constexpr int kSoloChannels = 16, kSoloOddF32 = 48;
template <typename T, class F> static void mix_tiles(long long nb, long long L, int C, F go)
{
    auto count = [&](int vec) { return nb * ((L + 32 * vec - 1) / (32 * vec)); };
    const int vec = L % 4 == 0 && count(4) >= 1024 ? 4 : L % 2 == 0 && count(2) >= 1024 ? 2 : 1;
    const long long tiles = count(vec);
    int nw = 4;
    while (nw < 32 && tiles * nw < 4096 && nw * 8 < C) nw *= 2;
    const dim3 grid((unsigned)((L + 32 * vec - 1) / (32 * vec)), (unsigned)nb);
    const std::integral_constant<int, 0> solo{};
    const std::integral_constant<int, 1> one{};
    const std::integral_constant<int, 2> two{};
    const std::integral_constant<int, 4> four{};
    if ((C <= kSoloChannels && tiles >= 1024) || (vec == 1 && tiles >= 4096 && (sizeof(T) == 2 || C <= kSoloOddF32))) {
        const dim3 g((unsigned)((L + kMixThreads * vec - 1) / (kMixThreads * vec)), (unsigned)nb);
        return vec == 4 ? go(four, solo, g) : vec == 2 ? go(two, solo, g) : go(one, solo, g);
    }
    // 16 warps on tiles of 64 tokens, from 128 such tiles on: where tiles of 32 tokens would take 32 warps for at most 8 channels each,
    // and for bf16 at 256 to 384 channels, which stay in registers (24 per thread) between the outer norm's sum and its result.
    // Eq. 2 without the synthesis against those tiles, 196 to 5280 tokens, 1 to 32 entries: the first 0.99 to 1.11 times as fast, the
    // second 0.98 to 1.06 (4 x 4096 tokens of 384 channels: outer norm 17.6 -> 14.0 us); but bf16 of 128 to 192 channels 0.96 to 1.02, of
    // 512 and more 0.86 to 1.05, other fp32 0.92 to 1.02.
    if (vec == 1 && L % 2 == 0 && count(2) >= 128 && ((nw == 32 && C <= 256) || (sizeof(T) == 2 && C >= 256 && C <= 384)))
        return go(two, std::integral_constant<int, 16>{}, dim3((unsigned)((L + 63) / 64), (unsigned)nb));
    if (vec == 4) return go(four, four, grid);               // (1024 tiles of 4 warps)
    if (vec == 2) return go(two, four, grid);
    if (nw == 4) go(one, four, grid);
    else if (nw == 8) go(one, std::integral_constant<int, 8>{}, grid);
    else if (nw == 16) go(one, std::integral_constant<int, 16>{}, grid);
    else go(one, std::integral_constant<int, 32>{}, grid);
}

template <typename T, bool GATES>
static void token_scale_t(const T *q, const T *k, const T *v, const float *g_in, float eps, long long nb, int C, long long L, float *scale,
                          float *qz, float *kz, float *vz, cudaStream_t st)
{
    mix_tiles<T>(nb, L, C, [&](auto vec, auto nw, dim3 grid) {
        constexpr int VEC = decltype(vec)::value, NW = decltype(nw)::value;
        if constexpr (NW == 0) launch_pdl(token_solo_kernel<T, VEC, GATES>, grid, kMixThreads, 0, st, q, k, v, g_in, eps, C, L, scale, qz, kz, vz);
        else launch_pdl(token_scale_kernel<T, VEC, NW, GATES>, grid, NW * 32, 0, st, q, k, v, g_in, eps, C, L, scale, qz, kz, vz);
    });
}

int launch_token_scale(const void *q, const void *k, float eps, int dtype, long long nb, int C, long long L, float *scale, cudaStream_t st)
{
    for (long long b0 = 0; b0 < nb; b0 += 65535) {           // (limit of a grid's second dimension)
        const long long n = nb - b0 < 65535 ? nb - b0 : 65535, off = b0 * C * L;
        if (dtype == 0) token_scale_t<float, false>((const float *)q + off, (const float *)k + off, nullptr, nullptr, eps, n, C, L, scale + b0 * L, nullptr, nullptr, nullptr, st);
        else token_scale_t<bf16, false>((const bf16 *)q + off, (const bf16 *)k + off, nullptr, nullptr, eps, n, C, L, scale + b0 * L, nullptr, nullptr, nullptr, st);
    }
    return 1;
}

int launch_mixer_gates(const void *q, const void *k, const void *v, const float *g_in, float eps, int dtype,
                       long long nb, int C, long long L, float *qz, float *kz, float *vz, cudaStream_t st)
{
    for (long long b0 = 0; b0 < nb; b0 += 65535) {
        const long long n = nb - b0 < 65535 ? nb - b0 : 65535, off = b0 * C * L;
        if (dtype == 0) token_scale_t<float, true>((const float *)q + off, (const float *)k + off, (const float *)v + off, g_in, eps, n, C, L, nullptr, qz + off, kz + off, vz ? vz + off : nullptr, st);
        else token_scale_t<bf16, true>((const bf16 *)q + off, (const bf16 *)k + off, (const bf16 *)v + off, g_in, eps, n, C, L, nullptr, qz + off, kz + off, vz ? vz + off : nullptr, st);
    }
    return 1;
}

template <typename T> static void mixer_post_t(const float *o, const float *g_out, float eps, long long nb, int C, long long L, T *y, cudaStream_t st)
{
    mix_tiles<T>(nb, L, C, [&](auto vec, auto nw, dim3 grid) {
        constexpr int VEC = decltype(vec)::value, NW = decltype(nw)::value;
        if constexpr (NW == 0) {
            launch_pdl(post_solo_kernel<T, VEC>, grid, kMixThreads, 0, st, o, g_out, eps, C, L, y);
        } else {
            const int per = (C + NW - 1) / NW;               // channels per thread
            if (per <= 4) launch_pdl(mixer_post_kernel<T, VEC, NW, 4>, grid, NW * 32, 0, st, o, g_out, eps, C, L, y);
            else if (per <= 16) launch_pdl(mixer_post_kernel<T, VEC, NW, 16>, grid, NW * 32, 0, st, o, g_out, eps, C, L, y);
            else {
                if constexpr (VEC == 2 && NW == 16) {        // (1024 threads have 64 registers each: 24 channels would spill)
                    if (per <= 24) return launch_pdl(mixer_post_kernel<T, VEC, NW, 24>, grid, NW * 32, 0, st, o, g_out, eps, C, L, y);
                }
                launch_pdl(mixer_post_kernel<T, VEC, NW, 0>, grid, NW * 32, 0, st, o, g_out, eps, C, L, y);
            }
        }
    });
}

int launch_mixer_post(const float *o, const float *g_out, float eps, int dtype, long long nb, int C, long long L,
                      void *y, cudaStream_t st)
{
    for (long long b0 = 0; b0 < nb; b0 += 65535) {
        const long long n = nb - b0 < 65535 ? nb - b0 : 65535, off = b0 * C * L;
        if (dtype == 0) mixer_post_t(o + off, g_out, eps, n, C, L, (float *)y + off, st);
        else mixer_post_t(o + off, g_out, eps, n, C, L, (bf16 *)y + off, st);
    }
    return 1;
}

int launch_widen(const void *src, int dtype, long long n, float *dst, cudaStream_t st)
{
    const int grid = mix_grid(n);
    if (grid <= 0) return 0;
    if (dtype == 0) widen_kernel<float><<<grid, kMixThreads, 0, st>>>((const float *)src, n, dst);
    else widen_kernel<bf16><<<grid, kMixThreads, 0, st>>>((const bf16 *)src, n, dst);
    return 1;
}

}  // namespace hn
