// Long 1-D path, warp-engine kernels (same decomposition as ct1d.cu: P = P1*P2,
// t = t1*P2 + t2, f = f1 + P1*f2; Appendix B.3 of the paper).
//
//   cols_fwd_w   tile of adjacent column pairs fetched with tensor copies, 8-byte asynchronous copies or, where a
//                slice starts off their boundaries, element by element (eight loads in flight),
//                one warp-group per column pair: transform along t1 (upper half of the
//                padded input is zero), separate the two real columns, multiply by the
//                inter-pass twiddle, coalesced store of [f1][t2].
//   hspec_w      per-sample filters only: transform each kept row along t2 in place and fold in 1/P.
//   core_w       one warp-group per row: transform along t2, multiply by the filter
//                spectrum (Eq. 12), inverse transform chained in registers, undo twiddle.  The
//                rows of a filter shared over the batch are transformed here, once per group of
//                the slices that it serves.
//   cols_inv_w   rebuild the mirrored half, inverse along f1 keeping t < P/2, crop, gate
//                with q, coalesced store.
#include <type_traits>
#include <cstring>
#include <cstdlib>
#include "common.cuh"
#include "tma_util.cuh"
#include "ct1d.cuh"
#include "plane_util.cuh"
#include "tmem_util.cuh"

namespace hn {

// column kernels: CTAs of four warps, several per SM (they synchronise at barriers; more, smaller CTAs keep the schedulers busy)
constexpr int kCtThreads = 128;

template <int BYTES> __device__ __forceinline__ void cp_async_n(void *smem_dst, const void *gmem_src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    HN_G(gmem_src, BYTES);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(gmem_src), "n"(BYTES) : "memory");
}

struct TwoLevelW {
    const float2 *coarse, *fine;
    int lo;
};
__device__ __forceinline__ float2 twp_w(const TwoLevelW &t, unsigned j)
{
    HN_G(t.coarse + (j >> t.lo), 8);
    HN_G(t.fine + (j & ((1u << t.lo) - 1)), 8);
    const float2 c = __ldg(t.coarse + (j >> t.lo));
    const float2 f = __ldg(t.fine + (j & ((1u << t.lo) - 1)));
    return cmul(c, f);
}

// ---- columns, forward ---------------------------------------------------------------------------

struct ColsFwdWArgs {
    const void *a, *b;        // k, v (b == nullptr: plain copy of a, used for a causal filter)
    float2 *out;              // [slices][P1/2+1][P2]
    long long slices;
    long long in_slice;       // elements per slice of the input
    int len;                  // valid elements (<= P/2)
    int *status;              // device word set when a bounded wait on a tensor copy gives up (may be NULL)
    int log2p2;
    const float2 *tw1;        // P1-point table
    TwoLevelW twp;
};

// Tile geometry of the column kernels, one line (column pair) per group of lanes.  Spectra travel as NH halves of rows of ROWB bytes
// (the swizzle span); the rows below P1/2 in boxes, the last one by an untiled copy of its own (a multiple of 8 rows in, where the
// swizzle is the identity), so that the tile is no larger than its rows.
template <typename T, int LOG2P1> struct CtGeo {
    using F = WF<LOG2P1, false>;
    using FI = WF<LOG2P1, true>;
    static constexpr int P1 = 1 << LOG2P1, HP1 = P1 / 2, F1 = HP1 + 1, TPL = F::TPL;
    static constexpr int TX = kCtThreads / TPL, TH = TX < 8 ? TX : 8, NH = TX / TH;           // pairs per tile and per half
    static constexpr unsigned ROWB = TH * 16, HALFB_ALIGN = NH > 1 ? 1024 : 256,
                              HALFB = (F1 * ROWB + HALFB_ALIGN - 1) / HALFB_ALIGN * HALFB_ALIGN;
    static constexpr int BOXR = HP1 < 256 ? HP1 : 256, NB = HP1 / BOXR;                       // boxes of a tile
    // tiles of the real tensors: HP1 rows of TX pairs
    static constexpr unsigned QROW = TX * 2 * sizeof(T), QBYTES = HP1 * QROW;
    static constexpr int QSW = QROW == 32 || QROW == 64 || QROW == 128 ? (int)QROW : 0;
    static constexpr unsigned QMASK = QSW == 128 ? 0x70u : QSW == 64 ? 0x30u : QSW == 32 ? 0x10u : 0u;
    static constexpr size_t QAL = QSW ? QSW * 8 : 128;       // the swizzle's period
    // (groups of 16 lanes and more fill a half warp: any stride does)
    static constexpr int PHN = F::ph(P1 - 1) > FI::ph(P1 - 1) ? F::ph(P1 - 1) : FI::ph(P1 - 1);
    static constexpr int LS = TPL >= 16 ? (PHN + 2) / 2 * 2 : plane_ls(P1);
    static constexpr size_t LINEB = sizeof(float2) * TX * LS;
    static __host__ __device__ constexpr int fit(size_t total, int cap)
    {
        const int n = (int)(227 * 1024 / (total + 1024));
        return n < cap ? n : cap;
    }
    // address of pair x of row t1 in a tile of a real tensor
    static __device__ __forceinline__ unsigned at(int t1, int x)
    {
        const unsigned o = (unsigned)t1 * QROW + (unsigned)x * 2 * sizeof(T);
        return o ^ ((o >> 3) & QMASK);
    }
};
template <typename T, int LOG2P1, bool HAS_B> struct CtFwdGeo : CtGeo<T, LOG2P1> {
    using B = CtGeo<T, LOG2P1>;
    using Tw = PassTw<LOG2P1, false>;
    // result tile over the lines, then the input tiles
    static constexpr size_t OUTB = (size_t)B::NH * B::HALFB, LINES = 0, RAW = ((OUTB > B::LINEB ? OUTB : B::LINEB) + 1023) / 1024 * 1024,
                            TW = RAW + (HAS_B ? 2 : 1) * (size_t)B::QBYTES, BARS = TW + sizeof(float2) * Tw::TOTAL, TOTAL = BARS + 8;
    // by shared memory, and at 128 registers a thread for the long transforms, 80 for the short ones
    static constexpr int PER_SM = B::fit(TOTAL, LOG2P1 >= 9 ? 4 : 6);
};

// A CTA of four warps works on a tile of TX column pairs; the next tile's inputs travel while this one is transformed.  IN: how
// they come: 0 tensor copies, 1 asynchronous copies of 8 bytes, 2 element by element (slices that start
// off 8-byte boundaries, eight loads in flight).
// The separated bins leave as tensor copies from a swizzled tile over the lines.  262144 bf16 values, 512 rows: 383 us with two CTAs
// of eight warps per SM, 348 with four of four (4.6 TB/s); the filter's rows 184, 168.  Bound by the shared-memory pipe (75 %) and
// the barriers around the result tile.
template <typename T, int LOG2P1, bool HAS_B, int IN>
__global__ void __launch_bounds__(kCtThreads, (CtFwdGeo<T, LOG2P1, HAS_B>::PER_SM))
ct_cols_fwd_w_kernel(ColsFwdWArgs p, const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                     const __grid_constant__ CUtensorMap map_o)
{
    using G = CtFwdGeo<T, LOG2P1, HAS_B>;
    using F = typename G::F;
    constexpr int P1 = G::P1, HP1 = G::HP1, F1 = G::F1, TPL = G::TPL, TX = G::TX;
    constexpr int NF = (F1 + TPL - 1) / TPL;               // bins of a lane
    using P0 = typename F::template Pass<0>;
    static_assert(F::NP == 2, "two passes");
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    if (smem_u32(smem_dyn) & 1023u) {                      // (aligned as declared: room to align it here would cost a CTA per SM)
        if (threadIdx.x == 0 && p.status) atomicExch(p.status, 7);
        return;
    }
    unsigned char *to = smem_dyn + G::LINES, *raw = smem_dyn + G::RAW;
    float2 *twt = reinterpret_cast<float2 *>(smem_dyn + G::TW);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_dyn + G::BARS);
    const int tid = threadIdx.x, l = tid % TPL, x = tid / TPL;
    const unsigned m = F::group_mask(tid);
    float2 *line = reinterpret_cast<float2 *>(to) + x * G::LS;
    PassTw<LOG2P1, false>::build(twt, p.tw1, P1, tid, kCtThreads);
    const PassTw<LOG2P1, false> tw{twt};
    const int P2 = 1 << p.log2p2;
    const int tpc = (P2 / 2) / TX;                         // tiles per slice (P2/2 is a multiple of TX)
    const long long tiles = p.slices * tpc;
    auto ask = [&](long long t) {                          // inputs of tile t: one thread, or all of them
        const long long s = t / tpc;
        const int c0 = (int)(t % tpc) * TX;
        if constexpr (IN == 0) {
            if (tid) return;
            mbar_expect_tx(bar, (HAS_B ? 2 : 1) * G::QBYTES);
#pragma unroll
            for (int b = 0; b < G::NB; ++b) {
                tma_load_3d(raw + b * G::BOXR * G::QROW, &map_a, bar, 2 * c0, b * G::BOXR, (int)s);
                if (HAS_B) tma_load_3d(raw + G::QBYTES + b * G::BOXR * G::QROW, &map_b, bar, 2 * c0, b * G::BOXR, (int)s);
            }
        } else {
            const T *ta = (const T *)p.a + s * p.in_slice, *tb = (const T *)p.b + s * p.in_slice;
            if constexpr (IN == 1) {
                constexpr int PG = 8 / (2 * sizeof(T));    // column pairs per copy
                static_assert(HP1 * (TX / PG) % kCtThreads == 0, "whole rounds");
#pragma unroll 4
                for (int idx = tid; idx < HP1 * (TX / PG); idx += kCtThreads) {
                    const int t1 = idx / (TX / PG), xg = idx % (TX / PG) * PG;
                    const long long e0 = (long long)t1 * P2 + 2 * (c0 + xg);
                    unsigned char *d = raw + G::at(t1, xg);
                    if (e0 + 2 * PG <= p.len) {
                        cp_async_n<8>(d, ta + e0);
                        if (HAS_B) cp_async_n<8>(d + G::QBYTES, tb + e0);
                    } else {
                        for (int e = 0; e < 2 * PG; ++e) {
                            const bool ok = e0 + e < p.len;
                            if (ok) HN_G(ta + e0 + e, sizeof(T));
                            if (ok && HAS_B) HN_G(tb + e0 + e, sizeof(T));
                            reinterpret_cast<T *>(d)[e] = ok ? ta[e0 + e] : T(0.f);
                            if (HAS_B) reinterpret_cast<T *>(d + G::QBYTES)[e] = ok ? tb[e0 + e] : T(0.f);
                        }
                    }
                }
            } else {
                // neighbouring elements by neighbouring threads
                constexpr int EPR = 2 * TX, U = 8;         // elements per row of the tile
                static_assert(HP1 * EPR % (U * kCtThreads) == 0, "whole rounds");
                for (int i0 = tid; i0 < HP1 * EPR; i0 += U * kCtThreads) {
                    T va[U], vb[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int i = i0 + u * kCtThreads;
                        const long long e = (long long)(i / EPR) * P2 + 2 * c0 + i % EPR;
                        const bool ok = e < p.len;
                        if (ok) HN_G(ta + e, sizeof(T));
                        if (ok && HAS_B) HN_G(tb + e, sizeof(T));
                        va[u] = ok ? __ldg(ta + e) : T(0.f);
                        if (HAS_B) vb[u] = ok ? __ldg(tb + e) : T(0.f);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int i = i0 + u * kCtThreads;
                        unsigned char *d = raw + G::at(i / EPR, i % EPR / 2) + (i & 1) * sizeof(T);
                        *reinterpret_cast<T *>(d) = va[u];
                        if (HAS_B) *reinterpret_cast<T *>(d + G::QBYTES) = vb[u];
                    }
                }
            }
        }
    };
    if constexpr (IN == 0) {
        if (tid == 0) {
            mbar_init(bar, 1);
            fence_mbar_init();
        }
    }
    __syncthreads();
    long long t = blockIdx.x;
    if (t < tiles) ask(t);
    unsigned phase = 0;
    int failed = 0;
    for (; t < tiles; t += gridDim.x, phase ^= 1u) {
        const long long tn = t + gridDim.x, s = t / tpc;
        const int c0 = (int)(t % tpc) * TX;
        if constexpr (IN == 0) {
            if (!mbar_wait(bar, phase)) failed = 1;
        } else {
            cp_async_wait_all();
            __syncthreads();
        }
        float2 keep[P0::IPL][P0::R];
        F::template pass<0, PRUNE_IN>(l, tw,
            [&](int, int, int idx) {
                const unsigned char *d = raw + G::at(idx, x);
                float a0 = staged<T>(d, 0, 0), a1 = staged<T>(d, 0, 1);
                if (HAS_B) {
                    a0 *= staged<T>(d + G::QBYTES, 0, 0);
                    a1 *= staged<T>(d + G::QBYTES, 0, 1);
                }
                return make_float2(a0, a1);
            },
            [&](int i, int r, int, float2 v) { keep[i][r] = v; });
        if (tid == 0) tma_wait_read0();                    // the previous result tile has left the lines
        if (__syncthreads_or(failed)) break;               // and the input tile has been read
        if (tn < tiles) ask(tn);
#pragma unroll
        for (int i = 0; i < P0::IPL; ++i)
#pragma unroll
            for (int r = 0; r < P0::R; ++r) line[F::ph((l + i * TPL) * P0::R + r)] = keep[i][r];
        __syncwarp(m);
        F::template mid<1, 2>(l, m, tw, line);             // (the last pass, line to line)
        // separate the two real columns, apply W_P^(t2*f1)
        float2 A0[NF], A1[NF];
        const unsigned t2 = 2u * (unsigned)(c0 + x);
        {
            // W_P^(t2*f1) with f1 = l + i*TPL is the product of a per-lane factor W_P^(t2*l) (one
            // gathered lookup) and a per-line factor W_P^(t2*TPL*i) (the same address in all lanes)
            // The per-line factor is looked up every fourth step and advanced by W_P^(t2*TPL) in between
            // (at most three products after a table value).
            const float2 cl0 = twp_w(p.twp, t2 * (unsigned)l), cl1 = twp_w(p.twp, (t2 + 1u) * (unsigned)l);
            const float2 st0 = twp_w(p.twp, t2 * (unsigned)TPL), st1 = twp_w(p.twp, (t2 + 1u) * (unsigned)TPL);
            float2 w0 = cl0, w1 = cl1;
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const int f1 = l + i * TPL;
                if (i > 0) {
                    if (i % 4 == 0) {
                        w0 = cmul(cl0, twp_w(p.twp, t2 * (unsigned)(i * TPL)));
                        w1 = cmul(cl1, twp_w(p.twp, (t2 + 1u) * (unsigned)(i * TPL)));
                    } else {
                        w0 = cmul(w0, st0);
                        w1 = cmul(w1, st1);
                    }
                }
                if (f1 < F1) {
                    const float2 z1 = line[F::ph(f1)], z2 = line[F::ph((P1 - f1) & (P1 - 1))];
                    A0[i] = cmul(make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y)), w0);
                    A1[i] = cmul(make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x)), w1);
                }
            }
        }
        __syncthreads();                                   // every line has been read
        {
            unsigned char *th = to + (x / G::TH) * G::HALFB;
            const unsigned xi = (unsigned)(x % G::TH);
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const int f1 = l + i * TPL;
                const unsigned sw = G::ROWB == 128 ? ((unsigned)f1 & 7u) : (((unsigned)f1 >> 1) & 3u);
                if (f1 < F1) *reinterpret_cast<float4 *>(th + f1 * G::ROWB + ((xi ^ sw) << 4)) = make_float4(A0[i].x, A0[i].y, A1[i].x, A1[i].y);
            }
        }
        fence_async_smem();
        __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int hh = 0; hh < G::NH; ++hh) {
                const unsigned char *th = to + hh * G::HALFB;
#pragma unroll
                for (int b = 0; b < G::NB; ++b) tma_store_3d(&map_o, th + b * G::BOXR * G::ROWB, 4 * (c0 + hh * G::TH), b * G::BOXR, (int)s);
                float2 *last = p.out + (s * F1 + HP1) * (long long)P2 + 2 * (c0 + hh * G::TH);
                HN_G(last, G::ROWB);
                bulk_store(last, th + HP1 * G::ROWB, G::ROWB);
            }
            tma_commit();
        }
    }
    if (failed) {
        // a wait gave up: say so, then give the copy a bounded time to land before the buffers go away
        if (p.status) atomicExch(p.status, 7);
        mbar_wait(bar, phase);
    }
    if (tid == 0) tma_wait_all0();
}

// ---- filter rows: spectrum in place -----------------------------------------------------------------

struct HspecArgs {
    float2 *h;                // [rows][P2]
    long long rows;
    float scale;
    const float2 *tw2;
};

template <int LOG2P2>
__global__ void __launch_bounds__(256, 2) ct_hspec_w_kernel(HspecArgs p)
{
    using F = WF<LOG2P2, false>;
    constexpr int P2 = 1 << LOG2P2, TPL = F::TPL, G = 256 / TPL, LS = plane_ls(P2);
    extern __shared__ float2 smem[];
    float2 *twt = smem + G * LS;
    const int tid = threadIdx.x, l = tid % TPL, gid = tid / TPL;
    const unsigned m = F::group_mask(tid);
    float2 *line = smem + gid * LS;
    PassTw<LOG2P2, false>::build(twt, p.tw2, P2, tid, 256);
    __syncthreads();
    const PassTw<LOG2P2, false> tw{twt};
    for (long long r = (long long)blockIdx.x * G + gid; r < p.rows; r += (long long)gridDim.x * G) {
        float2 *row = p.h + r * P2;
        F::template run<PRUNE_NONE>(l, m, tw, line,
            [&](int, int, int idx) { HN_G(row + idx, 8); return row[idx]; },
            [&](int, int, int idx, float2 v) { HN_G(row + idx, 8); row[idx] = make_float2(v.x * p.scale, v.y * p.scale); });
        __syncwarp(m);
    }
}

// ---- core --------------------------------------------------------------------------------------------

struct CoreWArgs {
    float2 *u;                // [slices][F1][P2], in place
    const float2 *h;          // [filters][F1][P2]: spectra along t2 (scaled), or with FILT the rows they are made from
    long long slices;
    int f1n;
    long long h_mod, h_off;
    const float2 *tw2;
    TwoLevelW twp;
    // FILT only: a unit is one row of a channel's filter and the same row of the slices it serves
    int nb;                   // slices per unit
    float scale;              // 1/P, folded into the filter's spectrum
    // The slices are a range of the batch that need not be whole entries: slice s has the filter of channel (s + h_off) % h_mod, so
    // the first `channels` of them have a filter each, and slice i + j * channels that of slice i.
    __host__ __device__ long long channels() const { return slices < h_mod ? slices : h_mod; }
    __host__ __device__ long long units(int n) const       // with n slices per unit; units of no slice come last and are left out
    {
        const long long c = channels(), step = c * n, full = (slices - 1) / step, rest = slices - full * step;
        return (full * c + (rest < c ? rest : c)) * f1n;
    }
};

// Twiddles of a pass from tensor memory (they depend on the lane only): 16 columns, 8 legs, at a time.
struct TmemTw {
    unsigned addr;
    mutable float v[16];
    template <int S> __device__ __forceinline__ float2 get(int, int r, int, int) const
    {
        if (r == 1 || (r & 7) == 0) {
            TmemIO<16>::ld(v, addr + 16 * (r >> 3));
            tmem_wait_ld();
        }
        return make_float2(v[2 * (r & 7)], v[2 * (r & 7) + 1]);
    }
};

// FILT (a filter shared over the batch): a lane group transforms a row of the filter itself, parks the spectrum in its own
// lanes of tensor memory and takes the row of nb slices of its channel through it, so the filter crosses HBM once and its spectrum
// never.  In shared memory the spectra of 16 warps (8 KB each) do not fit beside their lines; in registers 64 more per thread
// leave 8 warps per SM.  262144 bf16 values, 2 x 256 rows: 167 us in a kernel of the filter's own plus 525 here, now 595.  Bound by
// instruction issue (64 % of the slots) and instruction fetch of the unrolled passes.  Three CTAs of four warps with twiddles in
// registers and rows that travel ahead as untiled copies: 662.  Filters of which no group holds all (3 x 800 rows of 262144 values in groups
// of 765, 2 x 390 of 524288 in groups of 383) are transformed once per slice; spectra made once and read here: 6517 -> 6567 us, 4894 -> 5079.
template <int LOG2P2, bool FILT>
__global__ void __launch_bounds__(256, 2) ct_core_w_kernel(CoreWArgs p)
{
    using F = WF<LOG2P2, false>;
    using FI = WF<LOG2P2, true>;
    constexpr int P2 = 1 << LOG2P2, TPL = F::TPL, NP = F::NP, G = 256 / TPL, LS = plane_ls(P2);
    using PL = typename F::LastPass;
    constexpr int NV = PL::IPL * PL::R, NC = 2 * NV;       // points of a lane, tensor-memory columns of a warp
    static_assert(NV % 16 == 0, "whole blocks of tensor memory");
    extern __shared__ float2 smem[];
    __shared__ unsigned tm_slot;
    float2 *twt = smem + G * LS;
    const int tid = threadIdx.x, l = tid % TPL, gid = tid / TPL, warp = tid >> 5;
    const unsigned m = F::group_mask(tid);
    float2 *line = smem + gid * LS;
    PassTw<LOG2P2, false>::build(twt, p.tw2, P2, tid, 256);
    PassTw<LOG2P2, true>::build(twt + P2, p.tw2, P2, tid, 256);
    // 1024 points: the twiddles of the forward passes sit in tensor memory too, beside the spectra (from shared memory they are a
    // third of that pipe's work: 621 us)
    constexpr bool TWTM = LOG2P2 == 10;
    constexpr int TCOLS = (FILT ? 2 * NC : 0) + (TWTM ? 2 * PL::R : 0), TALLOC = TCOLS > 128 ? 256 : TCOLS > 64 ? 128 : 64;
    if constexpr (TCOLS > 0) {
        if (warp == 0) tmem_alloc(smem_u32(&tm_slot), TALLOC);
        tmem_fence_before_sync();
    }
    __syncthreads();
    if constexpr (TCOLS > 0) tmem_fence_after_sync();
    const unsigned tm = FILT ? tmem_addr(tm_slot, warp, (warp >> 2) * NC) : 0u;
    const unsigned tmt = TWTM ? tmem_addr(tm_slot, warp, FILT ? 2 * NC : 0) : 0u;
    if constexpr (TWTM) {
        if (warp < 4) {
#pragma unroll
            for (int b = 0; b < PL::R / 8; ++b) {
                float v[16];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float2 w = 8 * b + e == 0 ? make_float2(1.f, 0.f) : twt[(8 * b + e - 1) * PL::NS + l];
                    v[2 * e] = w.x; v[2 * e + 1] = w.y;
                }
                TmemIO<16>::st(tmt + 16 * b, v);
            }
            tmem_wait_st();
        }
        tmem_fence_before_sync();
        __syncthreads();
        tmem_fence_after_sync();
    }
    using TwT = typename std::conditional<TWTM, TmemTw, PassTw<LOG2P2, false>>::type;
    TwT tw;
    if constexpr (TWTM) tw.addr = tmt; else tw.base = twt;
    const PassTw<LOG2P2, true> twi{twt + P2};

    // Two equal passes: the inverse is the forward transform with real and imaginary parts exchanged on both ends, so one copy of
    // the passes serves the filter's row, the forward and the inverse (three copies of 32-point butterflies are 70 KB of code,
    // and every fifth cycle of a warp waited for instructions).
    constexpr bool EQUAL = NP == 2 && F::radix(0) == F::radix(1);
    using X = float2[PL::IPL][PL::R];

    // x <- transform of x along t2; `in` fills the points of the first pass, in the order they also leave the last one
    auto forward = [&](X &x, auto in) {
        F::template pass<0, PRUNE_NONE>(l, tw, in, [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
        __syncwarp(m);
        F::template mid<1, NP - 1, PRUNE_NONE>(l, m, tw, line);
        F::template pass<NP - 1, PRUNE_NONE>(l, tw,
            [&](int, int, int idx) { return line[F::ph(idx)]; },
            [&](int i, int rr, int, float2 v) { x[i][rr] = v; });
        __syncwarp(m);
    };
    // undo the inter-pass twiddle W_P^(t2*f1), t2 = l + TPL*q: per-lane factor W_P^(f1*l) times a
    // per-row factor W_P^(f1*TPL*q) whose address is the same in all lanes
    // (the per-row factor is looked up every fourth leg and advanced by one leg's step in between)
    using PE = typename FI::LastPass;
    struct Undo { float2 cl, stp, w; };
    auto undo_init = [&](int f1) {
        Undo t;
        t.cl = twp_w(p.twp, (unsigned)f1 * (unsigned)l);
        t.stp = twp_w(p.twp, (unsigned)f1 * (unsigned)(P2 / PE::R));
        t.w = t.cl;
        return t;
    };
    auto undo_store = [&](Undo &t, float2 *row, int f1, bool on, int r, int idx, float2 v) {
        // legs of one item come in order r = 0, 1, ...: positions idx = l + i*TPL + r*(P2/R)
        if (r % 4 == 0) t.w = cmul(t.cl, twp_w(p.twp, (unsigned)f1 * (unsigned)(idx - l)));
        else t.w = cmul(t.w, t.stp);
        if (on) { HN_G(row + idx, 8); row[idx] = cmulc(v, t.w); }
    };
    // one row of u: forward along t2, product(x) for every point, back, inter-pass twiddle undone.  first: it is the filter's row,
    // whose spectrum goes to park(x) instead.
    // (rows go from global memory straight to the first pass: through the line they cost two more trips of the shared-memory pipe)
    auto row_through = [&](const float2 *src, float2 *row, int f1, bool on, bool first, auto park, auto product) {
        X x;
        if constexpr (EQUAL) {
#pragma unroll
            for (int r = 0; r < PL::R; ++r) {
                if (on) HN_G(src + l + r * TPL, 8);
                x[0][r] = on ? src[l + r * TPL] : make_float2(0.f, 0.f);
            }
#pragma unroll 1
            for (int way = 0;; ++way) {
                forward(x, [&](int i, int r, int) { return x[i][r]; });
                if (way) break;
                if (first) { park(x); return; }
                product(x);
#pragma unroll
                for (int r = 0; r < PL::R; ++r) x[0][r] = make_float2(x[0][r].y, x[0][r].x);
            }
            Undo t = undo_init(f1);
#pragma unroll
            for (int r = 0; r < PL::R; ++r) undo_store(t, row, f1, on, r, l + r * TPL, make_float2(x[0][r].y, x[0][r].x));
        } else {
            forward(x, [&](int, int, int idx) { if (on) HN_G(src + idx, 8); return on ? src[idx] : make_float2(0.f, 0.f); });
            if (first) { park(x); return; }
            product(x);
            FI::template pass<0, PRUNE_NONE>(l, twi,
                [&](int i, int rr, int) { return x[i][rr]; },
                [&](int, int, int idx, float2 v) { line[FI::ph(idx)] = v; });
            __syncwarp(m);
            FI::template mid<1, NP - 1, PRUNE_NONE>(l, m, twi, line);
            Undo t = undo_init(f1);
            FI::template pass<NP - 1, PRUNE_NONE>(l, twi,
                [&](int, int, int idx) { return line[FI::ph(idx)]; },
                [&](int, int r, int idx, float2 v) { undo_store(t, row, f1, on, r, idx, v); });
            __syncwarp(m);
        }
    };

    if constexpr (!FILT) {
        const long long rows = p.slices * p.f1n;
        for (long long r = (long long)blockIdx.x * G + gid; r < rows; r += (long long)gridDim.x * G) {
            const long long s = r / p.f1n;
            const int f1 = (int)(r % p.f1n);
            const long long hs = p.h_mod ? (s + p.h_off) % p.h_mod : s;
            const float2 *hrow = p.h + (hs * p.f1n + f1) * P2;
            row_through(p.u + r * P2, p.u + r * P2, f1, true, false, [](X &) {}, [&](X &Y) {
                // product with the precomputed filter spectrum (coalesced loads, no stores between)
#pragma unroll
                for (int i = 0; i < PL::IPL; ++i)
#pragma unroll
                    for (int rr = 0; rr < PL::R; ++rr) {
                        HN_G(hrow + F::last_pos(l, i, rr), 8);
                        Y[i][rr] = cmul(Y[i][rr], __ldg(hrow + F::last_pos(l, i, rr)));
                    }
            });
        }
    } else {
        const long long ch = p.channels(), per = ch * p.f1n, units = p.units(p.nb);
        constexpr int LPW = 32 / TPL;
        // (a warp's groups go round together: tensor memory is reached by whole warps)
        for (long long u0 = (long long)blockIdx.x * G + warp * LPW; u0 < units; u0 += (long long)gridDim.x * G) {
            const long long u = u0 + (gid - warp * LPW);
            const bool live = u < units;
            const long long s0 = live ? u / per * p.nb * ch : 0;
            const int rc = live ? (int)(u % per) : 0, i = rc / p.f1n, f1 = rc % p.f1n;
            const float2 *hrow = p.h + ((i + p.h_off) % p.h_mod * p.f1n + f1) * P2;
            float2 *const row0 = p.u + (s0 * p.f1n + rc) * P2;
            const long long left = live ? p.slices - s0 - i : -ch;
#pragma unroll 1
            for (int j = -1; j < p.nb; ++j) {
                const bool first = j < 0, on = j * ch < left;
                if (!__any_sync(0xffffffffu, on)) break;
                float2 *row = row0 + j * per * P2;
                row_through(first ? hrow : row, row, f1, on, first,
                    [&](X &H) {
                        __syncwarp();
#pragma unroll
                        for (int b = 0; b < NC / 32; ++b) {
                            float Hc[32];
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                const float2 v = H[(16 * b + e) / PL::R][(16 * b + e) % PL::R];
                                Hc[2 * e] = v.x * p.scale;
                                Hc[2 * e + 1] = v.y * p.scale;
                            }
                            TmemIO<32>::st(tm + 32 * b, Hc);
                        }
                        tmem_wait_st();
                    },
                    [&](X &Y) {
                        __syncwarp();
#pragma unroll
                        for (int b = 0; b < NC / 32; ++b) {
                            float Hc[32];
                            TmemIO<32>::ld(Hc, tm + 32 * b);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                float2 &y = Y[(16 * b + e) / PL::R][(16 * b + e) % PL::R];
                                y = cmul(y, make_float2(Hc[2 * e], Hc[2 * e + 1]));
                            }
                        }
                    });
            }
        }
    }
    if constexpr (TCOLS > 0) {
        tmem_fence_before_sync();
        __syncthreads();
        tmem_fence_after_sync();
        if (warp == 0) tmem_dealloc(tm_slot, TALLOC);
    }
}

// ---- columns, inverse ------------------------------------------------------------------------------------

struct ColsInvWArgs {
    const float2 *in;         // [slices][F1][P2]
    const void *q;
    void *y;
    long long slices;
    int len;                  // L
    int log2p2;
    const float2 *tw1;
    int *status;              // device word set when a bounded wait on a tensor copy gives up (may be NULL)
};

// Gate and store of a tile of lines (`lines`: position t1 < P1/2 of line x holds the two real outputs of columns 2x, 2x+1).
template <typename T, int LOG2P1, int TX, int LS, bool PAIR>
__device__ __forceinline__ void ct_inv_epilogue(const ColsInvWArgs &p, const float2 *lines, long long s, int c0, int P2, int tid)
{
    using FI = WF<LOG2P1, true>;
    constexpr int HP1 = (1 << LOG2P1) / 2;
    const T *pq = (const T *)p.q;
    T *py = (T *)p.y;
        const long long base = s * (long long)p.len + 2 * c0;
    // a half warp takes 8 pairs of two neighbouring rows: line stride and skew then spread its
    // 16 reads over all banks, and each row still receives whole 32-byte sectors
    constexpr int NE = HP1 * TX / kCtThreads;
    static_assert(HP1 * TX % kCtThreads == 0, "whole epilogue rounds");
    constexpr int XB = TX >= 8 ? TX / 8 : 1;
    const int x = TX < 8 ? tid % TX : (tid & 7) + 8 * ((tid >> 4) % XB);
    const int tb = TX < 8 ? tid / TX : ((tid >> 3) & 1) + 2 * ((tid >> 4) / XB);
    constexpr int TSTEP = kCtThreads / TX;
    using Q2 = typename std::conditional<sizeof(T) == 4, float2, __nv_bfloat162>::type;
    // gate values first (all requests in flight together), then products and stores
    const long long ox = base + 2 * x;
    if constexpr (!PAIR) {
        T qa[NE], qb[NE];
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int t1 = tb + e * TSTEP;
            const long long tt = (long long)t1 * P2 + 2 * (c0 + x), o = ox + (long long)t1 * P2;
            if (tt < p.len) HN_G(pq + o, sizeof(T));
            if (tt + 1 < p.len) HN_G(pq + o + 1, sizeof(T));
            qa[e] = tt < p.len ? __ldg(pq + o) : T(0.f);
            qb[e] = tt + 1 < p.len ? __ldg(pq + o + 1) : T(0.f);
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int t1 = tb + e * TSTEP;
            const long long tt = (long long)t1 * P2 + 2 * (c0 + x), o = ox + (long long)t1 * P2;
            const float2 z = lines[x * LS + FI::ph(t1)];
            if (tt < p.len) IO<T>::st(py, o, z.x * (float)qa[e]);
            if (tt + 1 < p.len) IO<T>::st(py, o + 1, z.y * (float)qb[e]);
        }
        return;
    }
    Q2 qv[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) {
        const int t1 = tb + e * TSTEP;
        const long long tt = (long long)t1 * P2 + 2 * (c0 + x);
        if (tt < p.len) HN_G(pq + ox + (long long)t1 * P2, 2 * sizeof(T));
        if (tt < p.len) qv[e] = __ldg(reinterpret_cast<const Q2 *>(pq + ox + (long long)t1 * P2));
    }
#pragma unroll
    for (int e = 0; e < NE; ++e) {
        const int t1 = tb + e * TSTEP;
        const long long tt = (long long)t1 * P2 + 2 * (c0 + x);
        if (tt < p.len) {
            const float2 z = lines[x * LS + FI::ph(t1)];
            const long long o = ox + (long long)t1 * P2;
            HN_G(py + o, 2 * sizeof(T));
            if constexpr (sizeof(T) == 4) {
                *reinterpret_cast<float2 *>(py + o) = make_float2(z.x * qv[e].x, z.y * qv[e].y);
            } else {
                *reinterpret_cast<__nv_bfloat162 *>(py + o) =
                    __floats2bfloat162_rn(z.x * __low2float(qv[e]), z.y * __high2float(qv[e]));
            }
        }
    }
}

template <typename T, int LOG2P1> struct CtInvGeo : CtGeo<T, LOG2P1> {
    using B = CtGeo<T, LOG2P1>;
    static constexpr size_t RAW = 0, Q = ((size_t)B::NH * B::HALFB + B::QAL - 1) / B::QAL * B::QAL, LINES = Q + B::QBYTES,
                            BARS = LINES + B::LINEB, TOTAL = BARS + 16;
    // by shared memory, and at 168 registers a thread for the long transforms, 96 for the short ones
    static constexpr int PER_SM = B::fit(TOTAL, LOG2P1 >= 9 ? 3 : 5);
};

// Tensor copies bring the tile of the spectra while the tile before it is transformed, and the gate tile under the last pass; the
// gated results take the gate's place and leave as a tensor copy.  QY: 0 gate and result as tensor copies, 1 pairs, 2 elements.
// Twiddles of the second pass in registers.  Bound by HBM: 262144 bf16 values, 512 rows, 456 us with 16 warps per SM that fetched
// their own tiles and waited for them, 267 with 12 warps here (6.0 TB/s).
template <typename T, int LOG2P1, int QY>
__global__ void __launch_bounds__(kCtThreads, (CtInvGeo<T, LOG2P1>::PER_SM))
ct_cols_inv_w_kernel(ColsInvWArgs p, const __grid_constant__ CUtensorMap map_u, const __grid_constant__ CUtensorMap map_q,
                     const __grid_constant__ CUtensorMap map_y)
{
    using G = CtInvGeo<T, LOG2P1>;
    using FI = typename G::FI;
    constexpr int P1 = G::P1, HP1 = G::HP1, F1 = G::F1, TPL = G::TPL, TX = G::TX;
    using P0 = typename FI::template Pass<0>;
    using PE = typename FI::LastPass;
    static_assert(FI::NP == 2, "two passes");
    using Q2 = typename std::conditional<sizeof(T) == 4, float2, __nv_bfloat162>::type;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char *base = smem_dyn;                        // (aligned as declared: room to align it here would cost a CTA per SM)
    if (smem_u32(base) & 1023u) {
        if (threadIdx.x == 0 && p.status) atomicExch(p.status, 8);
        return;
    }
    unsigned char *raw = base + G::RAW, *tq = base + G::Q;
    float2 *lines = reinterpret_cast<float2 *>(base + G::LINES);
    uint64_t *bar_u = reinterpret_cast<uint64_t *>(base + G::BARS), *bar_q = bar_u + 1;
    const int tid = threadIdx.x, l = tid % TPL, x = tid / TPL;
    const unsigned m = FI::group_mask(tid);
    float2 *line = lines + x * G::LS;
    if (tid == 0) {
        mbar_init(bar_u, 1);
        mbar_init(bar_q, 1);
        fence_mbar_init();
    }
    typename FI::template Hoist<1> tw;
    for (int t = tid; t < P1; t += kCtThreads) { HN_G(p.tw1 + t, 8); lines[t] = p.tw1[t]; }
    __syncthreads();
    tw.load(l, lines);
    __syncthreads();
    const int P2 = 1 << p.log2p2;
    const int tpc = (P2 / 2) / TX;
    const long long tiles = p.slices * tpc;
    auto issue_u = [&](long long t) {                      // one thread
        const long long s = t / tpc;
        const int c0 = (int)(t % tpc) * TX;
        mbar_expect_tx(bar_u, G::NH * F1 * G::ROWB);
#pragma unroll
        for (int hh = 0; hh < G::NH; ++hh) {
            unsigned char *d = raw + hh * G::HALFB;
#pragma unroll
            for (int b = 0; b < G::NB; ++b) tma_load_3d(d + b * G::BOXR * G::ROWB, &map_u, bar_u, 4 * (c0 + hh * G::TH), b * G::BOXR, (int)s);
            const float2 *last = p.in + (s * F1 + HP1) * (long long)P2 + 2 * (c0 + hh * G::TH);
            HN_G(last, G::ROWB);
            bulk_load(d + HP1 * G::ROWB, last, G::ROWB, bar_u);
        }
    };
    auto gate_boxes = [&](long long t, auto f) {
        const long long s = t / tpc;
        const int c0 = (int)(t % tpc) * TX;
#pragma unroll
        for (int b = 0; b < G::NB; ++b) f(tq + b * G::BOXR * G::QROW, 2 * c0, b * G::BOXR, (int)s);
    };
    long long t = blockIdx.x;
    if (tid == 0 && t < tiles) {
        issue_u(t);
        if constexpr (QY == 0) gate_boxes(t, [&](void *, int cx, int cy, int cz) { tma_prefetch_3d(&map_q, cx, cy, cz); });
    }
    // pair x of a tile row: its 16-byte chunk, XORed with address bits 7 and up, which the engine's strides (multiples of 8 rows)
    // leave alone, so it depends on the lane only; upwards for bins below P1/2, downwards for the mirrored ones
    const int xi = x % G::TH;
    const unsigned char *rx = raw + (x / G::TH) * G::HALFB;
    auto chunk = [&](int row) {
        const unsigned sw = G::ROWB == 128 ? ((unsigned)row & 7u) : (((unsigned)row >> 1) & 3u);
        return *reinterpret_cast<const float4 *>(rx + (size_t)row * G::ROWB + (((unsigned)xi ^ sw) << 4));
    };
    unsigned phase = 0;
    int failed = 0;
    for (; t < tiles; t += gridDim.x, phase ^= 1u) {
        const long long tn = t + gridDim.x, s = t / tpc;
        const int c0 = (int)(t % tpc) * TX;
        if (!mbar_wait(bar_u, phase)) failed = 1;
        // legs below half the first-pass radix read bins <= P1/2 directly, the others the mirrored bin
        // conjugated: known per leg at compile time, except where a leg starts at bin P1/2 itself
        constexpr int RH = P0::R / 2;
        FI::template pass<0, PRUNE_NONE>(l, tw,
            [&](int, int r, int idx) {
                if (r < RH) {
                    const float4 ab = chunk(idx);
                    return make_float2(ab.x - ab.w, ab.y + ab.z);
                }
                const float4 ab = chunk(P1 - idx);
                const float sg = (r == RH && idx == HP1) ? 1.f : -1.f;
                return make_float2(fmaf(-sg, ab.w, ab.x), fmaf(sg, ab.y, ab.z));
            },
            [&](int, int, int idx, float2 v) { line[FI::ph(idx)] = v; });
        if (__syncthreads_or(failed)) break;               // the tile buffer is free again
        if (tid == 0) {
            if (tn < tiles) issue_u(tn);
            if constexpr (QY == 0) {
                tma_wait_read0();                          // the results before these have left the gate's buffer
                mbar_expect_tx(bar_q, G::QBYTES);
                gate_boxes(t, [&](void *d, int cx, int cy, int cz) { tma_load_3d(d, &map_q, bar_q, cx, cy, cz); });
                if (tn < tiles) gate_boxes(tn, [&](void *, int cx, int cy, int cz) { tma_prefetch_3d(&map_q, cx, cy, cz); });
            }
        }
        // at t1 < P1/2 the two real outputs of columns 2x, 2x+1
        float2 z[PE::IPL][PE::R / 2];
        FI::template pass<1, PRUNE_OUT>(l, tw, [&](int, int, int idx) { return line[FI::ph(idx)]; },
                                        [&](int i, int r, int, float2 v) { z[i][r] = v; });
        __syncwarp(m);
        if constexpr (QY == 0) {
            if (!mbar_wait(bar_q, phase)) failed = 2;
#pragma unroll
            for (int i = 0; i < PE::IPL; ++i)
#pragma unroll
                for (int r = 0; r < PE::R / 2; ++r) {
                    Q2 *g = reinterpret_cast<Q2 *>(tq + G::at(l + i * TPL + r * (P1 / PE::R), x));
                    const Q2 qv = *g;
                    if constexpr (sizeof(T) == 4) *g = make_float2(z[i][r].x * qv.x, z[i][r].y * qv.y);
                    else *g = __floats2bfloat162_rn(z[i][r].x * __low2float(qv), z[i][r].y * __high2float(qv));
                }
            fence_async_smem();
            if (__syncthreads_or(failed)) break;
            if (tid == 0) {
                gate_boxes(t, [&](void *d, int cx, int cy, int cz) { tma_store_3d(&map_y, d, cx, cy, cz); });
                tma_commit();
            }
        } else {
#pragma unroll
            for (int i = 0; i < PE::IPL; ++i)
#pragma unroll
                for (int r = 0; r < PE::R / 2; ++r) line[FI::ph(l + i * TPL + r * (P1 / PE::R))] = z[i][r];
            __syncthreads();
            ct_inv_epilogue<T, LOG2P1, TX, G::LS, QY == 1>(p, lines, s, c0, P2, tid);
            __syncthreads();                               // the lines are free again
        }
    }
    if (failed) {
        // a wait gave up: say so, then give copies that may still be in flight a bounded time to land
        if (p.status) atomicExch(p.status, 8);
        mbar_wait(bar_u, phase);
        if (QY == 0 && failed == 2) mbar_wait(bar_q, phase);
        if (t + gridDim.x < tiles && failed == 2) mbar_wait(bar_u, phase ^ 1u);
    }
    if (tid == 0) tma_wait_all0();
}

// ---- launchers ----------------------------------------------------------------------------------------------

static int ctw_sms()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 148;
    }
    return n;
}

bool ct1d_w_supported(int log2p1, int log2p2)
{
    return log2p1 >= 7 && log2p1 <= 10 && log2p2 >= 7 && log2p2 <= 10 && tma_available();
}

// spectra [slice][P1/2+1][P2] complex, as fp32
template <class G> static bool spectra_map(CUtensorMap *m, const float2 *base, int P2, long long slices)
{
    const unsigned long long dims[3] = {2ull * P2, (unsigned long long)G::F1, (unsigned long long)slices};
    const unsigned long long strides[2] = {(unsigned long long)P2 * 8, (unsigned long long)G::F1 * P2 * 8};
    const unsigned box[3] = {G::TH * 4, G::BOXR, 1};
    return tma_encode_3d_cached(m, base, false, dims, strides, box, (int)G::ROWB);
}

// Whether the maps of a plan's workspace can be had.  They are made anew in each call, for the slices it works on; the address,
// strides and box are these.
bool ct1d_w_maps(const Ct1dPlan *c)
{
    if (!ct1d_w_supported(c->log2p1, c->log2p2)) return false;
    const int P2 = 1 << c->log2p2;
    alignas(64) CUtensorMap m;
    bool ok = false;
#define CALLM(L) ok = spectra_map<CtGeo<float, L>>(&m, c->wu, P2, c->slices_per_chunk) && spectra_map<CtGeo<float, L>>(&m, c->wh, P2, c->wh_slices)
    switch (c->log2p1) { case 7: CALLM(7); break; case 8: CALLM(8); break; case 9: CALLM(9); break; case 10: CALLM(10); break; }
#undef CALLM
    return ok;
}

// A tensor whose slices are whole numbers of rows of P2 elements, so that [slice][row][P2] is an exact view of it and rows past the
// data read as zeros; false where tensor copies do not apply.
template <class G, typename T> static bool rows_map(CUtensorMap *m, const void *base, int len, long long slice_elems, int P2, long long slices)
{
    if (len % P2 != 0 || G::QROW % 16 != 0) return false;
    const unsigned long long dims[3] = {(unsigned long long)P2, (unsigned long long)(len / P2), (unsigned long long)slices};
    const unsigned long long strides[2] = {(unsigned long long)P2 * sizeof(T), (unsigned long long)slice_elems * sizeof(T)};
    const unsigned box[3] = {2 * G::TX, G::BOXR, 1};
    return tma_encode_3d_cached(m, base, sizeof(T) == 2, dims, strides, box, G::QSW);
}

template <typename T, int LOG2P1, bool HAS_B, int IN>
static void launch_cols_fwd_w_in(const ColsFwdWArgs &a, const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &mo, long long pairs,
                                 cudaStream_t st)
{
    using G = CtFwdGeo<T, LOG2P1, HAS_B>;
    static DevOnce attr;
    if (attr.first())
        cudaFuncSetAttribute(ct_cols_fwd_w_kernel<T, LOG2P1, HAS_B, IN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::TOTAL);
    const long long tiles = pairs / G::TX, res = (long long)G::PER_SM * ctw_sms();
    ct_cols_fwd_w_kernel<T, LOG2P1, HAS_B, IN><<<(int)(tiles < res ? tiles : res), kCtThreads, G::TOTAL, st>>>(a, ma, mb, mo);
}

template <typename T, int LOG2P1, bool HAS_B> static int launch_cols_fwd_w_b(const ColsFwdWArgs &a, cudaStream_t st)
{
    using G = CtFwdGeo<T, LOG2P1, HAS_B>;
    const int P2 = 1 << a.log2p2;
    const long long pairs = a.slices * (P2 / 2);
    if (pairs <= 0) return 0;
    alignas(64) CUtensorMap ma, mb, mo;
    memset(&ma, 0, sizeof(ma));
    memset(&mb, 0, sizeof(mb));
    if (a.slices >= (1ll << 31) || !spectra_map<G>(&mo, a.out, P2, a.slices)) return -1;
    const bool vec = a.in_slice * sizeof(T) % 8 == 0 && (((uintptr_t)a.a | (uintptr_t)a.b) & 7) == 0;
    if (rows_map<G, T>(&ma, a.a, a.len, a.in_slice, P2, a.slices) && (!HAS_B || rows_map<G, T>(&mb, a.b, a.len, a.in_slice, P2, a.slices)))
        launch_cols_fwd_w_in<T, LOG2P1, HAS_B, 0>(a, ma, mb, mo, pairs, st);
    else if (vec) launch_cols_fwd_w_in<T, LOG2P1, HAS_B, 1>(a, ma, mb, mo, pairs, st);
    else launch_cols_fwd_w_in<T, LOG2P1, HAS_B, 2>(a, ma, mb, mo, pairs, st);
    return 1;
}

template <typename T, int LOG2P1> static int launch_cols_fwd_w_t(const ColsFwdWArgs &a, cudaStream_t st)
{
    return a.b ? launch_cols_fwd_w_b<T, LOG2P1, true>(a, st) : launch_cols_fwd_w_b<T, LOG2P1, false>(a, st);
}

template <typename T, int LOG2P1, int QY>
static void launch_cols_inv_w_qy(const ColsInvWArgs &a, const CUtensorMap &mu, const CUtensorMap &mq, const CUtensorMap &my, long long pairs,
                                 cudaStream_t st)
{
    using G = CtInvGeo<T, LOG2P1>;
    static DevOnce attr;
    if (attr.first())
        cudaFuncSetAttribute(ct_cols_inv_w_kernel<T, LOG2P1, QY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::TOTAL);
    const long long tiles = pairs / G::TX, res = (long long)G::PER_SM * ctw_sms();
    ct_cols_inv_w_kernel<T, LOG2P1, QY><<<(int)(tiles < res ? tiles : res), kCtThreads, G::TOTAL, st>>>(a, mu, mq, my);
}

template <typename T, int LOG2P1> static int launch_cols_inv_w_t(const ColsInvWArgs &a, cudaStream_t st)
{
    using G = CtInvGeo<T, LOG2P1>;
    const bool pair = a.len % 2 == 0 && (((uintptr_t)a.q | (uintptr_t)a.y) & (2 * sizeof(T) - 1)) == 0;
    const int P2 = 1 << a.log2p2;
    const long long pairs = a.slices * (P2 / 2);
    if (pairs <= 0) return 0;
    alignas(64) CUtensorMap mu, mq, my;
    memset(&mq, 0, sizeof(mq));
    memset(&my, 0, sizeof(my));
    if (a.slices >= (1ll << 31) || !spectra_map<G>(&mu, a.in, P2, a.slices)) return -1;
    if (rows_map<G, T>(&mq, a.q, a.len, a.len, P2, a.slices) && rows_map<G, T>(&my, a.y, a.len, a.len, P2, a.slices))
        launch_cols_inv_w_qy<T, LOG2P1, 0>(a, mu, mq, my, pairs, st);
    else if (pair) launch_cols_inv_w_qy<T, LOG2P1, 1>(a, mu, mq, my, pairs, st);
    else launch_cols_inv_w_qy<T, LOG2P1, 2>(a, mu, mq, my, pairs, st);
    return 1;
}

template <int LOG2P2> static int launch_rows_w_t(const HspecArgs *hs, const CoreWArgs *co, cudaStream_t st)
{
    using F = WF<LOG2P2, false>;
    constexpr int P2 = 1 << LOG2P2, G = 256 / F::TPL, LS = plane_ls(P2);
    const size_t sm = sizeof(float2) * ((size_t)G * LS + 2 * P2);
    static DevOnce attr;
    if (attr.first()) {
        cudaFuncSetAttribute(ct_hspec_w_kernel<LOG2P2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        cudaFuncSetAttribute(ct_core_w_kernel<LOG2P2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        cudaFuncSetAttribute(ct_core_w_kernel<LOG2P2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    }
    const long long slots = (long long)ctw_sms() * 2 * G;
    long long units = hs ? hs->rows : co->slices * co->f1n;
    CoreWArgs c{};
    if (co) c = *co;
    if (co && c.scale != 0.f) {
        // the count of slices per unit with the least work in the busiest slot: a transform for the filter, two per slice
        const long long most = (c.slices + c.channels() - 1) / c.channels();
        long long best = -1;
        for (int nb = 1; nb <= most && nb <= 64; ++nb) {
            const long long un = c.units(nb), cost = ((un + slots - 1) / slots) * (1 + 2 * nb);
            if (best < 0 || cost < best) { best = cost; c.nb = nb; units = un; }
        }
    }
    const long long want = (units + G - 1) / G;
    const int grid = (int)(want < (long long)ctw_sms() * 2 ? want : (long long)ctw_sms() * 2);
    if (grid <= 0) return 0;
    if (hs) ct_hspec_w_kernel<LOG2P2><<<grid, 256, sm, st>>>(*hs);
    else if (c.scale != 0.f) ct_core_w_kernel<LOG2P2, true><<<grid, 256, sm, st>>>(c);
    else ct_core_w_kernel<LOG2P2, false><<<grid, 256, sm, st>>>(c);
    return 1;
}

#define HN_SWITCH_CTW(x, CALL)                                                                  \
    switch (x) {                                                                                \
    case 7: CALL(7); break; case 8: CALL(8); break; case 9: CALL(9); break; case 10: CALL(10); break; \
    default: return -1;                                                                         \
    }

static int launch_rows_w(int log2p2, const HspecArgs *hs, const CoreWArgs *co, cudaStream_t st)
{
    int n = 0;
#define CALLR(L) n = launch_rows_w_t<L>(hs, co, st)
    HN_SWITCH_CTW(log2p2, CALLR)
#undef CALLR
    return n;
}

int ct1d_w_filter(Ct1dPlan *c, const void *h, long long n, bool shared, bool staged_ok, cudaStream_t st, int *launches, Prof *prof,
                  int (*fallback)(Ct1dPlan *, const char *, long long, cudaStream_t, int *, Prof *))
{
    const TwoLevelW twp{c->twp_coarse, c->twp_fine, c->lo};
    if (staged_ok) {
        ColsFwdWArgs a{};
        a.a = h; a.b = nullptr; a.out = c->wh; a.slices = n; a.in_slice = c->K; a.len = c->K; a.status = c->status;
        a.log2p2 = c->log2p2; a.tw1 = c->tw1; a.twp = twp;
        prof->begin(KID_CT_COLS_H, st);
        int r = 0;
#define CALLF(L) r = launch_cols_fwd_w_t<float, L>(a, st)
#define CALLB(L) r = launch_cols_fwd_w_t<bf16, L>(a, st)
        if (c->dt_h == 0) { HN_SWITCH_CTW(c->log2p1, CALLF) } else { HN_SWITCH_CTW(c->log2p1, CALLB) }
#undef CALLF
#undef CALLB
        prof->end(st);
        if (r < 0) return -1;
        *launches += r;
    } else if (fallback(c, (const char *)h, n, st, launches, prof)) {
        return -1;
    }
    if (shared) return 0;                                  // the core transforms the rows of a shared filter itself
    HspecArgs hs{};
    hs.h = c->wh; hs.rows = n * ((1 << c->log2p1) / 2 + 1); hs.scale = (float)ldexp(1.0, -c->log2p); hs.tw2 = c->tw2;
    prof->begin(KID_CT_HSPEC, st);
    int r = launch_rows_w(c->log2p2, &hs, nullptr, st);
    prof->end(st);
    if (r < 0) return -1;
    *launches += r;
    return 0;
}

int ct1d_w_body(Ct1dPlan *c, const void *q, const void *k, const void *v, long long n, bool shared, long long s0,
                void *y, cudaStream_t st, int *launches, Prof *prof)
{
    const TwoLevelW twp{c->twp_coarse, c->twp_fine, c->lo};
    ColsFwdWArgs a{};
    a.a = k; a.b = v; a.out = c->wu; a.slices = n; a.in_slice = c->L; a.len = c->L; a.status = c->status;
    a.log2p2 = c->log2p2; a.tw1 = c->tw1; a.twp = twp;
    prof->begin(KID_CT_COLS_U, st);
    int r = 0;
#define CALLF(L) r = launch_cols_fwd_w_t<float, L>(a, st)
#define CALLB(L) r = launch_cols_fwd_w_t<bf16, L>(a, st)
    if (c->dt_in == 0) { HN_SWITCH_CTW(c->log2p1, CALLF) } else { HN_SWITCH_CTW(c->log2p1, CALLB) }
#undef CALLF
#undef CALLB
    prof->end(st);
    if (r < 0) return -1;
    *launches += r;
    CoreWArgs co{};
    co.u = c->wu; co.h = c->wh; co.slices = n; co.f1n = (1 << c->log2p1) / 2 + 1;
    co.h_mod = shared ? c->C : 0; co.h_off = shared ? s0 % c->C : 0;
    co.scale = shared ? (float)ldexp(1.0, -c->log2p) : 0.f;
    co.tw2 = c->tw2; co.twp = twp;
    prof->begin(KID_CT_CORE, st);
    r = launch_rows_w(c->log2p2, nullptr, &co, st);
    prof->end(st);
    if (r < 0) return -1;
    *launches += r;
    ColsInvWArgs ci{};
    ci.in = c->wu; ci.q = q; ci.y = y; ci.slices = n; ci.len = c->L; ci.log2p2 = c->log2p2; ci.tw1 = c->tw1; ci.status = c->status;
    prof->begin(KID_CT_COLS_INV, st);
#define CALLF(L) r = launch_cols_inv_w_t<float, L>(ci, st)
#define CALLB(L) r = launch_cols_inv_w_t<bf16, L>(ci, st)
    if (c->dt_out == 0) { HN_SWITCH_CTW(c->log2p1, CALLF) } else { HN_SWITCH_CTW(c->log2p1, CALLB) }
#undef CALLF
#undef CALLB
    prof->end(st);
    if (r < 0) return -1;
    *launches += r;
    return 0;
}

}  // namespace hn
