// Fused spectral core along a strided axis for 64- to 1024-point lines, tiles moved by TMA.
//
// Same arithmetic as core_w.cu (forward transform of the filter lines, forward transform of the
// k*v lines, spectral product of Eq. 12 of the paper, inverse, cropped half written back in
// place), but the tiles -- 8 or 16 adjacent bins by all rows of the axis -- travel as tensor copies:
//
//   cp.async.bulk.tensor loads   filter tile (boxes of up to 256 rows; the wrapped placement of the
//                                taps is two row ranges) and k*v tile (one box; rows past the data
//                                and bins past the end come back as zeros)
//   cp.async.bulk.tensor store   the cropped result tile
//
// One elected thread issues them; nobody computes addresses or waits per element.  The boxes land
// row-major (one 64-byte row per axis position; the code also covers 128-byte rows) with the matching swizzle, which
// spreads the rows a group of lanes reads at once over the banks.  A tile buffer is free again as soon as the first pass
// has read it, so the next tile's copy runs under the rest of this tile's arithmetic.
//
// Every wait on a copy is bounded: if a barrier does not complete, the CTA records it in the
// status word, waits (bounded again) for what is still in flight and returns.
#include <cuda.h>
#include <cstdint>
#include "common.cuh"
#include "plane_util.cuh"
#include "core_tma.cuh"
#include "tma_util.cuh"

namespace hn {

// Threads per CTA: 128, several CTAs per SM (a CTA synchronises at two barriers per tile; more, smaller CTAs keep the
// schedulers busy while one of them waits), but one CTA of 256 threads for 1024-point lines.
// FULL (periodic axis: N rows in, N rows out) at 512 points: the result tile takes the k*v tile's buffer, which keeps two
// CTAs per SM; the next k*v tile is then asked for after the result has left, under the next filter tile's transforms.
template <int LOG2P, bool FULL> struct TmaCta {
    static constexpr int THREADS = len_of(LOG2P) >= 768 ? 256 : 128;
    // (512 points: 95 us with cp.async copies, 67 here, for 104x175x178; periodic 512x512 grids 1347 -> 1273.  192 and 384 points
    // share the buffer too: three CTAs per SM instead of two.)
    static constexpr int PER_SM = len_of(LOG2P) >= 768 ? 1 : LOG2P == kLen192 || LOG2P == kLen384 ? 3 : LOG2P == 9 ? 2 : FULL && LOG2P >= 7 ? 3 : 4;
    static constexpr bool SHARE = (FULL && LOG2P >= 9) || LOG2P == kLen192 || LOG2P == kLen384;
};

// Geometry of a tile for LOG2P-point lines: one line per group of TPL lanes, so TX = THREADS / TPL bins
// per tile and TX * 8 bytes per tile row (64 or 128: the swizzle span of the tensor maps).  A box holds at
// most 256 rows.
template <int LOG2P, bool FULL> struct TmaGeo {
    using F = WF<LOG2P, false>;
    static constexpr int N = len_of(LOG2P), HALF = N / 2;
    using CTA = TmaCta<LOG2P, FULL>;
    static constexpr int THREADS = CTA::THREADS;
    static constexpr int TX = THREADS / F::TPL;
    static constexpr unsigned ROWB = TX * 8;
    static constexpr int BOXR = HALF <= 256 ? HALF : HALF / 2;       // rows per box
    static constexpr int NB = HALF / BOXR;                           // boxes per half line
    static constexpr unsigned BOXB = BOXR * ROWB;
    static constexpr unsigned HALFB = HALF * ROWB;
    static constexpr unsigned UB = FULL ? 2 * HALFB : HALFB;         // k*v tile and result tile
    static constexpr int NBU = FULL ? 2 * NB : NB;                   // their boxes
    // 8- and 16-lane groups (several lines per warp): a half warp works on two lines (see the kernel), whose
    // strides are therefore 8 mod 16 entries, i.e. half a bank row apart
    static constexpr int PHN = F::ph(N - 1) > WF<LOG2P, true>::ph(N - 1) ? F::ph(N - 1) : WF<LOG2P, true>::ph(N - 1);
    static constexpr int LS = F::TPL <= 16 ? plane_ls(N) : ((PHN + 1 + 15) / 16 * 16 + 2);
    static_assert(PHN < LS, "a skewed line fits");
    static_assert(ROWB == 128 || ROWB == 64, "tile rows match a swizzle span");
    static constexpr int TWTAB = N + PlaneTw<LOG2P, false>::TABLE + PlaneTw<LOG2P, true>::TABLE;
    // shared memory: tile buffers first (1024-byte aligned, as the swizzle pattern repeats every 1024 bytes)
    static constexpr size_t TH = 0;                                  // filter tile, N rows
    static constexpr size_t TU = TH + 2 * HALFB;                     // k*v tile
    static constexpr size_t TO = CTA::SHARE ? TU : TU + UB;          // result tile
    static constexpr size_t LINES = TO + UB;                         // one skewed line per group
    static constexpr size_t TW = LINES + sizeof(float2) * TX * LS;
    static constexpr size_t BARS = TW + sizeof(float2) * TWTAB;
    static constexpr size_t TOTAL = BARS + 2 * sizeof(uint64_t) + 1024;    // + room to align the start
    static_assert(CTA::PER_SM * (TOTAL + 1024) <= 228 * 1024, "resident CTAs");
};

struct CoreTmaParams {
    long long n_outer;
    int tiles_per_outer;      // ceil(nc / TX)
    int h_shift;              // filter row (pos + h_shift) mod N sits at position pos
    long long h_mod, h_off;   // filter outer index = h_mod ? (o + h_off) % h_mod : o
    float scale;
    float scale_im;           // scale, or -scale where the product takes the conjugate of the filter spectrum
    const float2 *gtw;
    int gtw_n;
    int *status;              // device word: 0 ok, else which wait gave up
};

template <int LOG2P, bool FULL>
__global__ void __launch_bounds__(TmaCta<LOG2P, FULL>::THREADS, TmaCta<LOG2P, FULL>::PER_SM)
axis_core_tma_kernel(const __grid_constant__ CUtensorMap map_u, const __grid_constant__ CUtensorMap map_h, CoreTmaParams p)
{
    using G = TmaGeo<LOG2P, FULL>;
    using F = WF<LOG2P, false>;
    using FI = WF<LOG2P, true>;
    constexpr int N = G::N, TPL = F::TPL, NP = F::NP, kTmaThreads = G::THREADS;
    // two equal passes: the twiddles depend on the lane only and live in registers; the inverse uses the same values
    // conjugated, so one set serves both directions
    constexpr bool EQUAL = NP == 2 && F::radix(0) == F::radix(1);
    static_assert(NP == 2, "two passes");
    using PL = typename F::template Pass<NP - 1>;
    using P0 = typename F::template Pass<0>;
    using PE = typename FI::template Pass<NP - 1>;
    // float2 between a lane's first point and leg r of item i in a tile: multiples of 8 rows, which the swizzle repeats after
    constexpr int RF2 = (int)G::ROWB / 8;
    static_assert(TPL % 8 == 0 && (N / P0::R) % 8 == 0 && (N / PE::R) % 8 == 0, "legs keep the swizzle");
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    // the swizzle pattern is a function of the shared-memory address: start on a 1024-byte boundary
    unsigned char *smem_raw = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
    unsigned char *th = smem_raw + G::TH;
    unsigned char *tu = smem_raw + G::TU;
    unsigned char *to = smem_raw + G::TO;
    float2 *lines = reinterpret_cast<float2 *>(smem_raw + G::LINES);
    float2 *twt = reinterpret_cast<float2 *>(smem_raw + G::TW);
    uint64_t *bar_h = reinterpret_cast<uint64_t *>(smem_raw + G::BARS);
    uint64_t *bar_u = bar_h + 1;
    // Lanes of a warp: with one line per warp (32 lanes per line) lane = position.  With two lines per warp the
    // two are interleaved in blocks of 8 lanes (lanes 0-7 and 16-23 work on the first line, 8-15 and 24-31 on the
    // second): an 8-byte shared-memory access is served per half warp, and a half warp then reads 8 rows of BOTH
    // bins of a 16-byte tile chunk, 16 distinct 8-byte slots, instead of 16 rows of one bin, which share 8 slots.
    const int tid = threadIdx.x;
    const int l = TPL == 16 ? ((tid & 7) | ((tid >> 1) & 8)) : tid % TPL;
    const int gid = TPL == 16 ? ((tid >> 5) * 2 + ((tid >> 3) & 1)) : tid / TPL;
    const unsigned m = TPL == 16 ? (0x00ff00ffu << (tid & 8)) : F::group_mask(tid);
    float2 *line = lines + gid * G::LS;
    for (int t = tid; t < N; t += kTmaThreads) { HN_G(p.gtw + t * (p.gtw_n / N), 8); twt[t] = p.gtw[t * (p.gtw_n / N)]; }
    if (tid == 0) {
        mbar_init(bar_h, 1);
        mbar_init(bar_u, 1);
        fence_mbar_init();
    }
    __syncthreads();
    PlaneTw<LOG2P, false> tw;
    tw.init(l, twt, twt + N, tid, kTmaThreads);
    PlaneTw<LOG2P, true> twi_own;
    if constexpr (!EQUAL) {
        twi_own.init(l, twt, twt + N + PlaneTw<LOG2P, false>::TABLE, tid, kTmaThreads);
        __syncthreads();
    }
    const auto &twi = [&]() -> const auto & { if constexpr (EQUAL) return tw; else return twi_own; }();
    // Row z = l + TPL*r of bin `gid` inside a swizzled tile.  A row is ROWB bytes; the 16-byte chunk index
    // of an address is XORed with address bits 7 and up (3 bits for the 128-byte swizzle, 2 for the 64-byte
    // one), i.e. with a function of z that TPL*r does not change: every leg r is the same per-lane offset
    // plus a constant.
    constexpr unsigned ZSH = G::ROWB == 128 ? 0 : 1, ZMASK = G::ROWB == 128 ? 7u : 3u;
    const unsigned tile_off = (unsigned)l * G::ROWB
                            + ((((unsigned)gid >> 1) ^ (((unsigned)l >> ZSH) & ZMASK)) << 4) + ((unsigned)gid & 1u) * 8u;
    const long long tiles = p.n_outer * p.tiles_per_outer;
    auto issue_h = [&](long long t) {                  // one thread
        const long long o = t / p.tiles_per_outer;
        const int x = (int)(t % p.tiles_per_outer) * G::TX * 2;          // in floats
        const long long oh = p.h_mod ? (o + p.h_off) % p.h_mod : o;
        mbar_expect_tx(bar_h, 2 * G::HALFB);
#pragma unroll
        for (int b = 0; b < G::NB; ++b) {
            // positions [0, N/2) hold filter rows from h_shift on, positions [N/2, N) the rows before it (periodic: all in order)
            tma_load_3d(th + b * G::BOXB, &map_h, bar_h, x, p.h_shift + b * G::BOXR, (int)oh);
            tma_load_3d(th + G::HALFB + b * G::BOXB, &map_h, bar_h, x, (FULL ? G::HALF : p.h_shift - G::HALF) + b * G::BOXR, (int)oh);
        }
    };
    auto issue_u = [&](long long t) {
        const long long o = t / p.tiles_per_outer;
        const int x = (int)(t % p.tiles_per_outer) * G::TX * 2;
        mbar_expect_tx(bar_u, G::UB);
#pragma unroll
        for (int b = 0; b < G::NBU; ++b) tma_load_3d(tu + b * G::BOXB, &map_u, bar_u, x, b * G::BOXR, (int)o);
    };
    auto store_tile = [&](long long t) {               // one thread
        const long long o = t / p.tiles_per_outer;
        const int x = (int)(t % p.tiles_per_outer) * G::TX * 2;
#pragma unroll
        for (int b = 0; b < G::NBU; ++b) tma_store_3d(&map_u, to + b * G::BOXB, x, b * G::BOXR, (int)o);
        tma_commit();
    };
    long long t = blockIdx.x, tprev = 0;
    bool have_prev = false;
    pdl_join();
    if (tid == 0 && t < tiles) { issue_h(t); issue_u(t); }
    unsigned phase = 0;
    int failed = 0;
    for (; t < tiles; t += gridDim.x, phase ^= 1u) {
        const long long tn = t + gridDim.x;
        float2 H[PL::IPL][PL::R];
        // ---- filter lines: tile -> registers ------------------------------------------------------
        if (!mbar_wait(bar_h, phase)) failed = 1;
        {
            const float2 *src = reinterpret_cast<const float2 *>(th + tile_off);
            F::template pass<0, PRUNE_NONE>(l, tw,
                [&](int i, int r, int) { return src[(i * TPL + r * (N / P0::R)) * RF2]; },
                [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
        }
        if (__syncthreads_or(failed)) break;           // the filter tile buffer is free again; the previous result tile is complete
        if (tid == 0) {
            if (have_prev) store_tile(tprev);          // (its writers fenced before this barrier)
            if (tn < tiles) issue_h(tn);
        }
        F::template pass<NP - 1, PRUNE_NONE>(l, tw,
            [&](int, int, int idx) { return line[F::ph(idx)]; },
            [&](int i, int r, int, float2 v) { H[i][r] = make_float2(v.x * p.scale, v.y * p.scale_im); });
        __syncwarp(m);
        if constexpr (G::CTA::SHARE) {
            // the previous result tile has left the buffer it shares with the k*v tile
            if (tid == 0 && have_prev) { tma_wait_read0(); issue_u(t); }
        }
        // ---- k*v lines: tile -> spectrum, product, inverse ----------------------------------------
        if (!mbar_wait(bar_u, phase)) failed = 2;
        {
            const float2 *src = reinterpret_cast<const float2 *>(tu + tile_off);
            F::template pass<0, FULL ? PRUNE_NONE : PRUNE_IN>(l, tw,
                [&](int i, int r, int) { return src[(i * TPL + r * (N / P0::R)) * RF2]; },
                [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
        }
        if (!G::CTA::SHARE && tid == 0) tma_wait_read0();      // the previous result tile has left its buffer
        if (__syncthreads_or(failed)) break;           // the k*v tile buffer is free again
        if (!G::CTA::SHARE && tid == 0 && tn < tiles) issue_u(tn);
        float2 Y[PL::IPL][PL::R];
        F::template pass<NP - 1, PRUNE_NONE>(l, tw,
            [&](int, int, int idx) { return line[F::ph(idx)]; },
            [&](int i, int r, int, float2 v) { Y[i][r] = cmul(v, H[i][r]); });
        __syncwarp(m);
        FI::template pass<0, PRUNE_NONE>(l, twi,
            [&](int i, int r, int) { return Y[i][r]; },
            [&](int, int, int idx, float2 v) { line[FI::ph(idx)] = v; });
        __syncwarp(m);
        {
            float2 *dst = reinterpret_cast<float2 *>(to + tile_off);
            FI::template pass<NP - 1, FULL ? PRUNE_NONE : PRUNE_OUT>(l, twi,
                [&](int, int, int idx) { return line[FI::ph(idx)]; },
                [&](int i, int r, int, float2 v) { dst[(i * TPL + r * (N / PE::R)) * RF2] = v; });
        }
        __syncwarp(m);
        fence_async_smem();                            // generic-proxy writes visible to the copy engine
        // the tile is sent after the next barrier every thread passes (the first one of the next tile, or the
        // one after the loop): no barrier of its own
        tprev = t;
        have_prev = true;
    }
    if (t >= tiles) {
        __syncthreads();
        if (tid == 0 && have_prev) store_tile(tprev);
    }
    if (t < tiles) {
        // a wait gave up: say so, then give copies that may still be in flight a bounded time to land
        if (failed) atomicExch(p.status, failed);
        mbar_wait(bar_h, phase);
        mbar_wait(bar_u, phase);
    }
    if (tid == 0) tma_wait_all0();
}

// ---- host side -------------------------------------------------------------------------------------------

// [outer][rows][nc] complex fp32, seen as fp32 with 2*nc entries per row; box = one tile row of 2*TX floats
// by up to 256 rows, swizzled over the row's 64 or 128 bytes
static bool make_map(CUtensorMap *map, const float2 *base, long long outer, int rows, int nc, long long outer_stride_elems,
                     int tx, int box_rows)
{
    const unsigned long long dims[3] = {2ull * nc, (unsigned long long)rows, (unsigned long long)outer};
    const unsigned long long strides[2] = {(unsigned long long)nc * 8, (unsigned long long)outer_stride_elems * 8};
    const unsigned box[3] = {(unsigned)tx * 2, (unsigned)box_rows, 1};
    return tma_encode_3d(map, base, /*bf16=*/false, dims, strides, box, tx * 8);
}

bool core_tma_supported(const AxisArgs &a)
{
    if (!((a.log2p >= 6 && a.log2p <= 10) || (a.log2p >= kLen192 && a.log2p <= kLen768 && !a.full))) return false;
    const int n = len_of(a.log2p);
    const bool rows = a.full ? a.n_in == n && a.h_n_in == n && a.h_shift == 0 && a.log2p <= 9
                             : a.n_in >= 1 && a.n_in <= n / 2 && a.h_n_in >= 1 && a.h_n_in <= n;
    return rows && a.in == a.out && a.in_outer == a.out_outer && a.n_in == a.n_out && a.shift == 0 && a.h_shift >= 0 && a.h_shift < n &&
           (a.nc % 2) == 0 && a.n_outer < (1ll << 31) && tma_available();
}

#define HN_TMA_CASES(X) X(6) X(7) X(8) X(9) X(10) X(kLen192) X(kLen384) X(kLen768)

bool core_tma_make(CoreTmaMaps *m, const AxisArgs &a, long long max_outer, long long h_outer_count)
{
    m->valid = false;
    if (!core_tma_supported(a)) return false;
    static_assert(sizeof(m->u) >= sizeof(CUtensorMap) && sizeof(m->h) >= sizeof(CUtensorMap), "room for a tensor map");
    int tx = 0, br = 0;                                    // (tile width and box height do not depend on FULL)
#define HN_TMA_GEO(L) if (a.log2p == L) { tx = TmaGeo<L, false>::TX; br = TmaGeo<L, false>::BOXR; }
    HN_TMA_CASES(HN_TMA_GEO)
#undef HN_TMA_GEO
    if (!make_map(reinterpret_cast<CUtensorMap *>(m->u), a.in, max_outer, a.n_in, a.nc, a.in_outer, tx, br)) return false;
    if (!make_map(reinterpret_cast<CUtensorMap *>(m->h), a.h, h_outer_count, a.h_n_in, a.nc, a.h_outer, tx, br)) return false;
    m->in = a.in; m->h_base = a.h; m->nc = a.nc; m->n_in = a.n_in; m->h_n_in = a.h_n_in; m->log2p = a.log2p;
    m->in_outer = a.in_outer; m->h_outer = a.h_outer; m->max_outer = max_outer; m->h_outer_count = h_outer_count;
    m->valid = true;
    return true;
}

template <int LOG2P, bool FULL> static int launch_core_tma_t(const CoreTmaParams &p0, const CoreTmaMaps &m, int nc, cudaStream_t st)
{
    using G = TmaGeo<LOG2P, FULL>;
    CoreTmaParams p = p0;
    p.tiles_per_outer = (nc + G::TX - 1) / G::TX;
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 148;
    }
    static DevOnce attr;
    if (attr.first())
        cudaFuncSetAttribute(axis_core_tma_kernel<LOG2P, FULL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::TOTAL);
    const long long tiles = p.n_outer * p.tiles_per_outer;
    const long long res = (long long)sms * G::CTA::PER_SM;           // resident CTAs
    const int grid = (int)(tiles < res ? tiles : res);
    if (grid <= 0) return 0;
    launch_pdl(axis_core_tma_kernel<LOG2P, FULL>, grid, G::THREADS, G::TOTAL, st,
        *reinterpret_cast<const CUtensorMap *>(m.u), *reinterpret_cast<const CUtensorMap *>(m.h), p);
    return 1;
}

int launch_core_tma(const AxisArgs &a, const CoreTmaMaps &m, int *status, cudaStream_t st)
{
    // the maps describe fixed buffers: refuse anything else
    if (!m.valid || a.log2p != m.log2p || a.in != m.in || a.h != m.h_base || a.nc != m.nc || a.n_in != m.n_in ||
        a.h_n_in != m.h_n_in || a.in_outer != m.in_outer || a.h_outer != m.h_outer || a.n_outer > m.max_outer ||
        !core_tma_supported(a))
        return -1;
    const long long h_need = a.h_mod ? a.h_mod : a.n_outer;
    if (h_need > m.h_outer_count) return -1;
    CoreTmaParams p{};
    p.n_outer = a.n_outer;
    p.h_shift = a.h_shift; p.h_mod = a.h_mod; p.h_off = a.h_off;
    p.scale = a.scale; p.scale_im = a.h_conj ? -a.scale : a.scale; p.gtw = a.gtw; p.gtw_n = a.gtw_n; p.status = status;
    switch (a.log2p) {
    case 6: return a.full ? launch_core_tma_t<6, true>(p, m, a.nc, st) : launch_core_tma_t<6, false>(p, m, a.nc, st);
    case 7: return a.full ? launch_core_tma_t<7, true>(p, m, a.nc, st) : launch_core_tma_t<7, false>(p, m, a.nc, st);
    case 8: return a.full ? launch_core_tma_t<8, true>(p, m, a.nc, st) : launch_core_tma_t<8, false>(p, m, a.nc, st);
    case 9: return a.full ? launch_core_tma_t<9, true>(p, m, a.nc, st) : launch_core_tma_t<9, false>(p, m, a.nc, st);
    case kLen192: return launch_core_tma_t<kLen192, false>(p, m, a.nc, st);
    case kLen384: return launch_core_tma_t<kLen384, false>(p, m, a.nc, st);
    case kLen768: return launch_core_tma_t<kLen768, false>(p, m, a.nc, st);
    default: return launch_core_tma_t<10, false>(p, m, a.nc, st);
    }
}

}  // namespace hn
