// Spectral core of the backward pass along a strided axis: with H, U, G the transforms of a bin's filter line, k*v line and
// dy*q line,
//
//     U H       -> back, cropped  (dq's convolution)
//     G conj H  -> back, cropped  (the kernel at the opposite displacement: du)
//     G conj U  -> back, every displacement (dh)
//
// in place of three cores that transformed nine lines between them where six do, each reading its two operands again.
// Tiles (8 or 16 adjacent bins by all rows) travel as tensor copies as in core_tma.cu.  A group of lanes owns one bin: its
// column of a tile is nobody else's, so spectra that do not fit in registers wait in the column they came from and the
// results leave from there.  A CTA keeps one tile at a time; the other CTAs of the SM work while one waits for its copies.
// Issue slots 50 %, shared-memory pipe 54 % busy with ten warps per SM (192 points): latency of six transforms per bin, one after
// the other, against three tiles in and three out.  12 volumes of 96^3: 806 us at
// 256 points (a training step 3483 -> 2583 us), 468 at 192 points, where the copies alone need 209.
#include <cuda.h>
#include <cstdint>
#include "common.cuh"
#include "plane_util.cuh"
#include "core3_tma.cuh"
#include "tma_util.cuh"

namespace hn {

template <int LOG2P, bool FULL> struct Core3Geo {
    using F = WF<LOG2P, false>;
    static constexpr int N = len_of(LOG2P), HALF = N / 2;
    static constexpr int THREADS = N >= 768 ? 256 : N == 192 ? 64 : 128;     // (192: 468 us with 64 threads, 498 with 128, 12 volumes of 96^3)
    static constexpr int PER_SM = N >= 768 ? 1 : N == 192 ? 5 : N % 3 == 0 ? 2 : LOG2P == 9 ? (FULL ? 1 : 2) : LOG2P == 6 || (LOG2P == 8 && !FULL) ? 4 : 3;
    static constexpr int TX = THREADS / F::TPL;
    static constexpr unsigned ROWB = TX * 8;
    static_assert(ROWB == 128 || ROWB == 64, "tile rows match a swizzle span");
    static constexpr int BOXR = HALF <= 256 ? HALF : HALF / 2;       // rows per box
    static constexpr int NB = HALF / BOXR;                           // boxes per half line
    static constexpr unsigned BOXB = BOXR * ROWB, HALFB = HALF * ROWB;
    static constexpr unsigned UB = FULL ? 2 * HALFB : HALFB;         // k*v and dy*q tiles
    static constexpr int NBU = FULL ? 2 * NB : NB;
    static constexpr int PHN = F::ph(N - 1) > WF<LOG2P, true>::ph(N - 1) ? F::ph(N - 1) : WF<LOG2P, true>::ph(N - 1);
    static constexpr int LS = F::TPL <= 16 ? plane_ls(N) : ((PHN + 1 + 15) / 16 * 16 + 2);
    static_assert(PHN < LS, "a skewed line fits");
    static constexpr int TWTAB = N + PlaneTw<LOG2P, false>::TABLE + PlaneTw<LOG2P, true>::TABLE;
    static constexpr size_t TH = 0, TU = TH + 2 * HALFB, TG = TU + UB, LINES = TG + UB;
    static constexpr size_t TW = LINES + sizeof(float2) * TX * LS;
    static constexpr size_t BARS = TW + sizeof(float2) * TWTAB;
    static constexpr size_t TOTAL = BARS + sizeof(uint64_t) + 1024;  // + room to align the start
    static_assert(PER_SM * (TOTAL + 1024) <= 228 * 1024, "resident CTAs");
};

struct Core3Params {
    long long n_outer;
    int tiles_per_outer, h_shift, K;
    long long h_mod, h_off;
    float scale;
    const float2 *gtw;
    int gtw_n;
    int *status;
};

template <int LOG2P, bool FULL>
__global__ void __launch_bounds__(Core3Geo<LOG2P, FULL>::THREADS, Core3Geo<LOG2P, FULL>::PER_SM)
axis_core3_tma_kernel(const __grid_constant__ CUtensorMap map_u, const __grid_constant__ CUtensorMap map_g,
                      const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_dh, Core3Params p)
{
    using G = Core3Geo<LOG2P, FULL>;
    using F = WF<LOG2P, false>;
    using FI = WF<LOG2P, true>;
    constexpr int N = G::N, TPL = F::TPL, NP = F::NP, NT = G::THREADS;
    static_assert(NP == 2, "two passes");
    constexpr bool EQUAL = F::radix(0) == F::radix(1);               // one register set of twiddles serves both directions
    using P0 = typename F::template Pass<0>;
    using PL = typename F::template Pass<NP - 1>;                    // last forward pass == first inverse pass
    using PE = typename FI::template Pass<NP - 1>;
    constexpr int RF2 = (int)G::ROWB / 8;
    static_assert(TPL % 8 == 0 && (N / P0::R) % 8 == 0 && (N / PL::R) % 8 == 0 && (N / PE::R) % 8 == 0, "legs keep the swizzle");
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    // the swizzle pattern is a function of the shared-memory address: start on a 1024-byte boundary
    unsigned char *smem_raw = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
    unsigned char *th = smem_raw + G::TH, *tu = smem_raw + G::TU, *tg = smem_raw + G::TG;
    float2 *twt = reinterpret_cast<float2 *>(smem_raw + G::TW);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + G::BARS);
    // lanes: as in core_tma.cu (two 16-lane lines of a warp interleaved in blocks of 8 lanes)
    const int tid = threadIdx.x;
    const int l = TPL == 16 ? ((tid & 7) | ((tid >> 1) & 8)) : tid % TPL;
    const int gid = TPL == 16 ? ((tid >> 5) * 2 + ((tid >> 3) & 1)) : tid / TPL;
    const unsigned m = TPL == 16 ? (0x00ff00ffu << (tid & 8)) : F::group_mask(tid);
    float2 *line = reinterpret_cast<float2 *>(smem_raw + G::LINES) + gid * G::LS;
    for (int t = tid; t < N; t += NT) { HN_G(p.gtw + t * (p.gtw_n / N), 8); twt[t] = p.gtw[t * (p.gtw_n / N)]; }
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    PlaneTw<LOG2P, false> tw;
    tw.init(l, twt, twt + N, tid, NT);
    PlaneTw<LOG2P, true> twi_own;
    if constexpr (!EQUAL) twi_own.init(l, twt, twt + N + PlaneTw<LOG2P, false>::TABLE, tid, NT);
    __syncthreads();
    const auto &twi = [&]() -> const auto & { if constexpr (EQUAL) return tw; else return twi_own; }();
    // row z of this group's bin inside a swizzled tile; multiples of 8 rows add to it
    constexpr unsigned ZSH = G::ROWB == 128 ? 0 : 1, ZMASK = G::ROWB == 128 ? 7u : 3u;
    auto row_off = [&](unsigned z) {
        return z * G::ROWB + ((((unsigned)gid >> 1) ^ ((z >> ZSH) & ZMASK)) << 4) + ((unsigned)gid & 1u) * 8u;
    };
    const unsigned off = row_off((unsigned)l);
    float2 *ch = reinterpret_cast<float2 *>(th + off), *cu = reinterpret_cast<float2 *>(tu + off), *cg = reinterpret_cast<float2 *>(tg + off);
    const long long tiles = p.n_outer * p.tiles_per_outer;
    auto issue = [&](long long t) {                    // one thread
        const long long o = t / p.tiles_per_outer;
        const int x = (int)(t % p.tiles_per_outer) * G::TX * 2;          // in floats
        const long long oh = p.h_mod ? (o + p.h_off) % p.h_mod : o;
        mbar_expect_tx(bar, 2 * G::HALFB + 2 * G::UB);
#pragma unroll
        for (int b = 0; b < G::NB; ++b) {
            // positions [0, N/2) hold filter rows from h_shift on, positions [N/2, N) the rows before it (periodic: all in order)
            tma_load_3d(th + b * G::BOXB, &map_h, bar, x, p.h_shift + b * G::BOXR, (int)oh);
            tma_load_3d(th + G::HALFB + b * G::BOXB, &map_h, bar, x, (FULL ? G::HALF : p.h_shift - G::HALF) + b * G::BOXR, (int)oh);
        }
#pragma unroll
        for (int b = 0; b < G::NBU; ++b) {
            tma_load_3d(tu + b * G::BOXB, &map_u, bar, x, b * G::BOXR, (int)o);
            tma_load_3d(tg + b * G::BOXB, &map_g, bar, x, b * G::BOXR, (int)o);
        }
    };
    pdl_join();
    if (tid == 0 && (long long)blockIdx.x < tiles) issue(blockIdx.x);
    unsigned phase = 0;
    int failed = 0;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x, phase ^= 1u) {
        if (!mbar_wait(bar, phase)) failed = 4;
        constexpr int PRU = FULL ? PRUNE_NONE : PRUNE_IN;
        float2 U[PL::IPL][PL::R], W[PL::IPL][PL::R];
        // filter spectrum: back into the column (a lane's own points)
        F::template pass<0, PRUNE_NONE>(l, tw, [&](int i, int r, int) { return ch[(i * TPL + r * (N / P0::R)) * RF2]; },
            [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
        __syncwarp(m);
        F::template pass<NP - 1, PRUNE_NONE>(l, tw, [&](int, int, int idx) { return line[F::ph(idx)]; },
            [&](int i, int r, int, float2 v) { ch[(i * TPL + r * (N / PL::R)) * RF2] = v; });
        __syncwarp(m);
        F::template pass<0, PRU>(l, tw, [&](int i, int r, int) { return cu[(i * TPL + r * (N / P0::R)) * RF2]; },
            [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
        __syncwarp(m);
        F::template pass<NP - 1, PRUNE_NONE>(l, tw, [&](int, int, int idx) { return line[F::ph(idx)]; },
            [&](int i, int r, int, float2 v) { U[i][r] = make_float2(v.x * p.scale, v.y * p.scale); });
        __syncwarp(m);
        F::template pass<0, PRU>(l, tw, [&](int i, int r, int) { return cg[(i * TPL + r * (N / P0::R)) * RF2]; },
            [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
        __syncwarp(m);
        F::template pass<NP - 1, PRUNE_NONE>(l, tw, [&](int, int, int idx) { return line[F::ph(idx)]; },
            [&](int i, int r, int, float2 v) {
                float2 *hp = ch + (i * TPL + r * (N / PL::R)) * RF2;
                const float2 h = *hp, u = U[i][r];
                *hp = cmulc(v, u);
                U[i][r] = cmul(u, h);
                W[i][r] = cmulc(make_float2(v.x * p.scale, v.y * p.scale), h);
            });
        __syncwarp(m);
        FI::template pass<0, PRUNE_NONE>(l, twi, [&](int i, int r, int) { return U[i][r]; },
            [&](int, int, int idx, float2 v) { line[FI::ph(idx)] = v; });
        __syncwarp(m);
        FI::template pass<NP - 1, FULL ? PRUNE_NONE : PRUNE_OUT>(l, twi, [&](int, int, int idx) { return line[FI::ph(idx)]; },
            [&](int i, int r, int, float2 v) { cu[(i * TPL + r * (N / PE::R)) * RF2] = v; });
        __syncwarp(m);
        FI::template pass<0, PRUNE_NONE>(l, twi, [&](int i, int r, int) { return W[i][r]; },
            [&](int, int, int idx, float2 v) { line[FI::ph(idx)] = v; });
        __syncwarp(m);
        FI::template pass<NP - 1, FULL ? PRUNE_NONE : PRUNE_OUT>(l, twi, [&](int, int, int idx) { return line[FI::ph(idx)]; },
            [&](int i, int r, int, float2 v) { cg[(i * TPL + r * (N / PE::R)) * RF2] = v; });
        __syncwarp(m);
        FI::template pass<0, PRUNE_NONE>(l, twi, [&](int i, int r, int) { return ch[(i * TPL + r * (N / PL::R)) * RF2]; },
            [&](int, int, int idx, float2 v) { line[FI::ph(idx)] = v; });
        __syncwarp(m);
        // position d mod N is tap row (d + h_shift) mod N: the taps leave in their own order (a store may not start at a
        // negative row)
        FI::template pass<NP - 1, PRUNE_NONE>(l, twi, [&](int, int, int idx) { return line[FI::ph(idx)]; },
            [&](int i, int r, int idx, float2 v) {
                if constexpr (FULL) ch[(i * TPL + r * (N / PE::R)) * RF2] = v;
                else *reinterpret_cast<float2 *>(th + row_off((unsigned)ring<N>(idx + p.h_shift))) = v;
            });
        fence_async_smem();                            // generic-proxy writes visible to the copy engine
        if (__syncthreads_or(failed)) break;
        if (tid == 0) {
            const long long o = t / p.tiles_per_outer;
            const int x = (int)(t % p.tiles_per_outer) * G::TX * 2;
#pragma unroll
            for (int b = 0; b < G::NBU; ++b) {
                tma_store_3d(&map_u, tu + b * G::BOXB, x, b * G::BOXR, (int)o);
                tma_store_3d(&map_g, tg + b * G::BOXB, x, b * G::BOXR, (int)o);
            }
#pragma unroll
            for (int b = 0; b < 2 * G::NB; ++b)
                if (b * G::BOXR < p.K) tma_store_3d(&map_dh, th + b * G::BOXB, x, b * G::BOXR, (int)o);
            tma_commit();
            if (t + gridDim.x < tiles) {
                tma_wait_read0();
                issue(t + gridDim.x);
            }
        }
    }
    if (failed) {
        // a wait gave up: say so, then give copies that may still be in flight a bounded time to land
        atomicExch(p.status, failed);
        mbar_wait(bar, phase);
    }
    if (tid == 0) tma_wait_all0();
}

// ---- host side -------------------------------------------------------------------------------------------

#define HN_CORE3_CASES(X) X(6, false) X(7, false) X(8, false) X(9, false) X(10, false) X(kLen192, false) X(kLen384, false) X(kLen768, false) X(6, true) X(7, true) X(8, true) X(9, true)

bool core3_tma_supported(int log2p, int full, int nc)
{
    const bool len = (log2p >= 6 && log2p <= (full ? 9 : 10)) || (log2p >= kLen192 && log2p <= kLen768 && !full);
    return len && nc % 2 == 0 && tma_available();
}

static bool map_lines(unsigned char *map, const float2 *base, long long outer, int rows, int nc, long long outer_elems, int tx, int box_rows)
{
    const unsigned long long dims[3] = {2ull * nc, (unsigned long long)rows, (unsigned long long)outer};
    const unsigned long long strides[2] = {(unsigned long long)nc * 8, (unsigned long long)outer_elems * 8};
    const unsigned box[3] = {(unsigned)tx * 2, (unsigned)box_rows, 1};
    return tma_encode_3d(reinterpret_cast<CUtensorMap *>(map), base, /*bf16=*/false, dims, strides, box, tx * 8);
}

bool core3_tma_make(Core3Maps *m, const Core3Args &a, long long max_outer, long long h_count)
{
    static_assert(sizeof(m->u) >= sizeof(CUtensorMap), "room for a tensor map");
    m->valid = false;
    if (!core3_tma_supported(a.log2p, a.full, a.nc) || max_outer >= (1ll << 31) || h_count >= (1ll << 31)) return false;
    int tx = 0, br = 0;
#define HN_CORE3_GEO(L, FU) if (a.log2p == L && (a.full != 0) == FU) { tx = Core3Geo<L, FU>::TX; br = Core3Geo<L, FU>::BOXR; }
    HN_CORE3_CASES(HN_CORE3_GEO)
#undef HN_CORE3_GEO
    m->valid = map_lines(m->u, a.u, max_outer, a.L, a.nc, a.u_outer, tx, br) && map_lines(m->g, a.g, max_outer, a.L, a.nc, a.u_outer, tx, br) &&
               map_lines(m->h, a.h, h_count, a.K, a.nc, a.h_outer, tx, br) && map_lines(m->dh, a.dh, max_outer, a.K, a.nc, a.h_outer, tx, br);
    return m->valid;
}

template <int LOG2P, bool FULL> static int launch_core3_t(Core3Params p, const Core3Maps &m, int nc, cudaStream_t st)
{
    using G = Core3Geo<LOG2P, FULL>;
    p.tiles_per_outer = (nc + G::TX - 1) / G::TX;
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 148;
    }
    static DevOnce attr;
    if (attr.first()) cudaFuncSetAttribute(axis_core3_tma_kernel<LOG2P, FULL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::TOTAL);
    const long long tiles = p.n_outer * p.tiles_per_outer, res = (long long)sms * G::PER_SM;
    const int grid = (int)(tiles < res ? tiles : res);
    if (grid <= 0) return 0;
    auto map = [](const unsigned char *b) -> const CUtensorMap & { return *reinterpret_cast<const CUtensorMap *>(b); };
    launch_pdl(axis_core3_tma_kernel<LOG2P, FULL>, grid, G::THREADS, G::TOTAL, st, map(m.u), map(m.g), map(m.h), map(m.dh), p);
    return 1;
}

int launch_core3_tma(const Core3Args &a, const Core3Maps &m, int *status, cudaStream_t st)
{
    if (!m.valid) return -1;
    Core3Params p{};
    p.n_outer = a.n_outer; p.h_shift = a.h_shift; p.K = a.K; p.h_mod = a.h_mod; p.h_off = a.h_off; p.scale = a.scale;
    p.gtw = a.gtw; p.gtw_n = a.gtw_n; p.status = status;
#define HN_CORE3_LAUNCH(L, FU) if (a.log2p == L && (a.full != 0) == FU) return launch_core3_t<L, FU>(p, m, a.nc, st);
    HN_CORE3_CASES(HN_CORE3_LAUNCH)
#undef HN_CORE3_LAUNCH
    return -1;
}

}  // namespace hn
