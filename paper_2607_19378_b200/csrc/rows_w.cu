// Contiguous-axis passes of the N-D path, warp-engine version (padded row length 64..1024, 192, 384, 768).
//
//   rows_fwd_w   one group of lanes per pair of rows: the rows are fetched with 16-byte
//                asynchronous copies into the group's line, gated (k*v) and zero-padded on the
//                fly, transformed as one complex row (real part / imaginary part), separated
//                with the Hermitian symmetry and stored as P/2+1 bins per row.
//   rows_inv_w   the inverse: two half spectra are merged into one complex row, transformed
//                back keeping the cropped half, multiplied by q and stored.
#include "common.cuh"
#include "plane_util.cuh"
#include "tma_util.cuh"

namespace hn {

constexpr int kRowThreads = 256;

// One lane asks for n bytes from src on, inside the tensor [lo, hi): the 16-byte granules around them that lie wholly inside, byte b of
// src at dst + (src & 15) + b.  Every lane that calls counts as one arrival.
__device__ __forceinline__ void ask_row(unsigned char *dst, const unsigned char *src, int n, const unsigned char *lo, const unsigned char *hi,
                                        uint64_t *bar)
{
    const unsigned long long s = (unsigned long long)src, a = s & ~15ull, l0 = ((unsigned long long)lo + 15ull) & ~15ull,
                             h0 = (unsigned long long)hi & ~15ull;
    unsigned long long from = a > l0 ? a : l0, to = (s + n + 15ull) & ~15ull;
    to = to < h0 ? to : h0;
    const unsigned bytes = n > 0 && to > from ? (unsigned)(to - from) : 0u;
    mbar_expect_tx(bar, bytes);
    if (bytes) {
        HN_G((const void *)from, bytes);
        bulk_load(dst + (from - a), (const void *)from, bytes, bar);
    }
}
// What ask_row leaves out: elements of the row in the tensor's first and last granules where those are cut.
template <typename T, int TPL>
__device__ __forceinline__ void ragged_row(unsigned char *dst, const unsigned char *src, int n, const unsigned char *lo, const unsigned char *hi, int l)
{
    const unsigned long long s = (unsigned long long)src, l0 = ((unsigned long long)lo + 15ull) & ~15ull, h0 = (unsigned long long)hi & ~15ull;
    unsigned char *d = dst + (s & 15ull);
    auto copy = [&](int from, int to) {
        for (int b = from + l * (int)sizeof(T); b < to; b += TPL * (int)sizeof(T)) {
            HN_G(src + b, sizeof(T));
            *reinterpret_cast<T *>(d + b) = *reinterpret_cast<const T *>(src + b);
        }
    };
    if (s < l0) copy(0, (long long)(l0 - s) < n ? (int)(l0 - s) : n);
    if (s + n > h0) copy(h0 > s ? (int)(h0 - s) : 0, n);
}

// MODE 0: k*v rows (upper half zero), 1: filter rows with wrapped placement, 2: causal filter rows,
// 3: circular mode, rows of exactly P elements (k*v when b is given, else the filter): power-of-two, aligned rows
// that are read straight from global memory (no staging of misaligned odd-length rows is needed)
// One lane asks the memory system to bring [lo, hi) of an array into L2, trimmed inwards to 16-byte granules.
__device__ __forceinline__ void prefetch_rows_l2(const unsigned char *lo, const unsigned char *hi)
{
    const unsigned long long a0 = ((unsigned long long)lo + 15ull) & ~15ull, a1 = (unsigned long long)hi & ~15ull;
    if (a1 > a0) HN_G((const void *)a0, a1 - a0);
    if (a1 > a0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(a0), "r"((unsigned)(a1 - a0)) : "memory");
}

// LATE: the twiddles a lane keeps in registers are read after the wait for the preceding kernel instead of before it.  The
// compiler sinks such reads to where they are used when registers run out, but not past the wait: at 1024 points (32 x 32, 62
// registers of twiddles, 128 in all) reading them early costs spills in every row pair (fp32, bytes of spill loads per thread:
// staged k v rows 200 -> 256, rows back 136 -> 184; a forward of 512 x 512 grids 2654 -> 2701 us, late 2656).  Grids of fewer CTAs than SMs
// start while their predecessor runs and gain more from early reads: one 500 x 500 grid 38.0 us late, 33.7 early.
// AHEAD: a group's next rows travel by untiled copies into a buffer of its own while it works on the present ones; CTAs of four
// warps, three per SM, with the twiddles of the second pass in registers.  Else the rows arrive in the group's line and the group
// waits for them: CTAs of eight warps, two per SM.  Where which is taken: ahead_rows below.
template <typename T, int LOG2P, int MODE> constexpr bool kAheadRows = MODE != 3 && (LOG2P == 10 || (LOG2P == 9 && sizeof(T) == 4 && MODE == 1));
template <typename T, int LOG2P, int MODE, bool AHEAD> struct RowFwdGeo {
    using F = WF<LOG2P, false>;
    static constexpr int P = len_of(LOG2P), HP = P / 2, TPL = F::TPL;
    static constexpr int THREADS = AHEAD ? 128 : kRowThreads, PER_SM = AHEAD ? 3 : 2;
    static constexpr int G = THREADS / TPL, LS = plane_ls(P);
    static constexpr int NT = MODE == 0 ? 2 : 1;                                // tensors per row
    static constexpr int ROWMAX = (MODE == 1 ? P - 1 : HP) * (int)sizeof(T);    // longest row in bytes
    static constexpr int SLOT = (ROWMAX + 15) / 16 * 16 + 16;
    static constexpr size_t TW = sizeof(float2) * G * LS, ROWS = TW + (AHEAD ? 0 : sizeof(float2) * 2 * P),
                            BARS = ROWS + (AHEAD ? (size_t)G * 2 * NT * SLOT : 0), TOTAL = BARS + (AHEAD ? 8 * G : 0);
    static_assert(PER_SM * (TOTAL + 1024) <= 228 * 1024, "resident CTAs");
    static_assert(AHEAD || MODE == 3 || 2 * NT * SLOT <= LS * 8, "staged rows must fit the line");
    static_assert(G * LS >= P, "the lines hold the twiddle table at first");
};

template <typename T, int LOG2P, int MODE, bool LATE, bool AHEAD>
__global__ void __launch_bounds__(RowFwdGeo<T, LOG2P, MODE, AHEAD>::THREADS, RowFwdGeo<T, LOG2P, MODE, AHEAD>::PER_SM) rows_fwd_w_kernel(RowsArgs p)
{
    using GE = RowFwdGeo<T, LOG2P, MODE, AHEAD>;
    using F = typename GE::F;
    constexpr int P = GE::P, HP = GE::HP, TPL = GE::TPL, G = GE::G, LS = GE::LS, THREADS = GE::THREADS;
    constexpr int PR = (MODE == 1 || MODE == 3) ? PRUNE_NONE : PRUNE_IN;
    constexpr int NT = GE::NT, ROWMAX = GE::ROWMAX, SLOT = GE::SLOT;
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    float2 *lines = reinterpret_cast<float2 *>(smem_dyn), *twt = AHEAD ? lines : reinterpret_cast<float2 *>(smem_dyn + GE::TW);
    const int tid = threadIdx.x, l = tid % TPL, gid = tid / TPL;
    const unsigned m = F::group_mask(tid);
    float2 *line = lines + gid * LS;
    unsigned char *s = AHEAD ? smem_dyn + GE::ROWS + gid * 2 * NT * SLOT : reinterpret_cast<unsigned char *>(line);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_dyn + GE::BARS) + gid;
    if (AHEAD && l == 0) {
        mbar_init(bar, 2 * NT);
        fence_mbar_init();
    }
    if (p.gtw_fresh) pdl_wait();
    for (int t = tid; t < P; t += THREADS) { HN_G(p.gtw + t * (p.gtw_n / P), 8); twt[t] = p.gtw[t * (p.gtw_n / P)]; }
    __syncthreads();
    typename std::conditional<AHEAD, typename F::template Hoist<F::NP - 1>, PlaneTw<LOG2P, false>>::type tw;
    if constexpr (LATE) pdl_join();
    if constexpr (AHEAD) tw.load(l, twt); else tw.init(l, twt, twt + P, tid, THREADS);
    __syncthreads();
    if constexpr (!LATE) pdl_join();
    const unsigned char *ab = (const unsigned char *)p.a, *bb = (const unsigned char *)p.b;
    const unsigned char *ahi = ab + p.rows * (long long)p.len * sizeof(T);
    const unsigned char *bhi = bb + p.rows * (long long)p.len * sizeof(T);
    const long long pairs = (p.rows + 1) / 2;
    auto after = [&](long long rp) { return rp + (long long)gridDim.x * G; };      // (a step held in registers costs 8 bytes of spills)
    const int rowb = p.len * (int)sizeof(T);
    // lane j < 2 NT fetches row j of the pair: a0, a1, b0, b1
    auto ask = [&](long long rp) {
        if (l >= 2 * NT || rp >= pairs) return;
        const long long r = 2 * rp + (l & 1);
        const unsigned char *lo = l < 2 ? ab : bb;
        ask_row(s + l * SLOT, lo + r * rowb, r < p.rows ? rowb : 0, lo, l < 2 ? ahi : bhi, bar);
    };
    // the transform of a pair of rows, into the line
    auto transform = [&](long long rp, auto in) {
        if constexpr (AHEAD) {
            F::template pass<0, PR>(l, tw, in, [&](int, int, int idx, float2 v) { line[F::ph(idx)] = v; });
            fence_async_smem();                            // (blanked and ragged elements, before the copies that follow)
            __syncwarp(m);
            ask(after(rp));
            F::template mid<1, F::NP>(l, m, tw, line);
        } else {
            F::template run_to_line<PR, MODE != 3>(l, m, tw, line, in);
        }
    };
    unsigned phase = 0;
    int failed = 0;
    long long rp = (long long)blockIdx.x * G + gid;
    if constexpr (AHEAD) ask(rp);
    for (; rp < pairs; rp = after(rp), phase ^= 1u) {
        const long long r0 = 2 * rp, r1 = r0 + 1;
        const bool has1 = r1 < p.rows;
        if constexpr (MODE == 3) {
            const T *a0 = (const T *)p.a + r0 * P, *a1 = (const T *)p.a + (has1 ? r1 : r0) * P;
            const T *b0 = (const T *)p.b + r0 * P, *b1 = (const T *)p.b + (has1 ? r1 : r0) * P;
            const bool gated = p.b != nullptr;
            const float keep1 = has1 ? 1.f : 0.f;
            transform(rp, [&](int, int, int idx) {
                float a = IO<T>::ld(a0, idx), b = IO<T>::ld(a1, idx) * keep1;
                if (gated) { a *= IO<T>::ld(b0, idx); b *= IO<T>::ld(b1, idx); }
                return make_float2(a, b);
            });
        } else {
            const unsigned char *g0 = ab + r0 * rowb, *g1 = ab + r1 * rowb, *h0 = bb + r0 * rowb, *h1 = bb + r1 * rowb;
            if constexpr (AHEAD) {
                if (!mbar_wait(bar, phase)) failed = 1;
                if (__any_sync(m, failed)) break;
                ragged_row<T, TPL>(s, g0, rowb, ab, ahi, l);
                if (has1) ragged_row<T, TPL>(s + SLOT, g1, rowb, ab, ahi, l);
                if constexpr (MODE == 0) {
                    ragged_row<T, TPL>(s + 2 * SLOT, h0, rowb, bb, bhi, l);
                    if (has1) ragged_row<T, TPL>(s + 3 * SLOT, h1, rowb, bb, bhi, l);
                }
            } else {
                stage_row_u<TPL, ROWMAX>(s, g0, rowb, ab, ahi, l);
                if (has1) stage_row_u<TPL, ROWMAX>(s + SLOT, g1, rowb, ab, ahi, l);
                if (MODE == 0) {
                    stage_row_u<TPL, ROWMAX>(s + 2 * SLOT, h0, rowb, bb, bhi, l);
                    if (has1) stage_row_u<TPL, ROWMAX>(s + 3 * SLOT, h1, rowb, bb, bhi, l);
                }
                if (MODE != 1 && l == 0) {
                    // the k and v rows this group takes next travel to L2 while it works on these (measured: a gain for
                    // the short k*v rows, none for the long filter rows)
                    const long long rn = 2 * after(rp);
                    if (rn + 1 < p.rows) {
                        prefetch_rows_l2(ab + rn * rowb, ab + (rn + 2) * rowb);
                        if (MODE == 0) prefetch_rows_l2(bb + rn * rowb, bb + (rn + 2) * rowb);
                    }
                }
                cp_async_wait_all();
            }
            __syncwarp(m);
            const int f0 = (int)((unsigned long long)g0 & 15ull), f1 = (int)((unsigned long long)g1 & 15ull);
            const int fb0 = (int)((unsigned long long)h0 & 15ull), fb1 = (int)((unsigned long long)h1 & 15ull);
            if constexpr (MODE == 1) {
                // filter rows: blank the padding taps (and a missing second row) once, then no bounds tests
                zero_staged<T, TPL>(s, f0, p.len, P, l);
                zero_staged<T, TPL>(s + SLOT, f1, has1 ? p.len : 0, P, l);
                __syncwarp(m);
                const int cw = ring<P>(l + p.shift);
                transform(rp, [&](int i, int r, int) {
                    const int mm = ring<P>(cw + i * TPL + r * (P / F::template Pass<0>::R));
                    return make_float2(staged<T>(s, f0, mm), staged<T>(s + SLOT, f1, mm));
                });
            } else if (P % 3 != 0 && p.len == HP && has1) {
                // full rows: no bounds tests in the input functor (3 * 2^k points have few full rows, and with two copies of the first
                // pass 768 points spill 300 bytes per thread: 384x384 grids, 128 slices fp32, 470 -> 453 us with one, 257x257 393 -> 381)
                transform(rp, [&](int, int, int idx) {
                    float a = staged<T>(s, f0, idx), b = staged<T>(s + SLOT, f1, idx);
                    if (MODE == 0) {
                        a *= staged<T>(s + 2 * SLOT, fb0, idx);
                        b *= staged<T>(s + 3 * SLOT, fb1, idx);
                    }
                    return make_float2(a, b);
                });
            } else {
                transform(rp, [&](int, int, int idx) {
                    float a = 0.f, b = 0.f;
                    if (idx < p.len) {
                        a = staged<T>(s, f0, idx);
                        if (has1) b = staged<T>(s + SLOT, f1, idx);
                        if (MODE == 0) {
                            a *= staged<T>(s + 2 * SLOT, fb0, idx);
                            if (has1) b *= staged<T>(s + 3 * SLOT, fb1, idx);
                        }
                    }
                    return make_float2(a, b);
                });
            }
        }
        float2 *o0 = p.out + r0 * p.pitch, *o1 = p.out + r1 * p.pitch;
        for (int kx = l; kx <= HP; kx += TPL) {
            const float2 z1 = line[F::ph(kx)], z2 = line[F::ph(ring<P>(P - kx))];
            HN_G(o0 + kx, 8);
            if (has1) HN_G(o1 + kx, 8);
            o0[kx] = make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
            if (has1) o1[kx] = make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x));
        }
        __syncwarp(m);
    }
    if constexpr (AHEAD) {
        if (failed) {
            // a wait gave up: say so, and give the rows that may still be on their way a bounded time to land
            if (p.status) atomicExch(p.status, 11);
            mbar_wait(bar, phase);
        }
    }
}

// OUT: which outputs of a row are kept.  ROW_CROP the first len <= P/2; ROW_FULL (circular mode) all of them; ROW_SHIFT (rows of
// taps) positions (n - shift) mod P, n < len.
enum { ROW_CROP = 0, ROW_FULL = 1, ROW_SHIFT = 2 };
template <typename T, int LOG2P, int OUT, bool LATE>
__global__ void __launch_bounds__(kRowThreads, 2) rows_inv_w_kernel(RowsInvArgs p)
{
    constexpr bool FULL = OUT != ROW_CROP;
    using FI = WF<LOG2P, true>;
    constexpr int P = len_of(LOG2P), HP = P / 2, TPL = FI::TPL, G = kRowThreads / TPL, LS = plane_ls(P);
    constexpr int RS = HP + 2;                                   // slot of one staged half spectrum
    static_assert(2 * RS <= LS, "staged spectra must fit the line");
    extern __shared__ float2 smem[];
    float2 *twt = smem + G * LS;
    const int tid = threadIdx.x, l = tid % TPL, gid = tid / TPL;
    const unsigned m = FI::group_mask(tid);
    float2 *line = smem + gid * LS;
    for (int t = tid; t < P; t += kRowThreads) { HN_G(p.gtw + t * (p.gtw_n / P), 8); twt[t] = p.gtw[t * (p.gtw_n / P)]; }
    __syncthreads();
    PlaneTw<LOG2P, true> tw;
    if constexpr (LATE) pdl_join();
    tw.init(l, twt, twt + P, tid, kRowThreads);
    __syncthreads();
    if constexpr (!LATE) pdl_join();
    const T *pq = (const T *)p.q;
    T *py = (T *)p.y;
    const long long pairs = (p.rows + 1) / 2;
    for (long long rp = (long long)blockIdx.x * G + gid; rp < pairs; rp += (long long)gridDim.x * G) {
        const long long r0 = 2 * rp, r1 = r0 + 1;
        const bool has1 = r1 < p.rows;
        const float2 *i0 = p.in + r0 * p.pitch, *i1 = p.in + r1 * p.pitch;
        // rows of the workspace start on 16-byte boundaries (even pitch): two bins per copy
        for (int c = l; 2 * c <= HP; c += TPL) {
            cp_async16(line + 2 * c, i0 + 2 * c);
            if (has1) cp_async16(line + RS + 2 * c, i1 + 2 * c);
        }
        if (l == 0) {
            // the gate rows of the pair travel to L2 meanwhile
            const long long e0 = r0 * p.len, e1 = e0 + (has1 ? 2 : 1) * (long long)p.len;
            if (pq) prefetch_rows_l2((const unsigned char *)(pq + e0), (const unsigned char *)(pq + e1));
            if (p.q2) prefetch_rows_l2((const unsigned char *)((const T *)p.q2 + e0), (const unsigned char *)((const T *)p.q2 + e1));
        }
        cp_async_wait_all();
        __syncwarp(m);
        // Legs below half the first-pass radix read bins <= P/2 directly; the others read the mirrored bin
        // conjugated.  Which case applies is known per leg at compile time, except for the leg that starts at
        // P/2 (its first position is the unmirrored bin P/2 itself).
        if (!has1) for (int c = l; c <= HP; c += TPL) line[RS + c] = make_float2(0.f, 0.f);
        __syncwarp(m);
        constexpr int RH = FI::template Pass<0>::R / 2;
        FI::template run_to_line<FULL ? PRUNE_NONE : PRUNE_OUT, true>(l, m, tw, line, [&](int, int r, int idx) {
            if (r < RH) {
                const float2 A = line[idx], B = line[RS + idx];
                return make_float2(A.x - B.y, A.y + B.x);
            }
            const float2 A = line[P - idx], B = line[RS + P - idx];
            const float sg = (r == RH && idx == HP) ? 1.f : -1.f;
            return make_float2(fmaf(-sg, B.y, A.x), fmaf(sg, A.y, B.x));
        });
        auto at = [&](int n) { return line[FI::ph(OUT == ROW_SHIFT ? ring<P>(n + P - p.shift) : n)]; };
        // gate and store in rounds of eight values of each row, whose gate loads are in flight together (one iteration's at a time
        // the loads waited for memory each: periodic 512x512 grids, 256 slices fp32, 160 -> 131 us; 511x500 fp32 128 -> 96)
        auto rows_out = [&](const T *gq, T *gy) {
            const T *q0 = gq + r0 * p.len, *q1 = q0 + p.len;
            T *y0 = gy + r0 * p.len, *y1 = y0 + p.len;
            constexpr int U = 8;
#pragma unroll 1
            for (int n0 = l; n0 < p.len; n0 += U * TPL) {
                T qa[U], qb[U];                            // (converted where they are used: under the loads' conditions they would wait one by one)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int n = n0 + u * TPL;
                    const bool oa = n < p.len, ob = oa && has1;
                    if (oa) HN_G(q0 + n, sizeof(T));
                    if (ob) HN_G(q1 + n, sizeof(T));
                    qa[u] = oa ? __ldg(q0 + n) : T(1.f);
                    qb[u] = ob ? __ldg(q1 + n) : T(1.f);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int n = n0 + u * TPL;
                    if (n >= p.len) break;
                    const float2 z = at(n);
                    IO<T>::st(y0, n, z.x * (float)qa[u]);
                    if (has1) IO<T>::st(y1, n, z.y * (float)qb[u]);
                }
            }
        };
        if (!FULL && p.len == HP && has1 && pq) {
            // full rows: all gate loads of the pair are in flight together (they were asked into L2 above)
            float qa[HP / TPL], qb[HP / TPL];
#pragma unroll
            for (int t = 0; t < HP / TPL; ++t) {
                qa[t] = IO<T>::ld(pq, r0 * HP + l + t * TPL);
                qb[t] = IO<T>::ld(pq, r1 * HP + l + t * TPL);
            }
#pragma unroll
            for (int t = 0; t < HP / TPL; ++t) {
                const float2 z = line[FI::ph(l + t * TPL)];
                IO<T>::st(py, r0 * HP + l + t * TPL, z.x * qa[t]);
                IO<T>::st(py, r1 * HP + l + t * TPL, z.y * qb[t]);
            }
        } else if (pq) {
            rows_out(pq, py);
        } else {
            // no gate tensor: the rows leave as they are
            for (int n = l; n < p.len; n += TPL) {
                const float2 z = at(n);
                IO<T>::st(py, r0 * p.len + n, z.x);
                if (has1) IO<T>::st(py, r1 * p.len + n, z.y);
            }
        }
        if (p.y2) rows_out((const T *)p.q2, (T *)p.y2);    // second gate and result: the rows are still in the line
        __syncwarp(m);
    }
}

static int rows_sms()
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

// length and grid size from which the kernels take their LATE variant (rows ahead have none: no spills either way)
template <int LOG2P> constexpr bool kLateRows = LOG2P == 10;
static bool late_rows(long long ctas) { return ctas >= rows_sms(); }
// Rows ahead (GA) or staged (GS), for `pairs` pairs of rows.  1024 points: ahead (128 slices of 512x512, filter rows and k*v rows: fp32
// 206 and 102 us -> 184 and 91, bf16 190 and 94 -> 165 and 85; passes of 11 to 62 slices 1.05 to 1.10 times as fast as with staged
// rows), but for two ranges: pairs that are one round of the staged groups and more than one of those ahead (16 and 12 warps per SM),
// and pairs whose staged CTAs, of twice as many groups, are fewer than the SMs, so that they let the next kernel in early, while the
// CTAs ahead are not, or the rows are k*v rows, which the core waits for (staged / ahead: 10 slices of 100x400 fp32 28.3 and 29.2 us,
// bf16 28.6 and 29.0; 20 of 40x511 fp32 27.3 and 28.4; 5 of 100x400 25.1 and 25.0; 4 of 512x512 fp32, in both ranges, 38.0 and 39.9).
// 512 points: fp32 filter rows of three rounds and more (256x256, 70 to 257 slices: 1.01 to 1.09; 1788 to 9313 pairs 0.87 to 1.08,
// mostly by the larger last round); k*v rows are faster staged (fp32 0.80 to
// 0.95, bf16 52 and 29 us -> 53 and 32).  Shorter rows are a few hundred bytes, whose waits 16 warps cover (256 points: 63 and 35 ->
// 70 and 38).
template <int LOG2P, int MODE, class GA, class GS> static bool ahead_rows(long long pairs)
{
    const long long sms = rows_sms(), round_a = sms * GA::PER_SM * GA::G, round_s = sms * GS::PER_SM * GS::G;
    if (LOG2P != 10) return pairs >= 3 * round_a;
    const bool lets_in_early = pairs <= (sms - 1) * GS::G && (MODE == 0 || pairs > (sms - 1) * GA::G);
    return !lets_in_early && (pairs <= round_a || pairs > round_s);
}

bool rows_w_supported(int log2p) { return (log2p >= 6 && log2p <= 10) || (log2p >= kLen192 && log2p <= kLen768); }

template <typename T, int LOG2P> static int launch_rows_fwd_w_t(const RowsArgs &a, cudaStream_t st)
{
    constexpr int P = len_of(LOG2P);
    if (a.rows <= 0) return 0;
    auto go = [&](auto mode, auto late, auto ahead, long long want) {
        using GE = RowFwdGeo<T, LOG2P, decltype(mode)::value, decltype(ahead)::value>;
        auto fn = rows_fwd_w_kernel<T, LOG2P, decltype(mode)::value, decltype(late)::value, decltype(ahead)::value>;
        static DevOnce attr;
        if (attr.first()) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GE::TOTAL);
        const long long res = (long long)GE::PER_SM * rows_sms();
        launch_pdl(fn, (unsigned)(want < res ? want : res), GE::THREADS, GE::TOTAL, st, a);
    };
    auto launch = [&](auto mode) {
        constexpr int M = decltype(mode)::value;
        using GE = RowFwdGeo<T, LOG2P, M, false>;
        const long long pairs = (a.rows + 1) / 2, want = (pairs + GE::G - 1) / GE::G;
        if constexpr (kAheadRows<T, LOG2P, M>) {
            // (a wait that gives up has to be reported: calls without a status word take the rows without such waits)
            using GA = RowFwdGeo<T, LOG2P, M, true>;
            if (a.status && ahead_rows<LOG2P, M, GA, GE>(pairs)) return go(mode, std::false_type{}, std::true_type{}, (pairs + GA::G - 1) / GA::G);
        }
        if constexpr (kLateRows<LOG2P>) { if (late_rows(want)) return go(mode, std::true_type{}, std::false_type{}, want); }
        go(mode, std::false_type{}, std::false_type{}, want);
    };
    if (a.full_in) {
        if constexpr ((P & (P - 1)) == 0) launch(std::integral_constant<int, 3>{}); else return -1;      // (periodic grids are powers of two)
    }
    else if (a.b) launch(std::integral_constant<int, 0>{});
    else if (a.prune_in) launch(std::integral_constant<int, 2>{});
    else launch(std::integral_constant<int, 1>{});
    return 1;
}

template <typename T, int LOG2P> static int launch_rows_inv_w_t(const RowsInvArgs &a, cudaStream_t st)
{
    using F = WF<LOG2P, true>;
    constexpr int P = len_of(LOG2P), G = kRowThreads / F::TPL, LS = plane_ls(P);
    const size_t sm = sizeof(float2) * ((size_t)G * LS + 2 * P);
    const long long want = ((a.rows + 1) / 2 + G - 1) / G;
    const int grid = (int)(want < 2ll * rows_sms() ? want : 2ll * rows_sms());
    if (grid <= 0) return 0;
    auto go = [&](auto out, auto late) {
        auto fn = rows_inv_w_kernel<T, LOG2P, decltype(out)::value, decltype(late)::value>;
        static DevOnce attr;
        if (attr.first()) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        launch_pdl(fn, grid, kRowThreads, sm, st, a);
    };
    auto launch = [&](auto out) {
        if constexpr (kLateRows<LOG2P>) { if (late_rows(grid)) return go(out, std::true_type{}); }
        go(out, std::false_type{});
    };
    if (!a.full_out) launch(std::integral_constant<int, ROW_CROP>{});
    else if constexpr (P % 3 == 0) launch(std::integral_constant<int, ROW_SHIFT>{});      // (periodic grids are powers of two)
    else if (a.shift) launch(std::integral_constant<int, ROW_SHIFT>{});
    else launch(std::integral_constant<int, ROW_FULL>{});
    return 1;
}

#define HN_SWITCH_RW(x, CALL)                                                                  \
    switch (x) {                                                                               \
    case 6: CALL(6); break; case 7: CALL(7); break; case 8: CALL(8); break;                    \
    case 9: CALL(9); break; case 10: CALL(10); break;                                          \
    case kLen192: CALL(kLen192); break; case kLen384: CALL(kLen384); break; case kLen768: CALL(kLen768); break;     \
    default: return -1;                                                                        \
    }

int launch_rows_fwd_w(const RowsArgs &a, int dtype, cudaStream_t st)
{
    int n = 0;
#define CALLF(L) n = launch_rows_fwd_w_t<float, L>(a, st)
#define CALLB(L) n = launch_rows_fwd_w_t<bf16, L>(a, st)
    if (dtype == 0) { HN_SWITCH_RW(a.log2p, CALLF) } else { HN_SWITCH_RW(a.log2p, CALLB) }
#undef CALLF
#undef CALLB
    return n;
}

int launch_rows_inv_w(const RowsInvArgs &a, int dtype, cudaStream_t st)
{
    int n = 0;
#define CALLF(L) n = launch_rows_inv_w_t<float, L>(a, st)
#define CALLB(L) n = launch_rows_inv_w_t<bf16, L>(a, st)
    if (dtype == 0) { HN_SWITCH_RW(a.log2p, CALLF) } else { HN_SWITCH_RW(a.log2p, CALLB) }
#undef CALLF
#undef CALLB
    return n;
}

}  // namespace hn
