// Slice engine: the whole transform of one (b,c) slice in the shared memory of one group of threads.
//
// The padded grid P0 x P1 x P2 of reals is held as n0 x n1 x n2 complex points, n2 = P2 / 2, two neighbouring reals of
// the contiguous axis per point (real part x = 2 i, imaginary part x = 2 i + 1), M = n0 n1 n2 = 2^LM points.  A
// transform is a sequence of in-place passes: a thread reads R points a fixed stride apart, transforms them in
// registers and writes them back where they were.  Forward passes run from the slowest axis to the contiguous one,
// most significant digit first (decimation in frequency), and leave the spectrum in digit-reversed order; inverse
// passes undo them in the opposite order (decimation in time) and end in natural order, so nothing is ever reordered,
// one buffer serves a transform and one barrier separates two passes.  The first forward pass takes its points from a
// functor (global memory, gated and padded on the fly), the last inverse pass hands its results to one.
//
// Product.  With Z the M-point spectrum of a slice of reals packed this way and Z' its value at the mirrored frequency
// (-k on every axis), E = (Z + conj Z') / 2 and O = (Z - conj Z') / 2i are the spectra of the even and of the odd reals.
// The convolution's even and odd spectra are E_u E_h + W O_u O_h and E_u O_h + O_u E_h, W = exp(-2 pi i k2 / n2): the
// packed spectrum of the result needs no value but Z and Z' of either operand.
//
// Points sit at i + (i >> 4): with the last digit of the contiguous axis 16 points wide every pass reads and writes
// without bank conflicts (strides 1 and multiples of 16).
#pragma once
#include "fft_engine.cuh"

namespace hn {

// Digits of an axis of 2^b points, most significant (first forward pass) to least, at most 4 bits each.  The contiguous
// axis (`in`) ends in a digit of 4 bits; the others begin with their widest digit, so that the first pass, which waits for
// global memory, has most loads in flight per thread.
__host__ __device__ constexpr int sl_ndig(int b) { return (b + 3) / 4; }
__host__ __device__ constexpr int sl_dig(int b, int d, bool in)
{
    const int n = sl_ndig(b);
    if (n <= 1) return b;
    if (in && d == n - 1) return 4;
    const int rest = in ? b - 4 : b, m = in ? n - 1 : n;
    if (in) return rest / m + (d < rest % m ? 1 : 0);
    return d == 0 ? 4 : (b - 4) / (n - 1) + (d - 1 < (b - 4) % (n - 1) ? 1 : 0);
}
// bits above digit d of the axis (already transformed when pass d runs)
__host__ __device__ constexpr int sl_above(int b, int d, bool in)
{
    int s = 0;
    for (int i = 0; i < d; ++i) s += sl_dig(b, i, in);
    return s;
}

// position on an axis <-> frequency held there after the forward passes (digit reversal)
template <int B, bool IN> __device__ __forceinline__ int sl_freq(int pos)
{
    int k = 0;
#pragma unroll
    for (int d = 0; d < sl_ndig(B); ++d) {
        const int w = sl_dig(B, d, IN), ab = sl_above(B, d, IN);
        k |= ((pos >> (B - ab - w)) & ((1 << w) - 1)) << ab;
    }
    return k;
}
template <int B, bool IN> __device__ __forceinline__ int sl_pos(int k)
{
    int pos = 0;
#pragma unroll
    for (int d = 0; d < sl_ndig(B); ++d) {
        const int w = sl_dig(B, d, IN), ab = sl_above(B, d, IN);
        pos |= ((k >> ab) & ((1 << w) - 1)) << (B - ab - w);
    }
    return pos;
}

template <int L0_, int L1_, int L2_> struct SliceFft {
    static constexpr int L0 = L0_, L1 = L1_, L2 = L2_, LM = L0 + L1 + L2, M = 1 << LM;
    static_assert(L2 >= 4, "the contiguous axis ends in a digit of 16 points");
    static constexpr int PPT = 16;                           // points per thread
    static constexpr int T = M / PPT;                        // threads per slice
    static constexpr int BUF = M + M / 16;                   // float2 per buffer
    __host__ __device__ static constexpr int bits(int ax) { return ax == 0 ? L0 : ax == 1 ? L1 : L2; }
    __host__ __device__ static constexpr int stride_log(int ax) { return ax == 0 ? L1 + L2 : ax == 1 ? L2 : 0; }
    __host__ __device__ static constexpr int first_axis() { return L0 > 0 ? 0 : L1 > 0 ? 1 : 2; }
    static __device__ __forceinline__ int ph(int i) { return i + (i >> 4); }

    // Twiddle tables of all passes but the untwiddled last digits, one after the other, [leg - 1][j]; the first pass of
    // a 1-D slice keeps its twiddles in registers instead (they depend on the thread only).
    static constexpr bool HOIST = L0 == 0 && L1 == 0 && sl_ndig(L2) > 1;
    __host__ __device__ static constexpr int tab_size(int ax, int d)
    {
        if (d >= sl_ndig(bits(ax)) - 1) return 0;
        if (HOIST && ax == 2 && d == 0) return 0;
        return ((1 << sl_dig(bits(ax), d, ax == 2)) - 1) << (bits(ax) - sl_above(bits(ax), d, ax == 2) - sl_dig(bits(ax), d, ax == 2));
    }
    __host__ __device__ static constexpr int tab_off(int ax, int d)
    {
        int o = 0;
        for (int a = 0; a < 3; ++a)
            for (int i = 0; i < sl_ndig(bits(a)); ++i) {
                if (a == ax && i == d) return o;
                o += tab_size(a, i);
            }
        return o;
    }
    static constexpr int WTAB = tab_off(3, 0);               // then n2 / 16 entries exp(-2 pi i k / n2) for the product
    static constexpr int TAB = WTAB + (1 << (L2 - 4));

    template <int AX, int D> struct Pass {
        static constexpr int B = bits(AX), RB = sl_dig(B, D, AX == 2), R = 1 << RB, LS = B - sl_above(B, D, AX == 2);
        static constexpr int SL = stride_log(AX) + LS - RB;  // log2 of the distance between legs
        static constexpr int IPT = PPT / R;
        static constexpr bool TW = D < sl_ndig(B) - 1;
        static constexpr bool REG = HOIST && AX == 2 && D == 0;
        static __device__ __forceinline__ int base(int item) { return ((item >> SL) << (SL + RB)) | (item & ((1 << SL) - 1)); }
        static __device__ __forceinline__ int j(int item) { return (item & ((1 << SL) - 1)) >> stride_log(AX); }
        // physical distance of leg r from leg 0 (see the header: no carry out of the low bits)
        __host__ __device__ static constexpr int leg(int r) { return (r << SL) + ((r << SL) >> 4); }
    };
    using First = Pass<first_axis(), 0>;
    using Last = Pass<2, sl_ndig(L2) - 1>;
    static_assert(Last::R == 16 && Last::SL == 0, "last digit");

    struct Tw {
        const float2 *tab;
        float2 hw[HOIST ? First::IPT : 1][HOIST ? First::R : 1];
    };
    // gtw: global table of gtw_n >= max axis points; all nthr threads take part; t: thread of its slice; caller synchronises
    static __device__ __forceinline__ void init(Tw &tw, float2 *tab, const float2 *gtw, int gtw_n, int tid, int nthr, int t)
    {
        tw.tab = tab;
        fill<0, 0>(tab, gtw, gtw_n, tid, nthr);
        for (int e = tid; e < (1 << (L2 - 4)); e += nthr) { HN_G(gtw + e * (gtw_n >> L2), 8); tab[WTAB + e] = gtw[e * (gtw_n >> L2)]; }
        if constexpr (HOIST) {
#pragma unroll
            for (int i = 0; i < First::IPT; ++i)
#pragma unroll
                for (int r = 1; r < First::R; ++r) {
                    const float2 *g = gtw + (size_t)r * First::j(t + i * T) * (gtw_n >> L2);
                    HN_G(g, 8);
                    tw.hw[i][r] = __ldg(g);
                }
        }
    }
    template <int AX, int D> static __device__ __forceinline__ void fill(float2 *tab, const float2 *gtw, int gtw_n, int tid, int nthr)
    {
        if constexpr (AX < 3) {
            if constexpr (D < sl_ndig(bits(AX))) {
                if constexpr (tab_size(AX, D) > 0) {
                    using P = Pass<AX, D>;
                    constexpr int NJ = 1 << (P::LS - P::RB);
                    for (int e = tid; e < tab_size(AX, D); e += nthr) {
                        const int r = e / NJ + 1, j = e % NJ;
                        const float2 *g = gtw + (size_t)r * j * (gtw_n >> P::LS);
                        HN_G(g, 8);
                        tab[tab_off(AX, D) + e] = __ldg(g);
                    }
                }
                fill<AX, D + 1>(tab, gtw, gtw_n, tid, nthr);
            } else {
                fill<AX + 1, 0>(tab, gtw, gtw_n, tid, nthr);
            }
        }
    }
    template <int AX, int D> static __device__ __forceinline__ float2 twiddle(const Tw &tw, int i, int r, int j)
    {
        using P = Pass<AX, D>;
        if constexpr (P::REG) return tw.hw[i][r];
        else return tw.tab[tab_off(AX, D) + ((r - 1) << (P::LS - P::RB)) + j];
    }

    // ---- passes -----------------------------------------------------------------------------------------------
    // first forward pass: in(i, base, x) fills the NIN inputs of item i, leg r from array index base + (r << First::SL);
    // PRUNE: the upper half of the first axis is zero and not asked for
    template <bool PRUNE> static constexpr int NIN = PRUNE ? First::R / 2 : First::R;
    template <bool PRUNE, class In> static __device__ __forceinline__ void fwd_first(float2 *buf, const Tw &tw, int t, In in)
    {
        using P = First;
        constexpr int AX = first_axis();
        float2 z[P::IPT][P::R];
#pragma unroll
        for (int i = 0; i < P::IPT; ++i) in(i, P::base(t + i * T), z[i]);        // the loads of all items go out together
#pragma unroll
        for (int i = 0; i < P::IPT; ++i) {
            const int item = t + i * T;
            float2 (&x)[P::R] = z[i];
#pragma unroll
            for (int r = NIN<PRUNE>; r < P::R; ++r) x[r] = make_float2(0.f, 0.f);
            dft<P::R, false, PRUNE ? PRUNE_IN : PRUNE_NONE>(x);
            float2 *b = buf + ph(P::base(item));
            const int j = P::j(item);
#pragma unroll
            for (int r = 0; r < P::R; ++r) {
                if constexpr (P::TW) { if (r) x[r] = cmul(x[r], twiddle<AX, 0>(tw, i, r, j)); }
                b[P::leg(r)] = x[r];
            }
        }
    }
    // NB buffers one after the other (in a loop: one copy of the code, one barrier for all of them)
    template <int AX, int D, int NB = 1> static __device__ __forceinline__ void fwd_pass(float2 *buf, const Tw &tw, int t)
    {
        if constexpr (NB > 1) {
#pragma unroll 1
            for (int b = 0; b < NB; ++b) fwd_one<AX, D>(buf + b * BUF, tw, t);
        } else {
            fwd_one<AX, D>(buf, tw, t);
        }
    }
    template <int AX, int D> static __device__ __forceinline__ void fwd_one(float2 *buf, const Tw &tw, int t)
    {
        using P = Pass<AX, D>;
#pragma unroll
        for (int i = 0; i < P::IPT; ++i) {
            const int item = t + i * T;
            float2 *b = buf + ph(P::base(item));
            float2 x[P::R];
#pragma unroll
            for (int r = 0; r < P::R; ++r) x[r] = b[P::leg(r)];
            dft<P::R, false, PRUNE_NONE>(x);
            const int j = P::j(item);
#pragma unroll
            for (int r = 0; r < P::R; ++r) {
                if constexpr (P::TW) { if (r) x[r] = cmul(x[r], twiddle<AX, D>(tw, i, r, j)); }
                b[P::leg(r)] = x[r];
            }
        }
    }
    template <int AX, int D, int NB = 1> static __device__ __forceinline__ void inv_pass(float2 *buf, const Tw &tw, int t)
    {
        if constexpr (NB > 1) {
#pragma unroll 1
            for (int b = 0; b < NB; ++b) inv_one<AX, D>(buf + b * BUF, tw, t);
        } else {
            inv_one<AX, D>(buf, tw, t);
        }
    }
    template <int AX, int D> static __device__ __forceinline__ void inv_one(float2 *buf, const Tw &tw, int t)
    {
        using P = Pass<AX, D>;
#pragma unroll
        for (int i = 0; i < P::IPT; ++i) {
            const int item = t + i * T;
            float2 *b = buf + ph(P::base(item));
            const int j = P::j(item);
            float2 x[P::R];
#pragma unroll
            for (int r = 0; r < P::R; ++r) {
                x[r] = b[P::leg(r)];
                if constexpr (P::TW) { if (r) x[r] = cmulc(x[r], twiddle<AX, D>(tw, i, r, j)); }
            }
            dft<P::R, true, PRUNE_NONE>(x);
#pragma unroll
            for (int r = 0; r < P::R; ++r) b[P::leg(r)] = x[r];
        }
    }
    // last inverse pass: out(i, r, idx, value); PRUNE: the upper half of the first axis is not produced
    template <bool PRUNE, class Out> static __device__ __forceinline__ void inv_last(const float2 *buf, const Tw &tw, int t, Out out)
    {
        using P = First;
        constexpr int AX = first_axis();
#pragma unroll
        for (int i = 0; i < P::IPT; ++i) {
            const int item = t + i * T, base = P::base(item);
            const float2 *b = buf + ph(base);
            const int j = P::j(item);
            float2 x[P::R];
#pragma unroll
            for (int r = 0; r < P::R; ++r) {
                x[r] = b[P::leg(r)];
                if constexpr (P::TW) { if (r) x[r] = cmulc(x[r], twiddle<AX, 0>(tw, i, r, j)); }
            }
            dft<P::R, true, PRUNE ? PRUNE_OUT : PRUNE_NONE>(x);
            constexpr int NOUT = PRUNE ? P::R / 2 : P::R;
#pragma unroll
            for (int r = 0; r < NOUT; ++r) out(i, r, base + (r << P::SL), x[r]);
        }
    }
    // all forward passes between the first and the last one, and the inverse ones; sync() separates passes (called before
    // each of them)
    template <int NB = 1, class Sync> static __device__ __forceinline__ void fwd_mid(float2 *buf, const Tw &tw, int t, Sync sync)
    {
        fwd_from<first_axis(), 1, NB>(buf, tw, t, sync);
    }
    template <int AX, int D, int NB, class Sync> static __device__ __forceinline__ void fwd_from(float2 *buf, const Tw &tw, int t, Sync sync)
    {
        if constexpr (AX < 3) {
            if constexpr (D >= sl_ndig(bits(AX))) fwd_from<AX + 1, 0, NB>(buf, tw, t, sync);
            else if constexpr (!(AX == 2 && D == sl_ndig(L2) - 1)) {
                sync();
                fwd_pass<AX, D, NB>(buf, tw, t);
                fwd_from<AX, D + 1, NB>(buf, tw, t, sync);
            }
        }
    }
    template <int NB = 1, class Sync> static __device__ __forceinline__ void inv_mid(float2 *buf, const Tw &tw, int t, Sync sync)
    {
        inv_from<2, sl_ndig(L2) - 2, NB>(buf, tw, t, sync);
    }
    template <int AX, int D, int NB, class Sync> static __device__ __forceinline__ void inv_from(float2 *buf, const Tw &tw, int t, Sync sync)
    {
        if constexpr (AX >= first_axis()) {
            if constexpr (D < 0) {
                if constexpr (AX > first_axis()) inv_from<AX - 1, sl_ndig(bits(AX - 1)) - 1, NB>(buf, tw, t, sync);
            } else if constexpr (!(AX == first_axis() && D == 0)) {
                sync();
                inv_pass<AX, D, NB>(buf, tw, t);
                inv_from<AX, D - 1, NB>(buf, tw, t, sync);
            }
        }
    }
};

}  // namespace hn
