// Slice-fused forward kernel (see slice_fft.cuh for the engine): one group of M / 16 threads takes a slice from its
// tensors to its result, y = q * crop(IFFT(FFT(pad(k v)) FFT(pad(h)))), in two shared-memory buffers.
//
// Used wherever the engine has an instance (slice.cu): lines padded to at most 8192 points, small 2-D and 3-D grids.  The
// general path takes these shapes through four to eight kernels with the spectra in HBM and, for lines and axes below 64
// points, block-wide transforms with element-wise copies.  Measured, general path -> here: 12288 rows of 2000 bf16 values
// (shared filters) 2336 -> 150 us, 24576 grids of 15 x 14 527 -> 139 us.  What bounds it: instruction issue (63 % of the
// slots at 16 warps per SM for the 4096-point lines, FMA pipe 50 %), then the shared-memory pipe (55 %).
#pragma once
#include "slice.cuh"
#include "slice_fft.cuh"
#include "mix.cuh"

namespace hn {

template <class S> struct SliceCta {
    static constexpr int THREADS = S::T >= 128 ? S::T : 128;
    static constexpr int G = THREADS / S::T;                 // slices per CTA
    // groups of more than a warp synchronise through the CTA's barrier: they have the CTA to themselves
    static constexpr bool WARP = S::T <= 32;
    static constexpr int CT = WARP ? THREADS : S::T;         // threads launched
    static constexpr int NG = WARP ? G : 1;
    static constexpr int PER_SM = 512 / CT;                  // at most 128 registers per thread
    __host__ __device__ static constexpr size_t smem(int bufs) { return sizeof(float2) * ((size_t)NG * bufs * S::BUF + S::TAB); }
    static __device__ __forceinline__ void sync()
    {
        if constexpr (WARP) __syncwarp(); else __syncthreads();
    }
};

// Index of the complex point `idx` of a slice on its grid: rows (i0, i1) and the first of its two positions x.
template <class S> struct SliceIdx {
    int i0, i1, x;
    __device__ __forceinline__ explicit SliceIdx(int idx)
        : i0(S::L0 ? idx >> (S::L1 + S::L2) : 0), i1(S::L1 ? (idx >> S::L2) & ((1 << S::L1) - 1) : 0), x(2 * (idx & ((1 << S::L2) - 1))) {}
};

// ---- two neighbouring reals of a row ---------------------------------------------------------------------------------
// Loads are gathered for all legs of an item before the first value is used (a leg at a time, each under its own branch,
// exposed the memory latency once per leg: 374 us for 12288 rows of 2000 bf16 values, gathered 160).  EVEN: rows are whole
// pairs, one load per pair; else two loads, the second one where x + 1 is still in the row.
template <typename T, bool EVEN> struct SlPair;
template <> struct SlPair<float, true> {
    float2 v;
    __device__ __forceinline__ void load(const float *p, bool a, bool) { if (a) HN_G(p, 8); v = a ? __ldg(reinterpret_cast<const float2 *>(p)) : make_float2(0.f, 0.f); }
    __device__ __forceinline__ float2 get() const { return v; }
    static __device__ __forceinline__ void store(float *p, float2 w, bool a, bool) { if (a) { HN_G(p, 8); *reinterpret_cast<float2 *>(p) = w; } }
};
template <> struct SlPair<float, false> {
    float2 v;
    __device__ __forceinline__ void load(const float *p, bool a, bool b) { load2(p, p + 1, a, b); }
    __device__ __forceinline__ void load2(const float *p, const float *p1, bool a, bool b)
    {
        if (a) HN_G(p, 4);
        if (b) HN_G(p1, 4);
        v.x = a ? __ldg(p) : 0.f;
        v.y = b ? __ldg(p1) : 0.f;
    }
    __device__ __forceinline__ float2 get() const { return v; }
    static __device__ __forceinline__ void store(float *p, float2 w, bool a, bool b)
    {
        if (a) { HN_G(p, 4); p[0] = w.x; }
        if (b) { HN_G(p + 1, 4); p[1] = w.y; }
    }
};
template <> struct SlPair<bf16, true> {
    unsigned v;
    __device__ __forceinline__ void load(const bf16 *p, bool a, bool) { if (a) HN_G(p, 4); v = a ? __ldg(reinterpret_cast<const unsigned *>(p)) : 0u; }
    __device__ __forceinline__ float2 get() const { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }
    static __device__ __forceinline__ void store(bf16 *p, float2 w, bool a, bool)
    {
        if (a) { HN_G(p, 4); *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(w.x, w.y); }
    }
};
template <> struct SlPair<bf16, false> {
    unsigned short lo, hi;
    __device__ __forceinline__ void load(const bf16 *p, bool a, bool b) { load2(p, p + 1, a, b); }
    __device__ __forceinline__ void load2(const bf16 *p, const bf16 *p1, bool a, bool b)
    {
        if (a) HN_G(p, 2);
        if (b) HN_G(p1, 2);
        lo = a ? __ldg(reinterpret_cast<const unsigned short *>(p)) : (unsigned short)0;
        hi = b ? __ldg(reinterpret_cast<const unsigned short *>(p1)) : (unsigned short)0;
    }
    __device__ __forceinline__ float2 get() const { return make_float2(__uint_as_float((unsigned)lo << 16), __uint_as_float((unsigned)hi << 16)); }
    static __device__ __forceinline__ void store(bf16 *p, float2 w, bool a, bool b)
    {
        if (a) { HN_G(p, 2); p[0] = __float2bfloat16_rn(w.x); }
        if (b) { HN_G(p + 1, 2); p[1] = __float2bfloat16_rn(w.y); }
    }
};

// Where the legs of a first-pass item lie in a slice of the grid: leg r's pair at element o + r * step, its first element
// exists for r < na, its second one for r < nb (the legs of an item share all but one coordinate).
template <class S> struct SliceLegs {
    using P = typename S::First;
    static constexpr int AX = S::first_axis();
    static constexpr int D = P::SL - S::stride_log(AX);      // log2 of the legs' distance on the axis
    int o, na, nb, row;
    __device__ __forceinline__ SliceLegs(const SliceGeo &g, int base, bool on)
    {
        const SliceIdx<S> c(base);
        row = AX == 0 ? g.L[1] * g.L[2] : g.L[2];
        o = (S::L0 ? c.i0 * g.L[1] * g.L[2] : 0) + (S::L1 ? c.i1 * g.L[2] : 0) + c.x;
        if constexpr (AX == 2) {
            na = on ? (g.L[2] - c.x + (2 << D) - 1) >> (D + 1) : 0;
            nb = on ? (g.L[2] - 1 - c.x + (2 << D) - 1) >> (D + 1) : 0;
        } else {
            const int i = AX == 0 ? c.i0 : c.i1, L = AX == 0 ? g.L[0] : g.L[1];
            const bool in = on && c.x < g.L[2] && (AX == 1 || S::L1 == 0 || c.i1 < g.L[1]);
            na = in ? (L - i + (1 << D) - 1) >> D : 0;
            nb = c.x + 1 < g.L[2] ? na : 0;
        }
    }
    __device__ __forceinline__ int at(int r) const { return AX == 2 ? o + (r << (D + 1)) : o + (r << D) * row; }
};

// taps of an item's legs: positions x, x + 1 hold taps (x + shift) mod P2 and the one after it.  EVEN: unshifted rows of
// whole pairs (causal, circular).
template <class S, int NIN, bool EVEN, typename T>
__device__ __forceinline__ void slice_taps(const T *h, const SliceGeo &g, int base, bool on, float2 *x)
{
    using P = typename S::First;
    constexpr int AX = S::first_axis(), D = P::SL - S::stride_log(AX);
    SlPair<T, EVEN> w[NIN];
    const SliceIdx<S> c(base);
    constexpr int MX = (2 << S::L2) - 1, MA = (1 << (AX == 0 ? S::L0 : S::L1)) - 1;
    if constexpr (AX == 2) {
#pragma unroll
        for (int r = 0; r < NIN; ++r) {
            const int xr = c.x + (r << (D + 1));
            if constexpr (EVEN) {
                w[r].load(h + xr, on && xr < g.K[2], true);
            } else {
                const int ma = (xr + g.shift[2]) & MX, mb = (xr + 1 + g.shift[2]) & MX;
                w[r].load2(h + ma, h + mb, on && ma < g.K[2], on && mb < g.K[2]);
            }
        }
    } else {
        const int ma = (c.x + g.shift[2]) & MX, mb = (c.x + 1 + g.shift[2]) & MX;
        const int m1 = (AX == 0 && S::L1) ? (c.i1 + g.shift[1]) & ((1 << S::L1) - 1) : 0;
        const bool in = on && (AX == 1 || S::L1 == 0 || m1 < g.K[1]);
        const bool va = in && ma < g.K[2], vb = in && mb < g.K[2];
        const int row = AX == 0 ? g.K[1] * g.K[2] : g.K[2], Kax = AX == 0 ? g.K[0] : g.K[1];
        const int i = (AX == 0 ? c.i0 + g.shift[0] : c.i1 + g.shift[1]);
        const T *pa = h + (AX == 0 ? m1 * g.K[2] : 0) + ma, *pb = pa + (mb - ma);
#pragma unroll
        for (int r = 0; r < NIN; ++r) {
            const int m = (i + (r << D)) & MA, off = m * row;
            const bool ok = m < Kax;
            if constexpr (EVEN) w[r].load(pa + off, va && ok, true);
            else w[r].load2(pa + off, pb + off, va && ok, vb && ok);
        }
    }
#pragma unroll
    for (int r = 0; r < NIN; ++r) x[r] = w[r].get();
}

// the gated signal of an item's legs
template <class S, int NIN, bool EVEN, typename T>
__device__ __forceinline__ void slice_signal(const T *k, const T *v, const SliceLegs<S> &g, float2 *x)
{
    SlPair<T, EVEN> a[NIN], b[NIN];
#pragma unroll
    for (int r = 0; r < NIN; ++r) {
        a[r].load(k + g.at(r), r < g.na, r < g.nb);
        b[r].load(v + g.at(r), r < g.na, r < g.nb);
    }
#pragma unroll
    for (int r = 0; r < NIN; ++r) {
        const float2 u = a[r].get(), w = b[r].get();
        x[r] = make_float2(u.x * w.x, u.y * w.y);
    }
}

// the operator's signal of an item's legs: q scale g_in SiLU(k)
template <class S, int NIN, bool EVEN, typename T>
__device__ __forceinline__ void slice_mixed(const T *q, const T *k, const float *ts, float gin, const SliceLegs<S> &g, float2 *x)
{
    SlPair<T, EVEN> a[NIN], b[NIN];
    SlPair<float, EVEN> c[NIN];
#pragma unroll
    for (int r = 0; r < NIN; ++r) {
        a[r].load(q + g.at(r), r < g.na, r < g.nb);
        b[r].load(k + g.at(r), r < g.na, r < g.nb);
        c[r].load(ts + g.at(r), r < g.na, r < g.nb);
    }
#pragma unroll
    for (int r = 0; r < NIN; ++r) {
        const float2 u = a[r].get(), w = b[r].get(), sc = c[r].get();
        x[r] = make_float2(u.x * (sc.x * gin) * (w.x * mix_sigmoid(w.x)), u.y * (sc.y * gin) * (w.y * mix_sigmoid(w.y)));
    }
}

// the pair of tap gradients at array index idx: the inverse of the placement above
template <class S, typename T> __device__ __forceinline__ void slice_tap_store(T *dh, const SliceGeo &g, int idx, bool on, float2 w)
{
    const SliceIdx<S> c(idx);
    const int m0 = S::L0 ? (c.i0 + g.shift[0]) & ((1 << S::L0) - 1) : 0;
    const int m1 = S::L1 ? (c.i1 + g.shift[1]) & ((1 << S::L1) - 1) : 0;
    const int ma = (c.x + g.shift[2]) & ((2 << S::L2) - 1), mb = (c.x + 1 + g.shift[2]) & ((2 << S::L2) - 1);
    const bool row = on && (S::L0 == 0 || m0 < g.K[0]) && (S::L1 == 0 || m1 < g.K[1]);
    T *p = dh + ((S::L0 ? m0 * g.K[1] * g.K[2] : 0) + (S::L1 ? m1 * g.K[2] : 0));
    if (row && ma < g.K[2]) IO<T>::st(p, ma, w.x);
    if (row && mb < g.K[2]) IO<T>::st(p, mb, w.y);
}

// Mirrored frequency of a last-digit item: where the 16 legs of its partner sit.  Leg r's partner is leg (16 - r) mod 16
// of the partner item where the lower digits of k2 are zero, else leg 15 - r.
template <class S> struct SliceMirror {
    int pm;                   // physical index of the partner's leg for r = 1 .. 15 is pm - r
    int p0;                   // and for r = 0
    int klow;                 // k2 of leg 0
    __device__ __forceinline__ explicit SliceMirror(int item)
    {
        constexpr int NL = S::L2 - 4;                        // bits of k2 above the last digit's leg index
        const int b = item << 4;
        const int f0 = S::L0 ? sl_freq<S::L0, false>(b >> (S::L1 + S::L2)) : 0;
        const int f1 = S::L1 ? sl_freq<S::L1, false>((b >> S::L2) & ((1 << S::L1) - 1)) : 0;
        // the last digit is zero in b: the frequency of the contiguous axis is its low part
        klow = sl_freq<S::L2, true>(b & ((1 << S::L2) - 1));
        const int g0 = S::L0 ? sl_pos<S::L0, false>((-f0) & ((1 << S::L0) - 1)) : 0;
        const int g1 = S::L1 ? sl_pos<S::L1, false>((-f1) & ((1 << S::L1) - 1)) : 0;
        const int kl = (-klow) & ((1 << NL) - 1);
        const int pb = (((g0 << S::L1) | g1) << S::L2) | sl_pos<S::L2, true>(kl);
        const int base = S::ph(pb);
        pm = base + (klow == 0 ? 16 : 15);
        p0 = base + (klow == 0 ? 0 : 15);
    }
};

__device__ __forceinline__ float2 sl_even(float2 z, float2 m) { return make_float2(z.x + m.x, z.y - m.y); }       // 2 E
__device__ __forceinline__ float2 sl_odd(float2 z, float2 m) { return make_float2(z.y + m.y, m.x - z.x); }        // 2 O

// a * exp(-2 pi i R / 16), R a compile-time leg
template <int R> struct SlLeg { static __device__ __forceinline__ float2 rot(float2 a) { return mul_w16<R, false>(a); } };

// w * exp(-2 pi i r / 16) for a leg r known after unrolling
__device__ __forceinline__ float2 sl_rot16(float2 w, int r)
{
    switch (r) {
    case 1: return SlLeg<1>::rot(w); case 2: return SlLeg<2>::rot(w); case 3: return SlLeg<3>::rot(w); case 4: return SlLeg<4>::rot(w);
    case 5: return SlLeg<5>::rot(w); case 6: return SlLeg<6>::rot(w); case 7: return SlLeg<7>::rot(w); default: return w;
    }
}

template <int R, class F> __device__ __forceinline__ void sl_legs(F f)
{
    if constexpr (R < 16) { f(std::integral_constant<int, R>{}); sl_legs<R + 1>(f); }
}

// Asks a slice's tensor into L2, one prefetch per 128-byte line, dealt out to the slice's threads.
template <class S, typename T> __device__ __forceinline__ void slice_prefetch(const T *p, long long elems, int t)
{
    const char *b = reinterpret_cast<const char *>(p);
    for (long long o = (long long)t * 128; o < elems * (long long)sizeof(T); o += S::T * 128) {
        HN_G(b + o, 1);
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"(b + o) : "memory");
    }
}

// FULL: circular mode, else the upper half of the signal's first axis is padding.  EVEN: rows of whole pairs.
// MIX: Eq. 2 around the convolution.  k, v, q are then the operator's raw q, k, v: the signal is q scale g_in SiLU(k) with
// one scale per token (the l2 norm and the inner RMSNorm, mixer.cu), the outer gate Sigmoid(v), the result fp32 for the
// outer RMSNorm.
template <typename T, int L0, int L1, int L2, bool FULL, bool EVEN, bool MIX>
__global__ void __launch_bounds__(SliceCta<SliceFft<L0, L1, L2>>::CT, SliceCta<SliceFft<L0, L1, L2>>::PER_SM) slice_fwd_kernel(SliceArgs p)
{
    using S = SliceFft<L0, L1, L2>;
    using CT = SliceCta<S>;
    extern __shared__ float2 smem[];
    const int tid = threadIdx.x, t = tid % S::T, grp = CT::WARP ? tid / S::T : 0;
    float2 *bh = smem + (size_t)grp * 2 * S::BUF, *bu = bh + S::BUF;
    typename S::Tw tw;
    S::init(tw, smem + (size_t)CT::NG * 2 * S::BUF, p.gtw, p.gtw_n, tid, CT::CT, t);
    __syncthreads();
    pdl_join();
    auto sync = [] { CT::sync(); };
    const SliceGeo &g = p.g;
    const float sc = 0.25f / (float)S::M;                    // 1/M of the inverse, 1/4 of the two separations
    const bool shared = p.C > 0;
    const long long n = p.s1 - p.s0;
    // a unit is one filter and the slices it serves: one, or up to nb batch entries of one channel
    const long long c_first = shared ? p.s0 / p.C : 0;       // first batch entry in range
    const long long chunks = shared ? ((p.s1 - 1) / p.C - c_first + p.nb) / p.nb : 0;
    const long long units = shared ? chunks * p.C : n;
    const bool heven = g.shift[2] == 0 && (g.K[2] & 1) == 0;
    const SliceMirror<S> mir(t);
    const float2 w0 = tw.tab[S::WTAB + mir.klow];
    constexpr int NU = S::template NIN<!FULL>, NH = S::template NIN<false>;
    for (long long u0 = (long long)blockIdx.x * CT::NG; u0 < units; u0 += (long long)gridDim.x * CT::NG) {
        const long long u = u0 + grp;
        const bool live = u < units;
        const long long chan = shared ? u % p.C : 0, b0 = shared ? c_first + u / p.C * p.nb : 0;
        {
            const long long hs = (shared ? chan : p.s0 + u) * g.kvol;
            auto taps = [&](const auto *h) {
                S::template fwd_first<false>(bh, tw, t, [&](int, int base, float2 *x) {
                    // (unshifted rows of whole pairs: circular, or causal of even length)
                    if constexpr (FULL) slice_taps<S, NH, true>(h, g, base, live, x);
                    else if (S::L0 == 0 && S::L1 == 0 && heven) slice_taps<S, NH, true>(h, g, base, live, x);
                    else slice_taps<S, NH, false>(h, g, base, live, x);
                });
            };
            // (a plan of fp32 tensors may read bf16 taps, never the other way round)
            if (sizeof(T) == 2 || p.h_bf16) taps((const bf16 *)p.h + hs); else taps((const float *)p.h + hs);
        }
        S::fwd_mid(bh, tw, t, sync);
        sync();
        S::template fwd_pass<2, sl_ndig(L2) - 1>(bh, tw, t);
        const int nbu = shared ? p.nb : 1;
        for (int bi = 0; bi < nbu; ++bi) {
            const long long s = shared ? (b0 + bi) * p.C + chan : p.s0 + u;
            const bool on = live && s >= p.s0 && s < p.s1;
            if (!CT::WARP && !on) continue;                  // (the same for the whole CTA)
            const T *k = (const T *)p.k + s * g.vol, *v = (const T *)p.v + s * g.vol;
            if constexpr (MIX) {
                const float *ts = p.token_scale + (s / p.mix_C) * g.vol;
                HN_G(p.g_in + s % p.mix_C, 4);
                const float gin = on ? __ldg(p.g_in + s % p.mix_C) : 0.f;
                S::template fwd_first<!FULL>(bu, tw, t, [&](int, int base, float2 *x) { slice_mixed<S, NU, EVEN>(k, v, ts, gin, SliceLegs<S>(g, base, on), x); });
            } else {
                S::template fwd_first<!FULL>(bu, tw, t, [&](int, int base, float2 *x) { slice_signal<S, NU, EVEN>(k, v, SliceLegs<S>(g, base, on), x); });
            }
            {
                // what this group reads next travels to L2 under this slice's transforms
                const bool last = bi + 1 == nbu;
                const long long un = u + (long long)gridDim.x * CT::NG;
                const long long sn = !last ? s + p.C : shared ? (c_first + un / p.C * p.nb) * p.C + un % p.C : p.s0 + un;
                if ((!last || un < units) && sn >= p.s0 && sn < p.s1) {
                    slice_prefetch<S>((const T *)p.k + sn * g.vol, g.vol, t);
                    slice_prefetch<S>((const T *)p.v + sn * g.vol, g.vol, t);
                    slice_prefetch<S>((const T *)p.q + sn * g.vol, g.vol, t);
                    if (!shared) {
                        if (p.h_bf16) slice_prefetch<S>((const bf16 *)p.h + sn * g.kvol, g.kvol, t);
                        else slice_prefetch<S>((const float *)p.h + sn * g.kvol, g.kvol, t);
                    }
                }
            }
            S::fwd_mid(bu, tw, t, sync);
            sync();
            float2 z[16];
            float2 *bl = bu + S::ph(t << 4);
            {
#pragma unroll
                for (int r = 0; r < 16; ++r) z[r] = bl[r];
                dft<16, false, PRUNE_NONE>(z);
#pragma unroll
                for (int r = 0; r < 16; ++r) bl[r] = z[r];
            }
            sync();
            const float2 *hl = bh + S::ph(t << 4);
            sl_legs<0>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                const int pi = r == 0 ? mir.p0 : mir.pm - r;
                const float2 zm = bu[pi], hz = hl[r], hm = bh[pi];
                const float2 eu = sl_even(z[r], zm), ou = sl_odd(z[r], zm), eh = sl_even(hz, hm), oh = sl_odd(hz, hm);
                const float2 wo = SlLeg<r>::rot(cmul(cmul(ou, oh), w0));
                const float2 ee = cmul(eu, eh), eo = cmul(eu, oh), oe = cmul(ou, eh);
                const float2 ey = cadd(ee, wo), oy = cadd(eo, oe);
                z[r] = make_float2(ey.x - oy.y, ey.y + oy.x);
            });
            dft<16, true, PRUNE_NONE>(z);
            sync();                                          // every partner has been read
#pragma unroll
            for (int r = 0; r < 16; ++r) bl[r] = z[r];
            S::inv_mid(bu, tw, t, sync);
            // the gate values are requested before the last barrier
            const T *q = (const T *)p.q + s * g.vol;
            using TO = typename MixOut<T, MIX>::type;
            TO *y = (TO *)p.y + s * g.vol;
            SlPair<T, EVEN> gate[S::First::IPT][NU];
#pragma unroll
            for (int i = 0; i < S::First::IPT; ++i) {
                const SliceLegs<S> lg(g, S::First::base(t + i * S::T), on);
#pragma unroll
                for (int r = 0; r < NU; ++r) gate[i][r].load(q + lg.at(r), r < lg.na, r < lg.nb);
            }
            sync();
            S::template inv_last<!FULL>(bu, tw, t, [&](int i, int r, int, float2 w) {
                const SliceLegs<S> lg(g, S::First::base(t + i * S::T), on);
                float2 a = gate[i][r].get();
                if constexpr (MIX) a = make_float2(mix_sigmoid(a.x), mix_sigmoid(a.y));
                SlPair<TO, EVEN>::store(y + lg.at(r), make_float2(w.x * sc * a.x, w.y * sc * a.y), r < lg.na, r < lg.nb);
            });
        }
    }
}

template <typename T, int L0, int L1, int L2, bool FULL, bool EVEN, bool MIX> int launch_slice_t(const SliceArgs &a0, cudaStream_t st)
{
    using S = SliceFft<L0, L1, L2>;
    using CT = SliceCta<S>;
    constexpr size_t sm = CT::smem(2);
    auto fn = slice_fwd_kernel<T, L0, L1, L2, FULL, EVEN, MIX>;
    static int resident[64];
    const int ctas_fit = slice_resident(resident, (const void *)fn, CT::CT, sm);
    if (ctas_fit <= 0) return -1;
    SliceArgs a = a0;
    const long long n = a.s1 - a.s0, slots = (long long)ctas_fit * CT::NG;
    if (n <= 0) return 0;
    long long units = n;
    a.nb = 1;
    if (a.C > 0) {
        // Shared filter: a unit transforms the filter once and serves nb batch entries.  Units of unequal count per slot
        // leave slots idle at the end: nb is the one with the least work on the busiest slot, a unit costing one
        // transform for the filter and two per entry.
        const long long be = (a.s1 - 1) / a.C - a.s0 / a.C + 1;                  // batch entries touched
        long long best = -1;
        for (long long nb = 1; nb <= be && nb <= 64; ++nb) {
            const long long un = (be + nb - 1) / nb * a.C, cost = ((un + slots - 1) / slots) * (1 + 2 * nb);
            if (best < 0 || cost < best) { best = cost; a.nb = (int)nb; units = un; }
        }
    }
    const long long ctas = (units + CT::NG - 1) / CT::NG;
    const int grid = (int)(ctas < ctas_fit ? ctas : ctas_fit);
    launch_pdl(fn, grid, CT::CT, sm, st, a);
    return 1;
}

// (l1, l2) / (l0, l1, l2) instances of the 1-D, 2-D and 3-D translation units; -1: none
int launch_slice_1d_f32(const SliceArgs &a, cudaStream_t st);
int launch_slice_mix_1d_f32(const SliceArgs &a, cudaStream_t st);
int launch_slice_1d_bf16(const SliceArgs &a, cudaStream_t st);
int launch_slice_mix_1d_bf16(const SliceArgs &a, cudaStream_t st);
int launch_slice_2d_f32(const SliceArgs &a, cudaStream_t st);
int launch_slice_mix_2d_f32(const SliceArgs &a, cudaStream_t st);
int launch_slice_2d_bf16(const SliceArgs &a, cudaStream_t st);
int launch_slice_mix_2d_bf16(const SliceArgs &a, cudaStream_t st);
int launch_slice_3d_f32(const SliceArgs &a, cudaStream_t st);
int launch_slice_mix_3d_f32(const SliceArgs &a, cudaStream_t st);
int launch_slice_3d_bf16(const SliceArgs &a, cudaStream_t st);
int launch_slice_mix_3d_bf16(const SliceArgs &a, cudaStream_t st);

template <typename T, int A, int B, int C, bool MIX> int launch_slice_d(const SliceArgs &a, cudaStream_t st)
{
    if (a.g.full) return launch_slice_t<T, A, B, C, true, true, MIX>(a, st);          // (power-of-two rows)
    return (a.g.L[2] & 1) ? launch_slice_t<T, A, B, C, false, false, MIX>(a, st) : launch_slice_t<T, A, B, C, false, true, MIX>(a, st);
}
#define HN_SLICE_CASE(A, B, C)                                                                             \
    if (a.g.l0 == A && a.g.l1 == B && a.g.l2 == C) return launch_slice_d<HN_SLICE_T, A, B, C, HN_SLICE_MIX>(a, st);

// instances of the engine: 1-D lines of 128 .. 8192 reals; 2-D and 3-D grids of up to 8192 complex points
#define HN_SLICE_1D(X) X(0, 0, 6) X(0, 0, 7) X(0, 0, 8) X(0, 0, 9) X(0, 0, 10) X(0, 0, 11) X(0, 0, 12)
#define HN_SLICE_2D(X) X(0, 4, 4) X(0, 4, 5) X(0, 5, 4) X(0, 5, 5) X(0, 5, 6) X(0, 6, 4) X(0, 6, 5) X(0, 6, 6) X(0, 7, 4) X(0, 7, 5) X(0, 7, 6)
#define HN_SLICE_3D(X) X(4, 4, 4) X(4, 5, 4) X(5, 4, 4) X(4, 4, 5)

}  // namespace hn

