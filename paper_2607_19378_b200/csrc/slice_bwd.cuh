// Slice-fused backward kernel: dq, dk, dv and dh of one (b,c) slice from one group of M / 16 threads, in three
// shared-memory buffers (u = k v, h, g = dy q; see slice_fft.cuh for the engine).
//
// With the packed spectra's even and odd parts E, O and w = exp(-2 pi i k2 / n2):
//     h conv u             E = E_u E_h + w O_u O_h          O = E_u O_h + O_u E_h            -> dq
//     h' conv g, h'[d] = h[-d]   E' = conj E, O' = conj(w O) for the reversed factor, hence
//                          E = E_g E_h* + O_g O_h*          O = E_g (w O_h)* + O_g E_h*      -> dk, dv
//     g conv u'            the same with u for h                                             -> dh, at every displacement
// Each mirrored pair of frequencies belongs to one thread, which replaces both members in all three buffers, so the three
// inverse transforms run in place.  The ring of P >= 2L - 1 points per axis holds every displacement without wrap.
//
// Six transforms per slice on data read once.  The general path's backward took twenty launches for these shapes, the
// spectra of each stage through HBM; the fused 2-D path took two forwards of its own and five general kernels for dh.
//
// Issue slots 53 %, shared-memory pipe 54 % busy at 16 warps per SM, the rest is latency (the bytes alone need 31 us): 1536 bf16 slices of 64x64, training step
// 616 -> 407 us, of which this kernel 300.
#pragma once
#include "slice_fwd.cuh"

namespace hn {

// legs 0 .. 7 of an item with their partners, see SliceMirror: which leg the first iteration takes where the partner
// item shares leg 0 (k2 = 0 in the low digits): the smaller item takes the pair of legs 0, the larger one that of legs 8,
// an item that is its own partner both
template <class S> __device__ __forceinline__ int slice_self_leg(int t, const SliceMirror<S> &m)
{
    if (m.klow) return 0;
    return m.p0 < S::ph(t << 4) ? 8 : 0;
}

// one pair of packed frequencies (a at index i, its mirror at index j), w = W^k2 of the first
__device__ __forceinline__ void slice_bwd_pair(float2 *bu, float2 *bh, float2 *bg, int i, int j, float2 w)
{
    const float2 u = bu[i], um = bu[j], h = bh[i], hm = bh[j], g = bg[i], gm = bg[j];
    const float2 eu = sl_even(u, um), ou = sl_odd(u, um), eh = sl_even(h, hm), oh = sl_odd(h, hm), eg = sl_even(g, gm), og = sl_odd(g, gm);
    const float2 wou = cmul(ou, w), woh = cmul(oh, w);
    // packed spectrum E + iO at the frequency, conj(E) + i conj(O) at its mirror
    auto put = [&](float2 *b, float2 e, float2 o) {
        b[i] = make_float2(e.x - o.y, e.y + o.x);
        b[j] = make_float2(e.x + o.y, o.x - e.y);
    };
    put(bu, cadd(cmul(eu, eh), cmul(wou, oh)), cadd(cmul(eu, oh), cmul(ou, eh)));
    put(bh, cadd(cmulc(eg, eh), cmulc(og, oh)), cadd(cmulc(eg, woh), cmulc(og, eh)));
    put(bg, cadd(cmulc(eg, eu), cmulc(og, ou)), cadd(cmulc(eg, wou), cmulc(og, eu)));
}

template <typename T, int L0, int L1, int L2, bool FULL, bool EVEN>
__global__ void __launch_bounds__(SliceCta<SliceFft<L0, L1, L2>>::CT, SliceCta<SliceFft<L0, L1, L2>>::PER_SM) slice_bwd_kernel(SliceBwdArgs p)
{
    using S = SliceFft<L0, L1, L2>;
    using CT = SliceCta<S>;
    using P0 = typename S::First;
    extern __shared__ float2 smem[];
    const int tid = threadIdx.x, t = tid % S::T, grp = CT::WARP ? tid / S::T : 0;
    float2 *bu = smem + (size_t)grp * 3 * S::BUF, *bh = bu + S::BUF, *bg = bh + S::BUF;
    typename S::Tw tw;
    S::init(tw, smem + (size_t)CT::NG * 3 * S::BUF, p.gtw, p.gtw_n, tid, CT::CT, t);
    __syncthreads();
    pdl_join();                                              // (the tables built under the forward: one line of 4096 25.0 -> 23.6 us a step)
    auto sync = [] { CT::sync(); };
    const SliceGeo &g = p.g;
    const float sc = 0.25f / (float)S::M;
    const bool heven = g.shift[2] == 0 && (g.K[2] & 1) == 0;
    const SliceMirror<S> mir(t);
    const float2 w0 = tw.tab[S::WTAB + mir.klow];
    const int self = slice_self_leg<S>(t, mir);
    const bool own = mir.klow == 0 && mir.p0 == S::ph(t << 4);
    constexpr int NU = S::template NIN<!FULL>, NH = S::template NIN<false>;
    for (long long u0 = (long long)blockIdx.x * CT::NG; u0 < p.slices; u0 += (long long)gridDim.x * CT::NG) {
        const long long s = u0 + grp;
        const bool on = s < p.slices;
        const long long so = s * g.vol, hs = p.C > 0 ? s % p.C : s;
        const T *q = (const T *)p.q + so, *k = (const T *)p.k + so, *v = (const T *)p.v + so, *dy = (const T *)p.dy + so;
        const T *h = (const T *)p.h + hs * g.kvol;
        S::template fwd_first<false>(bh, tw, t, [&](int, int base, float2 *x) {
            if constexpr (FULL) slice_taps<S, NH, true>(h, g, base, on, x);
            else if (S::L0 == 0 && S::L1 == 0 && heven) slice_taps<S, NH, true>(h, g, base, on, x);
            else slice_taps<S, NH, false>(h, g, base, on, x);
        });
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            const T *a = i ? dy : k, *b = i ? q : v;
            S::template fwd_first<!FULL>(i ? bg : bu, tw, t, [&](int, int base, float2 *x) {
                slice_signal<S, NU, EVEN>(a, b, SliceLegs<S>(g, base, on), x);
            });
        }
        {
            const long long sn = s + (long long)gridDim.x * CT::NG;       // what this group reads next travels to L2
            if (sn < p.slices) {
                slice_prefetch<S>((const T *)p.q + sn * g.vol, g.vol, t);
                slice_prefetch<S>((const T *)p.k + sn * g.vol, g.vol, t);
                slice_prefetch<S>((const T *)p.v + sn * g.vol, g.vol, t);
                slice_prefetch<S>((const T *)p.dy + sn * g.vol, g.vol, t);
                if (p.C <= 0) slice_prefetch<S>((const T *)p.h + sn * g.kvol, g.kvol, t);
            }
        }
        // the three transforms side by side: one barrier serves a pass of all of them, and one copy of its code
        S::template fwd_mid<3>(bu, tw, t, sync);
        sync();
        S::template fwd_pass<2, sl_ndig(L2) - 1, 3>(bu, tw, t);
        sync();
        {
            const int b = S::ph(t << 4);
#pragma unroll
            for (int r = 1; r < 8; ++r) slice_bwd_pair(bu, bh, bg, b + r, mir.pm - r, sl_rot16(w0, r));
            // legs 0: the partner is leg 15, or where k2's low digits are zero a leg of the same number
            const int i0 = b + self, j0 = mir.p0 + self;
            slice_bwd_pair(bu, bh, bg, i0, j0, self ? make_float2(-w0.x, -w0.y) : w0);
            if (own) slice_bwd_pair(bu, bh, bg, b + 8, b + 8, make_float2(-w0.x, -w0.y));
        }
        sync();
        S::template inv_pass<2, sl_ndig(L2) - 1, 3>(bu, tw, t);
        S::template inv_mid<3>(bu, tw, t, sync);
        sync();
        // dq = dy * (h conv u)
        {
            SlPair<T, EVEN> gate[P0::IPT][NU];
#pragma unroll
            for (int i = 0; i < P0::IPT; ++i) {
                const SliceLegs<S> lg(g, P0::base(t + i * S::T), on);
#pragma unroll
                for (int r = 0; r < NU; ++r) gate[i][r].load(dy + lg.at(r), r < lg.na, r < lg.nb);
            }
            T *dq = (T *)p.dq + so;
            S::template inv_last<!FULL>(bu, tw, t, [&](int i, int r, int, float2 w) {
                const SliceLegs<S> lg(g, P0::base(t + i * S::T), on);
                const float2 a = gate[i][r].get();
                SlPair<T, EVEN>::store(dq + lg.at(r), make_float2(w.x * sc * a.x, w.y * sc * a.y), r < lg.na, r < lg.nb);
            });
        }
        // dk = v du, dv = k du
        {
            SlPair<T, EVEN> gk[P0::IPT][NU], gv[P0::IPT][NU];
#pragma unroll
            for (int i = 0; i < P0::IPT; ++i) {
                const SliceLegs<S> lg(g, P0::base(t + i * S::T), on);
#pragma unroll
                for (int r = 0; r < NU; ++r) {
                    gk[i][r].load(k + lg.at(r), r < lg.na, r < lg.nb);
                    gv[i][r].load(v + lg.at(r), r < lg.na, r < lg.nb);
                }
            }
            T *dk = (T *)p.dk + so, *dv = (T *)p.dv + so;
            S::template inv_last<!FULL>(bh, tw, t, [&](int i, int r, int, float2 w) {
                const SliceLegs<S> lg(g, P0::base(t + i * S::T), on);
                const float2 a = gk[i][r].get(), b = gv[i][r].get(), d = make_float2(w.x * sc, w.y * sc);
                SlPair<T, EVEN>::store(dk + lg.at(r), make_float2(d.x * b.x, d.y * b.y), r < lg.na, r < lg.nb);
                SlPair<T, EVEN>::store(dv + lg.at(r), make_float2(d.x * a.x, d.y * a.y), r < lg.na, r < lg.nb);
            });
        }
        // dh: the ring position of a displacement is where the taps were read from
        {
            const long long ho = s * g.kvol;
            auto taps_out = [&](auto *dh) {
                S::template inv_last<false>(bg, tw, t, [&](int, int, int idx, float2 w) { slice_tap_store<S>(dh + ho, g, idx, on, make_float2(w.x * sc, w.y * sc)); });
            };
            if (p.dh_f32) taps_out((float *)p.dh); else taps_out((T *)p.dh);
        }
        // (the next slice's first pass writes where this thread has just read)
    }
}

template <typename T, int L0, int L1, int L2, bool FULL, bool EVEN> int launch_slice_bwd_t(const SliceBwdArgs &a, cudaStream_t st)
{
    using CT = SliceCta<SliceFft<L0, L1, L2>>;
    constexpr size_t sm = CT::smem(3);
    auto fn = slice_bwd_kernel<T, L0, L1, L2, FULL, EVEN>;
    static int resident[64];
    const int slots = slice_resident(resident, (const void *)fn, CT::CT, sm);
    if (slots <= 0) return -1;
    const long long ctas = (a.slices + CT::NG - 1) / CT::NG;
    if (ctas <= 0) return 0;
    launch_pdl(fn, (unsigned)(ctas < slots ? ctas : slots), CT::CT, sm, st, a);
    return 1;
}

template <typename T, int A, int B, int C> int launch_slice_bwd_d(const SliceBwdArgs &a, cudaStream_t st)
{
    if (a.g.full) return launch_slice_bwd_t<T, A, B, C, true, true>(a, st);
    return (a.g.L[2] & 1) ? launch_slice_bwd_t<T, A, B, C, false, false>(a, st) : launch_slice_bwd_t<T, A, B, C, false, true>(a, st);
}
#define HN_SLICE_BWD_CASE(A, B, C)                                                                         \
    if (a.g.l0 == A && a.g.l1 == B && a.g.l2 == C) return launch_slice_bwd_d<HN_SLICE_T, A, B, C>(a, st);

int launch_slice_bwd_1d_f32(const SliceBwdArgs &a, cudaStream_t st);
int launch_slice_bwd_1d_bf16(const SliceBwdArgs &a, cudaStream_t st);
int launch_slice_bwd_2d_f32(const SliceBwdArgs &a, cudaStream_t st);
int launch_slice_bwd_2d_bf16(const SliceBwdArgs &a, cudaStream_t st);
int launch_slice_bwd_3d_f32(const SliceBwdArgs &a, cudaStream_t st);
int launch_slice_bwd_3d_bf16(const SliceBwdArgs &a, cudaStream_t st);

}  // namespace hn
