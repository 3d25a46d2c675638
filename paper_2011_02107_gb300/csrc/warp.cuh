// Warp sums and the paired double-float accesses of the stencil kernels.
#pragma once

#include "common.cuh"

namespace dacp {

__device__ __forceinline__ df32 shfl_xor_df(df32 v, int o) {
    return df32(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}

__device__ __forceinline__ df32 warp_shfl_xor(df32 v, int o) { return shfl_xor_df(v, o); }

// Sums V = 2^v values (double-float, or any type with + and warp_shfl_xor) per lane over the lanes of a warp and
// scatters the totals (a reduce-scatter butterfly): at each of the first v
// levels (lane offsets 16, 8, ...) a lane keeps the half of its values that its
// lane bit selects and adds the partner's copy of that half; the offsets left,
// down to OMIN, sum the one value kept. On return (OMIN = 1) lane L holds the
// total of value L / (32 / V), every lane of a group of 32 / V the same; with
// OMIN > 1 lanes that differ below OMIN keep separate sums. For V = 32 this is
// 31 double-float additions per lane on the float32 pipes, where a float64
// butterfly per value takes 5 V float64 additions: GB300 issues float64 at
// 1/64 of the float32 rate, and that once-per-tile reduction used to bound the
// float32 evolution kernel.
template <int V, int OMIN = 1, typename T>
__device__ __forceinline__ T warp_reduce_scatter(T (&x)[V], const int lane) {
    static_assert((V & (V - 1)) == 0 && V <= 32 / OMIN, "V a power of two, at most the lanes summed over");
#pragma unroll
    for (int half = V / 2, o = 16; half >= 1; half >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const T send = up ? x[i] : x[i + half];
            const T keep = up ? x[i + half] : x[i];
            x[i] = keep + warp_shfl_xor(send, o);
        }
    }
    T v = x[0];
#pragma unroll
    for (int o = 16 / V; o >= OMIN; o >>= 1) v = v + warp_shfl_xor(v, o);
    return v;
}

// The 16 bytes of a column pair are (hi_p, hi_{p+1} | lo_p, lo_{p+1}): the two
// register pairs of a DF2 as they are.
__device__ __forceinline__ DF2 ld_df2_s(const df32* p) {
    const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(p);
    return DF2{f.x, f.y};
}

template <bool COHERENT>
__device__ __forceinline__ DF2 ld_df2_g(const df32* p) {
    const ulonglong2 f = COHERENT ? __ldcg(reinterpret_cast<const ulonglong2*>(p))
                                  : __ldg(reinterpret_cast<const ulonglong2*>(p));
    return DF2{f.x, f.y};
}

template <bool COHERENT>
__device__ __forceinline__ DF2 ld_df2_rw(const df32* p) {
    const ulonglong2 f = COHERENT ? __ldcg(reinterpret_cast<const ulonglong2*>(p))
                                  : *reinterpret_cast<const ulonglong2*>(p);
    return DF2{f.x, f.y};
}

__device__ __forceinline__ void st_df2(df32* p, DF2 v) {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.hi, v.lo);
}

// lanes swapped: (x1 | x0)
__device__ __forceinline__ DF2 df2_swap(DF2 v) {
    float h0, h1, l0, l1;
    upk2(v.hi, h0, h1);
    upk2(v.lo, l0, l1);
    return DF2{pk2(h1, h0), pk2(l1, l0)};
}

__device__ __forceinline__ DF2 df2_shfl_xor(DF2 v, int o) {
    float h0, h1, l0, l1;
    upk2(v.hi, h0, h1);
    upk2(v.lo, l0, l1);
    return DF2{pk2(__shfl_xor_sync(0xffffffffu, h0, o), __shfl_xor_sync(0xffffffffu, h1, o)),
               pk2(__shfl_xor_sync(0xffffffffu, l0, o), __shfl_xor_sync(0xffffffffu, l1, o))};
}

// Moment sums of one state on its two threads (b = 4): thread h has the state's column pair h of
// w_k (A), of w_{k+1} (O), and the other pair of w_k (Cx).
// h = 0: (x0 x0 | x1 x1), (o0 x0 | o1 x1), (x0 x1 | o0 x1), (o0 x2 | o1 x3), (o0 x3 | o1 x2)
// h = 1: the same with columns 2, 3 for 0, 1, and <x_p, x_q> across the pairs
__device__ __forceinline__ void df4_moments_within(Dot2x2 (&mp)[3], DF2 A, DF2 O) {
    const DF2m Am = df2m(A);
    dot2x2_mad(mp[0], Am, A);
    dot2x2_mad(mp[1], Am, O);
    float ah0, ah1, al0, al1, oh0, oh1, ol0, ol1;
    upk2(A.hi, ah0, ah1);
    upk2(A.lo, al0, al1);
    upk2(O.hi, oh0, oh1);
    upk2(O.lo, ol0, ol1);
    const DF2 X01 = DF2{pk2(ah0, oh0), pk2(al0, ol0)};
    dot2x2_mad(mp[2], df2m(X01), DF2{pk2(ah1, ah1), pk2(al1, al1)});
}
__device__ __forceinline__ void df4_moments_across(Dot2x2 (&mp)[2], DF2 A, DF2 O, DF2 Cx, int h) {
    const DF2 U = h ? Cx : O, V = h ? A : Cx;
    const DF2m Um = df2m(U);
    dot2x2_mad(mp[0], Um, V);
    dot2x2_mad(mp[1], Um, df2_swap(V));
}

// The warp's ten sums per column pair, in the order (x0x0, x0x1, x1x1, o0x0, o0x1, o1x1, u0v0, u0v1,
// u1v0, u1v1); columns shifted by two for h = 1. The lane keeps sum e (e < 10) of its pair.
__device__ __forceinline__ df32 df4_warp_moments(const Dot2x2 (&in)[3], const Dot2x2 (&ac)[2], int lane, int& e) {
    Dot2 ms[10];
    dot2x2_split(in[0], ms[0], ms[2]);
    dot2x2_split(in[1], ms[3], ms[5]);
    dot2x2_split(in[2], ms[1], ms[4]);
    dot2x2_split(ac[0], ms[6], ms[9]);
    dot2x2_split(ac[1], ms[7], ms[8]);
    df32 xs[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) xs[i] = i < 10 ? dot2_final(ms[i]) : df32(0.f, 0.f);
    e = (lane >> 1) & 15;
    return warp_reduce_scatter<16, 2>(xs, lane);
}

// The two (equal) entries of sum e of pair h in the rows [<x_p, x_q>, <o_p, x_q>].
__device__ __forceinline__ int2 df4_moment_entry(int e, int h) {
    int blk, p, q;
    if (e < 6) {
        blk = e / 3;
        const int k = e % 3;
        p = 2 * h + (k == 2 ? 1 : 0);
        q = 2 * h + (k >= 1 ? 1 : 0);
    } else {
        blk = h == 0 ? 1 : 0;
        p = (e - 6) >> 1;
        q = 2 + ((e - 6) & 1);
    }
    return make_int2(blk * 16 + p * 4 + q, blk * 16 + q * 4 + p);
}

}  // namespace dacp
