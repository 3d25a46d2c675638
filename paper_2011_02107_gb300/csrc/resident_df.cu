// The double-float b = 4 recurrences, filter (Sec. II A) and evolution (Sec. II B), with
// the vectors of a realization resident in shared memory for the whole run.
//
// A cluster owns one realization, one CTA per tile of the per-order launch
// (2^(N - TB) tiles of 2^TB states). Its tiles of w_k and w_{k-1} (overwritten
// by w_{k+1}; the filter also of u = H w_k) and its diagonal stay in shared memory from the first order to
// the last, and one cluster barrier (0.23 us) separates the orders. A flip of
// a bit beyond the tile, and the global flip, reads the partner CTA's tile:
// each CTA also publishes its new tile to global memory, where it stays in L2
// (60 bytes per clock and SM, against 16 through distributed shared memory,
// both measured with 16-byte loads).
//
// Every vector and moment has the bits of tile_step_df4x2 (stencil.cu): the
// flips in rising bit order, the global flip, the diagonal, w_{k-1}; the moments
// of slots t, t + 256, ... of a tile make one running sum, 32 of these a warp's,
// the warps' sums are added in order and then the tiles'. The levels that the learned
// parameters resolve worst move with the last bits of the moments, so the
// launch a handle happens to take must not show in its results.

#include "common.cuh"
#include "ops.h"
#include "warp.cuh"

namespace dacp {

namespace {

constexpr int kDfThreads = 2 * kThreads;
constexpr int kRedRing = 3, kPartRing = 4;          // orders in flight between a sum and its moment row
constexpr int kRowSums = 32;                        // two rows of 4 x 4

// Scaled x-fields in shared memory, per spin (g.hi, g.hi, g.lo, g.lo) and (-g.hi, -g.hi): the register
// pairs of a DF2m. Entry kMaxSpins is the global flip.
struct Df4Fields {
    const ulonglong2* g;
    const uint64_t* ng;
    __device__ __forceinline__ DF2m operator[](const int i) const { return DF2m{g[i].x, ng[i], g[i].y}; }
};

__device__ __forceinline__ void df4_load_fields(float4* g_s, float2* ng_s, const df32 ch, const df32* gam,
                                                const double* gflip, const int N) {
    const int i = threadIdx.x;
    if (i < N || (i == kMaxSpins && gflip)) {
        const df32 g = ch * (i < N ? gam[i] : df32(*gflip));
        g_s[i] = make_float4(g.hi, g.hi, g.lo, g.lo);
        ng_s[i] = make_float2(-g.hi, -g.hi);
    }
}

// The flips of U slots (base, base + kDfThreads, ...) of the tile `cur`, in rising bit order, then the global
// flip; A: the slots themselves. pcur: the realization's published vector.
template <int TB, int U>
__device__ __forceinline__ void df4_flips(const ulonglong2* cur, const ulonglong2* pcur, const int base, const int rank,
                                          const int nb, const bool gflip, const Df4Fields gam, DF2 (&A)[U],
                                          Dot2x2 (&acc)[U]) {
    constexpr int kSlots = 2 << TB;
    auto at = [&](const int sl) {
        const ulonglong2 v = cur[sl];
        return DF2{v.x, v.y};
    };
    DF2 P[3][U];
#pragma unroll
    for (int u = 0; u < U; ++u) A[u] = at(base + kDfThreads * u);
    // partner tiles: loaded now, summed after the flips inside the tile
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const bool flip = j >= nb;                   // the first slot past the bits: the global flip
        if (j < nb || (j == nb && gflip && nb > 0)) {
            const ulonglong2* pp = pcur + (flip ? rank ^ ((1 << nb) - 1) : rank ^ (1 << j)) * kSlots;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int sl = base + kDfThreads * u;
                const ulonglong2 v = __ldcg(pp + (flip ? sl ^ (kSlots - 2) : sl));
                P[j][u] = DF2{v.x, v.y};
            }
        }
    }
    {
        const DF2m g = gam[0];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = dot2x2_prod(g, at((base + kDfThreads * u) ^ 2));
    }
#pragma unroll
    for (int i = 1; i < TB; ++i) {
        const DF2m g = gam[i];
        // the bit's distance in slots; two of them lie among the thread's own slots
        const int dist = 2 << i, du = dist / kDfThreads;
#pragma unroll
        for (int u = 0; u < U; ++u)
            dot2x2_mad(acc[u], g, du >= 1 && du < U ? A[u ^ du] : at((base + kDfThreads * u) ^ dist));
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if (j < nb || (j == nb && gflip && nb > 0)) {
            const DF2m g = gam[j < nb ? TB + j : kMaxSpins];
#pragma unroll
            for (int u = 0; u < U; ++u) dot2x2_mad(acc[u], g, P[j][u]);
        }
    }
    if (gflip && (nb == 0 || nb == 3)) {             // one tile, or no early slot left
        const DF2m g = gam[kMaxSpins];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int sl = (base + kDfThreads * u) ^ (kSlots - 2);
            const ulonglong2 v = nb == 0 ? cur[sl] : __ldcg(pcur + (rank ^ ((1 << nb) - 1)) * kSlots + sl);
            dot2x2_mad(acc[u], g, DF2{v.x, v.y});
        }
    }
}

__device__ __forceinline__ void df4_cluster_sync(const bool cluster) {
    if (cluster) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}

// Bound by the float32 pipe (248 lane operations per value and order at 13 spins and a global flip).
// Two passes an order, so that 16 warps of an SM work although the moments have 256 running sums of
// 10: first w_{k+1}, U slots (column pairs of a state) of a thread at a time, kDfThreads apart, so that the
// flips of two bits are register operands and a coefficient is read once per U slots; then the moments
// from shared memory, six of the ten sums on the first 256 threads and four on the others. (One pass on
// 256 threads: 12.9 us an order and wave with U = 4, 11.4 with U = 8 and 255 registers, against 16.3k
// clocks = 7.9 us of float32 work.) The sums of an order travel warp -> CTA -> cluster -> moment row one
// barrier at a time, on the last warp between its arrival and its wait, so no order waits for them.
template <int TB>
__global__ void __launch_bounds__(kDfThreads, 1) evolve_df4_resident_kernel(const DfResArgs a) {
    constexpr int kSlots = 2 << TB, NI = kSlots / kDfThreads, U = NI < 4 ? NI : 4;
    static_assert(NI >= 1, "a tile gives every thread a slot");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // per spin: (g.hi, g.hi, g.lo, g.lo) and (-g.hi, -g.hi), the register pairs of a DF2m
    __shared__ __align__(16) float4 gam_s[kMaxSpins + 1];        // slot kMaxSpins: the global flip
    __shared__ __align__(8) float2 ngam_s[kMaxSpins + 1];
    __shared__ double red_s[kRedRing][kThreads / 32][kRowSums];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, h = tid & 1;
    const int G = 1 << a.lg;
    const int group = blockIdx.x >> a.lg, rank = blockIdx.x & (G - 1);
    const int r = a.list[group];
    const RealInfo R = a.real[r];
    const int nb = R.N - TB;                                     // bits beyond the tile
    const bool active = rank < (1 << nb);
    const int orders = R.ne;
    ulonglong2* buf0 = reinterpret_cast<ulonglong2*>(smem_raw);
    ulonglong2* buf1 = buf0 + kSlots;
    df32* diag_s = reinterpret_cast<df32*>(buf1 + kSlots);
    const int64_t slot0 = R.off * 2 + static_cast<int64_t>(rank) * kSlots;
    const Df4Fields gam{reinterpret_cast<const ulonglong2*>(gam_s), reinterpret_cast<const uint64_t*>(ngam_s)};
    const bool gflip = a.gflip != nullptr;
    // 2 / E_max in every order: order 0 (w_1 = G w_0) takes half of its sum, which is exact
    const df32 ch = static_cast<df32>(2.0 / a.emax[r]);

    df4_load_fields(gam_s, ngam_s, ch, a.gam + r * kMaxSpins, gflip ? a.gflip + r : nullptr, R.N);
    if (active) {
        const ulonglong2* psi = static_cast<const ulonglong2*>(a.psi) + slot0;
        for (int i = tid; i < kSlots; i += kDfThreads) {
            const ulonglong2 v = psi[i];
            buf0[i] = v;
            if (nb > 0) a.pub0[slot0 + i] = v;
        }
        for (int i = tid; i < (1 << TB); i += kDfThreads)
            diag_s[i] = ch * a.diag[R.off + (static_cast<int64_t>(rank) << TB) + i];
    }

    double* part = a.part + static_cast<int64_t>(group) * kPartRing * G * kRowSums;
    // while order k's barrier is open: the CTA's sums of order k - 1, and the rows of order k - 3, whose
    // partials every CTA wrote before barrier k - 1. The warp may run behind by one order, hence the rings.
    auto moments_behind = [&](const int k) {
        if (active && k >= 1 && k <= orders) {
            double s = 0.0;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) s += red_s[(k - 1) % kRedRing][w][lane];
            __stcg(part + ((k - 1) % kPartRing * G + rank) * kRowSums + lane, s);
        }
        if (rank == 0 && k >= 3 && k - 3 < orders) {
            double s = 0.0;
            for (int j = 0; j < (1 << nb); ++j) s += __ldcg(part + ((k - 3) % kPartRing * G + j) * kRowSums + lane);
            a.mom[(R.mom_off + 2 * static_cast<int64_t>(k - 3)) * 16 + lane] = s;
        }
    };
    // sum e (of ten) of the warp's pair half h, as the two (equal) entries of its rows
    auto put_sum = [&](const int k, const int w, const int e, const df32 t, const bool valid) {
        if (!valid) return;
        const int2 pq = df4_moment_entry(e, h);
        red_s[k % kRedRing][w][pq.x] = static_cast<double>(t);
        red_s[k % kRedRing][w][pq.y] = static_cast<double>(t);
    };
    auto sync = [&](const int k) {
        const bool last = warp == kDfThreads / 32 - 1;
        if (a.lg > 0) {
            // (An arrival before the moments, its wait after them, was slower, 12.2 against 11.4 us an order:
            // its release waits for the stores just issued.)
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            if (last) moments_behind(k);
            __syncwarp();
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else {
            if (last) moments_behind(k);
            __syncthreads();
        }
    };
    sync(0);

    for (int k = 0; k < orders; ++k) {
        const ulonglong2* cur = (k & 1) ? buf1 : buf0;
        ulonglong2* oth = (k & 1) ? buf0 : buf1;
        const ulonglong2* pcur = ((k & 1) ? a.pub1 : a.pub0) + R.off * 2;
        ulonglong2* pnew = ((k & 1) ? a.pub0 : a.pub1) + slot0;
        if (active) {
#pragma unroll 1
            for (int base = tid; base < kSlots; base += kDfThreads * U) {
                DF2 A[U];
                Dot2x2 acc[U];
                df4_flips<TB, U>(cur, pcur, base, rank, nb, gflip, gam, A, acc);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int sl = base + kDfThreads * u;
                    dot2x2_mad(acc[u], df2m_bcast(diag_s[sl >> 1]), A[u]);
                    if (k > 0) {
                        const ulonglong2 y = oth[sl];
                        dot2x2_sub(acc[u], DF2{y.x, y.y});
                    }
                    DF2 O = dot2x2_final(acc[u]);
                    if (k == 0) {
                        const uint64_t half = pk2(0.5f, 0.5f);
                        O = DF2{mul2(O.hi, half), mul2(O.lo, half)};
                    }
                    oth[sl] = make_ulonglong2(O.hi, O.lo);
                    if (nb > 0) pnew[sl] = make_ulonglong2(O.hi, O.lo);
                }
            }
            __syncthreads();
            const int cls = tid & (kThreads - 1);                // running sum of slots cls, cls + 256, ...
            if (tid < kThreads) {
                Dot2x2 mp[3];
#pragma unroll
                for (int e = 0; e < 3; ++e) mp[e] = Dot2x2{0ull, 0ull};
#pragma unroll 4
                for (int sl = cls; sl < kSlots; sl += kThreads) {
                    const ulonglong2 av = cur[sl], ov = oth[sl];
                    df4_moments_within(mp, DF2{av.x, av.y}, DF2{ov.x, ov.y});
                }
                Dot2 ms[6];
                dot2x2_split(mp[0], ms[0], ms[2]);
                dot2x2_split(mp[1], ms[3], ms[5]);
                dot2x2_split(mp[2], ms[1], ms[4]);
                df32 xs[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) xs[e] = e < 6 ? dot2_final(ms[e]) : df32(0.f, 0.f);
                put_sum(k, warp, lane >> 2, warp_reduce_scatter<8, 2>(xs, lane), (lane >> 2) < 6);
            } else {
                Dot2x2 mp[2] = {Dot2x2{0ull, 0ull}, Dot2x2{0ull, 0ull}};
#pragma unroll 4
                for (int sl = cls; sl < kSlots; sl += kThreads) {
                    const ulonglong2 av = cur[sl], ov = oth[sl];
                    const DF2 A = DF2{av.x, av.y};
                    df4_moments_across(mp, A, DF2{ov.x, ov.y}, df2_shfl_xor(A, 1), h);
                }
                Dot2 ms[4];
                dot2x2_split(mp[0], ms[0], ms[3]);
                dot2x2_split(mp[1], ms[1], ms[2]);
                df32 xs[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) xs[e] = dot2_final(ms[e]);
                put_sum(k, warp - kThreads / 32, 6 + (lane >> 3), warp_reduce_scatter<4, 2>(xs, lane), true);
            }
        }
        sync(k);
    }
    for (int k = orders; k < orders + 3; ++k) sync(k);
}

// The filter's recurrence w_{k+1} = 2 F w_k - w_{k-1}, F = (H^2 - E_c) / E_0 (Sec. II A), with w_k, w_{k-1}
// (overwritten by w_{k+1}), u = H w_k and the diagonal resident: two passes and two cluster barriers an order.
// w_K ends in pub0 (K even) or pub1 (K odd), as the per-order launch leaves it. pub0 holds w_0 at the start.
// Bound by the float32 pipe, its issue and the last round of clusters: 500 orders of 64 sectors of 13 spins
// (36 clusters at a time) take 22.2 ms, 29.4 as two launches an order; the filter of 512, 715 orders at most,
// 149 and 166 ms.
template <int TB>
__global__ void __launch_bounds__(kDfThreads, 1) filter_df4_resident_kernel(const DfResArgs a) {
    constexpr int kSlots = 2 << TB, NI = kSlots / kDfThreads, U = NI < 4 ? NI : 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) float4 gam_s[2][kMaxSpins + 1];     // of u = H w_k, and of w_{k+1}
    __shared__ __align__(8) float2 ngam_s[2][kMaxSpins + 1];

    const int tid = threadIdx.x;
    const int group = blockIdx.x >> a.lg, rank = blockIdx.x & ((1 << a.lg) - 1);
    const int r = a.list[group];
    const RealInfo R = a.real[r];
    const int nb = R.N - TB;
    const bool active = rank < (1 << nb);
    const int orders = R.nf;
    ulonglong2* buf0 = reinterpret_cast<ulonglong2*>(smem_raw);
    ulonglong2* buf1 = buf0 + kSlots;
    ulonglong2* bufu = buf1 + kSlots;
    df32* diag_s = reinterpret_cast<df32*>(bufu + kSlots);
    const int64_t slot0 = R.off * 2 + static_cast<int64_t>(rank) * kSlots;
    const bool gflip = a.gflip != nullptr;
    // the coefficients of orders 1, 2, ...; order 0 takes half of their sum without w_{k-1}, which is exact
    const double* cf = a.coef + 8 * r + 3;
    const df32 ch = static_cast<df32>(cf[0]);
    const bool use1 = cf[1] != 0.0, sub1 = cf[1] == -1.0, use2 = cf[2] != 0.0, sub2v = cf[2] == -1.0;
    const DF2m C1 = df2m_bcast(static_cast<df32>(cf[1])), C2 = df2m_bcast(static_cast<df32>(cf[2]));
    for (int p = 0; p < 2; ++p)
        df4_load_fields(gam_s[p], ngam_s[p], p == 0 ? df32(1.0) : ch, a.gam + r * kMaxSpins, gflip ? a.gflip + r : nullptr,
                        R.N);
    if (active) {
        for (int i = tid; i < kSlots; i += kDfThreads) buf0[i] = a.pub0[slot0 + i];
        for (int i = tid; i < (1 << TB); i += kDfThreads)
            diag_s[i] = a.diag[R.off + (static_cast<int64_t>(rank) << TB) + i];
    }
    df4_cluster_sync(a.lg > 0);

    for (int k = 0; k < orders; ++k) {
        const ulonglong2* cur = (k & 1) ? buf1 : buf0;
        ulonglong2* oth = (k & 1) ? buf0 : buf1;
        const ulonglong2* pcur = ((k & 1) ? a.pub1 : a.pub0) + R.off * 2;
        ulonglong2* pnew = ((k & 1) ? a.pub0 : a.pub1) + slot0;
        for (int pass = 0; pass < 2; ++pass) {
            if (active) {
                const Df4Fields gam{reinterpret_cast<const ulonglong2*>(gam_s[pass]),
                                    reinterpret_cast<const uint64_t*>(ngam_s[pass])};
                const ulonglong2* x = pass == 0 ? cur : bufu;
                const ulonglong2* px = pass == 0 ? pcur : a.pubu + R.off * 2;
                ulonglong2* out = pass == 0 ? bufu : oth;
                ulonglong2* pout = pass == 0 ? a.pubu + slot0 : pnew;
                const df32 cd = pass == 0 ? df32(1.0) : ch;
                const bool publish = nb > 0 || (pass == 1 && k == orders - 1);
#pragma unroll 1
                for (int base = tid; base < kSlots; base += kDfThreads * U) {
                    DF2 A[U];
                    Dot2x2 acc[U];
                    df4_flips<TB, U>(x, px, base, rank, nb, gflip, gam, A, acc);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int sl = base + kDfThreads * u;
                        dot2x2_mad(acc[u], df2m_bcast(cd * diag_s[sl >> 1]), A[u]);
                        if (pass == 1) {
                            if (use1) {
                                const ulonglong2 y = cur[sl];
                                if (sub1) dot2x2_sub(acc[u], DF2{y.x, y.y});
                                else dot2x2_mad(acc[u], C1, DF2{y.x, y.y});
                            }
                            if (use2 && k > 0) {
                                const ulonglong2 z = oth[sl];
                                if (sub2v) dot2x2_sub(acc[u], DF2{z.x, z.y});
                                else dot2x2_mad(acc[u], C2, DF2{z.x, z.y});
                            }
                        }
                        DF2 O = dot2x2_final(acc[u]);
                        if (pass == 1 && k == 0) {
                            const uint64_t half = pk2(0.5f, 0.5f);
                            O = DF2{mul2(O.hi, half), mul2(O.lo, half)};
                        }
                        out[sl] = make_ulonglong2(O.hi, O.lo);
                        if (publish) pout[sl] = make_ulonglong2(O.hi, O.lo);
                    }
                }
            }
            df4_cluster_sync(a.lg > 0);
        }
    }
}

// Moments of one column (the kernel-polynomial pre-pass): a CTA owns a realization, with both vectors and the
// diagonal in shared memory, and no order needs more than the CTA's barrier. A slot holds two neighbouring
// states. The bits are those of tile_step<df32, 1, kEvolve> on tiles of 2^TB states: the diagonal, then the
// flips in rising bit order, the global flip, w_{k-1}; 256 running sums a tile, warps and tiles in order.
// Bound by the float32 pipe: 190 paired instructions per two states and order. As 64 launches of one pass each,
// the 512 tiles of 128 sectors of 13 spins waited on L2 and on the tail of every launch: the parameter choice of
// those sectors took 7.7 ms, and takes 4.8.
template <int TB>
__global__ void __launch_bounds__(kDfThreads, 1) moments_df1_resident_kernel(const DfResArgs a, const int orders,
                                                                             const int rows_fixed) {
    constexpr int kUnits = 1 << (TB - 1), U = kUnits / kThreads;     // slots of a tile, and of a thread
    static_assert(U >= 1, "a tile gives every thread a slot");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) float4 gam_s[kMaxSpins + 1];
    __shared__ __align__(8) float2 ngam_s[kMaxSpins + 1];
    __shared__ double red_s[2][8][kThreads / 32][2];                 // [order parity][tile][warp][xx, ox]

    const int tid = threadIdx.x, lane = tid & 31;
    const int r = a.list[blockIdx.x];
    const RealInfo R = a.real[r];
    const int slots = 1 << (R.N - 1), tiles = 1 << (R.N - TB);
    ulonglong2* buf0 = reinterpret_cast<ulonglong2*>(smem_raw);
    ulonglong2* buf1 = buf0 + slots;
    ulonglong2* diag_s = buf1 + slots;                               // (d0.hi, d1.hi | d0.lo, d1.lo)
    const Df4Fields gam{reinterpret_cast<const ulonglong2*>(gam_s), reinterpret_cast<const uint64_t*>(ngam_s)};
    const bool gflip = a.gflip != nullptr;
    const df32 ch = static_cast<df32>(2.0 / a.emax[r]);
    const df32* psi = static_cast<const df32*>(a.psi) + R.off;
    const df32* diag = a.diag + R.off;

    df4_load_fields(gam_s, ngam_s, ch, a.gam + r * kMaxSpins, gflip ? a.gflip + r : nullptr, R.N);
    auto pack = [](const df32 x, const df32 y) { return make_ulonglong2(pk2(x.hi, y.hi), pk2(x.lo, y.lo)); };
    for (int i = tid; i < slots; i += blockDim.x) {
        buf0[i] = pack(psi[2 * i], psi[2 * i + 1]);
        diag_s[i] = pack(ch * diag[2 * i], ch * diag[2 * i + 1]);
    }
    __syncthreads();
    double* mom = a.mom + static_cast<int64_t>(r) * rows_fixed;
    auto write_row = [&](const int k) {                              // lanes 0, 1: rows 2 k, 2 k + 1
        double tot = 0.0;
        for (int t = 0; t < tiles; ++t) {
            double s = 0.0;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) s += red_s[k & 1][t][w][lane];
            tot += s;
        }
        mom[2 * k + lane] = tot;
    };

    for (int k = 0; k < orders; ++k) {
        const ulonglong2* cur = (k & 1) ? buf1 : buf0;
        ulonglong2* oth = (k & 1) ? buf0 : buf1;
        auto at = [&](const int sl) {
            const ulonglong2 v = cur[sl];
            return DF2{v.x, v.y};
        };
        for (int t = tid / kThreads; t < tiles; t += blockDim.x / kThreads) {
            const int base = t * kUnits + (tid & (kThreads - 1));
            DF2 A[U];
            Dot2x2 acc[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                A[u] = at(base + kThreads * u);
                const ulonglong2 d = diag_s[base + kThreads * u];
                acc[u] = dot2x2_prod(df2m(DF2{d.x, d.y}), A[u]);
            }
            {
                const DF2m g = gam[0];
#pragma unroll
                for (int u = 0; u < U; ++u) dot2x2_mad(acc[u], g, df2_swap(A[u]));
            }
#pragma unroll 2
            for (int i = 1; i < R.N; ++i) {
                const DF2m g = gam[i];
#pragma unroll
                for (int u = 0; u < U; ++u) dot2x2_mad(acc[u], g, at((base + kThreads * u) ^ (1 << (i - 1))));
            }
            if (gflip) {
                const DF2m g = gam[kMaxSpins];
#pragma unroll
                for (int u = 0; u < U; ++u) dot2x2_mad(acc[u], g, df2_swap(at((base + kThreads * u) ^ (slots - 1))));
            }
            Dot2x2 ms = Dot2x2{0ull, 0ull};                          // (<x, x> | <o, x>)
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int sl = base + kThreads * u;
                if (k > 0) {
                    const ulonglong2 y = oth[sl];
                    dot2x2_sub(acc[u], DF2{y.x, y.y});
                }
                DF2 O = dot2x2_final(acc[u]);
                if (k == 0) {
                    const uint64_t half = pk2(0.5f, 0.5f);
                    O = DF2{mul2(O.hi, half), mul2(O.lo, half)};
                }
                oth[sl] = make_ulonglong2(O.hi, O.lo);
                const df32 x0 = df2_lane0(A[u]), x1 = df2_lane1(A[u]), o0 = df2_lane0(O), o1 = df2_lane1(O);
                dot2x2_mad(ms, df2m(DF2{pk2(x0.hi, o0.hi), pk2(x0.lo, o0.lo)}), DF2{pk2(x0.hi, x0.hi), pk2(x0.lo, x0.lo)});
                dot2x2_mad(ms, df2m(DF2{pk2(x1.hi, o1.hi), pk2(x1.lo, o1.lo)}), DF2{pk2(x1.hi, x1.hi), pk2(x1.lo, x1.lo)});
            }
            Dot2 s0, s1;
            dot2x2_split(ms, s0, s1);
            df32 v[2] = {dot2_final(s0), dot2_final(s1)};
            const df32 sum = warp_reduce_scatter<2>(v, lane);
            if ((lane & 15) == 0) red_s[k & 1][t][(tid & (kThreads - 1)) >> 5][lane >> 4] = static_cast<double>(sum);
        }
        __syncthreads();
        if (tid >= static_cast<int>(blockDim.x) - 32 && lane < 2) write_row(k);    // beside the next order
    }
}

template <int TB>
cudaError_t launch_moments_df1(const DfResArgs& a, int count, int max_N, int orders, int rows_fixed, cudaStream_t st) {
    auto* f = moments_df1_resident_kernel<TB>;
    const int smem = 24 << max_N;
    cudaError_t e = grow_smem_attr(reinterpret_cast<const void*>(f), smem);
    if (e != cudaSuccess) return e;
    f<<<count, max_N > TB ? kDfThreads : kThreads, smem, st>>>(a, orders, rows_fixed);
    return cudaGetLastError();
}

// Launch shape of `count` clusters of 2^lg CTAs; at: room for the cluster attribute.
cudaLaunchConfig_t df4_config(int TB, bool filter, int count, int lg, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(count) << lg);
    cfg.blockDim = dim3(kDfThreads);
    cfg.dynamicSmemBytes = (filter ? 104 : 72) << TB;     // three or two vectors of 32 bytes a state, and the diagonal
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << lg;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = lg > 0 ? 1 : 0;
    return cfg;
}

template <int TB>
cudaError_t launch_df4_resident(bool filter, const DfResArgs& a, int count, cudaStream_t st) {
    auto* f = filter ? filter_df4_resident_kernel<TB> : evolve_df4_resident_kernel<TB>;
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = df4_config(TB, filter, count, a.lg, at);
    cfg.stream = st;
    cudaError_t e = grow_smem_attr(reinterpret_cast<const void*>(f), static_cast<int>(cfg.dynamicSmemBytes));
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, f, a);
}

// Clusters of 2^lg CTAs of the filter, which takes the more shared memory, that the device holds at once.
template <int TB>
int df4_clusters(int lg) {
    auto* f = filter_df4_resident_kernel<TB>;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = df4_config(TB, true, 1, lg, at);
    int n = 0;
    if (grow_smem_attr(reinterpret_cast<const void*>(f), static_cast<int>(cfg.dynamicSmemBytes)) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace

// Tiles of 2^10 or 2^11 states (the sizes of tile_step_df4x2 whose two vectors and diagonal fit shared
// memory: 147 KB, with the filter's third vector 213 KB), at most 8 of them to a realization (a portable cluster).
bool df4_resident_fits(int tbits_uniform, int max_N) {
    return (tbits_uniform == 10 || tbits_uniform == 11) && max_N - tbits_uniform <= 3;
}

int df4_resident_clusters(int tbits, int lg) {
    switch (tbits) {
        case 10: return df4_clusters<10>(lg);
        case 11: return df4_clusters<11>(lg);
    }
    return 0;
}

// Filter or evolve the realizations a.list[0 .. count) in 2^a.lg CTAs each.
cudaError_t launch_df4_resident(int tbits, bool filter, const DfResArgs& a, int count, cudaStream_t st) {
    switch (tbits) {
        case 10: return launch_df4_resident<10>(filter, a, count, st);
        case 11: return launch_df4_resident<11>(filter, a, count, st);
    }
    return cudaErrorInvalidValue;
}

// Tiles of 2^9 to 2^11 states, and two vectors and the diagonal of a realization (24 bytes a state) in the
// shared memory of one CTA: up to 13 spins, in at most 8 tiles.
// Ahead at every batch size: the parameter choice of 1, 32, 152 and 512 sectors of 13 spins takes 3.5, 3.6, 4.2
// and 10.4 ms with it, 4.3, 4.7, 7.5 and 19.8 without (and without the kept scratch).
bool df1_resident_fits(int tbits_uniform, int max_N) {
    return tbits_uniform >= 9 && tbits_uniform <= 11 && max_N <= 13 && max_N - tbits_uniform <= 3;
}

// `orders` evolution orders of one column (a.psi) of the realizations a.list[0 .. count), rows at r * rows_fixed.
cudaError_t launch_moments_df1_resident(int tbits, const DfResArgs& a, int count, int max_N, int orders, int rows_fixed,
                                        cudaStream_t st) {
    switch (tbits) {
        case 9: return launch_moments_df1<9>(a, count, max_N, orders, rows_fixed, st);
        case 10: return launch_moments_df1<10>(a, count, max_N, orders, rows_fixed, st);
        case 11: return launch_moments_df1<11>(a, count, max_N, orders, rows_fixed, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dacp
