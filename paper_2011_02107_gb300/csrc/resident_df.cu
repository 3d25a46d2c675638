// The double-float b = 4 evolution w_{k+1} = 2 G w_k - w_{k-1} (Sec. II B) with
// both vectors of a realization resident in shared memory for the whole run.
//
// A cluster owns one realization, one CTA per tile of the per-order launch
// (2^(N - TB) tiles of 2^TB states). Its tiles of w_k and w_{k-1} (overwritten
// by w_{k+1}) and its diagonal stay in shared memory from the first order to
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
    const ulonglong2* g2 = reinterpret_cast<const ulonglong2*>(gam_s);
    const uint64_t* ng2 = reinterpret_cast<const uint64_t*>(ngam_s);
    const bool gflip = a.gflip != nullptr;
    // 2 / E_max in every order: order 0 (w_1 = G w_0) takes half of its sum, which is exact
    const df32 ch = static_cast<df32>(2.0 / a.emax[r]);

    if (tid < R.N) {
        const df32 g = ch * a.gam[r * kMaxSpins + tid];
        gam_s[tid] = make_float4(g.hi, g.hi, g.lo, g.lo);
        ngam_s[tid] = make_float2(-g.hi, -g.hi);
    }
    if (tid == kMaxSpins && gflip) {
        const df32 g = ch * df32(a.gflip[r]);
        gam_s[kMaxSpins] = make_float4(g.hi, g.hi, g.lo, g.lo);
        ngam_s[kMaxSpins] = make_float2(-g.hi, -g.hi);
    }
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
                auto at = [&](const int sl) {
                    const ulonglong2 v = cur[sl];
                    return DF2{v.x, v.y};
                };
                auto coef = [&](const int i) { return DF2m{g2[i].x, ng2[i], g2[i].y}; };
                DF2 A[U], P[3][U];
                Dot2x2 acc[U];
#pragma unroll
                for (int u = 0; u < U; ++u) A[u] = at(base + kDfThreads * u);
                // partner tiles: loaded now, summed after the flips inside the tile
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const bool flip = j >= nb;               // the first slot past the bits: the global flip
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
                    const DF2m g = coef(0);
#pragma unroll
                    for (int u = 0; u < U; ++u) acc[u] = dot2x2_prod(g, at((base + kDfThreads * u) ^ 2));
                }
#pragma unroll
                for (int i = 1; i < TB; ++i) {
                    const DF2m g = coef(i);
                    // the bit's distance in slots; two of them lie among the thread's own slots
                    const int dist = 2 << i, du = dist / kDfThreads;
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        dot2x2_mad(acc[u], g, du >= 1 && du < U ? A[u ^ du] : at((base + kDfThreads * u) ^ dist));
                }
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    if (j < nb || (j == nb && gflip && nb > 0)) {
                        const DF2m g = coef(j < nb ? TB + j : kMaxSpins);
#pragma unroll
                        for (int u = 0; u < U; ++u) dot2x2_mad(acc[u], g, P[j][u]);
                    }
                }
                if (gflip && (nb == 0 || nb == 3)) {         // one tile, or no early slot left
                    const DF2m g = coef(kMaxSpins);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int sl = (base + kDfThreads * u) ^ (kSlots - 2);
                        const ulonglong2 v = nb == 0 ? cur[sl] : __ldcg(pcur + (rank ^ ((1 << nb) - 1)) * kSlots + sl);
                        dot2x2_mad(acc[u], g, DF2{v.x, v.y});
                    }
                }
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

template <int TB>
cudaError_t launch_df4_resident(const DfResArgs& a, int count, cudaStream_t st) {
    auto* f = evolve_df4_resident_kernel<TB>;
    const int smem = 72 << TB;                      // two vectors of 32 bytes a state and the diagonal
    cudaError_t e = grow_smem_attr(reinterpret_cast<const void*>(f), smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(count) << a.lg);
    cfg.blockDim = dim3(kDfThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << a.lg;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = a.lg > 0 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, f, a);
}

}  // namespace

// Tiles of 2^10 or 2^11 states (the sizes of tile_step_df4x2 whose two vectors and diagonal fit shared
// memory, 147 KB), at most 8 of them to a realization (a portable cluster).
bool df4_resident_fits(int tbits_uniform, int max_N) {
    return (tbits_uniform == 10 || tbits_uniform == 11) && max_N - tbits_uniform <= 3;
}

// Evolve the realizations a.list[0 .. count) in 2^a.lg CTAs each.
cudaError_t launch_evolve_df4_resident(int tbits, const DfResArgs& a, int count, cudaStream_t st) {
    switch (tbits) {
        case 10: return launch_df4_resident<10>(a, count, st);
        case 11: return launch_df4_resident<11>(a, count, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dacp
