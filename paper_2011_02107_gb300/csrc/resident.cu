// The float64 Chebyshev evolution w_{k+1} = 2 G w_k - w_{k-1} (Sec. II B) with
// both vectors of a realization resident in shared memory for the whole run,
// in 59-bit fixed point on the integer multiply-add pipe.
//
// A group of 2^lg CTAs owns one realization: CTA `rank` holds the states whose
// top lg bits are `rank`. Its tile of w_k, its tile of w_{k-1} (overwritten by
// w_{k+1}) and its diagonal stay in shared memory from the first order to the
// last, and one group barrier separates the orders. A flip of one of the top
// lg bits (and the global flip) reads the partner CTA's tile: each CTA also
// publishes its new tile to global memory, where it stays in L2.
//
// Fixed point. A column of w_k has norm at most 1, because the spectrum of G
// lies in [-1, 1], so the values need no exponents: X = round(x 2^S) with one
// S per realization, |X| < 2^58, kept as two limbs X = xh 2^29 + xl with
// xl in [-2^28, 2^28). Coefficients are round(g 2^58) in the same limbs. A
// product then takes three 32 x 32 -> 64-bit multiply-adds (xh gh into one
// 64-bit sum, xh gl + xl gh into a second; xl gl is below the last place).
// GB300 takes 30 of them per clock and SM (measured) against 1.7 float64
// multiply-adds. The last place is 2^-58 of two to four times the largest |x|:
// an order's rounding is that of float64 in the norm of the vector, while its
// elements below 2^-6 of the largest keep fewer bits than in float64. Moments
// of 2000 orders at 10 spins came out 3 times closer to an 80-bit evaluation
// than in float64; levels of whole solves scatter as they do there (geometric
// mean over 24 start vectors 1.6e-11 against 1.4e-11 for the 10-spin chain,
// 6e-13 against 5e-13 and 4e-13 for sectors of 10 and 11 spins).
// The scale leaves 2 to 4 times the largest element as room. Random vectors
// stay inside; one whose elements are even (a product state, random signs)
// may concentrate and outgrow it, within some ten orders: the group then leaves
// the run (status kFxOutgrown) and is launched again with room for 32 to 64
// times the root mean square, the coarsest scale that any vector is given.
// Realizations that this does not suit leave status kFxUnsuited and are evolved
// by the floating-point kernels: a vector with an element above 16 times its
// root mean square, one that outgrows the coarse scale as well (E_max not a
// bound, or most of the norm in a few states), or couplings beyond the limbs.

#include <math.h>

#include <map>
#include <mutex>
#include <utility>

#include "common.cuh"
#include "ops.h"
#include "warp.cuh"

namespace dacp {

namespace {

constexpr int kFxMinTileBits = 3;      // states of a tile: at least 2^3 (fewer CTAs of the group work below that)
constexpr int kFxRedRing = 3, kFxPartRing = 4;   // orders in flight between a sum and its moment row
constexpr int kFxCheck = 32;           // orders between two looks at the overflow flag
constexpr uint64_t kFxWaitNs = 1000000000ull;

template <int B> struct FxSums { static constexpr int value = B == 4 ? 20 : (B == 2 ? 6 : 2); };

__device__ __forceinline__ uint64_t fx_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int2 fx_limbs(int64_t v) {
    const int lo = static_cast<int>(static_cast<uint32_t>(v) << 3) >> 3;
    return make_int2(static_cast<int>((v + (int64_t(1) << 28)) >> 29), lo);
}

__device__ __forceinline__ void fx_mad(int64_t& hh, int64_t& mm, const int2 g, const int xh, const int xl) {
    hh += static_cast<int64_t>(g.x) * xh;
    mm += static_cast<int64_t>(g.x) * xl;
    mm += static_cast<int64_t>(g.y) * xh;
}

// Moment sums of products of two values (both in limbs).
struct FxMom {
    int64_t hh, mm;
    __device__ __forceinline__ void mad(int ah, int al, int bh, int bl) {
        hh += static_cast<int64_t>(ah) * bh;
        mm += static_cast<int64_t>(ah) * bl;
        mm += static_cast<int64_t>(al) * bh;
    }
    // the sum in units of 2^58
    __device__ __forceinline__ int64_t value() const { return hh + ((mm + (int64_t(1) << 28)) >> 29); }
};

// A sum of moment products over lanes: hi 2^8 + lo, so that no vector can overflow it.
struct FxSum {
    int64_t hi;
    int lo;
};
__device__ __forceinline__ FxSum operator+(const FxSum a, const FxSum b) { return FxSum{a.hi + b.hi, a.lo + b.lo}; }
__device__ __forceinline__ FxSum warp_shfl_xor(const FxSum v, int o) {
    return FxSum{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ FxSum fx_sum(const int64_t v) { return FxSum{v >> 8, static_cast<int>(v & 255)}; }

// Barrier of the realization's group: the CTA alone, a cluster, or CTAs of a cooperative launch
// on a counter (bounded: false when one second passes, and then at every CTA of the group).
// `aux` runs on the CTA's last warp while the others wait (alone: before).
template <typename F>
__device__ __forceinline__ bool fx_group_sync(const FxArgs& a, const int group, const unsigned target, F aux) {
    const bool last = (threadIdx.x >> 5) == (blockDim.x >> 5) - 1;
    if (a.sync == kFxCluster) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (last) aux();
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return true;
    }
    if (a.sync == kFxAlone) {
        if (last) aux();
        __syncthreads();
        return true;
    }
    __shared__ int ok_s;
    __syncthreads();
    if (last) aux();
    if (threadIdx.x == 0) {
        unsigned* ctr = a.bar + group;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
        unsigned v;
        int ok = 1;
        const uint64_t t0 = fx_ns();
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
            if (v >= target) break;
            if (fx_ns() - t0 > kFxWaitNs) {
                ok = 0;
                atomicExch(a.err_flag, 2);
                break;
            }
        }
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// A 16-byte slot holds two consecutive values of [state][b]: a column pair of a
// state (b = 4: two slots per state, b = 2: one) or one column of two states (b = 1).
template <int B> __device__ __forceinline__ int fx_slot_bit(int i) { return B == 4 ? 2 << i : (B == 2 ? 1 << i : (1 << i) >> 1); }
template <int B> __device__ __forceinline__ int fx_slots(int states) { return B == 4 ? 2 * states : (B == 2 ? states : states >> 1); }

// Bound by the integer multiply-add pipe (62 multiply-adds per value and order at 13 spins and a
// global flip, b = 4), then by shared memory (14 16-byte accesses per two values). Each thread works
// on U slots at a time that differ in the top tile bits: their flips among each other are register
// operands, every coefficient is read from shared memory once per U slots, and U independent chains
// hide the multiply-add latency. The moment sums of an order travel warp -> CTA -> group -> moment row
// one barrier at a time, on one warp while it waits at the barrier, so no order waits for its sums.
template <int B, int U>
__global__ void __launch_bounds__(kFxThreads, 1) evolve_fx_kernel(const FxArgs a) {
    constexpr int NS = FxSums<B>::value;          // moment sums of a CTA
    constexpr int NT = B == 4 ? 10 : NS;          // of a thread
    constexpr int LU = U == 4 ? 2 : (U == 2 ? 1 : 0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int2 g_s[kMaxSpins + 1];            // 2 Gamma_i / E_max, then the global flip
    __shared__ FxSum red_s[kFxRedRing][kFxThreads / 32][NS];
    __shared__ float pro_s[3][kFxThreads / 32];
    __shared__ float max_s[4];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwork = blockDim.x, nwarps = nwork >> 5;
    const int G = 1 << a.lg;
    const int group = blockIdx.x >> a.lg, rank = blockIdx.x & (G - 1);
    const int r = a.list[group];
    const RealInfo R = a.real[r];
    const int lgr = R.N - kFxMinTileBits < a.lg ? (R.N > kFxMinTileBits ? R.N - kFxMinTileBits : 0) : a.lg;
    const bool active = rank < (1 << lgr);
    const int t = R.N - lgr, T = 1 << t, S = fx_slots<B>(T);
    const int64_t s0 = R.off + (static_cast<int64_t>(rank) << t);       // first state of the tile in the batch
    int4* buf0 = reinterpret_cast<int4*>(smem_raw);
    int4* buf1 = buf0 + a.slots_max;
    int2* diag_s = reinterpret_cast<int2*>(buf1 + a.slots_max);
    const int orders = a.nsteps_override > 0 ? a.nsteps_override : R.ne;
    const double emax = a.emax[r];
    unsigned target = 0;

    // ---- largest element, norm and diagonal of the realization -> scale ------------------------
    {
        float mx = 0.f, md = 0.f, ss = 0.f;
        if (active) {
            for (int i = tid; i < T * B; i += blockDim.x) {
                const float v = fabsf(static_cast<float>(a.psi[s0 * B + i]));
                mx = fmaxf(mx, v);
                ss = fmaf(v, v, ss);
            }
            for (int i = tid; i < T; i += blockDim.x) {
                const float v = fabsf(static_cast<float>(a.diag[s0 + i]));
                md = fmaxf(md, v);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
        }
        if (lane == 0) {
            pro_s[0][warp] = mx;
            pro_s[1][warp] = md;
            pro_s[2][warp] = ss;
        }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) {
                mx = fmaxf(mx, pro_s[0][w]);
                md = fmaxf(md, pro_s[1][w]);
                ss += pro_s[2][w];
            }
            __stcg(a.pro + (static_cast<int64_t>(group) << a.lg) + rank, make_float4(mx, md, ss, 0.f));
        }
        for (int i = tid; rank == 0 && i < kFxPartRing * NS; i += blockDim.x)
            __stcg(a.part + static_cast<int64_t>(group) * kFxPartRing * NS + i, make_longlong2(0, 0));
        if (!fx_group_sync(a, group, target += G, [] {})) return;
        if (warp == 0) {
            mx = md = ss = 0.f;
            for (int i = lane; i < G; i += 32) {
                const float4 v = __ldcg(a.pro + (static_cast<int64_t>(group) << a.lg) + i);
                mx = fmaxf(mx, v.x);
                md = fmaxf(md, v.y);
                ss += v.z;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
                ss += __shfl_xor_sync(0xffffffffu, ss, o);
            }
            if (lane == 0) {
                max_s[0] = mx;
                max_s[1] = md;
                max_s[2] = ss;
            }
        }
        __syncthreads();
    }
    const float mx = max_s[0], md = max_s[1], ss = max_s[2];
    int sexp = mx > 0.f ? 57 - (ilogbf(mx) + 1) : 0;                   // |x| < 2^(57 - sexp)
    const double c2 = 2.0 / emax;
    double gsum;
    bool fits = isfinite(ss) && mx > 0.f && isfinite(md) &&
                static_cast<double>(mx) * mx * ldexp(1.0, R.N) * B <= 256.0 * static_cast<double>(ss);
    {
        // sum of |coefficients| below 8: the limbs and the 64-bit sums hold
        double gs = md;
        for (int i = 0; i < R.N; ++i) gs += fabs(a.gam[r * kMaxSpins + i]);
        if (a.gflip) gs += fabs(a.gflip[r]);
        gsum = gs * c2;
        fits = fits && gsum < 7.9;
    }
    if (fits && a.coarse) {
        // 16 times the root mean square in the place of the largest element
        const int fine = sexp;
        sexp = 57 - (ilogb(16.0 * sqrt(static_cast<double>(ss) / (ldexp(1.0, R.N) * B))) + 1);
        fits = sexp < fine;
    }
    if (!fits) {                                    // the same at every CTA of the group
        if (rank == 0 && tid == 0) a.status[group] = kFxUnsuited;
        return;
    }
    // coefficients in units of 2^-(58 - ge): as fine as the sum of their magnitudes allows (limbs and 64-bit sums)
    const int ge = gsum < 3.95 ? 0 : 1;
    const double cg = ldexp(c2, 58 - ge);
    if (tid < R.N) g_s[tid] = fx_limbs(__double2ll_rn(cg * a.gam[r * kMaxSpins + tid]));
    if (tid == kMaxSpins) g_s[kMaxSpins] = a.gflip ? fx_limbs(__double2ll_rn(cg * a.gflip[r])) : make_int2(0, 0);
    const int64_t pslot0 = R.off * B / 2;           // the realization's first published slot (off is a multiple of 4)
    if (active) {
        const double sc = ldexp(1.0, sexp);
        for (int i = tid; i < T; i += blockDim.x)
            diag_s[i] = fx_limbs(__double2ll_rn(cg * a.diag[s0 + i]));
        for (int i = tid; i < S; i += blockDim.x) {
            const double* w = a.psi + s0 * B + 2 * i;            // 8-byte aligned only
            const int2 v0 = fx_limbs(__double2ll_rn(sc * w[0]));
            const int2 v1 = fx_limbs(__double2ll_rn(sc * w[1]));
            const int4 v = make_int4(v0.x, v0.y, v1.x, v1.y);
            buf0[i] = v;
            if (lgr > 0) a.pub0[pslot0 + static_cast<int64_t>(rank) * S + i] = v;
        }
    }
    if (!fx_group_sync(a, group, target += G, [] {})) return;

    const double unit = ldexp(1.0, 58 - 2 * sexp);
    const double square = ldexp(1.0 / 3.0, R.N + 56 - 2 * sexp);
    longlong2* part = a.part + static_cast<int64_t>(group) * kFxPartRing * NS;
    const int64_t row0 = a.mom_rows_fixed > 0 ? static_cast<int64_t>(r) * a.mom_rows_fixed : R.mom_off;
    // the rows of order k from the partials of its CTAs
    auto write_rows = [&](const int k) {
        if (lane < NS) {
            // exact integer sums over the CTAs, rounded once; the slot is free again for the order after next
            longlong2* slot = part + (k % kFxPartRing) * NS + lane;
            const longlong2 v = __ldcg(slot);
            __stcg(slot, make_longlong2(0, 0));
            double tot = unit * fma(static_cast<double>(v.x), 16777216.0, static_cast<double>(v.y));
            int blk, p, q;
            if (B == 4) {
                const int h = lane / 10, e = lane % 10;
                if (e < 6) {
                    blk = e / 3;
                    p = 2 * h + (e % 3 == 2 ? 1 : 0);
                    q = 2 * h + (e % 3 >= 1 ? 1 : 0);
                } else {
                    blk = h == 0 ? 1 : 0;
                    p = (e - 6) >> 1;
                    q = 2 + ((e - 6) & 1);
                }
            } else if (B == 2) {
                blk = lane / 3;
                p = lane % 3 == 2 ? 1 : 0;
                q = lane % 3 >= 1 ? 1 : 0;
            } else {
                blk = lane;
                p = q = 0;
            }
            // the dropped xl xl of a square is 2^56 / 3 in the mean
            if (blk == 0 && p == q) tot += square;
            double* m = a.mom + (row0 + 2 * static_cast<int64_t>(k) + blk) * B * B;
            m[p * B + q] = tot;
            m[q * B + p] = tot;
        }
    };

    // while order k's barrier is open: the CTA's sums of order k - 1, and the rows of order k - 3, whose
    // partials every CTA wrote before barrier k - 1. The warp may run behind by one order, hence the rings.
    auto moments_behind = [&](const int k) {
        if (active && lane < NS && k >= 1 && k <= orders) {
            long long hi = 0, lo = 0;
            for (int w = 0; w < nwarps; ++w) {
                const FxSum s = red_s[(k - 1) % kFxRedRing][w][lane];
                hi += s.hi >> 16;
                lo += (s.hi & 0xffff) * 256 + s.lo;
            }
            // integer sums: the order in which the CTAs add does not matter
            unsigned long long* slot = reinterpret_cast<unsigned long long*>(part + ((k - 1) % kFxPartRing) * NS + lane);
            atomicAdd(slot, static_cast<unsigned long long>(hi));
            atomicAdd(slot + 1, static_cast<unsigned long long>(lo));
        }
        if (rank == 0 && k >= 3 && k - 3 < orders) write_rows(k - 3);
    };

    // ---- the recurrence ------------------------------------------------------------------------
    const int q4 = S >> LU;                         // slots of one of the U parts of the tile
    const int sbits = t - LU;                       // tile bits that flip through shared memory
    const int flip_mask = S - 1 - (B == 4 ? 1 : 0);  // the global flip inside the tile: every state bit
    const bool gf = a.gflip != nullptr;
    const int yone = -(1 << (29 - ge));             // -1 in the units of the sums
    uint32_t chk = 0;
    auto order = [&](const int k) -> bool {
        const int4* cur = (k & 1) ? buf1 : buf0;
        int4* oth = (k & 1) ? buf0 : buf1;
        const int4* pcur = ((k & 1) ? a.pub1 : a.pub0) + pslot0;
        int4* pnew = ((k & 1) ? a.pub0 : a.pub1) + pslot0 + static_cast<int64_t>(rank) * S;
        FxMom ms[NT];
#pragma unroll
        for (int e = 0; e < NT; ++e) ms[e].hh = ms[e].mm = 0;
        if (active) {
            for (int qb = 0; qb < q4; qb += nwork) {
                const bool val = qb + tid < q4;
                const int q = (qb + tid) & (q4 - 1);     // idle lanes repeat a slot of w_k, and store and check nothing
                const int4* old = val ? oth : cur;       // a repeated slot of w_{k-1} is being overwritten
                int4 x[U];
                int64_t hh[U][2], mm[U][2];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    x[u] = cur[u * q4 + q];
                    hh[u][0] = hh[u][1] = 0;
                    mm[u][0] = mm[u][1] = int64_t(1) << (28 - ge);
                }
                if (k > 0) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int4 y = old[u * q4 + q];
                        hh[u][0] += static_cast<int64_t>(y.x) * yone;
                        mm[u][0] += static_cast<int64_t>(y.y) * yone;
                        hh[u][1] += static_cast<int64_t>(y.z) * yone;
                        mm[u][1] += static_cast<int64_t>(y.w) * yone;
                    }
                }
                // flips of the top tile bits: the thread's own slots
#pragma unroll
                for (int l = 0; l < LU; ++l) {
                    const int2 g = g_s[sbits + l];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        fx_mad(hh[u][0], mm[u][0], g, x[u ^ (1 << l)].x, x[u ^ (1 << l)].y);
                        fx_mad(hh[u][1], mm[u][1], g, x[u ^ (1 << l)].z, x[u ^ (1 << l)].w);
                    }
                }
                if (B == 1) {                            // bit 0: the slot's two states
                    const int2 g = g_s[0];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        fx_mad(hh[u][0], mm[u][0], g, x[u].z, x[u].w);
                        fx_mad(hh[u][1], mm[u][1], g, x[u].x, x[u].y);
                    }
                }
                for (int i = B == 1 ? 1 : 0; i < sbits; ++i) {
                    const int2 g = g_s[i];
                    const int q2 = q ^ fx_slot_bit<B>(i);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int4 v = cur[u * q4 + q2];
                        fx_mad(hh[u][0], mm[u][0], g, v.x, v.y);
                        fx_mad(hh[u][1], mm[u][1], g, v.z, v.w);
                    }
                }
                // flips of the group bits: partner tiles, published in L2
                for (int j = 0; j < lgr; ++j) {
                    const int2 g = g_s[t + j];
                    const int4* pp = pcur + static_cast<int64_t>(rank ^ (1 << j)) * S + q;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int4 v = __ldcg(pp + u * q4);
                        fx_mad(hh[u][0], mm[u][0], g, v.x, v.y);
                        fx_mad(hh[u][1], mm[u][1], g, v.z, v.w);
                    }
                }
                if (gf) {
                    const int2 g = g_s[kMaxSpins];
                    const int4* pp = pcur + static_cast<int64_t>(rank ^ ((1 << lgr) - 1)) * S;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int sl = (u * q4 + q) ^ flip_mask;
                        const int4 v = lgr > 0 ? __ldcg(pp + sl) : cur[sl];
                        fx_mad(hh[u][0], mm[u][0], g, B == 1 ? v.z : v.x, B == 1 ? v.w : v.y);
                        fx_mad(hh[u][1], mm[u][1], g, B == 1 ? v.x : v.z, B == 1 ? v.y : v.w);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int sl = u * q4 + q;
                    const int2 d0 = diag_s[B == 4 ? sl >> 1 : (B == 2 ? sl : 2 * sl)];
                    const int2 d1 = B == 1 ? diag_s[2 * sl + 1] : d0;
                    fx_mad(hh[u][0], mm[u][0], d0, x[u].x, x[u].y);
                    fx_mad(hh[u][1], mm[u][1], d1, x[u].z, x[u].w);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    int64_t o0 = (hh[u][0] << ge) + (mm[u][0] >> (29 - ge));
                    int64_t o1 = (hh[u][1] << ge) + (mm[u][1] >> (29 - ge));
                    if (k == 0) {                        // w_1 = G w_0: half of 2 G w_0
                        o0 = (o0 + 1) >> 1;
                        o1 = (o1 + 1) >> 1;
                    }
                    const int2 l0 = fx_limbs(o0), l1 = fx_limbs(o1);
                    const int4 o = make_int4(l0.x, l0.y, l1.x, l1.y);
                    if (val) {
                        oth[u * q4 + q] = o;
                        if (lgr > 0) pnew[u * q4 + q] = o;
                        // |o| < 2^58: the top bits of the high word are all sign
                        chk |= (static_cast<uint32_t>(static_cast<uint64_t>(o0) >> 32) + (1u << 26)) & ~((1u << 27) - 1u);
                        chk |= (static_cast<uint32_t>(static_cast<uint64_t>(o1) >> 32) + (1u << 26)) & ~((1u << 27) - 1u);
                    }
                    if constexpr (B == 4) {
                        // columns 2h, 2h + 1 of a state sit in the thread, the other pair in lane ^ 1 (the sums
                        // and their split over the pair are those of tile_step_df4 in stencil.cu)
                        const int4 c = make_int4(__shfl_xor_sync(0xffffffffu, x[u].x, 1), __shfl_xor_sync(0xffffffffu, x[u].y, 1),
                                                 __shfl_xor_sync(0xffffffffu, x[u].z, 1), __shfl_xor_sync(0xffffffffu, x[u].w, 1));
                        if (val) {
                            const bool h = tid & 1;
                            ms[0].mad(x[u].x, x[u].y, x[u].x, x[u].y);
                            ms[1].mad(x[u].x, x[u].y, x[u].z, x[u].w);
                            ms[2].mad(x[u].z, x[u].w, x[u].z, x[u].w);
                            ms[3].mad(o.x, o.y, x[u].x, x[u].y);
                            ms[4].mad(o.x, o.y, x[u].z, x[u].w);
                            ms[5].mad(o.z, o.w, x[u].z, x[u].w);
                            const int4 p = h ? c : o, v = h ? x[u] : c;
                            ms[6].mad(p.x, p.y, v.x, v.y);
                            ms[7].mad(p.x, p.y, v.z, v.w);
                            ms[8].mad(p.z, p.w, v.x, v.y);
                            ms[9].mad(p.z, p.w, v.z, v.w);
                        }
                    } else if constexpr (B == 2) {
                        if (val) {
                            ms[0].mad(x[u].x, x[u].y, x[u].x, x[u].y);
                            ms[1].mad(x[u].x, x[u].y, x[u].z, x[u].w);
                            ms[2].mad(x[u].z, x[u].w, x[u].z, x[u].w);
                            ms[3].mad(o.x, o.y, x[u].x, x[u].y);
                            ms[4].mad(o.x, o.y, x[u].z, x[u].w);
                            ms[5].mad(o.z, o.w, x[u].z, x[u].w);
                        }
                    } else {
                        if (val) {
                            ms[0].mad(x[u].x, x[u].y, x[u].x, x[u].y);
                            ms[0].mad(x[u].z, x[u].w, x[u].z, x[u].w);
                            ms[1].mad(o.x, o.y, x[u].x, x[u].y);
                            ms[1].mad(o.z, o.w, x[u].z, x[u].w);
                        }
                    }
                }
            }
            // the warp's sums, lane by lane
            if constexpr (B == 4) {
                FxSum v[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = fx_sum(e < 10 ? ms[e].value() : 0);
                const FxSum s = warp_reduce_scatter<16, 2>(v, lane);
                const int e = lane >> 1;
                if (e < 10) red_s[k % kFxRedRing][warp][(lane & 1) * 10 + e] = s;
            } else if constexpr (B == 2) {
                FxSum v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = fx_sum(e < 6 ? ms[e].value() : 0);
                const FxSum s = warp_reduce_scatter<8>(v, lane);
                if ((lane & 3) == 0 && (lane >> 2) < 6) red_s[k % kFxRedRing][warp][lane >> 2] = s;
            } else {
                FxSum v[2] = {fx_sum(ms[0].value()), fx_sum(ms[1].value())};
                const FxSum s = warp_reduce_scatter<2>(v, lane);
                if ((lane & 15) == 0) red_s[k % kFxRedRing][warp][lane >> 4] = s;
            }
        }
        return fx_group_sync(a, group, target += G, [&] { moments_behind(k); });
    };
    for (int k0 = 0; k0 < orders; k0 += kFxCheck) {
        const int k1 = k0 + kFxCheck < orders ? k0 + kFxCheck : orders;
        for (int k = k0; k < k1; ++k)
            if (!order(k)) return;
        // Outgrown in an earlier stretch? (The status is the larger the earlier: this stretch's, which some CTAs may
        // have set already, does not count, so that all CTAs of the group leave together.) A look at every order
        // would take 0.1 to 0.5 us of its 2 to 3.
        if (__ldcg(a.status + group) > 0x7fffffff - k0) return;
        if (chk) atomicMax(a.status + group, 0x7fffffff - k0);
    }
    for (int k = orders; k < orders + 3; ++k)
        if (!fx_group_sync(a, group, target += G, [&] { moments_behind(k); })) return;
}

std::mutex g_fx_mu;
std::map<std::pair<const void*, int>, bool> g_fx_ready;

// Allow the largest dynamic shared memory once per kernel and device.
cudaError_t fx_prepare(const void* f, int optin) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_fx_mu);
    bool& have = g_fx_ready[std::make_pair(f, dev)];
    if (have) return cudaSuccess;
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, f)) != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - static_cast<int>(fa.sharedSizeBytes));
    if (e == cudaSuccess) have = true;
    return e;
}

template <int B>
const void* fx_kernel_b(int u) {
    return u == 4 ? reinterpret_cast<const void*>(evolve_fx_kernel<B, 4>)
                  : (u == 2 ? reinterpret_cast<const void*>(evolve_fx_kernel<B, 2>) : reinterpret_cast<const void*>(evolve_fx_kernel<B, 1>));
}

const void* fx_kernel(int b, int u) { return b == 4 ? fx_kernel_b<4>(u) : (b == 2 ? fx_kernel_b<2>(u) : fx_kernel_b<1>(u)); }

constexpr int kFxStatic = 18432;        // static shared memory of the kernels, rounded up

int fx_smem(int b, int maxN, int lg) {
    const int64_t T = int64_t(1) << (maxN - lg > 0 ? maxN - lg : 0);
    const int64_t slots = T * b / 2 > 1 ? T * b / 2 : 1;
    return slots * 32 + T * 8 > (1 << 20) ? 1 << 20 : static_cast<int>(slots * 32 + T * 8);
}

}  // namespace

int fx_part_sums(int b) { return kFxPartRing * (b == 4 ? 20 : (b == 2 ? 6 : 2)); }

// Group size, threads and slots per thread for `count` realizations of at most maxN spins; false when a
// realization does not fit the shared memory of a group.
bool fx_plan(int b, int count, int minN, int maxN, FxPlan* p) {
    int dev = 0, optin = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    const int room = optin - kFxStatic;
    int lg = 0;
    while (lg < kFxMaxLg && (fx_smem(b, maxN, lg) > room)) ++lg;
    if (fx_smem(b, maxN, lg) > room || (1 << lg) > sms) return false;
    // more CTAs per realization while all realizations run at once and each thread keeps a slot
    auto slots = [&](int l) { return ((int64_t(1) << maxN) >> l) * b / 2; };
    while (lg < kFxMaxLg && (static_cast<int64_t>(count) << (lg + 1)) <= sms && slots(lg + 1) >= (lg < 3 ? 128 : 512)) ++lg;
    p->lg = lg;
    p->sync = lg == 0 ? kFxAlone : (lg <= 3 ? kFxCluster : kFxCounter);
    const int64_t S = slots(lg) > 1 ? slots(lg) : 1;
    p->u = S >= 4 * kFxThreads ? 4 : (S >= 2 * kFxThreads ? 2 : 1);
    if (minN < 6) p->u = 1;
    int64_t nt = (S / p->u + 31) / 32 * 32;
    p->threads = static_cast<int>(nt < kFxThreads ? nt : kFxThreads);
    p->slots_max = static_cast<int>(S);
    p->smem = fx_smem(b, maxN, lg);
    p->groups = sms >> lg;              // groups of a cooperative launch (one CTA per SM)
    return true;
}

// Evolve the realizations a.list[0 .. count) (order: longest first) under plan p.
cudaError_t launch_evolve_fx(int b, const FxPlan& p, const FxArgs& args, int count, cudaStream_t st) {
    const void* f = fx_kernel(b, p.u);
    int dev = 0, optin = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
        (e = fx_prepare(f, optin)) != cudaSuccess)
        return e;
    FxArgs a = args;
    a.lg = p.lg;
    a.sync = p.sync;
    a.slots_max = p.slots_max;
    const int per = p.sync == kFxCounter ? p.groups : count;
    for (int g0 = 0; g0 < count; g0 += per) {
        const int n = count - g0 < per ? count - g0 : per;
        FxArgs c = a;
        c.list = a.list + g0;
        c.bar = a.bar + g0;
        c.status = a.status + g0;
        c.pro = a.pro + (static_cast<int64_t>(g0) << p.lg);
        c.part = a.part + static_cast<int64_t>(g0) * fx_part_sums(b);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(n) << p.lg);
        cfg.blockDim = dim3(p.threads);
        cfg.dynamicSmemBytes = p.smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        if (p.sync == kFxCluster) {
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 1u << p.lg;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
        } else if (p.sync == kFxCounter) {
            at[0].id = cudaLaunchAttributeCooperative;
            at[0].val.cooperative = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
        }
        void* params[] = {&c};
        if ((e = cudaLaunchKernelExC(&cfg, f, params)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dacp
