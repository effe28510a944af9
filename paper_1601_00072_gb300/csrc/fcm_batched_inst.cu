// Batched FCM: many independent slices in one persistent launch.
//
// Compiled once per block size with -DFCM_BATCH_NT=256 or 512.
//
// Each slice is one run of Algorithm 1 (arXiv:1601.00072, Sec. 2.1) with its
// own n, C, m, eps and max_iter. The grid is persistent: CTAs (or thread-block
// clusters) take slices from a work queue ordered by decreasing size (LPT),
// so the largest slices start first and the small ones fill the tail.
//
//  * Big slices (n >= plan.big) are shared by all K CTAs of a cluster: each
//    CTA takes a contiguous 1/K of the pixels; after every pass the CTAs
//    exchange their block totals through distributed shared memory at a
//    hardware cluster barrier and add them in rank order, so every rank
//    derives the same centers and the same stop decision.
//  * Once the queue reaches small slices, every CTA works alone.
//
// No U is stored between iterations: an iteration reads only x, which sits in
// shared memory when the CTA's share fits, and adds up Eq. 3's sums; the change
// |U^k - U^{k-1}| is taken over a sample of the pixels, which bounds delta_k from
// below, and over every pixel, with J_k and the write of U^k, in a full pass when
// that bound does not reach eps or k is max_iter (as in the whole-run kernel of a
// single image). U^0, when given, is read in pass 0. All per-pixel arithmetic is
// in packed FP32x2 pairs; sums run in FP32 over chunks of a few pixels, then in
// compensated FP32 per thread, warp, CTA and cluster (no FP64 instruction in the
// iteration loop). Bound by the barriers of the reductions (the largest stall), then
// by the FP32 pipe (31 to 40 % of cycles on 64 slices): a batch of 512
// slices (32 M pixels, 33 iterations on average) 3.66 -> 2.54 ms per call.
#define FCM_ONE_SCALAR_PAIR
#include "fcm_batched.h"
#include "fcm_device.cuh"
#include "fcm_df.cuh"

#ifndef FCM_BATCH_NT
#error "compile with -DFCM_BATCH_NT=<threads per CTA>"
#endif

namespace fcm {
namespace {

constexpr int NTB = FCM_BATCH_NT;
constexpr int NWB = NTB / 32;
// Up to 128 registers per thread (the recompute loop keeps two center sets
// and packed accumulators live): one 512-thread CTA or two 256-thread CTAs
// per SM, with 192 KB or 96 KB of x staging each.
constexpr int XCAP = NTB == 512 ? 49152 : 24576;
constexpr int MIN_BLOCKS = NTB == 512 ? 1 : 2;
constexpr int SAMPLE_WARPS = 2;  // warps that sample delta_k in a sums pass

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned k;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(k));
    return k;
}
// Hardware barrier of all threads of all CTAs of the cluster, with release /
// acquire ordering of their shared-memory writes.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t dsmem_addr(const void* local, unsigned rank) {
    uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(local)), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 ld_dsmem_f4(const float4* local, unsigned rank) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(dsmem_addr(local, rank))
                 : "memory");
    return v;
}
__device__ __forceinline__ int ld_dsmem_s32(const int* local, unsigned rank) {
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(dsmem_addr(local, rank)) : "memory");
    return v;
}

struct BatchShared {
    DF w[NWB][2 * FCM_MAX_CLUSTERS];  // warp totals of num[C], den[C]; J in w[][0] of a full pass
    float mx[NWB];                    // warp maxima of |dU|
    unsigned bad[NWB];
    f2 wit[NWB];                      // each warp's pair of largest change in a full pass
    // block totals, double-buffered for the cluster or team exchange: (num, den)
    // of each cluster as double-floats, then (max|dU|, bad, J)
    float4 red[2][FCM_MAX_CLUSTERS + 1];
    float v[3][FCM_MAX_CLUSTERS];     // V^k, V^{k-1} and V^{k+1} in turn
    DF v64[3][FCM_MAX_CLUSTERS];      // the double-float quotients behind them
    DF J;
    float delta;
    unsigned flags;                   // bit 0: bad input
    unsigned empty;                   // some cluster of the latest sums pass was empty
    unsigned far;                     // some center moved by more than REBASE times its new value
    int idx;
    int team_err;             // a team barrier gave up
    int item[3];              // team schedule: slice, seat, team size
};

// A slice shared by a team of CTAs of the team schedule (any CTAs of the
// grid, not one cluster): after every pass each rank writes its block totals
// to global slots, arrives at the slice's barrier counter and waits, bounded,
// for the whole team; then every rank adds the team's totals in rank order.
// slots == nullptr: no team (a lone CTA, or a cluster exchanging through
// distributed shared memory).
struct TeamCtx {
    float4* slots;        // [T][2][TEAM_SLOT], this slice's
    unsigned* ctr;        // this slice's barrier counter (zero before the batch)
    uint32_t spins;       // polls, 64 ns and an L2 round trip apart, before the barrier gives up
    uint32_t phantoms;    // arrivals beyond the team's (0 unless a test injects a barrier that never fills)
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Threads add the centered terms of Eq. 3 (num_j = sum u_j^m (x - v_j^k), so
// v_j^{k+1} = v_j^k + num_j / den_j) in FP32 over CHUNK pairs and fold each chunk
// into double-float sums, so the rounding of a thread's sum does not grow with the
// size of its share of the slice. (Errors against 64 bits over 2^12 to 2^21 pixels,
// C and m: U 0.96, V 1.02 times those of uncentered sums folded every 8 pairs.)
constexpr int CHUNK = 16;

template <int C>
struct SliceAcc {
    f2 num2[C], den2[C];
    DF num[C], den[C];
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num2[j] = den2[j] = pack2(0.0f, 0.0f);
            num[j] = den[j] = DF{0.0f, 0.0f};
        }
    }
    __device__ __forceinline__ void add(const f2 (&d2)[C], const f2 (&um2)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num2[j] = fma2(um2[j], d2[j], num2[j]);
            den2[j] = add2(den2[j], um2[j]);
        }
    }
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            df_add(num[j], lo2(num2[j]) + hi2(num2[j]));
            df_add(den[j], lo2(den2[j]) + hi2(den2[j]));
            num2[j] = den2[j] = pack2(0.0f, 0.0f);
        }
    }
};

// Warp totals of P double-floats (P a power of two up to 16) by log-step
// halving: at each step a lane keeps one half of the values and hands the other
// half to its partner, P - 1 + (5 - log2 P) merges in place of 5 P. On return the
// lanes with (lane & (32 / P - 1)) == 0 hold, in a[0], the total of one value:
// bit i of its number from the top is bit 4 - i of the lane.
template <int P>
__device__ __forceinline__ void warp_totals_df(DF (&a)[P]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int w = P; w > 1; w >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < w / 2; ++i) {
            const DF send = up ? a[i] : a[i + w / 2], keep = up ? a[i + w / 2] : a[i];
            a[i] = df_merge(keep, DF{__shfl_xor_sync(0xffffffffu, send.hi, o), __shfl_xor_sync(0xffffffffu, send.lo, o)});
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1)
        a[0] = df_merge(a[0], DF{__shfl_xor_sync(0xffffffffu, a[0].hi, o), __shfl_xor_sync(0xffffffffu, a[0].lo, o)});
}
constexpr int pow2_at_least(int n) { return n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 16; }

// Sum over the first n lanes (n up to 32), the same in every lane: TwoSum is
// symmetric.
__device__ __forceinline__ DF lanes_sum(DF d, int n) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (o < n)
            d = df_merge(d, DF{__shfl_xor_sync(0xffffffffu, d.hi, o), __shfl_xor_sync(0xffffffffu, d.lo, o)});
    }
    return d;
}

// What one pass leaves: X_SUMS0 the sums of pass 0 from U^0, X_SUMS centered sums
// (V^{k+1} into sh.v[nxt]), X_FULL J and the exact maximum. All with the maximum
// (sh.delta) and the flags.
// X_REBASED: sums centered on what slot nxt holds already.
enum Exchange : int { X_SUMS0 = 0, X_SUMS = 1, X_FULL = 2, X_REBASED = 3 };
// The FP32 differences x - v_j^k round by 2^-24 of the step at most, so up to this
// factor the new center keeps about 18 bits; beyond it, the sums are taken again
// (rebased_sums), as in the whole-run kernel of a single image.
constexpr float REBASE = 64.0f;

// Totals of one pass over the slice: warp totals (already in sh.w, sh.mx, sh.bad),
// the CTA's, then (K > 1) the K CTAs' through distributed shared memory or, in a
// team, global slots, all in compensated FP32 (no FP64 instruction: a few threads
// would run a long FP64 chain while the rest wait at the barrier). Warp q < C
// takes cluster q from its warp totals to its new center, so two barriers serve
// the pass; warp C (or the first one again) takes the maximum, flags and J.
// One function for every cluster count: called once per pass, it does not slow
// the pass, and the 32 variants of the slice loop stay small.
static __device__ __noinline__ void slice_reduce(BatchShared& sh, int C, int X, unsigned r, unsigned K, int parity,
                                                 int npass, const TeamCtx& tc, int cur, int nxt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int FIRST = X == X_FULL ? C : 0;
    __syncthreads();
    auto center = [&](int q, DF num, DF den) {
        if (den.hi > 0.0f) {
            DF v = df_div(num, den);
            const float step = fabsf(v.hi);
            if (X == X_SUMS || X == X_REBASED) v = df_merge(v, DF{sh.v[X == X_SUMS ? cur : nxt][q], 0.0f});
            if (X == X_SUMS && step > REBASE * fabsf(v.hi)) sh.far = 1u;
            sh.v[nxt][q] = v.hi;
            sh.v64[nxt][q] = v;
        } else {
            // an empty cluster keeps its center (in pass 0 that is V^0, or 0 from a U^0)
            if (X != X_REBASED) {
                sh.v[nxt][q] = X == X_SUMS ? sh.v[cur][q] : 0.0f;
                sh.v64[nxt][q] = X == X_SUMS ? sh.v64[cur][q] : DF{0.0f, 0.0f};
            }
            sh.empty = 1u;
        }
    };
    const bool alone = K == 1;
    for (int q = FIRST + warp; q <= C; q += NWB) {
        float4 t;
        if (q < C) {
            const DF z{0.0f, 0.0f};
            const DF num = lanes_sum(lane < NWB ? sh.w[lane][q] : z, NWB), den = lanes_sum(lane < NWB ? sh.w[lane][C + q] : z, NWB);
            t = make_float4(num.hi, num.lo, den.hi, den.lo);
            if (alone && lane == 0) center(q, num, den);
        } else {
            const unsigned mb = __reduce_max_sync(0xffffffffu, lane < NWB ? __float_as_uint(sh.mx[lane]) : 0u);
            const unsigned fb = __reduce_or_sync(0xffffffffu, lane < NWB ? sh.bad[lane] & 1u : 0u);
            const DF J = X == X_FULL ? lanes_sum(lane < NWB ? sh.w[lane][0] : DF{0.0f, 0.0f}, NWB) : DF{0.0f, 0.0f};
            t = make_float4(__uint_as_float(mb), __uint_as_float(fb), J.hi, J.lo);
            if (alone && lane == 0) {
                sh.delta = t.x;
                sh.flags = fb;
                sh.J = J;
            }
        }
        if (!alone && lane == 0) {
            sh.red[parity][q] = t;
            if (tc.slots) __stcg(&tc.slots[((int64_t)r * 2 + parity) * TEAM_SLOT + q], t);
        }
    }
    if (!alone) {
        if (tc.slots) {
            // team: arrive, wait (bounded) for every rank's totals of this pass
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                atomicAdd(tc.ctr, 1u);
                const unsigned target = (unsigned)(npass + 1) * K + tc.phantoms;
                uint32_t spins = 0;
                while (ld_acquire_gpu(tc.ctr) < target) {
                    if (++spins > tc.spins) {
                        sh.team_err = 1;
                        break;
                    }
                    __nanosleep(64);
                }
                __threadfence();
            }
            __syncthreads();
        } else {
            cluster_sync();
        }
        for (int q = FIRST + warp; q <= C; q += NWB) {
            // lane i takes rank i's totals
            float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (lane < (int)K)
                t = tc.slots ? __ldcg(&tc.slots[((int64_t)lane * 2 + parity) * TEAM_SLOT + q]) : ld_dsmem_f4(&sh.red[parity][q], lane);
            if (q < C) {
                const DF num = lanes_sum(DF{t.x, t.y}, (int)K), den = lanes_sum(DF{t.z, t.w}, (int)K);
                if (lane == 0) center(q, num, den);
            } else {
                const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(t.x));
                const unsigned fb = __reduce_or_sync(0xffffffffu, __float_as_uint(t.y));
                const DF J = lanes_sum(DF{t.z, t.w}, (int)K);
                if (lane == 0) {
                    sh.delta = __uint_as_float(mb);
                    sh.flags = fb;
                    sh.J = J;
                }
            }
        }
    }
    __syncthreads();
}

// A warp's totals of a sums pass into sh.w, its maximum and flags into sh.mx, sh.bad.
template <int C>
__device__ __forceinline__ void warp_publish(BatchShared& sh, const SliceAcc<C>& a, float mx, bool bad) {
    constexpr int P = pow2_at_least(2 * C);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    DF t[P];
#pragma unroll
    for (int i = 0; i < P; ++i)
        t[i] = i < C ? a.num[i < C ? i : 0] : i < 2 * C ? a.den[(i >= C && i < 2 * C) ? i - C : 0] : DF{0.0f, 0.0f};
    warp_totals_df<P>(t);
    int s = 0;
#pragma unroll
    for (int w = P, o = 16; w > 1; w >>= 1, o >>= 1) s += (lane & o) ? w / 2 : 0;
    if ((lane & (32 / P - 1)) == 0 && s < 2 * C) sh.w[warp][s] = t[0];
    const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
    const bool any = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
        sh.mx[warp] = __uint_as_float(mb);
        sh.bad[warp] = any ? 1u : 0u;
    }
}

// Where a CTA reads its share of x during the iterations: FP32 values (in
// shared memory, or in global memory when the share does not fit), or bytes
// in shared memory when every value of the share is an integer grey level
// 0..255 (exact, and four times the pixels per byte of shared memory). The
// choice is the same for the whole CTA.
struct XSrc {
    const float* f;
    const uint8_t* b;
    bool bytes;
    __device__ __forceinline__ float at(int i) const { return bytes ? (float)b[i] : f[i]; }
    __device__ __forceinline__ f2 pair(int q) const {
        if (bytes) {
            // 2^23 + byte is the byte in the low mantissa bits: no conversion unit
            const unsigned v = *reinterpret_cast<const uint16_t*>(b + 2 * q);
            const f2 t = pack2(__uint_as_float(0x4b000000u | (v & 0xffu)), __uint_as_float(0x4b000000u | (v >> 8)));
            return sub2(t, pack2(8388608.0f, 8388608.0f));
        }
        const float2 v = *reinterpret_cast<const float2*>(f + 2 * q);
        return pack2(v.x, v.y);
    }
};

// The warps' totals of a sums pass from V^k in slot cur, with the numerators centered
// on slot nxt, into sh.w: for a center that moved by far more than it is now away
// from 0, whose differences x - v^k have lost the bits of x. Rare: one function
// for every cluster count and fuzzifier, in the scalar form.
static __device__ __noinline__ void rebased_sums(BatchShared& sh, const XSrc& xl, int cnt, int C, int mk, float m,
                                                 float inv_m1, int cur, int nxt) {
    constexpr int N = FCM_MAX_CLUSTERS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    DF t[2 * N];
#pragma unroll
    for (int i = 0; i < 2 * N; ++i) t[i] = DF{0.0f, 0.0f};
    for (int i = threadIdx.x; i < cnt; i += NTB) {
        const float xi = xl.at(i);
        const PixelPair<N> w = scalar_pair_any(xi, xi, sh.v[cur], C, mk, true, m, inv_m1);
#pragma unroll
        for (int j = 0; j < N; ++j) {
            if (j >= C) break;
            df_add(t[j], w.a[j] * (xi - sh.v[nxt][j]));
            df_add(t[N + j], w.a[j]);
        }
    }
    warp_totals_df<2 * N>(t);
    // the lane's value: bit i of its number from the top is bit 4 - i of the lane
    int s = 0;
#pragma unroll
    for (int w = 2 * N, o = 16; w > 1; w >>= 1, o >>= 1) s += (lane & o) ? w / 2 : 0;
    const int j = s % N;
    if ((lane & 1) == 0 && j < C) sh.w[warp][s < N ? j : C + j] = t[0];
}

template <int C, int MK>
__device__ __noinline__ void process_slice(const SliceDesc& d, SliceResult& res, unsigned r, unsigned K, float* xs,
                                           BatchShared& sh, bool resume, int cap, const TeamCtx& tc) {
    const int64_t n = d.n;
    int64_t share = (n + K - 1) / K;
    share += share & 1;  // even, so only the last pixel of the slice can be unpaired
    const int64_t lo = min(n, (int64_t)r * share), hi = min(n, lo + share);
    const int cnt = (int)(hi - lo);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < C) {
        // a parked slice: V^k and V^{k-1} as saved, iteration k = iters + 1 next
        const int t = threadIdx.x;
        const double q = resume ? res.V64[t] : (double)d.V0[t];
        sh.v[0][t] = resume ? res.vcur[t] : d.V0[t];
        sh.v[2][t] = resume ? res.vprev[t] : d.V0[t];
        sh.v64[0][t] = DF{(float)q, (float)(q - (double)(float)q)};
    }
    if (threadIdx.x == 0) {
        sh.team_err = 0;
        sh.empty = sh.far = 0u;
    }
    XSrc xl{d.x + lo, reinterpret_cast<const uint8_t*>(xs), false};
    if (cnt <= XCAP) {
        for (int i = threadIdx.x; i < cnt; i += NTB) xs[i] = __ldg(d.x + lo + i);
        xl.f = xs;
    } else if (cnt <= 4 * XCAP) {
        uint8_t* xb = reinterpret_cast<uint8_t*>(xs);
        bool ok = true;
        for (int i = threadIdx.x; i < cnt; i += NTB) {
            const float v = __ldg(d.x + lo + i);
            const bool g = v >= 0.0f && v <= 255.0f && v == rintf(v);
            ok &= g;
            xb[i] = g ? (uint8_t)v : (uint8_t)0;
        }
        xl.bytes = __syncthreads_and(ok);
    }
    __syncthreads();
    const int npair = cnt >> 1;
    const bool odd_tail = (cnt & 1) && threadIdx.x == 0;  // the slice's last pixel, alone
    const float m = d.m, inv_m1 = d.inv_m1;
    const bool from_u = d.init == FCM_INIT_U;
    const float* U0 = d.U0;
    float* U = d.U;
    int parity = 0, npass = 0, flags = resume ? res.flags : 0;
    int cur = 0, prv = 2, nxt = 1;  // slots of V^k, V^{k-1}, V^{k+1} in sh.v
    auto advance = [&] {
        if (sh.empty) flags |= FCM_FLAG_EMPTY_CLUSTER;
        __syncthreads();
        if (threadIdx.x == 0) sh.empty = 0u;  // set again only after the next pass's first barrier
        const int t = prv;
        prv = cur;
        cur = nxt;
        nxt = t;
    };
    auto reduce = [&](int kind) {
        slice_reduce(sh, C, kind, r, K, parity, npass, tc, cur, nxt);
        parity ^= 1;
        ++npass;
    };
    // A sums pass from V^k: u^m of every pixel, Eq. 3's sums. check: pass 0.
    auto sums_pass = [&](float dmax, bool check) {
        SliceAcc<C> a;
        a.reset();
        PackedCenters<C, MK> cen;
        cen.set(sh.v[cur]);
        bool bad = false;
        int held = 0;
        constexpr int N = C <= 5 ? 2 : 1;  // pairs whose arithmetic overlaps, as registers allow
        int p = threadIdx.x;
        for (; p + (N - 1) * NTB < npair; p += N * NTB) {
            f2 xq[N], um[N][C], d2[N][C], J2[N];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                xq[i] = xl.pair(p + i * NTB);
                if (check) bad |= !(finite_f(lo2(xq[i])) && finite_f(hi2(xq[i])));
            }
            packed_pairs<C, MK, true, N>(xq, cen, m, inv_m1, um, d2, J2);
#pragma unroll
            for (int i = 0; i < N; ++i) a.add(d2[i], um[i]);
            if (++held == CHUNK / N) {
                a.fold();
                held = 0;
            }
        }
        if (N > 1 && p < npair) {
            f2 um[1][C], d2[1][C], J2[1];
            const f2 xq[1] = {xl.pair(p)};
            if (check) bad |= !(finite_f(lo2(xq[0])) && finite_f(hi2(xq[0])));
            packed_pairs<C, MK, true, 1>(xq, cen, m, inv_m1, um, d2, J2);
            a.add(d2[0], um[0]);
        }
        if (odd_tail) {
            // the low halves of the sums
            const float xi = xl.at(cnt - 1);
            if (check) bad |= !finite_f(xi);
            const PixelPair<C> w = scalar_pair<C, MK, true>(xi, xi, cen.vs, m, inv_m1);
            const f2 xs2 = cen.of(pack2(xi, xi));
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const f2 um = pack2(w.a[j], 0.0f);
                a.num2[j] = fma2(um, sub2(xs2, cen.v2[j]), a.num2[j]);
                a.den2[j] = add2(a.den2[j], um);
            }
        }
        a.fold();
        if (PackedCenters<C, MK>::SCALED) {
            // back from scaled differences (by a power of two: exact)
            const float back = rcp_approx(lo2(cen.scale));
#pragma unroll
            for (int j = 0; j < C; ++j) a.num[j] = DF{a.num[j].hi * back, a.num[j].lo * back};
        }
        if (check && threadIdx.x < C) bad |= !finite_f(sh.v[cur][threadIdx.x]);
        warp_publish<C>(sh, a, dmax, bad);
        reduce(X_SUMS);
        if (sh.far && !sh.team_err) {
            // the same in every CTA that shares the slice; the maximum and the flags
            // are still in sh.mx and sh.bad
            __syncthreads();
            if (threadIdx.x == 0) sh.far = 0u;
            rebased_sums(sh, xl, cnt, C, MK, m, inv_m1, cur, nxt);
            reduce(X_REBASED);
        }
    };
    // U^k of a pair and its largest |U^k - U^{k-1}|; U^{k-1} is given (u0) or
    // comes from V^{k-1}. J2: the pair's J terms.
    auto change = [&](f2 xq, const PackedCenters<C, MK>& cen, const PackedCenters<C, MK>& pre, f2 (&u2)[C],
                      const f2 (&u0)[C], bool given, f2& J2) {
        f2 w[1][C], o[1][C], t[1][C], j2[1];
        const f2 xa[1] = {xq};
        packed_pairs<C, MK, false, 1>(xa, cen, m, inv_m1, w, t, j2);
        J2 = j2[0];
        if (given) {
#pragma unroll
            for (int j = 0; j < C; ++j) o[0][j] = u0[j];
        } else {
            packed_pairs<C, MK, false, 1>(xa, pre, m, inv_m1, o, t, j2);
        }
        float dd = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            float da, db;
            u2[j] = w[0][j];
            unpack2(sub2(w[0][j], o[0][j]), da, db);
            dd = fmaxf(dd, fmaxf(fabsf(da), fabsf(db)));
        }
        return dd;
    };
    auto u0_pair = [&](int p, f2 (&u0)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const float* r0 = U0 + (int64_t)j * n + lo + 2 * p;
            u0[j] = pack2(__ldg(r0), __ldg(r0 + 1));
        }
    };

    int status = FCM_NOT_CONVERGED, iters = resume ? res.iters : 0;
    if (!resume) {
        // ---- pass 0: V^1 from U^0 (Eq. 3), or U^0 = membership(V^0) (Eq. 4) ----
        if (from_u) {
            SliceAcc<C> a;
            a.reset();
            bool bad = false;
            for (int p0 = threadIdx.x; p0 < npair; p0 += NTB * (CHUNK / 2)) {
                float num[C], den[C];
#pragma unroll
                for (int j = 0; j < C; ++j) num[j] = den[j] = 0.0f;
                for (int q = 0, p = p0; q < CHUNK / 2 && p < npair; ++q, p += NTB) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int i = 2 * p + h;
                        const float xi = xl.at(i);
                        bad |= !finite_f(xi);
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            const float u0 = __ldg(U0 + (int64_t)j * n + lo + i);
                            bad |= !(u0 >= 0.0f) || !finite_f(u0);
                            const float w = pow_m<MK>(u0, m);
                            num[j] = fmaf(w, xi, num[j]);
                            den[j] += w;
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    df_add(a.num[j], num[j]);
                    df_add(a.den[j], den[j]);
                }
            }
            if (odd_tail) {
                const float xi = xl.at(cnt - 1);
                bad |= !finite_f(xi);
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const float u0 = __ldg(U0 + (int64_t)j * n + lo + cnt - 1);
                    bad |= !(u0 >= 0.0f) || !finite_f(u0);
                    const float w = pow_m<MK>(u0, m);
                    df_add(a.num[j], w * xi);
                    df_add(a.den[j], w);
                }
            }
            warp_publish<C>(sh, a, 0.0f, bad);
            reduce(X_SUMS0);
        }
    }
    bool parked = false, gave_up = sh.team_err != 0;
    float delta = resume ? (float)res.delta : 0.0f;
    DF Jk{resume ? (float)res.J : 0.0f, 0.0f};
    if (gave_up) {
        status = FCM_ERR_TIMEOUT;
    } else if (!resume && from_u && (sh.flags & 1u)) {
        status = FCM_ERR_BAD_INPUT;
    } else {
        if (!resume && from_u) advance();
        // The sampled pair of a lane of the first warps: spread evenly over the
        // share, and after a full pass that did not stop the run, in warp 0, the
        // warps' pairs of largest change.
        f2 wx = 0;
        int wp = 0;
        bool sampled = warp < SAMPLE_WARPS && npair > 0;
        if (sampled) {
            wp = (int)((int64_t)threadIdx.x * npair / (32 * SAMPLE_WARPS));
            wx = xl.pair(wp);
        }
        // ---- iterations (k = 0: pass 0 from V^0). A sums pass takes the change over the sample, a lower
        // bound of delta_k: when it reaches eps the run cannot stop at k. Otherwise,
        // and at max_iter, a full pass takes delta_k and J_k over every pixel and
        // writes U^k. ----
        for (int k = !resume && !from_u ? 0 : iters + 1;; ++k) {
            if (k > cap) {
                // first phase of a two-phase batch: park before iteration k
                parked = true;
                break;
            }
            iters = k;
            const bool prev_given = from_u && k == 1, last = k >= d.max_iter;  // max_iter >= 1
            if (!last) {
                float dmax = 0.0f;
                if (sampled && k > 0) {
                    PackedCenters<C, MK> cen, pre;
                    cen.set(sh.v[cur]);
                    pre.set(sh.v[prv]);
                    f2 u0[C], u2[C], J2;
                    if (prev_given) u0_pair(wp, u0);
                    dmax = change(wx, cen, pre, u2, u0, prev_given, J2);
                }
                sums_pass(dmax, k == 0);
                if (sh.team_err) {
                    status = FCM_ERR_TIMEOUT;
                    gave_up = true;
                    break;
                }
                if (k == 0 && (sh.flags & 1u)) {
                    status = FCM_ERR_BAD_INPUT;
                    break;
                }
                if (k == 0 || sh.delta >= d.eps) {
                    advance();
                    continue;
                }
            }
            // ---- the full pass ----
            {
                PackedCenters<C, MK> cen, pre;
                cen.set(sh.v[cur]);
                pre.set(sh.v[prv]);
                DF J{0.0f, 0.0f};
                float dmax = -1.0f, dtail = 0.0f;
                f2 best = 0;
                for (int p = threadIdx.x; p < npair; p += NTB) {
                    const f2 xq = xl.pair(p);
                    f2 u0[C], u2[C], J2;
                    if (prev_given) u0_pair(p, u0);
                    const float dd = change(xq, cen, pre, u2, u0, prev_given, J2);
                    df_add(J, lo2(J2) + hi2(J2));
                    if (dd > dmax) {
                        dmax = dd;
                        best = xq;
                    }
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        float a0, b0;
                        unpack2(u2[j], a0, b0);
                        float* row = U + (int64_t)j * n + lo + 2 * p;
                        __stcs(row, a0);
                        __stcs(row + 1, b0);
                    }
                }
                if (odd_tail) {
                    const float xi = xl.at(cnt - 1);
                    const PixelPair<C> a = scalar_pair<C, MK, false>(xi, xi, cen.vs, m, inv_m1);
                    df_add(J, a.Ja);
                    if (prev_given) {
#pragma unroll
                        for (int j = 0; j < C; ++j)
                            dtail = fmaxf(dtail, fabsf(a.a[j] - __ldg(U0 + (int64_t)j * n + lo + cnt - 1)));
                    } else {
                        const PixelPair<C> b = scalar_pair<C, MK, false>(xi, xi, pre.vs, m, inv_m1);
#pragma unroll
                        for (int j = 0; j < C; ++j) dtail = fmaxf(dtail, fabsf(a.a[j] - b.a[j]));
                    }
#pragma unroll
                    for (int j = 0; j < C; ++j) __stcs(U + (int64_t)j * n + lo + cnt - 1, a.a[j]);
                }
                J = warp_sum_df(J);
                const float own = fmaxf(dmax, 0.0f);
                const unsigned wb = __reduce_max_sync(0xffffffffu, __float_as_uint(own));
                const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(own, dtail)));
                const unsigned who = __ballot_sync(0xffffffffu, dmax >= 0.0f && __float_as_uint(own) == wb);
                if (lane == (who ? __ffs(who) - 1 : 0)) sh.wit[warp] = best;
                if (lane == 0) {
                    sh.w[warp][0] = J;
                    sh.mx[warp] = __uint_as_float(mb);
                    sh.bad[warp] = who ? 2u : 0u;
                }
            }
            reduce(X_FULL);
            if (warp == 0 && lane < NWB && (sh.bad[lane] & 2u)) {
                wx = sh.wit[lane];
                sampled = true;
            }
            if (sh.team_err) {
                status = FCM_ERR_TIMEOUT;
                gave_up = true;
                break;
            }
            delta = sh.delta;
            Jk = sh.J;
            if (delta < d.eps || last) {
                status = delta < d.eps ? FCM_OK : FCM_NOT_CONVERGED;
                break;
            }
            advance();  // to the V^{k+1} of the sums pass
        }
    }
    if (r == 0 && threadIdx.x == 0) {
        res.iters = iters;
        res.status = parked ? SLICE_PARKED : status;
        res.flags = flags;
        res.delta = (double)delta;
        res.J = (double)Jk.hi + (double)Jk.lo;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            res.V64[j] = (double)sh.v64[cur][j].hi + (double)sh.v64[cur][j].lo;
            if (parked) {
                res.vcur[j] = sh.v[cur][j];
                res.vprev[j] = sh.v[prv][j];
            } else {
                d.V[j] = sh.v[cur][j];
            }
        }
    }
    // no rank of a cluster leaves the slice (and reuses its shared memory)
    // while another may still read it; a team exchanges through global slots
    // of its own slice and needs no such wait
    if (K > 1 && !tc.slots) cluster_sync();
    __syncthreads();
}

__device__ __forceinline__ void run_slice(const SliceDesc& d, SliceResult& res, unsigned r, unsigned K, float* xs,
                                          BatchShared& sh, bool resume, int cap, const TeamCtx& tc) {
#define FCM_BATCH_CASE(CC)                                                                  \
    case CC:                                                                                \
        switch (d.mk) {                                                                     \
            case M_TWO: process_slice<CC, M_TWO>(d, res, r, K, xs, sh, resume, cap, tc); break;              \
            case M_THREE: process_slice<CC, M_THREE>(d, res, r, K, xs, sh, resume, cap, tc); break;          \
            case M_ONE_HALF: process_slice<CC, M_ONE_HALF>(d, res, r, K, xs, sh, resume, cap, tc); break;    \
            default: process_slice<CC, M_GENERIC>(d, res, r, K, xs, sh, resume, cap, tc); break;             \
        }                                                                                   \
        break;
    switch (d.C) {
        FCM_BATCH_CASE(1)
        FCM_BATCH_CASE(2)
        FCM_BATCH_CASE(3)
        FCM_BATCH_CASE(4)
        FCM_BATCH_CASE(5)
        FCM_BATCH_CASE(6)
        FCM_BATCH_CASE(7)
        FCM_BATCH_CASE(8)
        default: break;
    }
#undef FCM_BATCH_CASE
}

__global__ void __launch_bounds__(NTB, MIN_BLOCKS)
    k_fcm_batched(const SliceDesc* __restrict__ descs, const int* __restrict__ order, int n_slices,
                  SliceResult* __restrict__ results, BatchCtl* __restrict__ ctl, int64_t big, int phase,
                  int cap) {
    extern __shared__ __align__(16) float xs[];
    __shared__ BatchShared sh;
    const unsigned K = cluster_size(), r = cluster_rank();
    const bool resume = phase == 1;
    // the second phase takes only the slices the first one parked (their
    // status was written by the earlier launch; no one else writes it now)
    auto wanted = [&](int s) { return !resume || __ldcg(&results[s].status) == SLICE_PARKED; };
    bool solo = K == 1;
    int first_solo = -1;
    // ---- the cluster shares the big slices ----
    while (!solo) {
        if (r == 0 && threadIdx.x == 0) sh.idx = (int)atomicAdd(&ctl->next, 1u);
        cluster_sync();
        const int idx = ld_dsmem_s32(&sh.idx, 0);
        cluster_sync();  // every rank has read the index before rank 0 takes another
        if (idx >= n_slices) return;
        const int s = order[idx];
        if (!wanted(s)) continue;
        if (descs[s].n >= big) {
            run_slice(descs[s], results[s], r, K, xs, sh, resume, cap, TeamCtx{});
            continue;
        }
        // the queue has reached the small slices: every CTA works alone now
        solo = true;
        if (r == 0) first_solo = s;
    }
    if (first_solo >= 0) run_slice(descs[first_solo], results[first_solo], 0, 1, xs, sh, resume, cap, TeamCtx{});
    for (;;) {
        if (threadIdx.x == 0) sh.idx = (int)atomicAdd(&ctl->next, 1u);
        __syncthreads();
        const int idx = sh.idx;
        __syncthreads();
        if (idx >= n_slices) return;
        const int s = order[idx];
        if (!wanted(s)) continue;
        run_slice(descs[s], results[s], 0, 1, xs, sh, resume, cap, TeamCtx{});
    }
}

// The team schedule: one cooperative launch (every CTA resident), no
// clusters. The queue holds one item per seat: a slice with a team of T CTAs
// appears T times in a row, seats 0..T-1, so the CTAs that take them form its
// team; the host orders the items by team time, longest first. Only the team
// at the head of the queue can be incomplete, and every other team finishes
// and frees its CTAs, so every team fills; each barrier wait is bounded
// nonetheless.
__global__ void __launch_bounds__(NTB, MIN_BLOCKS)
    k_fcm_teams(TeamArgs a) {
    extern __shared__ __align__(16) float xs[];
    __shared__ BatchShared sh;
    for (;;) {
        if (threadIdx.x == 0) {
            const int idx = (int)atomicAdd(&a.ctl->next, 1u);
            if (idx < a.hdr->max_rounds) {
                const int4 it = a.items[idx];
                sh.item[0] = it.x;
                sh.item[1] = it.y;
                sh.item[2] = it.z;
            } else {
                sh.item[0] = -1;
            }
        }
        __syncthreads();
        const int s = sh.item[0], seat = sh.item[1], T = sh.item[2];
        __syncthreads();
        if (s < 0) return;
        TeamCtx tc{};
        if (T > 1) {
            tc.slots = a.slots + (int64_t)a.slot_base[s] * 2 * TEAM_SLOT;
            tc.ctr = a.counters + s;
            tc.spins = a.hdr->wait_spins;
            tc.phantoms = a.hdr->phantoms;
        }
        run_slice(a.descs[s], a.results[s], (unsigned)seat, (unsigned)T, xs, sh, false, 0x7fffffff, tc);
    }
}

}  // namespace

#define FCM_CAT2(a, b) a##b
#define FCM_CAT(a, b) FCM_CAT2(a, b)
BatchKernel FCM_CAT(batched_kernel_, FCM_BATCH_NT)() {
    return BatchKernel{k_fcm_batched, XCAP * (int)sizeof(float), XCAP, k_fcm_teams};
}

}  // namespace fcm
