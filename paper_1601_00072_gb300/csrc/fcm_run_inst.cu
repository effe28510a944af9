// The whole single-image run in one cooperative launch, instantiated for one
// cluster count.
//
// Compiled once per C in 1..8 with -DFCM_INST_C=<C>.
//
// Algorithm 1 (arXiv:1601.00072, Sec. 2.1) needs U^{k-1} only for the stopping
// quantity delta_k = max |U^k - U^{k-1}|, and delta_k only for the test
// delta_k < eps. So no U is kept between iterations:
//  * A sums pass (iteration k) reads x, forms u^m from V^k (Eq. 4) and adds up
//    the numerators and denominators of V^{k+1} (Eq. 3): 4 bytes per pixel
//    instead of 4 + 8C.
//  * In the same pass a few warps take max |U^k - U^{k-1}| over a sample of the
//    pixels (U^{k-1} again from V^{k-1}, or from U^0 at k = 1). The maximum over
//    a sample is a lower bound of delta_k: when it reaches eps the run cannot
//    stop at k, and the exact delta_k is not needed.
//  * When it does not, or k is max_iter, or a trace wants every iteration, a
//    full pass takes delta_k over every pixel and J_k (Eq. 1), and writes U^k
//    unless the sample has already shown that the run goes on. If the run goes
//    on all the same, the next samples hold the pixel of largest change that
//    every thread saw.
// The iterates, the stop decision and the outputs are those of the loop that
// takes delta_k in every iteration; U is written once instead of k times.
//
// What bounds it: on a large image the FP32 pipe (about 33 operations per pixel
// and iteration at C = 4, m = 2, in packed FP32x2 pairs); x comes from the L2
// (67 MB for a 256^3 volume) or, up to about 10 million pixels, partly from L1.
// On a small image the exchange between the blocks. 60 iterations on a GB300,
// before (U stored; plain loads and a launch per pass where n % 4 != 0) and
// after: 200x200 371 -> 215 us, 199x201 907 -> 247 us, 1024x1024 716 -> 413 us,
// 256^3 6.02 -> 1.85 ms.
//
// The exchange carries its own arrival: every block publishes (num_j, den_j)
// with a 64-bit tag (the run's number and the exchange's index) in one 16-byte
// store, and the warp that needs cluster j's totals polls the slots of all
// blocks until each shows the tag. That is one L2 round trip after the slowest
// block's store, where a barrier counter followed by reads of the partial sums
// takes three. Every block adds the blocks' totals in the same order in
// compensated FP32, so all derive the same V^{k+1} and the same decision.
// Every poll loop is bounded (fcm_set_limits): the run then ends with
// FCM_ERR_TIMEOUT.
#include "fcm_device.cuh"
#include "fcm_df.cuh"
#include "fcm_internal.h"
#include "fcm_run.h"

#ifndef FCM_INST_C
#error "compile with -DFCM_INST_C=<cluster count>"
#endif

namespace fcm {
namespace {

constexpr int SAMPLE_WARPS = 4;  // warps per block that sample delta_k: one per SM sub-partition

// ---- exchange slots: {float a, float b, u64 tag} moved as one 128-bit unit ----

__device__ __forceinline__ void st_slot(void* p, float a, float b, uint64_t tag) {
    const uint64_t v = (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "mov.b128 t, {%1, %2};\n\t"
        "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(v), "l"(tag)
        : "memory");
}
__device__ __forceinline__ void ld_slot(const void* p, float& a, float& b, uint64_t& tag) {
    uint64_t v;
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "ld.relaxed.gpu.global.b128 t, [%2];\n\t"
        "mov.b128 {%0, %1}, t;\n\t}"
        : "=l"(v), "=l"(tag)
        : "l"(p)
        : "memory");
    a = __uint_as_float((unsigned)v);
    b = __uint_as_float((unsigned)(v >> 32));
}

// One warp collects the slots of nb blocks: f(a, b) is called on every lane
// for blocks lane, lane + 32, ... in that order, once each slot shows `tag`.
// GRP loads per lane are in flight together (152 blocks: one group). After
// `limit` unsuccessful polls of a group it gives up and returns false.
template <typename F>
__device__ __forceinline__ bool collect(const char* slots, int nb, uint64_t tag, uint32_t limit, uint32_t phantoms,
                                        F&& f) {
    constexpr int GRP = 5;
    const int lane = threadIdx.x & 31;
    bool ok = true;
    for (int g0 = 0; g0 < nb; g0 += 32 * GRP) {
        float a[GRP], b[GRP];
        uint64_t t[GRP];
        uint32_t spins = 0;
        for (;;) {
            bool ready = phantoms == 0;
#pragma unroll
            for (int i = 0; i < GRP; ++i) {
                const int at = g0 + 32 * i + lane;
                t[i] = tag;
                a[i] = b[i] = 0.0f;
                if (at < nb) ld_slot(slots + (int64_t)at * RUN_SLOT_BYTES, a[i], b[i], t[i]);
            }
#pragma unroll
            for (int i = 0; i < GRP; ++i) ready &= t[i] == tag;
            if (__all_sync(0xffffffffu, ready)) break;
            if (++spins > limit) {
                ok = false;
                break;
            }
            if (spins > 64) __nanosleep(100);
        }
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < GRP; ++i)
            if (g0 + 32 * i + lane < nb) f(a[i], b[i]);
    }
    return ok;
}

// ---- warp totals of N values: log-step halving, N - 1 + (5 - log2 N) shuffles ----

constexpr int pow2_at_least(int n) { return n <= 1 ? 1 : n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 16; }

// Sums a[0..P) over the warp, P a power of two up to 16: at each step a lane
// keeps one half of the values and hands the other half to its partner. On
// return the lanes with (lane & (32 / P - 1)) == 0 hold, in a[0], the total of
// value slot_of_lane<P>(lane).
template <int P>
__device__ __forceinline__ void warp_totals(float (&a)[P]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int w = P; w > 1; w >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < w / 2; ++i) {
            const float send = up ? a[i] : a[i + w / 2];
            const float keep = up ? a[i + w / 2] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
}
template <int P>
__device__ __forceinline__ int slot_of_lane(int lane) {
    int s = 0;
#pragma unroll
    for (int w = P, o = 16; w > 1; w >>= 1, o >>= 1) s += (lane & o) ? w / 2 : 0;
    return s;
}

// ---- one pair of pixels in a sums pass ----

// The numerators are centered: num_j = sum u_j^m (x - v_j^k), so that
// v_j^{k+1} = v_j^k + num_j / den_j. The differences are at hand, and the FP32
// rounding of the sums is then relative to the pixels' distance from the center
// and not to their grey level, and vanishes from den as the run converges.
//
// Sums in two levels: pairs into num2/den2, those into num/den after every
// FOLD quads. A thread's share of a 256^3 volume is 54 quads; many of its terms
// are equal (a constant background), so a single chain of 108 additions rounds
// the same way again and again, in all threads alike. Uncentered and in one
// chain, the sums moved the iteration at which a random start of that volume
// breaks its symmetry by three.
constexpr int FOLD = 8;

template <int C>
struct SumAcc {
    f2 num2[C], den2[C], num[C], den[C];
    int held;
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int j = 0; j < C; ++j) num2[j] = den2[j] = num[j] = den[j] = pack2(0.0f, 0.0f);
        held = 0;
    }
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num[j] = add2(num[j], num2[j]);
            den[j] = add2(den[j], den2[j]);
            num2[j] = den2[j] = pack2(0.0f, 0.0f);
        }
        held = 0;
    }
    __device__ __forceinline__ void add(const f2 (&d2)[C], const f2 (&um2)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num2[j] = fma2(um2[j], d2[j], num2[j]);
            den2[j] = add2(den2[j], um2[j]);
        }
    }
};

// What the passes read of the run.
struct Px {
    const float* __restrict__ x;
    int64_t n;
    bool vec_x;   // x 16-byte aligned: quads of pixels
    bool vec_u;   // n % 4 == 0 and U, U^0 aligned too: quads of memberships
};

// Calls f(xa, xb) on packed pairs, the pixels (i, i+1) of a quad; tail(i) on
// the pixels past the last whole quad (at most three, on one thread). The
// loads run two steps ahead of their use.
template <typename F, typename T>
__device__ __forceinline__ void for_quads(const Px& px, int64_t t0, int64_t nt, F&& f, T&& tail) {
    const int64_t nq = px.n >> 2;
    const float4* x4 = reinterpret_cast<const float4*>(px.x);
    float4 a = t0 < nq ? __ldg(x4 + t0) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 b = t0 + nt < nq ? __ldg(x4 + t0 + nt) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t q = t0; q < nq; q += nt) {
        const float4 c = a;
        a = b;
        if (q + 2 * nt < nq) b = __ldg(x4 + q + 2 * nt);
        f(c, 4 * q);
    }
    if (t0 == nq % nt)
        for (int64_t i = 4 * nq; i < px.n; ++i) tail(i);
}

// The same for unaligned x or rows: a warp takes 128 consecutive pixels, a
// lane the pixels base + lane + 32 p, p = 0..3 (coalesced 32-bit accesses);
// whole tiles through f, the last partial one pixel by pixel through tail.
template <typename F, typename T>
__device__ __forceinline__ void for_tiles(const Px& px, int64_t t0, int64_t nt, F&& f, T&& tail) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = nt >> 5, w0 = t0 >> 5, tiles = (px.n + 127) >> 7;
    for (int64_t w = w0; w < tiles; w += nw) {
        const int64_t i = (w << 7) + lane;
        if ((w << 7) + 128 <= px.n) {
            const float4 c = make_float4(__ldg(px.x + i), __ldg(px.x + i + 32), __ldg(px.x + i + 64), __ldg(px.x + i + 96));
            f(c, i);
        } else {
#pragma unroll 1
            for (int64_t k = i; k < px.n; k += 32) tail(k);
        }
    }
}

template <int C>
struct RunShared {
    float red[RUN_NW][2 * C];  // warp totals of a sums pass; row 0..: J in red[w][0] of a full pass
    float mx[RUN_NW];
    unsigned bad[RUN_NW];
    DF vq[C];                  // V^{k+1} as double-float quotients
    int empty[C];
    DF J;
    float delta;
    unsigned flags;            // bit 0: bad input
    int err;
    float v[C], vp[C];         // V^k and V^{k-1}, for the rare scalar path and the sample
};

template <int C, int MK>
__global__ void __launch_bounds__(RUN_NT, 1) k_fcm_run(RunState* __restrict__ st, void* slots_raw, unsigned nonce) {
    constexpr int P = pow2_at_least(2 * C);
    constexpr bool SCALED = MK == M_ONE_HALF;
    __shared__ RunShared<C> sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * RUN_NT + threadIdx.x, nt = (int64_t)gridDim.x * RUN_NT;
    const int nb = (int)gridDim.x;
    const bool from_u = st->from_u != 0;
    const float* U0 = st->Uprev;  // may be U itself: each pixel is read, then written, by one thread
    float* U = st->U;
    Px px;
    px.x = st->x;
    px.n = st->n;
    px.vec_x = ((uintptr_t)px.x & 15) == 0;
    px.vec_u = px.vec_x && (px.n & 3) == 0 && ((uintptr_t)U & 15) == 0 && (!from_u || ((uintptr_t)U0 & 15) == 0);
    const int64_t n = px.n;
    const float m = st->m, inv_m1 = st->inv_m1, eps = st->eps;
    const int max_iter = st->max_iter;
    const uint32_t limit = st->lim.grid_spins, phantoms = st->lim.phantoms;
    double* const trace = st->trace;
    char* const slots = static_cast<char*>(slots_raw);

    if (threadIdx.x < C) sh.v[threadIdx.x] = sh.vp[threadIdx.x] = st->V0[threadIdx.x];
    if (threadIdx.x == 0) sh.err = 0;
    __syncthreads();
    f2 v2[C];
    DF v64[C];  // the double-float quotients behind V^k
#pragma unroll
    for (int j = 0; j < C; ++j) {
        v2[j] = pack2(sh.v[j], sh.v[j]);
        v64[j] = DF{sh.v[j], 0.0f};
    }
    int flags = 0;
    unsigned nx = 0;  // exchanges so far

    // Publishes this block's totals and collects every block's: the sums (or J)
    // of sh.red, the maximum of sh.mx and the flags of sh.bad. SUMS: cluster
    // totals -> sh.vq, sh.empty; otherwise J -> sh.J. centered: the numerators are
    // relative to V^k. Returns false when a wait gave up.
    auto exchange = [&](bool sums, bool centered) {
        __syncthreads();
        const uint64_t tag = ((uint64_t)nonce << 32) | ++nx;
        char* const mine = slots + (int64_t)(nx & 1) * (C + 1) * nb * RUN_SLOT_BYTES;
        const int nq = sums ? C : 1;
        if (warp < nq) {
            const int j = warp;
            float a = lane < RUN_NW ? sh.red[lane][j] : 0.0f, b = (sums && lane < RUN_NW) ? sh.red[lane][C + j] : 0.0f;
#pragma unroll
            for (int o = RUN_NW / 2; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                b += __shfl_xor_sync(0xffffffffu, b, o);
            }
            char* const row = mine + (int64_t)j * nb * RUN_SLOT_BYTES;
            if (lane == 0) st_slot(row + (int64_t)blockIdx.x * RUN_SLOT_BYTES, a, b, tag);
            DF na{0.0f, 0.0f}, da{0.0f, 0.0f};
            const bool ok = collect(row, nb, tag, limit, phantoms, [&](float p, float q) {
                df_add(na, p);
                df_add(da, q);
            });
            if (!ok && lane == 0) sh.err = 1;
            DF d[2] = {na, da};
            warp_sum_df_n<2>(d);
            if (lane == 0) {
                if (sums) {
                    const bool empty = !(d[1].hi > 0.0f);
                    DF q = empty ? DF{0.0f, 0.0f} : df_div(d[0], d[1]);
                    if (centered) {
                        if (SCALED) {
                            const float s = __frcp_rn(spread_scale<C>(v2));  // a power of two: exact
                            q = DF{q.hi * s, q.lo * s};
                        }
                        q = df_merge(q, DF{sh.v[j], 0.0f});
                    }
                    sh.vq[j] = q;
                    sh.empty[j] = empty;
                } else {
                    sh.J = d[0];
                }
            }
        } else if (warp == C) {
            unsigned mb = lane < RUN_NW ? __float_as_uint(sh.mx[lane]) : 0u, fb = lane < RUN_NW ? sh.bad[lane] : 0u;
            mb = __reduce_max_sync(0xffffffffu, mb);  // non-negative floats order as their bits
            fb = __reduce_or_sync(0xffffffffu, fb);
            char* const row = mine + (int64_t)C * nb * RUN_SLOT_BYTES;
            if (lane == 0) st_slot(row + (int64_t)blockIdx.x * RUN_SLOT_BYTES, __uint_as_float(mb), __uint_as_float(fb), tag);
            unsigned tm = 0u, tf = 0u;
            const bool ok = collect(row, nb, tag, limit, phantoms, [&](float p, float q) {
                tm = max(tm, __float_as_uint(p));
                tf |= __float_as_uint(q);
            });
            if (!ok && lane == 0) sh.err = 1;
            tm = __reduce_max_sync(0xffffffffu, tm);
            tf = __reduce_or_sync(0xffffffffu, tf);
            if (lane == 0) {
                sh.delta = __uint_as_float(tm);
                sh.flags = tf;
            }
        }
        __syncthreads();
        return sh.err == 0;
    };
    // This warp's totals of a sums pass into sh.red / sh.mx / sh.bad.
    auto warp_publish = [&](const float (&num)[C], const float (&den)[C], float mx, bool bad) {
        float a[P];
#pragma unroll
        for (int i = 0; i < P; ++i) a[i] = i < C ? num[i < C ? i : 0] : i < 2 * C ? den[i < 2 * C && i >= C ? i - C : 0] : 0.0f;
        warp_totals<P>(a);
        const int s = slot_of_lane<P>(lane);
        if ((lane & (32 / P - 1)) == 0 && s < 2 * C) sh.red[warp][s] = a[0];
        const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
        const bool any = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            sh.mx[warp] = __uint_as_float(mb);
            sh.bad[warp] = any ? 1u : 0u;
        }
    };

    // ---- a sums pass from V^k (also pass 0 from V^0, which checks x) ----
    SumAcc<C> a;
    auto sums_pass = [&](float dmax, bool check_x) {
        a.reset();
        float tn[C], td[C];  // pixels that do not fill a pair
#pragma unroll
        for (int j = 0; j < C; ++j) tn[j] = td[j] = 0.0f;
        bool bad = false;
        f2 vq2[C], s2;
        if (SCALED) {
            const float s = spread_scale<C>(v2);
            s2 = pack2(s, s);
        }
#pragma unroll
        for (int j = 0; j < C; ++j) vq2[j] = SCALED ? mul2(v2[j], s2) : v2[j];
        auto quad = [&](const float4& c, int64_t) {
            const f2 xa = pack2(c.x, c.y), xb = pack2(c.z, c.w);
            if (check_x) bad |= !(finite_f(c.x) && finite_f(c.y) && finite_f(c.z) && finite_f(c.w));
            f2 um[C], d2[C];
            powers_pair<C, MK>(xa, SCALED ? mul2(xa, s2) : xa, vq2, m, inv_m1, sh.v, um, d2);
            a.add(d2, um);
            powers_pair<C, MK>(xb, SCALED ? mul2(xb, s2) : xb, vq2, m, inv_m1, sh.v, um, d2);
            a.add(d2, um);
            if (++a.held == FOLD) a.fold();
        };
        auto single = [&](int64_t i) {
            const float xi = __ldg(px.x + i);
            if (check_x) bad |= !finite_f(xi);
            const Powers<C> w = powers_scalar<C, MK>(xi, xi, sh.v, m, inv_m1);
#pragma unroll
            for (int j = 0; j < C; ++j) {
                tn[j] = fmaf(w.a[j], SCALED ? lo2(mul2(pack2(xi, xi), s2)) - lo2(vq2[j]) : xi - lo2(vq2[j]), tn[j]);
                td[j] += w.a[j];
            }
        };
        if (px.vec_x) for_quads(px, t0, nt, quad, single);
        else for_tiles(px, t0, nt, quad, single);
        if (check_x && threadIdx.x < C) bad |= !finite_f(sh.v[threadIdx.x]);
        a.fold();
#pragma unroll
        for (int j = 0; j < C; ++j) {
            tn[j] += lo2(a.num[j]) + hi2(a.num[j]);
            td[j] += lo2(a.den[j]) + hi2(a.den[j]);
        }
        warp_publish(tn, td, dmax, bad);
    };

    // ---- pass 0: V^1 from U^0, or from U^0 = f(x, V^0) ----
    if (from_u) {
        // four pixels in FP32, then double-float: the pass waits for memory, and
        // the separation of the V^1 of a random start is of the order of 1e-5
        DF sn[C], sd[C];
        float num[C], den[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            sn[j] = sd[j] = DF{0.0f, 0.0f};
            num[j] = den[j] = 0.0f;
        }
        bool bad = false;
        auto one = [&](float xi, float u0, int j) {
            bad |= !(u0 >= 0.0f) || !finite_f(u0);
            const float w = pow_m<MK>(u0, m);
            num[j] = fmaf(w, xi, num[j]);
            den[j] += w;
        };
        auto fold = [&] {
#pragma unroll
            for (int j = 0; j < C; ++j) {
                df_add(sn[j], num[j]);
                df_add(sd[j], den[j]);
                num[j] = den[j] = 0.0f;
            }
        };
        auto quad_v = [&](const float4& c, int64_t i) {
            bad |= !(finite_f(c.x) && finite_f(c.y) && finite_f(c.z) && finite_f(c.w));
            float4 u[C];
#pragma unroll
            for (int j = 0; j < C; ++j) u[j] = __ldcs(reinterpret_cast<const float4*>(U0 + (int64_t)j * n + i));
#pragma unroll
            for (int j = 0; j < C; ++j) {
                one(c.x, u[j].x, j);
                one(c.y, u[j].y, j);
                one(c.z, u[j].z, j);
                one(c.w, u[j].w, j);
            }
            fold();
        };
        auto quad_t = [&](const float4& c, int64_t i) {
            bad |= !(finite_f(c.x) && finite_f(c.y) && finite_f(c.z) && finite_f(c.w));
#pragma unroll
            for (int p = 0; p < 4; ++p) {
#pragma unroll
                for (int j = 0; j < C; ++j) one(comp(c, p), __ldcs(U0 + (int64_t)j * n + i + 32 * p), j);
            }
            fold();
        };
        auto single = [&](int64_t i) {
            const float xi = __ldg(px.x + i);
            bad |= !finite_f(xi);
#pragma unroll
            for (int j = 0; j < C; ++j) one(xi, __ldcs(U0 + (int64_t)j * n + i), j);
        };
        if (px.vec_u) for_quads(px, t0, nt, quad_v, single);
        else for_tiles(px, t0, nt, quad_t, single);
        fold();
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num[j] = sn[j].hi + sn[j].lo;
            den[j] = sd[j].hi + sd[j].lo;
        }
        warp_publish(num, den, 0.0f, bad);
    } else {
        sums_pass(0.0f, true);
    }
    bool ok = exchange(true, !from_u);

    int status = FCM_NOT_CONVERGED, iters = 0;
    if (!ok) {
        status = FCM_ERR_TIMEOUT;
    } else if (sh.flags & 1u) {
        status = FCM_ERR_BAD_INPUT;
        ok = false;
    }
    // V^{k+1} of the last exchange becomes V^k (an empty cluster keeps its
    // center; in pass 0 that is V^0, or 0 from a U^0).
    auto advance = [&](bool first) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const float old = lo2(v2[j]);
            float nv = old;
            if (sh.empty[j]) {
                flags |= FCM_FLAG_EMPTY_CLUSTER;
                if (first && from_u) {
                    nv = 0.0f;
                    v64[j] = DF{0.0f, 0.0f};
                }
            } else {
                v64[j] = sh.vq[j];
                nv = v64[j].hi;
            }
            if (threadIdx.x == 0) {
                sh.vp[j] = old;
                sh.v[j] = nv;
            }
            v2[j] = pack2(nv, nv);
        }
        __syncthreads();
    };

    // The sampled pair of this thread: the first pair that a full pass gives it
    // (the same pairs, so the sample's changes are bit for bit those of the full
    // pass), until a full pass has found its pair of largest change.
    f2 wx = 0;
    const int64_t wi = px.vec_u ? 4 * t0 : ((t0 >> 5) << 7) + lane;
    const int ws = px.vec_u ? 1 : 32;
    bool sampled = px.vec_u ? t0 < (n >> 2) : ((t0 >> 5) << 7) + 128 <= n;
    bool wide = false;  // every warp samples (after a full pass that did not stop the run)
    if (sampled) wx = pack2(__ldg(px.x + wi), __ldg(px.x + wi + ws));
    // U^k of a pair and its largest |U^k - U^{k-1}|; U^{k-1} is given (u0) or
    // comes from V^{k-1}. J2: the pair's J terms.
    auto change = [&](f2 xq, f2 (&u2)[C], const f2 (&u0)[C], bool given, f2& J2) {
        f2 um2[C], uo2[C], vp2[C];
        J2 = membership_pair<C, MK>(xq, v2, m, inv_m1, sh.v, u2, um2);
        if (given) {
#pragma unroll
            for (int j = 0; j < C; ++j) uo2[j] = u0[j];
        } else {
#pragma unroll
            for (int j = 0; j < C; ++j) vp2[j] = pack2(sh.vp[j], sh.vp[j]);
            membership_pair<C, MK>(xq, vp2, m, inv_m1, sh.vp, uo2, um2);
        }
        float d = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            float da, db;
            unpack2(sub2(u2[j], uo2[j]), da, db);
            d = fmaxf(d, fmaxf(fabsf(da), fabsf(db)));
        }
        return d;
    };
    if (ok) advance(true);
    for (int k = 1; ok; ++k) {
        const bool last = k == max_iter, prev_u0 = from_u && k == 1;
        bool go_on = false;
        if (!last) {
            float dmax = 0.0f;
            if (sampled && (wide || warp < SAMPLE_WARPS)) {
                f2 u0[C], u2[C];
                if (prev_u0) {
#pragma unroll
                    for (int j = 0; j < C; ++j)
                        u0[j] = pack2(__ldcs(U0 + (int64_t)j * n + wi), __ldcs(U0 + (int64_t)j * n + wi + ws));
                }
                f2 J2;
                dmax = change(wx, u2, u0, prev_u0, J2);
            }
            sums_pass(dmax, false);
            if (!exchange(true, true)) {
                status = FCM_ERR_TIMEOUT;
                iters = k;
                break;
            }
            go_on = sh.delta >= eps;
        }
        if (!go_on || trace) {
            // ---- full pass: delta_k and J_k over every pixel, U^k ----
            const bool emit = !go_on;
            f2 J2 = pack2(0.0f, 0.0f);
            float J1 = 0.0f, dmax = 0.0f;
            auto pair = [&](f2 xq, f2 (&u2)[C], const f2 (&u0)[C]) {
                f2 j2;
                const float d = change(xq, u2, u0, prev_u0, j2);
                J2 = add2(J2, j2);
                if (d > dmax) {
                    dmax = d;
                    wx = xq;
                    sampled = true;
                }
            };
            auto quad_v = [&](const float4& c, int64_t i) {
                f2 ua[C], ub[C], u0a[C], u0b[C];
                if (prev_u0) {
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        const float4 u = __ldcs(reinterpret_cast<const float4*>(U0 + (int64_t)j * n + i));
                        u0a[j] = pack2(u.x, u.y);
                        u0b[j] = pack2(u.z, u.w);
                    }
                }
                pair(pack2(c.x, c.y), ua, u0a);
                pair(pack2(c.z, c.w), ub, u0b);
                if (emit) {
#pragma unroll
                    for (int j = 0; j < C; ++j) st_u4(U + (int64_t)j * n + i, make_float4(lo2(ua[j]), hi2(ua[j]), lo2(ub[j]), hi2(ub[j])));
                }
            };
            auto quad_t = [&](const float4& c, int64_t i) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    f2 u[C], u0[C];
                    const int64_t ia = i + 64 * h, ib = ia + 32;
                    if (prev_u0) {
#pragma unroll
                        for (int j = 0; j < C; ++j) u0[j] = pack2(__ldcs(U0 + (int64_t)j * n + ia), __ldcs(U0 + (int64_t)j * n + ib));
                    }
                    pair(h ? pack2(c.z, c.w) : pack2(c.x, c.y), u, u0);
                    if (emit) {
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            __stcs(U + (int64_t)j * n + ia, lo2(u[j]));
                            __stcs(U + (int64_t)j * n + ib, hi2(u[j]));
                        }
                    }
                }
            };
            auto single = [&](int64_t i) {
                const float xi = __ldg(px.x + i);
                float u[C], um[C], up[C], ump[C];
                float vv[C], vvp[C];
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    vv[j] = sh.v[j];
                    vvp[j] = sh.vp[j];
                }
                J1 += membership<C, MK>(xi, vv, m, inv_m1, u, um);
                if (prev_u0) {
#pragma unroll
                    for (int j = 0; j < C; ++j) up[j] = __ldcs(U0 + (int64_t)j * n + i);
                } else {
                    membership<C, MK>(xi, vvp, m, inv_m1, up, ump);
                }
                float d = 0.0f;
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    d = fmaxf(d, fabsf(u[j] - up[j]));
                    if (emit) __stcs(U + (int64_t)j * n + i, u[j]);
                }
                dmax = fmaxf(dmax, d);
            };
            if (px.vec_u) for_quads(px, t0, nt, quad_v, single);
            else for_tiles(px, t0, nt, quad_t, single);
            wide = true;
            J1 = warp_sum(J1 + lo2(J2) + hi2(J2));
            const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(dmax));
            if (lane == 0) {
                sh.red[warp][0] = J1;
                sh.mx[warp] = __uint_as_float(mb);
                sh.bad[warp] = 0u;
            }
            if (!exchange(false, false)) {
                status = FCM_ERR_TIMEOUT;
                iters = k;
                break;
            }
            const float delta = sh.delta;
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                st->delta = delta;
                st->J = df_to_double(sh.J);
                if (trace) {
                    double* t = trace + (int64_t)(k - 1) * (2 + C);
                    t[0] = delta;
                    t[1] = df_to_double(sh.J);
#pragma unroll
                    for (int j = 0; j < C; ++j) t[2 + j] = df_to_double(v64[j]);
                }
            }
            if (!go_on && (delta < eps || last)) {
                status = delta < eps ? FCM_OK : FCM_NOT_CONVERGED;
                iters = k;
                break;
            }
            // the run goes on from the V^{k+1} of the sums pass (still in sh.vq)
        }
        advance(false);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            st->V[j] = lo2(v2[j]);
            st->V64[j] = df_to_double(v64[j]);
        }
        st->status = status;
        st->iters = iters;
        st->k = iters;
        st->flags = flags;
        st->done = 1;
        st->Uprev = st->U;
    }
}

template <int C>
void fill(RunTable& t) {
    t.run[C][M_TWO] = k_fcm_run<C, M_TWO>;
    t.run[C][M_THREE] = k_fcm_run<C, M_THREE>;
    t.run[C][M_ONE_HALF] = k_fcm_run<C, M_ONE_HALF>;
    t.run[C][M_GENERIC] = k_fcm_run<C, M_GENERIC>;
}

}  // namespace

#define FCM_CAT2(a, b) a##b
#define FCM_CAT(a, b) FCM_CAT2(a, b)
void FCM_CAT(register_run_c, FCM_INST_C)(RunTable& t) { fill<FCM_INST_C>(t); }

}  // namespace fcm
