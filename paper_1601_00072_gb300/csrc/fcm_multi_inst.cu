// Multi-feature FCM: pixels with D channels (colour, or co-registered MR
// sequences), one cooperative launch per run.
//
// Compiled once per channel count with -DFCM_MULTI_D=1..4.
//
// Sec. 2.1 defines d_ij as a norm of x_i - v_j; with D channels it is the
// Euclidean norm over the channels, so Eq. 4 takes d_ij^2 = sum_d (x_id -
// v_jd)^2, Eq. 3 gives each center channel by channel, and Eq. 1 sums
// u_ij^m d_ij^2. The loop is Algorithm 1 with the readings of the scalar
// path (zero distance, L-infinity stopping test, empty clusters).
//
// As in the scalar whole-run kernel no U is stored between iterations: a sums
// pass reads x (4D bytes per pixel) and adds up Eq. 3's sums, centered on V^k, in
// packed FP32x2 pairs of pixels; the change |U^k - U^{k-1}| is taken over a sample,
// which bounds delta_k from below, and over every pixel (with J_k and the write of
// U^k) in a full pass only when that bound does not reach eps or k is max_iter.
// Every block adds the per-block sums (compensated FP32 pairs) in the same order
// after a bounded grid barrier, so all blocks take the same decisions.
// Bound by the block's and the grid's barriers, with the sums behind them (the
// largest stall at 4 M pixels too), then by the FP32 pipe (about 60 operations per
// pixel and iteration at C = 4, D = 3; 37 % of cycles).
// 3 channels of 2048^2 pixels, C = 4, 30 iterations: 1.50 -> 0.64 ms (memberships
// twice per iteration, scalar, double-float sums every four pixels before).
#include "fcm_device.cuh"
#include "fcm_df.cuh"
#include "fcm_multi.h"

#ifndef FCM_MULTI_D
#error "compile with -DFCM_MULTI_D=<channels>"
#endif

namespace fcm {
namespace {

constexpr int D = FCM_MULTI_D;
constexpr int MNT = MULTI_NT;
constexpr int MNW = MNT / 32;
constexpr int MFOLD = 8;         // pairs added in registers before they go to the second set of sums (FP32,
                                 // centered: errors against 64 bits are those of uncentered sums folded
                                 // into double-float every four pixels, over 2^12 to 2^22 pixels)
constexpr int MSAMPLE_WARPS = 2; // warps per block that sample delta_k
// The FP32 differences x - v_j^k round by 2^-24 of the step at most, so up to this
// factor (of the largest channel of the new center) the center keeps about 18 bits;
// beyond it, the sums are taken again, centered on the new one.
constexpr float REBASE = 64.0f;

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Memberships of one pixel from its squared distances d2[j] (Eq. 4 in the
// weight form w_j = (d2min / d2_j)^(1/(m-1)), u_j = w_j / sum_k w_k, with the
// zero-distance rule). A squared distance below the smallest normal float
// (2^-126) counts as zero, as the .ftz reciprocal and logarithm would read
// it. Returns the pixel's J term, d2min * S^(1-m).
template <int C, int MK>
__device__ __forceinline__ float membership_d2(const float (&d2)[C], float m, float inv_m1, float (&u)[C],
                                               float (&um)[C]) {
    float dmin = __int_as_float(0x7f800000);
#pragma unroll
    for (int j = 0; j < C; ++j) dmin = fminf(dmin, d2[j]);
    float Ji = 0.0f;
    if (dmin >= flt_min()) {
        float w[C];
        if (MK == M_TWO) {
#pragma unroll
            for (int j = 0; j < C; ++j) w[j] = dmin * rcp_approx(d2[j]);
        } else {
            const float l0 = lg2_approx(dmin);
#pragma unroll
            for (int j = 0; j < C; ++j) w[j] = ex2_approx(inv_m1 * (l0 - lg2_approx(d2[j])));
        }
        float S = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) S += w[j];
        const float r = rcp_approx(S);
#pragma unroll
        for (int j = 0; j < C; ++j) u[j] = w[j] * r;
        Ji = (MK == M_TWO) ? dmin * r : dmin * ex2_approx((1.0f - m) * lg2_approx(S));
    } else {
        int nz = 0;
#pragma unroll
        for (int j = 0; j < C; ++j) nz += (d2[j] < flt_min());
        const float share = __fdiv_rn(1.0f, (float)nz);
#pragma unroll
        for (int j = 0; j < C; ++j) u[j] = (d2[j] < flt_min()) ? share : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < C; ++j) um[j] = (MK == M_TWO) ? u[j] * u[j] : ex2_approx(m * lg2_approx(u[j]));
    return Ji;
}

template <int C>
__device__ __forceinline__ void dist2(const float (&xv)[D], const float* vs, float (&d2)[C]) {
#pragma unroll
    for (int j = 0; j < C; ++j) {
        float s = 0.0f;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const float t = xv[d] - vs[j * D + d];
            s = fmaf(t, t, s);
        }
        d2[j] = s;
    }
}

// Memberships of one pixel from centers vs[C * D] (the full pass and the sample).
template <int C, int MK>
__device__ __noinline__ float pixel_memberships(const float (&xv)[D], const float* vs, float m, float inv_m1, float* u) {
    float d2[C], ul[C], um[C];
    dist2<C>(xv, vs, d2);
    const float J = membership_d2<C, MK>(d2, m, inv_m1, ul, um);
#pragma unroll
    for (int j = 0; j < C; ++j) u[j] = ul[j];
    return J;
}

// u^m of a pair of pixels, and their differences t2 from the centers v2.
template <int C, int MK>
__device__ __forceinline__ void pair_powers(const f2 (&x2)[D], const f2 (&v2)[C][D], float m, float inv_m1,
                                            f2 (&um2)[C], f2 (&t2)[C][D]) {
    f2 b[C];
#pragma unroll
    for (int j = 0; j < C; ++j) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            t2[j][d] = sub2(x2[d], v2[j][d]);
            b[j] = d == 0 ? mul2(t2[j][d], t2[j][d]) : fma2(t2[j][d], t2[j][d], b[j]);
        }
    }
    if (MK == M_TWO) {
        // the product form of the scalar kernels: one reciprocal per pixel
        f2 P[C];
        co_products<C>(b, P);
        f2 S = P[0];
#pragma unroll
        for (int j = 1; j < C; ++j) S = add2(S, P[j]);
        float s0, s1;
        unpack2(S, s0, s1);
        if (max(__float_as_uint(s0) - 0x00800000u, __float_as_uint(s1) - 0x00800000u) < 0x7f000000u) {
            const f2 r = pack2(rcp_approx(s0), rcp_approx(s1));
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const f2 u = mul2(P[j], r);
                um2[j] = mul2(u, u);
            }
            return;
        }
    } else {
        float ta[C], tb[C], la = __int_as_float(0x7f800000), lb = la;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            ta[j] = lg2_approx(lo2(b[j]));  // a square below 2^-126 reads as 0: -inf
            tb[j] = lg2_approx(hi2(b[j]));
            la = fminf(la, ta[j]);
            lb = fminf(lb, tb[j]);
        }
        if (fminf(la, lb) >= -126.0f) {
            float Sa = 0.0f, Sb = 0.0f;
#pragma unroll
            for (int j = 0; j < C; ++j) {
                ta[j] = inv_m1 * (la - ta[j]);
                tb[j] = inv_m1 * (lb - tb[j]);
                Sa += ex2_approx(ta[j]);
                Sb += ex2_approx(tb[j]);
            }
            const float ga = lg2_approx(Sa), gb = lg2_approx(Sb);
#pragma unroll
            for (int j = 0; j < C; ++j) um2[j] = pack2(ex2_approx(m * (ta[j] - ga)), ex2_approx(m * (tb[j] - gb)));
            return;
        }
    }
    float da[C], db[C], u[C], ua[C], ub[C];
#pragma unroll
    for (int j = 0; j < C; ++j) unpack2(b[j], da[j], db[j]);
    membership_d2<C, MK>(da, m, inv_m1, u, ua);
    membership_d2<C, MK>(db, m, inv_m1, u, ub);
#pragma unroll
    for (int j = 0; j < C; ++j) um2[j] = pack2(ua[j], ub[j]);
}

// Sums of eight values over the warp by log-step halving (nine shuffles); the
// lanes with (lane & 3) == 0 end with the total of value `slot` in a[0].
__device__ __forceinline__ int warp_totals8(float (&a)[8]) {
    const int lane = threadIdx.x & 31;
    int slot = 0;
#pragma unroll
    for (int w = 8, o = 16; w > 1; w >>= 1, o >>= 1) {
        const bool up = lane & o;
        slot += up ? w / 2 : 0;
#pragma unroll
        for (int i = 0; i < w / 2; ++i) {
            const float send = up ? a[i] : a[i + w / 2], keep = up ? a[i + w / 2] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    return slot;
}

// A warp's sums from the centers `cur`, centered on `base`, into w[0..C D + C).
// Called, not inlined: rare, and the usual passes keep their registers.
template <int C, int MK>
__device__ __noinline__ void rebased_sums(const float* x, int64_t n, int64_t t0, int64_t nt, const float* cur,
                                          const float* base, float m, float inv_m1, DF* w) {
    for (int j = 0; j < C; ++j) {
        DF acc[D + 1];
#pragma unroll
        for (int d = 0; d <= D; ++d) acc[d] = DF{0.0f, 0.0f};
        for (int64_t i = t0; i < n; i += nt) {
            float xv[D], u[C];
#pragma unroll
            for (int d = 0; d < D; ++d) xv[d] = __ldg(x + (int64_t)d * n + i);
            pixel_memberships<C, MK>(xv, cur, m, inv_m1, u);
            const float um = (MK == M_TWO) ? u[j] * u[j] : ex2_approx(m * lg2_approx(u[j]));
            df_add(acc[D], um);
#pragma unroll
            for (int d = 0; d < D; ++d) df_add(acc[d], um * (xv[d] - base[j * D + d]));
        }
#pragma unroll
        for (int d = 0; d <= D; ++d) {
            const DF t = warp_sum_df(acc[d]);
            if ((threadIdx.x & 31) == 0) w[d < D ? j * D + d : C * D + j] = t;
        }
    }
}

// Pass 0 is INIT (V^1 from U^0, or from U^0 = f(x, V^0)).
template <int C, int MK, bool FROM_U>
__global__ void __launch_bounds__(MNT, 1) k_fcm_run_multi(MultiState* __restrict__ st, float* __restrict__ partials) {
    constexpr int NV = C * D + C;  // num[C][D], den[C] (compensated); a full pass uses slot 0 for J
    constexpr int S = NV + 3;      // then max|dU|, bad input, spare
    constexpr int NP = (NV + 7) / 8 * 8;
    extern __shared__ __align__(16) f2 second[];  // [NV][MNT] second set of the sums
    __shared__ float s_v[3][C * D];               // V^k, V^{k-1} and V^{k+1} in turn
    __shared__ DF s_v64[3][C * D];
    __shared__ DF s_w[MNW][NP];
    __shared__ float s_m[MNW];
    __shared__ int s_b[MNW];
    __shared__ DF s_df[NV];
    __shared__ float s_mx[2];
    __shared__ float s_wit[MNW][D];               // each warp's pixel of largest change in a full pass
    __shared__ int s_err, s_empty, s_far;

    const float* __restrict__ x = st->x;
    const float* U0 = st->U0;  // may be U itself: each pixel is read, then written, by one thread
    float* U = st->U;
    const int64_t n = st->n;
    const float m = st->m, inv_m1 = st->inv_m1, eps = st->eps;
    const int max_iter = st->max_iter;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nb = (int)gridDim.x;
    for (int t = threadIdx.x; t < C * D; t += MNT) {
        s_v[0][t] = st->V0[t];
        s_v64[0][t] = DF{st->V0[t], 0.0f};
    }
    if (threadIdx.x == 0) s_err = s_empty = s_far = 0;
    int flags = 0, parity = 0;
    unsigned arrived = 0;
    __syncthreads();

    const int64_t t0 = (int64_t)blockIdx.x * MNT + threadIdx.x, nt = (int64_t)nb * MNT, npair = n >> 1;
    // pairs of pixels with one 64-bit load per channel when every row allows it
    const bool vec = (n & 1) == 0 && ((uintptr_t)x & 7) == 0;
    auto load_pair = [&](int64_t q, f2 (&x2)[D]) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const float* p = x + (int64_t)d * n + 2 * q;
            if (vec) {
                const float2 v = __ldg(reinterpret_cast<const float2*>(p));
                x2[d] = pack2(v.x, v.y);
            } else {
                x2[d] = pack2(__ldg(p), __ldg(p + 1));
            }
        }
    };
    // The block's totals (s_w per warp, s_m, s_b) -> the grid's: s_df[0..nv), s_mx.
    // False when the bounded barrier gave up.
    auto exchange = [&](int nv) {
        __syncthreads();
        float* part = partials + (int64_t)parity * (2 * S) * nb;
        if (threadIdx.x < nv) {
            const int q = threadIdx.x;
            DF t = s_w[0][q];
            for (int w = 1; w < MNW; ++w) t = df_merge(t, s_w[w][q]);
            __stcg(part + (int64_t)(2 * q) * nb + blockIdx.x, t.hi);
            __stcg(part + (int64_t)(2 * q + 1) * nb + blockIdx.x, t.lo);
        } else if (threadIdx.x >= MNT - 32) {
            const unsigned mb = __reduce_max_sync(0xffffffffu, lane < MNW ? __float_as_uint(s_m[lane]) : 0u);
            const unsigned bb = __reduce_or_sync(0xffffffffu, lane < MNW ? (unsigned)s_b[lane] & 1u : 0u);
            if (lane == 0) {
                __stcg(part + (int64_t)(2 * NV) * nb + blockIdx.x, __uint_as_float(mb));
                __stcg(part + (int64_t)(2 * NV + 1) * nb + blockIdx.x, bb ? 1.0f : 0.0f);
            }
        }
        __syncthreads();
        ++arrived;
        // bounded by st->lim: grid_spins polls, for the grid's arrivals plus
        // st->lim.phantoms (0 unless a test injects a barrier that never fills)
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&st->ticket, 1u);
            const unsigned target = arrived * gridDim.x + st->lim.phantoms;
            const uint32_t limit = st->lim.grid_spins;
            uint32_t spins = 0;
            while (ld_acquire_u32(&st->ticket) < target) {
                if (++spins > limit) {
                    s_err = 1;
                    break;
                }
                __nanosleep(32);
            }
            __threadfence();
        }
        __syncthreads();
        if (s_err) return false;
        // the same fixed order in every block
        for (int q = warp; q <= nv; q += MNW) {
            const int slot = q < nv ? q : NV;
            const float* ph = part + (int64_t)(2 * slot) * nb;
            const float* pl = ph + nb;
            if (q < nv) {
                DF d{0.0f, 0.0f};
#pragma unroll 5
                for (int b = lane; b < nb; b += 32) d = df_merge(d, DF{__ldcg(ph + b), __ldcg(pl + b)});
                d = warp_sum_df(d);
                if (lane == 0) s_df[q] = d;
            } else {
                float t = 0.0f, f = 0.0f;
#pragma unroll 5
                for (int b = lane; b < nb; b += 32) {
                    t = fmaxf(t, __ldcg(ph + b));
                    f = fmaxf(f, __ldcg(pl + b));
                }
                t = warp_max(t);
                f = warp_max(f);
                if (lane == 0) {
                    s_mx[0] = t;
                    s_mx[1] = f;
                }
            }
        }
        parity ^= 1;
        __syncthreads();
        return true;
    };
    // V^{k+1} into slot nxt from the sums; cur: the slot the numerators are centered
    // on (nxt itself for rebased sums), or -1. An empty cluster keeps its center
    // (pass 0: V^0, or 0 from a U^0).
    auto centers = [&](int cur, int nxt) {
        if (threadIdx.x < C * D) {
            const int t = threadIdx.x, j = t / D;
            const DF den = s_df[C * D + j];
            DF v = cur >= 0 ? s_v64[cur][t] : DF{0.0f, 0.0f};
            if (den.hi > 0.0f) {
                v = df_div(s_df[t], den);
                if (cur >= 0) {
                    const float step = fabsf(v.hi);
                    v = df_merge(v, DF{s_v[cur][t], 0.0f});
                    if (step > REBASE * fabsf(v.hi)) s_far = 1;
                }
            } else {
                s_empty = 1;
            }
            s_v[nxt][t] = v.hi;
            s_v64[nxt][t] = v;
        }
        __syncthreads();
    };
    // s_far says that some channel of a center moved far: whether one moved by more
    // than its largest channel is worth, and then V^{k+1} again from sums centered on
    // slot nxt (the scalar form: rare). False when the barrier gave up.
    auto rebase = [&](int cur, int nxt) {
        bool far = false;
        for (int j = 0; j < C; ++j) {
            float step = 0.0f, size = 0.0f;
            for (int d = 0; d < D; ++d) {
                step = fmaxf(step, fabsf(s_v[nxt][j * D + d] - s_v[cur][j * D + d]));
                size = fmaxf(size, fabsf(s_v[nxt][j * D + d]));
            }
            far |= step > REBASE * size;
        }
        __syncthreads();
        if (threadIdx.x == 0) s_far = 0;
        if (!far) return true;
        rebased_sums<C, MK>(x, n, t0, nt, s_v[cur], s_v[nxt], m, inv_m1, s_w[warp]);
        if (!exchange(NV)) return false;
        centers(nxt, nxt);
        __syncthreads();
        if (threadIdx.x == 0) s_far = 0;
        return true;
    };
    auto publish = [&](float (&a)[NP], float mx, bool bad) {
#pragma unroll
        for (int g = 0; g < NP / 8; ++g) {
            float t[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) t[i] = a[8 * g + i];
            const int slot = warp_totals8(t);
            if ((lane & 3) == 0) s_w[warp][8 * g + slot] = DF{t[0], 0.0f};
        }
        const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
        const bool any = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            s_m[warp] = __uint_as_float(mb);
            s_b[warp] = any ? 1 : 0;
        }
    };
    // A sums pass from V^k in slot cur (check: pass 0 from V^0).
    auto sums_pass = [&](int cur, float dmax, bool check) {
        f2 v2[C][D], num2[C][D], den2[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            den2[j] = pack2(0.0f, 0.0f);
#pragma unroll
            for (int d = 0; d < D; ++d) {
                v2[j][d] = pack2(s_v[cur][j * D + d], s_v[cur][j * D + d]);
                num2[j][d] = pack2(0.0f, 0.0f);
            }
        }
        bool bad = check && threadIdx.x < C * D && !finite_f(s_v[cur][threadIdx.x]);
        f2* const set = second + threadIdx.x;
        int held = 0;
        bool folded = false;
        f2 nx2[D];
        if (t0 < npair) load_pair(t0, nx2);
#pragma unroll 1
        for (int64_t q = t0; q < npair; q += nt) {
            f2 x2[D], um2[C], t2[C][D];
#pragma unroll
            for (int d = 0; d < D; ++d) x2[d] = nx2[d];
            if (q + nt < npair) load_pair(q + nt, nx2);
            if (check) {
#pragma unroll
                for (int d = 0; d < D; ++d) bad |= !(finite_f(lo2(x2[d])) && finite_f(hi2(x2[d])));
            }
            pair_powers<C, MK>(x2, v2, m, inv_m1, um2, t2);
#pragma unroll
            for (int j = 0; j < C; ++j) {
                den2[j] = add2(den2[j], um2[j]);
#pragma unroll
                for (int d = 0; d < D; ++d) num2[j][d] = fma2(um2[j], t2[j][d], num2[j][d]);
            }
            if (++held == MFOLD) {
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    f2& a = i < C * D ? num2[i / D < C ? i / D : 0][i % D] : den2[i >= C * D ? i - C * D : 0];
                    f2* const p = set + i * MNT;
                    *p = folded ? add2(*p, a) : a;
                    a = pack2(0.0f, 0.0f);
                }
                folded = true;
                held = 0;
            }
        }
        float t[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            t[i] = 0.0f;
            if (i < NV) {
                f2 a = i < C * D ? num2[i / D < C ? i / D : 0][i % D] : den2[(i >= C * D && i < NV) ? i - C * D : 0];
                if (folded) a = add2(a, set[i * MNT]);
                t[i] = lo2(a) + hi2(a);
            }
        }
        if ((n & 1) && t0 == npair % nt) {
            // the last, unpaired pixel
            float xv[D], d2[C], u[C], um[C];
#pragma unroll
            for (int d = 0; d < D; ++d) {
                xv[d] = __ldg(x + (int64_t)d * n + n - 1);
                if (check) bad |= !finite_f(xv[d]);
            }
            dist2<C>(xv, s_v[cur], d2);
            membership_d2<C, MK>(d2, m, inv_m1, u, um);
#pragma unroll
            for (int j = 0; j < C; ++j) {
                t[C * D + j] += um[j];
#pragma unroll
                for (int d = 0; d < D; ++d) t[j * D + d] = fmaf(um[j], xv[d] - s_v[cur][j * D + d], t[j * D + d]);
            }
        }
        publish(t, dmax, bad);
        return exchange(NV);
    };

    // ---- pass 0 ----
    bool ok;
    if (FROM_U) {
        DF acc[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) acc[i] = DF{0.0f, 0.0f};
        bool bad = false;
        for (int64_t i = t0; i < n; i += nt) {
            float xv[D];
#pragma unroll
            for (int d = 0; d < D; ++d) {
                xv[d] = __ldg(x + (int64_t)d * n + i);
                bad |= !finite_f(xv[d]);
            }
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const float u0 = __ldcs(U0 + (int64_t)j * n + i);
                bad |= !(u0 >= 0.0f) || !finite_f(u0);
                const float um = (MK == M_TWO) ? u0 * u0 : ex2_approx(m * lg2_approx(u0));
                df_add(acc[C * D + j], um);
#pragma unroll
                for (int d = 0; d < D; ++d) df_add(acc[j * D + d], um * xv[d]);
            }
        }
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const DF t = warp_sum_df(acc[i]);
            if (lane == 0) s_w[warp][i] = t;
        }
        const bool any = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            s_m[warp] = 0.0f;
            s_b[warp] = any ? 1 : 0;
        }
        ok = exchange(NV);
    } else {
        ok = sums_pass(0, 0.0f, true);
    }
    int status = FCM_NOT_CONVERGED, iters = 0, cur = 0, prv = 2, nxt = 1;
    if (!ok) {
        status = FCM_ERR_TIMEOUT;
    } else if (s_mx[1] != 0.0f) {
        status = FCM_ERR_BAD_INPUT;
        ok = false;
    } else {
        centers(FROM_U ? -1 : 0, 1);
        if (!FROM_U && s_far && !rebase(0, 1)) {
            status = FCM_ERR_TIMEOUT;
            ok = false;
        }
    }
    auto advance = [&] {
        if (s_empty) flags |= FCM_FLAG_EMPTY_CLUSTER;
        const int t = prv;
        prv = cur;
        cur = nxt;
        nxt = t;
        __syncthreads();
        if (threadIdx.x == 0) s_empty = 0;  // set again only behind the next exchange
    };
    if (ok) advance();
    // The sampled pixel of a lane of the first warps: spread evenly over the
    // image, and after a full pass that did not stop the run, in warp 0, the
    // warps' pixels of largest change.
    float wx[D];
    int64_t wi = 0;
    const bool samples = warp < MSAMPLE_WARPS;
    if (samples) {
        wi = min(n - 1, (int64_t)(((double)blockIdx.x * 32 * MSAMPLE_WARPS + threadIdx.x) / ((double)nb * 32 * MSAMPLE_WARPS) * (double)n));
#pragma unroll
        for (int d = 0; d < D; ++d) wx[d] = __ldg(x + (int64_t)d * n + wi);
    }
    for (int k = 1; ok; ++k) {
        const bool last = k == max_iter, given = FROM_U && k == 1;
        if (!last) {
            float dmax = 0.0f;
            if (samples) {
                float u[C], up[C];
                pixel_memberships<C, MK>(wx, s_v[cur], m, inv_m1, u);
                if (given) {
#pragma unroll
                    for (int j = 0; j < C; ++j) up[j] = __ldcs(U0 + (int64_t)j * n + wi);
                } else {
                    pixel_memberships<C, MK>(wx, s_v[prv], m, inv_m1, up);
                }
#pragma unroll
                for (int j = 0; j < C; ++j) dmax = fmaxf(dmax, fabsf(u[j] - up[j]));
            }
            if (!sums_pass(cur, dmax, false)) {
                status = FCM_ERR_TIMEOUT;
                iters = k;
                break;
            }
            const bool go_on = s_mx[0] >= eps;
            centers(cur, nxt);
            if (go_on && !(s_far | s_empty)) {
                // as advance(), with no flag to note or clear
                const int t = prv;
                prv = cur;
                cur = nxt;
                nxt = t;
                continue;
            }
            if (s_far && !rebase(cur, nxt)) {
                status = FCM_ERR_TIMEOUT;
                iters = k;
                break;
            }
            if (go_on) {
                advance();
                continue;
            }
        }
        // ---- full pass: delta_k and J_k over every pixel, U^k ----
        DF J{0.0f, 0.0f};
        float dmax = -1.0f, best[D];
#pragma unroll
        for (int d = 0; d < D; ++d) best[d] = 0.0f;
        for (int64_t i = t0; i < n; i += nt) {
            float xv[D], u[C], up[C];
#pragma unroll
            for (int d = 0; d < D; ++d) xv[d] = __ldg(x + (int64_t)d * n + i);
            df_add(J, pixel_memberships<C, MK>(xv, s_v[cur], m, inv_m1, u));
            if (given) {
#pragma unroll
                for (int j = 0; j < C; ++j) up[j] = __ldcs(U0 + (int64_t)j * n + i);
            } else {
                pixel_memberships<C, MK>(xv, s_v[prv], m, inv_m1, up);
            }
            float dd = 0.0f;
#pragma unroll
            for (int j = 0; j < C; ++j) {
                dd = fmaxf(dd, fabsf(u[j] - up[j]));
                __stcs(U + (int64_t)j * n + i, u[j]);
            }
            if (dd > dmax) {
                dmax = dd;
#pragma unroll
                for (int d = 0; d < D; ++d) best[d] = xv[d];
            }
        }
        J = warp_sum_df(J);
        const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(dmax, 0.0f)));
        const unsigned who = __ballot_sync(0xffffffffu, dmax >= 0.0f && __float_as_uint(dmax) == mb);
        if (lane == (who ? __ffs(who) - 1 : 0)) {
#pragma unroll
            for (int d = 0; d < D; ++d) s_wit[warp][d] = best[d];
        }
        if (lane == 0) {
            s_w[warp][0] = J;
            s_m[warp] = __uint_as_float(mb);
            s_b[warp] = who ? 2 : 0;
        }
        if (!exchange(1)) {
            status = FCM_ERR_TIMEOUT;
            iters = k;
            break;
        }
        if (warp == 0 && lane < MNW && (s_b[lane] & 2)) {
#pragma unroll
            for (int d = 0; d < D; ++d) wx[d] = s_wit[lane][d];
        }
        const float delta = s_mx[0];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->delta = delta;
            st->J = df_to_double(s_df[0]);
        }
        if (delta < eps || last) {
            status = delta < eps ? FCM_OK : FCM_NOT_CONVERGED;
            iters = k;
            break;
        }
        advance();  // to the V^{k+1} of the sums pass
    }
    if (blockIdx.x == 0) {
        if (threadIdx.x < C * D) {
            st->V[threadIdx.x] = s_v[cur][threadIdx.x];
            st->V64[threadIdx.x] = df_to_double(s_v64[cur][threadIdx.x]);
        }
        if (threadIdx.x == 0) {
            st->status = status;
            st->iters = iters;
            st->flags = flags;
        }
    }
}

template <int C, int MK>
void fill(MultiTable& t) {
    t.run[D][C][MK == M_TWO ? 0 : 1][0] = k_fcm_run_multi<C, MK, true>;
    t.run[D][C][MK == M_TWO ? 0 : 1][1] = k_fcm_run_multi<C, MK, false>;
}

template <int C>
void fill_c(MultiTable& t) {
    fill<C, M_TWO>(t);
    fill<C, M_GENERIC>(t);
}

}  // namespace

#define FCM_CAT2(a, b) a##b
#define FCM_CAT(a, b) FCM_CAT2(a, b)
void FCM_CAT(register_multi_d, FCM_MULTI_D)(MultiTable& t) {
    fill_c<1>(t);
    fill_c<2>(t);
    fill_c<3>(t);
    fill_c<4>(t);
    fill_c<5>(t);
    fill_c<6>(t);
    fill_c<7>(t);
    fill_c<8>(t);
}

}  // namespace fcm
