// Device-side building blocks of the FCM pixel pass (sm_103a).
//
// Membership (Eq. 4 of arXiv:1601.00072) is evaluated in its weight form:
//   u_j = w_j / sum_k w_k,   w_j = (q_j)^(1/(m-1)),   q_j = d2min / d2_j,
// which equals 1 / sum_k (d_j / d_k)^(2/(m-1)) after dividing numerator and
// denominator by sum_k w_k; the common factor keeps every weight in (0, 1], so
// no weight or sum can overflow. When some squared distance d2 = (x - v)^2
// falls below the smallest normal float (2^-126) although the distances
// themselves are normal, q_j is formed as (|d|min / |d_j|)^2 instead, from the
// distances, which do not underflow.
// A pixel at distance 0 from one or more centers gives those clusters equal
// shares and the others 0 (Bezdek's rule; the paper leaves d = 0 open).
// "Distance 0" means |x - v| below 2^-126, i.e. zero once the FP32
// approximate instructions flush subnormal operands to zero.
//
// Specialisations of the fuzzifier avoid general powers on the hot path:
//   m = 2    w = q                u^m = u*u
//   m = 3    w = sqrt(q)          u^m = u*u*u
//   m = 1.5  w = q*q              u^m = u*sqrt(u)
//   other m  w = 2^((log2 q)/(m-1))   u^m = 2^(m log2 u)
// using the PTX approximate instructions (rcp, rsqrt, sqrt, lg2, ex2), whose
// documented error is at most a few ulp in FP32.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fcm.h"

namespace fcm {

enum MKind : int { M_TWO = 0, M_THREE = 1, M_ONE_HALF = 2, M_GENERIC = 3, M_KINDS = 4 };

__host__ __device__ inline int mkind_of(float m) {
    return m == 2.0f ? M_TWO : m == 3.0f ? M_THREE : m == 1.5f ? M_ONE_HALF : M_GENERIC;
}

__device__ __forceinline__ float rcp_approx(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float rsqrt_approx(float a) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float sqrt_approx(float a) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float lg2_approx(float a) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float ex2_approx(float a) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// u^m for the specialised fuzzifiers (u in [0, 1]).
template <int MK>
__device__ __forceinline__ float pow_m(float u, float m) {
    if (MK == M_TWO) return u * u;
    if (MK == M_THREE) return u * u * u;
    if (MK == M_ONE_HALF) return u * sqrt_approx(u);
    return ex2_approx(m * lg2_approx(u));  // lg2(0) = -inf -> ex2(-inf) = 0
}

// Smallest normal FP32 value: distances (and sums of products of distances)
// below it count as zero, as the .ftz instructions would read them.
__device__ __forceinline__ float flt_min() { return __int_as_float(0x00800000); }

// Memberships of one pixel x against C centers v (Eq. 4). Writes u[j] and
// um[j] = u[j]^m; returns this pixel's term of J_m, sum_j u_j^m d_j^2 (Eq. 1),
// through its closed form under Eq. 4: with u_j = w_j / S and
// w_j = (d2min / d2_j)^(1/(m-1)), u_j^m d2_j = d2min w_j / S^m, so the term is
// d2min * S^(1-m) (and 0 when the pixel sits on a center).
template <int C, int MK>
__device__ __forceinline__ float membership(float x, const float (&v)[C], float m, float inv_m1,
                                            float (&u)[C], float (&um)[C]) {
    float d2[C], ad[C];
    float dmin = __int_as_float(0x7f800000), amin = dmin;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const float d = x - v[j];
        ad[j] = fabsf(d);
        d2[j] = __fmul_rn(d, d);
        dmin = fminf(dmin, d2[j]);
        amin = fminf(amin, ad[j]);
    }
    float Ji = 0.0f;
    if (amin >= flt_min()) {
        float w[C];
        if (dmin >= flt_min()) {
            // every squared distance is a normal float: ratios of the squares
            if (MK == M_GENERIC) {
                const float l0 = lg2_approx(dmin);
#pragma unroll
                for (int j = 0; j < C; ++j) w[j] = ex2_approx(inv_m1 * (l0 - lg2_approx(d2[j])));
            } else if (MK == M_THREE) {
                const float s0 = sqrt_approx(dmin);
#pragma unroll
                for (int j = 0; j < C; ++j) w[j] = s0 * rsqrt_approx(d2[j]);
            } else {
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const float q = dmin * rcp_approx(d2[j]);
                    w[j] = (MK == M_ONE_HALF) ? q * q : q;
                }
            }
        } else {
            // tiny distances: ratios of the distances themselves
            if (MK == M_GENERIC) {
                const float l0 = lg2_approx(amin), e = 2.0f * inv_m1;
#pragma unroll
                for (int j = 0; j < C; ++j) w[j] = ex2_approx(e * (l0 - lg2_approx(ad[j])));
            } else {
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const float r = amin * rcp_approx(ad[j]);
                    const float q = r * r;
                    w[j] = (MK == M_THREE) ? r : (MK == M_ONE_HALF) ? q * q : q;
                }
            }
        }
        float S = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) S += w[j];
        const float r = rcp_approx(S);
#pragma unroll
        for (int j = 0; j < C; ++j) u[j] = w[j] * r;
        // dmin may be subnormal or 0 for tiny distances: the J term is then tiny or 0
        if (MK == M_TWO) Ji = dmin * r;
        else if (MK == M_THREE) Ji = dmin * r * r;
        else if (MK == M_ONE_HALF) Ji = dmin * sqrt_approx(r);
        else Ji = dmin * ex2_approx((1.0f - m) * lg2_approx(S));
    } else {
        int nz = 0;
#pragma unroll
        for (int j = 0; j < C; ++j) nz += (ad[j] < flt_min());
        const float share = __fdiv_rn(1.0f, (float)nz);
#pragma unroll
        for (int j = 0; j < C; ++j) u[j] = (ad[j] < flt_min()) ? share : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < C; ++j) um[j] = pow_m<MK>(u[j], m);
    return Ji;
}

// ---------------------------------------------------------------------------
// Two pixels at once with the packed FP32x2 instructions of sm_100+ (PTX
// add/sub/mul/fma.rn.f32x2). A pair lives in one 64-bit register pair:
// the low half is the first pixel.
// ---------------------------------------------------------------------------
typedef uint64_t f2;

__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 r, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ float lo2(f2 r) { float a, b; unpack2(r, a, b); return a; }
__device__ __forceinline__ float hi2(f2 r) { float a, b; unpack2(r, a, b); return b; }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 abs2(f2 a) { return a & 0x7fffffff7fffffffull; }

// Memberships of two pixels (packed x2) against C centers (each packed as
// (v_j, v_j)), Eq. 4. Writes u2[j], um2[j] = u^m and returns the pair of J
// terms sum_j u_j^m d_j^2.
//
// m = 2 and m = 3 use the product form: with b_j = d_j^2 (m = 2) or |d_j|
// (m = 3) the weights 1/b_j share the denominator prod_k b_k, so
//   u_j = P_j / sum_k P_k,   P_j = prod_{k != j} b_k,
// one reciprocal per pixel; a pixel equal to exactly one center gets u = 1
// there and 0 elsewhere without a special case. The J term is u_j b_j for any
// j when m = 2 (both equal 1 / sum_k 1/d_k^2), and (u_j b_j)^2 when m = 3.
// A pixel whose sum_k P_k is 0 (two or more centers hit exactly), below the
// smallest normal float (products of tiny distances), or not finite (products
// out of FP32 range) takes the scalar weight form above, as do the other
// fuzzifiers.
template <int C, int MK>
__device__ __forceinline__ f2 membership_pair(f2 x2, const f2 (&v2)[C], float m, float inv_m1,
                                              const float (&v)[C], f2 (&u2)[C], f2 (&um2)[C]) {
    if (MK == M_TWO || MK == M_THREE) {
        f2 b[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const f2 d = sub2(x2, v2[j]);
            b[j] = (MK == M_TWO) ? mul2(d, d) : abs2(d);
        }
        f2 P[C];
        if (C == 1) {
            P[0] = pack2(1.0f, 1.0f);
        } else {
            f2 pre[C], suf[C];
#pragma unroll
            for (int j = 1; j < C; ++j) pre[j] = (j == 1) ? b[0] : mul2(pre[j - 1], b[j - 1]);
#pragma unroll
            for (int j = C - 2; j >= 0; --j) suf[j] = (j == C - 2) ? b[C - 1] : mul2(suf[j + 1], b[j + 1]);
#pragma unroll
            for (int j = 0; j < C; ++j) P[j] = (j == 0) ? suf[0] : (j == C - 1) ? pre[C - 1] : mul2(pre[j], suf[j]);
        }
        f2 S = P[0];
#pragma unroll
        for (int j = 1; j < C; ++j) S = add2(S, P[j]);
        float s0, s1;
        unpack2(S, s0, s1);
        // a sum below the smallest normal float would be flushed to zero by
        // the reciprocal: those pixels take the scalar form
        const float inf = __int_as_float(0x7f800000);
        if (s0 >= flt_min() && s0 < inf && s1 >= flt_min() && s1 < inf) {
            const f2 r = pack2(rcp_approx(s0), rcp_approx(s1));
#pragma unroll
            for (int j = 0; j < C; ++j) {
                u2[j] = mul2(P[j], r);
                const f2 uu = mul2(u2[j], u2[j]);
                um2[j] = (MK == M_TWO) ? uu : mul2(uu, u2[j]);
            }
            const f2 t = mul2(u2[0], b[0]);
            return (MK == M_TWO) ? t : mul2(t, t);
        }
    }
    // scalar weight form, one pixel at a time
    float xa, xb;
    unpack2(x2, xa, xb);
    float ua[C], uma[C], ub[C], umb[C];
    const float ja = membership<C, MK>(xa, v, m, inv_m1, ua, uma);
    const float jb = membership<C, MK>(xb, v, m, inv_m1, ub, umb);
#pragma unroll
    for (int j = 0; j < C; ++j) {
        u2[j] = pack2(ua[j], ub[j]);
        um2[j] = pack2(uma[j], umb[j]);
    }
    return pack2(ja, jb);
}

// ---------------------------------------------------------------------------
// Two pixels at once for every fuzzifier, u^m alone (the passes that only add
// up Eq. 3's sums) or u with the J terms. The scalar weight form above is called,
// not inlined, for the rare pair that the packed forms cannot take: the packed
// code keeps its registers and stays small.
// ---------------------------------------------------------------------------

template <int C>
struct PixelPair {
    float a[C], b[C];  // u^m or u of the two pixels
    float Ja, Jb;
};
#ifdef FCM_ONE_SCALAR_PAIR
// One function for every cluster count and fuzzifier, for the kernels that hold
// all of them (nested calls of 32 variants compile for minutes): the C centers are
// padded with infinitely distant ones, whose weights are exactly 0.
static __device__ __noinline__ PixelPair<FCM_MAX_CLUSTERS> scalar_pair_any(float xa, float xb, const float* vs, int C,
                                                                          int mk, bool powers, float m, float inv_m1) {
    constexpr int N = FCM_MAX_CLUSTERS;
    float v[N], u[N], um[N];
    PixelPair<N> w;
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = j < C ? vs[j] : __int_as_float(0x7f800000);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const float x = h ? xb : xa;
        float J;
        switch (mk) {
            case M_TWO: J = membership<N, M_TWO>(x, v, m, inv_m1, u, um); break;
            case M_THREE: J = membership<N, M_THREE>(x, v, m, inv_m1, u, um); break;
            case M_ONE_HALF: J = membership<N, M_ONE_HALF>(x, v, m, inv_m1, u, um); break;
            default: J = membership<N, M_GENERIC>(x, v, m, inv_m1, u, um); break;
        }
#pragma unroll
        for (int j = 0; j < N; ++j) (h ? w.b : w.a)[j] = powers ? um[j] : u[j];
        (h ? w.Jb : w.Ja) = J;
    }
    return w;
}
template <int C, int MK, bool POWERS>
__device__ __forceinline__ PixelPair<C> scalar_pair(float xa, float xb, const float* vs, float m, float inv_m1) {
    const PixelPair<FCM_MAX_CLUSTERS> q = scalar_pair_any(xa, xb, vs, C, MK, POWERS, m, inv_m1);
    PixelPair<C> w;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        w.a[j] = q.a[j];
        w.b[j] = q.b[j];
    }
    w.Ja = q.Ja;
    w.Jb = q.Jb;
    return w;
}
#else
template <int C, int MK, bool POWERS>
__device__ __noinline__ PixelPair<C> scalar_pair(float xa, float xb, const float* vs, float m, float inv_m1) {
    float v[C], t[C];
    PixelPair<C> w;
#pragma unroll
    for (int j = 0; j < C; ++j) v[j] = vs[j];
    if (POWERS) {
        w.Ja = membership<C, MK>(xa, v, m, inv_m1, t, w.a);
        w.Jb = membership<C, MK>(xb, v, m, inv_m1, t, w.b);
    } else {
        w.Ja = membership<C, MK>(xa, v, m, inv_m1, w.a, t);
        w.Jb = membership<C, MK>(xb, v, m, inv_m1, w.b, t);
    }
    return w;
}
#endif

// Power-of-two factor that brings the centers' spread to [1, 2), for the
// products at m = 1.5 (1 when the spread is 0 or extreme). Scaling by it is
// exact, so it changes the products' range and nothing else.
template <int C>
__device__ __forceinline__ float spread_scale(const float* v) {
    float lo = v[0], hi = lo;
#pragma unroll
    for (int j = 1; j < C; ++j) {
        lo = fminf(lo, v[j]);
        hi = fmaxf(hi, v[j]);
    }
    const int e = (__float_as_int(hi - lo) >> 23) - 127;
    return (e < -60 || e > 60) ? 1.0f : __int_as_float((127 - e) << 23);
}

// Products P_j = prod_{k != j} b_k.
template <int C>
__device__ __forceinline__ void co_products(const f2 (&b)[C], f2 (&P)[C]) {
    if (C == 1) {
        P[0] = pack2(1.0f, 1.0f);
        return;
    }
    f2 pre[C], suf[C];
#pragma unroll
    for (int j = 1; j < C; ++j) pre[j] = (j == 1) ? b[0] : mul2(pre[j - 1], b[j - 1]);
#pragma unroll
    for (int j = C - 2; j >= 0; --j) suf[j] = (j == C - 2) ? b[C - 1] : mul2(suf[j + 1], b[j + 1]);
#pragma unroll
    for (int j = 0; j < C; ++j) P[j] = (j == 0) ? suf[0] : (j == C - 1) ? pre[C - 1] : mul2(pre[j], suf[j]);
}

// What the packed forms read of the centers: the centers themselves in memory
// (vs, for the scalar form), and as the differences use them (v2; at m = 1.5
// times the power of two `scale`, see spread_scale).
template <int C, int MK>
struct PackedCenters {
    f2 v2[C], scale;
    const float* vs;
    static constexpr bool SCALED = MK == M_ONE_HALF;
    __device__ __forceinline__ void set(const float* v) {
        vs = v;
        float s = 1.0f;
        if (SCALED) {
            s = spread_scale<C>(v);
            scale = pack2(s, s);
        }
#pragma unroll
        for (int j = 0; j < C; ++j) v2[j] = pack2(v[j] * s, v[j] * s);
    }
    __device__ __forceinline__ f2 of(f2 x) const { return SCALED ? mul2(x, scale) : x; }
};

// N pairs at once (N = 1 or 2: two pairs share one test for the scalar form, and
// their chains overlap). POWERS: w2[j] = u_j^m of each pair, and d2[j] = x - v_j
// (scaled). Otherwise w2[j] = u_j, and J2 each pair's J terms.
//   m = 2, 3  the product form of membership_pair.
//   m = 1.5   for u^m, with p_j = prod_{k != j} d_k^2: sqrt(u_j) = p_j / sqrt(
//             sum_k p_k^2), one reciprocal square root per pixel where the weight
//             form takes C reciprocals and C square roots; u^1.5 is its cube.
//             The products' roundings average out in the sums, but not in a
//             pixel's u (at C = 8 up to 7e-7, against 2e-7): u itself takes the
//             weight form, w_j = (d2min / d2_j)^2.
//   WEIGHTS takes the weight form of u at m = 2 and 3 too (w_j = d2min / d2_j, its
//   square root): the grey-level kernels, whose 256 bins are a pixel each.
//   other m   w_j = 2^t_j, t_j = (log2 d2min - log2 d2_j) / (m - 1), S = sum w:
//             u_j^m = 2^(m (t_j - log2 S)), without the C logarithms of u_j.
template <int C, int MK, bool POWERS, int N, bool WEIGHTS = MK == M_ONE_HALF>
__device__ __forceinline__ void packed_pairs(const f2 (&x2)[N], const PackedCenters<C, MK>& c, float m, float inv_m1,
                                             f2 (&w2)[N][C], f2 (&d2)[N][C], f2 (&J2)[N]) {
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const f2 xs = c.of(x2[p]);
#pragma unroll
        for (int j = 0; j < C; ++j) d2[p][j] = sub2(xs, c.v2[j]);
    }
    if (MK != M_GENERIC && WEIGHTS && !POWERS) {
        float mn[2 * N], low = __int_as_float(0x7f800000);
        f2 b[N][C];
#pragma unroll
        for (int p = 0; p < N; ++p) {
            mn[2 * p] = mn[2 * p + 1] = __int_as_float(0x7f800000);
#pragma unroll
            for (int j = 0; j < C; ++j) {
                b[p][j] = (MK == M_THREE) ? abs2(d2[p][j]) : mul2(d2[p][j], d2[p][j]);
                mn[2 * p] = fminf(mn[2 * p], lo2(b[p][j]));
                mn[2 * p + 1] = fminf(mn[2 * p + 1], hi2(b[p][j]));
            }
            low = fminf(low, fminf(mn[2 * p], mn[2 * p + 1]));
        }
        if (low >= flt_min()) {
#pragma unroll
            for (int p = 0; p < N; ++p) {
                const f2 mn2 = pack2(mn[2 * p], mn[2 * p + 1]);
                f2 S = pack2(0.0f, 0.0f);
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const f2 q = mul2(mn2, pack2(rcp_approx(lo2(b[p][j])), rcp_approx(hi2(b[p][j]))));
                    w2[p][j] = (MK == M_ONE_HALF) ? mul2(q, q) : q;
                    S = add2(S, w2[p][j]);
                }
                const float ra = rcp_approx(lo2(S)), rb = rcp_approx(hi2(S));
#pragma unroll
                for (int j = 0; j < C; ++j) w2[p][j] = mul2(w2[p][j], pack2(ra, rb));
                if (MK == M_ONE_HALF) {
                    // d2min S^(-1/2), back from scaled differences
                    const float q = rcp_approx(lo2(c.scale));  // of a power of two: exact
                    J2[p] = mul2(mul2(mn2, pack2(sqrt_approx(ra), sqrt_approx(rb))), pack2(q * q, q * q));
                } else {
                    // d2min / S (m = 2), d2min / S^2 (m = 3)
                    J2[p] = mul2(mn2, pack2(ra, rb));
                    if (MK == M_THREE) J2[p] = mul2(J2[p], J2[p]);
                }
            }
            return;
        }
    } else if (MK == M_TWO || MK == M_THREE || MK == M_ONE_HALF) {
        f2 b0[N], P[N][C];
        unsigned worst = 0u;  // of the sums' distances from the smallest normal float
        float s0[N], s1[N];
#pragma unroll
        for (int p = 0; p < N; ++p) {
            f2 b[C];
#pragma unroll
            for (int j = 0; j < C; ++j) b[j] = (MK == M_THREE) ? abs2(d2[p][j]) : mul2(d2[p][j], d2[p][j]);
            b0[p] = b[0];
            co_products<C>(b, P[p]);
            f2 S = (MK == M_ONE_HALF) ? mul2(P[p][0], P[p][0]) : P[p][0];
#pragma unroll
            for (int j = 1; j < C; ++j) S = (MK == M_ONE_HALF) ? fma2(P[p][j], P[p][j], S) : add2(S, P[p][j]);
            unpack2(S, s0[p], s1[p]);
            // a normal positive float has bits in [0x00800000, 0x7f800000): not
            // zero, subnormal, infinite or NaN
            worst = max(worst, max(__float_as_uint(s0[p]) - 0x00800000u, __float_as_uint(s1[p]) - 0x00800000u));
        }
        if (worst < 0x7f000000u) {
#pragma unroll
            for (int p = 0; p < N; ++p) {
                const f2 r = (MK == M_ONE_HALF) ? pack2(rsqrt_approx(s0[p]), rsqrt_approx(s1[p]))
                                                : pack2(rcp_approx(s0[p]), rcp_approx(s1[p]));
                if (!POWERS) {
                    // u_j d_j^2 (m = 2), (u_j |d_j|)^2 (m = 3), any j
                    J2[p] = mul2(mul2(P[p][0], r), b0[p]);
                    if (MK == M_THREE) J2[p] = mul2(J2[p], J2[p]);
                }
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const f2 u = mul2(P[p][j], r);
                    if (POWERS) {
                        w2[p][j] = mul2(u, u);
                        if (MK != M_TWO) w2[p][j] = mul2(w2[p][j], u);
                    } else {
                        w2[p][j] = u;
                    }
                }
            }
            return;
        }
    } else {
        float t[2 * N][C], l[2 * N], mn[2 * N], low = __int_as_float(0x7f800000);
#pragma unroll
        for (int p = 0; p < N; ++p) {
            l[2 * p] = l[2 * p + 1] = mn[2 * p] = mn[2 * p + 1] = __int_as_float(0x7f800000);
#pragma unroll
            for (int j = 0; j < C; ++j) {
                float q[2];
                unpack2(mul2(d2[p][j], d2[p][j]), q[0], q[1]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!POWERS) mn[2 * p + h] = fminf(mn[2 * p + h], q[h]);
                    t[2 * p + h][j] = lg2_approx(q[h]);  // a square below 2^-126 reads as 0: -inf
                    l[2 * p + h] = fminf(l[2 * p + h], t[2 * p + h][j]);
                }
            }
            low = fminf(low, fminf(l[2 * p], l[2 * p + 1]));
        }
        if (low >= -126.0f) {
#pragma unroll
            for (int p = 0; p < N; ++p) {
                const float la = l[2 * p], lb = l[2 * p + 1];
                f2 S = pack2(0.0f, 0.0f);
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    t[2 * p][j] = inv_m1 * (la - t[2 * p][j]);
                    t[2 * p + 1][j] = inv_m1 * (lb - t[2 * p + 1][j]);
                    w2[p][j] = pack2(ex2_approx(t[2 * p][j]), ex2_approx(t[2 * p + 1][j]));
                    S = add2(S, w2[p][j]);
                }
                const float ga = lg2_approx(lo2(S)), gb = lg2_approx(hi2(S));
                if (POWERS) {
#pragma unroll
                    for (int j = 0; j < C; ++j)
                        w2[p][j] = pack2(ex2_approx(m * (t[2 * p][j] - ga)), ex2_approx(m * (t[2 * p + 1][j] - gb)));
                } else {
                    const f2 r = pack2(rcp_approx(lo2(S)), rcp_approx(hi2(S)));
#pragma unroll
                    for (int j = 0; j < C; ++j) w2[p][j] = mul2(w2[p][j], r);
                    // d2min S^(1-m)
                    J2[p] = mul2(pack2(mn[2 * p], mn[2 * p + 1]),
                                 pack2(ex2_approx((1.0f - m) * ga), ex2_approx((1.0f - m) * gb)));
                }
            }
            return;
        }
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const PixelPair<C> w = scalar_pair<C, MK, POWERS>(lo2(x2[p]), hi2(x2[p]), c.vs, m, inv_m1);
#pragma unroll
        for (int j = 0; j < C; ++j) w2[p][j] = pack2(w.a[j], w.b[j]);
        if (!POWERS) J2[p] = pack2(w.Ja, w.Jb);
    }
}

// Compensated FP32 ("double-float") sum, hi + lo, with Knuth's TwoSum: long
// sums of the center numerators/denominators and of J carry about 44 bits
// while using only FP32 instructions.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ void df_add(DF& a, float b) {
    const float s = __fadd_rn(a.hi, b);
    const float bb = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    a.hi = s;
    a.lo = __fadd_rn(a.lo, e);
}
__device__ __forceinline__ DF df_merge(DF a, DF b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float bb = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
    const float lo = __fadd_rn(__fadd_rn(a.lo, b.lo), e);
    const float hi = __fadd_rn(s, lo);  // Fast2Sum renormalisation (|s| >= |lo|)
    return DF{hi, __fsub_rn(lo, __fsub_rn(hi, s))};
}

// The same without the renormalisation (two dependent steps shorter): for a
// few merges in a row, followed by df_norm.
__device__ __forceinline__ DF df_merge_raw(DF a, DF b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float bb = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
    return DF{s, __fadd_rn(__fadd_rn(a.lo, b.lo), e)};
}
__device__ __forceinline__ DF df_norm(DF a) {
    const float hi = __fadd_rn(a.hi, a.lo);
    return DF{hi, __fsub_rn(a.lo, __fsub_rn(hi, a.hi))};
}

// Warp-wide double-float sum (xor tree, fixed order).
__device__ __forceinline__ DF warp_sum_df(DF d) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        DF e{__shfl_xor_sync(0xffffffffu, d.hi, o), __shfl_xor_sync(0xffffffffu, d.lo, o)};
        d = (lane & o) ? df_merge(e, d) : df_merge(d, e);
    }
    return d;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float comp(const float4& a, int p) {
    return p == 0 ? a.x : p == 1 ? a.y : p == 2 ? a.z : a.w;
}
__device__ __forceinline__ void set_comp(float4& a, int p, float v) {
    if (p == 0) a.x = v; else if (p == 1) a.y = v; else if (p == 2) a.z = v; else a.w = v;
}

// Read-only streaming load of the intensities (non-coherent path).
__device__ __forceinline__ float4 ld_x4(const float* p) {
    return __ldg(reinterpret_cast<const float4*>(p));
}
// Memberships are read once and overwritten by the same thread: evict-first.
__device__ __forceinline__ float4 ld_u4(const float* p) {
    return __ldcs(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ void st_u4(float* p, float4 v) {
    __stcs(reinterpret_cast<float4*>(p), v);
}

__device__ __forceinline__ bool finite_f(float a) {
    return (__float_as_uint(a) & 0x7f800000u) != 0x7f800000u;
}

}  // namespace fcm
