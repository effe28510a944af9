// Algorithm 1 (arXiv:1601.00072, Sec. 2.1) on the 256-bin grey-level
// histogram: the loop of the histogram-domain run (brFCM, cited in Sec. 3),
// shared by the single-image kernel and the batch kernels (one CTA per run).
//
// Under Eq. 4 a pixel's memberships depend only on its grey level, so the
// center sums of Eq. 3 and J of Eq. 1 are sums over bins weighted by their
// pixel counts, and the stopping quantity is a maximum over the bins present.
#pragma once

#include "fcm_device.cuh"
#include "fcm_df.cuh"

namespace fcm {

constexpr int HNT = 256;  // threads of the pixel-pass CTAs

__device__ __forceinline__ bool grey_level(float v) {
    return v >= 0.0f && v <= 255.0f && v == rintf(v);  // false for NaN
}

// The grey level of v when v is an integer in [0, 255], else -1 (the same
// test as grey_level, with the index). Adding 1.5 * 2^23 rounds any
// |v| < 2^22 to an integer held in the low mantissa bits; v is that integer
// exactly when subtracting the constant gives v back. NaN fails the
// comparison; infinities and values outside [0, 255] give an index outside
// [0, 255] (as unsigned).
__device__ __forceinline__ int grey_index(float v) {
    constexpr float kShift = 12582912.0f;  // 1.5 * 2^23
    const float t = __fadd_rn(v, kShift);
    const int g = __float_as_int(t) - __float_as_int(kShift);
    return ((unsigned)g <= 255u && __fsub_rn(t, kShift) == v) ? g : -1;
}

// The loop runs in one CTA of BIN_NT threads, thread t holding the grey levels
// 2t and 2t + 1 as a packed pair. It is bound by latency: every iteration is one
// chain from the centers through the memberships and the sums back to the
// centers, so what counts is the length of that chain. The numerators are
// centered (sum u^m (b - v_j), so v_j moves by num_j / den_j). A sum over the bins
// is taken in two steps: in each warp a five-level FP32 tree that halves the
// number of values at every level (N - 1 + 5 - log2 N shuffles for N values), then
// the four warp totals in double-float, two levels, by groups of four lanes, group
// j holding cluster j; each group forms its center (double-float quotient) and the
// lanes of every warp fetch all C of them. Every warp does so alike, so all
// threads hold the same centers, and one barrier per iteration suffices: the warp
// totals are double-buffered by the parity `par`, which every reduction flips. J
// is added up once, after the last iteration. (With 256 threads, J in the loop and a
// full tree for every value an iteration took 1.2 us at C = 4.)
constexpr int BIN_NT = 128;
constexpr int BIN_NW = BIN_NT / 32;
static_assert(BIN_NW == 4 && FCM_MAX_CLUSTERS == 8, "groups of four lanes hold the warp totals of one cluster");

struct BinScratch {
    float w[2][BIN_NW][2 * FCM_MAX_CLUSTERS];  // [parity][warp] sums
    float mx[2][BIN_NW];
    float vs[BIN_NW][FCM_MAX_CLUSTERS];        // each warp's copy of the centers, for the scalar form
};

constexpr int bin_pow2(int n) { return n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 16; }

// Sums of P values over the warp by log-step halving; the lanes with
// (lane & (32 / P - 1)) == 0 end with the total of value `slot` in a[0].
template <int P>
__device__ __forceinline__ int bin_warp_totals(float (&a)[P]) {
    const int lane = threadIdx.x & 31;
    int o = 16, slot = 0;
#pragma unroll
    for (int w = P; w > 1; w >>= 1, o >>= 1) {
        const bool up = lane & o;
        slot += up ? w / 2 : 0;
#pragma unroll
        for (int i = 0; i < w / 2; ++i) {
            const float send = up ? a[i] : a[i + w / 2], keep = up ? a[i + w / 2] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    return slot;
}

// This thread's copy of the centers v, and the warp's for the scalar form.
template <int C, int MK>
__device__ __forceinline__ void bin_centers(BinScratch& sc, const float (&v)[C], PackedCenters<C, MK>& cen) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < C; ++j)
        if (lane == j) sc.vs[warp][j] = v[j];
    __syncwarp();
    cen.set(sc.vs[warp]);
}

// The CTA's sums of num and den (per thread, both grey levels) and its maximum;
// then the centers. base: what the numerators are relative to (bin_base). mine:
// the double-float center of cluster lane >> 2, kept where that cluster is empty.
// On return v and mine hold the new centers, mx the maximum, and the result tells
// whether some cluster was empty. All BIN_NT threads must call it.
template <int C>
__device__ __forceinline__ bool bin_reduce(BinScratch& sc, int& par, const f2 (&num2)[C], const f2 (&den2)[C],
                                           float& mx, const float (&base)[C], float (&v)[C], DF& mine) {
    constexpr int P = bin_pow2(2 * C);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float t[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const f2 q = i < C ? num2[i < C ? i : 0] : den2[(i >= C && i < 2 * C) ? i - C : 0];
        t[i] = i < 2 * C ? lo2(q) + hi2(q) : 0.0f;
    }
    const int slot = bin_warp_totals<P>(t);
    const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));  // non-negative
    if ((lane & (32 / P - 1)) == 0 && slot < 2 * C) sc.w[par][warp][slot] = t[0];
    if (lane == 0) sc.mx[par][warp] = __uint_as_float(mb);
    __syncthreads();
    const int g = lane >> 2, w = lane & 3;
    DF num{0.0f, 0.0f}, den{1.0f, 0.0f};
    float bg = 0.0f;
#pragma unroll
    for (int j = 0; j < C; ++j)
        if (g == j) bg = base[j];
    if (g < C) {
        num.hi = sc.w[par][w][g];
        den = DF{sc.w[par][w][C + g], 0.0f};
    }
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sc.mx[par][w])));
    par ^= 1;
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
        // TwoSum is symmetric: the four lanes of a group get the same totals
        num = df_merge(num, DF{__shfl_xor_sync(0xffffffffu, num.hi, o), __shfl_xor_sync(0xffffffffu, num.lo, o)});
        den = df_merge(den, DF{__shfl_xor_sync(0xffffffffu, den.hi, o), __shfl_xor_sync(0xffffffffu, den.lo, o)});
    }
    const bool empty = !(den.hi > 0.0f);
    if (!empty) mine = df_merge((den.hi > 1e-30f && den.hi < 1e30f) ? df_div_fast(num, den) : df_div(num, den), DF{bg, 0.0f});
#pragma unroll
    for (int j = 0; j < C; ++j) v[j] = __shfl_sync(0xffffffffu, mine.hi, 4 * j);
    return __any_sync(0xffffffffu, empty);
}

// The center of cluster lane >> 2 as a double-float.
template <int C>
__device__ __forceinline__ DF bin_mine(const float (&v)[C]) {
    float t = 0.0f;
#pragma unroll
    for (int j = 0; j < C; ++j)
        if ((int)((threadIdx.x & 31) >> 2) == j) t = v[j];
    return DF{t, 0.0f};
}

// The CTA's maximum of mx (non-negative), the same in every thread.
__device__ __forceinline__ float bin_max(BinScratch& sc, int& par, float mx) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
    if (lane == 0) sc.mx[par][warp] = __uint_as_float(mb);
    __syncthreads();
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sc.mx[par][lane & 3])));
    par ^= 1;
    return mx;
}

// What cluster j's numerator is centered on: its center, or the end of the grey
// scale that is nearest to it. Differences from a center far outside the scale (an
// initial one) would have lost the bits of the grey levels.
__device__ __forceinline__ float bin_base(float v) { return fminf(fmaxf(v, 0.0f), 255.0f); }

// u of this thread's grey levels b2 = (2t, 2t + 1), the J terms, and u^m with
// the differences from the bases.
template <int C, int MK>
__device__ __forceinline__ void bin_memberships(f2 b2, const PackedCenters<C, MK>& cen, const float (&base)[C], float m,
                                                float inv_m1, f2 (&u2)[C], f2 (&um2)[C], f2 (&d2)[C], f2& J2) {
    f2 w[1][C], d[1][C], j[1];
    const f2 x[1] = {b2};
    packed_pairs<C, MK, false, 1, true>(x, cen, m, inv_m1, w, d, j);
    J2 = j[0];
#pragma unroll
    for (int q = 0; q < C; ++q) {
        u2[q] = w[0][q];
        d2[q] = sub2(b2, pack2(base[q], base[q]));
        um2[q] = (MK == M_TWO)     ? mul2(u2[q], u2[q])
                 : (MK == M_THREE) ? mul2(mul2(u2[q], u2[q]), u2[q])
                                   : pack2(pow_m<MK>(lo2(u2[q]), m), pow_m<MK>(hi2(u2[q]), m));
    }
}

// V^1 on the bins with U^0 = f(b, V^0): U^0 of the grey levels into up2, V^1 into
// v. Returns whether some cluster was empty.
template <int C, int MK>
__device__ __forceinline__ bool bin_first_centers(BinScratch& sc, int& par, f2 cnt2, const float (&v0)[C], float m,
                                                  float inv_m1, f2 (&up2)[C], float (&v)[C], DF& mine) {
    const f2 b2 = pack2((float)(2 * threadIdx.x), (float)(2 * threadIdx.x + 1));
    PackedCenters<C, MK> cen;
    bin_centers<C, MK>(sc, v0, cen);
    float base[C];
#pragma unroll
    for (int j = 0; j < C; ++j) base[j] = bin_base(v0[j]);
    f2 um2[C], d2[C], J2, num2[C];
    bin_memberships<C, MK>(b2, cen, base, m, inv_m1, up2, um2, d2, J2);
#pragma unroll
    for (int j = 0; j < C; ++j) {
        um2[j] = mul2(cnt2, um2[j]);
        num2[j] = mul2(um2[j], d2[j]);
    }
    float mx = 0.0f;
    mine = bin_mine<C>(v0);
    return bin_reduce<C>(sc, par, num2, um2, mx, base, v, mine);
}

// Iterations k = 1, 2, ... of Algorithm 1 on the bins of one run, in one CTA.
//   cnt2  the pixel counts of this thread's grey levels (as floats).
//   from_u  the run started from U^0: its first stopping quantity is d1,
//         taken over the pixels (a run from centers has U^0 per grey level).
//   v, mine  in: V^1 (the same in every thread) and the double-float center of
//         cluster lane >> 2; out: those of V^k of the returned U^k.
//   up2   in: U^0 of the grey levels (runs from centers); out: their U^k.
//   J     out: J_k (Eq. 1).
// An empty cluster keeps its center and sets the flag.
template <int C, int MK>
__device__ __forceinline__ void solve_bins(BinScratch& sc, int& par, f2 cnt2, bool from_u, float d1, float (&v)[C],
                                           DF& mine, f2 (&up2)[C], float m, float inv_m1, float eps, int max_iter,
                                           int& flags, int& k_out, int& status_out, float& delta_out, DF& J) {
    const f2 b2 = pack2((float)(2 * threadIdx.x), (float)(2 * threadIdx.x + 1));
    const bool in0 = lo2(cnt2) > 0.0f, in1 = hi2(cnt2) > 0.0f;
    int status = FCM_NOT_CONVERGED, k;
    float delta = 0.0f;
    f2 J2;
#pragma unroll 1
    for (k = 1;; ++k) {
        PackedCenters<C, MK> cen;
        bin_centers<C, MK>(sc, v, cen);
        float base[C];
#pragma unroll
        for (int j = 0; j < C; ++j) base[j] = bin_base(v[j]);
        f2 u2[C], um2[C], d2[C], num2[C];
        bin_memberships<C, MK>(b2, cen, base, m, inv_m1, u2, um2, d2, J2);
        float ma = 0.0f, mb = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            float da, db;
            unpack2(sub2(u2[j], up2[j]), da, db);
            ma = fmaxf(ma, fabsf(da));
            mb = fmaxf(mb, fabsf(db));
            up2[j] = u2[j];
            um2[j] = mul2(cnt2, um2[j]);
            num2[j] = mul2(um2[j], d2[j]);
        }
        float mx = fmaxf(in0 ? ma : 0.0f, in1 ? mb : 0.0f);
        float vn[C];
        DF next = mine;
        const bool empty = bin_reduce<C>(sc, par, num2, um2, mx, base, vn, next);
        delta = (from_u && k == 1) ? d1 : mx;
        if (delta < eps) {
            status = FCM_OK;
            break;
        }
        if (k >= max_iter) break;
        // V^{k+1} (Eq. 3); an empty cluster keeps v_j
        if (empty) flags |= FCM_FLAG_EMPTY_CLUSTER;
        mine = next;
#pragma unroll
        for (int j = 0; j < C; ++j) v[j] = vn[j];
    }
    // J_k: an FP32 tree in each warp, then the warp totals in double-float
    const f2 jt = mul2(cnt2, J2);
    const float jw = warp_sum(lo2(jt) + hi2(jt));
    if ((threadIdx.x & 31) == 0) sc.w[par][threadIdx.x >> 5][0] = jw;
    __syncthreads();
    J = DF{sc.w[par][0][0], 0.0f};
#pragma unroll
    for (int w = 1; w < BIN_NW; ++w) J = df_merge(J, DF{sc.w[par][w][0], 0.0f});
    par ^= 1;
    __syncthreads();
    k_out = k;
    status_out = status;
    delta_out = delta;
}

}  // namespace fcm
