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
//  * A control warp beside the pixel warps takes max |U^k - U^{k-1}| over a
//    sample of the pixels (U^{k-1} again from V^{k-1}, or from U^0 at k = 1). The
//    maximum over a sample is a lower bound of delta_k: when it reaches eps in any
//    block the run cannot stop at k, and the exact delta_k is not needed.
//  * When it does not, or k is max_iter, or a trace wants every iteration, a
//    full pass takes delta_k over every pixel and J_k (Eq. 1), and writes U^k. If
//    the run goes on all the same, the next samples hold the pairs of largest
//    change that the pixel warps saw.
// The iterates, the stop decision and the outputs are those of the loop that
// takes delta_k in every iteration; U is written once instead of k times.
//
// What bounds it: on a large image the FP32 pipe (33 operations per pixel and
// iteration at C = 4, m = 2, in packed FP32x2 pairs: 14 us per iteration of a
// 256^3 volume at the pipe's rate, 27 measured; 15 pixel warps per SM, two pairs
// in flight each: 23 or 31 warps with fewer registers were slower). x is kept in
// shared memory up to 7 million pixels; beyond that, the rest of x comes from the
// L2, two steps ahead of its use. On a small image it is the latency of an
// iteration (1.9 us at 40,000 pixels): a single block of 512 pixels, whose exchange is
// an L2 round trip that no other block contends for, takes 1.4. 60 iterations on a GB300, before (U stored; plain
// loads and a launch per pass where n % 4 != 0) and after: 200x200 374 -> 153 us,
// 199x201 902 -> 191 us, 1024x1024 717 -> 273 us, 256^3 6.02 -> 1.77 ms.
//
// The exchange. Between iterations every block adds its totals of (num_j, den_j)
// as 64-bit fixed-point numbers to one word each, with a reduction in the L2; the
// top byte of a word counts the arrivals, so the word itself says when the sum
// is complete, and the warp that needs cluster j polls these two words and
// nothing else. Integer sums do not depend on the order of arrival: every block
// reads the same totals and forms the same V^{k+1}. (Slots that every block
// polls for every other one cost 5,000 cycles per exchange at 152 blocks, most
// of it contention of the polls: 7.5 us per iteration of a 1 M-pixel image.)
// The words are never cleared within a run: those of even and odd exchanges
// alternate, and a sum is the difference from the word's value two exchanges
// ago, which no block can have moved on from before all have read it. The
// fixed-point units come from n and the largest |x|, |V^0|, known after pass 0:
// 2^-53 of the largest num_j possible, 2^-46 of n (the error of den_j is relative
// to the center's step). A few outliers or a masked part at some sentinel value set
// the largest |x|, and the other clusters' totals may lie wholly below the unit:
// when all blocks' roundings together could move a center by 2^-26 of it and are
// not below 2^-16 of its step, when den_j is below 2^-16 n, or when some block's
// total is no number (it adds a mark instead), then (the same decision in every
// block) the totals go through the slots, in FP32, and so do the next ones until
// the words would do. Measured there: 40,000 pixels 1.9 -> 2.8 us per iteration,
// 1 M 3.8 -> 6.0. (A second word for what the first one leaves of num_j needs none
// of that, but costs every run: 40,000 pixels, 60 iterations, 151.6 -> 161.2 us with
// a line of its own, 172 on the same line.) Pass 0's totals and J's always go
// through the slots.
// Slots: a block's values with a 64-bit tag (the run's number and the exchange's
// index) in one 16-byte store, polled until each block's shows the tag, added in
// block order in compensated FP32.
// Every poll loop is bounded (fcm_set_limits): the run then ends with
// FCM_ERR_TIMEOUT.
#include <type_traits>

#include "fcm_bounds.cuh"
#include "fcm_device.cuh"
#include "fcm_df.cuh"
#include "fcm_internal.h"
#include "fcm_run.h"

#ifndef FCM_INST_C
#error "compile with -DFCM_INST_C=<cluster count>"
#endif

namespace fcm {
namespace {

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

// ---- exchange words ----

constexpr uint64_t ARRIVAL = 1ull << 56;  // the top byte counts blocks (at most 255)

__device__ __forceinline__ void red_add_u64(uint64_t* p, uint64_t v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void ld_words(const uint64_t* p, uint64_t& a, uint64_t& b) {
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "ld.relaxed.gpu.global.b128 t, [%2];\n\t"
        "mov.b128 {%0, %1}, t;\n\t}"
        : "=l"(a), "=l"(b)
        : "l"(p)
        : "memory");
}
__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) {
    uint64_t a;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    return a;
}
// The arrivals in a word's change since an earlier value; the sum in it may be
// negative, but is below 2^55 in magnitude.
__device__ __forceinline__ unsigned arrivals(uint64_t change) { return (unsigned)((change + (ARRIVAL >> 1)) >> 56); }
// v * unit, |v| < 2^55 and unit a power of two, to 2^-25 of itself or better: the
// upper part exactly, the lower 31 bits (signed) rounded; then renormalised.
__device__ __forceinline__ DF fixed_to_df(int64_t v, float unit) {
    const int top = (int)((v + (1ll << 30)) >> 31);
    const float a = (float)top * 2147483648.0f, b = (float)(int)(v - ((int64_t)top << 31));
    const float hi = __fadd_rn(a, b);
    return DF{hi * unit, __fsub_rn(b, __fsub_rn(hi, a)) * unit};
}
// Bits of the sum of an exchange word.
constexpr int NUM_BITS = 53, DEN_BITS = 46;
constexpr uint64_t DEN_MARK = 2ull << DEN_BITS;  // 255 of them stay below 2^55
// Iterations that a cluster's totals are taken to be resolved after an exchange
// through the slots has shown that they are.
constexpr int TRUST = 16;
// The units of the fixed-point numbers.
struct Fixed {
    float to_num, to_den, num_unit, den_unit;
    float num_max, den_max;  // no block's totals are above these
    float lost;              // all blocks' roundings to the unit, at most
    float thick;             // least den_j, in slots, that the words may have again
    // Whether a block's totals are numbers that the words can add.
    __device__ __forceinline__ bool fits(float a, float b) const { return fabsf(a) <= num_max && b <= den_max; }
    // Whether the roundings move a center v with the sums a, b by less than 2^-26 of
    // it, or are below 2^-16 of what moves it. slack > 1 asks for that much more room.
    __device__ __forceinline__ bool resolves(float a, float b, float v, float slack) const {
        return b * fabsf(v) >= (0x1p26f * slack) * lost || fabsf(a) >= (0x1p16f * slack) * lost;
    }
};
// 2^e for e in [-126, 127].
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

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

// ---- the sums of a sums pass ----

// The numerators are centered: num_j = sum u_j^m (x - v_j^k), so that
// v_j^{k+1} = v_j^k + num_j / den_j. The differences are at hand, and the FP32
// rounding of the sums is then relative to the pixels' distance from the center
// and not to their grey level, and vanishes from den as the run converges. (A
// center that moves by more than it is worth takes its sums again: rebased_pass.)
//
// Sums in two levels: pairs into num2/den2, those into a second set after every
// FOLD quads. A thread's share of a 256^3 volume is 27 quads; many of its terms
// are equal (a constant background), so a single chain of additions rounds the
// same way again and again, in all threads alike. Uncentered and in one chain of
// 108, the sums moved the iteration at which a random start of that volume
// breaks its symmetry by three. The second set is touched once in FOLD quads
// and lives in shared memory, not in registers.
constexpr int FOLD = 8;
static_assert(RUN_MAX_PW <= 16, "the block's totals are a tree over 16 lanes");
// Pairs of pixels whose arithmetic overlaps: as many as fit in the registers.
constexpr int run_pairs(int C) { return C <= 6 ? 2 : 1; }

template <int C>
struct SumAcc {
    f2 num2[C], den2[C];
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int j = 0; j < C; ++j) num2[j] = den2[j] = pack2(0.0f, 0.0f);
    }
    __device__ __forceinline__ void add(const f2 (&d2)[C], const f2 (&um2)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num2[j] = fma2(um2[j], d2[j], num2[j]);
            den2[j] = add2(den2[j], um2[j]);
        }
    }
    // Into the second set (of this thread: stride threads apart), or from it.
    __device__ __forceinline__ void fold(f2* set, int stride, bool first) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            f2* const a = set + (2 * j) * stride;
            f2* const b = a + stride;
            *a = first ? num2[j] : add2(*a, num2[j]);
            *b = first ? den2[j] : add2(*b, den2[j]);
        }
        reset();
    }
    __device__ __forceinline__ void finish(const f2* set, int stride, bool folded) {
        if (!folded) return;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            num2[j] = add2(num2[j], set[(2 * j) * stride]);
            den2[j] = add2(den2[j], set[(2 * j + 1) * stride]);
        }
    }
};

// The pixels of a pass. Pixel thread t0 of nt takes the quads (four consecutive
// pixels) t0, t0 + nt, ...; the first `resident` of them stay in shared memory
// for the whole run (at xs[step * pt], this thread's own place), the others are
// read again in every pass.
struct Px {
    const float* __restrict__ x;
    float4* xs;
    int64_t n, t0, nt;
    int pt;               // pixel threads of the block
    int steps, resident;  // this thread's quads; how many of them are kept
    bool vec_x;           // x is 16-byte aligned
    bool vec_u;           // so are the rows of U and U^0, and n % 4 == 0
    int64_t guard_n;      // a FCM_DEBUG_BOUNDS build checks every index against it
    unsigned* bounds;     // and reports here

    // Whether the pixels i .. i + count - 1 may be accessed.
    __device__ __forceinline__ bool in(int64_t i, int count) const { return in_bounds(i >= 0 && i + count <= guard_n, bounds); }
    __device__ __forceinline__ float4 load(int step) const {
        const int64_t q = t0 + (int64_t)step * nt;
        if (!in(4 * q, 4)) return make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec_x) return __ldg(reinterpret_cast<const float4*>(x) + q);
        const float* p = x + 4 * q;
        return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
    }
    // tail(i) on the pixels past the last whole quad (at most three, on one thread)
    template <typename T>
    __device__ __forceinline__ void tail(T&& f) const {
        if (t0 == (n >> 2) % nt) {
#pragma unroll 1
            for (int64_t i = n & ~(int64_t)3; i < n; ++i)
                if (in(i, 1)) f(i);
        }
    }
    // Reads the quads from global memory, two steps ahead, keeps the resident
    // ones and calls f(quad, index of its first pixel).
    template <typename F>
    __device__ __forceinline__ void stage(F&& f) const {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (steps > 0) a = load(0);
        if (steps > 1) b = load(1);
#pragma unroll 1
        for (int s = 0; s < steps; ++s) {
            const float4 c = a;
            a = b;
            if (s + 2 < steps) b = load(s + 2);
            if (s < resident) xs[s * pt] = c;
            const int64_t i = 4 * (t0 + (int64_t)s * nt);
            if (in(i, 4)) f(c, i);
        }
    }
    // The same, once the resident quads are in place.
    template <typename F>
    __device__ __forceinline__ void quads(F&& f) const {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (resident < steps) {
            a = load(resident);
            if (resident + 1 < steps) b = load(resident + 1);
        }
#pragma unroll 1
        for (int s = 0; s < steps; ++s) {
            float4 c;
            if (s < resident) {
                c = xs[s * pt];
            } else {
                c = a;
                a = b;
                if (s + 2 < steps) b = load(s + 2);
            }
            const int64_t i = 4 * (t0 + (int64_t)s * nt);
            if (in(i, 4)) f(c, i);
        }
    }
    // For unaligned rows of U: a warp takes 128 consecutive pixels, a lane the
    // pixels i + 32 p, p = 0..3 (coalesced 32-bit accesses); whole tiles through f,
    // the last partial one pixel by pixel through g.
    template <typename F, typename G>
    __device__ __forceinline__ void tiles(F&& f, G&& g) const {
        const int64_t nw = nt >> 5, all = (n + 127) >> 7;
#pragma unroll 1
        for (int64_t w = t0 >> 5; w < all; w += nw) {
            const int64_t i = (w << 7) + (threadIdx.x & 31);
            if ((w << 7) + 128 <= n) {
                if (in(w << 7, 128)) f(make_float4(__ldg(x + i), __ldg(x + i + 32), __ldg(x + i + 64), __ldg(x + i + 96)), i);
            } else {
#pragma unroll 1
                for (int64_t k = i; k < n; k += 32)
                    if (in(k, 1)) g(k);
            }
        }
    }
};

// This thread's pixels. second: the block's dynamic shared memory.
template <int C>
__device__ __forceinline__ Px run_px(const RunArgs& ra, f2* second) {
    Px px;
    px.x = ra.x;
    px.n = ra.n;
    px.pt = (int)blockDim.x - 32;
    px.xs = reinterpret_cast<float4*>(second + 2 * C * px.pt) + threadIdx.x;
    px.t0 = (int64_t)blockIdx.x * px.pt + threadIdx.x;
    px.nt = (int64_t)gridDim.x * px.pt;
    px.steps = (px.n >> 2) > px.t0 ? (int)(((px.n >> 2) - 1 - px.t0) / px.nt) + 1 : 0;
    px.resident = min(ra.resident, px.steps);
    px.guard_n = ra.guard_n;
    px.bounds = &ra.out->bounds;
    if (kBoundsChecks) {
        // the places of the resident quads lie in the block's dynamic shared memory
        unsigned smem;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem));
        if (!in_bounds((unsigned)(px.pt * 16 * (C + ra.resident)) <= smem, px.bounds)) px.resident = 0;
    }
    px.vec_x = ((uintptr_t)px.x & 15) == 0;
    px.vec_u = px.vec_x && (px.n & 3) == 0 && ((uintptr_t)ra.U & 15) == 0 && (!ra.from_u || ((uintptr_t)ra.U0 & 15) == 0);
    return px;
}

template <int C>
struct RunShared {
    float red[RUN_MAX_PW][2 * C];  // warp totals of a sums pass; J in red[w][0] of a full pass
    float mx[RUN_MAX_PW];
    unsigned bad[RUN_MAX_PW];      // bit 0: bad input; bit 1: wit holds a pair of the image
    f2 wit[RUN_MAX_PW];            // each warp's pair of largest change in a full pass
    float v[4][C];             // V^k in v[k % 4]
    DF v64[4][C];              // the double-float quotients behind them
    unsigned empty[4];         // whether some cluster was empty in the sums behind V^k
    // By the parity of the iteration: the control warp writes the next iteration's
    // while slower warps still read this one's (no barrier is between them).
    // x: a wait gave up; y: a sampled change reached eps; z: the exchange words do not
    // hold the sums, or (of an exchange through the slots) would not; w: some cluster
    // is empty, or a center moved by more than REBASE times its new value.
    int4 ctl[2];
    uint64_t seen[2][C][2];    // the words of each cluster after their last exchange, of even and odd parity
    uint64_t seen_ctl[2];      // and the control word
    int trust[C];              // see TRUST
    DF J;
    float delta;
    unsigned flags;            // bit 0: bad input
    WaitLimits lim;
};

// A pixel warp's totals of a sums pass into sh.red.
template <int C>
__device__ __forceinline__ void warp_sums(RunShared<C>& sh, float (&a)[pow2_at_least(2 * C)]) {
    constexpr int P = pow2_at_least(2 * C);
    const int lane = threadIdx.x & 31;
    warp_totals<P>(a);
    const int s = slot_of_lane<P>(lane);
    if ((lane & (32 / P - 1)) == 0 && s < 2 * C) sh.red[threadIdx.x >> 5][s] = a[0];
}

// A sums pass of a pixel warp from V^k in sh.v[cur]. FIRST: pass 0 from V^0,
// which reads x and calls see(x) on every pixel.
template <int C, int MK, bool FIRST, typename See>
__device__ __forceinline__ void sums_pass_body(const Px& px, RunShared<C>& sh, f2* second, int cur, float m,
                                               float inv_m1, See&& see) {
    constexpr int P = pow2_at_least(2 * C);
    SumAcc<C> a;
    a.reset();
    PackedCenters<C, MK> cen;
    cen.set(sh.v[cur]);
    f2* const set = second + threadIdx.x;
    int held = 0;
    bool folded = false;
    auto quad = [&](const float4& c, int64_t) {
        if (FIRST) see(c.x), see(c.y), see(c.z), see(c.w);
        if (run_pairs(C) == 2) {
            f2 um[2][C], d2[2][C], J2[2];
            const f2 xq[2] = {pack2(c.x, c.y), pack2(c.z, c.w)};
            packed_pairs<C, MK, true, 2>(xq, cen, m, inv_m1, um, d2, J2);
            a.add(d2[0], um[0]);
            a.add(d2[1], um[1]);
        } else {
            // one pair at a time: two would not fit in the registers
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                f2 um[1][C], d2[1][C], J2[1];
                const f2 xq[1] = {h ? pack2(c.z, c.w) : pack2(c.x, c.y)};
                packed_pairs<C, MK, true, 1>(xq, cen, m, inv_m1, um, d2, J2);
                a.add(d2[0], um[0]);
            }
        }
        if (++held == FOLD) {
            a.fold(set, px.pt, !folded);
            folded = true;
            held = 0;
        }
    };
    if (FIRST) px.stage(quad);
    else px.quads(quad);
    px.tail([&](int64_t i) {
        // a pixel past the last quad: the low halves of the sums
        const float xi = __ldg(px.x + i);
        if (FIRST) see(xi);
        const PixelPair<C> w = scalar_pair<C, MK, true>(xi, xi, cen.vs, m, inv_m1);
        const f2 xs = cen.of(pack2(xi, xi));
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const f2 um = pack2(w.a[j], 0.0f);
            a.num2[j] = fma2(um, sub2(xs, cen.v2[j]), a.num2[j]);
            a.den2[j] = add2(a.den2[j], um);
        }
    });
    a.finish(set, px.pt, folded);
    // back from scaled differences (by a power of two: exact)
    const float back = PackedCenters<C, MK>::SCALED ? rcp_approx(lo2(cen.scale)) : 1.0f;
    float t[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const f2 q = i < C ? a.num2[i < C ? i : 0] : a.den2[(i >= C && i < 2 * C) ? i - C : 0];
        t[i] = i < 2 * C ? lo2(q) + hi2(q) : 0.0f;
        if (PackedCenters<C, MK>::SCALED && i < C) t[i] *= back;
    }
    warp_sums<C>(sh, t);
}

template <int C, int MK>
__device__ __forceinline__ void sums_pass(const Px& px, RunShared<C>& sh, f2* second, int cur, float m, float inv_m1) {
    sums_pass_body<C, MK, false>(px, sh, second, cur, m, inv_m1, [](float) {});
}

// The sums of a sums pass once more, with the numerators centered on sh.v[basis]:
// for a center that moved by far more than it is now away from 0 (an initial
// center far outside the image, a center between two parts that are far apart),
// whose differences x - v^k have lost the bits of x. Called, not inlined, so that
// the usual passes keep their registers.
template <int C, int MK>
__device__ __noinline__ void rebased_pass(const RunArgs& ra, RunShared<C>& sh, f2* second, int cur, int basis) {
    constexpr int P = pow2_at_least(2 * C);
    const Px px = run_px<C>(ra, second);
    const float m = ra.m, inv_m1 = ra.inv_m1;
    SumAcc<C> a;
    a.reset();
    PackedCenters<C, MK> cen;
    cen.set(sh.v[cur]);
    f2* const set = second + threadIdx.x;
    int held = 0;
    bool folded = false;
    auto pair = [&](f2 x) {
        f2 um[1][C], d2[1][C], J2[1];
        const f2 xq[1] = {x};
        packed_pairs<C, MK, true, 1>(xq, cen, m, inv_m1, um, d2, J2);
#pragma unroll
        for (int j = 0; j < C; ++j) d2[0][j] = sub2(x, pack2(sh.v[basis][j], sh.v[basis][j]));
        a.add(d2[0], um[0]);
    };
    px.quads([&](const float4& c, int64_t) {
        pair(pack2(c.x, c.y));
        pair(pack2(c.z, c.w));
        if (++held == FOLD) {
            a.fold(set, px.pt, !folded);
            folded = true;
            held = 0;
        }
    });
    px.tail([&](int64_t i) {
        const float xi = __ldg(px.x + i);
        const PixelPair<C> w = scalar_pair<C, MK, true>(xi, xi, cen.vs, m, inv_m1);
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const f2 um = pack2(w.a[j], 0.0f);
            a.num2[j] = fma2(um, pack2(xi - sh.v[basis][j], 0.0f), a.num2[j]);
            a.den2[j] = add2(a.den2[j], um);
        }
    });
    a.finish(set, px.pt, folded);
    float t[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const f2 q = i < C ? a.num2[i < C ? i : 0] : a.den2[(i >= C && i < 2 * C) ? i - C : 0];
        t[i] = i < 2 * C ? lo2(q) + hi2(q) : 0.0f;
    }
    warp_sums<C>(sh, t);
}

// What an exchange adds up over the blocks.
enum Exchange : int { X_SUMS0 = 0, X_SUMS = 1, X_J = 2 };  // sums of pass 0 from U^0; centered sums; J

// The FP32 differences x - v_j^k round by 2^-24 of the step at most, so up to this
// factor the new center keeps about 18 bits; beyond it, the pass is taken again.
constexpr float REBASE = 64.0f;

template <int C, int MK>
__global__ void __launch_bounds__(run_max_pt(C) + 32, 1)
    k_fcm_run(const __grid_constant__ RunArgs ra) {
    constexpr int P = pow2_at_least(2 * C);
    extern __shared__ __align__(16) f2 second[];  // [2 C][pt] second set of the sums, then the resident quads
    __shared__ RunShared<C> sh;
    // the scratch has room for the grid's slots, and the words can count its blocks
    if (!in_bounds((int)gridDim.x <= ra.max_blocks, &ra.out->bounds)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pw = (int)(blockDim.x >> 5) - 1;  // pixel warps; the control warp follows
    const bool control = warp == pw;
    const int nb = (int)gridDim.x;
    char* const scratch = ra.scratch;
    const unsigned nonce = ra.nonce;
    RunState* const st = ra.out;
    const bool from_u = ra.from_u != 0;
    const float* U0 = ra.U0;  // may be U itself: each pixel is read, then written, by one thread
    float* U = ra.U;
    const int64_t n = ra.n;
    const Px px = run_px<C>(ra, second);
    const float m = ra.m, inv_m1 = ra.inv_m1, eps = ra.eps;
    const int max_iter = ra.max_iter;
    const bool tracing = ra.trace != nullptr;

    if (threadIdx.x < C) sh.trust[threadIdx.x] = 0;
    if (threadIdx.x < 4 * C) (&sh.seen[0][0][0])[threadIdx.x] = 0ull;
    if (threadIdx.x < C) {
        const float v0 = ra.Vin ? ra.Vin[threadIdx.x] : ra.V0[threadIdx.x];
        sh.v[0][threadIdx.x] = v0;
        sh.v64[0][threadIdx.x] = DF{v0, 0.0f};
    }
    if (threadIdx.x == 0) {
        sh.ctl[0] = sh.ctl[1] = make_int4(0, 0, 0, 0);
        sh.seen_ctl[0] = sh.seen_ctl[1] = 0ull;
        sh.empty[0] = sh.empty[1] = sh.empty[2] = sh.empty[3] = 0u;
        sh.lim = ra.lim;
    }
    __syncthreads();
    int flags = 0;    // thread 0 of block 0 only
    unsigned nx = 0;  // exchanges so far
    int it = 0;       // parity of the iteration (0 in pass 0)

    // The words of this run's bank (runs alternate between two; each run clears
    // the other one, which the next run uses): [parity][cluster] pairs and, in row
    // C, the control word, a 128-byte line each.
    auto word = [&](unsigned bank, unsigned x, int q) {
        return reinterpret_cast<uint64_t*>(scratch + RUN_WORD_BYTES * (((bank & 1) * 2 + (x & 1)) * (FCM_MAX_CLUSTERS + 1) + q));
    };
    if (blockIdx.x == 0 && threadIdx.x < 2 * (FCM_MAX_CLUSTERS + 1)) {
        uint64_t* const w = word(nonce + 1, threadIdx.x & 1, threadIdx.x >> 1);
        w[0] = w[1] = 0ull;
    }
    char* const slots_raw = scratch + RUN_WORDS_BYTES;
    Fixed fx{0.0f, 0.0f, 0.0f, 0.0f, -1.0f, -1.0f, 0.0f, 0.0f};  // nothing fits

    // This block's row of exchange nx + 1: cluster q's slots, or (q = C) the
    // maxima's and flags'.
    auto slot_row = [&](int q, unsigned x) {
        return slots_raw + ((int64_t)(x & 1) * (C + 1) + q) * nb * RUN_SLOT_BYTES;
    };
    // Control warp: publishes the block's maximum and flags and collects every
    // block's into sh.delta and sh.flags.
    auto exchange_max = [&](float mx, unsigned fl) {
        const uint64_t tag = ((uint64_t)nonce << 32) | (nx + 1);
        char* const row = slot_row(C, nx + 1);
        unsigned tm = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));  // non-negative floats order as their bits
        unsigned tf = __reduce_or_sync(0xffffffffu, fl);
        if (lane == 0) st_slot(row + (int64_t)blockIdx.x * RUN_SLOT_BYTES, __uint_as_float(tm), __uint_as_float(tf), tag);
        const bool ok = collect(row, nb, tag, sh.lim.grid_spins, sh.lim.phantoms, [&](float p, float r) {
            tm = max(tm, __float_as_uint(p));
            tf |= __float_as_uint(r);
        });
        tm = __reduce_max_sync(0xffffffffu, tm);
        tf = __reduce_or_sync(0xffffffffu, tf);
        if (lane == 0) {
            sh.delta = __uint_as_float(tm);
            sh.flags = tf;
            if (!ok) sh.ctl[it].x = 1;
        }
    };
    // V^{k+1}_q from the totals (one lane).
    auto new_center = [&](int q, DF na, DF da, bool centered, int cur, int nxt) {
        if (da.hi > 0.0f) {
            DF r = (da.hi > 1e-30f && da.hi < 1e30f) ? df_div_fast(na, da) : df_div(na, da);
            const float step = fabsf(r.hi);
            if (centered) r = df_merge(r, DF{sh.v[cur][q], 0.0f});
            sh.v[nxt][q] = r.hi;
            sh.v64[nxt][q] = r;
            if (centered && step > REBASE * fabsf(r.hi)) sh.ctl[it].w = 1;
        } else {
            // an empty cluster keeps its center (in pass 0 that is V^0, or 0 from a U^0)
            sh.v[nxt][q] = centered ? sh.v[cur][q] : 0.0f;
            sh.v64[nxt][q] = centered ? sh.v64[cur][q] : DF{0.0f, 0.0f};
            sh.empty[nxt] = 1u;
            sh.ctl[it].w = 1;
        }
    };
    // Warp q < C (q = 0 for X_J): the block's totals from the warp totals, then
    // the grid's. X_SUMS*: V^{k+1}_q into sh.v[nxt], sh.v64[nxt]; cur is the slot
    // of V^k, which centers the numerators. X_J: sh.J.
    auto exchange_sums = [&](auto kind, int q, int cur, int nxt) {
        constexpr int K = decltype(kind)::value;
        const uint64_t tag = ((uint64_t)nonce << 32) | (nx + 1);
        char* const row = slot_row(q, nx + 1);
        float a = lane < pw ? sh.red[lane][q] : 0.0f, b = (K != X_J && lane < pw) ? sh.red[lane][C + q] : 0.0f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            if (K != X_J) b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        if (lane == 0) st_slot(row + (int64_t)blockIdx.x * RUN_SLOT_BYTES, a, b, tag);
        DF na{0.0f, 0.0f}, da{0.0f, 0.0f};
        bool fits = true;
        float amax = 0.0f;  // the largest block's |num_j|
        const bool ok = collect(row, nb, tag, sh.lim.grid_spins, sh.lim.phantoms, [&](float p, float r) {
            if (K == X_SUMS) {
                fits &= fx.fits(p, r);
                amax = fmaxf(amax, fabsf(p));
            }
            df_add(na, p);
            if (K != X_J) df_add(da, r);
        });
        if (K == X_SUMS) {
            fits = __all_sync(0xffffffffu, fits);
            amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            // TwoSum is symmetric: every lane gets the same totals
            na = df_merge_raw(na, DF{__shfl_xor_sync(0xffffffffu, na.hi, o), __shfl_xor_sync(0xffffffffu, na.lo, o)});
            if (K != X_J)
                da = df_merge_raw(da, DF{__shfl_xor_sync(0xffffffffu, da.hi, o), __shfl_xor_sync(0xffffffffu, da.lo, o)});
        }
        if (lane != 0) return;
        if (!ok) sh.ctl[it].x = 1;
        na = df_norm(na);
        if (K == X_J) {
            sh.J = na;
            return;
        }
        da = df_norm(da);
        if (K == X_SUMS) {
            // Would the words do? A center near 0 that hardly moves any more is
            // resolved where the roundings are small against the largest block's part
            // of the sum (parts that cancel), or every part is 0.
            const bool ok2 = fx.resolves(amax, da.hi, sh.v[cur][q], 4.0f) || amax == 0.0f;
            sh.trust[q] = fits && ok2 ? TRUST : 0;
            if (!fits || !ok2 || !(da.hi >= fx.thick)) sh.ctl[it].z = 1;
        }
        new_center(q, na, da, K == X_SUMS, cur, nxt);
    };
    // Reads words until they are complete.
    auto poll = [&](auto&& complete) {
        const uint32_t limit = sh.lim.grid_spins, phantoms = sh.lim.phantoms;
        for (uint32_t spins = 0;;) {
            if (complete() && phantoms == 0) return true;
            if (++spins > limit) return false;
            if (spins > 256) __nanosleep(100);
        }
    };
    // Warp q < C between iterations: the block's totals into cluster q's words,
    // then V^{k+1}_q from the complete ones (one lane polls).
    auto exchange_words = [&](int q, int cur, int nxt) {
        uint64_t* const w = word(nonce, nx + 1, q);
        const float v = sh.v[cur][q];
        float a = lane < pw ? sh.red[lane][q] : 0.0f, b = lane < pw ? sh.red[lane][C + q] : 0.0f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        if (lane != 0) return;
        // Totals that are no numbers, or too large, add only a mark to den_j, beyond
        // every possible sum of them: nothing else may reach the arrival counts.
        const bool fits = fx.fits(a, b);
        red_add_u64(w, (uint64_t)__float2ll_rn(fits ? a * fx.to_num : 0.0f) + ARRIVAL);
        red_add_u64(w + 1, (uint64_t)__float2ll_rn(fits ? b * fx.to_den : (float)DEN_MARK) + ARRIVAL);
        uint64_t* const seen = sh.seen[(nx + 1) & 1][q];
        const uint64_t pa = seen[0], pb = seen[1];
        uint64_t va, vb;
        const bool ok = poll([&] {
            ld_words(w, va, vb);
            return arrivals(va - pa) == (unsigned)nb && arrivals(vb - pb) == (unsigned)nb;
        });
        const int64_t sa = (int64_t)(va - pa - (uint64_t)nb * ARRIVAL), sb = (int64_t)(vb - pb - (uint64_t)nb * ARRIVAL);
        seen[0] = va;
        seen[1] = vb;
        if (!ok) sh.ctl[it].x = 1;
        if (sb < (1ll << (DEN_BITS - 16)) || sb >= (int64_t)DEN_MARK) {
            sh.ctl[it].z = 1;
        } else {
            const DF na = fixed_to_df(sa, fx.num_unit), da = fixed_to_df(sb, fx.den_unit);
            new_center(q, na, da, true, cur, nxt);
            if (!fx.resolves(na.hi, da.hi, v, 1.0f) && --sh.trust[q] < 0) sh.ctl[it].z = 1;
        }
    };
    // Control warp: publishes whether this block's sample of iteration k reached
    // eps; collects, an iteration later, whether any block's did.
    auto publish_decision = [&](int k, float mx) {
        const bool ge = __any_sync(0xffffffffu, mx >= eps);
        if (lane == 0) red_add_u64(word(nonce, k, C), 1ull + (ge ? 1ull << 16 : 0ull));
    };
    auto collect_decision = [&](int k) {
        if (lane != 0) return;
        const uint64_t* const w = word(nonce, k, C);
        const uint64_t pa = sh.seen_ctl[k & 1];
        uint64_t va;
        const bool ok = poll([&] {
            va = ld_word(w);
            return ((va - pa) & 0xffffu) == (unsigned)nb;
        });
        sh.ctl[it].y = ((va - pa) >> 16) != 0;
        sh.seen_ctl[k & 1] = va;
        if (!ok) sh.ctl[it].x = 1;
    };
    // V^{k+1} in slot nxt again, with sums centered on what it holds, if a center moved
    // far. False when a wait gave up.
    auto rebase = [&](int cur, int nxt) {
        bool far = false;
#pragma unroll
        for (int j = 0; j < C; ++j) far |= fabsf(sh.v[nxt][j] - sh.v[cur][j]) > REBASE * fabsf(sh.v[nxt][j]);
        if (!far) return true;
        __syncthreads();
        if (!control) rebased_pass<C, MK>(ra, sh, second, cur, nxt);
        __syncthreads();
        if (warp < C) exchange_sums(std::integral_constant<int, X_SUMS>(), warp, nxt, nxt);
        ++nx;
        __syncthreads();
        return sh.ctl[it].x == 0;
    };
    // ---- pass 0: V^1 from U^0, or from U^0 = f(x, V^0) ----
    bool ok;
    {
        bool bad = false;
        float xmax = 0.0f;  // largest |x| (and |V^0|)
        auto see = [&](float xi) {
            bad |= !finite_f(xi);
            xmax = fmaxf(xmax, fabsf(xi));
        };
        if (control) {
            if (!from_u && lane < C) see(sh.v[0][lane]);
        } else if (from_u) {
            // four pixels in FP32, then double-float: the pass waits for memory, and
            // the separation of the V^1 of a random start is of the order of 1e-5
            DF sn[C], sd[C];
            float num[C], den[C];
#pragma unroll
            for (int j = 0; j < C; ++j) {
                sn[j] = sd[j] = DF{0.0f, 0.0f};
                num[j] = den[j] = 0.0f;
            }
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
            auto single = [&](int64_t i) {
                const float xi = __ldg(px.x + i);
                see(xi);
#pragma unroll
                for (int j = 0; j < C; ++j) one(xi, __ldcs(U0 + (int64_t)j * n + i), j);
            };
            if (px.vec_u) {
                px.stage([&](const float4& c, int64_t i) {
                    see(c.x), see(c.y), see(c.z), see(c.w);
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
                });
            } else {
                px.stage([&](const float4&, int64_t) {});
                px.tiles(
                    [&](const float4& c, int64_t i) {
                        see(c.x), see(c.y), see(c.z), see(c.w);
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
#pragma unroll
                            for (int j = 0; j < C; ++j) one(comp(c, p), __ldcs(U0 + (int64_t)j * n + i + 32 * p), j);
                        }
                        fold();
                    },
                    single);
            }
            fold();
            float t[P];
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const DF q = i < C ? sn[i < C ? i : 0] : sd[(i >= C && i < 2 * C) ? i - C : 0];
                t[i] = i < 2 * C ? q.hi + q.lo : 0.0f;
            }
            warp_sums<C>(sh, t);
        } else {
            sums_pass_body<C, MK, true>(px, sh, second, 0, m, inv_m1, see);
        }
        const unsigned wx = __reduce_max_sync(0xffffffffu, __float_as_uint(xmax));
        const bool wbad = __any_sync(0xffffffffu, bad);
        if (!control && lane == 0) {
            sh.bad[warp] = wbad ? 1u : 0u;
            sh.mx[warp] = __uint_as_float(wx);
        }
        __syncthreads();
        if (control) exchange_max(fmaxf(xmax, lane < pw ? sh.mx[lane] : 0.0f), (wbad ? 1u : 0u) | (lane < pw ? sh.bad[lane] : 0u));
        else if (warp < C && from_u) exchange_sums(std::integral_constant<int, X_SUMS0>(), warp, 0, 1);
        else if (warp < C) exchange_sums(std::integral_constant<int, X_SUMS>(), warp, 0, 1);
        ++nx;
        __syncthreads();
        ok = sh.ctl[0].x == 0;
        if (ok && !from_u && !(sh.flags & 1u)) ok = rebase(0, 1);
    }
    // The fixed-point units: |num_j| <= 2 n max(|x|, |V^0|) < 2^NUM_BITS units and
    // den_j <= n. Images whose FP32 sums could overflow never use the words.
    const int en = 64 - __clzll(n);                                        // n < 2^en
    const int ex = max(-100, (__float_as_int(sh.delta) >> 23) - 125);      // 2 max|x| < 2^ex
    const bool fixed = en + ex <= 126;
    if (fixed) {
        const int e = min(126, NUM_BITS - en - ex);
        fx = Fixed{pow2f(e), pow2f(DEN_BITS - en), pow2f(-e), pow2f(en - DEN_BITS), pow2f(min(127, en + ex)), 1.25f * pow2f(en),
                   (0.5f * (float)nb) * pow2f(-e), pow2f(en - 15)};
    }
    bool words = fixed;  // the next exchange of sums goes through the words (the same in every block)
    int status = FCM_NOT_CONVERGED, iters = 0;
    if (!ok) {
        status = FCM_ERR_TIMEOUT;
    } else if (sh.flags & 1u) {
        status = FCM_ERR_BAD_INPUT;
        ok = false;
    }
    // The control warp samples the change of one pair per lane. The pairs are
    // spread evenly over the image and are pairs of the full pass (so their
    // changes are bit for bit the full pass's); after a full pass that did not
    // stop the run, the lanes of the pixel warps' numbers hold those warps' pairs
    // of largest change.
    f2 wx = 0;
    int64_t wi = 0;
    int ws = 1;
    bool sampled = false;
    if (control) {
        const double at = ((double)blockIdx.x * 32 + lane) / ((double)nb * 32);
        const int64_t i = (int64_t)(at * (double)n);
        if (px.vec_u) {
            wi = min(i, n - 2) & ~(int64_t)1;
            sampled = px.in(wi, 2);
        } else {
            const int64_t whole = n >> 7;
            wi = (min(i >> 7, whole - 1) << 7) + lane;
            ws = 32;
            sampled = whole > 0 && px.in(wi, ws + 1);
        }
        if (sampled) wx = pack2(__ldg(px.x + wi), __ldg(px.x + wi + ws));
    }

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
        float d = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            float da, db;
            u2[j] = w[0][j];
            unpack2(sub2(w[0][j], o[0][j]), da, db);
            d = fmaxf(d, fmaxf(fabsf(da), fabsf(db)));
        }
        return d;
    };
    // The full pass of iteration k: delta_k and J_k over every pixel, and U^k.
    // False when a wait gave up.
    auto full_pass = [&](int k) {
        const int cur = k & 3, prv = (k - 1) & 3;
        const bool prev_u0 = from_u && k == 1;
        if (!control) {
            f2 J2 = pack2(0.0f, 0.0f), best = 0;
            float J1 = 0.0f, dmax = -1.0f, dtail = 0.0f;
            PackedCenters<C, MK> cen, pre;
            cen.set(sh.v[cur]);
            pre.set(sh.v[prv]);
            auto pair = [&](f2 xq, f2 (&u2)[C], const f2 (&u0)[C]) {
                f2 j2;
                const float d = change(xq, cen, pre, u2, u0, prev_u0, j2);
                J2 = add2(J2, j2);
                if (d > dmax) {
                    dmax = d;
                    best = xq;
                }
            };
            auto single = [&](int64_t i) {
                const float xi = __ldg(px.x + i);
                const PixelPair<C> a = scalar_pair<C, MK, false>(xi, xi, cen.vs, m, inv_m1);
                J1 += a.Ja;
                if (prev_u0) {
#pragma unroll
                    for (int j = 0; j < C; ++j) dtail = fmaxf(dtail, fabsf(a.a[j] - __ldcs(U0 + (int64_t)j * n + i)));
                } else {
                    const PixelPair<C> b = scalar_pair<C, MK, false>(xi, xi, pre.vs, m, inv_m1);
#pragma unroll
                    for (int j = 0; j < C; ++j) dtail = fmaxf(dtail, fabsf(a.a[j] - b.a[j]));
                }
                {
#pragma unroll
                    for (int j = 0; j < C; ++j) __stcs(U + (int64_t)j * n + i, a.a[j]);
                }
            };
            if (px.vec_u) {
                px.quads([&](const float4& c, int64_t i) {
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
                    {
#pragma unroll
                        for (int j = 0; j < C; ++j)
                            st_u4(U + (int64_t)j * n + i, make_float4(lo2(ua[j]), hi2(ua[j]), lo2(ub[j]), hi2(ub[j])));
                    }
                });
            } else {
                px.tiles(
                    [&](const float4& c, int64_t i) {
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            f2 u[C], u0[C];
                            const int64_t ia = i + 64 * h, ib = ia + 32;
                            if (prev_u0) {
#pragma unroll
                                for (int j = 0; j < C; ++j)
                                    u0[j] = pack2(__ldcs(U0 + (int64_t)j * n + ia), __ldcs(U0 + (int64_t)j * n + ib));
                            }
                            pair(h ? pack2(c.z, c.w) : pack2(c.x, c.y), u, u0);
                            {
#pragma unroll
                                for (int j = 0; j < C; ++j) {
                                    __stcs(U + (int64_t)j * n + ia, lo2(u[j]));
                                    __stcs(U + (int64_t)j * n + ib, hi2(u[j]));
                                }
                            }
                        }
                    },
                    single);
            }
            J1 = warp_sum(J1 + lo2(J2) + hi2(J2));
            const float own = fmaxf(dmax, 0.0f);
            const unsigned wb = __reduce_max_sync(0xffffffffu, __float_as_uint(own));
            const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(own, dtail)));
            const unsigned who = __ballot_sync(0xffffffffu, dmax >= 0.0f && __float_as_uint(own) == wb);
            if (lane == (who ? __ffs(who) - 1 : 0)) sh.wit[warp] = best;
            if (lane == 0) {
                sh.red[warp][0] = J1;
                sh.mx[warp] = __uint_as_float(mb);
                sh.bad[warp] = who ? 2u : 0u;
            }
        }
        __syncthreads();
        if (control) {
            if (lane < pw && (sh.bad[lane] & 2u)) {
                wx = sh.wit[lane];
                sampled = true;
            }
            exchange_max(lane < pw ? sh.mx[lane] : 0.0f, 0u);
        } else if (warp == 0) {
            exchange_sums(std::integral_constant<int, X_J>(), 0, 0, 0);
        }
        ++nx;
        __syncthreads();
        if (sh.ctl[it].x) return false;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->delta = sh.delta;
            st->J = df_to_double(sh.J);
            if (tracing) {
                double* t = ra.trace + (int64_t)(k - 1) * (2 + C);
                t[0] = sh.delta;
                t[1] = df_to_double(sh.J);
#pragma unroll
                for (int j = 0; j < C; ++j) t[2 + j] = df_to_double(sh.v64[cur][j]);
            }
        }
        return true;
    };
    // Iterations. The decision of iteration k - whether its sample shows that the
    // run goes on - is collected an iteration later, so that the control warp's
    // sample and exchange are never waited for: iteration k + 1 runs meanwhile, and
    // is dropped when the full pass of iteration k stops the run.
    auto give_up = [&](int k) {
        status = FCM_ERR_TIMEOUT;
        iters = k;
        return false;
    };
    if (ok && threadIdx.x == 0 && sh.empty[1]) flags |= FCM_FLAG_EMPTY_CLUSTER;
    bool empty = false;  // some cluster is in the sums behind V^k, k > 1
    for (int k = 1; ok; ++k) {
        const bool last = k == max_iter, prev_u0 = from_u && k == 1;
        const int cur = k & 3, prv = (k - 1) & 3, nxt = (k + 1) & 3;
        it = k & 1;
        if (!last) {
            if (control) {
                float d = 0.0f;
                if (sampled) {
                    PackedCenters<C, MK> cen, pre;
                    cen.set(sh.v[cur]);
                    pre.set(sh.v[prv]);
                    f2 u0[C], u2[C], J2;
                    if (prev_u0) {
#pragma unroll
                        for (int j = 0; j < C; ++j)
                            u0[j] = pack2(__ldcs(U0 + (int64_t)j * n + wi), __ldcs(U0 + (int64_t)j * n + wi + ws));
                    }
                    d = change(wx, cen, pre, u2, u0, prev_u0, J2);
                }
                publish_decision(k, d);
                if (k > 1) collect_decision(k - 1);
                __syncthreads();
            } else {
                if (threadIdx.x == 0) {
                    sh.empty[nxt] = 0u;
                    sh.ctl[it].z = sh.ctl[it].w = 0;
                }
                sums_pass<C, MK>(px, sh, second, cur, m, inv_m1);
                __syncthreads();
                if (warp < C) {
                    if (words) exchange_words(warp, cur, nxt);
                    else exchange_sums(std::integral_constant<int, X_SUMS>(), warp, cur, nxt);
                }
            }
            ++nx;
        } else {
            // no exchange, and so none counted: the full pass's slots are those of
            // the other parity than the last exchange's, which another block may
            // still be reading
            if (control && k > 1) collect_decision(k - 1);
            __syncthreads();
        }
        __syncthreads();
        const int4 ctl = sh.ctl[it];
        // nothing but the next iteration to do: one test, every warp waits for it
        const bool plain = words && !last && !tracing && !empty && (ctl.x | ctl.z | ctl.w) == 0 && (k == 1 || ctl.y);
        if (plain) continue;
        empty = ctl.w != 0;  // perhaps, behind V^{k+1}
        if (ctl.x) {
            ok = give_up(k);
            break;
        }
        if (!last && words && ctl.z) {
            // uniform over the grid: every block has read the same words
            words = false;
            __syncthreads();
            if (warp < C) exchange_sums(std::integral_constant<int, X_SUMS>(), warp, cur, nxt);
            ++nx;
            __syncthreads();
            if (sh.ctl[it].x) {
                ok = give_up(k);
                break;
            }
        } else if (!last && !words) {
            words = fixed && !ctl.z;
        }
        if (!last && !rebase(cur, nxt)) {
            ok = give_up(k);
            break;
        }
        // Iteration k - 1's full pass when its sample could not decide, iteration
        // k's when it is the last (and every one for a trace).
        const int from = (k > 1 && !ctl.y && !tracing) ? k - 1 : k, to = (last || tracing) ? k : k - 1;
#pragma unroll 1
        for (int r = from; ok && r <= to; ++r) {
            if (!full_pass(r)) {
                ok = give_up(r);
            } else if (sh.delta < eps || r == max_iter) {
                status = sh.delta < eps ? FCM_OK : FCM_NOT_CONVERGED;
                iters = r;
                ok = false;
            } else if (r < k && threadIdx.x == 0 && sh.empty[cur]) {
                flags |= FCM_FLAG_EMPTY_CLUSTER;
            }
        }
        if (from == k && k > 1 && threadIdx.x == 0 && sh.empty[cur]) flags |= FCM_FLAG_EMPTY_CLUSTER;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            st->V[j] = sh.v[iters & 3][j];
            if (ra.Vout) ra.Vout[j] = sh.v[iters & 3][j];
            st->V64[j] = df_to_double(sh.v64[iters & 3][j]);
        }
        st->status = status;
        st->iters = iters;
        st->flags = flags;
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
