// Host/device shared definitions of the single-image FCM path.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fcm.h"

namespace fcm {

constexpr int NT = 256;                                  // threads per block of the pass
constexpr int NWARP = NT / 32;
constexpr int WARP_TILE = 128;                           // pixels per warp tile of the TMA kernels
constexpr int SLOTS_MAX = 2 * FCM_MAX_CLUSTERS + 4;      // num[C], den[C], J, delta, 2 flags
constexpr int STATUS_RUNNING = 2;

// Bounds of the device-side waits of one run, set per handle from the host
// (fcm_set_limits). Every spin or suspension loop counts against one of them
// and, when it runs out, the kernel records FCM_ERR_TIMEOUT and returns.
struct WaitLimits {
    uint32_t grid_spins;  // polls, a fraction of a microsecond apart, of a grid-wide wait
    uint32_t tma_polls;   // suspensions, up to about 1 ms each, of a wait for TMA bytes
    uint32_t phantoms;    // arrivals every grid-wide barrier waits for beyond the
                          // grid's own: 0 in normal use; a test sets 1 to make
                          // every barrier give up (fault injection on the host side)
    uint32_t pad;
};
constexpr uint32_t DEFAULT_GRID_SPINS = 1u << 23;  // a few seconds
constexpr uint32_t DEFAULT_TMA_POLLS = 2048;       // about 2 s

// Which half-step a launch of the pass performs.
enum Pass : int {
    P_ACCUM0 = 0,  // V^1 from a given U^0 (Eq. 3); validates x and U^0
    P_INITV = 1,   // U^0 = membership(V^0) (Eq. 4), written to U; V^1 from it
    P_ITER = 2,    // U^k from V^k in place, delta_k, J_k, V^{k+1} (Eqs. 4, 1, 3)
    P_COUNT = 3
};

// Device-resident state of one run. The host writes the whole struct before a
// run; the passes read their inputs from it and the last block of each pass
// writes the evolving part. Kernels and graphs therefore never need new
// parameters when the caller's buffers change.
struct alignas(128) RunState {
    // per-run inputs
    const float* x;
    const float* Uprev;  // U^{k-1}: the caller's U^0 for the first pass, then U
    float* U;            // U^k, written in place
    double* trace;   // nullable: (max_iter) rows of (delta, J, V^k[C])
    int64_t n;
    float m;
    float inv_m1;    // 1 / (m - 1)
    float eps;
    int max_iter;
    int C;
    int pad0;
    float V0[FCM_MAX_CLUSTERS];
    // evolving
    float V[FCM_MAX_CLUSTERS];      // V^k used by the next pass
    double V64[FCM_MAX_CLUSTERS];   // the FP64 quotients V rounds
    double delta;
    double J;
    int k;          // index of the next iteration
    int status;
    int done;
    int flags;
    int iters;
    unsigned int ticket;  // last-block-done counter of the current pass
    int launches;         // passes started in this run (loop guard)
    WaitLimits lim;
    unsigned int bounds;  // FCM_FLAG_BOUNDS from a FCM_DEBUG_BOUNDS build's guards
};

typedef void (*PassFn)(RunState*, double*, cudaGraphConditionalHandle, int);

// Kernel table: [C][m kind][pass][variant], variant 0 = grid-stride scalar
// loads (any n), 1 = TMA ring (n % 4 == 0, 16-byte aligned rows); smem holds
// each kernel's dynamic shared memory in bytes.
struct SingleTable {
    PassFn k[FCM_MAX_CLUSTERS + 1][4][P_COUNT][2];
    int smem[FCM_MAX_CLUSTERS + 1][4][P_COUNT][2];
};

void register_single_c1(SingleTable&);
void register_single_c2(SingleTable&);
void register_single_c3(SingleTable&);
void register_single_c4(SingleTable&);
void register_single_c5(SingleTable&);
void register_single_c6(SingleTable&);
void register_single_c7(SingleTable&);
void register_single_c8(SingleTable&);

}  // namespace fcm
