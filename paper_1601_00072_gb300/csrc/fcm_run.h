// Kernel table of the whole-run kernel (fcm_run_inst.cu, compiled once per
// cluster count) and its exchange slots.
#pragma once

#include "fcm_internal.h"

namespace fcm {

// Threads per block of the whole-run kernel (one block per SM): pt pixel
// threads, then one control warp. At most 15 pixel warps at C <= 5 (128
// registers each; a 17th warp would leave 96) and 11 above (168 registers).
constexpr int run_max_pt(int C) { return C <= 5 ? 480 : 352; }
constexpr int RUN_MAX_PW = 15;
// The fewest pixel threads of a block, where an image is too small to give every
// SM's threads a quad: more blocks with fewer warps to meet at each barrier (40,000
// pixels at C = 4, m = 2: 1.92 us per iteration with 128 threads, 2.23 with 480).
constexpr int RUN_FEW_PT = 128;
// Dynamic shared memory: the second set of the sums (2 C pairs per pixel
// thread), then `resident` quads of x per pixel thread.
constexpr int run_smem(int C, int pt, int resident) { return pt * 16 * (C + resident); }
constexpr int RUN_SMEM_MAX = 222 * 1024;
constexpr int run_max_resident(int C, int pt) { return RUN_SMEM_MAX / (pt * 16) - C; }

// One 16-byte exchange slot: two values and the 64-bit tag of the exchange
// they belong to, written and read as a unit.
constexpr int RUN_SLOT_BYTES = 16;
// Slots of one exchange per block: (num_j, den_j) of each cluster, then the
// maximum and the flags; two exchanges are live at a time.
constexpr int run_slots(int C) { return 2 * (C + 1); }

// The scratch of the exchanges: the words of two banks (runs alternate), each
// [parity][cluster or control], a 128-byte line each; then the slots.
constexpr int RUN_WORD_BYTES = 128;
constexpr int RUN_WORDS_BYTES = 2 * 2 * (FCM_MAX_CLUSTERS + 1) * RUN_WORD_BYTES;
constexpr int RUN_MAX_BLOCKS = 255;  // a word's top byte counts them
constexpr size_t run_scratch_bytes(int blocks) {
    return RUN_WORDS_BYTES + (size_t)RUN_SLOT_BYTES * run_slots(FCM_MAX_CLUSTERS) * blocks;
}

// Arguments of one whole run, by value: a run is one launch, with no upload
// before it. Its results (V, V64, delta, J, iters, status, flags of RunState) go
// straight to `out`, pinned host memory or device memory, and V to Vout too.
struct RunArgs {
    const float* x;
    const float* U0;   // the initial memberships (from_u); may equal U
    float* U;
    const float* Vin;  // nullable: initial centers in device memory (else V0)
    float* Vout;       // nullable: device memory
    double* trace;     // nullable
    RunState* out;
    char* scratch;
    int64_t n;
    float m, inv_m1, eps;
    int max_iter;
    int from_u;        // 1 from U^0, 0 from V^0
    int resident;      // quads of x per pixel thread kept in shared memory
    int max_blocks;    // blocks that the scratch has room for
    int64_t guard_n;   // n, or fewer: what a FCM_DEBUG_BOUNDS build's guards take for n (run_guard_n)
    unsigned nonce;    // the run's number on its scratch, counting up by one from run to run
    WaitLimits lim;
    float V0[FCM_MAX_CLUSTERS];
};
typedef void (*WholeRunFn)(RunArgs);

struct RunTable {
    WholeRunFn run[FCM_MAX_CLUSTERS + 1][4];
};

void register_run_c1(RunTable&);
void register_run_c2(RunTable&);
void register_run_c3(RunTable&);
void register_run_c4(RunTable&);
void register_run_c5(RunTable&);
void register_run_c6(RunTable&);
void register_run_c7(RunTable&);
void register_run_c8(RunTable&);

// The kernel table, filled on first use.
const RunTable& run_table();

// Raises the kernel's dynamic shared memory limit; whether it can be launched.
bool run_kernel_fits(const void* kernel, int C);

// Launch shape of a run of n pixels when at most max_blocks blocks are
// co-resident (0 blocks: none): blocks, threads per block, quads of x per pixel
// thread kept in shared memory, and the dynamic shared memory that takes.
struct RunShape {
    int blocks, threads, resident, smem;
};
RunShape run_shape(int64_t n, int C, int64_t max_blocks);

// n; in a FCM_DEBUG_BOUNDS build FCM_DEBUG_BOUNDS_SHORT in the environment takes
// that many pixels off, so that a test can see the guards at work: they then skip
// accesses that are in bounds, and report them.
int64_t run_guard_n(int64_t n);

}  // namespace fcm
