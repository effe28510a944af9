// Kernel table of the whole-run kernel (fcm_run_inst.cu, compiled once per
// cluster count) and its exchange slots.
#pragma once

#include "fcm_internal.h"

namespace fcm {

constexpr int RUN_NT = 512;  // threads per block of the whole-run kernel, one block per SM
constexpr int RUN_NW = RUN_NT / 32;

// One 16-byte exchange slot: two values and the 64-bit tag of the exchange
// they belong to, written and read as a unit.
constexpr int RUN_SLOT_BYTES = 16;
// Slots of one exchange per block: (num_j, den_j) of each cluster, then the
// maximum and the flags; two exchanges are live at a time.
constexpr int run_slots(int C) { return 2 * (C + 1); }

typedef void (*WholeRunFn)(RunState*, void* slots, unsigned nonce);

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

// Grid of a run of n pixels when at most max_blocks blocks are co-resident.
int run_grid(int64_t n, int64_t max_blocks);

}  // namespace fcm
