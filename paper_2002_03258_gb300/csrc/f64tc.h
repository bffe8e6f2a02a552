// Host-side declarations of the binary64 tensor-core kernel (tsm2_f64tc.cu).
#pragma once

#include "internal.h"
#include "shift.h"

namespace tsm2 {

struct F64TCLaunch {
    GemmArgs g;          // k <= f64tc_kc()
    bool split;          // A with any alignment, through two column classes
    ColumnClasses a;     // otherwise map[0] alone: dims {m, n}, box {f64tc_rows(false), f64tc_step()}
    void *digits;        // f64tc_digit_bytes(n), 256-byte aligned
    void *slots;         // f64tc_slot_bytes(grid), 256-byte aligned
    int *counters;       // eight per row block, zero between launches
    unsigned *status;
    int64_t wait_ns;
    int grid;
    unsigned long long *trace;  // optional per-block timestamps (nullptr: off)
};
int f64tc_rows(bool split);  // rows per row block
int f64tc_step();  // inner columns per pipeline stage
int f64tc_kc();    // C columns per pass
size_t f64tc_digit_bytes(int64_t n);
size_t f64tc_slot_bytes(int64_t grid);
cudaError_t f64tc_launch(const F64TCLaunch &L, cudaStream_t stream);

}  // namespace tsm2
