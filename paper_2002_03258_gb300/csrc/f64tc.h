// Host-side declarations of the binary64 tensor-core kernel (tsm2_f64tc.cu).
#pragma once

#include "internal.h"
#include "shift.h"

namespace tsm2 {

// How A(m x n) lies in memory: column-major with 16-byte rows, column-major
// with any alignment (two column classes), or row-major with 16-byte rows.
enum class F64TCMode { Plain, Split, Transposed };

struct F64TCLaunch {
    GemmArgs g;          // k <= f64tc_kc()
    F64TCMode mode;
    ColumnClasses a;     // Split; otherwise map[0] alone: Plain dims {m, n}, box {f64tc_rows(Plain), f64tc_step()},
                         // Transposed dims {n, m}, box {f64tc_step(), f64tc_rows(Transposed)}, 128-byte swizzle
    void *digits;        // f64tc_digit_bytes(n), 256-byte aligned
    void *slots;         // f64tc_slot_bytes(grid), 256-byte aligned
    void *fails;         // f64tc_fail_bytes(g.m, mode), 256-byte aligned
    unsigned *status;
    int64_t wait_ns;
    int grid;
    int blocks;          // multiprocessors to use
    unsigned long long *trace;  // optional per-block timestamps (nullptr: off)
};
int f64tc_rows(F64TCMode mode);  // rows per row block
int f64tc_step();  // inner columns per pipeline stage
int f64tc_kc();    // C columns per pass
size_t f64tc_digit_bytes(int64_t n);
size_t f64tc_slot_bytes(int64_t grid);
size_t f64tc_fail_bytes(int64_t m, F64TCMode mode);
cudaError_t f64tc_launch(const F64TCLaunch &L, cudaStream_t stream);
cudaError_t f64tc_add(int64_t m, int k, const double *X, double *C, int64_t ldc, cudaStream_t stream);  // C += X, X m x k

}  // namespace tsm2
