// Host-side declarations of the binary64 tensor-core kernel for short inner
// dimensions (tsm2_f64s.cu).
#pragma once

#include "internal.h"
#include "shift.h"

namespace tsm2 {

constexpr int kF64SMaxK = 32;  // inner indices

struct F64SLaunch {
    int64_t M, N;        // C(M x N) [+]= A(M x K) B(K x N)
    int K;               // <= kF64SMaxK
    ColumnClasses a;     // A: map[0] alone, dims {M, K}, box {f64s_tile(), f64s_step()}, or split: column classes, box rows f64s_tile()
    bool split;          // (not with accumulate)
    const double *A;
    int64_t lda;
    const double *B;     // element (j, c) at B[j bes + c bcs]
    int64_t bes, bcs;
    double *C;
    int64_t ldc;
    bool accumulate;
    void *digits;        // f64s_digit_bytes(N, K), 256-byte aligned
    unsigned *status;
    int64_t wait_ns;
    int blocks;          // thread blocks at most
    unsigned long long *trace;  // optional per-block timestamps for grids of at most trace_blocks
    int64_t trace_blocks;
};
int f64s_tile();            // rows of a box
int f64s_rows(bool split);  // rows of a tile
int f64s_cols();  // columns of a group
int f64s_step();
size_t f64s_digit_bytes(int64_t N, int K);
cudaError_t f64s_launch(const F64SLaunch &L, cudaStream_t stream);

}  // namespace tsm2
