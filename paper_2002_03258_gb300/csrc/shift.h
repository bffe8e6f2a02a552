// Host-side declarations of the unaligned-operand kernel (tsm2_shift.cu).
#pragma once

#include "internal.h"

namespace tsm2 {

// Column classes of A for the bulk copies: columns j = q P + r (P = 16 / elem)
// of an A with any leading dimension have a stride of P lda elements, a
// multiple of 16 bytes, from a start that is rounded down to one.
struct ColumnClasses {
    CUtensorMap map[4];  // [r]: dims {m + shift[r], columns of the class}, box {256, 16 / P}
    int shift[4];        // elements by which the rows lie behind the rounded start
    int cols[4];         // columns of the class (0: none, map[r] is map[0])
};

struct ShiftLaunch {
    GemmArgs g;  // k <= shift_kc(elem, k)
    ColumnClasses a;
    int splits;      // shift_splits
    void *slots;     // shift_slot_bytes
    int *counters;   // one per row block, zero between launches (splits > 1)
    unsigned *status;
    int64_t wait_ns;
    int grid;
};
struct ShiftShape {
    const char *name;
    int elem, KC, R;
    int rows;  // rows per row block
    size_t slot;
};
constexpr int kShiftStep = 16;  // inner columns per pipeline stage
const ShiftShape *shift_shape(int elem, int kc, bool tall);
// Ranges that the inner dimension (upr stages) of every row block is cut into.
int shift_splits(const ShiftShape *shape, int64_t num_rb, int64_t upr, int blocks);
size_t shift_slot_bytes(const ShiftShape *shape, int64_t num_rb, int splits);
cudaError_t shift_launch(const ShiftShape *shape, const ShiftLaunch &L, cudaStream_t stream);

}  // namespace tsm2
