// sequence_rows.h -- which row of the inputs of a sequence a warp of its
// preparing kernel copies (sequence.cu).  Plain C++, so that the arithmetic can
// be run on the host.
#pragma once

#include <cstdint>

#if defined(__CUDACC__)
#define DARB_HOST_DEVICE __host__ __device__
#else
#define DARB_HOST_DEVICE
#endif

namespace darb {
namespace seq {

// Rows [0, H) are those of h0; the rest, I for each step, those of x.
struct PrepRow {
    bool of_x;
    int64_t t, k;   // step (0 for h0) and row
};

DARB_HOST_DEVICE inline PrepRow prep_row(int64_t row, int64_t H, int64_t I) {
    if (row < H) return {false, 0, row};   // before any division: without x (I = 0) these are all rows
    return {true, (row - H) / I, (row - H) % I};
}

}  // namespace seq
}  // namespace darb
