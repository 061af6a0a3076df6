// Layout of the line-block ILU(0) coefficients (ilu_lines.cu builds them,
// ilu_sweep.cu applies them).
#pragma once
#include "common.cuh"

namespace msrsb {

constexpr int kLineNbr = 5;   // neighbour lines in other blocks
constexpr int kLineOff = 16;  // 3 per neighbour line, rounded up to whole groups
constexpr int kLineIn = 12;   // 2 + 3 per other line of the block, rounded up
template <typename T>
constexpr int kLineGroup = 16 / (int)sizeof(T);
template <typename T>
__host__ __device__ constexpr int line_groups(int values) {
    return (values + kLineGroup<T> - 1) / kLineGroup<T>;
}

}  // namespace msrsb
