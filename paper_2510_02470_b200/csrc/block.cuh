// Shared by the two tensor-core kernels that read a block's planes.
#pragma once
#include "sage_internal.h"
#include "tc05.cuh"

namespace sage {
namespace tc {
// The three places of BlockMap as boxes of 32 rows x 128 bytes (128-byte swizzle).
bool block_tmaps(const BlockSource& src, const BlockMap& map, int64_t D, CUtensorMap* tmS, CUtensorMap* tmR, CUtensorMap* tmI);
// Where the 32 planes from p on (a multiple of 32) come from: 0 S, 1 R, 2 in place, and the row there (past the end: none, read as zeros).
struct BlockBox {
    int place, row;
};
__device__ __forceinline__ BlockBox block_box(const BlockMap& m, int p) {
    const int place = p < m.oR ? 0 : p < m.oI ? 1 : 2;
    return {place, p >= m.P ? 1 << 20 : place == 0 ? p : place == 1 ? p - m.oR : p - m.oI};
}
}  // namespace tc
}  // namespace sage
