// Shared by the two tensor-core kernels that read a block's planes.
#pragma once
#include "sage_internal.h"
#include "tc05.cuh"

namespace sage {
namespace tc {
// The three places of BlockMap.
struct Place {
    const void* base;
    int64_t ld;
    int rows;                      // planes
};
inline Place place_of(const BlockSource& src, const BlockMap& m, int i) {
    if (i == 0) return {src.S, src.pitch, 3 * m.s_rows};
    if (i == 1 || m.n_in == 0) return {src.R, src.pitch, i == 1 ? m.np * m.n_store : 0};
    return {src.in_place, src.ld_in, m.n_in};
}
// Where plane p (a multiple of 32) of the block is, and which plane of that place; past the block's end one that no place has.
__device__ __forceinline__ int block_place(const BlockMap& m, int p) { return p < m.oR ? 0 : p < m.oI ? 1 : 2; }
__device__ __forceinline__ int block_place_row(const BlockMap& m, int p, int place) {
    return p >= m.P ? 1 << 20 : place == 0 ? p : place == 1 ? p - m.oR : p - m.oI;
}
}  // namespace tc
}  // namespace sage
