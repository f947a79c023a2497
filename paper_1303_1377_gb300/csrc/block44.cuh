// Index arithmetic of 4^4 blocks, shared by the Dslash and the SAP kernels.
#pragma once

#include "common.cuh"

namespace ddamg {

// ---------------------------------------------------------------------------
// 4^4 blocks.  Local order of a block (common.cuh): parity p (even first), then rank = lex >> 1
// among the sites of that parity, lex = ((y0 * 4 + y1) * 4 + y2) * 4 + y3.  Neighbours follow from
// the in-block lexicographic index and the (warp-uniform) neighbouring blocks, with no table load
// per site.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int lex44_of_local(int l) {
    const int p = l >> 7, k = l & 127, row = k >> 1;  // row = y0 * 16 + y1 * 4 + y2
    const int q = __popc(row & 0x15) & 1;             // parity of y0 + y1 + y2
    return 4 * row + ((p ^ q) & 1) + 2 * (k & 1);     // y3 = (p - q) mod 2 + 2 (k mod 2)
}
// global index of the neighbour of local site (lex L, parity p) of block c in direction MU,
// forward or backward; bn = the neighbouring block in that direction
template <int MU, bool FWD>
__device__ __forceinline__ int nbr44(int L, int p, int c, int bn) {
    constexpr int SH = 2 * (3 - MU), S = 1 << SH;
    const int y = (L >> SH) & 3;
    const bool cross = FWD ? y == 3 : y == 0;
    const int L2 = FWD ? (cross ? L - 3 * S : L + S) : (cross ? L + 3 * S : L - S);
    return (cross ? bn : c) * 256 + (((p ^ 1) << 7) | (L2 >> 1));
}

}  // namespace ddamg
