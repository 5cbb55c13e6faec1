// The ring of K blocks of the fused-epilogue GEMM (layer_tc.cu): how many stages it has, and which
// gather warp writes which block.  Plain C++, so that a test can take the rule from here.
#pragma once

#ifdef __CUDACC__
#define LT_HD __host__ __device__
#else
#define LT_HD
#endif

namespace bcrown {
namespace lt {

// Stages of one K block (A: 128 x 64, B: Np x 64, BF16), as many as fit in shared memory beside the
// epilogue warps' lists (layer_tc.cu asserts that they do); at most 5 by TMA and one per gather warp.
constexpr int NS_MAX = 5, NS_GATHER = 4;
LT_HD constexpr int lt_stages(bool ta, int Np) {
  return ta ? (Np > 128 ? 3 : Np <= 64 ? 5 : 4) : (Np > 208 ? 3 : NS_GATHER);
}

// K block s of a CTA's (tile, K block) order lies in stage s % stages, and one gather warp owns each
// stage; with fewer stages than warps the others gather nothing.  A barrier's phase is told by one
// parity bit, so a warp may only wait for a stage whose previous block it has written itself: a warp
// that took the blocks of several stages in turn could come to one two rounds ahead, where the
// wait's parity is that of a round that has passed.
LT_HD constexpr int lt_gather_warp(int stage) { return stage; }

}  // namespace lt
}  // namespace bcrown
