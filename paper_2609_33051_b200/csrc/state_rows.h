// Which rows of a dense head's state a warp of the decode kernel reads, and which it asks into L2 before it does.  Plain host
// constants (no CUDA), so that a test can walk them.
#pragma once

#ifndef SKETCHSSM_BOTH
#ifdef __CUDACC__
#define SKETCHSSM_BOTH __host__ __device__
#else
#define SKETCHSSM_BOTH
#endif
#endif

namespace sketchssm {

// W warps share the K rows of a head, K / W each; warp `sub` owns rows first_row .. end_row - 1.
SKETCHSSM_BOTH constexpr int first_row(int K, int W, int sub) { return sub * (K / W); }
SKETCHSSM_BOTH constexpr int end_row(int K, int W, int sub) { return (sub + 1) * (K / W); }

// Rows asked for ahead of the ones that are read: this many, of the warp's own.  (K = 64 shared by four warps: 16 rows each.)
constexpr int kAhead = 32;
SKETCHSSM_BOTH constexpr int rows_asked_first(int K, int W) { return kAhead < K / W ? kAhead : K / W; }
// While rows i0 .. are read, those kAhead further on are asked for, if they are this warp's.
SKETCHSSM_BOTH constexpr bool asks_ahead(int K, int W, int sub, int i0) { return i0 + kAhead < end_row(K, W, sub); }

}  // namespace sketchssm
