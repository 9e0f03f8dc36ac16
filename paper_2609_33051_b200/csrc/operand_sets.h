// The two operand sets that the tiles of a flush take in turn, and the phases of the barriers that go with them.  Plain host
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

// Tile t of a CTA (counted from 0) fills set t & 1 for the (t >> 1)-th time; a barrier's phases alternate in parity.
SKETCHSSM_BOTH constexpr int set_of_tile(int t) { return t & 1; }
SKETCHSSM_BOTH constexpr unsigned parity_of_tile(int t) { return (unsigned)(t >> 1) & 1u; }
// After `tiles` fills, those that may still be on their way: the last one of each set, tiles first_unfinished .. tiles - 1.
SKETCHSSM_BOTH constexpr int first_unfinished(int tiles) { return tiles > 2 ? tiles - 2 : 0; }

}  // namespace sketchssm
