// How the staged H psi kernel's pieces are dealt out to the blocks that share a
// tile.  Host code, without CUDA.
#pragma once
#include <algorithm>
#include <cstdint>

namespace gocp {

// cut[0 .. K]: part q of K takes the pieces [cut[q], cut[q + 1]), about equal
// shares of the bytes off[0 .. P] (piece p: off[p] .. off[p + 1]) and at least
// one piece each (1 <= K <= P): a part without a piece would have no last piece
// to end at.  A piece of more than a share takes the room of the cuts that fall
// into it, so each cut lies at least one piece after the one before.
inline void tiled_cuts(const uint32_t* off, int P, int K, uint32_t* cut) {
  cut[0] = 0u;
  for (int q = 1; q < K; ++q) {
    const uint64_t want = (uint64_t)off[P] * (uint64_t)q / (uint64_t)K;
    const int p = (int)(std::lower_bound(off, off + P, want) - off);
    cut[q] = (uint32_t)std::min(std::max(p, (int)cut[q - 1] + 1), P - (K - q));
  }
  cut[K] = (uint32_t)P;
}

}  // namespace gocp
