// How many tiles of a batch or a serving step run at once.
#pragma once

#include <algorithm>
#include <cstdint>

namespace ahpp {

// Of n_tiles, with at most `most` groups of blocks: the configured number
// (0: left to this rule), never more than there are tiles, whose blocks would
// idle.  By the rule, tiles that run at once share L2: their gathered tables (of
// `table` bytes each) stay within its size (100k nodes, 20 MB a tile: 106 us a tile
// and round one at a time, 91 with two, 84 with four; 300k nodes, 60 MB: 270 with
// one or two).  A serving step takes the configured number as a cap only: it is
// about batches, and eight tiles at once on a graph whose tables L2 does not hold
// would slow every request down.
inline uint32_t groups_of(uint32_t configured, uint32_t n_tiles, uint32_t most, uint64_t table, bool serving) {
  most = std::max<uint32_t>(1, std::min(most, n_tiles));
  if (configured && !serving) return std::min(configured, most);
  if (configured) most = std::min(most, configured);
  const uint64_t fit = std::max<uint64_t>(1, (128ull << 20) / std::max<uint64_t>(table, 1));
  const uint32_t at_once = (uint32_t)std::min<uint64_t>(most, fit);
  const uint32_t waves = (std::max(n_tiles, 1u) + at_once - 1) / at_once;
  return (std::max(n_tiles, 1u) + waves - 1) / waves;    // the same number of waves, evenly
}

}  // namespace ahpp
