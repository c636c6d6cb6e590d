// Runs of consecutive chains that one launch of the dense-tile label kernel
// takes.  A block lists its chains (jobs, 16 bytes each) at the start of its
// shared memory: the run's tiles are dealt to the blocks in turn and a job has a
// tile at least, so a block lists at most min(chains, ceil(tiles / blocks)) of
// them.  A run ends where that would pass max_jobs; the tiles of a chain are
// labelled independently, so the split changes no result.  Plain C++: the same
// code builds for the host alone (tests).
#pragma once
#include <stdint.h>

#include <algorithm>
#include <vector>

// Most jobs of a block: 8 KB of its 227 KB, beside stages and segments of every K
// (a run is cut only in batches of more than 512 chains with more than 512 tiles
// a block).
constexpr int32_t kMaxTileJobs = 512;

// tiles[b]: tiles of chain b (0: not on the dense-tile engine).  Returns the first
// chain of each run and, last, the number of chains.
inline std::vector<int32_t> tile_runs(const std::vector<int32_t>& tiles, int32_t blocks,
                                      int32_t max_jobs) {
    std::vector<int32_t> starts(1, 0);
    int64_t chains = 0, sum = 0;
    for (int32_t b = 0; b < (int32_t)tiles.size(); ++b) {
        if (!tiles[b]) continue;
        const int64_t c = chains + 1, s = sum + tiles[b];
        if (std::min(c, (s + blocks - 1) / blocks) > max_jobs) {
            starts.push_back(b);
            chains = 1;
            sum = tiles[b];
        } else {
            chains = c;
            sum = s;
        }
    }
    starts.push_back((int32_t)tiles.size());
    return starts;
}
