// Which Pauli strings share a tile pass (host only).
#pragma once

#include <cstdint>
#include <vector>

namespace svg {

// Strings of one x mask that stay together: order[pos .. pos + m) of the strings sorted by x mask.
struct EvRun {
    int pos, m;
};
// A pass over tiles of 2^qubits amplitudes with the local qubits `lam` (qubits 0-4 among them).
struct EvTilePass {
    uint64_t lam = 31;
    std::vector<EvRun> runs;
};
struct EvTileLimits {
    int qubits, strings, groups;   // of a tile pass; a run makes up to two groups
    int passes;                    // passes of the one-mask kernel that a tile pass has to replace
    int per_pass;                  // strings of one x mask that the one-mask kernel takes
};

// First fit in run order: the tile passes, and in `left` the runs for the one-mask kernel.  x[r] is run
// r's x mask.  A pass ends its scan when it is full, and runs that fit no tile are set aside before
// the first: the scans of 50,000 runs take 0.1 s or less.
inline void plan_tiles(const std::vector<EvRun> &runs, const std::vector<uint64_t> &x, int n, const EvTileLimits &lim,
                       std::vector<EvTilePass> *tiles, std::vector<EvRun> *left)
{
    tiles->clear();
    left->clear();
    // the runs left, as a list: next[r] is the run after r - 1 (next[0] the first)
    std::vector<int> next(runs.size() + 1, -1);
    int tail = 0;
    for (size_t r = 0; r < runs.size(); ++r) {
        if (__builtin_popcountll(x[r] | 31u) > lim.qubits || runs[r].m > lim.strings) {
            left->push_back(runs[r]);
        } else {
            next[(size_t)tail] = (int)r;
            tail = (int)r + 1;
        }
    }
    while (next[0] >= 0) {
        EvTilePass t;
        int strings = 0, passes = 0;
        for (int prev = 0; next[(size_t)prev] >= 0;) {
            const int r = next[(size_t)prev];
            const uint64_t with = t.lam | x[(size_t)r];
            if (__builtin_popcountll(with) > lim.qubits || strings + runs[(size_t)r].m > lim.strings) {
                prev = r + 1;
                continue;
            }
            t.lam = with;
            strings += runs[(size_t)r].m;
            passes += (runs[(size_t)r].m + lim.per_pass - 1) / lim.per_pass;
            t.runs.push_back(runs[(size_t)r]);
            next[(size_t)prev] = next[(size_t)r + 1];
            if (strings == lim.strings || 2 * (int)(t.runs.size() + 1) > lim.groups) break;
        }
        if (passes < lim.passes) {
            left->insert(left->end(), t.runs.begin(), t.runs.end());
            continue;
        }
        for (int q = 5; q < n && __builtin_popcountll(t.lam) < lim.qubits; ++q) t.lam |= uint64_t(1) << q;   // whole tiles
        tiles->push_back(std::move(t));
    }
}

}  // namespace svg
