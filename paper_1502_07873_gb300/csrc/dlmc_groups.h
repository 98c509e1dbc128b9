// The groups of outer samples that the double loop's screening holds distances of (host code).
#pragma once
#include <algorithm>
#include <cstddef>

namespace oed {

constexpr int kScreenRows = 64;                     // outer samples of a tile of k_screen
constexpr size_t kScreenFloats = (size_t)1 << 25;   // distances held at once (128 MB), if a tile's rows allow
constexpr int kScreenTiles = 65535;                 // tiles of a group: the second dimension of k_screen's grid

// Rows of a group: N rows at most, whole tiles, between one tile and what a grid takes.  Up to seven
// inner samples, kScreenFloats distances alone would allow more tiles than that.
inline int dlmc_group_rows(int N, int M)
{
    const size_t tiles = kScreenFloats / M / kScreenRows;
    return (int)std::min((size_t)N, std::clamp(tiles, (size_t)1, (size_t)kScreenTiles) * kScreenRows);
}

// f(n0, n1) for every group of rows n0 .. n1 - 1 (counted in 64 bits: the end of the last group may
// lie above the largest int)
template <typename F>
inline void dlmc_for_groups(int N, int M, F f)
{
    const int rows = dlmc_group_rows(N, M);
    for (long long n0 = 0; n0 < N; n0 += rows) f((int)n0, (int)std::min((long long)N, n0 + rows));
}

}  // namespace oed
