// list_scratch.cuh -- how much scratch list building takes (lists.cu), plain C++
// so that it can be checked without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace idtx {

constexpr int64_t kScratchTile = 128;  // queries of a tile: chunks are whole tiles
constexpr size_t kListEntry = 8, kListMeta = 16;  // an entry (int2) and a query's meta (int4)

// Scratch entries per query of a list of `cap`: room for the 1.15 capacities
// that its radius is chosen for and their spread, or every sample.  Not smaller
// for a larger capacity, so that scratch for some capacities does for any
// smaller ones.
inline int buf_of(int cap, int64_t n)
{
    const int64_t all = (n + 31) / 32 * 32;
    const int64_t want = cap >= 2048 ? cap + cap / 2 : std::min(2 * cap, 3072);
    return (int)std::max<int64_t>(64, std::min<int64_t>(want, all));
}

inline size_t query_scratch(int64_t n, int cap_a, int cap_b)
{
    return ((size_t)buf_of(cap_a, n) + buf_of(cap_b, n)) * kListEntry + kListMeta;
}

// Scratch of one chunk of queries: enough of them to fill the GPU several
// times over, without another list-sized buffer for large n.
constexpr size_t kScratchBudget = size_t(5) << 28;
constexpr int64_t kMinChunk = 4096;

inline int64_t chunk_of(int64_t n, int cap_a, int cap_b)
{
    const int64_t fit = (int64_t)(kScratchBudget / query_scratch(n, cap_a, cap_b));
    // whole tiles: warps share their home tile
    return std::min(n, std::max(kMinChunk, fit / kScratchTile * kScratchTile));
}

// Bytes of a chunk's entries of both lists and metas, and to align the metas.
inline size_t chunk_bytes(int64_t n, int cap_a, int cap_b)
{
    return (size_t)chunk_of(n, cap_a, cap_b) * query_scratch(n, cap_a, cap_b) + 16;
}

// Enough for these capacities and for any smaller ones (whose chunks may be
// larger).
inline size_t list_scratch_bytes(int64_t n, int cap_a, int cap_b)
{
    const size_t per = query_scratch(n, cap_a, cap_b);
    return std::min((size_t)n * per, std::max(kScratchBudget, (size_t)kMinChunk * per)) + 512;
}

}  // namespace idtx
