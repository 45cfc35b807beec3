// footprint.h -- device bytes of a served job: what it holds once built, and a
// bound on what it holds at any time, from its sizes alone (admission).
//
// Compiles for the host alone, so the CPU tests count the bytes of the worst
// windows against the bound.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "window.cuh"

namespace sls {

// What the two coordinate arrays and the statistics take: held at all times.
inline size_t base_bytes(int64_t n, size_t stats_bytes) { return 32 * (size_t)n + stats_bytes; }

// Device bytes a job holds once built: coordinates, node offsets, adjacency
// words, the window stream, the numbering map, statistics.
inline size_t built_footprint(int64_t n, uint64_t adj_words, size_t stream_bytes, size_t stats_bytes)
{
    return base_bytes(n, stats_bytes) + 4 * (size_t)(n + 1) + 4 * (size_t)adj_words + stream_bytes + 4 * (size_t)n;
}

// A bound on the window stream (window.cuh): every subtile with rings of the
// longest kind and lists of 16 bits, windows of whichever width takes more (64
// nodes fill two of a window's four subtiles; the others have a meta row), and
// every neighbour (at most six a triangle) in a halo, whose ids fill whole rows.
inline size_t window_stream_bound(int64_t n, int64_t m)
{
    const size_t row = 128, header = 4 * win::kHeaderWords;
    const size_t sub = win::subtile_rows(win::kRingMax, win::kRingMax, 16);
    const size_t w128 = row * (4 * sub + win::kColdRows + 1) + header;
    const size_t w64 = row * (2 * sub + 2 + win::kColdRows + 1) + header;
    return std::max(w128 * ((size_t)n / 128 + 1), w64 * ((size_t)n / 64 + 1)) + 24 * (size_t)m;
}

// A bound on the adjacency words: records at fixed places (2 a node and 6 a
// triangle), or of exact lengths (a meta word per node; per corner of a triangle
// at most two neighbours and one triangle code).
inline uint64_t adjacency_bound(int64_t n, int64_t m)
{
    return (uint64_t)std::max(2 * n + 6 * m, n + 9 * m);
}

// A bound on what a job holds at any time: the largest of what stands during
// the spatial numbering (cell counts and offsets, both maps, a copy of the
// coordinates), during the adjacency build (both maps, incidences, counts and
// flags, the records; their neighbour scratch when they have exact lengths) and
// with the window stream.  Each step's scratch is freed in stream order before
// the next one's is taken.
inline size_t admission_bound(int64_t n, int64_t m, size_t stats_bytes)
{
    const size_t N = (size_t)n, M = (size_t)m, base = base_bytes(n, stats_bytes);
    const size_t numbering = base + 12 * M + 56 * N;
    const size_t records = base + (12 + 12 + 24) * M + (8 + 8 + 1 + 4 + 9) * N + 4 * (size_t)adjacency_bound(n, m);
    const size_t built = built_footprint(n, adjacency_bound(n, m), window_stream_bound(n, m), stats_bytes);
    return std::max(std::max(numbering, records), built) + 65536;
}

}  // namespace sls
