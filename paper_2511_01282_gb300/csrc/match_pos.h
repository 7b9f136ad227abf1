// match_pos.h -- the numbers of the retrieval kernels' candidates, for buffers of
// up to 2^31 - 1 tokens (positions are int32).  Rows hold 128 candidates, and the
// last row's numbers pass 2^31.  Plain C++, so that the edges can be checked on the
// host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define RS_HD __host__ __device__ __forceinline__
#else
#define RS_HD inline
#endif

namespace rs {

constexpr long long kMatMaxTokens = 0x7fffffff;

constexpr int kMatCluster = 8;        // the portable cluster size
constexpr int kMatClusterMax = 16;

// CTAs of a request's cluster in a call over B requests; few: the kernel's own
// limit for clusters of 16; wide: how many of these the context can run at once
// (more would run in turn).
RS_HD int match_cluster(int B, int few, int wide) { return B <= few && B <= wide ? kMatClusterMax : kMatCluster; }

// A scan's candidates: the buffer's positions, as quads of four on 16-byte
// boundaries.  t: tokens, al: positions that the buffer begins past a boundary.
// Unsigned: a position in front of the buffer wraps to a number past every buffer,
// and one comparison tests both ends.
struct ScanPos {
    uint32_t t, al;
    RS_HD uint32_t rows() const { return (t + al + 126u) / 128u; }  // the last holds position t - 2
    RS_HD uint32_t quad(int row, int lane) const { return 128u * (uint32_t)row + 4u * (uint32_t)lane - al; }
    RS_HD bool whole(uint32_t p0) const { return p0 < (t > 3u ? t - 3u : 0u); }  // positions p0 .. p0 + 3
    RS_HD bool in(uint32_t p) const { return p < t; }
    // whether a match of k tokens can end at p: k - 1 <= p <= t - 2 (1 <= k <= t)
    RS_HD bool end(uint32_t p, int k) const { return p - (uint32_t)(k - 1) < t - (uint32_t)k; }
};

// A query's n candidates: element e of lane l in row r is number 128 r + 32 e + l.
// A row's first number is one of them; those behind it are counted from there, so
// that a number is only formed where it is in range.
struct ListPos {
    int n;
    RS_HD int rows() const { return (int)(((uint32_t)n + 127u) / 128u); }
    RS_HD bool in(int row, int o) const { return o < n - 128 * row; }  // number 128 row + o; row < rows()
    RS_HD static int number(int row, int o) { return 128 * row + o; }
};

}  // namespace rs
