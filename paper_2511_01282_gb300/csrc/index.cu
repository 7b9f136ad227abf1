// index.cu -- an inverted index over the committed token buffers, kept up to
// date step by step, and the retrieval of Section 3.3 answered from it
// (rs_match_index_build, rs_match_index_append, rs_match_scan_indexed).  The
// two queries Algorithm 1 asks of its suffix automaton -- Contains(key) and
// RetrievePositions(key), key = the buffer's last k <= RS_MAX_L tokens -- are
// answered exactly from the ascending list of positions holding the key's
// last token: each is a candidate, verified against the other k - 1 key
// tokens.  Algorithm 1's Update (the step's committed tokens join the index)
// is rs_match_index_append.  A query touches O(occurrences of one token)
// instead of O(t); an append touches O(appended tokens).
//
// Layout of the index (per request b, sizes from rs_match_index_bytes):
//   first[b][0 .. V+1]  number of build-time tokens with an id below v (ids
//                       outside [0, V) count as id V, the last bucket;
//                       verification compares the real tokens), first[V + 1] =
//                       t_b.  Bucket v holds the ascending positions of id v:
//                       list slots start(v) .. start(v) + len[v) with
//                       start(v) = first[v] + first[v] / 4 + 2 v, so bucket v
//                       has room for at least count_v + count_v / 4 + 2
//                       entries (count_v: occurrences at build time) and no
//                       prefix over the rooms is needed;
//   len[b][0 .. V]      entries in each bucket;
//   list (per request, at base[b]): kOvf overflow slots, then the buckets.
//                       A position whose bucket is full goes to the overflow
//                       list (ascending; all of a token's overflow entries
//                       are newer than its bucket entries);
//   built[b]            positions 0 .. built[b] - 1 are in the index;
//                       later ones (tokens appended and not yet indexed, or
//                       left out when the overflow list was full) are tested
//                       one by one (a linear tail).
// base[b] = tok_off[b] + tok_off[b] / 4 + b (2 (V + 1) + kOvf) at build time:
// a bound that telescopes over the requests (start(V + 1) <= t_b + t_b / 4 +
// 2 (V + 1)).
//
// Build: the (request, bucket) keys of all tokens are sorted, with their
// positions, by a stable LSD radix sort over all requests at once (digits of
// at most 9 bits).  A pass is three kernels: the digit counts of every tile of
// keys, their offsets, and the stable scatter, which ranks a tile's keys with
// per-warp counters, orders the tile in shared memory and writes whole runs of
// equal digits.  No atomics on global memory: counting buckets with them made a
// text's most common tokens the bottleneck (270 of 700 us for 4 x 1M tokens).
// Keys of 10 to 18 bits (32K ids and 8 requests, 128K ids and two) take two
// passes, and the tiles of the second are cut where the first digit changes:
// the offsets at the first tile of a digit's keys are then where each bucket
// begins, so the second scatter writes the positions straight into the buckets
// and the bucket starts need no search.  Between its passes a key is 32 bits,
// its second digit over its position.  Other key lengths (and the shortest and
// longest buffers) sort in plain passes, find first[] by a binary search per
// bucket and move the sorted positions in one more pass.
// Append: one CTA per request takes the new positions in rounds of 256; each
// position's rank among the round's positions of its bucket gives its slot
// after the bucket's entries; full buckets spill to the overflow list in
// position order; if that is full too, indexing stops at the first such
// position (it and every later one stay in the linear tail, and the status
// word says so).
// Query: the candidates (the key's last token's bucket, the overflow list,
// then the tail) are tested by one cluster per request as match.cuh
// describes (70K candidates for a text's most common token: 79-120 us with one
// CTA, 7.5 so; a handful 4.1 to 4.9, the chain of reads; none 2.8).
#include <stddef.h>

#include <algorithm>

#include "match.cuh"

namespace rs {
namespace {

constexpr int kOvf = 4096;               // overflow slots per request
constexpr int kMaxDigitBits = 9;
constexpr int kMaxBins = 1 << kMaxDigitBits;
constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kAppThreads = 256;         // positions per append round

// Keys per tile: 4096, or 1024 for builds of at most kSmallBuild tokens, whose
// 4096-key tiles would leave most SMs idle (4 x 32K tokens: 32 tiles).
constexpr int kTileRounds = 16, kTileRoundsSmall = 4;
constexpr long long kSmallBuild = 1 << 19;
inline int tile_rounds(long long t_total) { return t_total <= kSmallBuild ? kTileRoundsSmall : kTileRounds; }
inline long long n_tiles(long long t_total) {
    const long long tile = (long long)tile_rounds(t_total) * kRadixThreads;
    return (t_total + tile - 1) / tile;
}

// bits of a sort key (request, bucket): buckets 0 .. V, requests 0 .. B - 1
inline int bits_for(long long n) {  // smallest b with n < 2^b
    int b = 0;
    while (b < 63 && (1ll << b) <= n) ++b;
    return b;
}
inline int key_bits(int B, int V) { return bits_for(V) + bits_for(B > 0 ? B - 1 : 0); }
// Whether the second pass's tiles are cut at the first digit (see above), with
// 32-bit keys between the passes.  Builds of a text so and in plain passes: 4 x 1M
// tokens 62.8 and 88.0 us, 4 x 200K 38.1 and 47.3, 8 x 60K 34.8 and 37.7, 4 x 32K
// 27.1 and 29.2.  Shorter ones are a few us of kernels between launches either
// way, and the counts of the cut tiles are a MB more of index.
constexpr long long kCutMin = 1 << 16;
inline int cut_lo_bits(int B, int V) { return (key_bits(B, V) + 1) / 2; }
inline int cut_pos_bits(long long t_total) { return bits_for(t_total - 1); }
inline bool cut_build(int B, int V, long long t_total) {
    const int bits = key_bits(B, V);
    return t_total >= kCutMin && bits > kMaxDigitBits && bits <= 2 * kMaxDigitBits &&
           bits - cut_lo_bits(B, V) + cut_pos_bits(t_total) <= 32;
}
// tiles of a pass, at most: with cuts, one more per digit and one past the end
inline long long hist_tiles(int B, int V, long long t_total) {
    return n_tiles(t_total) + (cut_build(B, V, t_total) ? kMaxBins + 1 : 0);
}

struct IndexView {
    int32_t *valid;         // 1 when the build's offsets were consistent (else the index holds nothing)
    int64_t *built, *base;  // per request: positions indexed, first list slot
    int32_t *ovf_n;         // per request: overflow entries
    int32_t *first;         // [B][V + 2]
    int32_t *len;           // [B][V + 1]
    int32_t *list;
    // build scratch
    uint2 *pair[2];         // (key, position) of every token
    int32_t *hist;          // [tiles][bins]
    int32_t *dtot;          // [2][kMaxBins]
};

inline long long list_slots(int B, int V, long long t_total) {
    return t_total + t_total / 4 + (long long)B * (2ll * (V + 1) + kOvf);
}

// Carves the index (and its build scratch) out of `base`; returns the bytes used.
inline size_t carve_index(void *base, int B, int V, long long t_total, IndexView *v) {
    Carve cv(base);
    v->valid = cv.take<int32_t>(1);
    v->built = cv.take<int64_t>((size_t)B);
    v->base = cv.take<int64_t>((size_t)B);
    v->ovf_n = cv.take<int32_t>((size_t)B);
    v->first = cv.take<int32_t>((size_t)B * (V + 2));
    v->len = cv.take<int32_t>((size_t)B * (V + 1));
    v->list = cv.take<int32_t>((size_t)list_slots(B, V, t_total));
    v->pair[0] = cv.take<uint2>((size_t)t_total);
    v->pair[1] = cv.take<uint2>((size_t)t_total);
    v->hist = cv.take<int32_t>((size_t)kMaxBins * hist_tiles(B, V, t_total));
    v->dtot = cv.take<int32_t>((size_t)2 * kMaxBins);
    return cv.used();
}
inline size_t index_bytes(int B, int V, long long t_total) {
    IndexView v;
    return carve_index(nullptr, B, V, t_total, &v);
}
__device__ __forceinline__ int bucket_of(int tok, int V) { return (tok >= 0 && tok < V) ? tok : V; }
__device__ __forceinline__ long long base_of(long long t0, int b, int V) {
    return t0 + t0 / 4 + (long long)b * (2ll * (V + 1) + kOvf);
}
__device__ __forceinline__ long long start_of(int first, int v) { return (long long)first + first / 4 + 2ll * v; }

// (0) the build's offsets: tok_off[0] = 0, ascending, tok_off[B] = t_total;
// every later build kernel does nothing unless they are
__global__ void __launch_bounds__(1024)
index_check(const int64_t *tok_off, int B, long long t_total, IndexView ix) {
    pdl_enter();
    int bad = threadIdx.x == 0 && (tok_off[0] != 0 || tok_off[B] != t_total);
    for (int b = threadIdx.x; b < B; b += blockDim.x) bad |= tok_off[b + 1] < tok_off[b];
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) *ix.valid = bad ? 0 : 1;
}

// The keys of a pass, by tile: pass 0 makes them from the tokens (the request
// of token i is the last b with tok_off[b] <= i), later passes read the pairs.
struct TokenKeys {
    const int32_t *tokens;
    const int64_t *tok_off;
    int B, V, vbits;
    uint32_t i0;         // the tile's first token
    const int32_t *tile;
    uint32_t high;       // the request bits of that token's key
    int own;             // the tile's tokens of the same request
    __device__ __forceinline__ int request(long long i) const {
        int lo = 0, hi = B - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tok_off[mid] <= i) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    }
    __device__ __forceinline__ uint32_t request_bits(int b) const { return vbits >= 32 ? 0u : (uint32_t)b << vbits; }
    __device__ __forceinline__ void begin(long long first) {
        i0 = (uint32_t)first;
        tile = tokens + first;
    }
    // the load, apart from what is made of it, so that a thread's loads are all
    // in flight before any is used
    __device__ __forceinline__ int load(int e) const { return tile[e]; }
    __device__ __forceinline__ void after_loads() {
        const int b = request(i0);
        const long long left = tok_off[b + 1] - (long long)i0;
        high = request_bits(b);
        own = (int)(left < 0x7fffffff ? left : 0x7fffffff);
    }
    __device__ __forceinline__ uint2 pair(int tok, int e) const {
        const uint32_t i = i0 + (uint32_t)e;
        return make_uint2((uint32_t)bucket_of(tok, V) | (e < own ? high : request_bits(request(i))), i);
    }
};
struct PairKeys {
    const uint2 *in;
    __device__ __forceinline__ void begin(long long first) { in += first; }
    __device__ __forceinline__ uint2 load(int e) const { return in[e]; }
    __device__ __forceinline__ void after_loads() {}
    __device__ __forceinline__ uint2 pair(uint2 x, int) const { return x; }
};

// Each radix kernel handles one tile of kR * 256 keys; a thread's keys are all
// loaded before any is used.
template <class Keys, int kR>
__global__ void __launch_bounds__(kRadixThreads)
radix_hist(Keys src, long long N, int shift, int bins, int32_t *hist, const int32_t *valid) {
    pdl_enter();
    if (!*valid) return;
    __shared__ int cnt[kMaxBins];
    const long long tile = blockIdx.x, i0 = tile * (kR * kRadixThreads);
    for (int d = threadIdx.x; d < bins; d += kRadixThreads) cnt[d] = 0;
    const int n = (int)(N - i0 < kR * kRadixThreads ? N - i0 : kR * kRadixThreads);
    src.begin(i0);
    decltype(src.load(0)) x[kR];
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = q * kRadixThreads + (int)threadIdx.x;
        x[q] = src.load(e < n ? e : 0);
    }
    src.after_loads();
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = q * kRadixThreads + (int)threadIdx.x;
        if (e < n) atomicAdd(&cnt[(src.pair(x[q], e).x >> shift) & (bins - 1)], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += kRadixThreads) hist[tile * bins + d] = cnt[d];
}

// The exclusive sum over the block of one value per thread.
__device__ __forceinline__ int radix_excl_scan(int v, int *s_w, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    int before = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) {
        const int y = s_w[w];
        before += w < warp ? y : 0;
        sum += y;
    }
    __syncthreads();
    *total = sum;
    return before + x - v;
}

// (tile, digit) offsets: each digit's exclusive prefix over the tiles, and
// its total.  A block takes eight digits (one 32-byte sector of a tile's
// counts); thread (group g, digit d) takes kT consecutive tiles a round, four
// groups to a warp.
// Two sizes: up to kOffFew tiles in one round of 256 threads (4096 tokens: 19.0 us
// for the whole build, 21.4 with 1024 threads), more in rounds of 1024 tiles by
// 512 threads (4 x 1M tokens: 65.7 us, 68.8 with 1024 threads; 8 x 60K tokens 31.7,
// 34.6 in rounds of 128).
constexpr int kOffDigits = 8;
constexpr int kOffManyT = 16, kOffFewT = 4, kOffFew = 128;
constexpr int off_threads(int per_thread) { return per_thread == kOffManyT ? 512 : 256; }
static_assert(kOffFew == off_threads(kOffFewT) / kOffDigits * kOffFewT, "one round");
template <int kT>
__global__ void __launch_bounds__(off_threads(kT))
radix_offsets(int32_t *hist, long long ntiles, int bins, int32_t *dtot,
              const int32_t *valid) {
    pdl_enter();
    if (!*valid) return;
    constexpr int kWarps = off_threads(kT) / 32, kGroups = off_threads(kT) / kOffDigits;
    __shared__ int s_sum[kWarps][kOffDigits];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = lane % kOffDigits, g = threadIdx.x / kOffDigits;
    int32_t *col = hist + blockIdx.x * kOffDigits + d;
    const bool live = (int)blockIdx.x * kOffDigits + d < bins;
    int carry = 0;
    for (long long base = 0; base < ntiles; base += kGroups * kT) {
        const long long t = base + g * kT;
        int c[kT], sum = 0;
#pragma unroll
        for (int q = 0; q < kT; ++q) c[q] = live && t + q < ntiles ? col[(t + q) * bins] : 0;
#pragma unroll
        for (int q = 0; q < kT; ++q) sum += c[q];
        int x = sum;
#pragma unroll
        for (int o = kOffDigits; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane >= 32 - kOffDigits) s_sum[warp][d] = x;
        __syncthreads();
        x += carry - sum;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const int y = s_sum[w][d];
            x += w < warp ? y : 0;
            carry += y;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kT; ++q) {
            if (live && t + q < ntiles) col[(t + q) * bins] = x;
            x += c[q];
        }
    }
    if (live && g == 0) dtot[blockIdx.x * kOffDigits + d] = carry;
}

// A tile of keys put in digit order in shared memory, stably.  Warp w takes the
// keys w 32 rounds .. of the tile, 32 at a time; a key's rank is the count of
// equal digits before it in the tile (earlier warps, earlier rounds of its
// warp, lower lanes of its round).
template <class W, int kR>
struct alignas(16) TileShared {
    union {
        W word[kR * kRadixThreads];
        uint32_t peers[kRadixWarps][kMaxBins];  // while ranking: the lanes of the warp's round with that digit
    };
    uint16_t cnt[kRadixWarps][kMaxBins];
    int w[kRadixWarps];
};
__device__ __forceinline__ int tile_rounds_of(int n) { return (n + kRadixThreads - 1) / kRadixThreads; }
__device__ __forceinline__ int tile_elem(int rounds, int q) {
    return ((int)(threadIdx.x >> 5) * rounds + q) * 32 + (int)(threadIdx.x & 31);
}
// k[q]: this thread's keys, those past the tile's last with the largest digit
// (they come after the others wherever they are counted); digit(k): a key's
// digit; starts(x, y): called by every thread with the places of its digits 2
// tid and 2 tid + 1 in the ordered tile.  Ends with a barrier.
//
// Bound by shared memory (a key's bit, count, place, and the key itself written
// and read, most at two to three lanes a bank).  The lanes of a round that
// share a digit: those of the first lane's by one ballot, the others set their
// bits in a word per digit.  The ballot takes the digit that many lanes have,
// as in text and in the later passes, where setting bits would run one lane
// after the other.  A build of 4 x 1M tokens with this against a ballot per digit
// bit: a text 63.0 and 85.7 us, uniform tokens 63.1 and 86.6, one token 53.5 and
// 81.2 (bits alone: text 71, match.any in the second pass: text 60.5, uniform
// 78.4).
template <class W, int kR, class Digit, class Starts>
__device__ __forceinline__ void order_tile(TileShared<W, kR> &sh, const W (&k)[kR], int rounds, Digit digit,
                                           Starts starts) {
    using Tile = TileShared<W, kR>;
    static_assert(offsetof(Tile, peers) % 16 == 0 && offsetof(Tile, cnt) % 16 == 0, "cleared by 16-byte words");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int x = tid; x < kRadixWarps * kMaxBins / 8; x += kRadixThreads) reinterpret_cast<uint4 *>(&sh.cnt[0][0])[x] = uint4{};
    for (int x = tid; x < kRadixWarps * kMaxBins / 4; x += kRadixThreads)
        reinterpret_cast<uint4 *>(&sh.peers[0][0])[x] = uint4{};
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    int rk[kR];
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        if (q >= rounds) break;
        const int dg = digit(k[q]);
        const bool as_first = dg == __shfl_sync(0xffffffffu, dg, 0);
        const unsigned firsts = __ballot_sync(0xffffffffu, as_first);
        if (!as_first) atomicOr(&sh.peers[warp][dg], 1u << lane);
        __syncwarp();
        const unsigned peers = as_first ? firsts : sh.peers[warp][dg];
        const int before = sh.cnt[warp][dg];
        __syncwarp();
        if ((peers & lt) == 0) {
            sh.cnt[warp][dg] = (uint16_t)(before + __popc(peers));
            if (!as_first) sh.peers[warp][dg] = 0;
        }
        __syncwarp();
        rk[q] = before + __popc(peers & lt);
    }
    __syncthreads();
    {  // each digit's counts over the warps, then over the digits
        int run[2] = {0, 0};
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) {
            uint32_t *p = reinterpret_cast<uint32_t *>(&sh.cnt[w][2 * tid]);
            const uint32_t c = *p;
            *p = (uint32_t)run[0] | ((uint32_t)run[1] << 16);
            run[0] += (int)(c & 0xffffu);
            run[1] += (int)(c >> 16);
        }
        int total;
        const int x = radix_excl_scan(run[0] + run[1], sh.w, &total);
        starts(x, x + run[0]);
        // the counters become places in the ordered tile
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) {
            uint32_t *p = reinterpret_cast<uint32_t *>(&sh.cnt[w][2 * tid]);
            const uint32_t c = *p;
            *p = ((c & 0xffffu) + (uint32_t)x) | (((c >> 16) + (uint32_t)(x + run[0])) << 16);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kR; ++q)
        if (q < rounds) sh.word[sh.cnt[warp][digit(k[q])] + rk[q]] = k[q];
    __syncthreads();
}

// This thread's digits 2 tid and 2 tid + 1 of a row of bins counts (bins is even).
__device__ __forceinline__ int2 two_digits(const int32_t *row, int bins) {
    return 2 * (int)threadIdx.x < bins ? *reinterpret_cast<const int2 *>(row + 2 * threadIdx.x) : make_int2(0, 0);
}

// What a scatter keeps of a key in its tile and writes: the pair itself, or
// (first pass of a cut build, digit: the low bits of the key) the key over its
// place in the tile, written as its other bits over its position.
template <int kR>
struct WholePair {
    using W = uint2;
    static constexpr int kBlocks = 3;
    int shift, bins;
    __device__ __forceinline__ W make(uint2 p, int) const { return p; }
    __device__ __forceinline__ W last() const { return make_uint2(0xffffffffu, 0u); }
    __device__ __forceinline__ int digit(W w) const { return (int)((w.x >> shift) & (bins - 1)); }
    __device__ __forceinline__ W out(W w, long long) const { return w; }
};
template <int kR>
struct Packed {
    using W = uint32_t;
    static constexpr int kBlocks = 4;
    static constexpr int kPlace = kR == kTileRounds ? 12 : 10;
    static_assert(kR * kRadixThreads == 1 << kPlace && 2 * kMaxDigitBits + kPlace <= 32, "a key and a place in 32 bits");
    int lo_bits, pos_bits;
    __device__ __forceinline__ W make(uint2 p, int e) const { return p.x << kPlace | (uint32_t)e; }
    __device__ __forceinline__ W last() const { return 0xffffffffu; }
    __device__ __forceinline__ int digit(W w) const { return (int)((w >> kPlace) & ((1u << lo_bits) - 1u)); }
    __device__ __forceinline__ W out(W w, long long i0) const {
        return ((w >> kPlace) >> lo_bits) << pos_bits | ((uint32_t)i0 + (w & ((1u << kPlace) - 1u)));
    }
};

// The stable scatter: equal digits -- consecutive addresses -- are written by
// neighbouring threads.
template <class Keys, int kR, class Words>
__global__ void __launch_bounds__(kRadixThreads, Words::kBlocks)
radix_scatter(Keys src, Words words, typename Words::W *out, long long N, int bins,
              const int32_t *hist, const int32_t *dtot, const int32_t *valid) {
    pdl_enter();
    if (!*valid) return;
    using W = typename Words::W;
    constexpr int kTile = kR * kRadixThreads;
    __shared__ TileShared<W, kR> sh;
    __shared__ int s_dst[kMaxBins];  // global index of the digit's first key, less its place in the tile
    const long long tile = blockIdx.x, i0 = tile * kTile;
    const int n = (int)(N - i0 < kTile ? N - i0 : kTile), rounds = tile_rounds_of(n);
    src.begin(i0);
    decltype(src.load(0)) x[kR];
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = tile_elem(rounds, q);
        x[q] = src.load(q < rounds && e < n ? e : 0);
    }
    src.after_loads();
    // where the tile's keys of each digit begin, within the digit and over all digits
    int2 g = two_digits(hist + tile * bins, bins);
    const int2 tot = two_digits(dtot, bins);
    W k[kR];
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = tile_elem(rounds, q);
        k[q] = q < rounds && e < n ? words.make(src.pair(x[q], e), e) : words.last();
    }
    int all;
    const int below = radix_excl_scan(tot.x + tot.y, sh.w, &all);
    g.x += below;
    g.y += below + tot.x;
    order_tile(
        sh, k, rounds, [&](W w) { return words.digit(w); },
        [&](int x0, int x1) {
            s_dst[2 * threadIdx.x] = g.x - x0;
            s_dst[2 * threadIdx.x + 1] = g.y - x1;
        });
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = q * kRadixThreads + threadIdx.x;
        if (e < n) {
            const W v = sh.word[e];
            out[(long long)s_dst[words.digit(v)] + e] = words.out(v, i0);
        }
    }
}

// ---- the second of two passes, with tiles cut at the first digit ----
// Tile `tile`: its keys [i0, i0 + n) share the first digit `digit`, whose keys
// begin with tile `first`; n = 0 past the last tile.  dtot: the first digit's
// totals.
struct __align__(16) CutTile {
    int digit, first, n, i0;
};
__device__ __forceinline__ CutTile cut_tile(const int32_t *dtot, int bins, int tile_keys, int tile, int *s_w, CutTile *s_out) {
    const int2 c = two_digits(dtot, bins);
    if (threadIdx.x == 0) s_out->n = 0;
    const int a = (c.x + tile_keys - 1) / tile_keys, b = (c.y + tile_keys - 1) / tile_keys;
    int all;
    const int tx = radix_excl_scan(a + b, s_w, &all);
    const int kx = radix_excl_scan(c.x + c.y, s_w, &all);
    if (tile >= tx && tile < tx + a + b) {
        const bool second = tile >= tx + a;
        const int first = second ? tx + a : tx, at = (tile - first) * tile_keys, cnt = second ? c.y : c.x;
        *s_out = CutTile{2 * (int)threadIdx.x + second, first, min(tile_keys, cnt - at), kx + (second ? c.x : 0) + at};
    }
    __syncthreads();
    return *s_out;
}

template <int kR>
__global__ void __launch_bounds__(kRadixThreads)
cut_hist(const uint32_t *in, int bins0, int pos_bits, int bins, const int32_t *dtot,
         int32_t *hist, CutTile *tiles, const int32_t *valid) {
    pdl_enter();
    if (!*valid) return;
    __shared__ int cnt[kMaxBins];
    __shared__ int s_w[kRadixWarps];
    __shared__ CutTile s_tile;
    for (int d = threadIdx.x; d < bins; d += kRadixThreads) cnt[d] = 0;
    const CutTile t = cut_tile(dtot, bins0, kR * kRadixThreads, blockIdx.x, s_w, &s_tile);
    if (threadIdx.x == 0) tiles[blockIdx.x] = t;
    uint32_t x[kR];
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = q * kRadixThreads + threadIdx.x;
        x[q] = e < t.n ? in[t.i0 + e] : 0u;
    }
#pragma unroll
    for (int q = 0; q < kR; ++q)
        if (q * kRadixThreads + (int)threadIdx.x < t.n) atomicAdd(&cnt[x[q] >> pos_bits], 1);
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += kRadixThreads) hist[(long long)blockIdx.x * bins + d] = cnt[d];  // 0 past the last tile
}

// Blocks [0, tiles): a tile's positions into their buckets.  With O[tile][h] the
// keys of second digit h in earlier tiles and base(h) those of smaller second
// digits, bucket (h, l) begins at sorted index base(h) + O[first tile of l][h].
// Blocks past them: first[] and len[] of 1024 buckets, from the same sums.
constexpr int kCutFirst = 1024;
template <int kR>
__global__ void __launch_bounds__(kRadixThreads, 4)
cut_scatter(const uint32_t *in, const CutTile *cuts, int tiles, int bins0, int lo_bits, int pos_bits, int bins,
            const int32_t *dtot, const int32_t *hist, const int64_t *tok_off, int B, int V, int vbits, IndexView ix) {
    pdl_enter();
    if (!*ix.valid) return;
    constexpr int kTile = kR * kRadixThreads;
    __shared__ TileShared<uint32_t, kR> sh;
    __shared__ long long s_list[kMaxBins];  // list slot of the digit's first key in the tile, less its place there
    __shared__ int s_t0[kMaxBins];
    const int tid = threadIdx.x;
    const uint32_t vmask = (1u << vbits) - 1u;  // vbits <= 18 here
    const int2 tot = two_digits(dtot + kMaxBins, bins);
    const CutTile t = (int)blockIdx.x < tiles ? cuts[blockIdx.x] : CutTile{};
    int all;
    if ((int)blockIdx.x >= tiles) {
        const int below = radix_excl_scan(tot.x + tot.y, sh.w, &all);
        int *s_base = s_t0, *s_first = reinterpret_cast<int *>(s_list);
        const int2 c = two_digits(dtot, bins0);
        const int a = (c.x + kTile - 1) / kTile, b = (c.y + kTile - 1) / kTile;
        const int tx = radix_excl_scan(a + b, sh.w, &all);
        s_base[2 * tid] = below;
        s_base[2 * tid + 1] = below + tot.x;
        s_first[2 * tid] = tx;
        s_first[2 * tid + 1] = tx + a;
        __syncthreads();
        const long long end = (long long)B * (V + 2);
        for (int q = 0; q < kCutFirst / kRadixThreads; ++q) {
            const long long i = (long long)((int)blockIdx.x - tiles) * kCutFirst + q * kRadixThreads + tid;
            if (i >= end) break;
            const int rb = (int)(i / (V + 2)), v = (int)(i - (long long)rb * (V + 2));
            const long long t0 = tok_off[rb];
            const int t = (int)(tok_off[rb + 1] - t0);
            auto first_of = [&](int w) -> int {
                if (w > V) return t;
                const uint32_t key = ((uint32_t)rb << vbits) | (uint32_t)w;
                const int lo = (int)(key & ((1u << lo_bits) - 1u)), hi = (int)(key >> lo_bits);
                return (int)(s_base[hi] + hist[(long long)s_first[lo] * bins + hi] - t0);
            };
            const int f = first_of(v);
            ix.first[i] = f;
            if (v <= V) ix.len[(long long)rb * (V + 1) + v] = first_of(v + 1) - f;
            if (v == 0) {
                ix.built[rb] = t;
                ix.base[rb] = base_of(t0, rb, V);
                ix.ovf_n[rb] = 0;
            }
        }
        return;
    }
    if (t.n == 0) return;
    const int rounds = tile_rounds_of(t.n);
    const uint32_t last = (uint32_t)(bins - 1) << pos_bits;
    uint32_t k[kR];
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = tile_elem(rounds, q);
        k[q] = q < rounds && e < t.n ? in[t.i0 + e] : last;
    }
    const int2 own = two_digits(hist + (long long)blockIdx.x * bins, bins);
    const int2 run = two_digits(hist + (long long)t.first * bins, bins);
    const int below = radix_excl_scan(tot.x + tot.y, sh.w, &all);
    const int base[2] = {below, below + tot.x};
    long long list[2] = {0, 0};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int d = 2 * tid + h;
        const uint32_t key = ((uint32_t)d << lo_bits) | (uint32_t)t.digit;
        const int b = (int)(key >> vbits), v = (int)(key & vmask);
        if (d < bins && b < B && v <= V) {
            const long long t0 = tok_off[b];
            const int o = h ? own.y : own.x, r = h ? run.y : run.x;
            const int f = (int)(base[h] + r - t0);
            list[h] = base_of(t0, b, V) + kOvf + start_of(f, v) + (o - r);
            s_t0[d] = (int)t0;
        }
    }
    order_tile(
        sh, k, rounds, [&](uint32_t w) { return (int)(w >> pos_bits); },
        [&](int x0, int x1) {
            s_list[2 * tid] = list[0] - x0;
            s_list[2 * tid + 1] = list[1] - x1;
        });
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int e = q * kRadixThreads + tid;
        if (e < t.n) {
            const uint32_t v = sh.word[e];
            const int d = (int)(v >> pos_bits);
            ix.list[s_list[d] + e] = (int32_t)((v & ((1u << pos_bits) - 1u)) - (uint32_t)s_t0[d]);
        }
    }
}
static_assert(kMaxBins == 2 * kRadixThreads, "two digits per thread");
static_assert(kTileRounds * kRadixThreads <= 65535, "16-bit tile counters");

// ---- after plain passes ----
// first[b][v]: where the keys of (b, v) begin in the sorted order, by binary
// search; the lengths are the differences.  Blocks of 256 threads cover 255
// buckets (the last thread only serves its neighbour).
constexpr int kFirstPer = 255;
__global__ void __launch_bounds__(kFirstPer + 1)
index_first(const uint2 *sorted, const int64_t *tok_off, int V, int vbits, IndexView ix) {
    pdl_enter();
    if (!*ix.valid) return;
    __shared__ int s_first[kFirstPer + 1];
    const int b = blockIdx.y, tid = threadIdx.x;
    const long long v = (long long)blockIdx.x * kFirstPer + tid;
    const long long t0 = tok_off[b], t1 = tok_off[b + 1];
    int f = (int)(t1 - t0);
    if (v <= V) {
        const uint32_t key = (uint32_t)v | (vbits >= 32 ? 0u : ((uint32_t)b << vbits));
        long long lo = t0, hi = t1;  // first key >= (b, v)
        while (lo < hi) {
            const long long mid = (lo + hi) >> 1;
            if (sorted[mid].x < key) lo = mid + 1;
            else hi = mid;
        }
        f = (int)(lo - t0);
    }
    s_first[tid] = f;
    __syncthreads();
    if (tid < kFirstPer && v <= V + 1) {
        ix.first[(long long)b * (V + 2) + v] = f;
        if (v <= V) ix.len[(long long)b * (V + 1) + v] = s_first[tid + 1] - f;
    }
    if (blockIdx.x == 0 && tid == 0) {
        ix.built[b] = t1 - t0;
        ix.base[b] = base_of(t0, b, V);
        ix.ovf_n[b] = 0;
    }
}

// Each sorted position into its bucket: its rank among the request's
// positions of that bucket is its sorted index minus the bucket's first.
constexpr int kPlacePer = 4;
__global__ void __launch_bounds__(256)
index_place(const uint2 *sorted, long long N, const int64_t *tok_off, int V, int vbits,
            IndexView ix) {
    pdl_enter();
    if (!*ix.valid) return;
    const uint32_t vmask = (vbits >= 32) ? 0xffffffffu : ((1u << vbits) - 1u);
    const long long j0 = (long long)blockIdx.x * (256 * kPlacePer) + threadIdx.x;
    uint2 p[kPlacePer];
    int f[kPlacePer];
#pragma unroll
    for (int q = 0; q < kPlacePer; ++q) p[q] = j0 + 256 * q < N ? sorted[j0 + 256 * q] : make_uint2(0u, 0u);
#pragma unroll
    for (int q = 0; q < kPlacePer; ++q) {
        const int b = (int)(vbits >= 32 ? 0 : (p[q].x >> vbits));
        f[q] = ix.first[(long long)b * (V + 2) + (p[q].x & vmask)];
    }
#pragma unroll
    for (int q = 0; q < kPlacePer; ++q) {
        const long long j = j0 + 256 * q;
        if (j >= N) break;
        const int b = (int)(vbits >= 32 ? 0 : (p[q].x >> vbits));
        const long long t0 = tok_off[b];
        ix.list[ix.base[b] + kOvf + start_of(f[q], (int)(p[q].x & vmask)) + (j - t0 - f[q])] = (int32_t)((long long)p[q].y - t0);
    }
}

// Append: the positions built[b] .. t_b - 1 of every request, in one round of a
// warp when they are few (an append of 5 tokens and its query 8.5 -> 8.0 us),
// else in rounds of kAppThreads; see the file comment.
__global__ void __launch_bounds__(kAppThreads)
index_append(const int32_t *tokens, const int64_t *tok_off, int V, IndexView ix,
             int32_t *status) {
    pdl_enter();
    constexpr int kW = kAppThreads / 32;
    __shared__ int s_bk[kAppThreads];
    __shared__ unsigned char s_ok[kAppThreads];  // in the index (p < cut) and in its bucket
    __shared__ int s_w[kW];
    __shared__ long long s_cut;
    __shared__ int s_novf;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    long long built = ix.built[b];  // read beside the offsets; unused in an index that holds nothing
    int novf = ix.ovf_n[b];
    const long long t0 = tok_off[b], t = tok_off[b + 1] - t0;
    // an index whose build saw inconsistent offsets holds nothing, and the
    // buffers hold tok_off[B] tokens: otherwise nothing is read or written
    if (!*ix.valid || t0 < 0 || t < 0 || t0 + t > tok_off[gridDim.x]) {
        if (tid == 0 && status) status[b] = RS_ST_BAD_OFFSET;
        return;
    }
    const int32_t *X = tokens + t0;
    const int32_t *first = ix.first + (long long)b * (V + 2);
    int32_t *len = ix.len + (long long)b * (V + 1);
    int32_t *ovf = ix.list + ix.base[b];
    int32_t *buckets = ovf + kOvf;
    bool full = false;
    if (built < t && t - built <= 32) {
        // a step's few tokens: one warp, no barriers
        if (tid >= 32) return;
        const bool valid = lane < (int)(t - built);
        const int p = (int)built + lane;
        const int bk = valid ? bucket_of(X[p], V) : -1 - lane;
        const int f0 = valid ? first[bk] : 0, f1 = valid ? first[bk + 1] : 0;
        const int held = valid ? len[bk] : 0;
        const unsigned peers = __match_any_sync(0xffffffffu, bk), lt = (1u << lane) - 1u;
        const int slot = held + __popc(peers & lt);
        const bool inb = valid && slot < (f1 - f0) + (f1 - f0) / 4 + 2;
        const unsigned ov = __ballot_sync(0xffffffffu, valid && !inb);
        const int oslot = novf + __popc(ov & lt);
        // the first position with no room anywhere ends the indexed ones
        const unsigned none = __ballot_sync(0xffffffffu, valid && !inb && oslot >= kOvf);
        const int cut = none ? __ffs(none) - 1 : (int)(t - built);
        const bool in = lane < cut;
        const unsigned put = __ballot_sync(0xffffffffu, in && inb);
        if (in && inb) {
            buckets[start_of(f0, bk) + slot] = p;
            if ((peers & put) >> lane == 1u) len[bk] = slot + 1;  // the bucket's last
        }
        if (in && valid && !inb) ovf[oslot] = p;
        if (lane == 0) {
            ix.built[b] = built + cut;
            ix.ovf_n[b] = novf + __popc(ov & (cut < 32 ? (1u << cut) - 1u : 0xffffffffu));
            if (status) status[b] = built + cut < t ? RS_ST_TRUNCATED : 0;
        }
        return;
    }
    for (long long r0 = built; r0 < t && !full; r0 += kAppThreads) {
        const long long p = r0 + tid;
        const bool valid = p < t;
        const int bk = valid ? bucket_of(X[p], V) : -1;
        s_bk[tid] = bk;
        if (tid == 0) s_cut = t;
        __syncthreads();
        const int lo = valid ? len[bk] : 0;
        const int f0 = valid ? first[bk] : 0, f1 = valid ? first[bk + 1] : 0;
        const long long start = start_of(f0, valid ? bk : 0);
        const int room = valid ? (f1 - f0) + (f1 - f0) / 4 + 2 : 0;
        const int nr = (int)(t - r0 < kAppThreads ? t - r0 : kAppThreads);  // positions of this round
        int rank = 0;
        for (int j = 0; j < tid && j < nr; ++j) rank += s_bk[j] == bk;
        const int slot = lo + rank;
        const bool inb = valid && slot < room;
        const bool ov = valid && !inb;
        // overflow ranks in position order
        int x = ov ? 1 : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        int before = 0, nov = 0;
        for (int w = 0; w < kW; ++w) {
            before += w < warp ? s_w[w] : 0;
            nov += s_w[w];
        }
        const int oslot = novf + before + x - (ov ? 1 : 0);
        if (ov && oslot >= kOvf) atomicMin(&s_cut, p);  // the first position with no room anywhere
        __syncthreads();
        const long long cut = s_cut;
        const bool in = valid && p < cut;
        s_ok[tid] = (unsigned char)(in && inb);
        if (in && inb) buckets[start + slot] = (int32_t)p;
        if (in && ov) ovf[oslot] = (int32_t)p;
        if (tid == 0) s_novf = 0;
        __syncthreads();
        // the last indexed position of a bucket in this round sets its length
        if (in && inb) {
            bool last = true;
            for (int j = tid + 1; j < nr; ++j)
                if (s_bk[j] == bk && s_ok[j]) last = false;
            if (last) len[bk] = slot + 1;
        }
        if (in && ov) atomicAdd(&s_novf, 1);
        __syncthreads();
        novf += s_novf;
        if (cut < t) {
            built = cut;
            full = true;
        } else {
            built = r0 + kAppThreads < t ? r0 + kAppThreads : t;
        }
        __syncthreads();  // s_bk, s_ok, s_cut reused by the next round
    }
    if (tid == 0) {
        ix.built[b] = built;
        ix.ovf_n[b] = novf;
        if (status) status[b] = built < t ? RS_ST_TRUNCATED : 0;
    }
}

// Query candidates, ascending: the bucket of the key's last token, the
// overflow list (every token's overflow entries are newer than its bucket's),
// then the positions not indexed (built .. t - 2); row r's element e of lane l
// is candidate 128 r + 32 e + l.
struct ListSource {
    static constexpr int kRows = 2;
    static constexpr int kThreads = kMatHalf, kFewB = 4;
    static constexpr int kWideRows = 128;  // 16384 candidates, each a read of its own
    static constexpr bool kLaneMajor = false;
    static constexpr bool kSparse = false;  // candidates of a list often match: the test costs 0.05 to 0.1 us
    static constexpr bool kBound = false;  // (its code, 16 registers more, costs every query 0.4 us)
    const int32_t *blist, *olist;
    int nb, no, tail0;
    ListPos at{0};  // at most 2^31 - 1 in all: no position is in two lists
    __device__ __forceinline__ int cand(int c) const {
        if (c < nb) return blist[c];
        c -= nb;
        return c < no ? olist[c] : tail0 + (c - no);
    }
    __device__ __forceinline__ int pos(int row, int lane, int e) const { return cand(at.number(row, 32 * e + lane)); }
    __device__ __forceinline__ uint32_t test(const MatReq &q, int r0, int end, int lane) const {
        int p[4 * kRows], x0[4 * kRows], x1[4 * kRows];
#pragma unroll
        for (int j = 0; j < 4 * kRows; ++j) {
            const int o = 32 * j + lane;  // rows follow one another
            p[j] = r0 + (j >> 2) < end && at.in(r0, o) ? cand(at.number(r0, o)) : -1;
        }
#pragma unroll
        for (int j = 0; j < 4 * kRows; ++j) {
            const bool in = p[j] >= q.k - 1 && p[j] <= q.t - 2;
            if (!in) p[j] = -1;
            x0[j] = in ? q.X[p[j]] : 0;
            x1[j] = in && q.k > 1 ? q.X[p[j] - 1] : 0;
        }
        const int kl = q.k1, k2 = q.k2;
        uint32_t hits = 0;
#pragma unroll
        for (int j = 0; j < 4 * kRows; ++j)
            if (p[j] >= 0 && x0[j] == kl && (q.k < 2 || x1[j] == k2)) hits |= 1u << j;
        if (q.k > 2) {
#pragma unroll
            for (int j = 0; j < 4 * kRows; ++j)
                if (((hits >> j) & 1u) && !mat_prefix(q, p[j])) hits &= ~(1u << j);
        }
        return hits;
    }
};

__global__ void __launch_bounds__(kMatHalf)
index_query(const int32_t *tokens, const int64_t *tok_off, int V, const int32_t *k_star, const uint8_t *gate_ok,
            const float *scores, IndexView ix, MatOut o) {
    __shared__ MatShared sh;
    mat_enter(sh);
    extern __shared__ __align__(16) uint32_t qry_bits[];
    const int crank = (int)cooperative_groups::this_cluster().block_rank();
    const int b = blockIdx.y;
    // an index whose build saw inconsistent offsets holds nothing: the request is not read
    const long long built = ix.built[b], base = ix.base[b];  // read beside the request's own records
    const int novf = ix.ovf_n[b];
    MatReq q;
    mat_request(q, tokens, tok_off, k_star, gate_ok, scores, b, gridDim.y, *ix.valid != 0);
    ListSource src{nullptr, nullptr, 0, 0, 0, ListPos{0}};
    if (q.run) {
        const int bk = bucket_of(q.k1, V);
        src.olist = ix.list + base;
        src.blist = src.olist + kOvf + start_of(ix.first[(long long)b * (V + 2) + bk], bk);
        src.nb = ix.len[(long long)b * (V + 1) + bk];
        src.no = novf;
        src.tail0 = (int)(built < q.t ? built : q.t);
        const int nt = q.t - 1 - src.tail0;  // tail: positions tail0 .. t - 2
        src.at.n = src.nb + src.no + (nt > 0 ? nt : 0);
    }
    const int rows = src.at.rows();
    q.threads = kMatHalf;
    const int nc = mat_ctas<ListSource>(rows, q.threads);
    if (crank >= nc) return;
    mat_body(src, q, rows, nc, b, crank, sh, qry_bits, o);
}

}  // namespace
}  // namespace rs

using namespace rs;

extern "C" size_t rs_match_index_bytes(int B, int V, int64_t t_total) {
    if (B < 0 || V < 1 || t_total < 0) return 0;
    return index_bytes(B, V, t_total);
}

static rs_status check_index(const char *who, int B, int V, int64_t t_total, const void *index,
                             size_t index_bytes_avail) {
    RS_CHECK_ARG(B >= 0 && B <= 65535, "%s: B=%d outside [0, 65535]", who, B);
    RS_CHECK_ARG(V >= 1 && V < (1 << 30), "%s: V=%d outside [1, 2^30)", who, V);
    RS_CHECK_ARG(t_total >= 0 && t_total < (1ll << 31), "%s: t_total outside [0, 2^31)", who);
    if (key_bits(B, V) > 32) {
        set_error("%s: B=%d requests with V=%d need more than 32 key bits", who, B, V);
        return RS_ERR_UNSUPPORTED;
    }
    const size_t need = index_bytes(B, V, t_total);
    if (index_bytes_avail < need || !index) {
        set_error("%s: index %zu bytes < %zu required", who, index_bytes_avail, need);
        return RS_ERR_CAPACITY;
    }
    return RS_OK;
}

static void radix_offsets_launch(int32_t *hist, long long ntiles, int bins, int32_t *dtot, const int32_t *valid,
                                 cudaStream_t st) {
    const dim3 grid((unsigned)(bins + kOffDigits - 1) / kOffDigits);
    if (ntiles <= kOffFew)
        launch_pdl(radix_offsets<kOffFewT>, grid, dim3(off_threads(kOffFewT)), 0, st, hist, ntiles, bins, dtot, valid);
    else
        launch_pdl(radix_offsets<kOffManyT>, grid, dim3(off_threads(kOffManyT)), 0, st, hist, ntiles, bins, dtot, valid);
}

// The digit counts of a pass over the keys `src` and their offsets, then the scatter.
template <int kR, class Keys, class Words>
static rs_status radix_pass(const Keys &src, const Words &words, typename Words::W *out, int shift, int bins, long long N,
                            const IndexView &ix, cudaStream_t st) {
    const long long nt = n_tiles(N);
    const dim3 grid((unsigned)nt), block(kRadixThreads);
    launch_pdl(radix_hist<Keys, kR>, grid, block, 0, st, src, N, shift, bins, ix.hist, ix.valid);
    RS_CHECK_LAUNCH("rs_match_index_build/radix_hist");
    radix_offsets_launch(ix.hist, nt, bins, ix.dtot, ix.valid, st);
    RS_CHECK_LAUNCH("rs_match_index_build/radix_offsets");
    launch_pdl(radix_scatter<Keys, kR, Words>, grid, block, 0, st, src, words, out, N, bins, ix.hist, ix.dtot, ix.valid);
    RS_CHECK_LAUNCH("rs_match_index_build/radix_scatter");
    return RS_OK;
}

// Plain passes, then the bucket starts and the placement.
template <int kR>
static rs_status build_plain(const int32_t *tokens, const int64_t *tok_off, int B, int V, long long N, const IndexView &ix,
                             cudaStream_t st) {
    const int vbits = bits_for(V), keybits = key_bits(B, V);
    const int passes = N > 0 ? (keybits + kMaxDigitBits - 1) / kMaxDigitBits : 0;
    for (int pass = 0; pass < passes; ++pass) {
        const int bits = (keybits + passes - 1) / passes, shift = pass * bits, bins = 1 << bits;
        const WholePair<kR> words{shift, bins};
        uint2 *out = ix.pair[pass & 1];
        const rs_status s =
            pass == 0 ? radix_pass<kR>(TokenKeys{tokens, tok_off, B, V, vbits, 0, nullptr, 0, 0}, words, out, shift, bins, N, ix, st)
                      : radix_pass<kR>(PairKeys{ix.pair[(pass & 1) ^ 1]}, words, out, shift, bins, N, ix, st);
        if (s != RS_OK) return s;
    }
    const uint2 *sorted = ix.pair[(passes - 1) & 1];
    launch_pdl(index_first, dim3((unsigned)((V + 2ll + kFirstPer - 1) / kFirstPer), B), dim3(kFirstPer + 1), 0, st, sorted,
        tok_off, V, vbits, ix);
    RS_CHECK_LAUNCH("rs_match_index_build/first");
    if (N == 0) return RS_OK;
    launch_pdl(index_place, dim3((unsigned)((N + 256 * kPlacePer - 1) / (256 * kPlacePer))), dim3(256), 0, st, sorted, N,
        tok_off, V, vbits, ix);
    RS_CHECK_LAUNCH("rs_match_index_build/place");
    return RS_OK;
}

// Two passes, the second over tiles cut at the first digit.
template <int kR>
static rs_status build_cut(const int32_t *tokens, const int64_t *tok_off, int B, int V, long long N, const IndexView &ix,
                           cudaStream_t st) {
    const int vbits = bits_for(V), keybits = key_bits(B, V);
    const int lo_bits = cut_lo_bits(B, V), pos_bits = cut_pos_bits(N), bins0 = 1 << lo_bits, bins = 1 << (keybits - lo_bits);
    uint32_t *words = reinterpret_cast<uint32_t *>(ix.pair[0]);
    CutTile *cuts = reinterpret_cast<CutTile *>(ix.pair[1]);  // at most N / 1024 + 514 records of 16 bytes, N >= kCutMin
    const rs_status s = radix_pass<kR>(TokenKeys{tokens, tok_off, B, V, vbits, 0, nullptr, 0, 0}, Packed<kR>{lo_bits, pos_bits}, words, 0,
                                       bins0, N, ix, st);
    if (s != RS_OK) return s;
    const int tiles = (int)n_tiles(N) + bins0 + 1;  // the last one is never used: O past every key
    const dim3 block(kRadixThreads);
    launch_pdl(cut_hist<kR>, dim3((unsigned)tiles), block, 0, st, words, bins0, pos_bits, bins, ix.dtot, ix.hist, cuts, ix.valid);
    RS_CHECK_LAUNCH("rs_match_index_build/cut_hist");
    radix_offsets_launch(ix.hist, (long long)tiles, bins, ix.dtot + kMaxBins, ix.valid, st);
    RS_CHECK_LAUNCH("rs_match_index_build/cut_offsets");
    const unsigned firsts = (unsigned)(((long long)B * (V + 2) + kCutFirst - 1) / kCutFirst);
    launch_pdl(cut_scatter<kR>, dim3((unsigned)tiles + firsts), block, 0, st, words, cuts, tiles, bins0, lo_bits, pos_bits, bins, ix.dtot,
        ix.hist, tok_off, B, V, vbits, ix);
    RS_CHECK_LAUNCH("rs_match_index_build/cut_scatter");
    return RS_OK;
}

extern "C" rs_status rs_match_index_build(const int32_t *tokens, const int64_t *tok_off, int B, int V,
                                          int64_t t_total, void *index, size_t index_bytes_avail, void *stream) {
    clear_error();
    const rs_status e = check_index("rs_match_index_build", B, V, t_total, index, index_bytes_avail);
    if (e != RS_OK) return e;
    RS_CHECK_ARG(B == 0 || (tok_off && (tokens || t_total == 0)), "rs_match_index_build: null pointer");
    if (B == 0) return RS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    IndexView ix;
    carve_index(index, B, V, t_total, &ix);
    launch_pdl(index_check, dim3(1), dim3(1024), 0, st, tok_off, B, (long long)t_total, ix);
    RS_CHECK_LAUNCH("rs_match_index_build/check");
    const bool small = tile_rounds(t_total) == kTileRoundsSmall;
    if (cut_build(B, V, t_total))
        return small ? build_cut<kTileRoundsSmall>(tokens, tok_off, B, V, t_total, ix, st)
                     : build_cut<kTileRounds>(tokens, tok_off, B, V, t_total, ix, st);
    return small ? build_plain<kTileRoundsSmall>(tokens, tok_off, B, V, t_total, ix, st)
                 : build_plain<kTileRounds>(tokens, tok_off, B, V, t_total, ix, st);
}

extern "C" rs_status rs_match_index_append(const int32_t *tokens, const int64_t *tok_off, int B, int V,
                                           int64_t t_total, void *index, size_t index_bytes_avail, int32_t *status,
                                           void *stream) {
    clear_error();
    const rs_status e = check_index("rs_match_index_append", B, V, t_total, index, index_bytes_avail);
    if (e != RS_OK) return e;
    RS_CHECK_ARG(B == 0 || (tokens && tok_off), "rs_match_index_append: null pointer");
    if (B == 0) return RS_OK;
    IndexView ix;
    carve_index(index, B, V, t_total, &ix);
    launch_pdl(index_append, dim3(B), dim3(kAppThreads), 0, (cudaStream_t)stream, tokens, tok_off, V, ix, status);
    RS_CHECK_LAUNCH("rs_match_index_append");
    return RS_OK;
}

extern "C" rs_status rs_match_scan_indexed(const int32_t *tokens, const int64_t *tok_off, int B,
                                           const int32_t *k_star, const uint8_t *gate_ok, const float *scores,
                                           rs_params p, int pos_cap, int32_t *count, int32_t *pos,
                                           int32_t *sel_pos, int32_t *sel_len, int32_t *spans, int32_t *n_sel,
                                           int32_t *status, int V, int64_t t_total, const void *index,
                                           size_t index_bytes_avail, void *stream) {
    clear_error();
    const rs_status e = check_index("rs_match_scan_indexed", B, V, t_total, index, index_bytes_avail);
    if (e != RS_OK) return e;
    RS_CHECK_ARG(pos_cap >= 0, "rs_match_scan_indexed: negative pos_cap");
    RS_CHECK_ARG(p.top_c >= 1 && p.top_c <= RS_MAX_TOPC, "rs_match_scan_indexed: top_c=%d outside [1, %d]",
                 p.top_c, RS_MAX_TOPC);
    RS_CHECK_ARG(p.span_len >= 1 && p.span_len <= RS_MAX_SPAN, "rs_match_scan_indexed: span_len=%d outside [1, %d]",
                 p.span_len, RS_MAX_SPAN);
    RS_CHECK_ARG(B == 0 || (tokens && tok_off && k_star && scores && count && sel_pos && sel_len && spans &&
                            n_sel && status && (pos || pos_cap == 0)),
                 "rs_match_scan_indexed: null pointer");
    if (B == 0) return RS_OK;
    IndexView ix;
    carve_index(const_cast<void *>(index), B, V, t_total, &ix);
    const MatOut o{count, pos, sel_pos, sel_len, spans, n_sel, status, p.theta_score, p.top_c, p.span_len, pos_cap};
    static MatWide wide;
    return mat_launch<ListSource>("rs_match_scan_indexed", wide, index_query, B, (cudaStream_t)stream, tokens, tok_off, V, k_star,
                                  gate_ok, scores, ix, o);
}
