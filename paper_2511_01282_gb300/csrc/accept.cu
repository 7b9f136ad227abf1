// accept.cu -- rs_accept: source-aware verification (Section 3.4, Eq. 6-7
// and the look-ahead tolerance procedure), longest accepted path and winner
// (Algorithm 1), EMA feedback (Eq. 4-5 and Algorithm 1's score update).
//
// Kernel 1 (accept_rows): one CTA per (row, 8192-logit chunk) streams the
// chunk once and produces its (max, sum e^(z - max)[, sum e^(z - max)
// (z - max)]) triple and its beta best (logit, id) pairs in the total order
// (logit desc, id asc); the top-beta is exact and sort-free apart from one
// 16-lane sort that sets the candidate threshold.  No dynamic register
// indexing.
// Row merge: two warps per row merge the chunk results into argmax, top-beta,
// log-sum-exp, the row's largest logit (workspace, for kernel 3)
// and (optionally) the row entropy.  When a row has at most 8 chunks the
// row's chunk CTAs form one cluster: each pushes its results into CTA 0's
// shared memory and CTA 0 merges them after the cluster barrier, so the row
// statistics need no second kernel.  Longer rows write their chunk results
// to the workspace and kernel 2 (accept_merge) merges them.
// Kernel 3 (accept_decide): one CTA per request checks the tree, verifies
// model nodes (ancestor sets against the set of greedy matches), runs the
// look-ahead procedure per chain (one lane per chain), picks the winner and
// updates the scores (one lane per selection).
#include <math.h>

#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "sm100.cuh"

namespace rs {
namespace {

namespace cg = cooperative_groups;

constexpr int kAccThreads = 256;
constexpr int kAccVpt = 32;
constexpr int kAccChunk = kAccThreads * kAccVpt;
constexpr int kNoId = 0x7fffffff;  // "no candidate": after every real (v, id)
constexpr int kCandCap = 64;        // a chunk's candidate buffer (logits at or above the threshold)
constexpr int kListBeta = 8;        // list merges hold this many candidates of a chunk in registers
constexpr float kFarLogit = 5e8f;   // from here on logits lie 32 or more apart
constexpr int kFuseMax = 8;         // rows of at most this many chunks merge inside their cluster

struct VI {
    float v;
    int i;
};

__device__ __forceinline__ VI vi_best(VI a, VI b) { return vi_before(b.v, b.i, a.v, a.i) ? b : a; }

__device__ __forceinline__ VI vi_shfl(VI a, int o) {
    VI b;
    b.v = __shfl_xor_sync(0xffffffffu, a.v, o);
    b.i = __shfl_xor_sync(0xffffffffu, a.i, o);
    return b;
}

__device__ __forceinline__ VI warp_vi_best(VI a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = vi_best(a, vi_shfl(a, o));
    return a;
}

// (max m, sum e^(z-m), sum e^(z-m) (z-m)) of a set of logits: the row's
// log-sum-exp is m + ln s and its entropy ln s - w / s.
struct MS {
    float m, s, w;
};

// How far a triple's maximum lies below the union's.  Bounded, so that its product
// with s stays finite: a slice of masked logits (-FLT_MAX, say) has s = the number
// of them, and 0 times infinity is no 0.
__device__ __forceinline__ float ms_below(float m, float M) { return fmaxf(m - M, -1e30f); }

// The triple of the union of one triple per lane, over aligned groups of G lanes
// (each lane of a group gets it): the maximum first, then one exponential a
// lane and plain sums.  A triple without mass (s = 0) counts for nothing.
template <int G>
__device__ __forceinline__ MS ms_union(MS t) {
    const bool some = t.s != 0.f;
    float M = some ? t.m : -INFINITY;  // of a triple without mass m may be +inf
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float d = ms_below(t.m, M), c = some ? __expf(d) : 0.f;
    float s = some ? t.s * c : 0.f, w = some ? c * (t.w + t.s * d) : 0.f;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        w += __shfl_xor_sync(0xffffffffu, w, o);
    }
    return MS{M, s, w};
}
__device__ __forceinline__ MS ms_merge(MS a, MS b) {
    if (a.s == 0.f) return b;
    if (b.s == 0.f) return a;
    const float M = fmaxf(a.m, b.m), da = ms_below(a.m, M), db = ms_below(b.m, M);
    const float ca = __expf(da), cb = __expf(db);
    return MS{M, a.s * ca + b.s * cb, ca * (a.w + a.s * da) + cb * (b.w + b.s * db)};
}

// Bitonic sort of one float per lane within aligned groups of G lanes (a
// power of two <= 32), every group ending in descending order: lane g G + i
// holds the group's (i + 1)-th largest value.
template <int G>
__device__ __forceinline__ float group_sort_desc(float x, int lane) {
#pragma unroll
    for (int k = 2; k <= G; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const float y = __shfl_xor_sync(0xffffffffu, x, j);
            const bool desc = (k == G) || ((lane & k) == 0);
            const bool keep_max = ((lane & j) == 0) == desc;
            x = keep_max ? fmaxf(x, y) : fminf(x, y);
        }
    }
    return x;
}

constexpr int kHalves = 2 * kAccThreads / 32;  // half-warps per CTA (16 >= RS_MAX_BETA)
static_assert(kHalves >= RS_MAX_BETA, "the bound needs beta half-warp maxima");

struct RowsShared {
    MS sms[kAccThreads / 32];
    float hmax[kHalves];
    VI wtop[kAccThreads / 32][RS_MAX_BETA];  // per-warp lists (tie fallback)
    VI cbuf[kCandCap];                       // the chunk's candidates
    VI rx_cand[kFuseMax * RS_MAX_BETA];      // CTA 0 of a row: every chunk's beta best
    MS rx_ms[kFuseMax];                      // and every chunk's triple
    int cnt;
};

// Per-row outputs of the row statistics.
struct RowOut {
    int32_t *argmax, *topk;
    float *lse, *entropy, *rowmax;  // entropy may be null
};

// Row r's log-sum-exp (and entropy) from its chunk triples, by one warp.
template <int G>
__device__ __forceinline__ void merge_triples(const MS *part, int nchunks, long long r, const RowOut &o, int lane) {
    MS ms{-INFINITY, 0.f, 0.f};
    for (int c = lane; c < nchunks; c += 32) ms = ms_merge(ms, part[c]);
    ms = ms_union<G>(ms);
    if (lane == 0) {
        o.lse[r] = ms.s > 0.f ? ms.m + __logf(ms.s) : -INFINITY;
        if (o.entropy) o.entropy[r] = ms.s > 0.f ? (__logf(ms.s) - ms.w / ms.s) : 0.f;
    }
}

// Another merges the chunk candidate lists into argmax and top-beta.  Lane c < G
// holds chunk c's list (nchunks <= G, beta <= kBeta); the
// best of the lists' heads wins a round and its lane moves on.  (Rounds over all
// candidates with a warp-wide "best after the previous winner" each made the
// whole merge of 16 chunks and beta = 5 4.3 us behind the row pass, this 2.1.)
template <int G, int kBeta>
__device__ __forceinline__ void merge_lists(const VI *cand, int nchunks, int beta, long long r, const RowOut &o,
                                            int lane) {
    VI cv[kBeta];
#pragma unroll
    for (int k = 0; k < kBeta; ++k)
        cv[k] = lane < nchunks && k < beta ? cand[lane * beta + k] : VI{-INFINITY, kNoId};
    for (int k = 0; k < beta; ++k) {
        VI best = cv[0];
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) best = vi_best(best, vi_shfl(best, off));
        if (cv[0].i == best.i) {
#pragma unroll
            for (int q = 0; q + 1 < kBeta; ++q) cv[q] = cv[q + 1];
            cv[kBeta - 1] = VI{-INFINITY, kNoId};
        }
        if (lane == 0) {
            const int id = best.i == kNoId ? -1 : best.i;
            o.topk[r * beta + k] = id;
            if (k == 0) {
                o.argmax[r] = id;
                o.rowmax[r] = best.v;
            }
        }
    }
}

// The same for more chunks than lanes or longer lists (ncand <= 32 kPer pairs,
// loaded once into registers): beta rounds of a warp-wide "best after the
// previous winner" reduction over all candidates.
template <int kPer>
__device__ __forceinline__ void merge_row(const VI *cand, int ncand, int beta, long long r, const RowOut &o, int lane) {
    VI cv[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int c = lane + 32 * q;
        cv[q] = c < ncand ? cand[c] : VI{-INFINITY, kNoId};
    }
    VI prev{INFINITY, -1};
    for (int k = 0; k < beta; ++k) {
        VI best{-INFINITY, kNoId};
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const VI x = cv[q];
            if (x.i != kNoId && vi_before(prev.v, prev.i, x.v, x.i) && vi_before(x.v, x.i, best.v, best.i))
                best = x;
        }
        best = warp_vi_best(best);
        prev = best;
        if (lane == 0) {
            const int id = best.i == kNoId ? -1 : best.i;
            o.topk[r * beta + k] = id;
            if (k == 0) {
                o.argmax[r] = id;
                o.rowmax[r] = best.v;
            }
        }
    }
}

// One CTA per (row, 8192-logit chunk) item: the chunk's (max, sum e^(z -
// max)[, sum e^(z - max) (z - max)]) triple and its beta best (logit, id)
// pairs in the order (logit desc, id asc).
//   * Each thread streams 32 logits into registers (eight 128-bit loads, or 32
//     single ones in rows of other alignments; the in-range test is dropped for
//     chunks that lie inside the row: with it, and the registers it spilled,
//     calls on rows of 128257 logits took 1.6 times those on 128256).
//   * Every lane exponentiates against its warp's maximum, so a warp's
//     triple is a plain shuffle sum; two logits an instruction where the unit
//     has the form (145 rows of 128256 logits: 20.9 -> 20.7 us).  Scaling and
//     subtracting in one fma leaves the rounding of max log2(e) in the exponent:
//     nothing beside the logits' own spacing, but a factor of 2^860 for a warp
//     whose logits are all masked with -1e10.  Where the spacing is 32 or more
//     only logits equal to the maximum count, and they are counted.
//   * Top-beta: the sixteen half-warp maxima are logits of sixteen disjoint
//     parts of the chunk, so the beta-th largest of them (one 16-lane sort)
//     is a lower bound T on the chunk's beta-th largest logit.  Only logits
//     >= T can be among the best beta; a lane looks at a group of four only
//     if the group's maximum clears T, appends the survivors to shared
//     memory, and warp 0 ranks them by counting (rank = the number of
//     candidates before it in the total order).  If ties at T overflow the
//     buffer, every warp ranks its own logits by beta "best after the
//     previous winner" rounds and warp 0 merges the eight lists (exact too).
//   * kFuse: the chunk's results go to CTA 0 of the row (the CTAs of a row
//     are one cluster, chunk = rank), which merges the row after the
//     cluster barrier; otherwise they go to the workspace for accept_merge.
template <bool kVec, bool kEnt, bool kFuse>
__global__ void __launch_bounds__(kAccThreads, 4)
accept_rows(const float *logits, int V, int nchunks, int beta, VI *cand, MS *part, RowOut o) {
    // the kernels behind this one read the caller's arrays before they wait for
    // it (accept_decide), so they may launch only once its own wait is over
    pdl_wait_prev();
    pdl_launch_next();
    __shared__ RowsShared sh;
    const long long blk = blockIdx.x;
    const long long r = blockIdx.x / (unsigned)nchunks;  // 32-bit division
    const int chunk = (int)(blk - r * nchunks);
    const int c0 = chunk * kAccChunk;
    const float *row = logits + r * (long long)V;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr float kL2E = 1.4426950408889634f;
    const bool clustered = kFuse && nchunks > 1;
    if (clustered) cluster_arrive_relaxed();
    if (tid == 0) sh.cnt = 0;
    VI *dcand = cand + blk * beta;  // where this chunk's beta best and triple go
    MS *dms = part + blk;
    if (kFuse) {
        dcand = &sh.rx_cand[chunk * beta];
        dms = &sh.rx_ms[chunk];
        if (clustered) {
            cg::cluster_group cl = cg::this_cluster();
            dcand = cl.map_shared_rank(dcand, 0);
            dms = cl.map_shared_rank(dms, 0);
        }
    }

    // logit id of register j (ids >= V are padding, held as -inf)
    auto id_of = [&](int j) -> int {
        if (kVec) return c0 + ((j >> 2) * kAccThreads + tid) * 4 + (j & 3);
        return c0 + j * kAccThreads + tid;
    };
    float v[kAccVpt];
    if (kVec) {
        const bool inside = c0 + kAccChunk <= V;
#pragma unroll
        for (int j = 0; j < kAccVpt / 4; ++j) {
            const int off = c0 + (j * kAccThreads + tid) * 4;
            float4 x = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (inside || off < V) x = ldg_stream4(reinterpret_cast<const float4 *>(row + off));  // V % 4 == 0
            v[4 * j + 0] = x.x;
            v[4 * j + 1] = x.y;
            v[4 * j + 2] = x.z;
            v[4 * j + 3] = x.w;
        }
    } else {
        const float *p = row + c0 + tid;
        if (c0 + kAccChunk <= V) {
#pragma unroll
            for (int j = 0; j < kAccVpt; ++j) v[j] = ldg_stream(p + j * kAccThreads);
        } else {
#pragma unroll
            for (int j = 0; j < kAccVpt; ++j) v[j] = c0 + j * kAccThreads + tid < V ? ldg_stream(p + j * kAccThreads) : -INFINITY;
        }
    }

    // group, lane, half-warp and warp maxima
    float g[kAccVpt / 4];
#pragma unroll
    for (int q = 0; q < kAccVpt / 4; ++q) g[q] = fmaxf(fmaxf(v[4 * q], v[4 * q + 1]), fmaxf(v[4 * q + 2], v[4 * q + 3]));
    const float mx = fmaxf(fmaxf(fmaxf(g[0], g[1]), fmaxf(g[2], g[3])), fmaxf(fmaxf(g[4], g[5]), fmaxf(g[6], g[7])));
    float hm = mx;
#pragma unroll
    for (int off = 1; off < 16; off <<= 1) hm = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, off));
    const float wmax = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, 16));
    if ((lane & 15) == 0) sh.hmax[2 * warp + (lane >> 4)] = hm;

    MS t{wmax, 0.f, 0.f};
    if (wmax != -INFINITY) {
        // base 2: u = (z - max) log2(e), e = 2^u; sum e (z - max) = ln 2 sum e u
        const float nb = -wmax * kL2E;
        const float2 k2{kL2E, kL2E}, n2{nb, nb};
        float2 s2[2] = {}, w2[2] = {};
#pragma unroll
        for (int j = 0; j < kAccVpt; j += 2) {
            const int h = (j >> 1) & 1;
            float2 u = fma2(float2{v[j], v[j + 1]}, k2, n2);
            if (kEnt) u = float2{fmaxf(u.x, -1e30f), fmaxf(u.y, -1e30f)};  // -inf -> -1e30: e = 0, e u = 0
            const float2 e{sm100::ex2(u.x), sm100::ex2(u.y)};
            s2[h] = add2(s2[h], e);
            if (kEnt) w2[h] = fma2(e, u, w2[h]);
        }
        float ss = (s2[0].x + s2[0].y) + (s2[1].x + s2[1].y);
        float ww = (w2[0].x + w2[0].y) + (w2[1].x + w2[1].y);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            ss += __shfl_xor_sync(0xffffffffu, ss, off);
            if (kEnt) ww += __shfl_xor_sync(0xffffffffu, ww, off);
        }
        t.s = ss;
        t.w = ww * 0.6931471805599453f;
        if (fabsf(wmax) >= kFarLogit) {  // (a logit of +inf leaves no finite sum: no mass)
            int n = 0;
#pragma unroll
            for (int j = 0; j < kAccVpt; ++j) n += __popc(__ballot_sync(0xffffffffu, v[j] == wmax));
            t.s = wmax < INFINITY ? (float)n : 0.f;
            t.w = 0.f;
        }
    }
    if (lane == 0) sh.sms[warp] = t;
    __syncthreads();

    // T = the beta-th largest half-warp maximum (both half-warps sort the same 16)
    const float thr = __shfl_sync(0xffffffffu, group_sort_desc<16>(sh.hmax[lane & 15], lane), beta - 1);
    if (mx >= thr) {
#pragma unroll
        for (int q = 0; q < kAccVpt / 4; ++q) {
            if (g[q] >= thr) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = 4 * q + e;
                    const int id = id_of(j);
                    if (v[j] >= thr && id < V) {
                        const int p = atomicAdd(&sh.cnt, 1);
                        if (p < kCandCap) sh.cbuf[p] = VI{v[j], id};
                    }
                }
            }
        }
    }
    __syncthreads();
    const int total = sh.cnt;
    if (clustered) cluster_wait();  // every CTA of the row runs: CTA 0's shared memory is live
    if (total <= kCandCap) {
        if (warp == 0) {
            VI x0 = lane < total ? sh.cbuf[lane] : VI{-INFINITY, kNoId};
            VI x1 = lane + 32 < total ? sh.cbuf[lane + 32] : VI{-INFINITY, kNoId};
            int r0 = 0, r1 = 0;
            for (int q = 0; q < total; ++q) {
                const VI y = sh.cbuf[q];
                r0 += vi_before(y.v, y.i, x0.v, x0.i);
                r1 += vi_before(y.v, y.i, x1.v, x1.i);
            }
            if (lane < total && r0 < beta) dcand[r0] = x0;
            if (lane + 32 < total && r1 < beta) dcand[r1] = x1;
            if (lane >= total && lane < beta) dcand[lane] = VI{-INFINITY, kNoId};
        }
    } else {
        VI prev{INFINITY, -1};
        for (int k = 0; k < beta; ++k) {
            VI best{-INFINITY, kNoId};
#pragma unroll
            for (int j = 0; j < kAccVpt; ++j) {
                const int id = id_of(j);
                if (id < V && vi_before(prev.v, prev.i, v[j], id) && vi_before(v[j], id, best.v, best.i))
                    best = VI{v[j], id};
            }
            best = warp_vi_best(best);
            prev = best;
            if (lane == 0) sh.wtop[warp][k] = best;
        }
        __syncthreads();
        if (warp == 0) {
            constexpr int kW = kAccThreads / 32;
            VI prevb{INFINITY, -1};
            for (int k = 0; k < beta; ++k) {
                VI best{-INFINITY, kNoId};
                for (int q = lane; q < kW * beta; q += 32) {
                    const VI x = sh.wtop[q / beta][q % beta];
                    if (x.i != kNoId && vi_before(prevb.v, prevb.i, x.v, x.i) &&
                        vi_before(x.v, x.i, best.v, best.i))
                        best = x;
                }
                best = warp_vi_best(best);
                prevb = best;
                if (lane == 0) dcand[k] = best;
            }
        }
    }
    if (warp == 1) {  // the eight warp triples
        const MS a = ms_union<kAccThreads / 32>(sh.sms[lane % (kAccThreads / 32)]);
        if (lane == 0) *dms = a;
    }
    if (kFuse) {
        if (clustered) {
            cluster_arrive_release();  // the pushes above are visible in CTA 0 after the wait
            cluster_wait();
        } else {
            __syncthreads();
        }
        if (chunk == 0 && warp == 0) {
            if (beta <= kListBeta) merge_lists<kFuseMax, kListBeta>(sh.rx_cand, nchunks, beta, r, o, lane);
            else merge_row<kFuseMax * RS_MAX_BETA / 32>(sh.rx_cand, nchunks * beta, beta, r, o, lane);
        }
        if (chunk == 0 && warp == 1) merge_triples<kFuseMax>(sh.rx_ms, nchunks, r, o, lane);
    }
}

// Row statistics of rows longer than kFuseMax chunks: two warps per row merge
// the chunk results from the workspace, the lists and the triples.
constexpr int kMergeThreads = 128;
constexpr int kMergeRows = kMergeThreads / 64;  // rows per block
constexpr int kCandPerLane = 8;

__global__ void __launch_bounds__(kMergeThreads)
accept_merge(const VI *cand, const MS *part, int nchunks, int beta, int R, RowOut o) {
    pdl_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long r = (long long)blockIdx.x * kMergeRows + (warp >> 1);
    if (r >= R) return;
    const int ncand = nchunks * beta;
    if (warp & 1) merge_triples<32>(part + r * nchunks, nchunks, r, o, lane);
    else if (nchunks <= 32 && beta <= kListBeta) merge_lists<32, kListBeta>(cand + r * ncand, nchunks, beta, r, o, lane);
    else merge_row<kCandPerLane>(cand + r * ncand, ncand, beta, r, o, lane);
}

// One thread per node (warps 0-7) and a warp for the chains and selections.
constexpr int kDecThreads = RS_MAX_NODES + 32;
static_assert(RS_MAX_TOPC <= 32, "one lane per selection");
constexpr int kNodeWords = RS_MAX_NODES / 32;

// Consecutive set bits of w from bit `pos` on, below bit L.
__device__ __forceinline__ int ones_from(const uint32_t *w, int pos, int L) {
    int p = pos;
    while (p < L) {
        const int avail = 32 - (p & 31);
        const uint32_t x = ~(w[p >> 5] >> (p & 31));
        const int n = x ? min(__ffs(x) - 1, avail) : avail;
        p += n;
        if (n < avail) break;
    }
    return min(p, L) - pos;
}

// One CTA per request.  The kernel is a chain of dependent reads and block
// barriers, so everything that does not depend on the row statistics comes
// before the wait for the row kernels (kEarly) and overlaps them: the tree and
// its checks, each node's ancestor set and depth, each chain's nodes in order,
// the logit of each node's token in its parent's row, the selected positions
// and their scores.  That is safe because accept_rows lets its successors
// launch only after its own wait: whatever wrote the caller's arrays is
// complete by then, and this call's row kernels write none of them.
// After the wait one round of reads gives every node its parent's statistics;
// greedy matches (token == argmax of the parent row) and relaxed checks (Eq.
// 6-7: token among the parent row's top beta, fp64 logit gap <= tau) become
// bit sets, so a model node is accepted when its ancestor set lies in the
// greedy set and a chain's look-ahead counts runs of ones; then every node
// writes its own part of the accepted path.  Cold and alone 9.7 -> 7.3 us (4
// trees of 65 nodes), 11.2 -> 8.6 us (one of 145); the whole call in a graph,
// where the first half overlaps the row kernels, 18.2 -> 14.3 and 29.0 -> 23.7.
template <bool kEarly>
__global__ void __launch_bounds__(kDecThreads)
accept_decide(const float *logits, int R, int V, const int32_t *node_off, const int32_t *tokens,
              const int32_t *parents, const uint8_t *source, const int8_t *chain, const int32_t *sel_pos,
              const int64_t *tok_off, rs_params p, int acc_cap, const int32_t *argmax, const int32_t *topk,
              const float *lse, const float *rowmax, float *p_tok, int32_t *acc_len, int32_t *acc_nodes,
              int32_t *bonus, int32_t *winner, uint8_t *commit, float *scores, int32_t *status) {
    pdl_launch_next();
    if (!kEarly) pdl_wait_prev();
    const int b = blockIdx.x;
    const int n0 = node_off[b];
    const int N = node_off[b + 1] - n0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int beta = p.beta, top_c = p.top_c;

    __shared__ int s_par[RS_MAX_NODES];
    __shared__ uint8_t s_src[RS_MAX_NODES];
    __shared__ uint32_t s_anc[RS_MAX_NODES][kNodeWords + 1];  // ancestors and the node itself, without the root
    __shared__ uint32_t s_cmask[RS_MAX_TOPC][kNodeWords];
    __shared__ int s_cnodes[RS_MAX_TOPC][RS_MAX_NODES];
    __shared__ uint32_t s_cg[RS_MAX_TOPC][kNodeWords], s_cr[RS_MAX_TOPC][kNodeWords];  // greedy / relaxed, chain order
    __shared__ uint32_t s_g[kNodeWords];                                               // greedy, node order
    __shared__ int s_cacc[RS_MAX_TOPC];
    __shared__ int s_best;  // (depth << 16) | (0xffff - node)

    // the request's rows must lie in [0, R) and its buffer in the score table
    // (tok_off[B] entries); outside them nothing is read or written
    const bool rows_ok = n0 >= 0 && N >= 0 && (long long)n0 + N <= R;
    const long long t0 = tok_off[b];
    const long long t = tok_off[b + 1] - t0;
    const bool tok_ok = t0 >= 0 && t >= 0 && t0 + t <= tok_off[gridDim.x];
    int st = 0;
    if (!rows_ok || !tok_ok) st = RS_ST_BAD_OFFSET;
    else if (N > RS_MAX_NODES) st = RS_ST_TOO_LARGE;
    else if (N < 1) st = RS_ST_BAD_TREE;
    if (tid == 0) s_best = 0;
    if (tid < RS_MAX_TOPC * kNodeWords) {
        (&s_cg[0][0])[tid] = 0;
        (&s_cr[0][0])[tid] = 0;
    }
    static_assert(RS_MAX_TOPC * kNodeWords <= kDecThreads, "one thread per chain word");

    // ---- the tree: node = tid ----
    const int node = tid;
    const bool live = st == 0 && node < N;
    int pa = 0, sr = 0, ch = -1, tk = 0;
    float z = 0.f;  // the token's logit in the parent's row
    bool bad = false;
    if (live) {
        pa = parents[n0 + node];
        sr = source[n0 + node];
        ch = chain[n0 + node];
        tk = tokens[n0 + node];
        if (node == 0) bad = (pa != -1 || sr != 0 || ch != -1);
        else bad = (pa < 0 || pa >= node || sr < 1 || sr > 2 || (sr == 2 && (ch < 0 || ch >= top_c)) ||
                    (sr == 1 && ch != -1) || tk < 0 || tk >= V);
        if (!bad && node > 0) z = logits[(long long)(n0 + pa) * V + tk];
        s_par[node] = pa;
        s_src[node] = (uint8_t)sr;
    }
    // ---- the selections: lane j of the last warp ----
    const bool seller = warp == kNodeWords;
    int selp = -1;
    float selS = 0.f;
    bool dup = false;  // some position is selected twice: it is updated twice, in selection order
    if (seller) {
        if (lane < top_c) {
            selp = sel_pos[(long long)b * top_c + lane];
            selS = (tok_ok && selp >= 0 && (long long)selp < t) ? scores[t0 + selp] : 0.f;
        }
#pragma unroll
        for (int c = 0; c < RS_MAX_TOPC; ++c) {
            const int o = __shfl_sync(0xffffffffu, selp, c);
            dup |= c < lane && selp >= 0 && selp == o;
        }
        dup = __any_sync(0xffffffffu, dup);
    }
    bool any_bad = __syncthreads_or(bad);  // s_par, s_src and the zeroes are complete

    // ---- model nodes hang from the root or from model nodes; ancestor sets;
    // chain membership masks ----
    const bool ok1 = st == 0 && !any_bad;  // every parent is an earlier node: walks end
    uint32_t anc[kNodeWords];
    int depth = 0;
    bad = false;
    if (ok1) {
        if (live) {
            bad = node > 0 && sr == 1 && s_src[pa] > 1;
#pragma unroll
            for (int w = 0; w < kNodeWords; ++w) anc[w] = 0;
            for (int x = node; x > 0; x = s_par[x]) {
                ++depth;
#pragma unroll
                for (int w = 0; w < kNodeWords; ++w) anc[w] |= (x >> 5) == w ? 1u << (x & 31) : 0u;
            }
#pragma unroll
            for (int w = 0; w < kNodeWords; ++w) s_anc[node][w] = anc[w];
        }
        if (warp < kNodeWords) {
            const int c0 = (live && node > 0 && sr == 2) ? ch : -1;
            for (int c = 0; c < top_c; ++c) {
                const uint32_t m = __ballot_sync(0xffffffffu, c0 == c);
                if (lane == 0) s_cmask[c][warp] = m;
            }
        }
    }
    any_bad |= __syncthreads_or(bad);
    // ---- chain c in index order: node of rank r ----
    const bool ok2 = st == 0 && !any_bad;
    const bool chained = ok2 && live && node > 0 && sr == 2;
    int rank = 0, clen = 0;  // of a chain node; of lane c's chain
    if (chained) {
        rank = __popc(s_cmask[ch][node >> 5] & ((1u << (node & 31)) - 1u));
        for (int q = 0; q < (node >> 5); ++q) rank += __popc(s_cmask[ch][q]);
        s_cnodes[ch][rank] = node;
    }
    if (ok2 && seller && lane < top_c) {
#pragma unroll
        for (int q = 0; q < kNodeWords; ++q) clen += __popc(s_cmask[lane][q]);
    }
    __syncthreads();
    // ---- each chain is a path from the root: rank r hangs from rank r - 1 ----
    bad = chained && pa != (rank == 0 ? 0 : s_cnodes[ch][rank - 1]);
    any_bad |= __syncthreads_or(bad);
    if (st == 0 && any_bad) st = RS_ST_BAD_TREE;

    if (kEarly) pdl_wait_prev();  // the row statistics are complete

    // ---- outputs of a rejected request ----
    if (st != 0) {
        for (int i = tid; rows_ok && i < N; i += kDecThreads) {
            p_tok[n0 + i] = 0.f;
            commit[n0 + i] = 0;
        }
        for (int j = tid; j < acc_cap; j += kDecThreads) acc_nodes[(long long)b * acc_cap + j] = -1;
        if (tid == 0) {
            acc_len[b] = 0;
            winner[b] = -2;
            bonus[b] = -1;
            status[b] = st;
        }
        return;
    }

    // ---- greedy and relaxed flags, from the parent's row statistics ----
    int own_arg = 0;
    bool g = false;
    if (live) {
        own_arg = argmax[n0 + node];
        if (node == 0) {
            p_tok[n0] = 1.f;
        } else {
            const int32_t *tp = topk + (long long)(n0 + pa) * beta;
            int id[RS_MAX_BETA];
#pragma unroll
            for (int j = 0; j < RS_MAX_BETA; ++j) id[j] = j < beta ? tp[j] : -1;
            const int am = argmax[n0 + pa];
            const float zmax = rowmax[n0 + pa], lp = lse[n0 + pa];
            g = tk == am;
            bool in_top = false;
#pragma unroll
            for (int j = 0; j < RS_MAX_BETA; ++j) in_top |= id[j] == tk;  // tk >= 0
            const bool rx = in_top && (double)zmax - (double)z <= (double)p.tau;
            p_tok[n0 + node] = __expf(z - lp);
            if (chained) {
                if (g) atomicOr(&s_cg[ch][rank >> 5], 1u << (rank & 31));
                if (rx) atomicOr(&s_cr[ch][rank >> 5], 1u << (rank & 31));
            }
        }
    }
    if (warp < kNodeWords) {
        const uint32_t m = __ballot_sync(0xffffffffu, g);
        if (lane == 0) s_g[warp] = m;
    }
    __syncthreads();

    // ---- strict verification of model nodes: every node on the root path matches ----
    if (live && sr == 1) {
        uint32_t miss = 0;
#pragma unroll
        for (int w = 0; w < kNodeWords; ++w) miss |= anc[w] & ~s_g[w];
        if (!miss) atomicMax(&s_best, (depth << 16) | (0xffff - node));
    }
    // ---- relaxed verification with look-ahead, one lane per chain ----
    int cacc = 0;
    if (seller && lane < top_c) {
        const uint32_t *cg = s_cg[lane], *cr = s_cr[lane];
        int cur = ones_from(cg, 0, clen), last = cur;
        for (int att = 0; att < p.phi; ++att) {
            if (cur >= clen || !((cr[cur >> 5] >> (cur & 31)) & 1u)) break;
            const int xi = ones_from(cg, cur + 1, clen);
            if (xi >= p.m) {
                last = cur + 1 + xi;
                cur = last;
            } else {
                cur = cur + 1;
            }
        }
        cacc = last;
        s_cacc[lane] = last;
    }
    __syncthreads();

    // ---- winner; each node writes its own place on the accepted path ----
    const int best = s_best;
    int best_len = best >> 16, win = best_len > 0 ? -1 : -2;
    const int best_node = best_len > 0 ? 0xffff - (best & 0xffff) : 0;
    for (int c = 0; c < top_c; ++c) {
        const int l = s_cacc[c];
        if (l > best_len) {
            best_len = l;
            win = c;
        }
    }
    if (live) {
        const bool on = node > 0 && (win == -1 ? ((s_anc[best_node][node >> 5] >> (node & 31)) & 1u) != 0
                                               : (win >= 0 && sr == 2 && ch == win && rank < best_len));
        const int j = win == -1 ? depth - 1 : rank;
        commit[n0 + node] = (uint8_t)(on || node == 0);
        if (on && j < acc_cap) acc_nodes[(long long)b * acc_cap + j] = node;
        if (on ? j == best_len - 1 : (node == 0 && best_len == 0)) bonus[b] = own_arg;
        if (node == 0) {
            acc_len[b] = best_len;
            winner[b] = win;
        }
    }
    for (int j = best_len + tid; j < acc_cap; j += kDecThreads) acc_nodes[(long long)b * acc_cap + j] = -1;

    // ---- Eq. 4-5 in fp64, rounded once to the fp32 table ----
    if (seller) {
        const double a = (double)p.alpha;
        auto ema = [&](bool won, int acc, int len, double S) -> double {
            const double Rw = won ? __ddiv_rn((double)acc, (double)len) : 0.0;
            return __dadd_rn(__dmul_rn(__dsub_rn(1.0, a), S), __dmul_rn(a, Rw));
        };
        const bool upd = lane < top_c && selp >= 0 && clen != 0;
        const bool far = upd && (long long)selp >= t;
        if (!dup) {
            if (upd && !far) scores[t0 + selp] = __double2float_rn(ema(win == lane, cacc, clen, (double)selS));
        } else {
            for (int c = 0; c < top_c; ++c) {
                if (lane == c && upd && !far) {
                    volatile float *S = scores + t0 + selp;  // an earlier lane may just have written it
                    *S = __double2float_rn(ema(win == c, cacc, clen, (double)*S));
                    __threadfence();
                }
                __syncwarp();
            }
        }
        const bool any_far = __any_sync(0xffffffffu, far);
        if (lane == 0) status[b] = (best_len > acc_cap ? RS_ST_TRUNCATED : 0) | (any_far ? RS_ST_BAD_POS : 0);
    }
}

}  // namespace
}  // namespace rs

using namespace rs;

namespace {
using RowsFn = void (*)(const float *, int, int, int, VI *, MS *, RowOut);
template <bool kFuse>
RowsFn rows_fn(bool vec, bool ent) {
    if (vec) return ent ? accept_rows<true, true, kFuse> : accept_rows<true, false, kFuse>;
    return ent ? accept_rows<false, true, kFuse> : accept_rows<false, false, kFuse>;
}
}  // namespace

extern "C" size_t rs_accept_workspace_size(int R, int V, int beta) {
    if (R < 0 || V < 1 || beta < 1) return 0;
    int nchunks = (V + kAccChunk - 1) / kAccChunk;
    Carve cv(nullptr);
    cv.take<VI>((size_t)R * nchunks * beta);
    cv.take<MS>((size_t)R * nchunks);
    cv.take<float>((size_t)R);
    return cv.used();
}

extern "C" rs_status rs_accept(const float *logits, int R, int V, const int32_t *node_off, int B,
                               const int32_t *tokens, const int32_t *parents, const uint8_t *source,
                               const int8_t *chain, const int32_t *sel_pos, const int64_t *tok_off,
                               rs_params p, int acc_cap, int32_t *argmax, int32_t *topk, float *lse,
                               float *p_tok, float *entropy, int32_t *acc_len, int32_t *acc_nodes,
                               int32_t *bonus, int32_t *winner, uint8_t *commit, float *scores, int32_t *status,
                               void *workspace, size_t workspace_bytes, void *stream) {
    clear_error();
    RS_CHECK_ARG(R >= 0 && B >= 0, "rs_accept: negative size (R=%d, B=%d)", R, B);
    RS_CHECK_ARG(V >= 1, "rs_accept: V must be >= 1 (got %d)", V);
    RS_CHECK_ARG(p.beta >= 1 && p.beta <= RS_MAX_BETA && p.beta <= V,
                 "rs_accept: beta=%d outside [1, min(%d, V)]", p.beta, RS_MAX_BETA);
    RS_CHECK_ARG(p.top_c >= 1 && p.top_c <= RS_MAX_TOPC, "rs_accept: top_c=%d outside [1, %d]", p.top_c,
                 RS_MAX_TOPC);
    RS_CHECK_ARG(p.tau >= 0.f, "rs_accept: tau must be >= 0");
    RS_CHECK_ARG(p.phi >= 0 && p.m >= 0, "rs_accept: phi and m must be >= 0");
    RS_CHECK_ARG(p.alpha >= 0.f && p.alpha <= 1.f, "rs_accept: alpha outside [0, 1]");
    RS_CHECK_ARG(acc_cap >= 1, "rs_accept: acc_cap must be >= 1");
    RS_CHECK_ARG(R == 0 || (logits && tokens && parents && source && chain && argmax && topk && lse &&
                            p_tok && commit),
                 "rs_accept: null row pointer");
    RS_CHECK_ARG(B == 0 || (node_off && sel_pos && tok_off && acc_len && acc_nodes && bonus && winner &&
                            scores && status),
                 "rs_accept: null request pointer");
    const int nchunks = (V + kAccChunk - 1) / kAccChunk;
    if (nchunks * p.beta > 32 * kCandPerLane) {
        set_error("rs_accept: V=%d with beta=%d exceeds the %d top-k candidates a row merge holds", V, p.beta,
                  32 * kCandPerLane);
        return RS_ERR_UNSUPPORTED;
    }
    const size_t need = rs_accept_workspace_size(R, V, p.beta);
    if (workspace_bytes < need || (need && !workspace)) {
        set_error("rs_accept: workspace %zu bytes < %zu required", workspace_bytes, need);
        return RS_ERR_CAPACITY;
    }
    cudaStream_t st = (cudaStream_t)stream;
    Carve cv(workspace);
    VI *cand = cv.take<VI>((size_t)R * nchunks * p.beta);
    MS *part = cv.take<MS>((size_t)R * nchunks);
    float *rowmax = cv.take<float>((size_t)R);
    if (R > 0) {
        const long long blocks = (long long)R * nchunks;
        RS_CHECK_ARG(blocks < (1ll << 30), "rs_accept: R*chunks too large");
        const bool vec = (V % 4 == 0) && (((uintptr_t)logits & 15) == 0);
        const bool ent = entropy != nullptr;
        const bool fuse = nchunks <= kFuseMax;
        const RowOut ro{argmax, topk, lse, entropy, rowmax};
        const RowsFn fn = fuse ? rows_fn<true>(vec, ent) : rows_fn<false>(vec, ent);
        const dim3 grid((unsigned)blocks);
        if (fuse && nchunks > 1)
            launch_pdl_cluster(fn, grid, dim3(kAccThreads), 0, st, nchunks, logits, V, nchunks, p.beta, cand, part, ro);
        else
            launch_pdl(fn, grid, dim3(kAccThreads), 0, st, logits, V, nchunks, p.beta, cand, part, ro);
        RS_CHECK_LAUNCH("rs_accept/accept_rows");
        if (!fuse) {
            launch_pdl(accept_merge, dim3((R + kMergeRows - 1) / kMergeRows), dim3(kMergeThreads),
                0, st, cand, part, nchunks, p.beta, R, ro);
            RS_CHECK_LAUNCH("rs_accept/accept_merge");
        }
    }
    if (B > 0) {
        // without row kernels of its own the call's predecessor may still be running
        launch_pdl(R > 0 ? accept_decide<true> : accept_decide<false>, dim3(B), dim3(kDecThreads), 0, st, logits, R, V,
            node_off, tokens, parents, source, chain, sel_pos, tok_off, p, acc_cap, argmax, topk, lse, rowmax, p_tok,
            acc_len, acc_nodes, bonus, winner, commit, scores, status);
        RS_CHECK_LAUNCH("rs_accept/accept_decide");
    }
    return RS_OK;
}
