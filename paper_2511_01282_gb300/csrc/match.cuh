// match.cuh -- the part that rs_match_scan and rs_match_scan_indexed share:
// one cluster of CTAs per request tests its candidate positions against the
// key, counts and lists the matches in ascending order, ranks those that clear
// theta_score and gathers the selected continuations.
//
// The candidates come from a source (every position of the buffer, or the
// index's lists) in rows of 128: element e = 0..3 of lane l.  A warp tests
// kRows rows at a time with all their loads in flight; the outcome is four
// ballots per row, kept in shared memory (16 bytes per 128 candidates), so
// that the ascending ranks come from one block scan of popcounts and no
// candidate is tested twice.  A request with few rows is handled by CTA 0
// alone (the others leave at once and no cluster barrier is used); otherwise
// the rows are split evenly, every CTA pushes its count to all peers and its
// best top_c to CTA 0 through distributed shared memory, and after the cluster
// barrier nobody touches another CTA's shared memory.
//
// What bounds it: a chain of dependent reads (offsets, key, candidates,
// scores, spans) of about 0.5 us each and the barriers between them, then for
// long buffers the reads of one request's SMs (~100 GB/s per SM), then, with
// many requests, the CTAs an SM holds.  So calls of few requests take clusters of
// 16 CTAs (match_cluster), of which a request of fewer rows than its source's
// kWideRows uses 8; others clusters of 8.  Scans do so while the GPU runs all of
// them at once, which with 512 threads is 7 (5 and 7 requests of 200000 tokens
// 9.5 and 12.5 us with 8 CTAs, 8.0 and 9.7 with 16; of 1M tokens 33 and 20; but 8
// of 20000 tokens 5.6 and 9.3: the eighth waits), queries up to 4 requests (5 to 14
// would gain 1 us of 7.6 for a text's common token, but short ones lose 0.1 of 4.8,
// and 8 to 14 with many matches 0.4 of 13).  CTAs have 512 threads in the scans of
// up to kMatMidB requests, whose reads in flight bound them (4 x 1M tokens: 17 us,
// 25 with 256), but only 256 stay for a request of one round of these, and 256 are
// launched for everything else: twice the warps at each barrier cost a query of
// 4 x 32K tokens 0.7 of 5.2 us, a scan of 30000 positions 1.0 of 6.8.
#pragma once

#include <cooperative_groups.h>
#include <math.h>
#include <stdlib.h>

#include <mutex>

#include "common.cuh"
#include "match_pos.h"

namespace rs {

constexpr int kMatMidB = 8;
constexpr int kMatThreads = 512, kMatHalf = kMatThreads / 2;
constexpr int kMatWarps = kMatThreads / 32;
constexpr int kMatCand = 512;             // matches ranked from the shared buffer
constexpr int kMatRankAll = 64;           // of which so many at once
constexpr int kMatBitRows = 2048;         // rows whose ballots a CTA keeps (262144 candidates)
constexpr size_t kMatSmem = (size_t)kMatBitRows * 4 * sizeof(uint32_t);

// (s, p) before (s2, p2): higher score first, then the more recent position
__device__ __forceinline__ bool sp_before(float s, int p, float s2, int p2) {
    return s > s2 || (s == s2 && p > p2);
}

// Rank of (s, p) among n distinct (score, position) pairs in shared memory:
// the number of pairs before it in (score desc, position desc) order.
__device__ __forceinline__ int sp_rank(float s, int p, const float *cs, const int *cp, int n) {
    int r = 0;
    for (int q = 0; q < n; ++q) r += sp_before(cs[q], cp[q], s, p);
    return r;
}

struct MatShared {
    float cs[kMatCand];  // matches with S >= theta_score (first kMatCand)
    int cp[kMatCand];
    float gs[kMatCand / 32 * RS_MAX_TOPC];  // the best of every 32 of them
    int gp[kMatCand / 32 * RS_MAX_TOPC];
    int ccnt;
    int warp_sums[kMatWarps];
    float wv[kMatWarps];
    int wp[kMatWarps];
    int peer_cnt[kMatClusterMax];           // match count of each CTA (pushed by its owner)
    float peer_s[kMatClusterMax][RS_MAX_TOPC];    // CTA 0: each CTA's best top_c
    int peer_p[kMatClusterMax][RS_MAX_TOPC];
    int peer_n[kMatClusterMax];
    float top_s[RS_MAX_TOPC];                  // this CTA's best top_c
    int top_p[RS_MAX_TOPC];
    int ntop;
    int sel[RS_MAX_TOPC];
};

struct MatOut {
    int32_t *count, *pos, *sel_pos, *sel_len, *spans, *n_sel, *status;
    float theta_score;
    int top_c, span_len, pos_cap;
};

// The request's token buffer and key, as both kernels read them first.
struct MatReq {
    const int32_t *X;
    const float *S;
    int t;      // tokens (0 for a request that is not read)
    int k, st;  // key length; status bits
    bool run;
    int key[RS_MAX_L];  // key[i] = X[t - k + i]
    int k1, k2;         // its last token, and the one before (-1: none)
    int threads;        // of the CTA at work on it
};

// A retrieval kernel's first act.  The one barrier that no read depends on comes
// before the wait for the predecessor, and no thread stops at it between the
// request's records and its candidates.
__device__ __forceinline__ void mat_enter(MatShared &sh) {
    pdl_launch_next();
    if (threadIdx.x == 0) sh.ccnt = 0;
    __syncthreads();
    pdl_wait_prev();
}

// ok: the caller's own condition for reading the request (its index is valid).
__device__ __forceinline__ void mat_request(MatReq &q, const int32_t *tokens, const int64_t *tok_off,
                                            const int32_t *k_star, const uint8_t *gate_ok, const float *scores, int b,
                                            int B, bool ok) {
    const long long t0 = tok_off[b], t1 = tok_off[b + 1], tend = tok_off[B];
    q.k = k_star[b];
    const bool gate = gate_ok == nullptr || gate_ok[b] != 0;
    const long long t = t1 - t0;
    // the buffers hold tok_off[B] tokens: a range outside them is not read, and
    // neither is one of more tokens than positions can name
    const bool off_ok = ok && t0 >= 0 && (unsigned long long)t <= kMatMaxTokens && t1 <= tend;
    q.X = tokens + (off_ok ? t0 : 0);
    q.S = scores + (off_ok ? t0 : 0);
    q.t = off_ok ? (int)t : 0;
    q.st = 0;
    q.run = off_ok && q.k > 0 && gate;
    if (!off_ok) {
        if (!ok || t0 < 0 || t1 < t0 || t1 > tend) q.st = RS_ST_BAD_OFFSET;
        else if (q.k > 0 && gate) q.st = RS_ST_TOO_LARGE;
    }
    if (q.run && q.k > RS_MAX_L) {
        q.st = RS_ST_TOO_LARGE;
        q.run = false;
    }
    if (q.run && q.k > q.t) q.run = false;
#pragma unroll
    for (int i = 0; i < RS_MAX_L; ++i) q.key[i] = (q.run && i < q.k) ? q.X[q.t - q.k + i] : -1;
    q.k1 = q.run ? q.X[q.t - 1] : -1;
    q.k2 = q.run && q.k > 1 ? q.X[q.t - 2] : -1;
}

// Whether the k - 1 tokens before position p (p >= k - 1) are the key's; every
// load is issued before the first comparison.
__device__ __forceinline__ bool mat_prefix(const MatReq &q, int p) {
    int v[RS_MAX_L];
#pragma unroll
    for (int j = 0; j < RS_MAX_L; ++j) v[j] = j < q.k - 1 ? q.X[p - (q.k - 1) + j] : -1;
    bool m = true;
#pragma unroll
    for (int j = 0; j < RS_MAX_L; ++j) m &= j >= q.k - 1 || v[j] == q.key[j];
    return m;
}

// Exclusive scan of one int per thread over the block; *total gets the sum.
__device__ __forceinline__ int mat_excl_scan(int v, int threads, MatShared &sh, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh.warp_sums[warp] = x;
    __syncthreads();
    int before = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < kMatWarps; ++w) {
        const int y = w < (threads >> 5) ? sh.warp_sums[w] : 0;
        before += w < warp ? y : 0;
        sum += y;
    }
    __syncthreads();  // warp_sums reusable
    *total = sum;
    return before + x - v;
}

// Best head of the block's register lists; every thread gets it.
__device__ __forceinline__ void mat_block_best(float hv, int hp, int threads, MatShared &sh, float *bv, int *bp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, hv, o);
            const int op = __shfl_xor_sync(0xffffffffu, hp, o);
            if (sp_before(ov, op, hv, hp)) {
                hv = ov;
                hp = op;
            }
        }
        if (r == 0) {
            if (lane == 0) {
                sh.wv[warp] = hv;
                sh.wp[warp] = hp;
            }
            __syncthreads();
            hv = lane < (threads >> 5) ? sh.wv[lane] : -INFINITY;
            hp = lane < (threads >> 5) ? sh.wp[lane] : -1;
        }
    }
    __syncthreads();  // wv / wp reusable
    *bv = hv;
    *bp = hp;
}

// The tests of a source's rows [r0, r0 + kRows) by one warp: this lane's hits,
// bit 4 u + e for element e of row r0 + u; rows at or past `end` give none.
// The warp's ballots go to bits[4 (r0 - base) ..] (rows below `end` and the kept ones only).
template <class Src>
__device__ __forceinline__ uint32_t mat_rows(const Src &src, const MatReq &q, int r0, int end, uint32_t *bits,
                                             int base) {
    const int lane = threadIdx.x & 31;
    const uint32_t hits = src.test(q, r0, end, lane);
    uint32_t mine = 0;
    if (!Src::kSparse || __any_sync(0xffffffffu, hits != 0)) {
#pragma unroll
        for (int j = 0; j < 4 * Src::kRows; ++j) {
            const uint32_t bal = __ballot_sync(0xffffffffu, (hits >> j) & 1u);
            mine = lane == j ? bal : mine;
        }
    }
    if (lane < 4 * Src::kRows && r0 + (lane >> 2) < end && r0 - base + (lane >> 2) < kMatBitRows) bits[4 * (r0 - base) + lane] = mine;
    return hits;
}

// The ballots of rows [w0, w0 + nr) again, for slices of more rows than are
// kept (not inlined: the common path keeps its registers).
template <class Src>
__device__ __noinline__ void mat_again(Src src, MatReq q, int w0, int nr, uint32_t *bits) {
    __syncthreads();  // the previous rows are consumed
    const int stride = (q.threads >> 5) * Src::kRows;
    for (int r0 = w0 + (threadIdx.x >> 5) * Src::kRows; r0 < w0 + nr; r0 += stride)
        (void)mat_rows(src, q, r0, w0 + nr, bits, w0);
    __syncthreads();
}

// Calls use(idx, position, load(position)) for the matches of rows [a, z) of the
// kept ballots (by one warp), idx counting them in order from `base`, below `cap`;
// w0: the row the ballots start at.  32 rows at a time, either a lane per row (few matches in
// each: every row's first at once) or row by row with all lanes (many: a
// row's matches at once), whichever takes fewer steps, as each may wait for a
// read: 999 positions of one token in a list took 57 us a lane per row, 12 so.
template <class Src, class L, class U>
__device__ __forceinline__ void mat_each(const Src &src, const uint32_t *bits, int w0, int a, int z, int base, int cap,
                                         L load, U use) {
    auto f = [&](int idx, int p) { use(idx, p, load(p)); };
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    for (int c0 = a; c0 < z && base < cap; c0 += 32) {
        const int own = c0 + lane;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (own < z) w = *reinterpret_cast<const uint4 *>(bits + 4 * own);
        const int n = __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        int idx = base + incl - n;
        base += __shfl_sync(0xffffffffu, incl, 31);
        uint32_t rows = __ballot_sync(0xffffffffu, n > 0 && idx < cap);
        if (__reduce_max_sync(0xffffffffu, (unsigned)n) <= (unsigned)__popc(rows)) {
            if (Src::kLaneMajor) {
                uint32_t any = w.x | w.y | w.z | w.w;
                for (; any && idx < cap; any &= any - 1) {
                    const int l = __ffs(any) - 1;
                    uint32_t es =
                        ((w.x >> l) & 1u) | ((w.y >> l) & 1u) << 1 | ((w.z >> l) & 1u) << 2 | ((w.w >> l) & 1u) << 3;
                    for (; es && idx < cap; es &= es - 1) f(idx++, src.pos(w0 + own, l, __ffs(es) - 1));
                }
            } else {
#pragma unroll 1
                for (int e = 0; e < 4; ++e) {
                    uint32_t we = e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w;
                    for (; we && idx < cap; we &= we - 1) f(idx++, src.pos(w0 + own, __ffs(we) - 1, e));
                }
            }
            __syncwarp();
            continue;
        }
        for (; rows; rows &= rows - 1) {
            const int q = __ffs(rows) - 1, r = c0 + q;
            const uint4 v = *reinterpret_cast<const uint4 *>(bits + 4 * r);
            const uint32_t we[4] = {v.x, v.y, v.z, v.w};
            int at = __shfl_sync(0xffffffffu, idx, q);
            if (Src::kLaneMajor) at += __popc(v.x & lt) + __popc(v.y & lt) + __popc(v.z & lt) + __popc(v.w & lt);
            int p[4], k[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool hit = (we[e] >> lane) & 1u;
                k[e] = Src::kLaneMajor ? at : at + __popc(we[e] & lt);
                at += Src::kLaneMajor ? (int)hit : __popc(we[e]);
                if (!hit) k[e] = cap;
                p[e] = hit ? src.pos(w0 + r, lane, e) : 0;
            }
            float s[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = k[e] < cap ? load(p[e]) : 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (k[e] < cap) use(k[e], p[e], s[e]);
        }
        __syncwarp();
    }
}

// The whole of a request once its source is known (see the file comment).
// rows: candidate rows; nc: the CTAs that share them, 1 for CTA 0 alone.
template <class Src>
__device__ __forceinline__ void mat_body(const Src &src, const MatReq &q, int rows, int nc, int b, int crank,
                                         MatShared &sh, uint32_t *bits, const MatOut &o) {
    namespace cg = cooperative_groups;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nthreads = q.threads;
    const int top_c = o.top_c, pos_cap = o.pos_cap;
    const bool solo = nc == 1;
    if (!solo) cluster_arrive_relaxed();  // this CTA runs; the wait sits before the first push
    const int per = (rows + nc - 1) / nc;
    const int lo = min(per * crank, rows), hi = min(lo + per, rows);

    // ---- every candidate once: ballots, count, the matches that clear theta ----
    // (consecutive rows per warp, as the positions are written)
    const int mr = (hi - lo + (nthreads >> 5) - 1) / (nthreads >> 5);
    const int wa = min(lo + warp * mr, hi), wz = min(wa + mr, hi);
    int cnt = 0;
    for (int r0 = wa; r0 < wz; r0 += Src::kRows) {
        const uint32_t hits = mat_rows(src, q, r0, wz, bits, lo);
        cnt += __popc(hits);
        // their scores, four of each lane at once; one slot count per warp and
        // round.  Once the buffer has run over, its contents count no more
        for (uint32_t rem = hits; __any_sync(0xffffffffu, rem != 0);) {
            if (__any_sync(0xffffffffu, *(volatile int *)&sh.ccnt > kMatCand)) break;
            int p[4], at[4], n = 0;
            float s[4];
            bool pass[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = __ffs(rem) - 1;
                p[e] = rem ? src.pos(r0 + (j >> 2), lane, j & 3) : -1;
                s[e] = rem ? q.S[p[e]] : 0.f;
                rem &= rem - 1;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                pass[e] = p[e] >= 0 && s[e] >= o.theta_score;
                const uint32_t bal = __ballot_sync(0xffffffffu, pass[e]);
                at[e] = n + __popc(bal & ((1u << lane) - 1u));
                n += __popc(bal);
            }
            if (n == 0) continue;
            int slot = 0;
            if (lane == 0) slot = atomicAdd(&sh.ccnt, n);
            slot = __shfl_sync(0xffffffffu, slot, 0);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (pass[e] && slot + at[e] < kMatCand) {
                    sh.cs[slot + at[e]] = s[e];
                    sh.cp[slot + at[e]] = p[e];
                }
            }
        }
    }
    cnt = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
    if (lane == 0) sh.warp_sums[warp] = cnt;
    __syncthreads();
    int cta_total = 0, before = 0;  // before: the matches of the earlier warps
#pragma unroll
    for (int w = 0; w < kMatWarps; ++w) {
        const int y = w < (nthreads >> 5) ? sh.warp_sums[w] : 0;
        before += w < warp ? y : 0;
        cta_total += y;
    }
    // the CTA's best top_c: rank every buffered match by counting
    const int ncand = sh.ccnt;
    const bool over = ncand > kMatCand;
    bool kept = true;  // the ballots are still those of [lo, lo + kMatBitRows)
    if (!over || Src::kBound) {
        const float *cs = sh.cs;
        const int *cp = sh.cp;
        int n = Src::kBound ? min(ncand, kMatCand) : ncand;
        if (n > kMatRankAll) {
            // the best top_c of every 32 first (300 matches of a list: 12.5 us with
            // all ranked against each other, 9.3 so)
            for (int g = warp; g * 32 < n; g += nthreads >> 5) {
                const int e = g * 32 + lane;
                const float sv = e < n ? cs[e] : -INFINITY;
                const int pv = e < n ? cp[e] : -1 - lane;  // after every match
                int r = 0;
#pragma unroll 8
                for (int i = 0; i < 32; ++i)
                    r += sp_before(__shfl_sync(0xffffffffu, sv, i), __shfl_sync(0xffffffffu, pv, i), sv, pv);
                if (r < top_c) {
                    sh.gs[g * top_c + r] = sv;
                    sh.gp[g * top_c + r] = pv;
                }
            }
            __syncthreads();
            n = (n + 31) / 32 * top_c;
            cs = sh.gs;
            cp = sh.gp;
        }
        for (int e = tid; e < n; e += nthreads) {
            const float sv = cs[e];
            const int pv = cp[e];
            const int r = sp_rank(sv, pv, cs, cp, n);
            if (r < top_c) {
                sh.top_s[r] = sv;
                sh.top_p[r] = pv;
            }
        }
        if (tid == 0) sh.ntop = ncand < top_c ? ncand : top_c;
    }
    if (over) {  // more than the buffer holds: every thread's best of its rows, then the block's best of those
        // kBound: only those not behind the best top_c of the buffer (read
        // before the first of these is replaced, behind a barrier): 16 x 300000
        // positions, half of them matches, 98.5 -> 58.7 us
        float ts = -INFINITY;
        int tp = -1;
        if (Src::kBound) {
            __syncthreads();
            ts = sh.top_s[top_c - 1];
            tp = sh.top_p[top_c - 1];
        }
        float ls[RS_MAX_TOPC];
        int lp[RS_MAX_TOPC];
#pragma unroll
        for (int i = 0; i < RS_MAX_TOPC; ++i) {
            ls[i] = -INFINITY;
            lp[i] = -1;
        }
        for (int w0 = lo; w0 < hi; w0 += kMatBitRows) {
            const int nr = min(hi - w0, kMatBitRows);
            if (w0 != lo) {
                mat_again(src, q, w0, nr, bits);
                kept = false;
            }
            const int per_warp = (nr + (nthreads >> 5) - 1) / (nthreads >> 5);
            const int a = min(warp * per_warp, nr), z = min(a + per_warp, nr);
            mat_each(src, bits, w0, a, z, 0, 0x7fffffff, [&](int p) { return q.S[p]; },
                     [&](int, int p, float s) {
                if (s >= o.theta_score && !(Src::kBound && sp_before(ts, tp, s, p)) && sp_before(s, p, ls[RS_MAX_TOPC - 1], lp[RS_MAX_TOPC - 1])) {
                    float cs = s;
                    int cp = p;
#pragma unroll
                    for (int i = 0; i < RS_MAX_TOPC; ++i) {
                        if (sp_before(cs, cp, ls[i], lp[i])) {
                            const float ts = ls[i];
                            const int tp = lp[i];
                            ls[i] = cs;
                            lp[i] = cp;
                            cs = ts;
                            cp = tp;
                        }
                    }
                }
            });
        }
        int ntop = 0;
        for (int c = 0; c < top_c; ++c) {
            float bv;
            int bp;
            mat_block_best(ls[0], lp[0], nthreads, sh, &bv, &bp);
            if (bp < 0) break;
            if (tid == 0) {
                sh.top_s[c] = bv;
                sh.top_p[c] = bp;
            }
            ntop = c + 1;
            if (lp[0] == bp) {  // the owner pops its head
#pragma unroll
                for (int i = 0; i < RS_MAX_TOPC - 1; ++i) {
                    ls[i] = ls[i + 1];
                    lp[i] = lp[i + 1];
                }
                ls[RS_MAX_TOPC - 1] = -INFINITY;
                lp[RS_MAX_TOPC - 1] = -1;
            }
        }
        if (tid == 0) sh.ntop = ntop;
    }

    // ---- the slice's global rank (pushed counts) ----
    int offset = 0, total = cta_total;
    __syncthreads();  // this CTA's top list is complete
    if (!solo) {
        cg::cluster_group cluster = cg::this_cluster();
        cluster_wait();  // every CTA of the cluster is running (or has left: those share no rows)
        if (tid < nc) *cluster.map_shared_rank(&sh.peer_cnt[crank], tid) = cta_total;
        if (tid < RS_MAX_TOPC && tid < sh.ntop) {
            *cluster.map_shared_rank(&sh.peer_s[crank][tid], 0) = sh.top_s[tid];
            *cluster.map_shared_rank(&sh.peer_p[crank][tid], 0) = sh.top_p[tid];
        }
        if (tid == 0) *cluster.map_shared_rank(&sh.peer_n[crank], 0) = sh.ntop;
        cluster_arrive_release();  // every push is visible after the wait
        cluster_wait();
        total = 0;
        for (int r = 0; r < nc; ++r) {
            const int c = sh.peer_cnt[r];
            if (r < crank) offset += c;
            total += c;
        }
    }

    // ---- positions in ascending order ----
    int32_t *pos = o.pos + (long long)b * pos_cap;
    auto none = [](int) { return 0.f; };
    auto put = [&](int i, int p, float) { pos[i] = p; };
    if (kept && hi - lo <= kMatBitRows) {
        if (cnt > 0) mat_each(src, bits, lo, wa - lo, wz - lo, offset + before, pos_cap, none, put);
    } else {
        int base = offset;
        for (int w0 = lo; w0 < hi && base < pos_cap; w0 += kMatBitRows) {
            const int nr = min(hi - w0, kMatBitRows);
            if (w0 != lo || !kept) mat_again(src, q, w0, nr, bits);
            const int per_warp = (nr + (nthreads >> 5) - 1) / (nthreads >> 5);
            const int a = min(warp * per_warp, nr), z = min(a + per_warp, nr);
            int n = 0;
            for (int r = a + lane; r < z; r += 32) {
                const uint4 w = *reinterpret_cast<const uint4 *>(bits + 4 * r);
                n += __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
            }
            int wtotal = 0;
            const int idx = __shfl_sync(0xffffffffu, base + mat_excl_scan(n, nthreads, sh, &wtotal), 0);
            mat_each(src, bits, w0, a, z, idx, pos_cap, none, put);
            base += wtotal;
        }
    }
    if (crank != 0) return;

    // ---- CTA 0: merge the per-CTA lists, selection outputs ----
    for (int i = min(total, pos_cap) + tid; i < pos_cap; i += nthreads) pos[i] = -1;
    int nsel;
    if (solo) {
        nsel = sh.ntop;
        if (tid < nsel) sh.sel[tid] = sh.top_p[tid];  // already ranked
    } else {
        // the cluster's candidates (at most kMatClusterMax * RS_MAX_TOPC), ranked by counting
        float *ms = sh.cs;  // reused: the CTA's own buffer is no longer needed
        int *mp = sh.cp;
        int nm = 0;
        for (int r = 0; r < nc; ++r) {
            const int n = sh.peer_n[r];
            if (tid < n) {
                ms[nm + tid] = sh.peer_s[r][tid];
                mp[nm + tid] = sh.peer_p[r][tid];
            }
            nm += n;
        }
        __syncthreads();
        if (tid < nm) {
            const int r = sp_rank(ms[tid], mp[tid], ms, mp, nm);
            if (r < top_c) sh.sel[r] = mp[tid];
        }
        nsel = nm < top_c ? nm : top_c;
    }
    __syncthreads();
    for (int i = tid; i < top_c * o.span_len; i += nthreads) {
        const int c = i / o.span_len, j = i - c * o.span_len;
        int v = -1;
        if (c < nsel) {
            const int p = sh.sel[c];
            if (j < q.t - 1 - p) v = q.X[p + 1 + j];
        }
        o.spans[(long long)b * top_c * o.span_len + i] = v;
    }
    if (tid < top_c) {
        int sp = -1, sl = 0;
        if (tid < nsel) {
            sp = sh.sel[tid];
            sl = min(q.t - 1 - sp, o.span_len);
        }
        o.sel_pos[(long long)b * top_c + tid] = sp;
        o.sel_len[(long long)b * top_c + tid] = sl;
    }
    if (tid == 0) {
        o.count[b] = total;
        o.n_sel[b] = nsel;
        o.status[b] = q.st | (total > pos_cap ? RS_ST_TRUNCATED : 0);
    }
}

// The CTAs of the cluster that share a request's rows: one round of CTA 0's
// warps needs no others.
template <class Src>
__device__ __forceinline__ int mat_ctas(int rows, int threads) {
    if (rows <= (threads >> 5) * Src::kRows) return 1;
    const int nc = gridDim.x;
    return nc > kMatCluster && rows < Src::kWideRows ? kMatCluster : nc;
}

static_assert(sizeof(MatShared) + kMatSmem <= 48 * 1024, "within what a kernel may use without asking");

// How many clusters of kMatClusterMax CTAs the current context can run at once: 0
// where it has no GPC of so many SMs (a part of a GPU).  Remembered with the
// context's id, as the attribute that allows them goes with the context.
// RS_DEBUG_MATCH_CLUSTER=8 (a test hook, read where this is asked) answers 0.
class MatWide {
    std::mutex mu_;
    unsigned long long ctx_[64] = {};
    int n_[64] = {};

public:
    int ask(const void *kern, int threads) {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
        const unsigned long long id = context_id();
        std::lock_guard<std::mutex> lk(mu_);
        if (id != 0 && ctx_[dev] == id) return n_[dev];
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kMatClusterMax);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = kMatSmem;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kMatClusterMax;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
            n = 0;
            (void)cudaGetLastError();  // smaller clusters do as well
        }
        if (const char *e = getenv("RS_DEBUG_MATCH_CLUSTER"))
            if (atoi(e) == kMatCluster) n = 0;
        n_[dev] = n;
        ctx_[dev] = context_id();  // the questions made the context current if it was not
        return n;
    }
};

// Launches the retrieval kernel of a source over B requests; wide: the kernel's own.
template <class Src, typename... KArgs, typename... Args>
inline rs_status mat_launch(const char *who, MatWide &wide, void (*kern)(KArgs...), int B, cudaStream_t st, Args... args) {
    const int nc = match_cluster(B, Src::kFewB, B <= Src::kFewB ? wide.ask(reinterpret_cast<const void *>(kern), Src::kThreads) : 0);
    const int threads = B <= kMatMidB ? Src::kThreads : kMatHalf;
    launch_pdl_cluster(kern, dim3(nc, B), dim3(threads), kMatSmem, st, nc, args...);
    RS_CHECK_LAUNCH(who);
    return RS_OK;
}

}  // namespace rs
