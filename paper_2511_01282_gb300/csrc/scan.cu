// scan.cu -- rs_match_scan: retrieval and feedback-driven candidate
// selection (Section 3.3 "Selection Algorithm"; Algorithm 1's retrieval).
//
// One cluster of CTAs per request; match.cuh has the split, the ranks and
// the selection.  The candidates are the buffer's positions, as quads of four
// tokens on 16-byte boundaries: a lane reads four quads (one 128-bit load
// each, all in flight), compares the last token of the key, filters on the
// one before it from its neighbour's register, and only what is left reads
// the other key tokens and, if it matches, its score.  Nothing is staged in
// shared memory and nothing is read twice.  Staging 8192-position windows of
// tokens and scores (4-byte asynchronous copies, a second staging for the
// positions) took 47 us on 4 x 262144 tokens of text, a key of two; this takes
// 7.3 (graph), the reads of 64 SMs at 4 MB and the dependent rounds around
// them.  Short calls take as long as they did: no match in 300 tokens of one
// request 3.4 us (3.3 before), in 2000 of 16 requests 3.7 (4.3).
#include "match.cuh"

namespace rs {
namespace {

struct ScanSource {
    // (eight rows: 2 x 1.3M tokens 17.6 us instead of 18.8, but every call of a
    // round or two 1.2 us longer)
    static constexpr int kRows = 4;
    static constexpr int kThreads = kMatThreads, kFewB = kMatMidB;
    static constexpr int kWideRows = 1024;  // 131072 positions: below, 8 CTAs are as fast as 16
    static constexpr bool kLaneMajor = true;
    // most rows of a scan hold no match and need no ballots (4 x 262144 tokens of
    // text 7.8 -> 7.3 us, no match in 2000 tokens 3.6 -> 3.4; 0.03 more where all do)
    static constexpr bool kSparse = true;
    static constexpr bool kBound = true;
    ScanPos at;
    __device__ __forceinline__ int pos(int row, int lane, int e) const { return (int)(at.quad(row, lane) + (uint32_t)e); }
    __device__ __forceinline__ uint32_t test(const MatReq &q, int r0, int end, int lane) const {
        const uint32_t pb = at.quad(r0, lane);  // this lane's first position; row u's at pb + 128 u
        const int rows = min(end - r0, kRows);
        int4 x[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const uint32_t p0 = pb + 128u * u;
            x[u] = make_int4(0, 0, 0, 0);
            if (u < rows) {
                if (at.whole(p0)) {
                    x[u] = *reinterpret_cast<const int4 *>(q.X + p0);
                } else {  // the quad reaches past an end of the buffer
                    if (at.in(p0)) x[u].x = q.X[p0];
                    if (at.in(p0 + 1u)) x[u].y = q.X[p0 + 1u];
                    if (at.in(p0 + 2u)) x[u].z = q.X[p0 + 2u];
                    if (at.in(p0 + 3u)) x[u].w = q.X[p0 + 3u];
                }
            }
        }
        const int kl = q.k1, k2 = q.k2;
        const bool one = q.k < 2;
        uint32_t hits = 0;
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const int before = __shfl_up_sync(0xffffffffu, x[u].w, 1);
            const bool m0 = x[u].x == kl && (one || lane == 0 || before == k2);  // lane 0: not in a register
            const bool m1 = x[u].y == kl && (one || x[u].x == k2);
            const bool m2 = x[u].z == kl && (one || x[u].y == k2);
            const bool m3 = x[u].w == kl && (one || x[u].z == k2);
            hits |= ((m0 ? 1u : 0u) | (m1 ? 2u : 0u) | (m2 ? 4u : 0u) | (m3 ? 8u : 0u)) << (4 * u);
        }
        // what is left is checked one by one: the range of matches (k - 1 ..
        // t - 2), which the positions not loaded miss, and the key tokens the
        // registers did not show
        for (uint32_t rem = hits; rem; rem &= rem - 1) {
            const int j = __ffs(rem) - 1;
            const uint32_t p = pb + 128u * (uint32_t)(j >> 2) + (uint32_t)(j & 3);
            bool ok = (j >> 2) < rows && at.end(p, q.k);
            if (ok && !(one || (q.k == 2 && (lane != 0 || (j & 3) != 0)))) ok = mat_prefix(q, (int)p);
            if (!ok) hits &= ~(1u << j);
        }
        return hits;
    }
};

__global__ void __launch_bounds__(kMatThreads)
match_scan_kernel(const int32_t *tokens, const int64_t *tok_off, const int32_t *k_star, const uint8_t *gate_ok,
                  const float *scores, MatOut o) {
    __shared__ MatShared sh;
    mat_enter(sh);
    extern __shared__ __align__(16) uint32_t scan_bits[];
    const int crank = (int)cooperative_groups::this_cluster().block_rank();
    const int b = blockIdx.y;
    MatReq q;
    mat_request(q, tokens, tok_off, k_star, gate_ok, scores, b, gridDim.y, true);
    ScanSource src{ScanPos{(uint32_t)q.t, (uint32_t)(reinterpret_cast<uintptr_t>(q.X) >> 2) & 3u}};
    const int rows = q.run ? (int)src.at.rows() : 0;
    // with one round of half the warps of eight CTAs the other warps leave: they
    // would only make every barrier longer
    q.threads = rows <= kMatCluster * (kMatHalf / 32) * ScanSource::kRows ? kMatHalf : (int)blockDim.x;
    const int nc = mat_ctas<ScanSource>(rows, q.threads);
    if (crank >= nc || (int)threadIdx.x >= q.threads) return;
    mat_body(src, q, rows, nc, b, crank, sh, scan_bits, o);
}

}  // namespace
}  // namespace rs

using namespace rs;

extern "C" size_t rs_match_scan_workspace_size(int B) {
    (void)B;
    return 0;
}

extern "C" rs_status rs_match_scan(const int32_t *tokens, const int64_t *tok_off, int B, const int32_t *k_star,
                                   const uint8_t *gate_ok, const float *scores, rs_params p, int pos_cap,
                                   int32_t *count, int32_t *pos, int32_t *sel_pos, int32_t *sel_len,
                                   int32_t *spans, int32_t *n_sel, int32_t *status, void *workspace,
                                   size_t workspace_bytes, void *stream) {
    clear_error();
    (void)workspace;
    (void)workspace_bytes;
    RS_CHECK_ARG(B >= 0, "rs_match_scan: negative B");
    RS_CHECK_ARG(B <= 65535, "rs_match_scan: B=%d above 65535", B);
    RS_CHECK_ARG(pos_cap >= 0, "rs_match_scan: negative pos_cap");
    RS_CHECK_ARG(p.top_c >= 1 && p.top_c <= RS_MAX_TOPC, "rs_match_scan: top_c=%d outside [1, %d]", p.top_c,
                 RS_MAX_TOPC);
    RS_CHECK_ARG(p.span_len >= 1 && p.span_len <= RS_MAX_SPAN, "rs_match_scan: span_len=%d outside [1, %d]",
                 p.span_len, RS_MAX_SPAN);
    RS_CHECK_ARG(B == 0 || (tokens && tok_off && k_star && scores && count && sel_pos && sel_len && spans &&
                            n_sel && status && (pos || pos_cap == 0)),
                 "rs_match_scan: null pointer");
    if (B == 0) return RS_OK;
    const MatOut o{count, pos, sel_pos, sel_len, spans, n_sel, status, p.theta_score, p.top_c, p.span_len, pos_cap};
    static MatWide wide;
    return mat_launch<ScanSource>("rs_match_scan", wide, match_scan_kernel, B, (cudaStream_t)stream, tokens, tok_off, k_star, gate_ok,
                                  scores, o);
}
