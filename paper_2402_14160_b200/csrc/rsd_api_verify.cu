// C ABI of librsd (declared in include/rsd.h), verification half: rsd_verify_tree, rsd_verify_tree_rule and
// rsd_resample_residual.  Argument checks and kernel launches, nothing else.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

#include "rsd_api_common.h"
#include "rsd_verify.cuh"
#include "rsd_walk_cluster_args.h"
#include "rsd_walk_ring.cuh"

using namespace rsd_host;

namespace {
// The walk fed by the copy engine (rsd_walk_ring.cuh); a launch error stays pending for check_launch().
template <typename T>
void launch_ring_walk(const rsd::VerifyArgs& a, int B, cudaStream_t s) {
    using namespace rsd::walk_ring;
    // The attribute belongs to the (function, device) pair and setting it costs host time: once per device.
    static std::atomic<bool> raised[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    if (dev < 0 || dev >= 64 || !raised[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(verify_tree_ring_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes) != cudaSuccess)
            return;
        if (dev >= 0 && dev < 64) raised[dev].store(true, std::memory_order_release);
    }
    launch_overlapped(verify_tree_ring_kernel<T>, (unsigned)B, kThreads, kRingBytes, s, 0, a);
}

// The cluster that holds a row on chip.  Fewer tiles per warp walk faster, more leave room for more sequences at a time (148 SMs, 32,000
// entries; bf16 multi-round rule over (3, 2) trees, us at 40 / 75 / 148 / 222 sequences): one tile per warp, eight blocks, 48 resident: 15.6 / 28 / 48 / 68;
// two, four blocks, 71 resident: 17.0 / 28 / 41 / 53; four, two blocks, 148 resident: 21 / 23 / 26 / 46.  So the first of them that has all
// sequences resident, else the one with the most.  Rows of up to 8192 entries are held by one or two blocks with one tile per warp; beyond its
// residents that one stays ahead (V = 8096, 492 sequences: two blocks 57 us, one 63 us).  Rows beyond 65,536 entries: sixteen warps
// with two tiles (15 resident; 128,000 entries, 9 / 18 / 32 sequences 21 / 33 / 54 us), eight with four (33 resident; 22 / 25 / 31); beyond 131,072 no
// cluster holds them (C = 0).
rsd::walk_cluster::Shape cluster_shape(int B, int V) {
    rsd::walk_cluster::Shape best = {0, 0, 0, 0.0f};
    auto consider = [&](int W, int NT) {        // true: all sequences are resident
        int c = 1;
        while (c * W * NT * 512 < V) c *= 2;
        if (c > 8) return false;
        const rsd::walk_cluster::Shape s = {c, W, NT, (float)B / (float)rsd::walk_cluster::resident_clusters(c, W, NT)};
        if (best.C == 0 || V > 8192 || s.waves <= 1.0f) best = s;
        return s.waves <= 1.0f;
    };
    if (V > 65536) {
        if (!consider(16, 2)) consider(8, 4);
    } else if (!consider(8, 1) && !consider(8, 2) && V > 8192) {
        consider(8, 4);
    }
    return best;
}

// Whether the on-chip walk is taken, or else the ring walk or the one that reads its rows anew in every pass.
// Where fewer than four tiles per warp hold all sequences at a time it always is: in 7,500 such calls the other route took 1.02 to 15 times
// as long.  Rows of up to 8192 entries (a cluster of one or two blocks with one tile per warp) stay on chip, but where the ring takes them it is ahead
// from 1.3 waves on (8192 bf16, 260 / 300 sequences: 24 / 19 us on chip / ring, 24 / 21), and residual draws over 2-byte rows with two blocks a
// sequence meet a wave's end (8192, 200 / 300: 12.6 / 19 on chip / read anew, 22 / 22).
// With four tiles per warp two costs are compared.  A launch on chip takes as long as it has waves of clusters, each about the same whatever the row
// (sequences asked for over sequences resident); the other route as long as it has rounds of blocks (three or, for 4-byte rows read anew, two
// per SM), each in proportion to a constant and the row.  Sequences end at different times, so that half of a wave counts by its
// share and half as a whole one.  A round's cost in waves is a + b V / 10,000; a residual draw's pass over its rejected tokens raises it with the fourth root
// of their number.  Fitted to 12,100 calls with both routes timed (8,193 to 131,072 entries, 8 to 900 sequences, trees of 4 to 29 nodes, 1 to 32
// rejected tokens): the route taken is 0.7 % slower than the faster one in geometric mean (the limits per cluster size before: 2.7 %), and 54
// calls are more than a tenth slower than in the walks without a four-tile shape (222 before).
enum WalkKind { kRingRows, kReadAnew, kReadAnewTop1, kDraw, kDrawWhole };
bool on_chip_pays(const rsd::walk_cluster::Shape& c, int B, int V, bool f32, WalkKind kind, int rejected) {
    if (c.C == 0) return false;
    if (c.NT == 1 && V <= 8192) {
        if (kind == kRingRows) return c.waves <= 1.3f;
        if (kind == kDraw && c.C == 2 && !f32) return c.waves <= std::max(1.0f, 0.2f + (float)V / 9000.0f);
        return true;
    }
    if (c.NT < 4) return c.waves <= 1.0f;
    static const float cost[5][2][2] = {                 // [kind][4-byte rows]: a, b
        {{0.75f, 0.22f}, {0.60f, 0.40f}}, {{0.55f, 0.36f}, {0.30f, 0.52f}}, {{0.65f, 0.68f}, {0.80f, 0.60f}}, {{1.05f, 0.28f}, {0.65f, 0.68f}}, {{1.10f, 0.46f}, {0.75f, 1.00f}}};
    auto counted = [](float n) { return 0.5f * (std::ceil(n) + std::max(n, 1.0f)); };
    const float rounds = counted((float)B / (float)((f32 && kind != kRingRows ? 2 : 3) * sm_count()));
    const float passes = kind >= kDraw ? std::sqrt(std::sqrt((float)rejected / 3.0f)) : 1.0f;
    return counted(c.waves) <= rounds * passes * (cost[kind][f32][0] + cost[kind][f32][1] * (float)V / 10000.0f);
}

void launch_on_chip(const rsd::walk_cluster::ClusterArgs& a, int dtype, bool extra, int B, const rsd::walk_cluster::Shape& c, cudaStream_t s) {
    if (dtype == RSD_F32) rsd::walk_cluster::launch_f32(a, extra, B, c, s);
    else rsd::walk_cluster::launch_bf16(a, extra, B, c, s);
}

// Rows that no cluster holds: eight blocks a sequence up to about as many sequences as SMs (151,936 entries, us with eight blocks / one, 148
// sequences: residual draw fp32 251 / 259, multi-round 153 / 177; 222: 357 / 299, 220 / 194), plain walks up to half as many more
// (fp32, 222 / 256 sequences: 231 / 249, 262 / 258).
// 2-byte rows, one block a sequence: a block takes about 1.2 times as long where three share an SM (rsd_walk_stream.cuh), so three
// where that saves waves: multi-round over 32,000, 256 / 300 / 500 / 600 sequences 67 / 94 / 103 / 127 with two, 72 / 77 / 112 / 121 with three.
void launch_streamed(const rsd::walk_cluster::ClusterArgs& a, int dtype, bool extra, int B, bool fits_cluster, cudaStream_t s) {
    const int sms = sm_count();
    const int C = !fits_cluster && B <= (extra ? sms : sms + sms / 2) ? 8 : 1;
    const int waves2 = (B + 2 * sms - 1) / (2 * sms), waves3 = (B + 3 * sms - 1) / (3 * sms);
    if (dtype == RSD_F32) rsd::walk_cluster::launch_stream_f32(a, extra, B, C, 2, s);
    else rsd::walk_cluster::launch_stream_bf16(a, extra, B, C, 6 * waves3 < 5 * waves2 ? 3 : 2, s);
}
}  // namespace

extern "C" {

int rsd_verify_tree(const rsd_rows* draft, const rsd_rows* target, const rsd_tree* tree, int B, int V, uint64_t seed,
                    uint32_t step, uint32_t seq_base, int32_t* accepted_len, int32_t* accepted_node,
                    int32_t* accepted_token, int32_t* last_token, int32_t* stop_reason, float* dbg_theta,
                    int32_t* status, rsd_stream_t stream) {
    return rsd_verify_tree_rule(draft, target, tree, B, V, RSD_RULE_RRS, 1.0f, RSD_FINAL_INVERSE_CDF, seed, step, seq_base, accepted_len,
                                accepted_node, accepted_token, last_token, stop_reason, dbg_theta, status, stream);
}

int rsd_verify_tree_rule(const rsd_rows* draft, const rsd_rows* target, const rsd_tree* tree, int B, int V, int rule,
                         float gamma, int final_sampler, uint64_t seed, uint32_t step, uint32_t seq_base, int32_t* accepted_len,
                         int32_t* accepted_node, int32_t* accepted_token, int32_t* last_token, int32_t* stop_reason,
                         float* dbg_theta, int32_t* status, rsd_stream_t stream) {
    g_err[0] = 0;
    if (rule != RSD_RULE_RRS && rule != RSD_RULE_MULTIROUND && rule != RSD_RULE_KSEQ)
        return fail(RSD_ERR_INVALID_ARG, "unknown verification rule %d", rule);
    if (final_sampler != RSD_FINAL_INVERSE_CDF && final_sampler != RSD_FINAL_GUMBEL_TOP1)
        return fail(RSD_ERR_INVALID_ARG, "unknown sampler of the last token %d", final_sampler);
    if (rule == RSD_RULE_KSEQ && !(gamma >= 1.0f && gamma < 3.0e38f))
        return fail(RSD_ERR_INVALID_ARG, "K-SEQ: gamma = %g must be a finite number >= 1", (double)gamma);
    if (int e = check_vocab(V)) return e;
    if (int e = check_rows("draft", draft, V, true)) return e;
    if (int e = check_rows("target", target, V, true)) return e;
    if (draft->dtype != target->dtype) return fail(RSD_ERR_UNSUPPORTED, "draft and target rows must have the same dtype");
    if (!tree || !tree->parent || !tree->token) return fail(RSD_ERR_INVALID_ARG, "null tree");
    if (tree->num_levels < 0 || tree->num_nodes < 1 || tree->num_nodes > RSD_MAX_TREE_NODES)
        return fail(RSD_ERR_UNSUPPORTED, "num_levels = %d, num_nodes = %d", tree->num_levels, tree->num_nodes);
    if (B < 0) return fail(RSD_ERR_INVALID_ARG, "B = %d", B);
    if (!accepted_len || !accepted_node || !accepted_token || !last_token || !stop_reason || !status) return fail(RSD_ERR_INVALID_ARG, "null output");
    if (B == 0) return RSD_OK;
    rsd::VerifyArgs a;
    a.draft = {draft->data, draft->seq_stride, draft->row_stride, 1.0f / temperature_of(draft)};
    a.target = {target->data, target->seq_stride, target->row_stride, 1.0f / temperature_of(target)};
    a.V = V; a.L = tree->num_levels; a.num_nodes = tree->num_nodes; a.shared_topology = tree->topology_is_shared;
    a.rule = rule; a.gamma = rule == RSD_RULE_KSEQ ? gamma : 1.0f; a.final_sampler = final_sampler;
    a.parent = tree->parent; a.token = tree->token;
    a.seed_lo = (uint32_t)seed; a.seed_hi = (uint32_t)(seed >> 32); a.step = step; a.seq_base = seq_base;
    a.accepted_len = accepted_len; a.accepted_node = accepted_node; a.accepted_token = accepted_token;
    a.last_token = last_token; a.stop_reason = stop_reason; a.dbg_theta = dbg_theta; a.status = status;
    cudaStream_t s = (cudaStream_t)stream;
    const bool aligned = rows_aligned(draft) && rows_aligned(target);
    const bool plain = rule == RSD_RULE_RRS && final_sampler == RSD_FINAL_INVERSE_CDF;
    // the ring walk: rows on 16-byte boundaries, of at most 64 chunks (it keeps its chunks as bits of one word)
    const size_t row_bytes = (size_t)V * (draft->dtype == RSD_F32 ? 4 : 2);
    const bool ring = plain && aligned && (row_bytes + rsd::walk_ring::kRowChunkBytes - 1) / rsd::walk_ring::kRowChunkBytes <= 64;
    // The ring's sums and those of the other two are the same for the rows that it takes (ring_rows), and those of the other two
    // always: a batch and its parts give the same bits.
    const rsd::walk_cluster::Shape shape = cluster_shape(B, V);
    const WalkKind kind = ring ? kRingRows : final_sampler == RSD_FINAL_GUMBEL_TOP1 ? kReadAnewTop1 : kReadAnew;
    const bool on_chip = on_chip_pays(shape, B, V, draft->dtype == RSD_F32, kind, 0);
    rsd::walk_cluster::ClusterArgs ca;
    memset(&ca, 0, sizeof(ca));
    ca.v = a;
    ca.ring_rows = ring ? 1 : 0;
    if (on_chip) {
        launch_on_chip(ca, draft->dtype, !plain, B, shape, s);
    } else if (!ring) {
        launch_streamed(ca, draft->dtype, !plain, B, shape.C > 0, s);
    } else {
        if (draft->dtype == RSD_F32) launch_ring_walk<float>(a, B, s);
        else launch_ring_walk<__nv_bfloat16>(a, B, s);
    }
    return check_launch("rsd_verify_tree_rule");
}

int rsd_resample_residual(const rsd_rows* draft_row, const rsd_rows* target_row, int B, int V, const int32_t* rejected,
                          int max_k, const int32_t* rng_node, uint64_t seed, uint32_t step, uint32_t seq_base,
                          int32_t* out_token, float* out_residual, int32_t* status, rsd_stream_t stream) {
    g_err[0] = 0;
    if (int e = check_vocab(V)) return e;
    if (int e = check_rows("target_row", target_row, V, false)) return e;
    if (rejected) {
        if (int e = check_rows("draft_row", draft_row, V, false)) return e;
        if (draft_row->dtype != target_row->dtype) return fail(RSD_ERR_UNSUPPORTED, "draft and target rows must have the same dtype");
        if (max_k < 1 || max_k > RSD_MAX_K) return fail(RSD_ERR_UNSUPPORTED, "max_k = %d outside [1, %d]", max_k, (int)RSD_MAX_K);
    }
    if (B < 0) return fail(RSD_ERR_INVALID_ARG, "B = %d", B);
    if (!rng_node || !out_token || !status) return fail(RSD_ERR_INVALID_ARG, "null argument");
    if (B == 0) return RSD_OK;
    rsd::ResampleArgs a;
    a.target = {target_row->data, target_row->seq_stride, 0, 1.0f / temperature_of(target_row)};
    a.draft = rejected ? rsd::RowsDev{draft_row->data, draft_row->seq_stride, 0, 1.0f / temperature_of(draft_row)} : a.target;
    a.V = V; a.max_k = rejected ? max_k : 0; a.rejected = rejected; a.rng_node = rng_node;
    a.seed_lo = (uint32_t)seed; a.seed_hi = (uint32_t)(seed >> 32); a.step = step; a.seq_base = seq_base;
    a.out_token = out_token; a.out_residual = out_residual; a.status = status;
    cudaStream_t s = (cudaStream_t)stream;
    // A draw with nothing rejected is one sweep over the target row: a block per sequence, but a cluster for the few sequences of
    // rows beyond 16,384 entries that are resident at once (us, cluster / block, bf16: 32,000 entries, 1 / 64 / 148 sequences 6.2 / 7.3 / 20,
    // 6.8 / 7.0 / 7.1; 128,000, 1 / 16 / 64: 7.2 / 15 / 36, 17 / 17 / 17).  So, too, with four tiles per warp: eight blocks 0.34 to 0.67 of the block's time
    // (90,624 entries with the distribution, 16 sequences, bf16: 13 / 36), four 0.6 to 0.75 with the distribution, without it 0.9 for 4-byte rows and 1.2 for 2-byte ones.
    rsd::walk_cluster::ClusterArgs ca;
    memset(&ca, 0, sizeof(ca));
    ca.r = a;
    ca.resample = 1;
    ca.v.draft = a.draft; ca.v.target = a.target;
    ca.v.V = V; ca.v.num_nodes = 1;
    ca.v.seed_lo = a.seed_lo; ca.v.seed_hi = a.seed_hi; ca.v.step = step; ca.v.seq_base = seq_base;
    const rsd::walk_cluster::Shape shape = cluster_shape(B, V);
    const bool f32 = target_row->dtype == RSD_F32;
    const bool draw_on_chip = shape.C > 2 && shape.waves <= 1.0f && (shape.NT < 4 || shape.C == 8 || f32 || out_residual);
    if (!a.max_k && !draw_on_chip) {
        if (f32) rsd::walk_cluster::launch_draw_f32(a, B, s);
        else rsd::walk_cluster::launch_draw_bf16(a, B, s);
    } else if (!a.max_k || on_chip_pays(shape, B, V, f32, out_residual ? kDrawWhole : kDraw, a.max_k)) {
        launch_on_chip(ca, target_row->dtype, true, B, shape, s);
    } else {
        launch_streamed(ca, target_row->dtype, true, B, shape.C > 0, s);
    }
    return check_launch("rsd_resample_residual");
}

}  // extern "C"
