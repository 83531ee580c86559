// C ABI of librsd (declared in include/rsd.h), verification half: rsd_verify_tree, rsd_verify_tree_rule and
// rsd_resample_residual.  Argument checks and kernel launches, nothing else.
#include <algorithm>
#include <atomic>
#include <cstring>

#include "rsd_api_common.h"
#include "rsd_verify.cuh"
#include "rsd_walk_cluster_args.h"
#include "rsd_walk_ring.cuh"

using namespace rsd_host;

namespace {
// SMs of the current device (asked once per device; 148 if the query fails)
int sm_count() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (cached[dev] == 0) {
        int n = 0;
        cached[dev] = (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) ? n : 148;
    }
    return cached[dev];
}

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

// The smallest cluster that holds a row, with one tile per warp (three blocks an SM) as long as all sequences are
// resident at once, else with two (two blocks an SM), which costs a sequence about 10 % more time and 25 % fewer SM-cycles
// (V = 32,000, bf16: 42 against 47 us at 64 sequences, 122 against 102 us at 256).  Rows of up to 8192 entries stay with one
// tile per warp: a cluster of one block has nobody to share with (V = 8096, 492 sequences: two blocks 57 us, one 63 us).
// Rows beyond 65,536 entries take sixteen warps, one block an SM; beyond 131,072 no cluster holds them (C = 0).
rsd::walk_cluster::Shape cluster_shape(int B, int V) {
    auto blocks = [&](int per_block) {
        int c = 1;
        while (c * per_block < V) c *= 2;
        return c;
    };
    const float sms = (float)sm_count();
    int c = blocks(8 * 512);
    if (c <= 2 || (c <= 8 && (float)B * (float)c <= 3.0f * sms)) return {c, 8, 1, (float)B * (float)c / (3.0f * sms)};
    c = blocks(16 * 512);
    if (c <= 8) return {c, 8, 2, (float)B * (float)c / (2.0f * sms)};
    c = blocks(32 * 512);
    if (c <= 8) return {c, 16, 2, (float)B * (float)c / sms};
    return {0, 0, 0, 0.0f};
}

// Up to how many waves of clusters the on-chip walk is taken.
//   Rows that the ring takes (us, ring / cluster): from about two waves on the ring is ahead (trees of (3, 2, 2) / (4, 2, 2, 1, 1) / (3, 2, 1);
// 32,000 bf16 entries, 130 sequences: 36 / 37, 51 / 49, 41 / 34, 148: 36 / 44, 53 / 59, 41 / 44; fp32, 148: 47 / 48, 71 / 63, 51 / 47; 64,000 bf16, 80:
// 53 / 51, 78 / 63, 54 / 50), with clusters of one or two blocks from 1.3 (16,000 bf16, 180: 35 / 34, 44 / 41, 32 / 31, 222: 36 / 37, 47 / 49, 33 / 34).
//   Others: clusters of one or two blocks stay (8001 entries, 300 / 1000: 34 / 89 on chip, 41 / 102 read anew).  Beyond, a launch on
// chip takes as long as it has waves, one that reads the rows anew as long as they are, up to the 296 or 444 sequences that are
// resident at once: 20,000 entries, multi-round, 148 / 222: 46 / 66 on chip, 43 / 49 read anew; 32,001, plain, 200 / 250: 68 / 88, 73 / 75;
// 65,001, 148 / 200: 124 / 160, 134 / 150; 100,000, 80 / 128: 139 / 228, 149 / 151, fp32 128: 270, 275.
//   Gumbel-Top-1 draws take two rounds of Philox calls when rows are read anew: 32,000 entries, 256 / 400: 104 / 154 on chip, 108 / 132
// read anew; 100,000, 74 / 128: 141 / 240, 216 / 227; fp32, 400 / 512 of 32,000: 176 / 226, 195 / 220.
float most_waves(const rsd::walk_cluster::Shape& c, int V, bool f32, bool ring, bool top1) {
    if (ring) return c.C <= 2 ? 1.3f : (c.C == 4 && !f32 ? 1.8f : 2.0f);
    if (c.C <= 2) return 1e30f;
    if (top1) return f32 ? 7.0f : std::min(1.6f + (float)V / 16000.0f, 6.6f);
    return std::min(1.0f + (float)V / 18000.0f, f32 ? 7.0f : 4.8f);
}

// The same for residual draws with rejected tokens (a pass per token, always both rows; us, on chip / read anew).  Where the
// distribution itself is not asked for: bf16 8,096 entries, 256 sequences: 24 / 20; 32,000, 148 / 256 / 512: 38 / 53 / 103, 40 / 44 / 86; 128,000, 64 / 256: 74 / 259,
// 105 / 139; fp32 16,000, 512: 55 / 61; 32,000, 256 / 512: 58 / 108, 53 / 102.  The pass that writes it costs reading anew more: bf16
// 32,000, 256 / 1024: 63 / 237, 59 / 212; 128,000, 64 / 148: 85 / 173, 149 / 151; fp32 32,000, 256 / 1024: 64 / 234, 68 / 279; 64,000, the same on both sides;
// 128,000, 148 / 256: 190 / 332, 207 / 251.
float most_waves_resample(const rsd::walk_cluster::Shape& c, int V, bool f32, bool whole) {
    const float v = (float)V;
    if (c.C <= 1 || (c.C == 2 && (f32 || whole))) return 1e30f;
    if (c.C == 2) return 0.2f + v / 9000.0f;
    if (!whole) return std::min(1.0f + v / 18000.0f, f32 ? 7.0f : 4.8f);
    if (f32) return V > 65536 ? 9.0f : 1e30f;
    return std::min(1.5f + v / 16000.0f, 6.5f);
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
    const bool on_chip = shape.C > 0 && shape.waves <= most_waves(shape, V, draft->dtype == RSD_F32, ring, final_sampler == RSD_FINAL_GUMBEL_TOP1);
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
    // 6.8 / 7.0 / 7.1; 128,000, 1 / 16 / 64: 7.2 / 15 / 36, 17 / 17 / 17).
    rsd::walk_cluster::ClusterArgs ca;
    memset(&ca, 0, sizeof(ca));
    ca.r = a;
    ca.resample = 1;
    ca.v.draft = a.draft; ca.v.target = a.target;
    ca.v.V = V; ca.v.num_nodes = 1;
    ca.v.seed_lo = a.seed_lo; ca.v.seed_hi = a.seed_hi; ca.v.step = step; ca.v.seq_base = seq_base;
    const rsd::walk_cluster::Shape shape = cluster_shape(B, V);
    const bool f32 = target_row->dtype == RSD_F32;
    if (!a.max_k && !(shape.C > 2 && shape.waves <= 1.0f)) {
        if (f32) rsd::walk_cluster::launch_draw_f32(a, B, s);
        else rsd::walk_cluster::launch_draw_bf16(a, B, s);
    } else if (shape.C > 0 && shape.waves <= most_waves_resample(shape, V, f32, out_residual != nullptr)) {
        launch_on_chip(ca, target_row->dtype, true, B, shape, s);
    } else {
        launch_streamed(ca, target_row->dtype, true, B, shape.C > 0, s);
    }
    return check_launch("rsd_resample_residual");
}

}  // extern "C"
