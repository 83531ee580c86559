// The walk of rsd_walk_cluster.cuh for rows that a cluster does not hold on chip, and for batches so large that holding them
// there costs more than it saves: the same control warp and commands, but the working warps read the two rows anew in every
// pass.  One block per sequence (C = 1) in large batches, a cluster of eight in small ones.
//
// A block's eight working warps take its 512-element tiles in turn, so with one block per sequence warp w owns summation
// class w and its lanes carry the class's sums in registers; with eight blocks every block is one class, and its warps
// leave their tiles' sums in shared memory to be added in order.  Weights, sums and draws are those of the on-chip walk to the
// bit: which of the two runs, with how many blocks, does not show in any result.
//
// Bound by latency: a warp's eight tiles of a pass over 32,000 entries come one after the other, 64 exponentials per lane between
// their loads.  2-byte rows either have the next tile on its way meanwhile (two blocks an SM, 96 registers) or a third block (72
// registers); per batch of 256 / 400 sequences of 32,000, multi-round rule: 67 / 100 against 72 / 80 us.  4-byte rows have the
// registers for neither (with the next target tile on its way: 62 -> 70 us).  A loop of its own for each frequent pass took
// spills out of all of them (512 sequences, 155 -> 109 us).  The register-fed kernels that this replaces had sums of their own
// and took 68 / 82 us there, and 1000 sequences of 32,001 2-byte entries 344 us on chip are 210 here.
#pragma once
#include <type_traits>

#include "rsd_walk_cluster.cuh"

namespace rsd {
namespace walk_cluster {

constexpr int kStreamWarps = 8;
constexpr int kStreamThreads = (kStreamWarps + 1) * 32;

// C = 8: a block has up to 64 tiles
template <int C>
using StreamSmem = Smem<kStreamWarps, C == 1 ? 1 : kMaxTiles / kClasses, kMaxTiles>;

// A tile on its way: load_tile() in two halves, so that a warp's next tile travels while it works on this one.  Of a row off 16-byte
// boundaries a lane asks for the aligned word that its piece starts in; the one behind is the next lane's.
template <typename T>
struct Incoming {
    static constexpr int kElem = (int)sizeof(T), kPer = 16 / kElem, kPieces = 16 / kPer;
    Packed<T> pk;
    uint4 last;             // lane 31: the word behind its last piece
    bool shifted;

    __device__ __forceinline__ void ask(const char* row, int tile, int lane, int V) {
        const char* at = row + ((int64_t)tile * kTileElems + lane * kPer) * kElem;
        const uint32_t m = (uint32_t)(uintptr_t)row & 15u;
        const int after = V - (tile + 1) * kTileElems;      // elements behind the tile
        shifted = m != 0 && tile > 0 && after >= kPer;
        if (shifted) {
#pragma unroll
            for (int i = 0; i < kPieces; ++i) pk.w[i] = ld_stream(at + 512 * i - m);
            if (lane == 31) last = ld_stream(at + 512 * (kPieces - 1) - m + 16);
        } else {
            load_tile<T>(pk, row, tile, lane, V);
        }
    }
    __device__ __forceinline__ void take(Packed<T>& out, const char* row, int lane) const {
        out = pk;
        if (!shifted) return;
        const uint32_t m = (uint32_t)(uintptr_t)row & 15u;
        const int src = (lane + 1) & 31;
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
            const bool wrap = lane == 0 && i + 1 < kPieces;   // lane 31's next word is lane 0's next piece
            const uint4 mine = wrap ? pk.w[i + 1 < kPieces ? i + 1 : i] : pk.w[i];
            uint4 next = make_uint4(__shfl_sync(0xFFFFFFFFu, mine.x, src), __shfl_sync(0xFFFFFFFFu, mine.y, src),
                                    __shfl_sync(0xFFFFFFFFu, mine.z, src), __shfl_sync(0xFFFFFFFFu, mine.w, src));
            if (lane == 31 && i + 1 == kPieces) next = last;
            out.w[i] = window16(pk.w[i], next, m);
        }
    }
};

// kAhead: the warp's next tile travels while it works on this one.
template <typename T, int C, int MODE, bool kAhead>
__device__ __forceinline__ void work_stream(StreamSmem<C>& sm, float* frozen_w, const Place& pl, const WorkRows& rows) {
    static_assert(C == 1 || C == kClasses, "a warp or a block per summation class");
    constexpr int kAll = kStreamThreads, kWorkers = kStreamWarps * 32;
    constexpr int kPer = 16 / (int)sizeof(T), kRuns = 16 / kPer;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int V = pl.V;
    const int n_mine = pl.n_local > warp ? (pl.n_local - warp + kStreamWarps - 1) / kStreamWarps : 0;   // this warp's tiles
    int flags = kBuffer, node = 0;                   // (the next command is the first, an even one)
    float a_hi = 0.0f, a_lo = 0.0f;
    const char *rowq = rows.q, *rowp = rows.p;       // of the node that was opened last
    bool relative = false, dirty = false;            // its exponentials are relative to sm.ref_q, sm.ref_p; its rows may hold NaN
    int n_frozen = 0, frozen_tile = -1;              // tokens of sm.gone_tok that keep the weight frozen_w (kResample); lane i: the i-th one's tile
    Incoming<T> in_q, in_p;
    int held = -1;                                   // the tile whose rows they hold,
    bool held_p = false;                             // with the draft's
    auto ask = [&](int tile, bool with_p) {
        in_q.ask(rowq, tile, lane, V);
        if (with_p) in_p.ask(rowp, tile, lane, V);
        held = tile;
        held_p = with_p;
    };
    auto next_tile = [&](Packed<T>& rq, Packed<T>& rp, int tile, int after, bool with_p) {   // after: the tile behind it, or -1
        if (kAhead) {
            in_q.take(rq, rowq, lane);
            if (with_p) in_p.take(rp, rowp, lane);
            if (after >= 0) ask(after, with_p);
        } else {
            load_tile<T>(rq, rowq, tile, lane, V);
            if (with_p) load_tile<T>(rp, rowp, tile, lane, V);
        }
    };
    cluster_wait();                                  // every block's mbarriers are in place
    for (;;) {
        {
            const int odd = flags & kBuffer ? 0 : 1;
            cmd_sync<kAll>(odd);
            const Cmd cmd = sm.cmd[odd];
            flags = cmd.flags;
            node = cmd.node;
            a_hi = cmd.a_hi;
            a_lo = cmd.a_lo;
        }
        const int kind = flags & kKindMask, mode = flags >> kModeShift, buf = flags & kBuffer ? 1 : 0;
        if (kind == kEnd) return;
        if (kind == kOpen || kind == kOpenTarget) {
            rowq = rows.q + (int64_t)node * rows.stride_q;
            rowp = rows.p + (int64_t)node * rows.stride_p;
            relative = flags & kRelative;
            dirty = flags & kClean;
            held = -1;
        }
        if (MODE == kResample && kind == kWrite) dump_sync<kAll>();   // everyone has read the command
        if (MODE == kResample && kind == kResidualPass && (flags & kFreeze)) {
            if (lane == n_frozen) frozen_tile = sm.gone_tok[n_frozen] / kTileElems;
            ++n_frozen;
        }
        const bool use_p = kind >= kDump ? mode != 0 : kind != kOpenTarget && kind != kPlainPass;
        // the warp's tiles: i, i + way, ... of the block's (a dump: the one that is asked for)
        int todo = n_mine, i = flags & kBackward ? warp + kStreamWarps * (n_mine - 1) : warp;
        const int way = flags & kBackward ? -kStreamWarps : kStreamWarps;
        if (kind == kDump) {
            i = (node - pl.rank) / C;
            todo = i % kStreamWarps == warp ? 1 : 0;
        }
        // (passes over a node alternate in direction: a pass starts with the tile the one before has ended with)
        if (kAhead && todo > 0 && (held != pl.rank + C * i || (use_p && !held_p))) ask(pl.rank + C * i, use_p);
        float sum_q = 0.0f, sum_p = 0.0f, top_q = kNegInf, top_p = kNegInf;
        bool saw_nan = false;
        Top1 top1;
        auto count = [&](float s, float sp, bool with_p) {   // a tile's sums
            if (C == 1) {
                sum_q += s;
                if (with_p) sum_p += sp;
            } else {
                sm.lane_sum[0][i][lane] = s;
                if (with_p) sm.lane_sum[1][i][lane] = sp;
            }
            if (flags & kStoreTiles) {
                const float ts = warp_sum_f32(s);
                const int tile = pl.rank + C * i;
                if (lane < C) send_word(remote_addr(&sm.tile_sum[tile], lane), ts, remote_addr(&sm.red_bar[buf], lane));
            }
        };
        // (kResample) removed tokens keep the weight that they had when they were removed
        auto freeze = [&](int tile, float (&q)[16], float (&p)[16]) {
            for (unsigned here = __ballot_sync(0xFFFFFFFFu, frozen_tile == tile); here; here &= here - 1u) {
                const int f = __ffs(here) - 1, o = sm.gone_tok[f] - tile * kTileElems;
                int l_, j_;
                walk_ring::piece_of<T>(o, l_, j_);
                if (l_ != lane) continue;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j == j_) {      // (this lane alone reads and writes its tokens' frozen weights)
                        if ((flags & kFreeze) && f == n_frozen - 1) frozen_w[f] = residual_weight(q[j], p[j], sm.freeze_hi, sm.freeze_lo);
                        q[j] = frozen_w[f];
                        p[j] = 0.0f;
                    }
            }
        };
        // The passes that a walk consists of, each as a loop of its own: nothing of the others holds registers or splits the block of
        // instructions that the next tile's loads travel behind.
        auto sweep = [&](auto which) {
            constexpr int KIND = decltype(which)::value;
            constexpr bool WITH_P = KIND != kOpenTarget;
            for (; todo > 0; --todo, i += way) {
                Packed<T> rq, rp;
                next_tile(rq, rp, pl.rank + C * i, todo > 1 ? pl.rank + C * (i + way) : -1, WITH_P);
                float q[16], p[16];
                rq.unpack(q);
                exp16_precise(q, rows.kq, q);
                if (WITH_P) {
                    rp.unpack(p);
                    exp16_precise(p, rows.kp, p);
                }
                if (KIND == kOpen) {
                    count(tree_sum16(q), tree_sum16(p), true);
                } else {
                    float w[16];
                    if (KIND == kResidualPass) {
                        if (MODE == kResample) freeze(pl.rank + C * i, q, p);
                        residual16(q, p, a_hi, a_lo, w);
                        count(tree_sum16(w), 0.0f, false);
                    } else if (KIND == kOverlapPass) {
                        weights16<kSeqOverlap>(q, p, a_hi, a_lo, 0.0f, w);
                        count(tree_sum16(w), 0.0f, false);
                    } else if (KIND == kSeqPass) {
                        weights16<kSeqResidual>(q, p, a_hi, a_lo, sm.c_seq, w);
                        count(tree_sum16(w), 0.0f, false);
                    } else {
                        count(tree_sum16(q), 0.0f, false);
                    }
                }
            }
        };
        if (!relative && !dirty) {
            if (kind == kOpen) sweep(std::integral_constant<int, kOpen>());
            else if (kind == kOpenTarget) sweep(std::integral_constant<int, kOpenTarget>());
            else if (kind == kResidualPass) sweep(std::integral_constant<int, kResidualPass>());
            if constexpr (MODE == kRuleWalk) {
                if (kind == kOverlapPass) sweep(std::integral_constant<int, kOverlapPass>());
                else if (kind == kSeqPass) sweep(std::integral_constant<int, kSeqPass>());
            }
        }
        // everything else, and rows with NaN or far from 0
#pragma unroll 1
        for (; todo > 0; --todo, i += way) {
            const int tile = pl.rank + C * i;
            Packed<T> rq, rp;
            next_tile(rq, rp, tile, todo > 1 ? tile + C * way : -1, use_p);
            if (dirty) {
                top_q = fmaxf(top_q, clean_tile(rq, saw_nan));
                if (use_p) top_p = fmaxf(top_p, clean_tile(rp, saw_nan));
            }
            float q[16], p[16], w[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) p[j] = 0.0f;
            rq.unpack(q);
            if (relative) exp16(q, rows.kq, sm.ref_q, q);
            else exp16_precise(q, rows.kq, q);
            if (use_p) {
                rp.unpack(p);
                if (relative) exp16(p, rows.kp, sm.ref_p, p);
                else exp16_precise(p, rows.kp, p);
            }
            if (MODE == kResample) freeze(tile, q, p);
            if (kind == kResidualPass) {
                residual16(q, p, a_hi, a_lo, w);
            } else if (kind == kRestPass) {
#pragma unroll
                for (int j = 0; j < 16; ++j) w[j] = p[j];
                for (int f = 0; f < sm.n_gone_tok; ++f) {
                    const int o = sm.gone_tok[f] - tile * kTileElems;
                    if (o < 0 || o >= kTileElems) continue;
                    int l_, j_;
                    walk_ring::piece_of<T>(o, l_, j_);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (l_ == lane && j == j_) w[j] = 0.0f;
                }
            } else if (MODE == kRuleWalk && kind == kOverlapPass) {
                weights16<kSeqOverlap>(q, p, a_hi, a_lo, 0.0f, w);
            } else if (MODE == kRuleWalk && kind == kSeqPass) {
                weights16<kSeqResidual>(q, p, a_hi, a_lo, sm.c_seq, w);
            } else if (kind >= kDump) {
                mode_weights<MODE == kRuleWalk>(mode, q, p, a_hi, a_lo, MODE == kRuleWalk ? sm.c_seq : 0.0f, w);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) w[j] = q[j];
            }
            if (kind < kDump) {
                count(tree_sum16(w), kind == kOpen ? tree_sum16(p) : 0.0f, kind == kOpen);
            } else if (kind == kDump) {
#pragma unroll
                for (int r = 0; r < kRuns; ++r)
#pragma unroll
                    for (int j = 0; j < kPer; ++j) sm.tile_w[(r * 32 + lane) * kPer + j] = w[r * kPer + j];
            } else if (MODE == kRuleWalk && kind == kTop1) {
                const uint32_t word = top1.look<T>(rows.key, (uint32_t)node, tile, lane, w);
                top1.bound = -warp_max(-top1.bound);
                top1.take<T>(rows.key, (uint32_t)node, tile, lane, w, word);
            } else if (MODE == kResample && kind == kWrite) {
                write_tile<T>(rows.out_residual, tile, lane, V, w, sm.inv_total);
            }
        }
        if (kind == kDump) {
            dump_sync<kAll>();
        } else if (MODE == kRuleWalk && kind == kTop1) {
            top1_report<kStreamWarps>(sm, pl, flags, top1.best);
        } else if (kind < kDump) {
            if (flags & kClean) {
                top_q = warp_max(top_q);
                top_p = warp_max(top_p);
                if (lane == 0) { sm.warp_top[0][warp] = top_q; sm.warp_top[1][warp] = top_p; }
                if (saw_nan) sm.nan_seen = 1;
            }
            if (C == 1) {
                sum_q = warp_sum_f32(sum_q);
                sum_p = warp_sum_f32(sum_p);
                if (lane < (kind == kOpen ? 2 : 1))
                    send_word(remote_addr(&sm.class_sum[buf][lane * kClasses + warp], 0), lane ? sum_p : sum_q, remote_addr(&sm.red_bar[buf], 0));
                if (flags & kClean) workers_sync<kWorkers>();
            } else {
                workers_sync<kWorkers>();           // the lanes' sums are in place
                send_class_sums<kStreamWarps>(sm, pl, flags);
            }
            if (flags & kClean) send_tops<kStreamWarps>(sm, pl, flags);
        }
    }
}

// BLOCKS: blocks per SM
template <typename T, int C, int MODE, int BLOCKS>
__global__ void __launch_bounds__(kStreamThreads, BLOCKS) walk_stream_kernel(const __grid_constant__ ClusterArgs ca) {
    __shared__ StreamSmem<C> sm;
    __shared__ float frozen_w[MODE == kResample ? 32 : 1];
    run_walk<T, MODE, kStreamWarps>(sm, ca, [&](const Place& pl, const WorkRows& rows) {
        work_stream<T, C, MODE, sizeof(T) == 2 && BLOCKS == 2>(sm, frozen_w, pl, rows);
    });
}

}  // namespace walk_cluster
}  // namespace rsd
