// Recursive rejection sampling along the draft tree (Eqs. 1-4, Algorithm 1; Section 3.2.2, Algorithm 6), its two
// baseline rules and the stand-alone residual draw, by a thread block cluster per sequence that holds the weights of the
// node it is at on chip.
//
// A walk is a chain of dependent passes (open a node, one residual pass per rejected child), so with one block per
// sequence its latency is the number of passes times a sweep over two rows by one SM.  Here the vocabulary is dealt out
// to the blocks of a cluster, 512-element tiles in turn (tile t to block t mod C), and within a block to its working
// warps, NT tiles each.  Opening a node loads both rows once, turns them into exponentials and leaves these in registers;
// a rejected child then costs a fused multiply-add, a clamp and a sum per element, nothing is read or exponentiated
// again.  The blocks' partial sums travel to all blocks through distributed shared memory (st.async onto an mbarrier),
// and the control warp of every block takes the same decisions from the same numbers.  A control warp is one warp running
// dependent scalar code (5-6 cycles per instruction), so whatever does not depend on the running pass is done while it
// runs, one child per lane: tokens, row values, uniforms, the next node's children.
//
// Sums are taken in the order of the ring walk (rsd_walk_ring.cuh): per lane over the tiles of equal index modulo 8, in
// pass direction, then over the lanes, then a tree over the eight classes in double.  For the rows that the ring walk takes
// (plain walks, rows on 16-byte boundaries) the weights are its weights as well, so the two give the same bits; elsewhere the
// exponentials keep the rounding of their exponents (exp16_precise()), here and in the walk that reads the rows in every pass
// (rsd_walk_stream.cuh).  Which kernel runs, with how many blocks (a matter of batch size and vocabulary), does not show
// in any result.
// Every wait on an mbarrier is bounded (about a second); a wait that runs out abandons the walk with RSD_ST_TIMEOUT.
#pragma once
#include "rsd_walk_cluster_args.h"
#include "rsd_walk_ring.cuh"

namespace rsd {
namespace walk_cluster {

using walk_ring::kSumFloor;
using walk_ring::kTileElems;
using walk_ring::warp_sum_f32;

constexpr int kClasses = 8;              // summation classes: tiles of equal index modulo 8
constexpr int kMaxListed = 64;           // rejected tokens remembered per node

// What a kernel is compiled for: recursive rejection sampling with the inverse-CDF last draw; the other rules and the
// Gumbel-Top-1 draw; the stand-alone residual draw.  (One kernel for the last two spilled four times as many registers.)
enum { kPlainWalk = 0, kRuleWalk = 1, kResample = 2 };

// Cmd::flags: what a pass does (low four bits) and options
enum {
    kEnd = 0,
    kOpen = 1,           // load both rows of a node; sums of exp(lt k_q - c_q) and exp(ld k_p - c_p)
    kOpenTarget = 2,     // load its target row; sum of exp(lt k_q - c_q)
    kResidualPass = 3,   // sum of (q - a p)+
    kPlainPass = 4,      // sum of q
    kRestPass = 5,       // sum of p without the listed tokens
    kOverlapPass = 6,    // K-SEQ: sum of min(a_hi p, a_lo q)
    kSeqPass = 7,        // K-SEQ: sum of (q - c min(a_hi p, a_lo q))+
    kDump = 8,           // the weights of one tile in token order
    kTop1 = 9,           // Gumbel-Top-1 over the weights
    kWrite = 10,         // the normalised weights to global memory
    kKindMask = 15,
    kClean = 16,         // kOpen, kOpenTarget: NaN counts as -inf; the rows' maxima are reported
    kRelative = 32,      // kOpen, kOpenTarget: exponentials relative to sm.ref_q, sm.ref_p (else to 0)
    kStoreTiles = 64,    // the sum of every tile goes to every block's tile_sum
    kBackward = 128,     // order of the lanes' sums
    kBuffer = 256,       // an odd command: the second place, and the second half of class_sum / red_bar
    kFreeze = 512,       // kResidualPass: first sm.freeze_x leaves the draft and keeps its weight
    kFirst = 1024,       // (a working warp's own mark: no command yet)
    kModeShift = 12      // kDump, kTop1, kWrite: weights are 0 q, kResidual (q - a p)+, kSeqResidual K-SEQ's residual
};

struct __align__(16) Cmd {
    int flags;
    int node;            // kOpen, kOpenTarget: the node; kDump: the tile; kTop1: the node of the random stream
    float a_hi, a_lo;
};

// WARPS working warps; LISTED tiles of the block whose lanes' sums are kept; TILES tiles of all blocks
template <int WARPS, int LISTED, int TILES>
struct Smem {
    unsigned long long red_bar[2];
    Cmd cmd[2];                              // command n: cmd[n & 1]
    float ref_q, ref_p;                      // references of the exponentials, in units of log2
    float c_seq;                             // K-SEQ's factor of its residual
    int freeze_x;
    float freeze_hi, freeze_lo;              // the coefficient under which the frozen token's weight is taken
    double inv_total;                        // kWrite
    float class_sum[2][2 * kClasses];        // [buffer][target or only sum: 8 classes, draft sum: 8 classes]
    float extra[2][3][kClasses];             // [buffer][maxima of target and draft, NaN seen][block]
    unsigned long long top1[kClasses];       // [block] smallest key of the Gumbel draw with its token
    unsigned long long warp_key[WARPS];
    float lane_sum[2][LISTED][32];           // [target / only sum, draft][local tile][lane]
    float warp_top[2][WARPS];
    int nan_seen;
    int gave_up;                             // rank 0: some block's wait ran out
    float tile_sum[TILES];
    __align__(16) float tile_w[kTileElems];  // (read as float4)
    int par[kMaxCachedNodes], tok[kMaxCachedNodes];
    int kid_node[32];
    int gone_tok[kMaxListed];
    int n_gone_tok;
};
template <int WARPS, int NT>
using ChipSmem = Smem<WARPS, WARPS * NT, kClasses * WARPS * NT>;

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t remote_addr(const void* p, uint32_t rank) {   // p: this block's shared memory
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
// store a word in a block's shared memory and count its four bytes on that block's mbarrier
__device__ __forceinline__ void send_word(uint32_t addr, float v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}
// (every barrier is met by whole warps: the lanes are brought together first)
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void store_remote(uint32_t addr, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
template <int THREADS>
__device__ __forceinline__ void named_sync(int id) {
    __syncwarp();
    asm volatile("barrier.cta.sync.aligned %0, %1;" ::"r"(id), "n"(THREADS) : "memory");
}
// The command barriers: for command n the control warp arrives at one, the working warps wait there; commands take two places
// and two barriers in turn (kBuffer in its flags: the odd ones).  Command n + 2 follows the sums (or the dump barrier) of command n + 1, which no working
// warp runs before it has read command n: nobody arrives twice at one barrier, and no command is overwritten unread.
// That holds for the end of a walk whose wait for the sums of command n has run out as well: it is command n + 1.
__device__ __forceinline__ int cmd_barrier(int odd) { return odd ? 4 : 1; }
template <int THREADS>
__device__ __forceinline__ void cmd_arrive(int odd) {
    __syncwarp();
    asm volatile("barrier.cta.arrive.aligned %0, %1;" ::"r"(cmd_barrier(odd)), "n"(THREADS) : "memory");
}
template <int THREADS>
__device__ __forceinline__ void cmd_sync(int odd) { named_sync<THREADS>(cmd_barrier(odd)); }
template <int THREADS>
__device__ __forceinline__ void workers_sync() { named_sync<THREADS>(2); }
template <int THREADS>
__device__ __forceinline__ void dump_sync() { named_sync<THREADS>(3); }

// A lane's 16 values of a tile: the 16-byte pieces lane, lane + 32, ... (the order of the ring walk), -inf beyond the
// row's end.  Rows on 16-byte boundaries take one load a piece.  Others take the two aligned words around it, shifted;
// tiles at the ends of such a row, and every row's partial tile, are put together from single elements.
template <typename T>
__device__ __forceinline__ void load_tile(Packed<T>& pk, const char* row, int tile, int lane, int V) {
    constexpr int kElem = (int)sizeof(T), kPer = 16 / kElem, kPieces = 16 / kPer;
    const char* at = row + ((int64_t)tile * kTileElems + lane * kPer) * kElem;
    const uint32_t m = (uint32_t)(uintptr_t)row & 15u;
    const int after = V - (tile + 1) * kTileElems;      // elements behind the tile
    if (m == 0 && after >= 0) {
#pragma unroll
        for (int i = 0; i < kPieces; ++i) pk.w[i] = ld_stream(at + 512 * i);
    } else if (tile > 0 && after >= kPer) {
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
            const uint4 a = *(const uint4*)(at + 512 * i - m), b = *(const uint4*)(at + 512 * i - m + 16);
            pk.w[i] = window16(a, b, m);
        }
    } else {
        const int x0 = tile * kTileElems + lane * kPer;
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (kElem == 4) {
                    const int x = x0 + i * 32 * kPer + j;
                    w[j] = x < V ? ((const uint32_t*)row)[x] : 0xFF800000u;
                } else {
                    const int x = x0 + i * 32 * kPer + 2 * j;
                    const uint32_t lo = x < V ? ((const uint16_t*)row)[x] : 0xFF80u, hi = x + 1 < V ? ((const uint16_t*)row)[x + 1] : 0xFF80u;
                    w[j] = lo | (hi << 16);
                }
            }
            pk.w[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// the tile's largest value, with NaN turned into -inf (and noted)
template <typename T>
__device__ __forceinline__ float clean_tile(Packed<T>& pk, bool& saw_nan) {
    float m = group_max_nan(pk);
    if (m != m) { saw_nan = true; pk.clean_nan(); m = group_max_nan(pk); }
    return m;
}

// exp16() relative to 0 with the exponents' rounding put back in: v k = x + d with x = fl(v k), 2^(v k) = 2^x (1 + d ln 2).
// Relative to 0 an exponent of ten or so is rounded by 5e-7, where one relative to the row's maximum would be exact for
// the entries that matter.  (-inf would make d a NaN: it enters as -1e30, whose weight is 0 as well.)
__device__ __forceinline__ void exp16_precise(const float (&v)[16], float k, float (&e)[16]) {
    const unsigned long long k2 = f32x2(k, k), minus_k = f32x2(-k, -k), zero = f32x2(0.0f, 0.0f), minus_ln2 = f32x2(-0.69314718f, -0.69314718f);
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        const unsigned long long vv = f32x2(max_nan(v[j], -1e30f), max_nan(v[j + 1], -1e30f));
        const unsigned long long x = fma_f32x2(vv, k2, zero), minus_d = fma_f32x2(vv, minus_k, x);
        float a, b;
        split_f32x2(x, a, b);
        const unsigned long long w = f32x2(ex2_approx(a), ex2_approx(b));
        split_f32x2(fma_f32x2(fma_f32x2(w, minus_ln2, zero), minus_d, w), e[j], e[j + 1]);
    }
}
__device__ __forceinline__ float weight_precise(float l, float k) {
    if (!(l > -1e30f)) return 0.0f;
    const float x = l * k, w = ex2_approx(x);
    return fmaf(w * 0.69314718f, fmaf(l, k, -x), w);
}

// weights of a lane's 16 values under the mode of a drawing pass
template <bool EXTRA>
__device__ __forceinline__ void mode_weights(int mode, const float (&q)[16], const float (&p)[16], float a_hi, float a_lo, float c, float (&w)[16]) {
    if (mode == kResidual) {
        residual16(q, p, a_hi, a_lo, w);
    } else if (EXTRA && mode == kSeqResidual) {
        weights16<kSeqResidual>(q, p, a_hi, a_lo, c, w);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) w[j] = q[j];
    }
}

// The draft row's share of a warp: NT tiles of weights, 16 a lane, in registers.
template <typename T, int NT>
struct DraftTiles {
    static constexpr bool kShared = false;
    float v[NT][16];
    Packed<T> raw[NT];
    __device__ __forceinline__ explicit DraftTiles(float4*) {
#pragma unroll
        for (int k = 0; k < NT; ++k)
#pragma unroll
            for (int j = 0; j < 16; ++j) v[k][j] = 0.0f;
    }
    __device__ __forceinline__ void clear(int k) { raw[k].fill_neg_inf(); }
    __device__ __forceinline__ void ask(int k, const char* row, int tile, int lane, int V) { load_tile<T>(raw[k], row, tile, lane, V); }
    __device__ __forceinline__ void landed() const {}
    __device__ __forceinline__ void get_raw(int k, Packed<T>& out) const { out = raw[k]; }
    __device__ __forceinline__ void put_raw(int k, const Packed<T>& in) { raw[k] = in; }
    __device__ __forceinline__ void get(int k, float (&out)[16]) const {
#pragma unroll
        for (int j = 0; j < 16; ++j) out[j] = v[k][j];
    }
    __device__ __forceinline__ void put(int k, const float (&in)[16]) {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[k][j] = in[j];
    }
};
// Four tiles a warp: in shared memory, where the rows land by themselves (cp.async) while the target's are on their way to
// registers.  Value j of a lane is word j % 4 of its 16-byte place j / 4; a lane reads and writes its own places only.
template <typename T>
struct DraftTiles<T, 4> {
    static constexpr bool kShared = true;
    static constexpr int kPieces = (int)sizeof(T);
    float4* const at;                                    // this lane's first place
    __device__ __forceinline__ explicit DraftTiles(float4* warp_tiles) : at(warp_tiles + (threadIdx.x & 31)) {}
    __device__ __forceinline__ float4* place(int k, int i) const { return at + (k * 4 + i) * 32; }
    __device__ __forceinline__ void clear(int k) {
        Packed<T> none;
        none.fill_neg_inf();
        put_raw(k, none);
    }
    __device__ __forceinline__ void ask(int k, const char* row, int tile, int lane, int V) {
        if (((uintptr_t)row & 15u) == 0 && (tile + 1) * kTileElems <= V) {
            const char* from = row + (int64_t)tile * kTileElems * (int)sizeof(T) + lane * 16;
#pragma unroll
            for (int i = 0; i < kPieces; ++i)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(place(k, i))), "l"(from + 512 * i) : "memory");
        } else {
            Packed<T> pk;
            load_tile<T>(pk, row, tile, lane, V);
            put_raw(k, pk);
        }
    }
    __device__ __forceinline__ void landed() const { asm volatile("cp.async.wait_all;" ::: "memory"); }
    __device__ __forceinline__ void get_raw(int k, Packed<T>& out) const {
#pragma unroll
        for (int i = 0; i < kPieces; ++i) out.w[i] = *(const uint4*)place(k, i);
    }
    __device__ __forceinline__ void put_raw(int k, const Packed<T>& in) {
#pragma unroll
        for (int i = 0; i < kPieces; ++i) *(uint4*)place(k, i) = in.w[i];
    }
    __device__ __forceinline__ void get(int k, float (&out)[16]) const {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 f = *place(k, i);
            out[4 * i] = f.x; out[4 * i + 1] = f.y; out[4 * i + 2] = f.z; out[4 * i + 3] = f.w;
        }
    }
    __device__ __forceinline__ void put(int k, const float (&in)[16]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) *place(k, i) = make_float4(in[4 * i], in[4 * i + 1], in[4 * i + 2], in[4 * i + 3]);
    }
};
// shared memory that the draft tiles of a block of WARPS working warps take beside its Smem
template <int NT, int WARPS>
constexpr size_t draft_tiles_bytes() { return NT == 4 ? (size_t)WARPS * NT * kTileElems * 4 : 0; }

// A block's place in its cluster and the row's tiles.
struct Place {
    int rank, C, V, n_tiles, n_local;   // n_local: tiles rank, rank + C, ...
    int per_block;                      // summation classes of a block
};

// What the working warps need to know about the sequence.
struct WorkRows {
    const char* q;               // its rows of node 0 ...
    const char* p;
    int64_t stride_q, stride_p;  // ... and the bytes from node to node
    float kq, kp;                // log2(e) / temperature
    bool with_draft;             // the first node probably needs its draft row as well
    bool precise;                // exponentials by exp16_precise() while they are relative to 0
    RngKey key;                  // kTop1
    float* out_residual;         // kWrite
};

// Gumbel-Top-1 draw (Algorithm 6's last step): arg max over y of log w(y) + G(y), which is the arg min of E(y) / w(y) with
// E(y) = exp(-G(y)) = t(U_M) / 16 + [y mod 16 != a] t(U_y), the group-wise noise in its exponential form (streams
// kTagFinalGumbelCoarse / Fine of the node).  Entries without weight are left out; equal keys go to the smaller token.
// E >= t(U_M) / 16 with equality at position a: the smallest key at the positions a, from fast logarithms rounded up, bounds
// the winner from above, and only entries whose lower bound reaches it are taken exactly.  The result is that of taking
// every entry.  (Exact logarithms and a second round of Philox calls for every group made this pass 25 us of a walk's 73.
// The fast logarithms lie within the margins below for each of the 2^28 words a group can have.)
struct Top1 {
    float bound;
    unsigned long long best;                     // key bits << 32 | token: keys are >= 0, so the order is that of (key, token)

    __device__ __forceinline__ Top1() : bound(-kNegInf), best(~0ull) {}

    // t(U_M) / 16 of a group's word, down (up = -1) or up (+1) to a bound
    __device__ __forceinline__ static float group_bound(uint32_t word, float up) {
        const float t_hat = -__logf(fmaf((float)(word >> 4), 3.725290298461914e-09f, 1.862645149230957e-09f));
        return fmaxf(fmaf(up, fmaf(t_hat, 1e-6f, 2.5e-7f), t_hat), 0.0f) * 0.0625f;
    }
    // The lane of whose group a lane's piece i is part (a tile is 32 groups; RUNS lanes share one).
    template <int RUNS>
    __device__ __forceinline__ static int group_lane(int i, int lane) { return (i * 32 + lane) / RUNS; }
    // The coarse word of group `lane` of a tile; `bound` from the entries at the groups' positions a.  (Every lane takes one group's word
    // and bounds and hands them to the lanes that hold its entries: each lane for its own pieces took RUNS times the Philox calls and
    // logarithms.)
    template <typename T>
    __device__ __forceinline__ uint32_t look(const RngKey& key, uint32_t node, int tile, int lane, const float (&w)[16]) {
        constexpr int RUNS = (int)sizeof(T), kPer = 16 / RUNS;
        const uint32_t g = (uint32_t)(tile * 32 + lane);
        const uint32_t word = coarse_select(rng_draw(key, node, kTagFinalGumbelCoarse, coarse_index(g)), g);
        const float hi = group_bound(word, 1.0f);
#pragma unroll
        for (int i = 0; i < RUNS; ++i) {
            const int from = group_lane<RUNS>(i, lane);
            const float tg_hi = __shfl_sync(0xFFFFFFFFu, hi, from);
            const int ja = (int)(__shfl_sync(0xFFFFFFFFu, word, from) & 15u) - (lane % RUNS) * kPer;
            float wa = 0.0f;
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (j == ja) wa = w[i * kPer + j];
            if (wa > 0.0f) bound = fminf(bound, tg_hi / wa * 1.00001f);
        }
        return word;
    }
    // the exact keys of the entries that can reach `bound`
    template <typename T>
    __device__ __forceinline__ void take(const RngKey& key, uint32_t node, int tile, int lane, const float (&w)[16], uint32_t group_word) {
        constexpr int RUNS = (int)sizeof(T), kPer = 16 / RUNS;
        const float lo = group_bound(group_word, -1.0f);
#pragma unroll
        for (int i = 0; i < RUNS; ++i) {
            const int x0 = tile * kTileElems + (i * 32 + lane) * kPer, from = group_lane<RUNS>(i, lane);
            const float tg_lo = __shfl_sync(0xFFFFFFFFu, lo, from);
            const uint32_t word = __shfl_sync(0xFFFFFFFFu, group_word, from);
            uint32_t todo = 0;
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (w[i * kPer + j] > 0.0f && tg_lo <= bound * w[i * kPer + j] * 1.00001f) todo |= 1u << j;
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                float wj = 0.0f;
#pragma unroll
                for (int jj = 0; jj < kPer; ++jj)
                    if (jj == j) wj = w[i * kPer + jj];
                float e = neg_log_group_uniform_f32(word) * 0.0625f;
                if (j != (int)(word & 15u) - (x0 & 15)) {
                    const uint4 fw = rng_draw(key, node, kTagFinalGumbelFine, (uint32_t)(x0 + j) >> 2);
                    const uint32_t sel = (uint32_t)(x0 + j) & 3u;
                    e += neg_log_uniform_f32(sel < 2 ? (sel == 0 ? fw.x : fw.y) : (sel == 2 ? fw.z : fw.w));
                }
                const float key_j = e / wj;
                if (key_j < __int_as_float(0x7F800000)) best = min(best, ((unsigned long long)__float_as_uint(key_j) << 32) | (uint32_t)(x0 + j));
            }
            __syncwarp();
        }
    }
};
// the block's smallest key goes to every block
template <int WARPS, typename SM>
__device__ __forceinline__ void top1_report(SM& sm, const Place& pl, int flags, unsigned long long best) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if (lane == 0) sm.warp_key[warp] = best;
    workers_sync<WARPS * 32>();
    for (int w = 0; w < WARPS; ++w) best = min(best, sm.warp_key[w]);
    if (warp == 0 && lane < pl.C) {
        const uint32_t bar = remote_addr(&sm.red_bar[flags & kBuffer ? 1 : 0], lane), at = remote_addr(&sm.top1[pl.rank], lane);
        send_word(at, __uint_as_float((uint32_t)best), bar);
        send_word(at + 4u, __uint_as_float((uint32_t)(best >> 32)), bar);
    }
}
// The pass over tiles held in registers: the bound is the block's, from all its tiles.
template <typename T, int NT, int WARPS>
__device__ __forceinline__ void top1_pass(ChipSmem<WARPS, NT>& sm, const Place& pl, const RngKey& key, uint32_t node, int flags, float a_hi, float a_lo,
                                          const float (&q)[NT][16], DraftTiles<T, NT>& draft) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t words[NT];
    Top1 top1;
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        float p[16], w[16];
        draft.get(k, p);
        mode_weights<true>(flags >> kModeShift, q[k], p, a_hi, a_lo, sm.c_seq, w);
        const int tile = pl.rank + pl.C * (warp + WARPS * k);    // (beyond the row: no weight)
        words[k] = top1.look<T>(key, node, tile, lane, w);
        if (draft.kShared) draft.put(k, w);                      // (a walk's last pass: nothing needs the draft row any more)
    }
    top1.bound = -warp_max(-top1.bound);
    if (lane == 0) sm.warp_top[0][warp] = top1.bound;
    workers_sync<WARPS * 32>();
    top1.bound = -warp_max(-(lane < WARPS ? sm.warp_top[0][lane] : top1.bound));
    if constexpr (DraftTiles<T, NT>::kShared) {                  // (one copy of the code: four of them spilled)
#pragma unroll 1
        for (int k = 0; k < NT; ++k) {
            uint32_t word = words[0];
#pragma unroll
            for (int i = 1; i < NT; ++i) word = i == k ? words[i] : word;
            float w[16];
            draft.get(k, w);
            top1.take<T>(key, node, pl.rank + pl.C * (warp + WARPS * k), lane, w, word);
        }
    } else {
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            float p[16], w[16];
            draft.get(k, p);
            mode_weights<true>(flags >> kModeShift, q[k], p, a_hi, a_lo, sm.c_seq, w);
            top1.take<T>(key, node, pl.rank + pl.C * (warp + WARPS * k), lane, w, words[k]);
        }
    }
    top1_report<WARPS>(sm, pl, flags, top1.best);
}

// The lanes' sums in sm.lane_sum, added per summation class in the order of the pass, to every block.
template <int WARPS, typename SM>
__device__ __forceinline__ void send_class_sums(SM& sm, const Place& pl, int flags) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per_block = pl.per_block, buf = flags & kBuffer ? 1 : 0;
    for (int i = warp; i < ((flags & kKindMask) == kOpen ? 2 * per_block : per_block); i += WARPS) {
        const int which = i >= per_block ? 1 : 0, cl = i - which * per_block;
        const int n = pl.n_local > cl ? (pl.n_local - cl + per_block - 1) / per_block : 0;
        const int step = flags & kBackward ? -per_block : per_block, at = flags & kBackward ? cl + per_block * (n - 1) : cl;
        float acc = 0.0f;
        for (int m0 = 0; m0 < n; m0 += 8) {
            float v[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = m0 + m < n ? sm.lane_sum[which][at + step * (m0 + m)][lane] : 0.0f;
#pragma unroll
            for (int m = 0; m < 8; ++m) acc += v[m];
        }
        acc = warp_sum_f32(acc);
        if (lane < pl.C)
            send_word(remote_addr(&sm.class_sum[buf][which * kClasses + pl.rank + pl.C * cl], lane), acc, remote_addr(&sm.red_bar[buf], lane));
    }
}
// kClean: the rows' maxima and whether a NaN was met, to every block
template <int WARPS, typename SM>
__device__ __forceinline__ void send_tops(SM& sm, const Place& pl, int flags) {
    const int lane = threadIdx.x & 31, buf = flags & kBuffer ? 1 : 0;
    if ((threadIdx.x >> 5) != WARPS - 1) return;
    const float mq = warp_max(lane < WARPS ? sm.warp_top[0][lane] : kNegInf), mp = warp_max(lane < WARPS ? sm.warp_top[1][lane] : kNegInf);
    if (lane < pl.C) {
        const uint32_t bar = remote_addr(&sm.red_bar[buf], lane);
        send_word(remote_addr(&sm.extra[buf][0][pl.rank], lane), mq, bar);
        send_word(remote_addr(&sm.extra[buf][1][pl.rank], lane), mp, bar);
        send_word(remote_addr(&sm.extra[buf][2][pl.rank], lane), sm.nan_seen ? 1.0f : 0.0f, bar);
    }
}
// a tile's normalised weights to global memory
template <typename T>
__device__ __forceinline__ void write_tile(float* out, int tile, int lane, int V, const float (&w)[16], double inv) {
    constexpr int kPer = 16 / (int)sizeof(T);
    const bool vec = ((uintptr_t)out & 15u) == 0;
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const int x = tile * kTileElems + ((i / kPer) * 32 + lane) * kPer + i % kPer;
        float o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) o[j] = (float)((double)w[i + j] * inv);
        if (vec && x + 4 <= V) {
            *(float4*)(out + x) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (x + j < V) out[x + j] = o[j];
        }
    }
}

// The working warps: the passes they are told to run.  The root's rows are asked for before the first command is there.
// MODE: which of the rarer passes exist.
template <typename T, int NT, int WARPS, int MODE>
__device__ __forceinline__ void work(ChipSmem<WARPS, NT>& sm, float4* draft_sm, const Place& pl, const WorkRows& rows) {
    constexpr int kAll = (WARPS + 1) * 32, kWorkers = WARPS * 32;
    constexpr int kPer = 16 / (int)sizeof(T), kRuns = 16 / kPer;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = pl.C, V = pl.V, n_tiles = pl.n_tiles;
    const int tile0 = pl.rank + C * warp, tile_step = C * WARPS;   // this warp's tiles: tile0, tile0 + tile_step, ...
    float q[NT][16];
    DraftTiles<T, NT> draft(draft_sm + warp * NT * 128);
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
        for (int j = 0; j < 16; ++j) q[k][j] = 0.0f;
    int flags = (rows.with_draft ? kOpen : kOpenTarget) | kFirst, node = 0;
    float a_hi = 0.0f, a_lo = 0.0f;
    for (;;) {
        int kind = flags & kKindMask;
        float s[NT];
        if (kind == kOpen || kind == kOpenTarget) {
            Packed<T> rq[NT];
            const char* rowq = rows.q + (int64_t)node * rows.stride_q;
            const char* rowp = rows.p + (int64_t)node * rows.stride_p;
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                const int tile = tile0 + tile_step * k;
                rq[k].fill_neg_inf();
                if (!draft.kShared || tile >= n_tiles) draft.clear(k);
                if (tile < n_tiles) {
                    load_tile<T>(rq[k], rowq, tile, lane, V);
                    if (kind == kOpen) draft.ask(k, rowp, tile, lane, V);
                }
            }
            if (flags & kFirst) {
                cluster_wait();         // every block's mbarriers are in place
                cmd_sync<kAll>(0);
                flags = sm.cmd[0].flags;   // the root's rows, with or without the draft row
                kind = flags & kKindMask;
            }
            float cq = 0.0f, cp = 0.0f;
            const bool precise = rows.precise && !(flags & kRelative);
            if (flags & (kClean | kRelative)) {
                if (flags & kRelative) { cq = sm.ref_q; cp = sm.ref_p; }
                if (flags & kClean) {
                    float mq = kNegInf, mp = kNegInf;
                    bool saw_nan = false;
#pragma unroll
                    for (int k = 0; k < NT; ++k) {
                        mq = fmaxf(mq, clean_tile(rq[k], saw_nan));
                        if (kind == kOpen) {
                            if (k == 0) draft.landed();
                            Packed<T> rp;
                            draft.get_raw(k, rp);
                            mp = fmaxf(mp, clean_tile(rp, saw_nan));
                            draft.put_raw(k, rp);
                        }
                    }
                    mq = warp_max(mq);
                    mp = warp_max(mp);
                    if (lane == 0) { sm.warp_top[0][warp] = mq; sm.warp_top[1][warp] = mp; }
                    if (saw_nan) sm.nan_seen = 1;
                }
            }
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                rq[k].unpack(q[k]);
                if (precise) exp16_precise(q[k], rows.kq, q[k]);
                else exp16(q[k], rows.kq, cq, q[k]);
                s[k] = tree_sum16(q[k]);
            }
            draft.landed();
            if (kind == kOpen) {
#pragma unroll
                for (int k = 0; k < NT; ++k) {
                    Packed<T> rp;
                    draft.get_raw(k, rp);
                    float p[16];
                    rp.unpack(p);
                    if (precise) exp16_precise(p, rows.kp, p);
                    else exp16(p, rows.kp, cp, p);
                    draft.put(k, p);
                    sm.lane_sum[1][warp + WARPS * k][lane] = tree_sum16(p);
                }
            }
        } else if (kind == kResidualPass) {
            if (MODE == kResample && (flags & kFreeze)) {
                const int x = sm.freeze_x;
                int l_, j_;
                walk_ring::piece_of<T>(x % kTileElems, l_, j_);
#pragma unroll
                for (int k = 0; k < NT; ++k)
                    if (tile0 + tile_step * k == x / kTileElems && l_ == lane) {
                        float p[16];
                        draft.get(k, p);
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (j == j_) { q[k][j] = residual_weight(q[k][j], p[j], sm.freeze_hi, sm.freeze_lo); p[j] = 0.0f; }
                        draft.put(k, p);
                    }
            }
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                float p[16], w[16];
                draft.get(k, p);
                residual16(q[k], p, a_hi, a_lo, w);
                s[k] = tree_sum16(w);
            }
        } else if (kind == kPlainPass) {
#pragma unroll
            for (int k = 0; k < NT; ++k) s[k] = tree_sum16(q[k]);
        } else if (kind == kRestPass) {
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                uint32_t gone = 0;
                for (int i = 0; i < sm.n_gone_tok; ++i) {
                    const int o = sm.gone_tok[i] - (tile0 + tile_step * k) * kTileElems;
                    if (o < 0 || o >= kTileElems) continue;
                    int l_, j_;
                    walk_ring::piece_of<T>(o, l_, j_);
                    if (l_ == lane) gone |= 1u << j_;
                }
                float p[16], w[16];
                draft.get(k, p);
#pragma unroll
                for (int j = 0; j < 16; ++j) w[j] = ((gone >> j) & 1u) ? 0.0f : p[j];
                s[k] = tree_sum16(w);
            }
        } else if (MODE == kRuleWalk && (kind == kOverlapPass || kind == kSeqPass)) {
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                float p[16], w[16];
                draft.get(k, p);
                if (kind == kOverlapPass) weights16<kSeqOverlap>(q[k], p, a_hi, a_lo, 0.0f, w);
                else weights16<kSeqResidual>(q[k], p, a_hi, a_lo, sm.c_seq, w);
                s[k] = tree_sum16(w);
            }
        } else if (kind == kDump) {
#pragma unroll
            for (int k = 0; k < NT; ++k)
                if (tile0 + tile_step * k == node) {
                    float p[16], w[16];
                    draft.get(k, p);
                    mode_weights<MODE == kRuleWalk>(flags >> kModeShift, q[k], p, a_hi, a_lo, MODE == kRuleWalk ? sm.c_seq : 0.0f, w);
#pragma unroll
                    for (int i = 0; i < kRuns; ++i)
#pragma unroll
                        for (int j = 0; j < kPer; ++j) sm.tile_w[(i * 32 + lane) * kPer + j] = w[i * kPer + j];
                }
            dump_sync<kAll>();
        } else if (MODE == kResample && kind == kWrite) {
            dump_sync<kAll>();                  // everyone has read the command
            const double inv = sm.inv_total;
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                const int tile = tile0 + tile_step * k;
                if (tile >= n_tiles) continue;
                float p[16], w[16];
                draft.get(k, p);
                mode_weights<false>(flags >> kModeShift, q[k], p, a_hi, a_lo, 0.0f, w);
                write_tile<T>(rows.out_residual, tile, lane, V, w, inv);
            }
        } else if (MODE == kRuleWalk && kind == kTop1) {
            top1_pass<T, NT, WARPS>(sm, pl, rows.key, (uint32_t)node, flags, a_hi, a_lo, q, draft);
        } else {
            return;                             // kEnd
        }
        if (kind < kDump) {                     // the pass reports sums
#pragma unroll
            for (int k = 0; k < NT; ++k) sm.lane_sum[0][warp + WARPS * k][lane] = s[k];
            workers_sync<kWorkers>();           // the lanes' sums are in place
            const int buf = flags & kBuffer ? 1 : 0;
            send_class_sums<WARPS>(sm, pl, flags);
            if (flags & kStoreTiles) {
#pragma unroll
                for (int k = 0; k < NT; ++k) {
                    const int tile = tile0 + tile_step * k;
                    const float ts = warp_sum_f32(s[k]);
                    if (lane < C && tile < n_tiles) send_word(remote_addr(&sm.tile_sum[tile], lane), ts, remote_addr(&sm.red_bar[buf], lane));
                }
            }
            if (flags & kClean) send_tops<WARPS>(sm, pl, flags);
        }
        const int odd = flags & kBuffer ? 0 : 1;   // the next command
        cmd_sync<kAll>(odd);
        const Cmd cmd = sm.cmd[odd];
        flags = cmd.flags;
        node = cmd.node;
        a_hi = cmd.a_hi;
        a_lo = cmd.a_lo;
    }
}

// Sum over the eight classes in lanes 8 i .. 8 i + 7 as ((0+1)+(2+3))+((4+5)+(6+7)), on each of those lanes.
__device__ __forceinline__ double class_tree(double v) {
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__device__ __forceinline__ bool sum_usable(double s) { return s >= (double)kSumFloor && s < 1e300; }

// The control warp: the walk itself, the same in every block of the cluster.
template <typename T, typename SM, int WARPS, int MODE>
struct Control {
    static constexpr int kAll = (WARPS + 1) * 32;
    SM& sm;
    const ClusterArgs& ca;
    const VerifyArgs& a;
    const Place& pl;
    const int b;
    const bool precise;
    const int lane;
    const RngKey key;
    int cmd_no, backward;           // (the passes are the first commands: a walk's dump and end come last)
    bool aborted;
    float kq, kp, mq, mp;           // log2(e) / temperature; references of the exponentials (raw units)
    double Sq, Sp, inv_Sq, inv_Sp, ratio;
    double A, Z;                    // closed-form chain (see rsd_verify.cuh)
    float a_hi, a_lo;               // A Sq / Sp as a two-float sum
    int status;

    __device__ __forceinline__ Control(SM& sm_, const ClusterArgs& ca_, const Place& pl_, int b_, bool precise_)
        : sm(sm_), ca(ca_), a(ca_.v), pl(pl_), b(b_), precise(precise_), lane(threadIdx.x & 31),
          key{ca_.v.seed_lo, ca_.v.seed_hi, ca_.v.step, ca_.v.seq_base + (uint32_t)b_}, cmd_no(0), backward(0), aborted(false),
          kq(kLog2e * ca_.v.target.inv_temp), kp(kLog2e * ca_.v.draft.inv_temp), mq(0.0f), mp(0.0f), A(0.0), Z(1.0), a_hi(0.0f), a_lo(0.0f),
          status(0) {}

    __device__ __forceinline__ void publish(int flags, int node) {
        const int odd = cmd_no & 1;
        if (lane == 0) {
            Cmd cmd;
            cmd.flags = flags | (odd ? kBuffer : 0);
            cmd.node = node;
            cmd.a_hi = a_hi;
            cmd.a_lo = a_lo;
            sm.cmd[odd] = cmd;
        }
        cmd_arrive<kAll>(odd);
        ++cmd_no;
    }
    // publish a pass that reports `words` words to every block
    __device__ __forceinline__ void issue(int flags, int node, int words) {
        if (lane == 0) mbar_expect_tx(&sm.red_bar[cmd_no & 1], 4u * (uint32_t)words);
        publish(flags | (backward ? kBackward : 0), node);
        backward ^= 1;
    }
    // wait for the words of the latest pass; sets `aborted` when they do not come
    __device__ __forceinline__ int land() {
        const int n = cmd_no - 1, buf = n & 1;
        int late = 0;
        wait_bar(&sm.red_bar[buf], (uint32_t)(n >> 1) & 1u, &late);
        if (__any_sync(0xFFFFFFFFu, late)) aborted = true;
        return buf;
    }
    __device__ __forceinline__ double collect() {        // one sum
        const int buf = land();
        return __shfl_sync(0xFFFFFFFFu, class_tree((double)sm.class_sum[buf][lane & (kClasses - 1)]), 0);
    }
    __device__ __forceinline__ void collect2(double& s0, double& s1) {
        const int buf = land();
        const double v = class_tree((double)sm.class_sum[buf][lane & (2 * kClasses - 1)]);
        s0 = __shfl_sync(0xFFFFFFFFu, v, 0);
        s1 = __shfl_sync(0xFFFFFFFFu, v, kClasses);
    }

    __device__ __forceinline__ void issue_open(int node, bool with_draft, int options) {
        issue((with_draft ? kOpen : kOpenTarget | kStoreTiles) | options, node,
              (with_draft ? 2 * kClasses : kClasses + pl.n_tiles) + (options & kClean ? 3 * pl.C : 0));
    }
    // The sums of a node whose first pass, relative to 0, has been issued.  If they are not finite, or so small that
    // underflow may have eaten them, a cleaning pass finds the rows' maxima and the pass is run again relative to them.
    __device__ __forceinline__ void open_sums(int node, bool with_draft) {
        A = 0.0; Z = 1.0; a_hi = a_lo = 0.0f; mq = mp = 0.0f;
        double s0, s1;
        collect2(s0, s1);
        if (!with_draft) s1 = 1.0;
        if (!(sum_usable(s0) && sum_usable(s1)) && !aborted) {
            issue_open(node, with_draft, kClean);
            collect2(s0, s1);
            if (!with_draft) s1 = 1.0;
            const int buf = (cmd_no - 1) & 1;
            float top_q = kNegInf, top_p = kNegInf;
            bool saw_nan = false;
            for (int i = 0; i < pl.C; ++i) {
                top_q = fmaxf(top_q, sm.extra[buf][0][i]);
                top_p = fmaxf(top_p, sm.extra[buf][1][i]);
                saw_nan |= sm.extra[buf][2][i] != 0.0f;
            }
            if (saw_nan) status |= 1;              // RSD_ST_NAN_INPUT
            if (!(sum_usable(s0) && sum_usable(s1)) && !aborted) {
                if (top_q > kNegInf) mq = top_q;
                if (with_draft && top_p > kNegInf) mp = top_p;
                if (lane == 0) { sm.ref_q = mq * kq; sm.ref_p = mp * kp; }
                issue_open(node, with_draft, (saw_nan ? kClean : 0) | kRelative);
                collect2(s0, s1);
                if (!with_draft) s1 = 1.0;
            }
            if (lane == 0) sm.nan_seen = 0;        // (published with the next command)
        }
        Sq = s0;
        Sp = s1;
    }
    __device__ __forceinline__ void set_a(double A_) {
        A = A_;
        const double aa = A * ratio;
        a_hi = (float)aa;
        a_lo = (float)(aa - (double)a_hi);
    }
    // weight of a token with row value l as the working warps take it (NaN: 0)
    __device__ __forceinline__ float weight(float l, float k, float m) const {
        if (precise && m == 0.0f) return weight_precise(l, k);
        return l == l ? ex2_approx(fmaf(l, k, -m * k)) : 0.0f;
    }
    __device__ __forceinline__ void take_in(double Z_new, double A_old, bool& kept) {
        if (Z_new > 0.0 && Z_new < 1.7e308) {
            Z = Z_new;
            kept = true;
        } else {
            status |= 4;   // RSD_ST_ZERO_RESIDUAL: keep the previous residual
            set_a(A_old);
            kept = false;
        }
    }

    // a node's first 32 children after node `after`, in stored order, one per lane (-1: none)
    __device__ __forceinline__ int children(int of, int after, const int32_t* par, const int32_t* tok, bool cached) {
        int found = 0;
        sm.kid_node[lane] = -1;
        __syncwarp();
        for (int c0 = after + 1; c0 < a.num_nodes && found < 32; c0 += 32) {
            const int cc = c0 + lane;
            bool ok = false;
            if (cc < a.num_nodes) {
                const int pn = cached ? sm.par[cc] : par[cc];
                const int t = cached ? sm.tok[cc] : tok[cc];
                ok = pn == of && t >= 0 && t < pl.V;
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, ok);
            const int at = found + __popc(m & ((1u << lane) - 1u));
            if (ok && at < 32) sm.kid_node[at] = cc;
            found += __popc(m);
        }
        __syncwarp();
        const int r = sm.kid_node[lane];
        __syncwarp();
        return r;
    }

    // The last token under the weights of `mode` and its block's outputs.  Every block knows the tile sums; the block
    // that holds the crossing's tile ends the draw.  Returns true on the block that has the token in `last`.
    __device__ __forceinline__ bool draw(int mode, uint32_t node, int& last) {
        const uint4 rw = rng_draw(key, node, kTagResample, 0u);
        const double u = ((double)rw.x + 0.5) * (1.0 / 4294967296.0);
        walk_ring::TilePick t;
        walk_ring::pick_tile(sm.tile_sum, pl.n_tiles, u, t);
        if (t.tile < 0) { last = -1; return pl.rank == 0; }
        if (t.tile % pl.C != pl.rank) return false;
        publish(kDump | (mode << kModeShift), t.tile);
        dump_sync<kAll>();
        float w[16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 f = *(const float4*)&sm.tile_w[16 * lane + 4 * i];
            w[4 * i] = f.x; w[4 * i + 1] = f.y; w[4 * i + 2] = f.z; w[4 * i + 3] = f.w;
        }
        last = walk_ring::pick_in_tile(w, t);
        return true;
    }
    __device__ __forceinline__ bool draw_top1(int mode, uint32_t node, int& last) {
        issue(kTop1 | (mode << kModeShift), (int)node, 2 * pl.C);
        land();
        unsigned long long best = ~0ull;
        for (int i = 0; i < pl.C; ++i) best = min(best, sm.top1[i]);
        last = aborted || best == ~0ull ? -1 : (int)(uint32_t)best;
        return pl.rank == 0;
    }
    // after a walk whose latest pass does not hold the tile sums of what the last token is drawn from
    __device__ __forceinline__ double refresh_tiles(bool residual) {
        issue((residual ? kResidualPass : kPlainPass) | kStoreTiles, 0, kClasses + pl.n_tiles);
        return collect();
    }
    __device__ __forceinline__ void end_work() {
        publish(kEnd, 0);
        if (aborted) {
            status |= 32;            // RSD_ST_TIMEOUT
            if (lane == 0) store_remote(remote_addr(&sm.gave_up, 0), 1);
        }
    }
    // What is left of the draft once subtraction has lost its accuracy: summed anew without the rejected tokens.
    __device__ __forceinline__ double rest(int n_removed) {
        if (lane == 0) sm.n_gone_tok = n_removed;
        issue(kRestPass, 0, kClasses);
        return collect() * inv_Sp;
    }

    __device__ __forceinline__ void walk() {
        const int32_t* par = a.parent + (a.shared_topology ? 0 : (int64_t)b * a.num_nodes);
        const int32_t* tok = a.token + (int64_t)b * a.num_nodes;
        const bool cached = a.num_nodes <= kMaxCachedNodes;
        const int rule = (MODE == kRuleWalk) ? a.rule : 0;
        const int64_t out0 = (int64_t)b * a.L;
        if (cached) {
#pragma unroll 4
            for (int n = lane; n < a.num_nodes; n += 32) { sm.par[n] = par[n]; sm.tok[n] = tok[n]; }
            __syncwarp();
        }
        int cur = 0, len = 0, reason = 0, seq_kids = 0;
        bool tiles_valid = false, with_draft;
        int child_node = children(0, 0, par, tok, cached);
        unsigned kids = __ballot_sync(0xFFFFFFFFu, child_node >= 0);
        with_draft = kids != 0u && a.L > 0;
        cluster_wait();                               // every block's mbarriers are in place
        issue_open(0, with_draft, 0);
        if (pl.rank == 0) {
            for (int i = lane; i < a.L; i += 32) {
                a.accepted_node[out0 + i] = -1;
                a.accepted_token[out0 + i] = -1;
            }
            if (a.dbg_theta)
                for (int n = lane; n < a.num_nodes; n += 32) a.dbg_theta[(int64_t)b * a.num_nodes + n] = __int_as_float(0x7FC00000);
            __syncwarp();
        }
        for (;;) {
            // ---- the node `cur` is being opened: what its children need, one child per lane ---------------------------------
            if (!with_draft) {
                open_sums(cur, false);
                tiles_valid = true;
                reason = len >= a.L ? 2 : 1;          // RSD_STOP_LEAF : RSD_STOP_NO_CHILDREN
                break;
            }
            const char* rowq = row_ptr<T>(a.target, b, cur);
            const char* rowp = row_ptr<T>(a.draft, b, cur);
            int j0 = 0, n_removed = 0;                // children are looked at 32 at a time: j0 is the rank of lane 0's
            int child_x;
            float lq, lp;
            double Ud;
            bool repeated, p_none;                    // p_none: the draft row gives the token no mass (-inf or NaN)
            float qh, ph;                             // the token's weights under the two rows
            walk_ring::WeightRatio qp_rows;
            auto child_weights = [&] {
                qh = weight(lq, kq, mq);
                ph = weight(lp, kp, mp);
                p_none = !(lp > kNegInf);
                qp_rows = walk_ring::WeightRatio(lq, kq, mq * kq, lp, kp, mp * kp);
            };
            auto fetch_children = [&] {
                child_x = -1;
                lq = lp = 0.0f;
                if (child_node >= 0) {
                    child_x = cached ? sm.tok[child_node] : tok[child_node];
                    lq = RowIO<T>::scalar(rowq, child_x);
                    lp = RowIO<T>::scalar(rowp, child_x);
                }
                const uint4 rw = rng_draw(key, (uint32_t)cur, kTagAccept, (uint32_t)(j0 + lane));
                Ud = (double)(rw.x >> 8) * (1.0 / 16777216.0);
                // an earlier sibling with the same token: rejected by the time this one is tested, its draft mass is gone (Eq. 1)
                const unsigned same = __match_any_sync(0xFFFFFFFFu, child_x);
                repeated = (same & ((1u << lane) - 1u)) != 0u;
                if (j0 > 0) {
                    bool listed = false;
                    for (int i = 0; i < n_removed; ++i) listed |= sm.gone_tok[i] == child_x;
                    if (n_removed + 32 > kMaxListed) {   // (the ring walk does not know a token again that it has not listed)
                        const int first = __ffs(same) - 1;
                        const unsigned fresh = __ballot_sync(0xFFFFFFFFu, !listed && !repeated);
                        repeated = repeated && n_removed + __popc(fresh & ((1u << first) - 1u)) < kMaxListed;
                    }
                    repeated |= listed;
                }
                if (rule != 0) repeated = false;      // (the baselines never change the draft)
            };
            fetch_children();
            mq = mp = 0.0f;
            child_weights();
            int next_kid = children(__shfl_sync(0xFFFFFFFFu, child_node, 0), 0, par, tok, cached);
            open_sums(cur, true);
            if (aborted) break;
            inv_Sq = 1.0 / Sq;
            inv_Sp = 1.0 / Sp;
            ratio = Sq * inv_Sp;
            const double sp_over_sq = Sp * inv_Sq;
            double qpd;                               // q(x) / p(x)
            unsigned none_left, repeats;              // children that the draft cannot produce any more; those among them that repeat
            auto weigh_children = [&] {
                // Precise weights: the quotient of the very weights that the sums are made of, as long as they are in range, so
                // that their errors cancel where the token carries much of the residual.
                if (precise && qh > 1e-30f && ph > 1e-30f) qpd = (double)qh / (double)ph * sp_over_sq;
                else qpd = qp_rows.times(sp_over_sq);
                none_left = __ballot_sync(0xFFFFFFFFu, repeated || p_none);
                repeats = __ballot_sync(0xFFFFFFFFu, repeated);
            };
            if (mq != 0.0f || mp != 0.0f) child_weights();   // (the references have moved)
            weigh_children();
            // 1 - P of the closed form (see the ring walk: summed anew once subtraction loses accuracy)
            double one_mP = 1.0, one_mP_err = 0.0, inv_1mP = 1.0;
            int j = 0, accepted_lane = -1;            // j: lane of the child under test
            for (;;) {
                // Eq. 3 in closed form: accept iff U < min(1, (q/p - A)+ (1 - P) / Z).  Every lane tests its own child, lane j's
                // counts.  A child the draft cannot produce any more is taken iff it has residual mass (RSD_ST_ZERO_DRAFT_PROB).
                double g = fmax(qpd - A, 0.0) * one_mP;
                bool take = Ud * Z < g;
                if ((MODE == kRuleWalk) && rule == 2) {   // K-SEQ: min(1, q / (gamma p))
                    g = qpd / (double)a.gamma;
                    take = Ud < g;
                }
                if ((none_left >> j) & 1u) {
                    status |= 8;
                    const double qx = (double)qh * inv_Sq;
                    const bool any = (MODE == kRuleWalk) && rule == 2 ? qx > 0.0 : fmax(qx - A * ((double)ph * inv_Sp), 0.0) > 0.0;
                    if (lane == j) {
                        take = any;
                        g = any ? ((MODE == kRuleWalk) && rule == 2 ? 1.0 : Z) : 0.0;
                    }
                }
                const unsigned taken = __ballot_sync(0xFFFFFFFFu, take);
                if (a.dbg_theta && pl.rank == 0 && lane == j)
                    a.dbg_theta[(int64_t)b * a.num_nodes + child_node] = (float)fmin(1.0, ((MODE == kRuleWalk) && rule == 2) ? g : g / Z);
                if ((taken >> j) & 1u) { accepted_lane = j; break; }
                // rejected.  Eqs. 1-2 in closed form: A_{j+1} = A_j + Z_j / (1 - P_j), Z_{j+1} = sum (q - A_{j+1} p)+
                const bool more_here = j < 31 && ((kids >> (j + 1)) & 1u);
                const int more_nodes = (j == 31 && kids == 0xFFFFFFFFu) ? children(cur, __shfl_sync(0xFFFFFFFFu, child_node, 31), par, tok, cached) : -1;
                const bool more = more_here || __any_sync(0xFFFFFFFFu, more_nodes >= 0);
                const double A_old = A;
                if (!((MODE == kRuleWalk) && rule == 2)) {
                    set_a(fma(Z, inv_1mP, A));
                    issue(kResidualPass | (more ? 0 : kStoreTiles), 0, kClasses + (more ? 0 : pl.n_tiles));
                }
                const int x = __shfl_sync(0xFFFFFFFFu, child_x, j);
                const bool rep = (repeats >> j) & 1u;
                const double px = ((MODE == kRuleWalk) && rule != 0) || ((none_left >> j) & 1u) ? 0.0 : (double)__shfl_sync(0xFFFFFFFFu, ph, j) * inv_Sp;
                double one_mP_new = one_mP - px, err_new = one_mP_err + 4e-7 * px;   // (px = 0 for a repeated token)
                if (!rep && n_removed < kMaxListed) {
                    if (lane == 0) sm.gone_tok[n_removed] = x;
                    ++n_removed;
                    __syncwarp();
                }
                inv_1mP = 1.0 / one_mP_new;
                if (more) {
                    if (more_here) {
                        ++j;
                    } else {                          // the next 32 children
                        child_node = more_nodes;
                        kids = __ballot_sync(0xFFFFFFFFu, child_node >= 0);
                        j0 += 32;
                        j = 0;
                        fetch_children();
                        child_weights();
                        weigh_children();
                    }
                    next_kid = children(__shfl_sync(0xFFFFFFFFu, child_node, j), 0, par, tok, cached);
                }
                if (!((MODE == kRuleWalk) && rule == 2)) {
                    const double Z_new = collect() * inv_Sq;
                    if (aborted) break;
                    bool kept;
                    take_in(Z_new, A_old, kept);
                    tiles_valid = kept && !more;
                }
                if (!((MODE == kRuleWalk) && rule != 0)) {
                    if (more && err_new > 2e-6 * one_mP_new && n_removed < kMaxListed) {   // (every rejected token is listed)
                        one_mP_new = rest(n_removed);
                        if (aborted) break;
                        err_new = 4e-7 * one_mP_new;
                        inv_1mP = 1.0 / one_mP_new;
                    }
                    one_mP = one_mP_new;
                    one_mP_err = err_new;
                    if (!(one_mP > 0.0)) { status |= 16; break; }   // RSD_ST_DRAFT_EXHAUSTED
                }
                if (!more) { ++j; break; }
            }
            if (aborted) break;
            if (accepted_lane < 0) {   // RSD_STOP_ALL_REJECTED: the last token comes from the residual in force
                reason = 0;
                seq_kids = j0 + j;
                break;
            }
            const int x = __shfl_sync(0xFFFFFFFFu, child_x, accepted_lane);
            cur = __shfl_sync(0xFFFFFFFFu, child_node, accepted_lane);
            child_node = next_kid;
            kids = __ballot_sync(0xFFFFFFFFu, child_node >= 0);
            with_draft = kids != 0u && len + 1 < a.L;
            backward = 0;
            tiles_valid = false;
            issue_open(cur, with_draft, 0);
            if (lane == 0 && pl.rank == 0) {
                a.accepted_node[out0 + len] = cur;
                a.accepted_token[out0 + len] = x;
            }
            ++len;
        }
        int mode = with_draft && A != 0.0 ? (int)kResidual : 0;
        if ((MODE == kRuleWalk) && !aborted && rule == 2 && with_draft) {
            // K-SEQ after all K children were rejected: beta = sum min{p, q / gamma}, then the residual
            // (q - min{p, q / gamma} (1 - (1 - beta)^K) / beta)+
            a_hi = (float)(Sq / Sp);
            a_lo = (float)(1.0 / (double)a.gamma);
            issue(kOverlapPass, 0, kClasses);
            const double beta = collect() / Sq;
            double miss = 1.0;
            for (int i = 0; i < seq_kids; ++i) miss *= 1.0 - beta;
            const float c = (float)(beta > 0.0 ? (1.0 - miss) / beta : (double)seq_kids);
            if (!aborted) {
                if (lane == 0) sm.c_seq = c;
                issue(kSeqPass | kStoreTiles, 0, kClasses + pl.n_tiles);
                const double t = collect();
                tiles_valid = t > 0.0 && t < 1.7e308;
                if (tiles_valid) mode = kSeqResidual;
                else status |= 4;                     // RSD_ST_ZERO_RESIDUAL: draw from the target row itself
            }
        }
        const bool top1 = (MODE == kRuleWalk) && a.final_sampler == 1;
        if (!aborted && !tiles_valid && !top1) refresh_tiles(mode == kResidual);
        int last = -1;
        bool mine = pl.rank == 0;
        if (!aborted) mine = top1 ? draw_top1(mode, (uint32_t)cur, last) : draw(mode, (uint32_t)cur, last);
        end_work();
        if (lane == 0) {
            if (mine) a.last_token[b] = last;
            if (pl.rank == 0) {
                a.accepted_len[b] = len;
                a.stop_reason[b] = reason;
                a.status[b] = status;
            }
        }
    }

    // The stand-alone residual draw: the tokens of a list are rejected in order, then one token is drawn.  A listed token
    // keeps the residual mass it has when it is removed (its draft probability is 0 afterwards): the pass after freezes it.
    __device__ __forceinline__ void resample() {
        const ResampleArgs& r = ca.r;
        int tok = -1;
        if (r.rejected && lane < r.max_k) tok = r.rejected[(int64_t)b * r.max_k + lane];
        if (tok < 0 || tok >= pl.V) tok = -1;
        unsigned left = __ballot_sync(0xFFFFFFFFu, tok >= 0);
        const bool with_draft = left != 0u;
        cluster_wait();
        issue_open(0, with_draft, 0);
        const char* rowp = row_ptr<T>(a.draft, b, 0);
        const float lp = tok >= 0 ? RowIO<T>::scalar(rowp, tok) : 0.0f;
        const bool repeated = (__match_any_sync(0xFFFFFFFFu, tok) & ((1u << lane) - 1u)) != 0u;   // listed twice
        const uint32_t node = (uint32_t)r.rng_node[b];
        open_sums(0, with_draft);
        inv_Sq = 1.0 / Sq;
        inv_Sp = 1.0 / Sp;
        ratio = Sq * inv_Sp;
        double total = Sq;
        bool tiles_valid = !with_draft;
        const double px_row = (double)weight(lp, kp, mp) * inv_Sp;
        double one_mP = 1.0, one_mP_err = 0.0;
        int n_removed = 0, freeze = 0;
        while (left && !aborted) {
            const int j = __ffs(left) - 1;
            left &= left - 1u;
            const double A_old = A;
            set_a(A + Z / one_mP);
            issue(kResidualPass | freeze | (left ? 0 : kStoreTiles), 0, kClasses + (left ? 0 : pl.n_tiles));
            freeze = 0;
            const bool rep = (__ballot_sync(0xFFFFFFFFu, repeated) >> j) & 1u;
            const int x = __shfl_sync(0xFFFFFFFFu, tok, j);
            const double px = rep ? 0.0 : __shfl_sync(0xFFFFFFFFu, px_row, j);
            const double zhat = collect();
            if (aborted) break;
            bool kept;
            take_in(zhat * inv_Sq, A_old, kept);
            if (kept) total = zhat;
            tiles_valid = kept && !left;
            if (!rep) {
                if (lane == 0) { sm.gone_tok[n_removed] = x; sm.freeze_x = x; sm.freeze_hi = a_hi; sm.freeze_lo = a_lo; }
                ++n_removed;
                freeze = kFreeze;
            }
            one_mP -= px;
            one_mP_err += 4e-7 * px;
            if (one_mP_err > 2e-6 * one_mP && left) {
                one_mP = rest(n_removed);
                one_mP_err = 4e-7 * one_mP;
            }
            if (!(one_mP > 0.0)) { status |= 16; break; }   // RSD_ST_DRAFT_EXHAUSTED
        }
        const int mode = with_draft && A != 0.0 ? (int)kResidual : 0;
        if (!aborted && !tiles_valid) total = refresh_tiles(mode == kResidual);
        int last = -1;
        bool mine = pl.rank == 0;
        if (!aborted) {
            mine = draw(mode, node, last);
            if (r.out_residual) {
                if (lane == 0) sm.inv_total = total > 0.0 ? 1.0 / total : 0.0;
                publish(kWrite | (mode << kModeShift), 0);
                dump_sync<kAll>();   // (the command has been read: its place may take the next one)
            }
        }
        end_work();
        if (lane == 0) {
            if (mine) r.out_token[b] = last;
            if (pl.rank == 0) r.status[b] = status;
        }
    }
};

// By a thread of rank 0 when the cluster is through: a wait ran out in some block, which the sequence's outputs say.  (That block need
// not be the one that has written them; what was written so far is ordered before this by the cluster's barrier.)
template <int MODE>
__device__ __forceinline__ void report_timeout(const ClusterArgs& ca, int b) {
    (MODE == kResample ? ca.r.out_token : ca.v.last_token)[b] = -1;
    (MODE == kResample ? ca.r.status : ca.v.status)[b] |= 32;   // RSD_ST_TIMEOUT
}

// A walk by the blocks of a cluster: `work` is what the working warps do.
template <typename T, int MODE, int WARPS, typename SM, typename F>
__device__ __forceinline__ void run_walk(SM& sm, const ClusterArgs& ca, F&& work) {
    const VerifyArgs& a = ca.v;
    Place pl;
    pl.rank = (int)cluster_rank();
    pl.C = (int)cluster_size();
    pl.V = a.V;
    pl.n_tiles = (a.V + kTileElems - 1) / kTileElems;
    pl.per_block = kClasses / pl.C;
    pl.n_local = pl.n_tiles > pl.rank ? (pl.n_tiles - pl.rank + pl.C - 1) / pl.C : 0;
    const int b = blockIdx.x / pl.C;
    // Rows that the ring walk does not take, the baseline rules and the residual draw have no bits to match.
    const bool precise = MODE != kPlainWalk || !ca.ring_rows;
    if (threadIdx.x == WARPS * 32) {
        mbar_init(&sm.red_bar[0], 1);
        mbar_init(&sm.red_bar[1], 1);
        sm.nan_seen = 0;
        sm.gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_arrive();
    grid_wait();   // the tree, and whatever else the stream has on the way
    if (threadIdx.x < WARPS * 32) {
        WorkRows rows;
        rows.q = row_ptr<T>(a.target, b, 0);
        rows.p = row_ptr<T>(a.draft, b, 0);
        rows.stride_q = a.target.row_stride * RowIO<T>::kBytes;
        rows.stride_p = a.draft.row_stride * RowIO<T>::kBytes;
        rows.kq = kLog2e * a.target.inv_temp;
        rows.kp = kLog2e * a.draft.inv_temp;
        rows.with_draft = MODE == kResample ? ca.r.max_k > 0 : (a.L > 0 && a.num_nodes > 1);
        rows.precise = precise;
        rows.key = RngKey{a.seed_lo, a.seed_hi, a.step, a.seq_base + (uint32_t)b};
        rows.out_residual = MODE == kResample && ca.r.out_residual ? ca.r.out_residual + (int64_t)b * a.V : nullptr;
        work(pl, rows);
        grid_started();
        cluster_arrive();   // nothing is on its way to a block that has left
        cluster_wait();
    } else {
        Control<T, SM, WARPS, MODE> control(sm, ca, pl, b, precise);
        if constexpr (MODE == kResample) control.resample();
        else control.walk();
        grid_started();
        cluster_arrive();
        cluster_wait();
        if (threadIdx.x == WARPS * 32 && sm.gave_up) report_timeout<MODE>(ca, blockIdx.x / cluster_size());
    }
}

template <typename T, int NT, int WARPS, int MODE>
__global__ void __launch_bounds__((WARPS + 1) * 32, WARPS == 8 ? (NT == 1 ? 3 : 2) : 1) walk_cluster_kernel(const __grid_constant__ ClusterArgs ca) {
    __shared__ ChipSmem<WARPS, NT> sm;
    extern __shared__ __align__(16) float4 draft_sm[];
    run_walk<T, MODE, WARPS>(sm, ca, [&](const Place& pl, const WorkRows& rows) { work<T, NT, WARPS, MODE>(sm, draft_sm, pl, rows); });
}

}  // namespace walk_cluster
}  // namespace rsd
