// The residual draw with no rejected token: one token from softmax(target row), by one block per sequence.
//
// One sweep over the row leaves the sum of every 512-element tile, one warp finds the tile that the uniform falls into and takes
// that tile once more.  Tiles, exponentials and the order of all sums are those of the walk kernels (rsd_walk_cluster.cuh,
// rsd_walk_stream.cuh), which draw from few long rows: which of them runs does not show.
//
// Bound by latency, then by the exponentials.  There is no control warp and nothing to hand around, so a short row costs little more
// than its launch; two tiles of a warp are under way at a time, and four blocks on an SM (three or five: 71 or 62 us for 1024
// sequences of 128,000).  us for 1 / 256 / 1024 sequences, bf16, cluster against this: 1000 entries 6.2 / 6.9 / 20, 3.8 / 4.2 / 7.3;
// 32,000 6.2 / 27 / 101, 6.8 / 8.2 / 20; 128,000 7.2 / 130 / 503, 17 / 26 / 59.
#pragma once
#include "rsd_walk_cluster.cuh"

namespace rsd {
namespace walk_cluster {

constexpr int kDrawWarps = kClasses;     // a warp per summation class

struct DrawSmem {
    float tile_sum[kMaxTiles];
    float class_sum[kClasses];
    float top[kDrawWarps];
    int nan_seen;
};

template <typename T>
__global__ void __launch_bounds__(kDrawWarps * 32, 4) draw_target_kernel(const ResampleArgs r) {
    __shared__ DrawSmem sm;
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int V = r.V, n_tiles = (V + kTileElems - 1) / kTileElems;
    const char* row = row_ptr<T>(r.target, b, 0);
    const float k = kLog2e * r.target.inv_temp;
    bool dirty = false, relative = false;
    float c = 0.0f;                                    // reference of the exponentials, in units of log2
    if (threadIdx.x == 0) sm.nan_seen = 0;
    grid_wait();                                       // the row, and whatever else the stream has on the way
    auto weights = [&](Packed<T>& pk, float (&w)[16], bool& saw_nan) {   // returns the tile's largest value where that is looked at
        float top = kNegInf;
        if (dirty) top = clean_tile(pk, saw_nan);
        pk.unpack(w);
        if (relative) exp16(w, k, c, w);
        else exp16_precise(w, k, w);
        return top;
    };
    double S = 0.0;
    int status = 0;
    // As it is; without NaN if the sum is not usable; relative to the row's largest value if it still is not.  (The passes alternate in
    // direction, like those of the walks.)
    for (int pass = 0; pass < 3; ++pass) {
        float acc = 0.0f, top = kNegInf;
        bool saw_nan = false;
        const int n = n_tiles > warp ? (n_tiles - warp + kDrawWarps - 1) / kDrawWarps : 0;
        const int way = pass & 1 ? -kDrawWarps : kDrawWarps;
        int tile = pass & 1 ? warp + kDrawWarps * (n - 1) : warp;
        auto take = [&](Packed<T>& pk, int at) {
            float w[16];
            top = fmaxf(top, weights(pk, w, saw_nan));
            const float s = tree_sum16(w);
            acc += s;
            const float ts = walk_ring::warp_sum_f32(s);
            if (lane == 0) sm.tile_sum[at] = ts;
        };
        int m = 0;
        for (; m + 1 < n; m += 2, tile += 2 * way) {   // two tiles under way at a time
            Packed<T> pk0, pk1;
            load_tile<T>(pk0, row, tile, lane, V);
            load_tile<T>(pk1, row, tile + way, lane, V);
            take(pk0, tile);
            take(pk1, tile + way);
        }
        if (m < n) {
            Packed<T> pk;
            load_tile<T>(pk, row, tile, lane, V);
            take(pk, tile);
        }
        acc = walk_ring::warp_sum_f32(acc);
        top = warp_max(top);
        if (lane == 0) { sm.class_sum[warp] = acc; sm.top[warp] = top; }
        if (saw_nan) sm.nan_seen = 1;
        __syncthreads();
        S = class_tree((double)sm.class_sum[lane & (kClasses - 1)]);
        S = __shfl_sync(0xFFFFFFFFu, S, 0);
        if (sum_usable(S) || pass == 2) break;
        if (pass == 0) {
            dirty = true;
        } else {
            for (int i = 0; i < kDrawWarps; ++i) top = fmaxf(top, sm.top[i]);
            dirty = sm.nan_seen != 0;
            relative = true;
            c = (top > kNegInf ? top : 0.0f) * k;
        }
        __syncthreads();                               // everyone has read what the next pass overwrites
    }
    if (sm.nan_seen) status |= 1;                      // RSD_ST_NAN_INPUT
    if (r.out_residual) {
        const double inv = S > 0.0 ? 1.0 / S : 0.0;
        for (int tile = warp; tile < n_tiles; tile += kDrawWarps) {
            Packed<T> pk;
            load_tile<T>(pk, row, tile, lane, V);
            float w[16];
            bool dummy = false;
            weights(pk, w, dummy);
            write_tile<T>(r.out_residual + (int64_t)b * V, tile, lane, V, w, inv);
        }
    }
    grid_started();
    if (warp != 0) return;
    const RngKey key = {r.seed_lo, r.seed_hi, r.step, r.seq_base + (uint32_t)b};
    const uint4 rw = rng_draw(key, (uint32_t)r.rng_node[b], kTagResample, 0u);
    walk_ring::TilePick t;
    walk_ring::pick_tile(sm.tile_sum, n_tiles, ((double)rw.x + 0.5) * (1.0 / 4294967296.0), t);
    int last = -1;
    if (t.tile >= 0) {
        float w[16];                                   // tokens 16 lane .. 16 lane + 15 of the tile
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int x = t.tile * kTileElems + 16 * lane + j;
            w[j] = x < V ? RowIO<T>::scalar(row, x) : kNegInf;
            if (dirty && w[j] != w[j]) w[j] = kNegInf;
        }
        if (relative) exp16(w, k, c, w);
        else exp16_precise(w, k, w);
        last = walk_ring::pick_in_tile(w, t);
    }
    if (lane == 0) {
        r.out_token[b] = last;
        r.status[b] = status;
    }
}

}  // namespace walk_cluster
}  // namespace rsd
