// Logit warping of vocabulary rows: top-k and nucleus (top-p) filtering after the temperature (Section 4's sampling
// settings: temperature 0.3 / 1.0, nucleus 0.95).  A filtered token counts as log-probability -inf from then on, which
// is how the drafting and verification kernels already treat masked entries (Algorithms 4 and 9 drop them).
//
//   top-k   keep the k largest values (equal values: the smaller token first)
//   top-p   of what is left, in order of decreasing probability (equal values: the smaller token first), the
//           shortest prefix whose share of the mass reaches top_p (at least one token)
//
// One block per row.  The row is copied to shared memory once (NaN turned into -inf on the way); both cuts are then
// found without sorting, by a search for the value of the last kept token over the ordered bit patterns of the
// values:
//   sweep   the row once into a histogram of 1024 bins of equal width in value (where the tokens spread evenly).  A token
//           adds its weight exp(value / T) as a 32-bit fixed-point number, in two halves to two 32-bit counters, so the
//           sums are integers and do not depend on the order.  (Top-k: it adds 1.)
//   pick    the bin that brings the tally to what is needed, by a prefix sum over the block
//   gather  the few hundred tokens of that bin into a list, by tests on whole 16-byte words
//   finish  by one warp alone, the others waiting at a barrier: 32-way narrowing of the list's code interval down to one
//           value, then the last kept token among its equals
// A bin that holds more tokens than the list is swept again, into bins of equal width in code.
//
// Bound by instruction issue (58 %), the histogram's bank conflicts (3.6 wavefronts per addition) and the barriers between
// a row's serial steps.  A row of 32,000 bf16 entries takes 37,400 warp instructions; it took 67,000 before the sweep went
// without returned atomics and with packed arithmetic, and before the search behind it was left to one warp: 43,600, 1344 rows
// 146 -> 104 us.  Three blocks per SM for rows of up to 64,000 bytes, and 1024 threads for rows of which only one fits on an
// SM (32 rows of 32,000 fp32 with both cuts 47 -> 23 us).
// Since then, with lists in registers, a thread's words tested before its tokens, top-k from the threads' largest values and an output that compares once a word:
// 1500 rows of 32,000 bf16, top-p 0.95, 107 -> 90 us, the 1344 98 -> 84, the 32 rows 22 -> 14.7.
#pragma once
#include "rsd_device.cuh"
#include "rsd_scan.cuh"   // ex2_approx, packed arithmetic

namespace rsd {

constexpr int kBins = 1024;                      // bins of a sweep over the row
constexpr int kListCap = 1024;                   // tokens gathered into a list
constexpr int kNarrow = 32;                      // sub-intervals per turn of the list's search
constexpr float kValueRange = 24.0f;             // value-linear bins cover this many nats of value / T below the row's top

struct FilterArgs {
    const void* data;
    void* out;                                   // [B][R][V], the rows' element type
    int64_t seq_stride, row_stride;              // elements
    int R, V;
    int top_k;                                   // 0: none
    float top_p;                                 // >= 1: none
    float log2e_over_t;                          // log2(e) / temperature
    int32_t* kept;                               // [B][R] or null
    int32_t* status;                             // [B], OR-ed into, or (one row a sequence) written
};

struct FilterSmem {
    union {
        struct {
            uint32_t lo[kBins];                  // the sweep's histogram: low halves of the weights (or counts),
            uint32_t hi[kBins];                  // high halves
        } hist;
        struct {
            uint32_t lo[kNarrow], hi[kNarrow], count[kNarrow];   // the same for a turn of the list's search
            uint32_t tie[kListCap];              // tokens equal to the value found
        } fine;
    };
    uint32_t list[kListCap];                     // indices of the tokens still in play, in no particular order
    unsigned long long scan_w[32];
    unsigned long long pick_above;               // tally above the picked bin
    unsigned long long row_bar;                  // mbarrier of the row's bulk copy
    double above;                                // what the list's search found: the mass or number of the tokens strictly above
    uint32_t cut_code;                           // the last kept value, its code and
    int cut_tok;                                 // the last kept token among its equals
    uint32_t top, ext_lo, ext_hi;                // codes of the row's largest value, of a bin's smallest and largest
    float low;                                   // the smallest finite value in a sample of the row
    int pick_bin, n_list, n_all, not_finite, n_kept;
    int copy_gave_up, needs_cleaning, nan_flag;
    int scan_i[32];
};

// ordered code of a value's bit pattern: larger value <=> larger code, equal values <=> equal codes; NaN counts as -inf.
// 2-byte rows: the 16-bit pattern (all that distinguishes two bf16 values); 4-byte rows: all 32 bits.
template <typename T>
struct RowCodes;
template <>
struct RowCodes<__nv_bfloat16> {
    static constexpr int kBits = 16;
    static constexpr int kPerVec = 8;                                               // values in 16 bytes
    __device__ static __forceinline__ uint32_t code_of_bits(uint32_t h) {       // h: the 16-bit pattern
        if ((h & 0x7FFFu) > 0x7F80u) h = 0xFF80u;                                  // NaN -> -inf
        if (h == 0x8000u) h = 0u;                                                  // -0 and +0 are one value
        return (h & 0x8000u) ? (~h & 0xFFFFu) : (h | 0x8000u);
    }
    __device__ static __forceinline__ uint32_t bits(const unsigned char* row, int i) { return ((const uint16_t*)row)[i]; }
    __device__ static __forceinline__ uint32_t code(const unsigned char* row, int i) { return code_of_bits(bits(row, i)); }
    __device__ static __forceinline__ float value_of_bits(uint32_t h) { return __uint_as_float(h << 16); }
    __device__ static __forceinline__ float value_of_code(uint32_t c) {
        const uint32_t h = (c & 0x8000u) ? (c & 0x7FFFu) : (~c & 0xFFFFu);
        return __uint_as_float(h << 16);
    }
    __device__ static __forceinline__ bool bits_nan(uint32_t h) { return (h & 0x7FFFu) > 0x7F80u; }
    __device__ static __forceinline__ uint32_t code_of_float(float v) { return code_of_bits(__float_as_uint(v) >> 16); }   // (truncated)
    // the 16-bit patterns of the 8 values of a 16-byte word
    __device__ static __forceinline__ void unpack_bits(const uint4& w, uint32_t (&h)[8]) {
        const uint32_t q[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) { h[2 * j] = q[j] & 0xFFFFu; h[2 * j + 1] = q[j] >> 16; }
    }
    __device__ static __forceinline__ uint4 pack_bits(const uint32_t (&h)[8]) {
        return make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
    }
    static constexpr uint32_t kNegInfCode = 0x007Fu;                               // code of -inf (0xFF80)
    static constexpr uint32_t kNegInfBits = 0xFF80u;
};
template <>
struct RowCodes<float> {
    static constexpr int kBits = 32;
    static constexpr int kPerVec = 4;
    __device__ static __forceinline__ uint32_t code_of_bits(uint32_t u) {
        if ((u & 0x7FFFFFFFu) > 0x7F800000u) u = 0xFF800000u;
        if (u == 0x80000000u) u = 0u;                                              // -0 and +0 are one value
        return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    }
    __device__ static __forceinline__ uint32_t bits(const unsigned char* row, int i) { return ((const uint32_t*)row)[i]; }
    __device__ static __forceinline__ uint32_t code(const unsigned char* row, int i) { return code_of_bits(bits(row, i)); }
    __device__ static __forceinline__ float value_of_bits(uint32_t u) { return __uint_as_float(u); }
    __device__ static __forceinline__ float value_of_code(uint32_t c) {
        return __uint_as_float((c & 0x80000000u) ? (c & 0x7FFFFFFFu) : ~c);
    }
    __device__ static __forceinline__ bool bits_nan(uint32_t u) { return (u & 0x7FFFFFFFu) > 0x7F800000u; }
    __device__ static __forceinline__ uint32_t code_of_float(float v) { return code_of_bits(__float_as_uint(v)); }
    __device__ static __forceinline__ void unpack_bits(const uint4& w, uint32_t (&h)[4]) { h[0] = w.x; h[1] = w.y; h[2] = w.z; h[3] = w.w; }
    __device__ static __forceinline__ uint4 pack_bits(const uint32_t (&h)[4]) { return make_uint4(h[0], h[1], h[2], h[3]); }
    static constexpr uint32_t kNegInfCode = 0x007FFFFFu;
    static constexpr uint32_t kNegInfBits = 0xFF800000u;
};

// Largest value of a 16-byte word of the row (NaN ignored); `odd` is set when the word holds a NaN or a -inf.
template <typename T>
struct RowStats;
template <>
struct RowStats<__nv_bfloat16> {
    __device__ static __forceinline__ float largest(const uint4& w, bool& odd) {
        const uint32_t q[4] = {w.x, w.y, w.z, w.w};
        uint32_t m = 0xFF80FF80u, bad = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t le;
            asm("max.bf16x2 %0, %0, %1;" : "+r"(m) : "r"(q[j]));
            asm("set.leu.u32.bf16x2 %0, %1, %2;" : "=r"(le) : "r"(q[j]), "r"(0xFF80FF80u));   // <= -inf, or NaN
            bad |= le;
        }
        if (bad) odd = true;
        return fmaxf(__uint_as_float(m << 16), __uint_as_float(m & 0xFFFF0000u));
    }
};
template <>
struct RowStats<float> {
    __device__ static __forceinline__ float largest(const uint4& w, bool& odd) {
        const float v[4] = {__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w)};
        float m = kNegInf;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            m = fmaxf(m, v[j]);
            if (!(v[j] > kNegInf)) odd = true;
        }
        return m;
    }
};

// Tests on a whole 16-byte word of the row.  They compare values; as values and as codes +0 and -0 are one.  between() is a superset (2-byte
// rows: bounds cut to 16 bits) that gather() checks by code.  at_least() is final: outside the cut's word the output and the number of the kept are
// what it says, so its bound is a value of the rows' type, and a bound of NaN (the code behind +inf) keeps nothing.
template <typename T>
struct RowVec;
template <>
struct RowVec<__nv_bfloat16> {
    __device__ static __forceinline__ uint32_t twice(float v) { return (__float_as_uint(v) >> 16) * 0x00010001u; }
    // bit j set when first <= entry j <= last
    __device__ static __forceinline__ uint32_t between(const uint4& w, float first, float last) {
        const uint32_t q[4] = {w.x, w.y, w.z, w.w}, f2 = twice(first), l2 = twice(last);
        uint32_t acc = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t ge, le;
            asm("set.ge.u32.bf16x2 %0, %1, %2;" : "=r"(ge) : "r"(q[j]), "r"(f2));
            asm("set.le.u32.bf16x2 %0, %1, %2;" : "=r"(le) : "r"(q[j]), "r"(l2));
            acc |= ge & le & ((1u << (2 * j)) | (1u << (2 * j + 17)));
        }
        return (acc | (acc >> 16)) & 0xFFu;
    }
    // the word with -inf at the entries below `cut`; `kept`: the number of the others
    __device__ static __forceinline__ uint4 at_least(const uint4& w, float cut, int& kept) {
        const uint32_t q[4] = {w.x, w.y, w.z, w.w}, c2 = twice(cut);
        uint32_t o[4], acc = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t ge;
            asm("set.ge.u32.bf16x2 %0, %1, %2;" : "=r"(ge) : "r"(q[j]), "r"(c2));
            o[j] = (q[j] & ge) | (0xFF80FF80u & ~ge);
            acc |= ge & ((1u << (2 * j)) | (1u << (2 * j + 17)));
        }
        kept = __popc(acc);
        return make_uint4(o[0], o[1], o[2], o[3]);
    }
};
template <>
struct RowVec<float> {
    __device__ static __forceinline__ uint32_t between(const uint4& w, float first, float last) {
        const float v[4] = {__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w)};
        uint32_t acc = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) acc |= (v[j] >= first && v[j] <= last) ? 1u << j : 0u;
        return acc;
    }
    __device__ static __forceinline__ uint4 at_least(const uint4& w, float cut, int& kept) {
        const uint32_t q[4] = {w.x, w.y, w.z, w.w};
        uint32_t o[4];
        kept = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool ge = __uint_as_float(q[j]) >= cut;
            o[j] = ge ? q[j] : 0xFF800000u;
            kept += ge ? 1 : 0;
        }
        return make_uint4(o[0], o[1], o[2], o[3]);
    }
};

// A cut in the order (value descending, token ascending): a token is at or before the cut iff its code is larger,
// or equal with a token index not beyond `tok`.
struct Cut {
    uint32_t code;
    int tok;
};
__device__ __forceinline__ bool within(const Cut& c, uint32_t code, int i) { return code > c.code || (code == c.code && i <= c.tok); }

// inclusive prefix sum of a 64-bit word over the block; `total` = the sum over all threads
template <int NT>
__device__ __forceinline__ unsigned long long block_scan_u64(unsigned long long v, unsigned long long* scratch, unsigned long long& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long up = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += up;
    }
    if (lane == 31) scratch[warp] = v;
    __syncthreads();
    // every warp adds up the warps' sums by itself
    const unsigned long long mine = lane < NT / 32 ? scratch[lane] : 0ull;
    unsigned long long s = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long up = __shfl_up_sync(0xFFFFFFFFu, s, o);
        if (lane >= o) s += up;
    }
    total = __shfl_sync(0xFFFFFFFFu, s, 31);
    return v + __shfl_sync(0xFFFFFFFFu, s - mine, warp);
}

// Bins over an interval of codes [lo, hi], bin 0 at the top: of equal width in value (values further than the range below
// hi fall into the last bin), or, where `shift` >= 0, of 2^shift codes each.
struct BinMap {
    float scale, offset;     // bin = round(offset - value * scale), at most kBins - 1
    uint32_t lo, hi;
    int shift;
    __device__ __forceinline__ static int of_position(float d) {   // round to nearest, in the low mantissa bits
        return (int)(__float_as_uint(fminf(d, (float)(kBins - 1)) + 12582912.0f) & (uint32_t)(kBins - 1));
    }
    __device__ __forceinline__ int of(float v, uint32_t code) const {
        return shift >= 0 ? (int)((hi - code) >> shift) : of_position(fmaf(v, -scale, offset));
    }
};

template <typename T, int NT>
struct RowFilter {
    FilterSmem& sm;
    const unsigned char* row;   // shared memory, NaN already turned into -inf
    int V;
    float k, neg_c;             // weight of a value: 2^(value * k + neg_c)
    bool all_finite;            // nothing in the row is -inf
    int frac_bits, split;       // fixed point of the sweep's weights; bits of a low half

    using Codes = RowCodes<T>;
    static constexpr int kPerVec = Codes::kPerVec;

    __device__ __forceinline__ float weight_of_value(float v) const { return ex2_approx(fmaf(v, k, neg_c)); }
    __device__ __forceinline__ float weight(uint32_t code) const { return weight_of_value(Codes::value_of_code(code)); }
    __device__ __forceinline__ float to_fixed() const { return __uint_as_float((uint32_t)(127 + frac_bits) << 23); }
    __device__ __forceinline__ int words() const { return (V + kPerVec - 1) / kPerVec; }   // (the last one is padded with -inf)

    __device__ __forceinline__ void clear_histogram() {
        for (int q = threadIdx.x; q < kBins; q += NT) { sm.hist.lo[q] = 0u; sm.hist.hi[q] = 0u; }
    }

    // Every token of the row into the histogram (cleared), bins of equal width in value.  MASKED: the row holds entries of -inf, left out.
    template <bool BY_MASS, bool MASKED>
    __device__ __forceinline__ void sweep_all(const BinMap& bm) {
        const unsigned long long ns = f32x2(-bm.scale, -bm.scale), of = f32x2(bm.offset, bm.offset), magic = f32x2(12582912.0f, 12582912.0f),
                                 k2 = f32x2(k, k), c2 = f32x2(neg_c, neg_c), fx = f32x2(to_fixed(), to_fixed()), zero = f32x2(0.0f, 0.0f);
        const uint32_t low_mask = (1u << split) - 1u;
        auto two = [&](unsigned long long v) {
            float d0, d1;
            bool in0 = true, in1 = true;
            split_f32x2(fma_f32x2(v, ns, of), d0, d1);
            if (MASKED) { in0 = d0 < -kNegInf; in1 = d1 < -kNegInf; }   // (an entry of -inf lies infinitely far below the top)
            split_f32x2(add_f32x2(f32x2(fminf(d0, (float)(kBins - 1)), fminf(d1, (float)(kBins - 1))), magic), d0, d1);
            const int q0 = (int)(__float_as_uint(d0) & (uint32_t)(kBins - 1)), q1 = (int)(__float_as_uint(d1) & (uint32_t)(kBins - 1));
            if (BY_MASS) {
                float x0, x1;
                split_f32x2(fma_f32x2(v, k2, c2), x0, x1);
                split_f32x2(fma_f32x2(f32x2(ex2_approx(x0), ex2_approx(x1)), fx, zero), x0, x1);
                const uint32_t w0 = __float2uint_rn(x0), w1 = __float2uint_rn(x1);
                if (in0) {
                    atomicAdd(&sm.hist.lo[q0], w0 & low_mask);
                    atomicAdd(&sm.hist.hi[q0], w0 >> split);
                }
                if (in1) {
                    atomicAdd(&sm.hist.lo[q1], w1 & low_mask);
                    atomicAdd(&sm.hist.hi[q1], w1 >> split);
                }
            } else {
                if (in0) atomicAdd(&sm.hist.lo[q0], 1u);
                if (in1) atomicAdd(&sm.hist.lo[q1], 1u);
            }
        };
        const int n_vec = V / kPerVec;
        for (int m = threadIdx.x; m < n_vec; m += NT) {
            uint32_t h[kPerVec];
            Codes::unpack_bits(((const uint4*)row)[m], h);
#pragma unroll
            for (int j = 0; j < kPerVec; j += 2) two(f32x2(Codes::value_of_bits(h[j]), Codes::value_of_bits(h[j + 1])));
        }
        for (int i = n_vec * kPerVec + threadIdx.x; i < V; i += NT) {
            const float v = Codes::value_of_bits(Codes::bits(row, i));
            if (!MASKED || v > kNegInf) add_one<BY_MASS>(bm.of(v, 0u), v);
        }
    }
    template <bool BY_MASS>
    __device__ __forceinline__ void add_one(int q, float v) {
        if (BY_MASS) {
            const uint32_t w = __float2uint_rn(weight_of_value(v) * to_fixed());
            atomicAdd(&sm.hist.lo[q], w & ((1u << split) - 1u));
            atomicAdd(&sm.hist.hi[q], w >> split);
        } else {
            atomicAdd(&sm.hist.lo[q], 1u);
        }
    }
    // f(i, value, code) for the tokens within `inside` with a code in [bm.lo, bm.hi]
    template <typename F>
    __device__ __forceinline__ void for_tokens(const BinMap& bm, const Cut& inside, F f) const {
        for (int m = threadIdx.x; m < words(); m += NT) {
            uint32_t h[kPerVec];
            Codes::unpack_bits(((const uint4*)row)[m], h);
#pragma unroll
            for (int j = 0; j < kPerVec; ++j) {
                const uint32_t code = Codes::code_of_bits(h[j]);
                const int i = m * kPerVec + j;
                if (code >= bm.lo && code <= bm.hi && within(inside, code, i) && code > Codes::kNegInfCode) f(i, Codes::value_of_bits(h[j]), code);
            }
        }
    }

    // values that may lie in bin `pick`: its edges and a little more (2-byte rows compare against the bounds cut to 16 bits)
    __device__ __forceinline__ void bin_edges(const BinMap& bm, int pick, float& v_first, float& v_last) const {
        if (bm.shift >= 0) {
            const uint32_t hi = bm.hi - ((uint32_t)pick << bm.shift), w = (1u << bm.shift) - 1u;
            v_first = Codes::value_of_code(hi - bm.lo < w ? bm.lo : hi - w);
            v_last = Codes::value_of_code(hi);
        } else {
            const float slack = 0.5f + 1e-3f + 4e-7f * fabsf(bm.offset);
            v_last = pick == 0 ? -kNegInf : (bm.offset - ((float)pick - slack)) / bm.scale;
            v_first = pick == kBins - 1 ? kNegInf : (bm.offset - ((float)pick + slack)) / bm.scale;
            v_last += fabsf(v_last) * 0.0079f;
            v_first -= fabsf(v_first) * 0.0079f;
        }
    }
    // The tokens with a value in [v_first, v_last] that f(value, code) accepts (and that are within `inside`) into the list;
    // sm.n_list, cleared before, is their number, or more than the list holds.
    template <typename F>
    __device__ __forceinline__ void gather(float v_first, float v_last, uint32_t lo, uint32_t hi, const Cut& inside, F f) {
        // (Few words hold such a token, but a warp's 32 words mostly do: taken word by word, every word of a thread waited for the
        // longest of the warp's.  1344 rows of 32,000 bf16, top-p: 9.8 k cycles a row.)
        constexpr int kWords = 32 / kPerVec;             // their entries are the bits of one mask
        for (int m0 = threadIdx.x; m0 < words(); m0 += kWords * NT) {
            uint32_t in = 0u;
#pragma unroll
            for (int g = 0; g < kWords; ++g)
                if (m0 + g * NT < words()) in |= RowVec<T>::between(((const uint4*)row)[m0 + g * NT], v_first, v_last) << (g * kPerVec);
            while (in) {
                const int j = __ffs(in) - 1;
                in &= in - 1u;
                const int i = (m0 + (j / kPerVec) * NT) * kPerVec + j % kPerVec;
                const uint32_t h = Codes::bits(row, i), code = Codes::code_of_bits(h);
                if (code < lo || code > hi || code <= Codes::kNegInfCode || !within(inside, code, i) || !f(Codes::value_of_bits(h), code)) continue;
                const int at = atomicAdd(&sm.n_list, 1);
                if (at < kListCap) sm.list[at] = (uint32_t)i;
                else in = 0u;                            // (too many: one more addition tells)
            }
        }
        __syncthreads();
    }

    // The j-th (1-based, in token order) of the tokens with code `code` within `inside`: for runs of equal values that do not
    // fit the list.  Threads own consecutive runs; one prefix count over the block.
    __device__ __forceinline__ int nth_with_code(uint32_t code, int j, const Cut& inside) {
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        const int per = (V + NT - 1) / NT;
        const int m0 = min(V, tid * per), m1 = min(V, m0 + per);
        int mine = 0;
        for (int i = m0; i < m1; ++i) mine += (Codes::code(row, i) == code && within(inside, code, i)) ? 1 : 0;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += up;
        }
        __syncthreads();
        if (lane == 31) sm.scan_i[warp] = incl;
        if (tid == 0) sm.cut_tok = V;
        __syncthreads();
        int before = incl - mine;
        for (int w = 0; w < warp; ++w) before += sm.scan_i[w];
        if (mine > 0 && before < j && j <= before + mine) {
            int seen = before;
            for (int i = m0; i < m1; ++i)
                if (Codes::code(row, i) == code && within(inside, code, i) && ++seen == j) { sm.cut_tok = i; break; }
        }
        __syncthreads();
        return sm.cut_tok;
    }

    // how many of `ties` tokens of code t stay so that the tally reaches `need`
    template <bool BY_MASS>
    __device__ __forceinline__ int ties_to_keep(uint32_t t, int ties, double above, double need) const {
        if (!BY_MASS) return max(1, min(ties, (int)(need - above)));
        const double w = (double)weight(t);
        if (!(w > 0.0)) return ties;
        const double want = ceil((need - above) / w);
        int j = want < 1.0 ? 1 : (want > (double)ties ? ties : (int)want);
        while (j > 1 && above + (double)(j - 1) * w >= need) --j;
        while (j < ties && above + (double)j * w < need) ++j;
        return j;
    }

    // The cut within the list (n tokens), by one warp: the largest code t with F(t) >= need, F(t) = `above` plus the number
    // or weight of the list's tokens whose code is >= t, and the last kept token among its equals.
    // (HELD: up to kHeld tokens a lane, read once; a longer list costs two dependent reads of shared memory per token and turn.  A comparison
    // of each token with all others in place of the turns: 1500 rows of 32,000 bf16, top-p, 99 -> 152 us.)
    static constexpr int kHeld = 4;
    template <bool BY_MASS>
    __device__ __forceinline__ void finish(int n, double above, double need, const Cut& inside) {
        if (n <= 32 * kHeld) finish_list<BY_MASS, true>(n, above, need, inside);
        else finish_list<BY_MASS, false>(n, above, need, inside);
    }
    template <bool BY_MASS, bool HELD>
    __device__ __forceinline__ void finish_list(int n, double above, double need, const Cut& inside) {
        const int lane = threadIdx.x & 31;
        uint32_t lo = 0xFFFFFFFFu, hi = 0u;
        uint32_t held_x[HELD ? kHeld : 1], held_c[HELD ? kHeld : 1];
        if (HELD) {
#pragma unroll
            for (int e = 0; e < kHeld; ++e) held_x[HELD ? e : 0] = lane + 32 * e < n ? sm.list[lane + 32 * e] : 0u;
#pragma unroll
            for (int e = 0; e < kHeld; ++e) held_c[HELD ? e : 0] = Codes::code(row, (int)held_x[HELD ? e : 0]);
        }
        auto each = [&](auto f) {                          // f(code) for this lane's tokens
            if (HELD) {
#pragma unroll
                for (int e = 0; e < kHeld; ++e)
                    if (lane + 32 * e < n) f(held_c[HELD ? e : 0]);
            } else {
                for (int i = lane; i < n; i += 32) f(Codes::code(row, (int)sm.list[i]));
            }
        };
        each([&](uint32_t c) {
            lo = min(lo, c);
            hi = max(hi, c);
        });
        lo = __reduce_min_sync(0xFFFFFFFFu, lo);
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);
        // weights as 32-bit fixed point relative to the list's largest: exact unless they spread over more than a factor of 128
        const float w_top = weight(hi);
        const int e = max((int)((__float_as_uint(w_top) >> 23) & 255u), 1) - 127;
        const float up_a = __uint_as_float((uint32_t)(127 + (31 - e) / 2) << 23), up_b = __uint_as_float((uint32_t)(127 + (31 - e) - (31 - e) / 2) << 23);
        const double unit = 1.0 / ((double)up_a * (double)up_b);
        while (lo < hi) {
            const int shift = max(0, 32 - __clz(hi - lo) - 5);
            sm.fine.lo[lane] = 0u;
            sm.fine.hi[lane] = 0u;
            sm.fine.count[lane] = 0u;
            __syncwarp();
            each([&](uint32_t c) {
                if (c < lo || c > hi) return;
                const int q = (int)((hi - c) >> shift);
                atomicAdd(&sm.fine.count[q], 1u);
                if (BY_MASS) {
                    const uint32_t w = __float2uint_rn((weight(c) * up_a) * up_b);
                    atomicAdd(&sm.fine.lo[q], w & 0xFFFFu);
                    atomicAdd(&sm.fine.hi[q], w >> 16);
                }
            });
            __syncwarp();
            const uint32_t count = sm.fine.count[lane];
            unsigned long long sum = BY_MASS ? ((unsigned long long)sm.fine.hi[lane] << 16) + sm.fine.lo[lane] : (unsigned long long)count;
            __syncwarp();
            const unsigned long long mine = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long s = __shfl_up_sync(0xFFFFFFFFu, sum, o);
                if (lane >= o) sum += s;
            }
            const double per = BY_MASS ? unit : 1.0;
            const unsigned reached = __ballot_sync(0xFFFFFFFFu, count > 0u && above + (double)sum * per >= need), some = __ballot_sync(0xFFFFFFFFu, count > 0u);
            const int pick = reached ? __ffs(reached) - 1 : 31 - __clz(some);   // (rounding: the last one that holds anything)
            above += (double)__shfl_sync(0xFFFFFFFFu, sum - mine, pick) * per;
            const uint32_t new_hi = hi - ((uint32_t)pick << shift), width = (1u << shift) - 1u;
            lo = new_hi - lo < width ? lo : new_hi - width;
            hi = new_hi;
        }
        // the tokens equal to the value found, in no particular order
        int ties = 0;
        auto note = [&](bool eq, uint32_t x) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, eq);
            if (eq) sm.fine.tie[ties + __popc(m & ((1u << lane) - 1u))] = x;
            ties += __popc(m);
        };
        if (HELD) {
#pragma unroll
            for (int e = 0; e < kHeld; ++e) note(lane + 32 * e < n && held_c[HELD ? e : 0] == lo, held_x[HELD ? e : 0]);
        } else {
            for (int i0 = 0; i0 < n; i0 += 32) {
                const uint32_t x = i0 + lane < n ? sm.list[i0 + lane] : 0u;
                note(i0 + lane < n && Codes::code(row, (int)x) == lo, x);
            }
        }
        __syncwarp();
        const int j = ties_to_keep<BY_MASS>(lo, ties, above, need);
        int tok = lo == inside.code ? inside.tok : V;      // (all of them stay)
        if (j < ties) {
            if (ties <= 32) {
                const uint32_t x = lane < ties ? sm.fine.tie[lane] : 0xFFFFFFFFu;
                int rank = 0;
                for (int i = 0; i < ties; ++i) rank += __shfl_sync(0xFFFFFFFFu, x, i) < x ? 1 : 0;
                tok = (int)__shfl_sync(0xFFFFFFFFu, x, __ffs(__ballot_sync(0xFFFFFFFFu, lane < ties && rank == j - 1)) - 1);
            } else {                                       // smallest token with j ties up to it
                int a_ = 0, b_ = V - 1;
                while (a_ < b_) {
                    const int mid = (a_ + b_) >> 1;
                    int c = 0;
                    for (int i = lane; i < ties; i += 32) c += (int)sm.fine.tie[i] <= mid ? 1 : 0;
                    if (__reduce_add_sync(0xFFFFFFFFu, c) >= j) b_ = mid; else a_ = mid + 1;
                }
                tok = a_;
            }
        }
        if (lane == 0) { sm.cut_code = lo; sm.cut_tok = tok; }
    }

    // The reach of top_few()'s bins below the row's largest value, and whether the part of the slack in bin_edges() that follows the value
    // itself is at most a twelfth of it.
    __device__ __forceinline__ float few_width(float v_hi) const { return fminf(kValueRange * kLog2e / k, sm.low < v_hi ? 1.25f * (v_hi - sm.low) : 3.0e38f); }
    __device__ __forceinline__ bool slack_is_small(uint32_t top) const {
        const float v_hi = Codes::value_of_code(top);
        return fabsf(v_hi) * (0.0079f * 12.0f) <= few_width(v_hi);
    }

    // Top-k for few tokens, and top-p among them (top_p < 1), without a histogram of the row: the threads' largest values (of distinct tokens)
    // go into the bins, the n-th largest of them bounds the n-th largest token from below, and what reaches it fits the list
    // (n = 50 of 1024 threads: about 55 tokens).  false: it does not; nothing is decided.  The histogram is clear; mine_top: this thread's largest value.
    __device__ __forceinline__ bool top_few(uint32_t top, float mine_top, int n_wanted, float top_p, Cut& cut) {
        const int tid = threadIdx.x, lane = tid & 31;
        const Cut all = {Codes::kNegInfCode, V};
        BinMap bm;
        bm.shift = -1;
        bm.lo = Codes::kNegInfCode + 1u;
        bm.hi = top;
        const float v_hi = Codes::value_of_code(top), width = few_width(v_hi);
        bm.scale = (float)(kBins - 1) / width;
        bm.offset = v_hi * bm.scale;
        if (!(width > 0.0f) || !(width < 3.0e38f) || !(fabsf(bm.offset) < 1.0e6f)) return false;
        if (mine_top > kNegInf) atomicAdd(&sm.hist.lo[bm.of(mine_top, 0u)], 1u);
        if (tid == 0) { sm.pick_bin = -1; sm.n_list = 0; }
        __syncthreads();
        unsigned long long mine, incl, seen;
        prefix(mine, incl, seen);
        pick_bin((double)n_wanted, 0.0, 1.0, mine, incl);
        if (sm.pick_bin < 0) return false;
        float v_first, v_last;
        bin_edges(bm, sm.pick_bin, v_first, v_last);
        gather(v_first, -kNegInf, bm.lo, bm.hi, all, [](float, uint32_t) { return true; });
        const int n = sm.n_list;
        if (n < n_wanted || n > kListCap) return false;
        if (tid < 32) {
            finish<false>(n, 0.0, (double)n_wanted, all);
            __syncwarp();
            if (top_p < 1.0f) {                                                  // (the kept tokens' total in the sweep's fixed point)
                const Cut inside = {sm.cut_code, sm.cut_tok};
                unsigned long long total = 0;
                int kept = 0;
                for (int i0 = 0; i0 < n; i0 += 32) {
                    const uint32_t x = i0 + lane < n ? sm.list[i0 + lane] : 0u;
                    const uint32_t code = Codes::code(row, (int)x);
                    const bool in = i0 + lane < n && within(inside, code, (int)x);
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
                    if (in) {
                        sm.list[kept + __popc(m & ((1u << lane) - 1u))] = x;
                        total += __float2uint_rn(weight(code) * to_fixed());
                    }
                    kept += __popc(m);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, o);
                __syncwarp();
                finish<true>(kept, 0.0, (double)top_p * ((double)total / (double)(1ull << frac_bits)), inside);
            }
        }
        __syncthreads();
        cut = {sm.cut_code, sm.cut_tok};
        return true;
    }

    // Sums of this thread's bins and of all bins up to them, from the top bin down.
    static constexpr int kOwnBins = kBins / NT;
    __device__ __forceinline__ unsigned long long bin_sum(int q) const { return ((unsigned long long)sm.hist.hi[q] << split) + sm.hist.lo[q]; }
    __device__ __forceinline__ void prefix(unsigned long long& mine, unsigned long long& incl, unsigned long long& total) {
        mine = 0;
#pragma unroll
        for (int e = 0; e < kOwnBins; ++e) mine += bin_sum((int)threadIdx.x * kOwnBins + e);
        incl = block_scan_u64<NT>(mine, sm.scan_w, total);
    }
    // The bin that brings the tally to `need` (sm.pick_bin, -1 before) and what lies above it; ends with a barrier.
    __device__ __forceinline__ void pick_bin(double need, double above, double unit, unsigned long long mine, unsigned long long incl) {
        unsigned long long run = incl - mine;   // everything above this thread's bins
        auto tally = [&](unsigned long long w) { return above + (double)w * unit; };
        if (tally(run) < need && tally(incl) >= need) {
#pragma unroll
            for (int e = 0; e < kOwnBins; ++e) {
                const int q = (int)threadIdx.x * kOwnBins + e;
                const unsigned long long w = bin_sum(q);
                if (tally(run) < need && tally(run + w) >= need) { sm.pick_bin = q; sm.pick_above = run; }
                run += w;
            }
        }
        __syncthreads();
    }

    // The cut at which the number (BY_MASS = false) or the weight of the tokens within `inside` reaches need_abs, or, when that
    // is negative, need_frac of their total weight.  Nothing within `inside` lies above code `top`.  The histogram is clear.
    template <bool BY_MASS>
    __device__ __forceinline__ Cut search(uint32_t bottom, uint32_t top, double need_abs, double need_frac, const Cut& inside, bool everything) {
        const int tid = threadIdx.x;
        double need = need_abs, above = 0.0;
        BinMap bm;
        bm.lo = bottom;
        bm.hi = top;
        for (int level = 0;; ++level) {
            // bins of equal width in value first; in code where the interval is narrow or infinite, and on every further level
            bm.shift = -1;
            const float v_hi = Codes::value_of_code(bm.hi);
            float v_lo = fmaxf(Codes::value_of_code(bm.lo), v_hi - kValueRange * kLog2e / k);
            if (sm.low < v_hi) v_lo = fmaxf(v_lo, v_hi - 1.25f * (v_hi - sm.low));   // (what lies further down falls into the last bin)
            const float width = v_hi - v_lo;
            bm.scale = (float)(kBins - 1) / width;
            bm.offset = v_hi * bm.scale;
            if (level > 0 || bm.hi - bm.lo < (uint32_t)kBins || !(width > 0.0f) || !(width < 3.0e38f) || !(fabsf(bm.offset) < 1.0e6f))   // (rows far from 0: the position's rounding must stay below half a bin)
                bm.shift = max(0, 32 - __clz(bm.hi - bm.lo) - 10);   // ((hi - lo) >> shift) < 1024
            if (bm.shift < 0 && everything && all_finite) sweep_all<BY_MASS, false>(bm);
            else if (bm.shift < 0 && everything) sweep_all<BY_MASS, true>(bm);
            else for_tokens(bm, inside, [&](int, float v, uint32_t code) { add_one<BY_MASS>(bm.of(v, code), v); });
            __syncthreads();
            // ---- tally from the top bin down -------------------------------------------------------------------------------
            unsigned long long mine, incl, total;
            prefix(mine, incl, total);
            const double unit = BY_MASS ? 1.0 / (double)(1ull << frac_bits) : 1.0;
            if (level == 0 && need_abs < 0.0) need = need_frac * ((double)total * unit);
            if (tid == 0) { sm.pick_bin = -1; sm.pick_above = 0ull; sm.n_list = 0; }
            __syncthreads();
            pick_bin(need, above, unit, mine, incl);
            // The tallies are exact sums of integers, and bins of a further level share out the picked bin's, so `need` is
            // reached; a bin is missing only where nothing in the row has a weight (`need` and all tallies 0): then the first.
            const int pick = max(sm.pick_bin, 0);
            above += (double)sm.pick_above * unit;
            float v_first, v_last;
            bin_edges(bm, pick, v_first, v_last);
            gather(v_first, v_last, bm.lo, bm.hi, inside, [&](float v, uint32_t code) { return bm.of(v, code) == pick; });   // (ends with a barrier)
            const int n = sm.n_list;
            if (n > 0 && n <= kListCap) {
                if (tid < 32) finish<BY_MASS>(n, above, need, inside);
                __syncthreads();
                return {sm.cut_code, sm.cut_tok};
            }
            // ---- more tokens than the list holds: the codes the bin spans, then once more over these ------------------------
            if (tid == 0) { sm.ext_lo = 0xFFFFFFFFu; sm.ext_hi = 0u; sm.n_all = 0; }
            __syncthreads();
            uint32_t c_lo = 0xFFFFFFFFu, c_hi = 0u;
            int members = 0;
            for_tokens(bm, inside, [&](int, float v, uint32_t code) {
                if (bm.of(v, code) == pick) { c_lo = min(c_lo, code); c_hi = max(c_hi, code); ++members; }
            });
            c_lo = __reduce_min_sync(0xFFFFFFFFu, c_lo);
            c_hi = __reduce_max_sync(0xFFFFFFFFu, c_hi);
            members = __reduce_add_sync(0xFFFFFFFFu, members);
            if ((tid & 31) == 0) { atomicMin(&sm.ext_lo, c_lo); atomicMax(&sm.ext_hi, c_hi); atomicAdd(&sm.n_all, members); }
            clear_histogram();
            __syncthreads();
            bm.lo = sm.ext_lo;
            bm.hi = sm.ext_hi;
            if (bm.lo >= bm.hi) {                        // a run of equal values
                return {bm.hi, nth_with_code(bm.hi, ties_to_keep<BY_MASS>(bm.hi, sm.n_all, above, need), inside)};
            }
        }
    }
};

template <typename T, int NT>
__global__ void __launch_bounds__(NT, NT == 512 ? 3 : 1) filter_rows_kernel(const FilterArgs a) {
    extern __shared__ __align__(16) unsigned char row_sm[];   // the row, padded with -inf to whole 16-byte words
    __shared__ FilterSmem sm;
    constexpr int kElem = (int)sizeof(T);
    constexpr int kPerVec = RowCodes<T>::kPerVec;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x / a.R, r = blockIdx.x % a.R, V = a.V;
    const unsigned char* src = (const unsigned char*)a.data + ((int64_t)b * a.seq_stride + (int64_t)r * a.row_stride) * kElem;
    unsigned char* dst = (unsigned char*)a.out + ((int64_t)b * a.R + r) * (int64_t)V * kElem;
    const int n_vec = V / kPerVec;                               // whole 16-byte words of the row
    const int n_all = (V + kPerVec - 1) / kPerVec;               // with the padded word

    const bool only_row = a.R == 1;                              // (its status is stored; no kernel ahead clears it)
    if (only_row) grid_wait();
    auto report = [&](int bits) {
        if (only_row) {
            a.status[b] = bits;
        } else {
            grid_wait();                                         // (status[] has been cleared)
            if (bits) atomicOr(&a.status[b], bits);
        }
    };
    // ---- the row into shared memory, NaN as -inf; its largest value and the number of finite entries ------------------
    // Rows that start on a 16-byte boundary come in by one bulk copy of the whole words, the others by plain loads.  A
    // first look takes the largest value and notes whether anything is NaN or -inf; only then is the row gone over
    // entry by entry to replace and count them.
    const bool bulk = ((uintptr_t)src & 15u) == 0 && n_vec > 0;
    if (tid == 0) {
        sm.nan_flag = 0;
        sm.copy_gave_up = 0;
        sm.needs_cleaning = 0;
        sm.not_finite = 0;
        sm.n_kept = 0;
        sm.top = RowCodes<T>::kNegInfCode;
        if (bulk) {
            mbar_init(&sm.row_bar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            // (an mbarrier counts at most 2^20 - 1 bytes per phase, a row has fewer)
            mbar_expect_tx(&sm.row_bar, (uint32_t)n_vec * 16u);
            bulk_load(row_sm, src, (uint32_t)n_vec * 16u, &sm.row_bar);
        }
    }
    for (int q = tid; q < kBins; q += NT) { sm.hist.lo[q] = 0u; sm.hist.hi[q] = 0u; }
    if (!bulk) {
        const uint32_t m = (uint32_t)(uintptr_t)src & 15u;
        if (m != 0 && n_vec > 2 && m % kElem == 0) {             // in the aligned words around each, shifted; the ends one by one
            for (int i = 1 + tid; i < n_vec - 1; i += NT) {
                const uint4* p = (const uint4*)(src + (size_t)i * 16 - m);
                ((uint4*)row_sm)[i] = window16(ld_shared_word(p), ld_shared_word(p + 1), m);
            }
        }
        const bool ends = m != 0 && n_vec > 2 && m % kElem == 0;
        for (int i = tid; i < (ends ? 2 * kPerVec : n_vec * kPerVec); i += NT) {
            const int x = ends && i >= kPerVec ? (n_vec - 2) * kPerVec + i : i;
            if (kElem == 2) ((uint16_t*)row_sm)[x] = (uint16_t)RowCodes<T>::bits(src, x);
            else ((uint32_t*)row_sm)[x] = RowCodes<T>::bits(src, x);
        }
    }
    if (tid < kPerVec && n_vec * kPerVec < V) {                  // the last, partial word, padded with -inf
        const int i = n_vec * kPerVec + tid;
        const uint32_t h = i < V ? RowCodes<T>::bits(src, i) : RowCodes<T>::kNegInfBits;
        if (kElem == 2) ((uint16_t*)row_sm)[i] = (uint16_t)h;
        else ((uint32_t*)row_sm)[i] = h;
    }
    __syncthreads();
    if (bulk && warp == 0) wait_bar(&sm.row_bar, 0, &sm.copy_gave_up);   // one warp polls, the others sleep at the barrier
    __syncthreads();
    if (bulk && warp != 0 && !sm.copy_gave_up) wait_bar(&sm.row_bar, 0, &sm.copy_gave_up);   // (done: every thread has now seen the copy's completion itself)
    float vtop = kNegInf;                                        // this thread's largest value
    {
        bool odd = false;                                        // something is NaN or -inf
        for (int m = tid; m < n_vec; m += NT) vtop = fmaxf(vtop, RowStats<T>::largest(((const uint4*)row_sm)[m], odd));
        for (int i = n_vec * kPerVec + tid; i < V; i += NT) {
            const float v = RowCodes<T>::value_of_bits(RowCodes<T>::bits(row_sm, i));
            vtop = fmaxf(vtop, v);
            odd |= !(v > kNegInf);
        }
        if (odd) sm.needs_cleaning = 1;
        // The last warp, which may have a word less than the others, looks at 32 words spread over the row for how far down its
        // values reach: the bins of the first sweep go about as far.  (A flat row would fall into a few of them: 200 rows of 32,000
        // bf16 within 0.1 of each other, 81 -> 28 us.  All warps looking at a word each cost every row 0.4 us, this one 0.2.)
        if (warp == NT / 32 - 1) {
            float low = -kNegInf;
            if (n_vec > 0) {
                uint32_t h[kPerVec];
                RowCodes<T>::unpack_bits(((const uint4*)row_sm)[(int)((unsigned)lane * (unsigned)n_vec / 32u)], h);
#pragma unroll
                for (int j = 0; j < kPerVec; ++j) {
                    const float v = RowCodes<T>::value_of_bits(h[j]);
                    if (v > kNegInf) low = fminf(low, v);
                }
            }
            const uint32_t lowest = __reduce_min_sync(0xFFFFFFFFu, float_to_ordered(low));
            if (lane == 0) sm.low = ordered_to_float(lowest);
        }
        // (a largest value of -0 has the code of +0)
        uint32_t top = vtop == 0.0f ? RowCodes<T>::code_of_float(0.0f) : (vtop > kNegInf ? RowCodes<T>::code_of_float(vtop) : RowCodes<T>::kNegInfCode);
        top = __reduce_max_sync(0xFFFFFFFFu, top);
        if (lane == 0) atomicMax(&sm.top, top);
    }
    __syncthreads();
    if (sm.copy_gave_up) {                                        // the copy never landed: report, write nothing
        if (tid == 0) report(32);                                 // RSD_ST_TIMEOUT
        return;
    }
    if (sm.needs_cleaning) {
        bool saw_nan = false;
        int not_finite = 0;
        for (int m = tid; m < n_all; m += NT) {
            uint32_t h[kPerVec];
            RowCodes<T>::unpack_bits(((const uint4*)row_sm)[m], h);
#pragma unroll
            for (int j = 0; j < kPerVec; ++j) {
                if (RowCodes<T>::bits_nan(h[j])) { saw_nan = true; h[j] = RowCodes<T>::kNegInfBits; }
                not_finite += (h[j] == RowCodes<T>::kNegInfBits && m * kPerVec + j < V) ? 1 : 0;
            }
            ((uint4*)row_sm)[m] = RowCodes<T>::pack_bits(h);
        }
        not_finite = __reduce_add_sync(0xFFFFFFFFu, not_finite);
        if (lane == 0 && not_finite) atomicAdd(&sm.not_finite, not_finite);
        if (saw_nan) sm.nan_flag = 1;
        __syncthreads();
    }
    const uint32_t top = sm.top;
    const int finite = V - sm.not_finite;

    const float vmax = RowCodes<T>::value_of_code(top);
    const bool plus_inf = vmax == -kNegInf;                       // a +inf entry: it alone carries the mass
    // Fixed point of the weights: 32 fraction bits up to 32,767 entries, 31 up to 65,535, 30 beyond (the conversion saturates
    // at 2^32 - 1, which only the row's largest value can reach); the halves are such that V of them fit 32 bits.  A weight is
    // off by at most half a unit, so the tally is within V 2^-(bits + 1) of the exact sum relative to the row's largest
    // weight: in the worst case V 2^-33, V 2^-32 and V 2^-31 in the three ranges (4e-6 for 32,000 entries, 5e-5 for the longest
    // rows; around 1e-8 in practice).
    const int frac_bits = V < 32768 ? 32 : V < 65536 ? 31 : 30;
    // The reference is rounded down, so that no exponent is above 0: in a row far from 0 the product is off by up to 1e-4, and a
    // largest weight that much above 1 would saturate while all others keep the factor.
    RowFilter<T, NT> f = {sm, row_sm, V, a.log2e_over_t, (finite > 0 && !plus_inf) ? __fmul_rd(-vmax, a.log2e_over_t) : 0.0f, sm.not_finite == 0, frac_bits,
                          V < 65536 ? 16 : 15};
    Cut cut = {RowCodes<T>::kNegInfCode, V};                      // everything finite
    int kept = finite;
    bool everything = true, count_kept = false;

    // ---- top-k: the value of the k-th largest entry, then the last kept token among its equals -------------------------
    const bool want_p = a.top_p > 0.0f && a.top_p < 1.0f && finite > 0 && !plus_inf;
    bool found_p = false;
    if (a.top_k > 0 && a.top_k < V && finite > a.top_k) {
        // (top_few() pays while what reaches the bound, a few more tokens than asked for, stays in the registers of finish(); 512 threads, rows of 8,192 to
        // 50,000 entries, 4-byte with top-k alone, 64 / 100 / 128 / 256 tokens: 0.87 / 0.92 / 1.08 / 1.38 of the time of a histogram of the row; with a nucleus behind
        // it 0.81 / 0.74 / 0.89 / 1.13; 2-byte top-k alone 0.82 / 0.88 / 0.94 / 1.06; 1024 threads, 160 / 256: 0.89 / 0.93, 4-byte 1.00 / 1.13, with a nucleus 0.94 / 0.97.  Rows of four words a
        // thread on: from 16,384 2-byte or 8192 4-byte entries, 32 rows of 8192 fp32, top-k 50 and top-p 0.9 14.6 -> 10.9 us.  And while the slack that bin_edges() gives the bound,
        // which follows the values' distance from 0, is small beside the bins' reach: 110 rows of 11,336 fp32 around 300 take 33.2 us where it is not heeded, 14.6 here.)
        const bool few = a.top_k <= (kElem == 2 || want_p ? NT / 4 : NT / 8) && n_vec >= 4 * NT && f.slack_is_small(top);
        if (few && f.top_few(top, vtop, a.top_k, want_p ? a.top_p : 1.0f, cut)) {
            found_p = want_p;
        } else {
            if (few) {
                __syncthreads();
                f.clear_histogram();
                __syncthreads();
            }
            cut = f.template search<false>(RowCodes<T>::kNegInfCode + 1u, top, (double)a.top_k, 0.0, cut, true);
        }
        kept = a.top_k;
        everything = false;
    }
    // ---- top-p: of what is left, the shortest prefix (value descending, token ascending) whose mass reaches top_p -------
    if (want_p) {
        if (found_p) {
            // (with the top-k)
        } else if (!everything && kept <= kListCap) {
            // the kept tokens all fit the list: one warp does the rest (their total in the sweep's fixed point)
            if (tid == 0) sm.n_list = 0;
            __syncthreads();
            f.gather(RowCodes<T>::value_of_code(cut.code), vmax, cut.code, top, cut, [](float, uint32_t) { return true; });
            if (tid < 32) {
                unsigned long long total = 0;
                const int n = sm.n_list;
                for (int i = lane; i < n; i += 32)
                    total += __float2uint_rn(f.weight(RowCodes<T>::code(row_sm, (int)sm.list[i])) * f.to_fixed());
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, o);
                f.template finish<true>(n, 0.0, (double)a.top_p * ((double)total / (double)(1ull << frac_bits)), cut);
            }
            __syncthreads();
            cut = {sm.cut_code, sm.cut_tok};
        } else {
            if (!everything) {
                __syncthreads();
                f.clear_histogram();
                __syncthreads();
            }
            cut = f.template search<true>(everything ? RowCodes<T>::kNegInfCode + 1u : cut.code, top, -1.0, (double)a.top_p, cut, everything);
        }
        count_kept = a.kept != nullptr;
    }

    grid_started();
    // ---- the row with -inf at the filtered entries ------------------------------------------------------------------------------
    {
        auto keeps = [&](int i, uint32_t h) {
            const uint32_t c = RowCodes<T>::code_of_bits(h);
            return c > RowCodes<T>::kNegInfCode && within(cut, c, i);
        };
        const bool dst16 = ((uintptr_t)dst & 15u) == 0;
        // Entries that equal the cut's value stay up to the cut's token: words ahead of its word keep what is at least the value, words
        // behind it what is at least the next larger one (as values +0 and -0 are one here, as they are one code).  In its word the tokens decide.
        const float cut_value = RowCodes<T>::value_of_code(cut.code), next_value = RowCodes<T>::value_of_code(cut.code + 1u);
        const int cut_word = cut.tok / kPerVec;
        int n_kept = 0;
        for (int m = tid; m < n_vec; m += NT) {
            const uint4 w = ((const uint4*)row_sm)[m];
            int n_here;
            uint4 o = RowVec<T>::at_least(w, m <= cut_word ? cut_value : next_value, n_here);
            if (m == cut_word) {
                uint32_t h[kPerVec];
                RowCodes<T>::unpack_bits(w, h);
                n_here = 0;
#pragma unroll
                for (int j = 0; j < kPerVec; ++j) {
                    if (keeps(m * kPerVec + j, h[j])) ++n_here;
                    else h[j] = RowCodes<T>::kNegInfBits;
                }
                o = RowCodes<T>::pack_bits(h);
            }
            n_kept += n_here;
            if (dst16) {
                ((uint4*)dst)[m] = o;
            } else {
                uint32_t h[kPerVec];
                RowCodes<T>::unpack_bits(o, h);
#pragma unroll
                for (int j = 0; j < kPerVec; ++j) {
                    if (kElem == 2) ((uint16_t*)dst)[m * kPerVec + j] = (uint16_t)h[j];
                    else ((uint32_t*)dst)[m * kPerVec + j] = h[j];
                }
            }
        }
        for (int i = n_vec * kPerVec + tid; i < V; i += NT) {
            const uint32_t h0 = RowCodes<T>::bits(row_sm, i);
            const bool stays = keeps(i, h0);
            const uint32_t h = stays ? h0 : RowCodes<T>::kNegInfBits;
            n_kept += stays ? 1 : 0;
            if (kElem == 2) ((uint16_t*)dst)[i] = (uint16_t)h;
            else ((uint32_t*)dst)[i] = h;
        }
        if (count_kept) {
            n_kept = __reduce_add_sync(0xFFFFFFFFu, n_kept);
            if (lane == 0) atomicAdd(&sm.n_kept, n_kept);
            __syncthreads();
            kept = sm.n_kept;
        }
    }
    if (tid == 0) {
        if (a.kept) a.kept[(int64_t)b * a.R + r] = kept;
        report(sm.nan_flag ? 1 : 0);                              // RSD_ST_NAN_INPUT
    }
}

}  // namespace rsd
