// Step 3: the extra token of a verification step: a draw from the normalised
// residual max(0, p - q') at the first rejection, with q'(.) of Eq. (2), or
// from p itself (the free token) when every proposal was accepted (notation
// paragraph of Section 3; Section 3.1, Eq. (2); Algorithm 1, rejection and
// free-token lines).
//
// Inverse-CDF sampling in target-id order over tiles of 256 ids (8 consecutive
// ids per lane of one warp, so a tile needs shuffles only, no block barrier).
// Values are carried unnormalised: e(t) = exp2((x_t - M)*scale) = p(t)*S and
// r'(t) = max(0, e(t) - q'(t)*S).
//   pass 1  every warp takes a run of tiles of row j = n_b; per tile one coalesced
//           128-bit load of the logits per lane, the drafter's probabilities of the ids
//           that have one, r' of its eight ids (with the two ids Eq. (2) singles out) and
//           a warp sum: the tile's value;
//   pass 2  the running sum over the tile values passes the target = u * total in one
//           tile, and one warp evaluates r'(t) of that single tile id by id and scans
//           inside it. Without residual mass the draw is from p_j (the tile values are
//           redone with e alone).
//
// Where pass 1 has the drafter's probabilities from (they lie in draft-id order):
//   same tokenizer on both sides: the row itself, two 128-bit loads per lane and tile, or id by id
//           where rows are not whole vectors (FROM_ROW; 256 rows of 32000 ids: step 44.2 -> 40.1 us);
//   else    shared memory, in target-id order (STAGED): a block gathers the mapped ids of
//           its tiles once, from a list in DRAFT-id order (od_sample_plan), so that the 32
//           lanes of a load sit within a few lines, and finds them in pass 1 by counting
//           mapped ids. Gathered tile by tile through the inverse map instead, every mapped
//           id costs a 32-byte sector and every id four bytes of the map, from L2: 834 MB
//           for 512 rows of 152064 ids, the rate of L2 (9.3 TB/s) for 75 us;
//   else    (more mapped ids in a part of the row than shared memory holds, and the
//           vocabulary shards) the inverse map and a gather (FROM_MAP), the map's entries
//           of the next pair of tiles requested before the gathers of the current one.
//
// A lane adds its eight values in fp32 and a tile's value is the fp32 warp sum of the
// lanes (fixed trees); sums and scans across tiles, and the scan inside the chosen
// tile, are fp64 in a fixed order: the result is reproducible, and the only difference
// to exact arithmetic is the fp32 rounding of the terms and of the tile sums.
//
// Vocabulary shards (the rows split by columns over several GPUs) use the same
// kernel in two further modes. A shard owns a window of whole tiles:
//   mode 1  pass 1 over the window, then the last block adds the window's tile
//           values: the shard's share of the residual mass (and, when that is
//           zero, of the mass of p_j, for the fallback);
//   mode 2  after the shares of all shards were exchanged: every shard forms the
//           same total and target = u * total, finds the shard in which the running
//           sum over shards crosses the target, and that shard alone scans its
//           window (offset by the shares before it) as in pass 2.
#include <float.h>

#include <vector>

#include "od_common.cuh"
#include "od_decide.cuh"

namespace {

constexpr int WARPS = OD_SAMPLE_THREADS / 32;
constexpr int EPT = OD_SAMPLE_TILE / 32;                  // ids per lane per tile (8)

// A 16-byte load of logits, which are read once: past L1, whose lines are better spent on the
// drafter's row, which the gathers come back to, and on the inverse map, which the blocks of
// other sequences on the same multiprocessor read too (od_sample_residual 14.7 -> 14.2 us on
// the batched workload; the inverse map past L1 as well: 15.5 us).
__device__ __forceinline__ uint4 ld_once(const void *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
struct SampleArgs {
    const void *logits;
    int64_t row_stride, seq_stride;
    int32_t B, K_max, v_p, v_q;
    int32_t ntiles, tiles_per_warp;
    const float *row_max, *row_sum, *q_rows;
    const int32_t *draft_ids, *tgt_ids;
    const float *q_prime;
    const int32_t *span_start, *span_len, *m;
    const uint8_t *tail_kind;
    const int32_t *n_accepted;
    const float *temperature;
    const uint64_t *seed;
    uint64_t step;
    const int32_t *vocab_map, *inv_map;
    // the context's lists for this launch's number of parts (od_sample_lists)
    const uint32_t *list_word, *octet;
    const int32_t *list_base, *list_part;
    int32_t part_tiles, slots;          // tiles of a part; room for staged probabilities
    int32_t same_ids;                   // 1: target id t is draft id t (t < v_q)
    int32_t row_vec;                    // 1: v_q is a multiple of 4 and the drafter's rows are 16-byte aligned
    int32_t map_serial;                 // of the map this launch was laid out for
    const int32_t *map_serial_now;
    int32_t *out_token;
    float *resid_mass;
    uint32_t *flags;
    double *tile_val;                   // [B][ntiles] sum over the tile of r'
    unsigned int *ticket;
    // vocabulary shards: this shard's tiles are [tile_lo, tile_hi); `logits` points at
    // its first column (target id col0), v_p is the id one past its last column
    int32_t tile_lo, tile_hi, col0;
    int32_t n_shards, shard_index;
    const double *mass_all;             // [n_shards][B][2] (residual share, share of p_j or 0)
    double *mass_out;                   // [B][2] this shard's shares
    int32_t early;                      // 1: the translation's outputs may be read before griddepcontrol.wait
    // od_step: no decide kernel ran; the decisions of step 2 are taken here, by every block of a
    // sequence alike, from the partials the streaming pass left, and the sequence's block 0
    // writes step 2's outputs (the w_ pointers; row_max, row_sum, n_accepted above are not read)
    StreamPlan plan;
    float *w_row_max, *w_row_sum, *w_p_sel, *w_ratio;
    int32_t *w_n_accepted, *w_n_draft;
    uint32_t *w_vflags;
};

// what one sequence's warps need to evaluate r(t)
struct SeqState {
    const char *row;
    const float *q_row;
    float c, S, scale;      // e(t) = exp2(fma(x_t, scale, -c)); S is the row sum relative to c
    bool residual;
    bool from_row;          // the drafter's probabilities are read at the target ids
    int32_t ngram_token, prefix_token;
    float ngram_prob, prefix_val;
};

// Values are carried UNNORMALISED: with c = fl(M*scale), e(t) = exp2(x_t*scale - c) and
// S = (row sum relative to M) * exp2(M*scale - c), so that p(t) = e(t)/S exactly as
// before but one fused multiply-add per id replaces a subtraction and a product,
//   residual   r'(t) = max(0, e(t) - q'(t)*S) = S * max(0, p(t) - q'(t))
//   free token r'(t) = e(t)
// so one multiplication by 1/S at the very end replaces one per element, and the
// inverse-CDF pick (target = u * sum r') is unchanged by the common factor.
__device__ __forceinline__ float resid_of(const SeqState &q, float x, float qq)
{
    return fmaxf(0.f, fmaf(-qq, q.S, od_ex2(fmaf(x, q.scale, -q.c))));
}

// Eq. (2): the two ids whose q' is not the drafter's row. Only the lane that owns such
// an id (its ids are t0 .. t0 + EPT - 1) redoes it: prefix sub-token first, the n-gram
// token last.
template <int DTYPE>
__device__ __forceinline__ void eq2_ids(const SeqState &q, const SampleArgs &a, int t0, float *r)
{
    const int dp = q.prefix_token - t0, dn = q.ngram_token - t0;
    if ((unsigned)dp < (unsigned)EPT && q.prefix_token < a.v_p) {
        const float v = resid_of(q, od_load_logit<DTYPE>(q.row, q.prefix_token), q.prefix_val);
#pragma unroll
        for (int e = 0; e < EPT; ++e) r[e] = e == dp ? v : r[e];
    }
    if ((unsigned)dn < (unsigned)EPT && q.ngram_token < a.v_p) {
        const float v = resid_of(q, od_load_logit<DTYPE>(q.row, q.ngram_token), q.ngram_prob);
#pragma unroll
        for (int e = 0; e < EPT; ++e) r[e] = e == dn ? v : r[e];
    }
}

// The drafter's probabilities of the EPT ids from t0 where target ids are draft ids: nothing looked up;
// ids >= v_q have none. Two 16-byte loads where the rows allow them (v_q a multiple of 4, so that no
// vector straddles the end), else id by id (256 sequences of 50257 ids, the step: staged, in one block of
// 201 KB per multiprocessor, 89.2 us; through the inverse map 56.8; so 51.4).
__device__ __forceinline__ void same_id_probs(const SeqState &q, const SampleArgs &a, int t0, float *qq)
{
    if (!a.row_vec) {
#pragma unroll
        for (int e = 0; e < EPT; ++e) qq[e] = t0 + e < a.v_q ? __ldg(q.q_row + t0 + e) : 0.f;
        return;
    }
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 v0 = t0 < a.v_q ? __ldg((const float4 *)(q.q_row + t0)) : z;
    const float4 v1 = t0 + 4 < a.v_q ? __ldg((const float4 *)(q.q_row + t0) + 1) : z;
    qq[0] = v0.x; qq[1] = v0.y; qq[2] = v0.z; qq[3] = v0.w;
    qq[4] = v1.x; qq[5] = v1.y; qq[6] = v1.z; qq[7] = v1.w;
}

// Where the drafter's probabilities of a tile come from: the inverse map and the row in global
// memory, the row alone (target ids are draft ids), or, for the tiles of this block's part, shared
// memory, in target-id order.
enum { FROM_MAP, FROM_ROW, STAGED, FREE };
struct StagedRow {
    const float *q;                     // [mapped ids of the part]
    const uint32_t *octet;
    uint32_t rank0;                     // the part's first rank
};
__device__ __forceinline__ void staged_probs(const StagedRow &sr, uint32_t oct, float *qq)
{
    uint32_t i = (oct >> 8) - sr.rank0;
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const uint32_t has = oct >> e & 1u;
        qq[e] = has ? sr.q[i] : 0.f;
        i += has;
    }
}

// r'(t) of the EPT consecutive ids this lane owns in `tile`; ids >= v_p give 0
template <int DTYPE>
__device__ __forceinline__ void tile_values(const SeqState &q, const SampleArgs &a, bool residual,
                                            int tile, int lane, float *r, const StagedRow *sr = nullptr)
{
    const int t0 = tile * OD_SAMPLE_TILE + lane * EPT;
    if (t0 + EPT <= a.v_p) {
        float x[EPT];
        if (DTYPE == OD_BF16) {
            const uint4 v = ld_once(q.row + (size_t)t0 * 2);
            x[0] = od_bf16_lo(v.x); x[1] = od_bf16_hi(v.x); x[2] = od_bf16_lo(v.y); x[3] = od_bf16_hi(v.y);
            x[4] = od_bf16_lo(v.z); x[5] = od_bf16_hi(v.z); x[6] = od_bf16_lo(v.w); x[7] = od_bf16_hi(v.w);
        } else {
            const float4 v0 = __ldg((const float4 *)(q.row + (size_t)t0 * 4));
            const float4 v1 = __ldg((const float4 *)(q.row + (size_t)t0 * 4) + 1);
            x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w;
            x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
        }
        if (residual) {
            float qq[EPT];
            if (q.from_row) {
                same_id_probs(q, a, t0, qq);
            } else if (sr) {
                staged_probs(*sr, __ldg(sr->octet + (t0 >> 3)), qq);
            } else {
                const int4 i0 = __ldg((const int4 *)(a.inv_map + t0));
                const int4 i1 = __ldg((const int4 *)(a.inv_map + t0) + 1);
                const int32_t d[EPT] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
#pragma unroll
                for (int e = 0; e < EPT; ++e) qq[e] = d[e] >= 0 ? __ldg(q.q_row + d[e]) : 0.f;
            }
#pragma unroll
            for (int e = 0; e < EPT; ++e) r[e] = resid_of(q, x[e], qq[e]);
        } else {
#pragma unroll
            for (int e = 0; e < EPT; ++e) r[e] = od_ex2(fmaf(x[e], q.scale, -q.c));
        }
    } else {
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int t = t0 + e;
            r[e] = 0.f;
            if (t < a.v_p) {
                const float xv = od_load_logit<DTYPE>(q.row, t);
                if (residual) {
                    const int32_t dv = __ldg(a.inv_map + t);
                    r[e] = resid_of(q, xv, dv >= 0 ? __ldg(q.q_row + dv) : 0.f);
                } else {
                    r[e] = od_ex2(fmaf(xv, q.scale, -q.c));
                }
            }
        }
    }
    if (residual) eq2_ids<DTYPE>(q, a, t0, r);
}

// inside the picked tile a lane's eight values are added in fp32 in index order (pass 1 adds a tile in
// pairs); everything across lanes and tiles is fp64
__device__ __forceinline__ double lane_sum(const float *r)
{
    float s = r[0];
#pragma unroll
    for (int e = 1; e < EPT; ++e) s += r[e];
    return (double)s;
}

// e(t) of the EPT consecutive ids this lane owns in `tile`; ids >= v_p give 0
template <int DTYPE>
__device__ __forceinline__ void tile_e_values(const SeqState &q, const SampleArgs &a, int tile, int lane, float *r)
{
    const int t0 = tile * OD_SAMPLE_TILE + lane * EPT;
    if (t0 + EPT <= a.v_p) {
        float x[EPT];
        if (DTYPE == OD_BF16) {
            const uint4 v = ld_once(q.row + (size_t)t0 * 2);
            x[0] = od_bf16_lo(v.x); x[1] = od_bf16_hi(v.x); x[2] = od_bf16_lo(v.y); x[3] = od_bf16_hi(v.y);
            x[4] = od_bf16_lo(v.z); x[5] = od_bf16_hi(v.z); x[6] = od_bf16_lo(v.w); x[7] = od_bf16_hi(v.w);
        } else {
            const float4 v0 = __ldg((const float4 *)(q.row + (size_t)t0 * 4));
            const float4 v1 = __ldg((const float4 *)(q.row + (size_t)t0 * 4) + 1);
            x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w;
            x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
        }
#pragma unroll
        for (int e = 0; e < EPT; ++e) r[e] = od_ex2(fmaf(x[e], q.scale, -q.c));
    } else {
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int t = t0 + e;
            r[e] = t < a.v_p ? od_ex2(fmaf(od_load_logit<DTYPE>(q.row, t), q.scale, -q.c)) : 0.f;
        }
    }
}

__device__ __forceinline__ float warp_sum_f32(float v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    return v;
}

// Where a warp's tile values go. one(): every lane holds the tile's value; pair(): lanes 0..15
// hold tile t's, lanes 16..31 tile t + 1's (if `two`).
struct GlobalTiles {                                        // [ntiles] of one sequence
    double *val;
    int lane;
    __device__ __forceinline__ void one(int t, float v) { if (lane == 0) val[t] = (double)v; }
    __device__ __forceinline__ void pair(int t, float v, bool two)
    {
        if ((lane & 15) == 0 && (lane == 0 || two)) val[t + (lane >> 4)] = (double)v;
    }
};
struct WarpTiles {                                          // the warp's own run in shared memory, and its sum
    float *val;
    int lane, t_lo;
    double total;                                           // lanes 0..15 and 16..31 each hold a share
    __device__ __forceinline__ void one(int t, float v)
    {
        v = fmaxf(0.f, v);                                  // (a tile with NaN has no mass)
        if (lane == 0) val[t - t_lo] = v;
        if (lane < 16) total += (double)v;
    }
    __device__ __forceinline__ void pair(int t, float v, bool two)
    {
        v = lane < 16 || two ? fmaxf(0.f, v) : 0.f;
        if ((lane & 15) == 0 && (lane == 0 || two)) val[t - t_lo + (lane >> 4)] = v;
        total += (double)v;
    }
    __device__ __forceinline__ double sum() const
    {
        return __shfl_sync(0xFFFFFFFFu, total, 0) + __shfl_sync(0xFFFFFFFFu, total, 16);
    }
};

// Pass 1, tile by tile (the free token, ragged last tiles, and the fallback of pass 2): every
// id of a tile looks up its draft id in the inverse map (coalesced) and gathers the drafter's
// probability if it has one; NT tiles are in flight per warp.
template <int DTYPE, int NT, typename Sink>
__device__ __forceinline__ void warp_tiles_dense(const SeqState &q, const SampleArgs &a, bool residual, int t_lo,
                                                 int t_hi, int lane, Sink &out)
{
    for (int t = t_lo; t < t_hi; t += NT) {
        float r[NT][EPT];
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            if (t + i < t_hi) {
                if (residual) tile_values<DTYPE>(q, a, true, t + i, lane, r[i]);
                else tile_e_values<DTYPE>(q, a, t + i, lane, r[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            if (t + i < t_hi) {
                float s = r[i][0];
#pragma unroll
                for (int e = 1; e < EPT; ++e) s += r[i][e];
                out.one(t + i, warp_sum_f32(s));
            }
        }
    }
}

// A lane's ids of one whole tile as they are stored, and the tile's residual from them
template <int DTYPE>
constexpr int RAW = DTYPE == OD_BF16 ? 1 : 2;               // 16-byte vectors of logits per lane and tile
template <int DTYPE>
__device__ __forceinline__ void load_tile(const SeqState &q, int tile, int lane, uint4 *raw)
{
    const uint4 *src = (const uint4 *)(q.row + (size_t)(tile * OD_SAMPLE_TILE + lane * EPT) * (DTYPE == OD_BF16 ? 2 : 4));
    raw[0] = ld_once(src);
    if (DTYPE != OD_BF16) raw[1] = ld_once(src + 1);
}
// A lane's eight ids of a whole tile: the sum of their residuals, or of e alone. A tile is 256
// ids of work for one warp, and its instructions bound a large batch: 276 a tile and 66.8 us for
// 296 staged rows of 152064 ids with a branch per id, 195 and 51.9 us with a select per id,
// 154 and 44.8 us so: an unmapped id's multiply-add is predicated off, and Eq. (2)'s two ids are
// looked for only in the tiles that hold them. (The clamp at zero as the multiply-add's own .sat is 0.8 % of
// the step faster, but clamps at one too, which e(M) may exceed by c's rounding; with the residuals as
// halves, to allow for that, it is no faster than the maximum.)
template <int DTYPE>
__device__ __forceinline__ void tile_e(const SeqState &q, const uint4 *raw, float *e)
{
    float x[EPT];
    if (DTYPE == OD_BF16) {
        const uint4 v = raw[0];
        x[0] = od_bf16_lo(v.x); x[1] = od_bf16_hi(v.x); x[2] = od_bf16_lo(v.y); x[3] = od_bf16_hi(v.y);
        x[4] = od_bf16_lo(v.z); x[5] = od_bf16_hi(v.z); x[6] = od_bf16_lo(v.w); x[7] = od_bf16_hi(v.w);
    } else {
        const uint4 v0 = raw[0], v1 = raw[DTYPE == OD_BF16 ? 0 : 1];
        x[0] = __uint_as_float(v0.x); x[1] = __uint_as_float(v0.y); x[2] = __uint_as_float(v0.z); x[3] = __uint_as_float(v0.w);
        x[4] = __uint_as_float(v1.x); x[5] = __uint_as_float(v1.y); x[6] = __uint_as_float(v1.z); x[7] = __uint_as_float(v1.w);
    }
    const uint64_t scale2 = f2_pack(q.scale, q.scale), nc2 = f2_pack(-q.c, -q.c);
#pragma unroll
    for (int k = 0; k < EPT; k += 2) {
        f2_unpack(f2_fma(f2_pack(x[k], x[k + 1]), scale2, nc2), e[k], e[k + 1]);
        e[k] = od_ex2(e[k]); e[k + 1] = od_ex2(e[k + 1]);
    }
}
__device__ __forceinline__ float sum_of_eight(const float *r)
{
    float s0, s1;
    f2_unpack(f2_add(f2_add(f2_pack(r[0], r[1]), f2_pack(r[2], r[3])), f2_add(f2_pack(r[4], r[5]), f2_pack(r[6], r[7]))), s0, s1);
    return s0 + s1;
}
template <int DTYPE>
__device__ __forceinline__ float with_eq2_ids(const SeqState &q, const SampleArgs &a, int tile, int lane, float *r)
{
    if (tile == q.prefix_token / OD_SAMPLE_TILE || tile == q.ngram_token / OD_SAMPLE_TILE)
        eq2_ids<DTYPE>(q, a, tile * OD_SAMPLE_TILE + lane * EPT, r);
    return sum_of_eight(r);
}
template <int DTYPE>
__device__ __forceinline__ float tile_lane_sum(const SeqState &q, const SampleArgs &a, int tile, int lane, const uint4 *raw,
                                               const float *qq)
{
    float r[EPT];
    tile_e<DTYPE>(q, raw, r);
#pragma unroll
    for (int k = 0; k < EPT; ++k) r[k] = fmaxf(0.f, fmaf(-qq[k], q.S, r[k]));
    return with_eq2_ids<DTYPE>(q, a, tile, lane, r);
}
// the same with the probabilities in shared memory at `rank_at` (the address of the lane's first
// mapped id's; `oct` says which of the eight are mapped)
template <int DTYPE>
__device__ __forceinline__ float tile_lane_sum_staged(const SeqState &q, const SampleArgs &a, int tile, int lane, const uint4 *raw,
                                                      uint32_t oct, uint32_t rank_at)
{
    float r[EPT];
    tile_e<DTYPE>(q, raw, r);
    const float nS = -q.S;
#pragma unroll
    for (int k = 0; k < EPT; ++k)
        // (read for every id, mapped or not: the last rank has a word behind it)
        asm("{.reg .pred p; .reg .b32 t; .reg .f32 v;\n\t"
            "and.b32 t, %3, %4; setp.ne.u32 p, t, 0;\n\t"
            "ld.shared.f32 v, [%1];\n\t"
            "@p fma.rn.f32 %0, v, %2, %0;\n\t"
            "@p add.u32 %1, %1, 4; max.f32 %0, %0, 0f00000000;}"
            : "+f"(r[k]), "+r"(rank_at) : "f"(nS), "r"(oct), "r"(1u << k) : "memory");
    return with_eq2_ids<DTYPE>(q, a, tile, lane, r);
}

// The lanes' sums of two tiles: lanes 0..15 end with the first tile's value, lanes 16..31 with the second's.
__device__ __forceinline__ float pair_sum(float s0, float s1, int lane)
{
    const bool up = lane & 16;
    float v = (up ? s1 : s0) + __shfl_xor_sync(0xFFFFFFFFu, up ? s0 : s1, 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    return v;
}

// Inverse-map entries of a warp's first pair of whole tiles [t_lo, t_hi).
__device__ __forceinline__ void first_pair_entries(const SampleArgs &a, int t_lo, int t_hi, int lane, int4 (&ni)[2][2])
{
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int t0 = (t_lo + i < t_hi ? t_lo + i : t_lo) * OD_SAMPLE_TILE + lane * EPT;
        ni[i][0] = __ldg((const int4 *)(a.inv_map + t0));
        ni[i][1] = __ldg((const int4 *)(a.inv_map + t0) + 1);
    }
}

// The same pass for a residual draw, software-pipelined over pairs of WHOLE tiles: the
// inverse-map entries of the next pair are requested before the current pair's gathers,
// so a pair costs one memory round trip, not two. ni: the first pair's entries
// (first_pair_entries), which the caller requested early: they belong to the context and
// depend on nothing the launch in front writes.
template <int DTYPE, typename Sink>
__device__ __forceinline__ void warp_tiles_dense_piped(const SeqState &q, const SampleArgs &a, int t_lo, int t_hi,
                                                       int lane, Sink &out, int4 (&ni)[2][2])
{
    for (int t = t_lo; t < t_hi; t += 2) {
        int32_t d[2][EPT];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            d[i][0] = ni[i][0].x; d[i][1] = ni[i][0].y; d[i][2] = ni[i][0].z; d[i][3] = ni[i][0].w;
            d[i][4] = ni[i][1].x; d[i][5] = ni[i][1].y; d[i][6] = ni[i][1].z; d[i][7] = ni[i][1].w;
        }
        if (t + 2 < t_hi) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int t0 = (t + 2 + i < t_hi ? t + 2 + i : t + 2) * OD_SAMPLE_TILE + lane * EPT;
                ni[i][0] = __ldg((const int4 *)(a.inv_map + t0));
                ni[i][1] = __ldg((const int4 *)(a.inv_map + t0) + 1);
            }
        }
        const bool two = t + 1 < t_hi;
        uint4 raw[2][RAW<DTYPE>];
#pragma unroll
        for (int i = 0; i < 2; ++i) load_tile<DTYPE>(q, i == 0 || two ? t + i : t, lane, raw[i]);
        float qq[2][EPT];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) qq[i][e] = d[i][e] >= 0 ? __ldg(q.q_row + d[i][e]) : 0.f;
        }
        const float s0 = tile_lane_sum<DTYPE>(q, a, t, lane, raw[0], qq[0]);
        const float s1 = tile_lane_sum<DTYPE>(q, a, t + 1, lane, raw[1], qq[1]);
        out.pair(t, pair_sum(s0, s1, lane), two);
    }
}

// A whole tile's loads other than through the inverse map: the logits, and
//   FROM_ROW  the drafter's probabilities where target ids are draft ids
//   STAGED    which of the ids are mapped, and the rank of the first
//   FREE      nothing else (the free token is drawn from p itself)
template <int DTYPE, int SOURCE>
struct TileLoads {
    uint4 raw[RAW<DTYPE>];
    float qq[SOURCE == FROM_ROW ? EPT : 1];
    uint32_t oct;
    __device__ __forceinline__ void load(const SeqState &q, const SampleArgs &a, int tile, int lane)
    {
        load_tile<DTYPE>(q, tile, lane, raw);
        if (SOURCE == FROM_ROW) same_id_probs(q, a, tile * OD_SAMPLE_TILE + lane * EPT, qq);
        if (SOURCE == STAGED) oct = __ldg(a.octet + tile * (OD_SAMPLE_TILE / 8) + lane);
    }
    __device__ __forceinline__ float sum(const SeqState &q, const SampleArgs &a, const StagedRow &sr, int tile, int lane) const
    {
        if (SOURCE == STAGED)
            return tile_lane_sum_staged<DTYPE>(q, a, tile, lane, raw, oct,
                                               (uint32_t)__cvta_generic_to_shared(sr.q) + ((oct >> 8) - sr.rank0) * 4u);
        if (SOURCE == FREE) {
            float e[EPT];
            tile_e<DTYPE>(q, raw, e);
            return sum_of_eight(e);
        }
        return tile_lane_sum<DTYPE>(q, a, tile, lane, raw, qq);
    }
};

// Pass 1 over whole tiles [t_lo, t_hi) without the inverse map: the loads of the next tiles are
// issued before the current ones are worked on. cur: the first two tiles', which the caller
// requested (FROM_ROW keeps one tile ahead only, for its registers).
template <int DTYPE, int SOURCE, typename Sink>
__device__ __forceinline__ void warp_tiles_ahead(const SeqState &q, const SampleArgs &a, const StagedRow &sr, int t_lo, int t_hi,
                                                 int lane, Sink &out, TileLoads<DTYPE, SOURCE> (&cur)[SOURCE == FROM_ROW ? 1 : 2])
{
#pragma unroll 1
    for (int t = t_lo; t < t_hi; t += 2) {
        const bool two = t + 1 < t_hi;
        float s0, s1;
        if (SOURCE == FROM_ROW) {
            TileLoads<DTYPE, SOURCE> nx;
            nx.load(q, a, two ? t + 1 : t, lane);
            s0 = cur[0].sum(q, a, sr, t, lane);
            if (t + 2 < t_hi) cur[0].load(q, a, t + 2, lane);
            s1 = nx.sum(q, a, sr, t + 1, lane);
        } else {
            TileLoads<DTYPE, SOURCE> nx[2];
            if (t + 2 < t_hi) {
                nx[0].load(q, a, t + 2, lane);
                nx[1].load(q, a, min(t + 3, t_hi - 1), lane);
            }
            s0 = cur[0].sum(q, a, sr, t, lane);
            s1 = cur[SOURCE == FROM_ROW ? 0 : 1].sum(q, a, sr, t + 1, lane);
            cur[0] = nx[0]; cur[SOURCE == FROM_ROW ? 0 : 1] = nx[1];
        }
        out.pair(t, pair_sum(s0, s1, lane), two);
    }
}
template <int DTYPE, int SOURCE>
__device__ __forceinline__ void first_tiles(const SeqState &q, const SampleArgs &a, int t_lo, int t_hi, int lane,
                                            TileLoads<DTYPE, SOURCE> (&cur)[SOURCE == FROM_ROW ? 1 : 2])
{
    if (t_lo >= t_hi) return;
    cur[0].load(q, a, t_lo, lane);
    if (SOURCE != FROM_ROW) cur[SOURCE == FROM_ROW ? 0 : 1].load(q, a, min(t_lo + 1, t_hi - 1), lane);
}

// Sum of s_val[my_lo, my_hi) over the block's threads in the order of the scan of
// pass 2 (a thread's run, lanes in order, warps in order); every thread gets it.
__device__ __forceinline__ double block_total(const double *s_val, int my_lo, int my_hi, double *s_warp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double inc = 0.0;
    for (int t = my_lo; t < my_hi; ++t) inc += s_val[t];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double v = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += v;
    }
    __syncthreads();                                // s_warp may still be read from an earlier call
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    double tot = 0.0;
    for (int w = 0; w < WARPS; ++w) tot += s_warp[w];
    return tot;
}

// ---- what both kernels prepare and decide alike -------------------------------------------

// What a block can load before the verification kernels have finished: what the translation
// kernel wrote, for every position the step can stop at. Lane k of every warp prepares
// position k. Two memory round trips, not a chain of four: everything that is addressed by
// (b, lane) alone is requested at once, whether or not it will be used (lane < K keeps the
// addresses inside the arrays); what is addressed by those values comes second.
struct Ahead {
    int mb;
    bool stop;
    float T;
    int32_t l_len, l_tgt;               // piece `lane`: its length, target id
    float l_qp;                         // and q'
    int32_t s0, len, tgt, d1, pm;       // position `lane`: row of the drafter, length of the piece there (1 at a stop);
    float qp, qd1;                      // of a merged piece: target, q', first sub-token, its image and probability
};
__device__ __forceinline__ Ahead load_ahead(const SampleArgs &a, int b, int lane)
{
    const int K = a.K_max;
    Ahead h;
    int mb = a.m[b];
    h.stop = a.tail_kind[b] == OD_TAIL_UNMAPPED_STOP;
    h.T = a.temperature[b];
    int32_t l_s0 = 0, l_did = -1;
    h.l_len = 1; h.l_tgt = -1; h.l_qp = 0.f;
    if (lane < K) {
        const size_t o = (size_t)b * K + lane;
        l_s0 = a.span_start[o];
        h.l_len = a.span_len[o];
        h.l_tgt = a.tgt_ids[o];
        h.l_qp = a.q_prime[o];
        l_did = a.draft_ids[o];
    }
    h.mb = mb < 0 ? 0 : (mb > K ? K : mb);
    h.s0 = 0; h.len = 1; h.tgt = -1; h.d1 = -1; h.pm = -1; h.qp = 0.f; h.qd1 = 0.f;
    const bool live = lane < K && lane <= h.mb;
    if (live) {
        h.s0 = l_s0 < 0 ? 0 : (l_s0 >= K ? K - 1 : l_s0);
        h.len = lane < h.mb ? h.l_len : 1;
    }
    const int32_t d1 = __shfl_sync(0xFFFFFFFFu, l_did, h.s0);       // the span's first draft token
    if (live && h.len >= 2) {
        h.tgt = h.l_tgt;
        h.qp = h.l_qp;
        if (d1 >= 0 && d1 < a.v_q) {
            h.d1 = d1;
            h.pm = __ldg(a.vocab_map + d1);
            h.qd1 = __ldg(a.q_rows + ((size_t)b * K + h.s0) * a.v_q + d1);
        }
    }
    return h;
}

// What the draw at position j needs; rm, rs: lane k holds the statistics of row k. A shard's row
// pointer is moved back by the shard's first column (col0), and only ids of the window are read.
template <int DTYPE>
__device__ __forceinline__ SeqState seq_state(const SampleArgs &a, const Ahead &h, int b, int j, float rm, float rs, int col0,
                                              bool planned)
{
    const size_t esz = DTYPE == OD_BF16 ? 2 : 4;
    SeqState q;
    q.row = (const char *)a.logits + ((size_t)b * a.seq_stride + (size_t)j * a.row_stride) * esz - (size_t)col0 * esz;
    q.scale = 1.4426950408889634f / h.T;
    {
        // reference exponent c = fl(M*scale), od_verify's own, so that the errors of e(t) are those of the
        // row sum (a margin on it, to keep e(t) below one, made the residual mass's mean error 5 to 10 %
        // larger, and at |M|/T > 8.8e7 zero of everything); its rounding goes into S exactly:
        // sum_t exp2(x_t*scale - c) = (sum_t exp2((x_t - M)*scale)) * exp2(M*scale - c)
        const float M = __shfl_sync(0xFFFFFFFFu, rm, j);
        q.c = fmaxf(M * q.scale, -FLT_MAX);
        q.S = __shfl_sync(0xFFFFFFFFu, rs, j) * od_ex2(fmaf(M, q.scale, -q.c));
    }
    q.residual = (j < h.mb) || h.stop;
    q.from_row = a.same_ids && planned;
    q.ngram_token = -1; q.prefix_token = -1; q.ngram_prob = 0.f; q.prefix_val = 0.f;
    q.q_row = a.q_rows;
    // position j's preparation (j < K whenever the draw is a residual one)
    const int src = j < a.K_max ? j : 0;
    const int32_t s0 = __shfl_sync(0xFFFFFFFFu, h.s0, src), len = __shfl_sync(0xFFFFFFFFu, h.len, src);
    const int32_t tgt = __shfl_sync(0xFFFFFFFFu, h.tgt, src), d1 = __shfl_sync(0xFFFFFFFFu, h.d1, src);
    const int32_t pm = __shfl_sync(0xFFFFFFFFu, h.pm, src);
    const float qp = __shfl_sync(0xFFFFFFFFu, h.qp, src), qd1 = __shfl_sync(0xFFFFFFFFu, h.qd1, src);
    if (q.residual) {
        q.q_row = a.q_rows + ((size_t)b * a.K_max + s0) * a.v_q;
        if (len >= 2) {
            q.ngram_token = tgt;
            q.ngram_prob = qp;
            if (d1 >= 0) {
                q.prefix_token = pm;
                q.prefix_val = qd1 - q.ngram_prob;
            }
        }
    }
    return q;
}

// The gathers of pass 1 come two round trips from now: have the copy engine pull this block's
// share of the drafter's row into L2 meanwhile (one thread calls).
__device__ __forceinline__ void prefetch_q_row(const SampleArgs &a, const SeqState &q, unsigned part, unsigned nparts)
{
    const size_t row_bytes = (size_t)a.v_q * 4 / 16 * 16;
    const size_t lo = (row_bytes / nparts * part) / 16 * 16;
    const size_t hi = part + 1 == nparts ? row_bytes : (row_bytes / nparts * (part + 1)) / 16 * 16;
    const char *base = (const char *)q.q_row;
    if (((uintptr_t)base & 15u) == 0 && hi > lo)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + lo), "r"((uint32_t)(hi - lo)) : "memory");
}

// A warp's run of tiles [t_lo, t_hi): whole tiles pipelined, the row's ragged last tile (if it is
// this warp's) on its own. ni: the first pair's inverse-map entries (not read where ids are shared).
template <int DTYPE, int SOURCE, typename Sink>
__device__ __forceinline__ void warp_run(const SeqState &q, const SampleArgs &a, int t_lo, int t_hi, int hi_w, int lane,
                                         Sink &out, int4 (&ni)[2][2])
{
    const StagedRow none = {};
    if (t_lo >= t_hi) return;
    if (!q.residual) {
        TileLoads<DTYPE, FREE> cur[2];
        first_tiles<DTYPE, FREE>(q, a, t_lo, hi_w, lane, cur);
        warp_tiles_ahead<DTYPE, FREE>(q, a, none, t_lo, hi_w, lane, out, cur);
    } else if (SOURCE == FROM_ROW) {
        TileLoads<DTYPE, FROM_ROW> cur[1];
        first_tiles<DTYPE, FROM_ROW>(q, a, t_lo, hi_w, lane, cur);
        warp_tiles_ahead<DTYPE, FROM_ROW>(q, a, none, t_lo, hi_w, lane, out, cur);
    } else if (SOURCE == FROM_MAP && t_lo < hi_w) {
        warp_tiles_dense_piped<DTYPE>(q, a, t_lo, hi_w, lane, out, ni);
    }
    if (hi_w < t_hi) warp_tiles_dense<DTYPE, 1>(q, a, q.residual, max(hi_w, t_lo), t_hi, lane, out);
}

// One warp draws inside tile t_pick, whose ids begin at the running sum `before`: id by id, the
// first at which the sum passes `target` (or the tile's last one with mass, where rounding put the
// target past its end). Writes the outputs; false if the tile holds no mass after all.
template <int DTYPE>
__device__ __forceinline__ bool pick_in_tile(const SeqState &q, const SampleArgs &a, int b, bool residual, int t_pick,
                                             double before, double target, double Rn, uint32_t flags, int lane,
                                             const StagedRow *sr = nullptr)
{
    float r[EPT];
    if (residual) tile_values<DTYPE>(q, a, true, t_pick, lane, r, sr);
    else tile_e_values<DTYPE>(q, a, t_pick, lane, r);
    const double mine = lane_sum(r);
    double incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += v;
    }
    const double lbase = before + (incl - mine);            // sum before this lane's first id
    const int t0 = t_pick * OD_SAMPLE_TILE + lane * EPT;
    int my_pick = 0x7FFFFFFF, my_last = -1;
    double lo = 0.0, hi = 0.0, c = lbase;
    float run = 0.f;                                        // same fp32 order as lane_sum
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        run = e == 0 ? r[0] : run + r[e];
        const double nc = lbase + (double)run;
        if (r[e] > 0.f) my_last = t0 + e;
        if (my_pick == 0x7FFFFFFF && nc > target) { my_pick = t0 + e; lo = c; hi = nc; }
        c = nc;
    }
    int pick = my_pick, last = my_last;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        pick = min(pick, __shfl_xor_sync(0xFFFFFFFFu, pick, off));
        last = max(last, __shfl_xor_sync(0xFFFFFFFFu, last, off));
    }
    const float R = (float)(Rn / (double)q.S);              // residual mass (1 for the free token)
    if (pick != 0x7FFFFFFF) {
        if (my_pick == pick) {                              // exactly one lane owns the picked id
            uint32_t f = flags;
            if (fmin(target - lo, hi - target) <= OD_TAU_SAMPLE * Rn) f |= OD_SF_BOUNDARY;
            a.out_token[b] = pick; a.resid_mass[b] = R; a.flags[b] = f;
        }
        return true;
    }
    if (last >= 0) {
        // rounding: the target lies beyond the tile's last edge
        if (lane == 0) { a.out_token[b] = last; a.resid_mass[b] = R; a.flags[b] = flags | OD_SF_BOUNDARY; }
        return true;
    }
    return false;
}

// ---- the whole step on full rows -------------------------------------------------------------
//
// Grid (P, B), clusters of P blocks (od_sample_parts) of 16 warps: one cluster draws for one sequence. Pass 1 as
// above, the tile values of a warp's run staying in its block's shared memory. A block sends its
// sum to all blocks of the cluster (distributed shared memory), and behind ONE cluster barrier
// every warp has the blocks' sums and its own block's runs, scans both and knows whether the draw
// falls into its run: that warp, alone and without a further barrier, finds the tile and the id.
// Stamps, last tile done -> token: 2.6 us, of which the exchange is 1.0 and the picked tile 1.0
// (4.5 us for blocks of 8 warps that hand over through a ticket, reload the tile values and scan
// them block-wide; 3.2 with all P * 16 run sums exchanged and scanned by every warp).
// The whole step, device time: one sequence of 32000 fp32 ids 13.3 -> 12.0 us, 24 of 128256 bf16
// ids 24.2 -> 22.6, 64 31.7 -> 29.7, 512 of 152064 286 -> 273, 256 of 32000 (same tokenizer) 44.2 -> 37.0.
// FUSED: the launch in front is the streaming pass of od_verify itself; its decide kernel is
// folded into this kernel's prologue (see SampleArgs).
constexpr int CWARPS = 16, CTHREADS = CWARPS * 32;

// No usable residual mass (rare): one block draws from p_j. Redoes the row's tile values with e
// alone, in global memory, and walks them.
template <int DTYPE>
__device__ __forceinline__ void draw_from_p(const SeqState &q, const SampleArgs &a, int b, float u, uint32_t flags)
{
    __shared__ double s_sum[CTHREADS];
    __shared__ int s_crossing, s_lastmass, s_done;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    GlobalTiles out = {a.tile_val + (size_t)b * a.ntiles, lane};
    for (int t = warp * 2; t < a.ntiles; t += CWARPS * 2)
        warp_tiles_dense<DTYPE, 2>(q, a, false, t, t + 2 < a.ntiles ? t + 2 : a.ntiles, lane, out);
    if (threadIdx.x == 0) { s_crossing = 0x7FFFFFFF; s_lastmass = -1; s_done = 0; }
    __syncthreads();
    const int per = (a.ntiles + CTHREADS - 1) / CTHREADS;
    const int lo = min((int)threadIdx.x * per, a.ntiles), hi = min(lo + per, a.ntiles);
    double loc = 0.0;
    for (int t = lo; t < hi; ++t) loc += fmax(0.0, out.val[t]);
    s_sum[threadIdx.x] = loc;
    __syncthreads();
    double before = 0.0, tot = 0.0;
    for (int i = 0; i < CTHREADS; ++i) {
        if (i == (int)threadIdx.x) before = tot;
        tot += s_sum[i];
    }
    const double target = (double)u * tot;
    int mine = -1, last = -1;
    double c = before, at = 0.0;
    for (int t = lo; t < hi; ++t) {
        const double v = fmax(0.0, out.val[t]);
        if (v > 0.0) last = t;
        if (mine < 0 && c + v > target) { mine = t; at = c; }
        c += v;
    }
    if (tot > 0.0) {
        if (mine >= 0) atomicMin(&s_crossing, mine);
        if (last >= 0) atomicMax(&s_lastmass, last);
    }
    __syncthreads();
    const int t_pick = s_crossing != 0x7FFFFFFF ? s_crossing : s_lastmass;
    if (t_pick >= 0 && t_pick == mine) s_sum[0] = at;
    else if (t_pick >= lo && t_pick < hi) {                 // rounding hid the crossing: the last tile with mass
        c = before;
        for (int t = lo; t < t_pick; ++t) c += fmax(0.0, out.val[t]);
        s_sum[0] = c;
    }
    __syncthreads();
    if (warp == 0 && t_pick >= 0 && pick_in_tile<DTYPE>(q, a, b, false, t_pick, s_sum[0], target, tot, flags, lane) && lane == 0)
        s_done = 1;
    __syncthreads();
    if (threadIdx.x == 0 && !s_done) {                      // no mass at all (non-finite input)
        a.out_token[b] = -1;
        a.resid_mass[b] = (float)(tot / (double)q.S);
        a.flags[b] = flags;
    }
}

template <int DTYPE, bool FUSED, int SOURCE>
__global__ void __launch_bounds__(CTHREADS, 2)
od_sample_kernel(const SampleArgs a)
{
    __shared__ float s_M[FUSED ? OD_MAX_K + 1 : 1], s_S[FUSED ? OD_MAX_K + 1 : 1];
    __shared__ int s_red[2][CWARPS];
    __shared__ unsigned int s_vbits;
    __shared__ int s_bare;
    __shared__ double s_run[CWARPS], s_part[OD_SAMPLE_MAX_PARTS];   // sums of the block's runs, of the cluster's blocks
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const unsigned part = blockIdx.x, nparts = gridDim.x;
    const int b = blockIdx.y;
    const int K = a.K_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the staged probabilities, then the warps' tile values
    float *s_q = (float *)s_dyn, *s_val = s_q + (SOURCE == STAGED ? a.slots : 0) + warp * a.tiles_per_warp;

    // Under programmatic dependent launch this grid is resident while the verification
    // kernels still run. What the translation kernel wrote (it finished before them) is
    // read now. (a.early = 0: the launch before this one was not od_verify; everything waits.)
    asm volatile("griddepcontrol.launch_dependents;");
    if (!a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int32_t map_serial = SOURCE == FROM_ROW ? __ldg(a.map_serial_now) : a.map_serial;
    const Ahead h = load_ahead(a, b, lane);
    const int mb = h.mb;

    // FUSED, still before the wait: where the rows' partials will be (sums of m), and position
    // k's inputs of the acceptance test in lane k
    int before = 0, total = 0;
    float d_xt = 0.f, d_u = 0.f;
    bool d_tok = false;
    if (threadIdx.x == 0) { s_vbits = 0; s_bare = 0; }
    if (FUSED) {
        for (int i = threadIdx.x; i < a.B; i += CTHREADS) {
            const int v = clamp_m(a.m[i], K);
            total += v;
            if (i < b) before += v;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            before += __shfl_xor_sync(0xFFFFFFFFu, before, off);
            total += __shfl_xor_sync(0xFFFFFFFFu, total, off);
        }
        if (lane == 0) { s_red[0][warp] = before; s_red[1][warp] = total; }
        if (lane < mb) {
            d_tok = h.l_tgt >= 0 && h.l_tgt < a.v_p;
            const char *row_k = (const char *)a.logits +
                                ((size_t)b * a.seq_stride + (size_t)lane * a.row_stride) * (DTYPE == OD_BF16 ? 2 : 4);
            if (d_tok) d_xt = od_load_logit<DTYPE>(row_k, h.l_tgt);
            d_u = od_uniform(a.seed[b], a.step, (uint32_t)lane, 0u);
        }
        __syncthreads();
        before = 0; total = 0;
        for (int w = 0; w < CWARPS; ++w) { before += s_red[0][w]; total += s_red[1][w]; }
    }

    // pass 1's tiles of this warp, and the inverse-map entries of their first pair
    int p_hi = min((int)(part + 1) * a.part_tiles, a.ntiles);
    const int p_lo = min((int)part * a.part_tiles + warp * a.tiles_per_warp, p_hi);
    p_hi = min(p_lo + a.tiles_per_warp, p_hi);
    int p_hi_w = min(p_hi, a.v_p / OD_SAMPLE_TILE);
    int4 ni[2][2] = {};
    if (SOURCE == FROM_MAP && p_lo < p_hi_w) first_pair_entries(a, p_lo, p_hi_w, lane, ni);
    // STAGED: the first entries of the part's list
    constexpr int EB = 6;                                   // groups per warp and batch
    uint32_t word[EB];
    int32_t base[EB];
    int4 my_part = {};
    int g_at = 0;
    auto load_words = [&]() {
#pragma unroll
        for (int e = 0; e < EB; ++e) {
            const bool in = g_at + e * CWARPS < my_part.y;
            word[e] = in ? __ldg(a.list_word + (size_t)(g_at + e * CWARPS) * 32 + lane) : 0xFFFFu;
            base[e] = in ? __ldg(a.list_base + g_at + e * CWARPS) : 0;
        }
        g_at += EB * CWARPS;
    };
    if (SOURCE == STAGED) {
        my_part = __ldg((const int4 *)a.list_part + part);
        if (my_part.w != a.map_serial) { my_part.y = 0; p_hi_w = p_lo; }   // another map: nothing is staged, all is looked up
        g_at = my_part.x + warp;
        load_words();
    }

    // n_accepted and the row statistics come from the verification kernels
    if (a.early) asm volatile("griddepcontrol.wait;" ::: "memory");

    int j = 0;
    float rm = 0.f, rs = 0.f;                      // lane k: statistics of row k
    if (FUSED) {
        // ---- step 2's decisions (what od_verify_decide_kernel does, same arithmetic, same order)
        const bool bad_T = !(h.T > 0.f);
        const float dscale = bad_T ? 0.f : 1.4426950408889634f / h.T;
        for (int r = warp; r <= mb; r += CWARPS) {
            const int row_slot = b * (K + 1) + r;
            float c, sum, mx;
            merge_row_partials(a.plan, row_slot, row_partial_segments(a.plan, b, r, before, total), lane, c, sum, mx);
            if (lane == 0) {
                const float S = row_sum_of(c, sum, mx, dscale);
                s_M[r] = mx; s_S[r] = S;
                if (part == 0) { a.w_row_max[row_slot] = mx; a.w_row_sum[row_slot] = S; }
                if (!(S > 0.f) || !(S <= FLT_MAX)) atomicOr(&s_vbits, 1u);
            }
        }
        __syncthreads();
        // every warp takes the decisions for itself (lane k = position k holds the inputs in
        // every warp): no second barrier; warp 0 of the sequence's first block stores them
        bool acc = false, bnd = false;
        Acceptance d = {};
        if (lane <= mb) { rm = s_M[lane]; rs = s_S[lane]; }
        if (lane < mb) {
            d = accept_position(rm, rs, dscale, d_tok, d_xt, h.l_qp, d_u);
            acc = d.accept; bnd = d.boundary;
        }
        const unsigned int accmask = __ballot_sync(0xFFFFFFFFu, acc);
        while (j < mb && (accmask >> j & 1u)) ++j;
        if (bad_T) j = 0;
        if (part == 0 && warp == 0) {
            if (lane < mb) { a.w_p_sel[(size_t)b * K + lane] = d.p; a.w_ratio[(size_t)b * K + lane] = d.ratio; }
            const unsigned int bndmask = __ballot_sync(0xFFFFFFFFu, bnd);
            int nd = lane < j ? h.l_len : 0;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) nd += __shfl_xor_sync(0xFFFFFFFFu, nd, off);
            if (lane == 0) {
                uint32_t f = bndmask & OD_VF_BOUNDARY_MASK;
                if (s_vbits & 1u) f |= OD_VF_NONFINITE;
                if (bad_T) f |= OD_VF_BAD_TEMPERATURE;
                a.w_n_accepted[b] = j; a.w_n_draft[b] = nd; a.w_vflags[b] = f;
            }
        }
    } else {
        if (lane <= mb) { rm = a.row_max[b * (K + 1) + lane]; rs = a.row_sum[b * (K + 1) + lane]; }
        j = a.n_accepted[b];
        j = j < 0 ? 0 : (j > mb ? mb : j);
    }
    if (!(h.T > 0.f)) {                            // every block of the sequence leaves here
        if (part == 0 && threadIdx.x == 0) { a.out_token[b] = -1; a.resid_mass[b] = 0.f; a.flags[b] = OD_SF_BAD_TEMPERATURE; }
        return;
    }
    // FROM_ROW: the map is still the one this launch was laid out for
    const bool planned = map_serial == a.map_serial;
    od_cluster_arrive_relaxed();                   // this block runs: the others may store to it (waited for below)
    const SeqState q = seq_state<DTYPE>(a, h, b, j, rm, rs, 0, planned);
    if (SOURCE == FROM_MAP && q.residual && threadIdx.x == 0) prefetch_q_row(a, q, part, nparts);

    // ---- pass 1: the value of every tile; the ragged last one (all of them, if the map is another) one by one ----
    WarpTiles out = {s_val, lane, p_lo, 0.0};
    const int hi_w = planned ? p_hi_w : p_lo;
    const uint64_t seed_b = a.seed[b];
    const StagedRow sr = {s_q, a.octet, (uint32_t)my_part.z};
    if (SOURCE == STAGED && q.residual) {
        TileLoads<DTYPE, STAGED> cur[2];
        first_tiles<DTYPE, STAGED>(q, a, p_lo, hi_w, lane, cur);
        // the part's probabilities, gathered in draft-id order, to their ranks in shared memory
        for (;;) {
            float x[EB];
            uint32_t at[EB];
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                at[e] = word[e] & 0xFFFFu;
                if (at[e] != 0xFFFFu) x[e] = __ldg(q.q_row + base[e] + (int)(word[e] >> 16));
            }
            const bool more = g_at < my_part.y;             // the same for every lane of a warp
            if (more) load_words();
#pragma unroll
            for (int e = 0; e < EB; ++e)
                if (at[e] != 0xFFFFu) s_q[at[e]] = x[e];
            if (!more) break;
        }
        __syncthreads();
        warp_tiles_ahead<DTYPE, STAGED>(q, a, sr, p_lo, hi_w, lane, out, cur);
        if (hi_w < p_hi) warp_tiles_dense<DTYPE, 1>(q, a, true, max(hi_w, p_lo), p_hi, lane, out);
    } else {
        warp_run<DTYPE, SOURCE>(q, a, p_lo, p_hi, hi_w, lane, out, ni);
    }
    const float u = od_uniform(seed_b, a.step, (uint32_t)j, 1u);

    // ---- the sums: of the runs inside the block, of the block to every block of the cluster
    const double run_sum = out.sum();
    if (lane == 0) s_run[warp] = run_sum;
    __syncthreads();
    // every warp holds the block's runs in lanes 0..15 (and again in 16..31), summed up
    const double mine = s_run[lane & 15];
    double incl = mine;
#pragma unroll
    for (int off = 1; off < CWARPS; off <<= 1) {
        const double v = __shfl_up_sync(0xFFFFFFFFu, incl, off, CWARPS);
        if ((lane & 15) >= off) incl += v;
    }
    const double block_sum = __shfl_sync(0xFFFFFFFFu, incl, 15);
    od_cluster_wait();
    if (warp == 0 && lane < (int)nparts) od_cluster_store(&s_part[part], (uint32_t)lane, block_sum);
    od_cluster_arrive();
    od_cluster_wait();

    // ---- every warp scans the blocks' sums: is the draw in its block, in its run?
    const uint32_t flags = q.residual ? 0u : OD_SF_BONUS;
    const double p_sum = (lane & 15) < (int)nparts ? s_part[lane & 15] : 0.0;
    double p_incl = p_sum;
#pragma unroll
    for (int off = 1; off < OD_SAMPLE_MAX_PARTS; off <<= 1) {
        const double v = __shfl_up_sync(0xFFFFFFFFu, p_incl, off, OD_SAMPLE_MAX_PARTS);
        if ((lane & 15) >= off) p_incl += v;
    }
    const double Rn = __shfl_sync(0xFFFFFFFFu, p_incl, 15);  // unnormalised total
    bool bare = !(Rn > 0.0);                                 // the same in every warp of the cluster
    if (!bare) {
        const double target = (double)u * Rn;
        // the first block, then its first run, at whose end the sum passes the target; if rounding
        // hid it, the last with mass
        const auto first_past = [&](double before, double sum, double upto) {
            const unsigned past = __ballot_sync(0xFFFFFFFFu, sum > 0.0 && before + upto > target) & 0xFFFFu;
            const unsigned held = __ballot_sync(0xFFFFFFFFu, sum > 0.0) & 0xFFFFu;
            return past ? __ffs(past) - 1 : 31 - __clz(held);   // -1: no mass
        };
        const int p_hit = first_past(0.0, p_sum, p_incl);
        int run = -1;
        double at = __shfl_sync(0xFFFFFFFFu, p_incl - p_sum, p_hit & 15);
        if (p_hit == (int)part) {
            run = first_past(at, mine, incl);
            at += __shfl_sync(0xFFFFFFFFu, incl - mine, run & 15);
        }
        // ---- the warp whose run it is finds the tile, then the id
        if (run == warp) {
            const int n = p_hi - p_lo;
            int pick = -1, held = -1;
            double at_pick = 0.0, at_held = 0.0;
            for (int t0 = 0; t0 < n && pick < 0; t0 += 32) {
                const double v = t0 + lane < n ? (double)s_val[t0 + lane] : 0.0;
                double s = v;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const double w = __shfl_up_sync(0xFFFFFFFFu, s, off);
                    if (lane >= off) s += w;
                }
                const unsigned cross = __ballot_sync(0xFFFFFFFFu, v > 0.0 && at + s > target);
                const unsigned mass = __ballot_sync(0xFFFFFFFFu, v > 0.0);
                if (mass) {
                    const int l = cross ? __ffs(cross) - 1 : 31 - __clz(mass);
                    held = t0 + l;
                    at_held = at + __shfl_sync(0xFFFFFFFFu, s - v, l);
                    if (cross) { pick = held; at_pick = at_held; }
                }
                at += __shfl_sync(0xFFFFFFFFu, s, 31);
            }
            if (pick < 0) { pick = held; at_pick = at_held; }        // rounding hid it: the last tile with mass
            const bool drawn = pick >= 0 && pick_in_tile<DTYPE>(q, a, b, q.residual, p_lo + pick, at_pick, target, Rn, flags, lane,
                                                                 SOURCE == STAGED && my_part.y ? &sr : nullptr);
            if (lane == 0 && !drawn) s_bare = 1;             // the tile holds no mass after all
        }
        __syncthreads();
        bare = s_bare;
    } else if (part != 0) {
        return;
    }
    if (bare) draw_from_p<DTYPE>(q, a, b, u, flags | OD_SF_ZERO_MASS);
}

// ---- vocabulary shards: MODE 1, a shard's mass shares; MODE 2, a shard's pick ---------------
template <int DTYPE, int MODE>
__global__ void __launch_bounds__(OD_SAMPLE_THREADS, 4)
od_sample_shard_kernel(const SampleArgs a)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];   // ntiles x 8 bytes
    double *s_val = (double *)s_dyn;                         // pass 2: tile values
    __shared__ double s_warp[WARPS];
    __shared__ unsigned int s_last;
    __shared__ int s_tile, s_lastmass, s_done;
    __shared__ double s_before;
    __shared__ double s_cross[OD_SAMPLE_THREADS];           // pass 2: the sum in front of a thread's crossing tile

    // grid = (sequences, parts of a row): blocks with neighbouring indices, which often end up on
    // one multiprocessor, then work on the same tiles of different sequences and share the
    // inverse-map entries in L1
    const int b = blockIdx.x;
    const unsigned int part = blockIdx.y, nparts = gridDim.y;
    const int K = a.K_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    asm volatile("griddepcontrol.launch_dependents;");
    if (!a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    const Ahead h = load_ahead(a, b, lane);
    const int mb = h.mb;
    const float T = h.T;
    const bool planned = __ldg(a.map_serial_now) == a.map_serial;   // (as in od_sample_kernel)

    // a shard's tiles and ids keep their numbers of the full row
    const int tile_lo = a.tile_lo, tile_hi = a.tile_hi;
    // pass 1's whole tiles of this warp, and the inverse-map entries of their first pair
    const int p_lo = tile_lo + ((int)part * WARPS + warp) * a.tiles_per_warp;
    int p_hi = p_lo + a.tiles_per_warp;
    if (p_hi > tile_hi) p_hi = tile_hi;
    const int p_hi_w = p_hi < a.v_p / OD_SAMPLE_TILE ? p_hi : a.v_p / OD_SAMPLE_TILE;
    int4 ni[2][2] = {};
    if (MODE != 2 && !a.same_ids && p_lo < p_hi_w) first_pair_entries(a, p_lo, p_hi_w, lane, ni);

    // n_accepted and the row statistics come from the verification kernels
    if (a.early) asm volatile("griddepcontrol.wait;" ::: "memory");

    if (!(T > 0.f)) {                              // every block of the sequence leaves here
        if (part == 0 && threadIdx.x == 0) {
            if (MODE == 1) {
                a.mass_out[2 * b] = 0.0; a.mass_out[2 * b + 1] = 0.0;
            } else {
                a.out_token[b] = -1; a.resid_mass[b] = 0.f; a.flags[b] = OD_SF_BAD_TEMPERATURE;
            }
        }
        return;
    }
    float rm = 0.f, rs = 0.f;                      // lane k: statistics of row k
    if (lane <= mb) {
        rm = a.row_max[b * (K + 1) + lane];
        rs = a.row_sum[b * (K + 1) + lane];
    }
    int j = a.n_accepted[b];
    j = j < 0 ? 0 : (j > mb ? mb : j);
    const SeqState q = seq_state<DTYPE>(a, h, b, j, rm, rs, a.col0, planned);
    if (MODE != 2 && q.residual && threadIdx.x == 0) prefetch_q_row(a, q, part, nparts);

    const int ntiles = a.ntiles;
    double *tile_val = a.tile_val + (size_t)b * ntiles;
    GlobalTiles out = {tile_val, lane};

    if (MODE != 2) {
        // ---- pass 1: the value of every tile ----
        const int hi_w = planned || !a.same_ids ? p_hi_w : p_lo;
        if (a.same_ids) warp_run<DTYPE, FROM_ROW>(q, a, p_lo, p_hi, hi_w, lane, out, ni);
        else warp_run<DTYPE, FROM_MAP>(q, a, p_lo, p_hi, hi_w, lane, out, ni);
        // The tile values are read by another block: the barrier orders this block's stores
        // before thread 0's fence, the fence before its ticket (release); the block that
        // draws the last ticket fences again before anyone in it reads (acquire).
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(a.ticket + b, 1u) == nparts - 1 ? 1u : 0u;
            __threadfence();
        }
        __syncthreads();
        if (!s_last) return;
    }

    // ---- pass 2 (one block per sequence) ----
    bool residual = q.residual;
    uint32_t flags = residual ? 0u : OD_SF_BONUS;
    const int per = (tile_hi - tile_lo + OD_SAMPLE_THREADS - 1) / OD_SAMPLE_THREADS;
    const int my_lo = tile_lo + threadIdx.x * per < tile_hi ? tile_lo + threadIdx.x * per : tile_hi;
    const int my_hi = my_lo + per < tile_hi ? my_lo + per : tile_hi;
    // tile values (rounding can leave a tile without residual mass slightly negative): four
    // requests per thread at a time, and the draw's uniform worked out while they travel
    float u = 0.f;
    const uint64_t seed_b = MODE == 1 ? 0ull : a.seed[b];   // requested with the tile values, used behind them
    for (int t0 = tile_lo + threadIdx.x, first = 1; first || t0 < tile_hi; t0 += 4 * OD_SAMPLE_THREADS, first = 0) {
        double v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = t0 + i * OD_SAMPLE_THREADS;
            v[i] = t < tile_hi ? __ldcg(tile_val + t) : 0.0;
        }
        if (MODE != 1 && first) u = od_uniform(seed_b, a.step, (uint32_t)j, 1u);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = t0 + i * OD_SAMPLE_THREADS;
            if (t < tile_hi) s_val[t] = fmax(0.0, v[i]);
        }
    }
    if (MODE != 2 && threadIdx.x == 0) a.ticket[b] = 0;
    __syncthreads();

    if (MODE == 1) {
        // ---- this shard's shares ----
        const double mass_r = block_total(s_val, my_lo, my_hi, s_warp);
        double mass_e = 0.0;
        if (residual && !(mass_r > 0.0)) {
            // no residual mass here: should no shard have any, the draw is from p_j
            for (int t_lo = tile_lo + warp * 2; t_lo < tile_hi; t_lo += WARPS * 2)
                warp_tiles_dense<DTYPE, 2>(q, a, false, t_lo, t_lo + 2 < tile_hi ? t_lo + 2 : tile_hi, lane, out);
            __syncthreads();
            for (int t = tile_lo + threadIdx.x; t < tile_hi; t += OD_SAMPLE_THREADS) s_val[t] = fmax(0.0, tile_val[t]);
            __syncthreads();
            mass_e = block_total(s_val, my_lo, my_hi, s_warp);
        }
        if (threadIdx.x == 0) { a.mass_out[2 * b] = mass_r; a.mass_out[2 * b + 1] = mass_e; }
        return;
    }

    double shard_before = 0.0, shard_total = 0.0;      // MODE 2: sums over the shards before this one / all
    if (MODE == 2) {
        double tot_r = 0.0, tot_e = 0.0;
        for (int s = 0; s < a.n_shards; ++s) {
            tot_r += a.mass_all[((size_t)s * a.B + b) * 2];
            tot_e += a.mass_all[((size_t)s * a.B + b) * 2 + 1];
        }
        const bool use_e = residual && !(tot_r > 0.0);
        if (use_e) { residual = false; flags |= OD_SF_ZERO_MASS; }   // the tile values then hold p_j's
        shard_total = use_e ? tot_e : tot_r;
        // the shard in which the running sum crosses the target (else the last one with mass)
        int owner = -1;
        if (shard_total > 0.0) {
            const double target = (double)u * shard_total;
            double c = 0.0;
            int last = -1;
            for (int s = 0; s < a.n_shards; ++s) {
                const double v = a.mass_all[((size_t)s * a.B + b) * 2 + (use_e ? 1 : 0)];
                if (s == a.shard_index) shard_before = c;
                if (v > 0.0) last = s;
                if (c + v > target) { owner = s; break; }
                c += v;
            }
            if (owner < 0) owner = last;
        }
        if (owner != a.shard_index) {
            if (threadIdx.x == 0) {
                const bool report = owner < 0 && a.shard_index == 0;   // no mass anywhere: shard 0 says so
                a.out_token[b] = -1;
                a.resid_mass[b] = report ? (float)(shard_total / (double)q.S) : 0.f;
                a.flags[b] = report ? (flags | OD_SF_ZERO_MASS) : 0u;
            }
            return;
        }
    }

    // exclusive scan of the tile values: thread i owns `per` consecutive tiles
    double loc = 0.0;
    for (int t = my_lo; t < my_hi; ++t) loc += s_val[t];
    double inc = loc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double v = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += v;
    }
    if (lane == 31) s_warp[warp] = inc;
    if (threadIdx.x == 0) { s_tile = 0x7FFFFFFF; s_lastmass = -1; s_done = 0; }
    __syncthreads();
    double base = shard_before, tot = 0.0;
    for (int w = 0; w < WARPS; ++w) {
        if (w == warp) base += tot;
        tot += s_warp[w];
    }
    double target = 0.0;
    if (shard_total > 0.0) {
        target = (double)u * shard_total;
        double c = base + inc - loc;
        int last = -1;
        for (int t = my_lo; t < my_hi; ++t) {
            const double v = s_val[t];
            if (v > 0.0) last = t;
            if (c + v > target) {
                // first crossing of this run: the tile, and with it who found it, so that
                // the sum before the tile needs no barrier of its own
                s_cross[threadIdx.x] = c;
                atomicMin(&s_tile, t * OD_SAMPLE_THREADS + (int)threadIdx.x);
                break;
            }
            c += v;
        }
        if (last >= 0) atomicMax(&s_lastmass, last);
    }
    __syncthreads();
    // cumulative sums never decrease, so the smallest reported tile is the crossing;
    // if rounding hid it, take the last tile that has mass
    int t_pick = -1;
    if (shard_total > 0.0) {
        if (s_tile != 0x7FFFFFFF) {
            t_pick = s_tile / OD_SAMPLE_THREADS;
            if (threadIdx.x < 32) s_before = s_cross[s_tile % OD_SAMPLE_THREADS];   // warp 0 reads it back below
            __syncwarp();
        } else {
            t_pick = s_lastmass;
            if (t_pick >= my_lo && t_pick < my_hi) {    // its owner publishes the sum before it
                double c = base + inc - loc;
                for (int t = my_lo; t < t_pick; ++t) c += s_val[t];
                s_before = c;
            }
            __syncthreads();                            // (block-uniform: s_tile is the same for all)
        }
    }
    if (t_pick >= 0 && warp == 0 &&
        pick_in_tile<DTYPE>(q, a, b, residual, t_pick, s_before, target, shard_total, flags, lane) && lane == 0)
        s_done = 1;
    __syncthreads();
    if (threadIdx.x == 0 && !s_done) {                  // no mass at all (non-finite input)
        a.out_token[b] = -1;
        a.resid_mass[b] = (float)(shard_total / (double)q.S);
        a.flags[b] = flags | OD_SF_ZERO_MASS;
    }
}

}  // namespace

// Dynamic shared memory of the kernel for rows of `ntiles` tiles: the tile values of pass 2.
size_t od_sample_smem_bytes(int32_t ntiles) { return (size_t)ntiles * 8; }

template <typename K>
static cudaError_t allow_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <int DTYPE, bool FUSED, int SOURCE>
static cudaError_t allow_cluster16(size_t bytes)
{
    cudaError_t e = allow_smem(od_sample_kernel<DTYPE, FUSED, SOURCE>, bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(od_sample_kernel<DTYPE, FUSED, SOURCE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}
template <int DTYPE>
static cudaError_t prepare_kernels()
{
    const size_t bytes = OD_SAMPLE_SMEM_MAX;
    const size_t staged = (size_t)(OD_SAMPLE_MAX_SLOTS + 1) * 4 + 8 * 1024;
    cudaError_t e = allow_cluster16<DTYPE, false, FROM_MAP>(bytes);
    if (e == cudaSuccess) e = allow_cluster16<DTYPE, true, FROM_MAP>(bytes);
    if (e == cudaSuccess) e = allow_cluster16<DTYPE, false, FROM_ROW>(bytes);
    if (e == cudaSuccess) e = allow_cluster16<DTYPE, true, FROM_ROW>(bytes);
    if (e == cudaSuccess) e = allow_cluster16<DTYPE, false, STAGED>(staged);
    if (e == cudaSuccess) e = allow_cluster16<DTYPE, true, STAGED>(staged);
    if (e == cudaSuccess) e = allow_smem(od_sample_shard_kernel<DTYPE, 1>, bytes);
    if (e == cudaSuccess) e = allow_smem(od_sample_shard_kernel<DTYPE, 2>, bytes);
    return e;
}

// Rows beyond 6144 tiles (and the staged probabilities) need more dynamic shared memory than a
// kernel gets by default, and clusters of 16 blocks are not portable: opt in, to the same limit in every
// context (it is the kernel's: a smaller one would take it from a context made earlier), and ask how many
// clusters of each size are resident at a time (0: the device has no room for one; the device must be
// current; allocates nothing).
cudaError_t od_sample_prepare_device(int32_t *clusters)
{
    cudaError_t e = prepare_kernels<OD_BF16>();
    if (e == cudaSuccess) e = prepare_kernels<OD_F32>();
    if (e != cudaSuccess) return e;
    for (int level = 0; level < OD_SAMPLE_LEVELS; ++level) {
        cudaLaunchConfig_t cfg = {};
        const unsigned parts = (unsigned)od_sample_parts(level);
        cfg.gridDim = dim3(parts); cfg.blockDim = dim3(CTHREADS); cfg.dynamicSmemBytes = 64 * 1024;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = parts; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, od_sample_kernel<OD_BF16, true, STAGED>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        clusters[level] = n;
    }
    return cudaSuccess;
}

template <int DTYPE>
static cudaError_t launch_step(const cudaLaunchConfig_t &cfg, const SampleArgs &a, bool fused, int source)
{
    if (source == STAGED)
        return fused ? cudaLaunchKernelEx(&cfg, od_sample_kernel<DTYPE, true, STAGED>, a)
                     : cudaLaunchKernelEx(&cfg, od_sample_kernel<DTYPE, false, STAGED>, a);
    if (source == FROM_ROW)
        return fused ? cudaLaunchKernelEx(&cfg, od_sample_kernel<DTYPE, true, FROM_ROW>, a)
                     : cudaLaunchKernelEx(&cfg, od_sample_kernel<DTYPE, false, FROM_ROW>, a);
    return fused ? cudaLaunchKernelEx(&cfg, od_sample_kernel<DTYPE, true, FROM_MAP>, a)
                 : cudaLaunchKernelEx(&cfg, od_sample_kernel<DTYPE, false, FROM_MAP>, a);
}

// mode 0: od_sample_residual; 1 / 2: the two calls of a vocabulary shard
static cudaError_t launch_sample(od_ctx *c, int mode, int32_t B, int32_t K_max, const void *logits,
                                 int32_t dtype, int64_t row_stride, int64_t seq_stride,
                                 const float *row_max, const float *row_sum, const float *q_rows,
                                 const int32_t *draft_ids, const int32_t *tgt_ids,
                                 const float *q_prime, const int32_t *span_start,
                                 const int32_t *span_len, const int32_t *m,
                                 const uint8_t *tail_kind, const int32_t *n_accepted,
                                 const float *temperature, const uint64_t *seed, uint64_t step,
                                 int32_t *out_token, float *resid_mass, uint32_t *flags,
                                 int32_t shard_lo, int32_t shard_len, int32_t n_shards, int32_t shard_index,
                                 const double *mass_all, double *mass_out, cudaStream_t s,
                                 const od_fused_verify *fuse = nullptr)
{
    if (B == 0) return cudaSuccess;
    const int ntiles = c->tiles_per_row;
    const int tile_lo = mode == 0 ? 0 : shard_lo / OD_SAMPLE_TILE;
    const int tile_hi = mode == 0 ? ntiles : (shard_lo + shard_len + OD_SAMPLE_TILE - 1) / OD_SAMPLE_TILE;
    const int wtiles = tile_hi - tile_lo;
    int64_t tpw = c->opt_sample_tiles_per_warp;
    int blocks_x = 1, level = 0, part_tiles = 0;
    if (mode == 0) {
        // Parts (blocks) per sequence: as many as still make one resident wave of clusters, and no more
        // than have a tile for every warp (19 sequences of 100277 ids, the three calls: 25.2 us with 4 parts, 23.3
        // with 8, 27.0 with 16, which is two waves); under the option, the fewest of a power of two that
        // keep to it. 3 and 6 are for batches that just miss 4 and 8 (device time of the step, 37 and 73
        // sequences of 128256 bf16 ids: 23.7 -> 23.0 and 35.1 -> 32.9 us, of 152064 fp32 ids 35.6 -> 33.8 and 58.5
        // -> 52.9), where they save a warp two tiles (else they only add blocks: 37 of 32000 ids 14.4 us with 6,
        // 14.1 with 4). 12 was slower than 8 (19 sequences: 20.9 us, 18.4): a large cluster waits long for its place.
        int most = OD_SAMPLE_LEVELS - 1;
        while (most > 0 && c->sample_clusters[most] <= 0) --most;
        for (int next = 1; next <= most; ++next) {
            const int32_t tiles = od_sample_part_tiles(c->v_p, level), parts = od_sample_parts(next);
            const bool doubling = (parts & (parts - 1)) == 0;
            if (tpw > 0) {
                if (doubling && tiles > tpw * CWARPS) level = next;
            } else {
                if (B > c->sample_clusters[next]) break;
                const int32_t then = od_sample_part_tiles(c->v_p, next);
                if (doubling ? tiles > CWARPS : (tiles + CWARPS - 1) / CWARPS >= (then + CWARPS - 1) / CWARPS + 2) level = next;
            }
        }
        // staged probabilities of over 100 KB would leave room for one block per multiprocessor
        while (level < most && !c->map_same_ids && c->sample_slots[level] * 4 > 100 * 1024) ++level;
        blocks_x = od_sample_parts(level);
        part_tiles = od_sample_part_tiles(c->v_p, level);
        tpw = (part_tiles + CWARPS - 1) / CWARPS;
    } else {
        if (tpw <= 0) {
            // one resident wave (four 256-thread blocks per SM) over the whole batch
            const int64_t want = (int64_t)c->sm_count * 4;
            int64_t per_row = want / B;
            if (per_row < 1) per_row = 1;
            tpw = (wtiles + per_row * WARPS - 1) / (per_row * WARPS);
            if (tpw < 1) tpw = 1;
        }
        const int64_t tiles_per_block = tpw * WARPS;
        if (mode == 1) blocks_x = (int)((wtiles + tiles_per_block - 1) / tiles_per_block);
    }
    SampleArgs a = {};
    a.logits = logits; a.row_stride = row_stride; a.seq_stride = seq_stride;
    a.B = B; a.K_max = K_max; a.v_p = mode == 0 ? c->v_p : shard_lo + shard_len; a.v_q = c->v_q;
    a.ntiles = ntiles; a.tiles_per_warp = (int32_t)tpw;
    a.row_max = row_max; a.row_sum = row_sum; a.q_rows = q_rows;
    a.draft_ids = draft_ids; a.tgt_ids = tgt_ids; a.q_prime = q_prime;
    a.span_start = span_start; a.span_len = span_len; a.m = m; a.tail_kind = tail_kind;
    a.n_accepted = n_accepted; a.temperature = temperature; a.seed = seed; a.step = step;
    a.vocab_map = c->d_vocab_map; a.inv_map = c->d_inv_map;
    a.part_tiles = part_tiles;
    a.map_serial = c->map_serial; a.map_serial_now = c->d_map_serial;
    a.same_ids = c->map_same_ids;
    a.row_vec = c->v_q % 4 == 0 && ((uintptr_t)q_rows & 15u) == 0;
    a.out_token = out_token; a.resid_mass = resid_mass; a.flags = flags;
    a.tile_val = c->d_tile_sums; a.ticket = c->d_samp_ticket;
    a.tile_lo = tile_lo; a.tile_hi = tile_hi; a.col0 = mode == 0 ? 0 : shard_lo;
    a.n_shards = n_shards; a.shard_index = shard_index; a.mass_all = mass_all; a.mass_out = mass_out;
    // the translation kernel releases its successor before it has written anything: directly
    // after it, nothing may be read early
    a.early = c->last_was_map ? 0 : 1;
    if (fuse) {
        a.plan.W = fuse->W; a.plan.n_chunks = fuse->n_chunks; a.plan.span_min = fuse->span_min;
        a.plan.span_a = fuse->span_a; a.plan.seg_warps = fuse->seg_warps; a.plan.partials = c->d_partials;
        a.w_row_max = fuse->row_max; a.w_row_sum = fuse->row_sum; a.w_p_sel = fuse->p_sel; a.w_ratio = fuse->ratio;
        a.w_n_accepted = fuse->n_accepted; a.w_n_draft = fuse->n_draft_accepted; a.w_vflags = fuse->flags;
    }
    c->last_was_map = false;
    if (mode != 2) {
        c->info[2] = (int64_t)blocks_x * B;
        c->info[3] = tpw;
    }

    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = c->opt_pdl ? attr : attr + 1;
    const bool bf = dtype == OD_BF16;
    if (mode == 0) {
        cfg.gridDim = dim3((unsigned)blocks_x, (unsigned)B);
        cfg.blockDim = dim3(CTHREADS);
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)blocks_x; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = c->opt_pdl ? 2 : 1;
        const int source = a.same_ids ? FROM_ROW
                                      : c->sample_slots[level] <= OD_SAMPLE_MAX_SLOTS && part_tiles <= 2048 ? STAGED : FROM_MAP;
        if (source == STAGED) {
            const OdSampleLists l = od_sample_lists(c->d_sample_lists, c->v_q, c->v_p);
            a.list_word = l.word + (size_t)level * l.groups * 32; a.list_base = l.base + (size_t)level * l.groups;
            a.list_part = l.part + level * OD_SAMPLE_MAX_PARTS * 4; a.octet = l.octet;
            a.slots = c->sample_slots[level] + 1;
        }
        cfg.dynamicSmemBytes = ((size_t)a.slots + (size_t)tpw * CWARPS) * sizeof(float);
        return bf ? launch_step<OD_BF16>(cfg, a, fuse != nullptr, source) : launch_step<OD_F32>(cfg, a, fuse != nullptr, source);
    }
    cfg.gridDim = dim3((unsigned)B, (unsigned)blocks_x);
    cfg.blockDim = dim3(OD_SAMPLE_THREADS);
    cfg.dynamicSmemBytes = od_sample_smem_bytes(ntiles);
    cfg.numAttrs = c->opt_pdl ? 1 : 0;
    if (mode == 1)
        return bf ? cudaLaunchKernelEx(&cfg, od_sample_shard_kernel<OD_BF16, 1>, a)
                  : cudaLaunchKernelEx(&cfg, od_sample_shard_kernel<OD_F32, 1>, a);
    return bf ? cudaLaunchKernelEx(&cfg, od_sample_shard_kernel<OD_BF16, 2>, a)
              : cudaLaunchKernelEx(&cfg, od_sample_shard_kernel<OD_F32, 2>, a);
}

cudaError_t od_launch_sample(od_ctx *c, int32_t B, int32_t K_max, const void *logits,
                             int32_t dtype, int64_t row_stride, int64_t seq_stride,
                             const float *row_max, const float *row_sum, const float *q_rows,
                             const int32_t *draft_ids, const int32_t *tgt_ids,
                             const float *q_prime, const int32_t *span_start,
                             const int32_t *span_len, const int32_t *m,
                             const uint8_t *tail_kind, const int32_t *n_accepted,
                             const float *temperature, const uint64_t *seed, uint64_t step,
                             int32_t *out_token, float *resid_mass, uint32_t *flags,
                             cudaStream_t s, const od_fused_verify *fuse)
{
    return launch_sample(c, 0, B, K_max, logits, dtype, row_stride, seq_stride, row_max, row_sum, q_rows,
                         draft_ids, tgt_ids, q_prime, span_start, span_len, m, tail_kind, n_accepted,
                         temperature, seed, step, out_token, resid_mass, flags, 0, 0, 1, 0, nullptr, nullptr, s,
                         fuse);
}

cudaError_t od_launch_sample_shard_mass(od_ctx *c, int32_t B, int32_t K_max, int32_t shard_lo,
                                        int32_t shard_len, const void *logits, int32_t dtype,
                                        int64_t row_stride, int64_t seq_stride, const float *row_max,
                                        const float *row_sum, const float *q_rows, const int32_t *draft_ids,
                                        const int32_t *tgt_ids, const float *q_prime,
                                        const int32_t *span_start, const int32_t *span_len, const int32_t *m,
                                        const uint8_t *tail_kind, const int32_t *n_accepted,
                                        const float *temperature, double *mass, cudaStream_t s)
{
    return launch_sample(c, 1, B, K_max, logits, dtype, row_stride, seq_stride, row_max, row_sum, q_rows,
                         draft_ids, tgt_ids, q_prime, span_start, span_len, m, tail_kind, n_accepted,
                         temperature, nullptr, 0, nullptr, nullptr, nullptr, shard_lo, shard_len, 1, 0,
                         nullptr, mass, s);
}

cudaError_t od_launch_sample_shard_pick(od_ctx *c, int32_t B, int32_t K_max, int32_t n_shards,
                                        int32_t shard_index, int32_t shard_lo, int32_t shard_len,
                                        const double *mass_all, const void *logits, int32_t dtype,
                                        int64_t row_stride, int64_t seq_stride, const float *row_max,
                                        const float *row_sum, const float *q_rows, const int32_t *draft_ids,
                                        const int32_t *tgt_ids, const float *q_prime,
                                        const int32_t *span_start, const int32_t *span_len, const int32_t *m,
                                        const uint8_t *tail_kind, const int32_t *n_accepted,
                                        const float *temperature, const uint64_t *seed, uint64_t step,
                                        int32_t *out_token, float *resid_mass, uint32_t *flags, cudaStream_t s)
{
    return launch_sample(c, 2, B, K_max, logits, dtype, row_stride, seq_stride, row_max, row_sum, q_rows,
                         draft_ids, tgt_ids, q_prime, span_start, span_len, m, tail_kind, n_accepted,
                         temperature, seed, step, out_token, resid_mass, flags, shard_lo, shard_len, n_shards,
                         shard_index, mass_all, nullptr, s);
}


// What the sampler knows about the vocabulary map, on the host, in the layout of od_sample_lists.
// slots: [levels] most mapped ids of a part.
void od_sample_plan(int32_t v_q, int32_t v_p, const OdMappedIds &mapped, int32_t serial, void *out, int32_t *slots)
{
    const OdSampleLists l = od_sample_lists(out, v_q, v_p);
    const int32_t total = (int32_t)mapped.target.size(), octets = (v_p + 7) / 8;
    for (int32_t o = 0; o < octets; ++o) l.octet[o] = 0u;
    for (int32_t t : mapped.target) l.octet[t >> 3] |= 1u << (t & 7);
    for (int32_t o = 0, rank = 0; o < octets; ++o) {
        const uint32_t mask = l.octet[o];
        l.octet[o] = (uint32_t)rank << 8 | mask;
        rank += __builtin_popcount(mask);
    }
    // the mapped ids in draft-id order
    std::vector<int32_t> rank_of((size_t)v_q, -1), draft((size_t)v_q + 1);
    for (int32_t r = 0; r < total; ++r) rank_of[mapped.draft[r]] = r;
    for (int32_t d = 0, n = 0; d < v_q; ++d) {
        draft[n] = d;
        n += rank_of[d] >= 0 ? 1 : 0;
    }
    std::vector<int32_t> rank((size_t)total), tile((size_t)total);
    for (int32_t i = 0; i < total; ++i) {
        rank[i] = rank_of[draft[i]];
        tile[i] = mapped.target[rank[i]] / OD_SAMPLE_TILE;
    }
    std::vector<uint8_t> part_of((size_t)(v_p + OD_SAMPLE_TILE - 1) / OD_SAMPLE_TILE);
    for (int level = 0; level < OD_SAMPLE_LEVELS; ++level) {
        const int32_t parts = od_sample_parts(level), tiles = od_sample_part_tiles(v_p, level);
        for (size_t t = 0; t < part_of.size(); ++t) part_of[t] = (uint8_t)((int32_t)t / tiles);
        const auto rank_at = [&](int32_t part) {             // of the first mapped id of a part
            const int64_t t = (int64_t)part * tiles * OD_SAMPLE_TILE;
            return t < v_p ? (int32_t)(l.octet[t >> 3] >> 8) : total;
        };
        uint32_t *words = l.word + (size_t)level * l.groups * 32, *next[OD_SAMPLE_MAX_PARTS];   // a part's next entry
        int32_t *bases = l.base + (size_t)level * l.groups, rank0[OD_SAMPLE_MAX_PARTS], group = 0;
        slots[level] = 0;
        for (int32_t k = 0; k < parts; ++k) {
            const int32_t n = rank_at(k + 1) - (rank0[k] = rank_at(k));
            int32_t *p = l.part + (level * OD_SAMPLE_MAX_PARTS + k) * 4;
            p[0] = p[1] = group; p[2] = rank0[k]; p[3] = serial;
            next[k] = words + (size_t)group * 32;
            group += (n + 31) / 32 + v_q / 65536;
            if (n > slots[level]) slots[level] = n;
        }
        // a part's entries in draft-id order; groups end with 65536 draft ids, of which the first is their base
        for (int32_t i = 0, page = 0; page < v_q; page += 65536) {
            // (a part of more than OD_SAMPLE_MAX_SLOTS ids is not staged: the cut of its ranks does not matter)
            for (; i < total && draft[i] - page < 65536; ++i) {
                const int32_t k = part_of[tile[i]];
                *next[k]++ = (uint32_t)(draft[i] - page) << 16 | (uint32_t)((rank[i] - rank0[k]) & 0xFFFF);
            }
            for (int32_t k = 0; k < parts; ++k) od_end_group(words, next[k], bases, page, l.part[(level * OD_SAMPLE_MAX_PARTS + k) * 4 + 1]);
        }
    }
}
