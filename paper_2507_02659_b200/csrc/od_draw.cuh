// The extra token of one sequence (see od_sample.cu): the device code that the sampler's kernels and the
// whole step in one launch (od_step.cu) share.
#pragma once

#include <float.h>

#include "od_common.cuh"
#include "od_decide.cuh"

namespace {

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
// The same, and the sum of the warp's. With fp32 rows the tile loop spills by it, so it is kept in shared memory (a rank's
// mass of 256 sequences, half of 152064 ids, in registers and in shared memory: fp32 28.8 and 27.3 us, bf16 23.4 and 24.6).
template <int DTYPE>
struct SummedTiles {
    double *val, *s_sum;                                    // s_sum: two of the warp's own (fp32)
    int lane;
    double total;                                           // (bf16) lanes 0..15 and 16..31 each hold a share
    __device__ __forceinline__ void clear()
    {
        total = 0.0;
        if (DTYPE == OD_BF16) return;
        __syncwarp();
        if (lane < 2) s_sum[lane] = 0.0;
        __syncwarp();
    }
    __device__ __forceinline__ void one(int t, float v)
    {
        if (lane == 0) val[t] = (double)v;
        v = fmaxf(0.f, v);                                  // (a tile with NaN has no mass)
        if (DTYPE == OD_BF16) {
            if (lane < 16) total += (double)v;
        } else if (lane == 0) {
            s_sum[0] += (double)v;
        }
    }
    __device__ __forceinline__ void pair(int t, float v, bool two)
    {
        if (DTYPE == OD_BF16) total += lane < 16 || two ? (double)fmaxf(0.f, v) : 0.0;
        if ((lane & 15) != 0 || (lane != 0 && !two)) return;
        val[t + (lane >> 4)] = (double)v;
        if (DTYPE != OD_BF16) s_sum[lane >> 4] += (double)fmaxf(0.f, v);
    }
    __device__ __forceinline__ double sum() const
    {
        if (DTYPE == OD_BF16) return __shfl_sync(0xFFFFFFFFu, total, 0) + __shfl_sync(0xFFFFFFFFu, total, 16);
        __syncwarp();
        return s_sum[0] + s_sum[1];
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
    // tile t's value is another; then, with all tiles as they stay, the sum of the run's first n anew, in the order of the
    // pass: correcting it by the difference would lose what is small beside the old value (and give NaN where that is infinite)
    __device__ __forceinline__ void replace(int t, float v)
    {
        __syncwarp();
        if (lane == 0) val[t - t_lo] = fmaxf(0.f, v);
    }
    __device__ __forceinline__ void sum_anew(int n)
    {
        __syncwarp();
        total = 0.0;
#pragma unroll 1                                            // (unrolled by eight: 0.8 % of the step of 296, in the pass's registers)
        for (int i = lane >> 4; i < n; i += 2) total += (double)val[i];
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
    // (fp32 rows through L1, where the draw finds its tile again: the step of 19 sequences of 100277 ids 14.8 -> 14.3 us, 148
    // 46.3 -> 43.9, 296 86.0 -> 79.1, 512 162 -> 148; of 32000 shared ids 100 19.6 -> 19.0, 512 64.1 -> 63.8. Only 296 of 65000 shared ids,
    // one block to each and a whole chip of them, lose: 59.1 -> 60.5. bf16 rows gain nothing by it, a batch of 296 loses 2.5 %)
    if (DTYPE == OD_BF16) {
        raw[0] = ld_once(src);
    } else {
        raw[0] = __ldg(src); raw[RAW<DTYPE> - 1] = __ldg(src + 1);
    }
}
// A lane's eight ids of a whole tile: the sum of their residuals, or of e alone. A tile is 256
// ids of work for one warp, and its instructions bound a large batch: 276 a tile and 66.8 us for
// 296 staged rows of 152064 ids with a branch per id, 195 and 51.9 us with a select per id,
// 154 and 44.8 us with an unmapped id's multiply-add predicated off and Eq. (2)'s two ids looked for in every tile. Now
// those tiles are evaluated once more behind the pass (a test less in each tile), and the staging does without a base
// for each group of its list: the step of 296 such rows 89.9 -> 87.4 us, 512 with eight tokens 271.4 -> 266.8, 64 of 128256 ids
// 28.65 -> 28.1, 100 of 90001 fp32 ids 43.0 -> 41.8. (The clamp at zero as the multiply-add's own .sat is 0.8 % of
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
__device__ __forceinline__ float tile_lane_sum_staged(const SeqState &q, const uint4 *raw, uint32_t oct, uint32_t rank_at)
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
    return sum_of_eight(r);
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
            return tile_lane_sum_staged<DTYPE>(q, raw, oct, (uint32_t)__cvta_generic_to_shared(sr.q) + ((oct >> 8) - sr.rank0) * 4u);
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
// LONE: many warps have one tile alone (the step in one launch), and do not work on it twice.
template <int DTYPE, int SOURCE, bool LONE, typename Sink>
__device__ __forceinline__ void warp_tiles_ahead(const SeqState &q, const SampleArgs &a, const StagedRow &sr, int t_lo, int t_hi,
                                                 int lane, Sink &out, TileLoads<DTYPE, SOURCE> (&cur)[SOURCE == FROM_ROW ? 1 : 2])
{
#pragma unroll 1
    for (int t = t_lo; t < t_hi; t += 2) {
        const bool two = t + 1 < t_hi;
        float s0, s1;
        if (SOURCE == FROM_ROW) {
            TileLoads<DTYPE, SOURCE> nx;
            if (!LONE || two) nx.load(q, a, two ? t + 1 : t, lane);
            s0 = cur[0].sum(q, a, sr, t, lane);
            if (t + 2 < t_hi) cur[0].load(q, a, t + 2, lane);
            s1 = !LONE || two ? nx.sum(q, a, sr, t + 1, lane) : 0.f;
        } else {
            TileLoads<DTYPE, SOURCE> nx[2];
            if (t + 2 < t_hi) {
                nx[0].load(q, a, t + 2, lane);
                nx[1].load(q, a, min(t + 3, t_hi - 1), lane);
            }
            s0 = cur[0].sum(q, a, sr, t, lane);
            s1 = !LONE || two ? cur[SOURCE == FROM_ROW ? 0 : 1].sum(q, a, sr, t + 1, lane) : 0.f;
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

// ---- what both kernels prepare and decide alike -------------------------------------------

// What a block can load before the verification kernels have finished: what the translation
// kernel wrote, for every position the step can stop at. Lane k of every warp prepares
// position k. Two memory round trips, not a chain of four: everything that is addressed by
// (b, lane) alone is requested at once, whether or not it will be used (lane < K keeps the
// addresses inside the arrays); what is addressed by those values comes second.
struct Ahead {
    int mb;
    bool stop;
    float T, scale;                     // scale: log2(e) / T
    float u_draw;                       // the uniform of a draw at position `lane` (where it was worked out ahead)
    int32_t l_len, l_tgt;               // piece `lane`: its length, target id
    float l_qp;                         // and q'
    int32_t s0, len, tgt, d1, pm;       // position `lane`: row of the drafter, length of the piece there (1 at a stop);
    float qp, qd1;                      // of a merged piece: target, q', first sub-token, its image and probability
};
// position `lane` from its piece: s0 its first draft token's position, d1 that token's id
__device__ __forceinline__ void prepare_positions(const SampleArgs &a, Ahead &h, int b, int lane, int s0, int32_t d1)
{
    const int K = a.K_max;
    h.s0 = 0; h.len = 1; h.tgt = -1; h.d1 = -1; h.pm = -1; h.qp = 0.f;
    if (lane < K && lane <= h.mb) {
        h.s0 = s0;
        h.len = lane < h.mb ? h.l_len : 1;
    }
    if (h.len >= 2) {
        h.tgt = h.l_tgt;
        h.qp = h.l_qp;
        if (d1 >= 0 && d1 < a.v_q) {
            h.d1 = d1;
            h.pm = __ldg(a.vocab_map + d1);
        }
    }
}
// Its probability, from the drafter's row. The rows are the first thing of the caller's that a draw alone reads: whatever
// is directly in front of it may write them, so the load is behind griddepcontrol.wait. What is requested in front of it
// is the line, for L2, where such a writer's stores arrive too: then the load is back with those of the rows' statistics
// (device time of the three calls: 4 sequences of 128256 ids 16.2 us without the request, 16.0 with it, 19 of 100277 22.1,
// 22.0, 64 32.5, 32.4; a rank's five calls on a quarter of 128256 ids 26.4, 26.45: the shards' kernels do without).
__device__ __forceinline__ const float *first_probability(const SampleArgs &a, const Ahead &h, int b)
{
    return a.q_rows + ((size_t)b * a.K_max + h.s0) * a.v_q + h.d1;
}
__device__ __forceinline__ void request_first_probability(const SampleArgs &a, const Ahead &h, int b)
{
    if (h.d1 >= 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(first_probability(a, h, b)));
}
__device__ __forceinline__ void load_first_probability(const SampleArgs &a, Ahead &h, int b)
{
    h.qd1 = h.d1 >= 0 ? __ldg(first_probability(a, h, b)) : 0.f;
}
__device__ __forceinline__ Ahead load_ahead(const SampleArgs &a, int b, int lane)
{
    const int K = a.K_max;
    Ahead h;
    int mb = a.m[b];
    h.stop = a.tail_kind[b] == OD_TAIL_UNMAPPED_STOP;
    h.T = a.temperature[b];
    h.scale = 1.4426950408889634f / h.T;
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
    const int s0 = l_s0 < 0 ? 0 : (l_s0 >= K ? K - 1 : l_s0);
    prepare_positions(a, h, b, lane, s0, __shfl_sync(0xFFFFFFFFu, l_did, lane < K && lane <= h.mb ? s0 : 0));
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
    q.scale = h.scale;
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
template <int DTYPE, int SOURCE, bool LONE, typename Sink>
__device__ __forceinline__ void warp_run(const SeqState &q, const SampleArgs &a, int t_lo, int t_hi, int hi_w, int lane,
                                         Sink &out, int4 (&ni)[2][2])
{
    const StagedRow none = {};
    if (t_lo >= t_hi) return;
    if (!q.residual) {
        TileLoads<DTYPE, FREE> cur[2];
        first_tiles<DTYPE, FREE>(q, a, t_lo, hi_w, lane, cur);
        warp_tiles_ahead<DTYPE, FREE, LONE>(q, a, none, t_lo, hi_w, lane, out, cur);
    } else if (SOURCE == FROM_ROW) {
        TileLoads<DTYPE, FROM_ROW> cur[1];
        first_tiles<DTYPE, FROM_ROW>(q, a, t_lo, hi_w, lane, cur);
        warp_tiles_ahead<DTYPE, FROM_ROW, LONE>(q, a, none, t_lo, hi_w, lane, out, cur);
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
    const int pick = __reduce_min_sync(0xFFFFFFFFu, my_pick), last = __reduce_max_sync(0xFFFFFFFFu, my_last);
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
// A block costs about 10 us whatever its share of the tiles (512 sequences with 1, 2, 4 parts: 270, 278, 308 us), and every
// warp of it goes through the same chain, so its instructions count sixteen times: integer sums and
// minima in one instruction, the draw's uniform for every position ahead of the wait, the divisions that find a row's
// partials too, no second tile for a warp with one: 256 of 32000 34.7 -> 33.8, 64 of 128256 28.1 -> 27.5, one of 32000 fp32 8.66 -> 8.3.
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

// ---- one block's part of a sequence ------------------------------------------------------

// What a block knows before anything of the step: the tiles of this warp, the inverse-map entries of their
// first pair (FROM_MAP), the first entries of the part's list (STAGED). All of it belongs to the context.
template <int SOURCE>
struct Part {
    static constexpr int EB = 6;                            // groups of the list per warp and batch
    int p_lo, p_hi, p_hi_w;
    int4 ni[2][2];
    uint32_t word[EB];
    int4 list;
    int g_at;                                               // the group of word[0]
    __device__ __forceinline__ void load_words(const SampleArgs &a, int lane)
    {
#pragma unroll
        for (int e = 0; e < EB; ++e)
            word[e] = g_at + e * CWARPS < list.y ? __ldg(a.list_word + (size_t)(g_at + e * CWARPS) * 32 + lane) : 0xFFFFu;
    }
    __device__ __forceinline__ void prepare(const SampleArgs &a, int part, int warp, int lane)
    {
        p_hi = min((part + 1) * a.part_tiles, a.ntiles);
        p_lo = min(part * a.part_tiles + warp * a.tiles_per_warp, p_hi);
        p_hi = min(p_lo + a.tiles_per_warp, p_hi);
        p_hi_w = min(p_hi, a.v_p / OD_SAMPLE_TILE);
        if (SOURCE == FROM_MAP && p_lo < p_hi_w) first_pair_entries(a, p_lo, p_hi_w, lane, ni);
        list = make_int4(0, 0, 0, 0);
        g_at = 0;
        if (SOURCE == STAGED) {
            list = __ldg((const int4 *)a.list_part + part);
            if (list.w != a.map_serial) { list.y = 0; p_hi_w = p_lo; }   // another map: nothing is staged, all is looked up
            g_at = list.x + warp;
            load_words(a, lane);
        }
    }
};

// Step 2's decisions from the rows' statistics (rm, rs: lane k holds row k's; the other inputs position k's),
// by every warp of every block of a sequence alike: the accepted pieces. `store`: this warp writes step 2's
// per-position and per-sequence outputs.
__device__ __forceinline__ int decide(const SampleArgs &a, const Ahead &h, int b, int lane, float rm, float rs, bool t_ok,
                                      float x_t, float u, unsigned int vbits, bool store)
{
    const int K = a.K_max, mb = h.mb;
    const bool bad_T = !(h.T > 0.f);
    bool acc = false, bnd = false;
    Acceptance d = {};
    if (lane < mb) {
        d = accept_position(rm, rs, bad_T ? 0.f : h.scale, t_ok, x_t, h.l_qp, u);
        acc = d.accept; bnd = d.boundary;
    }
    const unsigned int accmask = __ballot_sync(0xFFFFFFFFu, acc);
    const int j = bad_T ? 0 : __ffs((int)~accmask) - 1;     // (no position beyond mb <= OD_MAX_K is accepted)
    if (store) {
        if (lane < mb) { a.w_p_sel[(size_t)b * K + lane] = d.p; a.w_ratio[(size_t)b * K + lane] = d.ratio; }
        const unsigned int bndmask = __ballot_sync(0xFFFFFFFFu, bnd);
        const int nd = __reduce_add_sync(0xFFFFFFFFu, lane < j ? h.l_len : 0);
        if (lane == 0) {
            uint32_t f = bndmask & OD_VF_BOUNDARY_MASK;
            if (vbits & 1u) f |= OD_VF_NONFINITE;
            if (bad_T) f |= OD_VF_BAD_TEMPERATURE;
            a.w_n_accepted[b] = j; a.w_n_draft[b] = nd; a.w_vflags[b] = f;
        }
    }
    return j;
}

// The draw at position j by the cluster of a sequence (every thread calls). STARTED: the cluster has met at
// a barrier already, so every block of it runs; else the caller has arrived (relaxed) at the first one.
// AHEAD: h.u_draw is there.
template <int DTYPE, int SOURCE, bool STARTED, bool AHEAD>
__device__ __forceinline__ void draw(const SampleArgs &a, const Ahead &h, Part<SOURCE> &my, int b, unsigned part, unsigned nparts,
                                     int warp, int lane, int j, float rm, float rs, bool planned, float *s_q, float *s_val)
{
    __shared__ int s_bare;
    __shared__ double s_run[CWARPS], s_part[OD_SAMPLE_MAX_PARTS];   // sums of the block's runs, of the cluster's blocks
    constexpr int EB = Part<SOURCE>::EB;
    if (threadIdx.x == 0) s_bare = 0;
    const int p_lo = my.p_lo, p_hi = my.p_hi;
    const SeqState q = seq_state<DTYPE>(a, h, b, j, rm, rs, 0, planned);
    if (SOURCE == FROM_MAP && q.residual && threadIdx.x == 0) prefetch_q_row(a, q, part, nparts);

    // ---- pass 1: the value of every tile; the ragged last one (all of them, if the map is another) one by one ----
    WarpTiles out = {s_val, lane, p_lo, 0.0};
    const int hi_w = planned ? my.p_hi_w : p_lo;
    const uint64_t seed_b = AHEAD ? 0ull : a.seed[b];
    const StagedRow sr = {s_q, a.octet, (uint32_t)my.list.z};
    if (SOURCE == STAGED && q.residual) {
        TileLoads<DTYPE, STAGED> cur[2];
        first_tiles<DTYPE, STAGED>(q, a, p_lo, hi_w, lane, cur);
        // the part's probabilities, gathered in draft-id order, to their ranks in shared memory
        for (;;) {
            float x[EB];
            uint32_t at[EB];
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                at[e] = my.word[e] & 0xFFFFu;
                if (at[e] == 0xFFFFu) continue;
                const float *from = q.q_row + (my.word[e] >> 16);
                if (a.v_q > 65536) from += __ldg(a.list_base + my.g_at + e * CWARPS);   // (else there is one page of draft ids)
                x[e] = __ldg(from);
            }
            my.g_at += EB * CWARPS;
            const bool more = my.g_at < my.list.y;             // the same for every lane of a warp
            if (more) my.load_words(a, lane);
#pragma unroll
            for (int e = 0; e < EB; ++e)
                if (at[e] != 0xFFFFu) s_q[at[e]] = x[e];
            if (!more) break;
        }
        __syncthreads();
        warp_tiles_ahead<DTYPE, STAGED, STARTED>(q, a, sr, p_lo, hi_w, lane, out, cur);
        // Eq. (2)'s two ids, which the pass above does not look for: their tiles once more
        bool other = false;
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            const int id = i == 0 ? q.prefix_token : q.ngram_token, t = id / OD_SAMPLE_TILE;
            if (id < 0 || t < p_lo || t >= hi_w) continue;
            float r[EPT];
            tile_values<DTYPE>(q, a, true, t, lane, r, &sr);
            out.replace(t, warp_sum_f32(sum_of_eight(r)));
            other = true;
        }
        if (other) out.sum_anew(hi_w - p_lo);
        if (hi_w < p_hi) warp_tiles_dense<DTYPE, 1>(q, a, true, max(hi_w, p_lo), p_hi, lane, out);
    } else {
        warp_run<DTYPE, SOURCE, STARTED>(q, a, p_lo, p_hi, hi_w, lane, out, my.ni);
    }
    const float u = AHEAD ? __shfl_sync(0xFFFFFFFFu, h.u_draw, j) : od_uniform(seed_b, a.step, (uint32_t)j, 1u);

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
    // one block to a sequence has nothing to exchange (256 sequences of 32000 ids 33.9 -> 33.4 us; in the staged kernels the
    // branch costs registers and 1.5 % of a step of 64)
    const bool alone = SOURCE == FROM_ROW && !STARTED && nparts == 1;
    if (!alone) {
        if (!STARTED) od_cluster_wait();
        if (warp == 0 && lane < (int)nparts) od_cluster_store(&s_part[part], (uint32_t)lane, block_sum);
        od_cluster_arrive();
        od_cluster_wait();
    }

    // ---- every warp scans the blocks' sums: is the draw in its block, in its run?
    const uint32_t flags = q.residual ? 0u : OD_SF_BONUS;
    const double p_sum = (lane & 15) < (int)nparts ? alone ? block_sum : s_part[lane & 15] : 0.0;
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
                                                                 SOURCE == STAGED && my.list.y ? &sr : nullptr);
            if (lane == 0 && !drawn) s_bare = 1;             // the tile holds no mass after all
        }
        __syncthreads();
        bare = s_bare;
    } else if (part != 0) {
        return;
    }
    if (bare) draw_from_p<DTYPE>(q, a, b, u, flags | OD_SF_ZERO_MASS);
}

// ---- host: how many blocks draw for one of B sequences, and what a launch of that many is told ----

// clusters of `parts` blocks that are resident at a time (0: the device has no room for one)
template <typename Kern>
int resident_clusters(Kern kern, int parts, size_t smem, int threads = CTHREADS)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)parts); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)parts; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess) return n;
    cudaGetLastError();
    return 0;
}

inline int draw_level(const od_ctx *c, int32_t B)
{
    const int64_t tpw = c->opt_sample_tiles_per_warp;
    int level = 0;
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
        if (parts == 5) continue;                           // (od_step.cu's)
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
    for (int next = level + 1; next <= most && !c->map_same_ids && c->sample_slots[level] * 4 > 100 * 1024; ++next)
        if (od_sample_parts(next) != 5) level = next;
    return level;
}

// of the context: its maps, its scratch
inline void context_args(const od_ctx *c, SampleArgs &a)
{
    a.v_q = c->v_q; a.ntiles = c->tiles_per_row;
    a.vocab_map = c->d_vocab_map; a.inv_map = c->d_inv_map;
    a.map_serial = c->map_serial; a.map_serial_now = c->d_map_serial;
    a.same_ids = c->map_same_ids;
    a.row_vec = c->v_q % 4 == 0 && ((uintptr_t)a.q_rows & 15u) == 0;
    a.tile_val = c->d_tile_sums;
}

// the cut of a row into the level's parts, and the level's lists
struct DrawPlan {
    int source;
    size_t smem;                        // dynamic shared memory
};
inline DrawPlan plan_draw(const od_ctx *c, int level, SampleArgs &a)
{
    DrawPlan p;
    a.part_tiles = od_sample_part_tiles(c->v_p, level);
    a.tiles_per_warp = (a.part_tiles + CWARPS - 1) / CWARPS;
    p.source = a.same_ids ? FROM_ROW
                          : c->sample_slots[level] <= OD_SAMPLE_MAX_SLOTS && a.part_tiles <= 2048 ? STAGED : FROM_MAP;
    if (p.source == STAGED) {
        const OdSampleLists l = od_sample_lists(c->d_sample_lists, c->v_q, c->v_p);
        a.list_word = l.word + (size_t)level * l.groups * 32; a.list_base = l.base + (size_t)level * l.groups;
        a.list_part = l.part + level * OD_SAMPLE_MAX_PARTS * 4; a.octet = l.octet;
        a.slots = c->sample_slots[level] + 1;
    }
    p.smem = ((size_t)a.slots + (size_t)a.tiles_per_warp * CWARPS) * sizeof(float);
    return p;
}

}  // namespace
