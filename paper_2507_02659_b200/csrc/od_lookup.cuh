// Lookups in the n-gram table: what the translation kernel and the whole step in one launch share.
#pragma once

#include "od_common.cuh"

namespace {

// Resolves a lookup whose first group g is already loaded (keys in k_lane, values in
// v_lane): the slot that holds `key` and its value, or -1. Walks at most ngroups groups,
// so it ends on any table contents.
__device__ __forceinline__ int32_t probe_continue(const uint64_t *__restrict__ keys, const int32_t *__restrict__ vals,
                                                  uint64_t ngroups, uint64_t key, uint64_t g,
                                                  uint64_t k_lane, int32_t v_lane, int lane, int32_t *value)
{
    for (uint64_t step = 0; step < ngroups; ++step) {
        unsigned match = __ballot_sync(0xFFFFFFFFu, k_lane == key);
        if (match) {
            const int src = __ffs(match) - 1;
            *value = __shfl_sync(0xFFFFFFFFu, v_lane, src);
            return (int32_t)(g * OD_GROUP + src);
        }
        unsigned empty = __ballot_sync(0xFFFFFFFFu, k_lane == 0ULL);
        if (empty) return -1;
        g = (g + 1) & (ngroups - 1);
        k_lane = __ldg(keys + g * OD_GROUP + lane);
        v_lane = __ldcg(vals + g * OD_GROUP + lane);
    }
    return -1;
}

// One warp looks up the runs of 2, 3 and 4 ids that begin at offset s of a proposal of K ids (id_at(i), which
// every lane calls): the target and the table slot of each, or -1.
template <typename IdAt>
__device__ __forceinline__ void probe_offset(IdAt id_at, int s, int K, int32_t v_q, const uint64_t *__restrict__ keys,
                                             const int32_t *__restrict__ vals, int64_t cap, int lane,
                                             int32_t (&hit)[OD_NGRAM_MAX + 1], int32_t (&slot)[OD_NGRAM_MAX + 1])
{
#pragma unroll
    for (int L = 0; L <= OD_NGRAM_MAX; ++L) hit[L] = slot[L] = -1;
    if (cap > 0) {
        const uint64_t ngroups = (uint64_t)cap / OD_GROUP;
        uint64_t key[OD_NGRAM_MAX + 1], grp[OD_NGRAM_MAX + 1], kl[OD_NGRAM_MAX + 1];
        int32_t vl[OD_NGRAM_MAX + 1];
        bool valid[OD_NGRAM_MAX + 1];
        // ids of a run must lie in the draft vocabulary; the run must fit
        bool ok = true;
        uint64_t k = 0;
#pragma unroll
        for (int L = 1; L <= OD_NGRAM_MAX; ++L) {
            int32_t id = (s + L - 1 < K) ? id_at(s + L - 1) : -1;
            ok = ok && (s + L <= K) && id >= 0 && id < v_q;
            k |= (uint64_t)(uint32_t)(id + 1) << (16 * (L - 1));
            valid[L] = ok && L >= 2;
            key[L] = k;
            grp[L] = od_hash64(k) & (ngroups - 1);
        }
#pragma unroll
        for (int L = 2; L <= OD_NGRAM_MAX; ++L) {
            kl[L] = valid[L] ? __ldg(keys + grp[L] * OD_GROUP + lane) : 0ULL;
            // the values of the group come with its keys, so a hit costs one round trip
            // (a concurrent batch insert writes an entry's value last: read it past L1)
            vl[L] = valid[L] ? __ldcg(vals + grp[L] * OD_GROUP + lane) : -1;
        }
#pragma unroll
        for (int L = 2; L <= OD_NGRAM_MAX; ++L)
            if (valid[L]) {
                int32_t value = -1;
                slot[L] = probe_continue(keys, vals, ngroups, key[L], grp[L], kl[L], vl[L], lane, &value);
                // an entry whose value is not set yet does not exist
                if (slot[L] >= 0) hit[L] = value;
            }
    }
}

// The piece of the proposal that begins at offset s, by one warp: the longest cached run, else the direct map.
// Lane k holds position k's id and probability. (length, 0 without either; target id; table slot or -1; bits of q')
__device__ __forceinline__ int4 look_up_piece(int32_t id, float q, int s, int K, int32_t v_q, const int32_t *__restrict__ vocab_map,
                                              const uint64_t *__restrict__ keys, const int32_t *__restrict__ vals, int64_t cap, int lane)
{
    const int32_t here = __shfl_sync(0xFFFFFFFFu, id, s);
    const int32_t direct = here >= 0 && here < v_q ? __ldg(vocab_map + here) : -1;
    int32_t hit[OD_NGRAM_MAX + 1], slot[OD_NGRAM_MAX + 1];
    probe_offset([&](int i) { return __shfl_sync(0xFFFFFFFFu, id, i); }, s, K, v_q, keys, vals, cap, lane, hit, slot);
    float prod = __shfl_sync(0xFFFFFFFFu, q, s);
    int4 piece = make_int4(direct >= 0 ? 1 : 0, direct, -1, __float_as_int(prod));
#pragma unroll
    for (int L = 2; L <= OD_NGRAM_MAX; ++L) {
        prod *= __shfl_sync(0xFFFFFFFFu, q, min(s + L - 1, 31));
        if (hit[L] >= 0) piece = make_int4(L, hit[L], slot[L], __float_as_int(prod));
    }
    return piece;
}

// The left-to-right walk, by one warp whose lane k holds the piece at offset k: m pieces, lane k's from draft
// position `start`; stopped: at a token without a piece, position `start` of lane m.
struct Walk {
    int m, start;
    bool stopped;
    int32_t len, tgt, slot, first_id;   // lane k's piece, and the id of its first token
    float q;
};
__device__ __forceinline__ Walk walk_proposal(int4 piece, int32_t id, int K, int lane)
{
    Walk w;
    int pos = 0;
    w.m = 0; w.start = 0;
    while (pos < K) {
        if (lane == w.m) w.start = pos;
        const int L = __shfl_sync(0xFFFFFFFFu, piece.x, pos);
        if (L == 0) break;
        ++w.m; pos += L;
    }
    w.stopped = pos < K;
    w.len = __shfl_sync(0xFFFFFFFFu, piece.x, w.start);
    w.tgt = __shfl_sync(0xFFFFFFFFu, piece.y, w.start);
    w.slot = __shfl_sync(0xFFFFFFFFu, piece.z, w.start);
    w.q = __int_as_float(__shfl_sync(0xFFFFFFFFu, piece.w, w.start));
    w.first_id = __shfl_sync(0xFFFFFFFFu, id, w.start);
    return w;
}

// Where the translation of one sequence goes; one warp writes it.
struct MapOut {
    int32_t *tgt_ids, *span_start, *span_len, *m;
    float *q_prime;
    uint8_t *tail_kind;
    uint32_t *counters, *stamp, *freq, clock;
};
__device__ __forceinline__ void store_walk(const MapOut &out, const Walk &w, int b, int K_max, int32_t v_q, int lane)
{
    const size_t o = (size_t)b * K_max + lane;
    if (lane < w.m) {
        out.tgt_ids[o] = w.tgt; out.q_prime[o] = w.q;
        out.span_start[o] = w.start; out.span_len[o] = w.len;
        if (out.stamp && w.slot >= 0) {                     // an access: recency and frequency of the entry
            atomicMax(out.stamp + w.slot, out.clock);
            atomicAdd(out.freq + w.slot, 1u);
        }
    } else if (lane == w.m && w.stopped) {
        out.span_start[o] = w.start; out.span_len[o] = 1;
    }
    const unsigned hits = __popc(__ballot_sync(0xFFFFFFFFu, lane < w.m && w.len >= 2));
    const int32_t stop_id = __shfl_sync(0xFFFFFFFFu, w.first_id, w.m & 31);
    if (lane != 0) return;
    out.m[b] = w.m;
    out.tail_kind[b] = w.stopped ? OD_TAIL_UNMAPPED_STOP : OD_TAIL_COMPLETE;
    if (!out.counters) return;
    if (hits) atomicAdd(out.counters + OD_CNT_CACHE_HITS, hits);
    if (w.stopped) atomicAdd(out.counters + OD_CNT_UNMAPPED_STOPS, 1u);
    if (w.stopped && (stop_id < 0 || stop_id >= v_q)) atomicAdd(out.counters + OD_CNT_INVALID_IDS, 1u);
    if (w.m) atomicAdd(out.counters + OD_CNT_MAPPED_TOKENS, (uint32_t)w.m);
}

inline MapOut map_out(const od_ctx *c, int32_t *tgt_ids, float *q_prime, int32_t *span_start, int32_t *span_len, int32_t *m,
                      uint8_t *tail_kind, uint32_t *counters)
{
    return MapOut{tgt_ids, span_start, span_len, m, q_prime, tail_kind, counters,
                  c->dyn ? c->d_stamp : nullptr, c->dyn ? c->d_freq : nullptr, c->clock};
}

}  // namespace
