// Online n-gram cache: insertion of unseen n-grams (Algorithm 1, cache-update line)
// and bounded size with LRU / LFU eviction (App. D.5, cache scalability).
//
// The table is the open-addressing table od_map_proposals probes (groups of 32
// slots), with three more words per slot: clock of the last access, access
// frequency, clock of insertion. Nothing is ever deleted in place, so lookups stay
// lock-free and simple; eviction rebuilds the table.
//   insert  one thread per candidate claims the first empty slot of its probe
//           sequence with a compare-and-swap on the key; candidates of one batch
//           that carry the same run settle on the one with the lowest index
//           (atomicMin on a claim word) and that one writes the value last, so a
//           concurrent or later lookup sees either nothing or the whole entry, and
//           the result does not depend on thread timing.
//   trim    with k = size - max_entries > 0 entries too many, the k entries that
//           come first in the order (inserted at the current clock?, score, run key)
//           are dropped, score = last-access clock (LRU) or frequency (LFU). A first
//           pass counts the entries by score, in 256 bins (trim_count_kernel); that
//           says for almost every entry whether it stays: a second pass copies those
//           that do straight into their own group of the spare table (trim_split_kernel)
//           and lists the entries of the one bin in which the k-th falls. The k-th of
//           those is found by a most-significant-digit radix select over the 104-bit order
//           key, by one cluster of blocks (trim_select_kernel). Tables too large for that take
//           a chain of 13 histogram launches: a pass copies the entries that still match
//           the decided prefix into the next list whenever that at least halves it, every
//           block works out the digit the pass before it decided from that pass's 256-bin
//           histogram, and a digit of (new?, score) that is the same in every listed entry
//           costs no histogram. Then the rest of the survivors go from the list into the
//           spare table (by that cluster, or trim_place_kernel), which becomes the table. No kernel waits for another.
#include <algorithm>
#include <stddef.h>
#include <string.h>
#include <utility>
#include <vector>

#include "od_common.cuh"

namespace {

constexpr int PASSES = 13;      // 5 bytes of (new?, score), 8 bytes of the run key

// What is known at the start of pass p: the digits before p of the k-th order key, the rank
// still to resolve among the candidates that match them, and where those candidates are.
struct SelState {
    unsigned long long pre_hi, pre_lo, mask_hi, mask_lo;
    unsigned int k_rem;         // rank (1-based) among the matching candidates
    unsigned int n_in;          // entries of the current candidate list
    unsigned int n_match;       // of them, how many match the decided prefix
    unsigned int cur;           // the current list: 0 = the dense list, 1, 2 = the scratch lists
};

struct TrimState {
    unsigned int size;          // live entries of the current table
    unsigned int k;             // entries to drop in this trim
    unsigned int invalid;       // malformed candidates seen by od_cache_insert
    unsigned int dropped;       // candidates that found no free slot on their whole probe sequence
    // The pass that counts sets these back, and the last kernel the bins: a trim that is replayed from a CUDA
    // graph starts like the one that was captured.
    unsigned int k_rem;         // of the listed entries, how many to drop
    unsigned int n_list;        // entries listed because their bin has both kinds
    unsigned int n_late;        // survivors that are not in the group their run hashes to, listed from the other end
    unsigned long long hi_and, hi_or;       // AND / OR of (new?, score) over the listed entries: bits that never vary
    unsigned long long thr_hi, thr_lo;      // trim_select_kernel: the k-th order key
    unsigned int bins[256];     // live entries by score (score_bin)
    // LRU: where the bins begin, a clock before which hardly an entry was accessed (that of the last entry which the trim before
    // dropped), and what becomes of it behind a trim without a list. What stays and what goes does not depend on it.
    unsigned int oldest, next_oldest;
    SelState sel[PASSES];       // sel[p]: written by block 0 of pass p
    unsigned int n_out[PASSES]; // entries pass p copied into its output list
    unsigned int hist[PASSES][256];
};

// Trim scratch for a table of `cap` slots: the listed entries (order key and slot in the old table)
// and two lists of (hi, lo) candidates.
struct TrimLists {
    unsigned long long *r_hi, *r_key;
    unsigned int *r_slot;
    unsigned long long *l_hi[2], *l_lo[2];
};
__host__ __device__ inline TrimLists trim_lists(void *base, int64_t cap)
{
    TrimLists t;
    unsigned long long *q = (unsigned long long *)base;
    t.r_hi = q; t.r_key = q + cap;
    t.l_hi[0] = q + 2 * cap; t.l_lo[0] = q + 3 * cap;
    t.l_hi[1] = q + 4 * cap; t.l_lo[1] = q + 5 * cap;
    t.r_slot = (unsigned int *)(q + 6 * cap);
    return t;
}
constexpr size_t TRIM_LIST_BYTES_PER_SLOT = 6 * 8 + 4;
// Slots taken in each group (a count may run past the group's 32), for a table of `cap` slots: read four groups at a time
inline size_t fill_words(int64_t cap) { return (size_t)(cap / OD_GROUP < 4 ? 4 : cap / OD_GROUP); }

// order key of a live entry: hi = (inserted at the current clock) << 32 | score, lo = run key
__device__ __forceinline__ void order_key(int policy, unsigned int clock, unsigned long long key,
                                          unsigned int stamp, unsigned int freq, unsigned int born,
                                          unsigned long long &hi, unsigned long long &lo)
{
    hi = ((unsigned long long)(born == clock ? 1u : 0u) << 32) | (policy == 0 ? stamp : freq);
    lo = key;
}

__device__ __forceinline__ unsigned int digit_of(int pass, unsigned long long hi, unsigned long long lo)
{
    return pass < 5 ? (unsigned int)(hi >> (8 * (4 - pass))) & 0xFFu
                    : (unsigned int)(lo >> (8 * (12 - pass))) & 0xFFu;
}

// The kernels of an insertion and of a trim form chains in which each needs what the one
// before it wrote. They are launched with programmatic stream serialization and wait at once:
// the launch latency of a kernel is spent while its predecessor still runs. The first kernel of a chain releases the
// next behind its wait: what runs behind the chain may read its inputs early, and is promised that what was in front of
// the chain is done.
__device__ __forceinline__ void chain_wait(bool first = false)
{
    if (!first) asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (first) asm volatile("griddepcontrol.launch_dependents;");
}

// launch with or without programmatic stream serialization (the context's "pdl" option)
template <typename... Params, typename... Args>
cudaError_t chain_launch(void (*kernel)(Params...), unsigned grid, unsigned block, cudaStream_t s, bool pdl, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(block); cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}


__global__ void insert_claim_kernel(int32_t N, int32_t v_q, int32_t v_p, const int32_t *__restrict__ runs,
                                    const int32_t *__restrict__ len, const int32_t *__restrict__ target,
                                    unsigned long long *keys, const int32_t *vals, int64_t cap,
                                    unsigned int *owner, int32_t *cand_slot, unsigned int *fill, TrimState *st)
{
    chain_wait(true);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    cand_slot[i] = -1;
    // one round trip: every load goes out before the first is looked at
    const int L = len[i], tgt = target[i];
    int32_t ids[OD_NGRAM_MAX];
#pragma unroll
    for (int j = 0; j < OD_NGRAM_MAX; ++j) ids[j] = runs[(size_t)i * OD_NGRAM_MAX + j];
    bool ok = L >= 2 && L <= OD_NGRAM_MAX && tgt >= 0 && tgt < v_p;
#pragma unroll
    for (int j = 0; j < OD_NGRAM_MAX; ++j) ok = ok && (j >= L || (ids[j] >= 0 && ids[j] < v_q));
    if (!ok) { atomicAdd(&st->invalid, 1u); return; }
    const unsigned long long key = od_pack_run(ids, L);
    const uint64_t ngroups = (uint64_t)cap / OD_GROUP;
    uint64_t g = od_hash64(key) & (ngroups - 1);
    for (uint64_t step = 0; step < ngroups; ++step) {       // bounded: ends on any table contents
        // A group is filled from slot 0 without holes, and in a table at most half full it
        // rarely holds more than sixteen entries: its first sixteen keys are read at once
        // (one round trip instead of one per occupied slot), the rest one by one.
        constexpr int HEAD = 16;
        unsigned long long head[HEAD];
#pragma unroll
        for (int h = 0; h < HEAD / 2; ++h) {
            const ulonglong2 a = __ldcg((const ulonglong2 *)(keys + g * OD_GROUP) + h);
            head[2 * h] = a.x; head[2 * h + 1] = a.y;
        }
        int s0 = HEAD;                                      // the first slot that is empty or holds the key
#pragma unroll
        for (int h = HEAD - 1; h >= 0; --h)
            if (head[h] == 0ull || head[h] == key) s0 = h;
        for (int s = s0; s < OD_GROUP; ++s) {
            const int64_t slot = (int64_t)(g * OD_GROUP + s);
            // the slot as it was read with its group: empty, or the candidate's run (then its value tells
            // whether it is an entry or another candidate's claim); a slot that was empty has no value
            unsigned long long seen = 0ull;
            if (s < HEAD) {
#pragma unroll
                for (int h = 0; h < HEAD; ++h) seen = h == s ? head[h] : seen;
            } else {
                seen = keys[slot];
            }
            const unsigned long long cur = seen == 0ull ? atomicCAS(keys + slot, 0ull, key) : seen;
            if (cur == 0ull) atomicAdd(fill + g, 1u);
            if (cur == 0ull || cur == key) {
                // an entry with a value was there before this batch: nothing to add
                if (seen == 0ull || ((volatile const int32_t *)vals)[slot] < 0) {
                    atomicMin(owner + slot, (unsigned int)i);
                    cand_slot[i] = (int32_t)slot;
                }
                return;
            }
        }
        g = (g + 1) & (ngroups - 1);
    }
    atomicAdd(&st->dropped, 1u);                            // the table is full: the candidate is lost
}

__global__ void insert_commit_kernel(int32_t N, const int32_t *__restrict__ target, int32_t *vals,
                                     unsigned int *stamp, unsigned int *freq, unsigned int *born,
                                     unsigned int *owner, const int32_t *__restrict__ cand_slot,
                                     unsigned int clock, TrimState *st)
{
    chain_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int32_t slot = cand_slot[i], tgt = target[i];
    if (slot < 0 || owner[slot] != (unsigned int)i) return; // a candidate with a lower index carries this run
    stamp[slot] = clock; freq[slot] = 1u; born[slot] = clock;
    __threadfence();
    vals[slot] = tgt;                                        // the entry exists from here on
    owner[slot] = 0xFFFFFFFFu;
    atomicAdd(&st->size, 1u);
}

__global__ void trim_begin_kernel(TrimState *st)
{
    chain_wait(true);
    for (int p = 0; p < PASSES; ++p) st->hist[p][threadIdx.x] = 0u;
    if (threadIdx.x < PASSES) st->n_out[threadIdx.x] = 0u;
}

// Exclusive offset of this thread's `n` items within the block's `total` (one block scan).
__device__ __forceinline__ unsigned int block_offsets(unsigned int n, unsigned int *s_warp, unsigned int &total)
{
    const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    unsigned int inc = n;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned int t = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += t;
    }
    __syncthreads();                                        // s_warp may still be read from the last call
    if (lane == 31u) s_warp[warp] = inc;
    __syncthreads();
    unsigned int base = 0;
    total = 0;
    for (unsigned int w = 0; w < blockDim.x / 32u; ++w) {
        if (w < warp) base += s_warp[w];
        total += s_warp[w];
    }
    return base + inc - n;
}

// ---- the two passes over the table ---------------------------------------------------------
//
// Sixteen lanes take a group's first sixteen slots (a table at most half full often has no more: a group is filled from
// slot 0), then the rest where the sixteenth is taken, up to four groups at a time. How far a group is filled is kept for
// each, so that no slot is cleared that was not taken. Neither pass has an atomic per entry: a survivor stays in the
// group it is in. Bound by the chain of round trips and by L2 (262144 entries: 13 MB read, 12 MB written). Before,
// one pass packed all live entries into a list, the select walked through it, and a rebuild put every survivor into the slot that
// its group's counter gave. Device time of an insertion, a trim and a translation, before -> now: 262144 entries and 16384 new
// ones 53.6 -> 36.7 us, by frequency 70.0 -> 64.7; 4096 and 512 24.5 -> 20.4; 32768 and 4096 by frequency 35.0 -> 31.9. (The
// whole trim in one cluster of 1 to 16 blocks, for tables of up to 131072 slots: 26.5 and 37.7 us on the last two; a step
// of it is a chain of trips as long as a launch's.)
// QUAD: groups of a half-warp at a time, 1, 2 or 4: see trim_quad.
constexpr int TRIM_THREADS = 256, TRIM_HALVES = TRIM_THREADS / 16;

// (new?, score) to one of 256 bins, in the order of trims: 255 new; else by frequency (LFU), or by the clock from the oldest
// on (LRU), exact for 128 of them, four bins to an octave beyond. LRU drops the oldest, so their clocks have bins of their own
// whatever the step of the clock: by age, exact for the last 127 clocks, the entries of several batches shared the bin where
// the k-th is (16384 entries, 256 new ones, an insertion and a trim, with a clock that goes on by 1000: 25.9 us by age, 18.0 so).
__device__ __forceinline__ unsigned int log_bin(unsigned int v)
{
    const int e = 31 - __clz((int)v);
    return v < 128u ? v : 128u + ((unsigned int)(e - 7) << 2) + (v >> (e - 2) & 3u);   // at most 227
}
// the least value of a bin (of one beyond the last: 2^32)
__device__ __forceinline__ unsigned long long log_bin_floor(unsigned int bin)
{
    return bin < 128u ? bin : (unsigned long long)(4u + (bin & 3u)) << (((bin - 128u) >> 2) + 5u);
}
__device__ __forceinline__ unsigned int score_bin(int policy, unsigned int oldest, unsigned int score, bool is_new)
{
    if (is_new) return 255u;
    if (policy != 0) return log_bin(score);
    return score < oldest ? 0u : 1u + log_bin(score - oldest);
}
// whether all of a bin's entries have one (new?, score), and which
__device__ __forceinline__ bool exact_bin(int policy, unsigned int oldest, unsigned int bin, unsigned long long &hi)
{
    hi = policy == 0 ? (unsigned long long)(oldest + bin - 1u) : (unsigned long long)bin;
    return policy == 0 ? bin >= 1u && bin <= 128u : bin < 128u;
}

// Count digit `d` of the lanes with `ok` into hist: digits are heavily tied (scores, the upper
// bytes of short runs), so lanes that agree count as one add.
__device__ __forceinline__ void count_digit(unsigned int *hist, unsigned int d, bool ok)
{
    const unsigned int same = __match_any_sync(0xFFFFFFFFu, ok ? d : 256u);
    if (ok && __ffs(same) - 1 == (int)(threadIdx.x & 31)) atomicAdd(hist + d, (unsigned int)__popc(same));
}

// The live entries by score.
template <int QUAD>
__global__ void __launch_bounds__(TRIM_THREADS)
trim_count_kernel(int policy, unsigned int clock, const int32_t *vals, const unsigned int *score, const unsigned int *born,
                  int64_t cap, TrimState *st)
{
    __shared__ unsigned int s_bins[256];
    s_bins[threadIdx.x] = 0u;
    const int64_t quads = (cap / OD_GROUP + QUAD - 1) / QUAD;
    const int at = threadIdx.x & 15;
    chain_wait(true);
    const unsigned int oldest = __ldcg(&st->oldest);
    if (blockIdx.x == 0 && threadIdx.x == 0) { st->n_list = 0u; st->n_late = 0u; st->hi_and = ~0ull; st->hi_or = 0ull; }
    __syncthreads();
    for (int64_t q0 = (int64_t)blockIdx.x * TRIM_HALVES; q0 < quads; q0 += (int64_t)gridDim.x * TRIM_HALVES) {
        const int64_t quad = q0 + (threadIdx.x >> 4);
        bool more = false;                                  // a group's sixteenth slot is taken: the others too
        for (int s = at; s < OD_GROUP && (s < 16 || __any_sync(0xFFFFFFFFu, more)); s += 16) {
            int32_t v[QUAD];
            unsigned int sc[QUAD], bn[QUAD];
#pragma unroll
            for (int e = 0; e < QUAD; ++e) {
                const int64_t slot = (quad * QUAD + e) * OD_GROUP + s;
                v[e] = -1;
                if (slot < cap) { v[e] = __ldcg(vals + slot); sc[e] = __ldcg(score + slot); bn[e] = __ldcg(born + slot); }
            }
#pragma unroll
            for (int e = 0; e < QUAD; ++e) {
                count_digit(s_bins, score_bin(policy, oldest, sc[e], bn[e] == clock), v[e] >= 0);   // (a slot without a value is no entry)
                more = more || (at == 15 && v[e] >= 0);
            }
        }
    }
    __syncthreads();
    if (s_bins[threadIdx.x]) atomicAdd(st->bins + threadIdx.x, s_bins[threadIdx.x]);
}

// A slot of the old table, as it goes into the new one
struct Entry {
    unsigned long long key;
    int32_t v;
    unsigned int stamp, freq, born;
};
struct Table {
    unsigned long long *keys;                               // an empty slot has no value (-1)
    int32_t *vals;
    unsigned int *stamp, *freq, *born, *fill;
    __device__ __forceinline__ Entry load(int64_t slot) const
    {
        return Entry{__ldcg(keys + slot), __ldcg(vals + slot), __ldcg(stamp + slot), __ldcg(freq + slot), __ldcg(born + slot)};
    }
    __device__ __forceinline__ void store(int64_t slot, const Entry &e) const
    {
        keys[slot] = e.key; vals[slot] = e.v; stamp[slot] = e.stamp; freq[slot] = e.freq; born[slot] = e.born;
    }
};

// An entry into the new table. A group is filled from its slot 0 without holes (od_cache_insert stops at the first empty
// slot). Every placement takes the next slot of its group from the group's count: no two entries ever want the same
// slot, so there is nothing to retry. A full group (32 entries: rare in a table at most half full) sends
// the entry on to the next group, as a probe would go.
__device__ __forceinline__ void place_entry(const Table &to, int64_t cap, const Entry &en)
{
    const uint64_t ngroups = (uint64_t)cap / OD_GROUP;
    uint64_t g = od_hash64(en.key) & (ngroups - 1);
    for (uint64_t step = 0; step < ngroups; ++step) {
        const unsigned int at = atomicAdd(to.fill + g, 1u);
        if (at < (unsigned int)OD_GROUP) { to.store((int64_t)(g * OD_GROUP + at), en); break; }
        g = (g + 1) & (ngroups - 1);
    }
}

// How far QUAD neighbouring groups are filled
template <int QUAD> struct FillWord;
template <> struct FillWord<1> { typedef unsigned int type; };
template <> struct FillWord<2> { typedef uint2 type; };
template <> struct FillWord<4> { typedef uint4 type; };
template <int QUAD>
__device__ __forceinline__ void load_fill(const unsigned int *fill, int64_t quad, unsigned int (&n)[QUAD])
{
    typedef typename FillWord<QUAD>::type Word;
    const Word v = __ldcg((const Word *)fill + quad);
    memcpy(n, &v, sizeof(v));
}
template <int QUAD>
__device__ __forceinline__ void store_fill(unsigned int *fill, int64_t quad, const unsigned int (&n)[QUAD])
{
    typename FillWord<QUAD>::type v;
    memcpy(&v, n, sizeof(v));
    ((typename FillWord<QUAD>::type *)fill)[quad] = v;
}

// Which bin the k-th entry is in; then every group's survivors into the same group of the new table, and into the list what
// cannot be said yet. The table has not been written since before the pass that counts waited, so the first
// groups are loaded in front of this kernel's own wait.
template <int QUAD>
__global__ void __launch_bounds__(TRIM_THREADS, 4)
trim_split_kernel(int policy, unsigned int clock, unsigned int max_entries, const Table from, const Table to, int64_t cap,
                  void *lists, TrimState *st)
{
    __shared__ unsigned int s_warp[TRIM_THREADS / 32], s_base[2], s_bin, s_rem, s_in;
    __shared__ unsigned long long s_and, s_or;
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t groups = cap / OD_GROUP, quads = (groups + QUAD - 1) / QUAD;
    const int at = threadIdx.x & 15, half = threadIdx.x >> 4 & 1;
    const TrimLists L = trim_lists(lists, cap);
    unsigned int run[QUAD];
    Entry en[QUAD];
    int64_t q0 = (int64_t)blockIdx.x * TRIM_HALVES, quad = q0 + (threadIdx.x >> 4);
    const auto load = [&](int s, unsigned int which) {
#pragma unroll
        for (int e = 0; e < QUAD; ++e) {
            const int64_t slot = (quad * QUAD + e) * OD_GROUP + s;
            en[e].v = -1;
            if (slot < cap && (which >> e & 1u)) en[e] = from.load(slot);
        }
    };
    load(at, 0xFu);
    // An entry is in another group than its run hashes to only if all groups from there on were full: where none of the
    // groups in front of the half-warp's is, nobody asks (the hash is a third of the pass's instructions).
    const auto behind_a_full_group = [&]() {
        if (quad >= quads) return false;
        unsigned int f[QUAD], most = __ldcg(from.fill + ((quad * QUAD - 1) & (groups - 1)));
        load_fill<QUAD>(from.fill, quad, f);
#pragma unroll
        for (int e = 0; e + 1 < QUAD; ++e) most = max(most, f[e]);
        return most >= (unsigned int)OD_GROUP;
    };
    bool ask = behind_a_full_group();
    if (threadIdx.x == 0) { s_and = ~0ull; s_or = 0ull; s_bin = 256u; s_rem = 0u; s_in = 0u; }
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- the first bin at which the running count reaches k (none: everything goes)
    const unsigned int oldest = __ldcg(&st->oldest), size = __ldcg(&st->size), k = size > max_entries ? size - max_entries : 0u;
    const unsigned int mine = __ldcg(st->bins + threadIdx.x);
    unsigned int total;
    const unsigned int before = block_offsets(mine, s_warp, total);
    if (k > before && k - before <= mine) { s_bin = threadIdx.x; s_rem = k - before; s_in = mine; }
    __syncthreads();
    const bool whole = s_rem == s_in;                       // the bin goes as a whole: nothing is left to find out
    const unsigned int first_kept = k == 0u ? 0u : s_bin + (whole ? 1u : 0u), mixed = k == 0u || whole ? 512u : s_bin;
    unsigned long long bin_hi;
    const bool exact = exact_bin(policy, oldest, mixed & 255u, bin_hi);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->k = k; st->k_rem = mixed < 256u ? s_rem : 0u;
        // (bins up to s_bin went: the least clock of the next)
        st->next_oldest = k == 0u || s_bin >= 256u ? oldest : (unsigned int)min((unsigned long long)clock, oldest + log_bin_floor(s_bin));
        if (exact) { st->hi_and = bin_hi; st->hi_or = bin_hi; }
    }

    for (;;) {
        const bool in = quad < quads, ask_here = __any_sync(0xFFFFFFFFu, ask);
        unsigned int had[QUAD];
#pragma unroll
        for (int e = 0; e < QUAD; ++e) { run[e] = 0u; had[e] = 0u; }
        // the groups whose sixteenth slot is taken: their other slots too
        unsigned int more = 0u;
        if (at == 15) {
#pragma unroll
            for (int e = 0; e < QUAD; ++e) more |= en[e].v >= 0 ? 1u << e : 0u;
        }
        const int rounds = __syncthreads_or((int)more) ? 2 : 1;
        for (int round = 0; round < rounds; ++round) {
            const int s = at + 16 * round;
            if (round) { more = __shfl_sync(0xFFFFFFFFu, more, 16 * half + 15); load(s, more); }
            if (round + 1 == rounds && in) load_fill<QUAD>(to.fill, quad, had);
            unsigned int listed = 0u, late = 0u;            // of this thread's four: bit e
            unsigned long long t_and = ~0ull, t_or = 0ull;
            if (round == 0 || __any_sync(0xFFFFFFFFu, more != 0u))
#pragma unroll
                for (int e = 0; e < QUAD; ++e) {
                    const int64_t g = quad * QUAD + e;
                    const bool is_new = en[e].born == clock;
                    const unsigned int score = policy == 0 ? en[e].stamp : en[e].freq;
                    const unsigned int bin = en[e].v >= 0 ? score_bin(policy, oldest, score, is_new) : 0u;
                    const bool live = en[e].v >= 0;
                    bool home = true;
                    if (ask_here) home = (int64_t)(od_hash64(en[e].key) & (uint64_t)(groups - 1)) == g;
                    const bool keep = live && bin >= first_kept && bin != mixed;
                    if (live && bin == mixed) {
                        listed |= 1u << e;
                        unsigned long long hi, lo;
                        order_key(policy, clock, en[e].key, en[e].stamp, en[e].freq, en[e].born, hi, lo);
                        t_and &= hi; t_or |= hi;
                    }
                    if (keep && !home) late |= 1u << e;
                    const unsigned int stays = __ballot_sync(0xFFFFFFFFu, keep && home) >> (16 * half) & 0xFFFFu;
                    if (keep && home) to.store(g * OD_GROUP + run[e] + __popc(stays & ((1u << at) - 1u)), en[e]);
                    run[e] += __popc(stays);
                }
            // ---- the lists: one append per block
            unsigned int sum;
            unsigned int ofs = block_offsets(__popc(listed) | __popc(late) << 16, s_warp, sum);
            if (sum == 0u) continue;                        // (the same for every thread of the block)
            if (threadIdx.x == 0) s_base[0] = sum & 0xFFFFu ? atomicAdd(&st->n_list, sum & 0xFFFFu) : 0u;
            if (threadIdx.x == 32) s_base[1] = sum >> 16 ? atomicAdd(&st->n_late, sum >> 16) : 0u;
            if (!exact && (sum & 0xFFFFu)) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    t_and &= __shfl_xor_sync(0xFFFFFFFFu, t_and, off);
                    t_or |= __shfl_xor_sync(0xFFFFFFFFu, t_or, off);
                }
                if ((threadIdx.x & 31) == 0) { atomicAnd(&s_and, t_and); atomicOr(&s_or, t_or); }
            }
            __syncthreads();
            int64_t i_list = (int64_t)s_base[0] + (ofs & 0xFFFFu), i_late = cap - 1 - ((int64_t)s_base[1] + (ofs >> 16));
#pragma unroll
            for (int e = 0; e < QUAD; ++e) {
                const unsigned int slot = (unsigned int)((quad * QUAD + e) * OD_GROUP + s);
                if (listed >> e & 1u) {
                    if (i_list < cap) {                     // (never beyond the list)
                        order_key(policy, clock, en[e].key, en[e].stamp, en[e].freq, en[e].born, L.r_hi[i_list], L.r_key[i_list]);
                        L.r_slot[i_list] = slot;
                    }
                    ++i_list;
                }
                if (late >> e & 1u) {
                    if (i_late >= 0) L.r_slot[i_late] = slot;
                    --i_late;
                }
            }
        }
        // ---- the slots that are free now and were taken, and how far each group is filled
#pragma unroll
        for (int e = 0; e < QUAD; ++e)
            for (unsigned int s = run[e] + at; s < min(had[e], (unsigned int)OD_GROUP); s += 16) {
                const int64_t slot = (quad * QUAD + e) * OD_GROUP + s;
                to.keys[slot] = 0ull; to.vals[slot] = -1;
            }
        if (in && at == 0) store_fill<QUAD>(to.fill, quad, run);
        q0 += (int64_t)gridDim.x * TRIM_HALVES;
        if (q0 >= quads) break;
        quad = q0 + (threadIdx.x >> 4);
        load(at, 0xFu);
        ask = behind_a_full_group();
    }
    if (!exact && threadIdx.x == 0 && (s_and != ~0ull || s_or != 0ull)) { atomicAnd(&st->hi_and, s_and); atomicOr(&st->hi_or, s_or); }
}

// ---- the k-th order key in one launch ------------------------------------------------------
//
// One cluster of P blocks, each with a slice of the list: a most-significant-digit radix
// select in which a pass is a histogram in shared memory, ONE cluster barrier and the sum of the
// P histograms over distributed shared memory, by every block alike. The bits of (new?, score)
// that vary are settled first, over the slices; the keys of the entries that tie at that score
// then stay in shared memory for the run key, and the select ends as soon as
// every candidate that is left is among the k (usually two passes in all, three by frequency: a pass costs 2.5 us or so,
// of which the barrier and the sums are most). As a chain of 13 launches of the whole grid the passes took
// 52 us for the 262144 entries of a table.
// How long the list is, only the device knows: one batch where a clock is one batch's, but most of the table where it was
// loaded at one clock, and by LFU as a rule. As many blocks take part as the list gives an entry a thread to; the others leave (4096
// entries and 512 new ones: 23.9 us with 16 blocks, 22.8 with one). Such a list stays in registers, and the cluster places what
// stays of it. A longer one is left to trim_place_kernel on the whole chip, which is launched where the table may have one
// (`follow`). An insertion and a trim by LRU of 262144 entries that were loaded at one clock, 16384 new ones: 72.1 us placed by the
// cluster, 54.9 so; 16000 and 256: 62.3 -> 31.6. (As many clusters as are resident, each with the whole select and a
// share of the placing, in place of the second launch: 58.3 and 32.1, and 39.3 where the list is short: 37.0.)
constexpr int SELECT_THREADS = 1024, SELECT_MAX_BLOCKS = 16;

__global__ void __launch_bounds__(SELECT_THREADS, 1)
trim_select_kernel(unsigned int room, const Table from, const Table to, int64_t cap, void *lists, TrimState *st, int follow)
{
    extern __shared__ __align__(16) unsigned long long s_keys[];   // [room]
    __shared__ unsigned int s_hist[2][256], s_sum[256];
    __shared__ unsigned int s_n, s_digit, s_run, s_in;
    const unsigned int rank = blockIdx.x, lane = threadIdx.x & 31u;
    chain_wait(true);                                       // (the next kernel reads the list in front of its own wait)
    const unsigned int n = (unsigned int)min((int64_t)__ldcg(&st->n_list), cap), k = __ldcg(&st->k_rem);
    const unsigned long long hi_and = __ldcg(&st->hi_and), hi_or = __ldcg(&st->hi_or);
    const TrimLists L = trim_lists(lists, cap);
    if (rank == 0 && threadIdx.x == 0) {
        st->size = __ldcg(&st->size) - __ldcg(&st->k);
        if (n == 0u) st->oldest = __ldcg(&st->next_oldest);
    }
    if (rank == 0 && threadIdx.x < 256) st->bins[threadIdx.x] = 0u;   // for the next trim
    const bool one = n <= gridDim.x * SELECT_THREADS, place = one || !follow;
    if (place) {
        const unsigned int late = __ldcg(&st->n_late);
        for (unsigned int i = rank * SELECT_THREADS + threadIdx.x; i < late; i += gridDim.x * SELECT_THREADS)
            place_entry(to, cap, from.load(__ldcg(L.r_slot + (cap - 1 - (int64_t)i))));
    }
    // the blocks that take part: a cluster's barrier waits for the threads that have not left
    const unsigned int P = min(gridDim.x, (n + SELECT_THREADS - 1) / SELECT_THREADS);
    if (rank >= P) return;
    const unsigned int per = (n + P - 1) / P, lo = min(rank * per, n), hi_end = min(lo + per, n);
    // An entry for a thread at most: it stays in registers, and what goes into the new table is on its way while the
    // digits are counted.
    const bool have = one && lo + threadIdx.x < hi_end;
    unsigned long long my_hi = 0ull;
    Entry mine = {};
    if (have) {
        my_hi = __ldcg(L.r_hi + lo + threadIdx.x);
        mine = from.load(__ldcg(L.r_slot + lo + threadIdx.x));
    }
    for (int i = threadIdx.x; i < 512; i += SELECT_THREADS) s_hist[i >> 8][i & 255] = 0u;
    if (threadIdx.x == 0) s_n = 0u;
    __syncthreads();

    unsigned int k_rem = k, n_match = n, buf = 0;
    // the first digit at which the running count over all blocks reaches k_rem
    auto settle = [&]() -> unsigned int {
        od_cluster_arrive(); od_cluster_wait();             // every block's histogram is complete
        if (threadIdx.x < 256) {
            unsigned int h[SELECT_MAX_BLOCKS], t = 0;       // all loads before the first use: one trip, not P
#pragma unroll
            for (unsigned int r = 0; r < SELECT_MAX_BLOCKS; ++r) h[r] = r < P ? od_cluster_load(&s_hist[buf][threadIdx.x], r) : 0u;
#pragma unroll
            for (unsigned int r = 0; r < SELECT_MAX_BLOCKS; ++r) t += h[r];
            s_sum[threadIdx.x] = t;
            s_hist[buf ^ 1][threadIdx.x] = 0u;              // (read by the others before the barrier above)
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            unsigned int mine = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) mine += s_sum[lane * 8 + i];
            unsigned int inc = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                if (lane >= (unsigned)off) inc += v;
            }
            const unsigned int reach = __ballot_sync(0xFFFFFFFFu, inc >= k_rem);
            const unsigned int owner = reach ? __ffs(reach) - 1 : 31;
            if (lane == owner) {
                unsigned int run = inc - mine, d = lane * 8;
                for (; d < lane * 8 + 7 && run + s_sum[d] < k_rem; ++d) run += s_sum[d];
                s_digit = d; s_run = run; s_in = s_sum[d];
            }
        }
        __syncthreads();
        buf ^= 1u;
        k_rem -= s_run; n_match = s_in;
        return s_digit;
    };

    // ---- (new?, score): the bits that vary, over the slice, up to eight a pass. They rarely are whole bytes (the
    // clocks of the last dozen batches and whether an entry is new: one pass, a byte at a time it was two).
    const unsigned long long vary = hi_or & ~hi_and;
    unsigned long long thr_hi = hi_and, todo = vary;
    while (todo != 0ull && n_match > k_rem) {
        // the highest ones, in at most two runs: sh1, sh2 their lowest bits, w1, w2 how many they are
        const int top = 63 - __clzll((long long)todo);
        const int w1 = min(8, __clzll((long long)~(todo << (63 - top)))), sh1 = top - w1 + 1;
        const unsigned long long rest = todo & ((1ull << sh1) - 1ull);
        int w2 = 0, sh2 = 0;
        if (w1 < 8 && rest) {
            const int top2 = 63 - __clzll((long long)rest);
            w2 = min(8 - w1, __clzll((long long)~(rest << (63 - top2))));
            sh2 = top2 - w2 + 1;
        }
        const unsigned int m1 = (1u << w1) - 1u, m2 = (1u << w2) - 1u;
        const unsigned long long known = ~todo;
        const auto digit = [&](unsigned long long h) { return ((unsigned int)(h >> sh1) & m1) << w2 | ((unsigned int)(h >> sh2) & m2); };
        constexpr int U = 9;
        if (one) count_digit(s_hist[buf], digit(my_hi), have && (my_hi & known) == (thr_hi & known));
        for (unsigned int i0 = one ? hi_end : lo; i0 < hi_end; i0 += SELECT_THREADS * U) {
            unsigned long long h[U];
#pragma unroll
            for (int e = 0; e < U; ++e) {
                const unsigned int i = i0 + e * SELECT_THREADS + threadIdx.x;
                h[e] = i < hi_end ? __ldcg(L.r_hi + i) : 0ull;
            }
#pragma unroll
            for (int e = 0; e < U; ++e)
                count_digit(s_hist[buf], digit(h[e]), i0 + e * SELECT_THREADS + threadIdx.x < hi_end && (h[e] & known) == (thr_hi & known));
        }
        const unsigned int d = settle();
        const unsigned long long bits = (unsigned long long)m1 << sh1 | (unsigned long long)m2 << sh2;
        thr_hi = (thr_hi & ~bits) | (unsigned long long)(d >> w2) << sh1 | (unsigned long long)(d & m2) << sh2;
        todo &= ~bits;
    }
    thr_hi |= todo;                                         // (every candidate left is among the k, whatever these bits)
    // ---- the run keys of the entries that tie at that score
    unsigned long long thr_lo = 0ull, decided = 0ull, least = 0ull;
    if (n_match > k_rem) {
        // The first digit tells runs of two, three and four ids apart (of equal score the shorter run's key is the
        // smaller: the upper fields are zero) and has the leading bits of the last id. A byte at a time the select
        // walked through the empty fields: five or six passes where two are enough.
        const auto first_digit = [](unsigned long long key) -> unsigned int {
            const unsigned int f3 = (unsigned int)(key >> 48), f2 = (unsigned int)(key >> 32) & 0xFFFFu;
            return f3 ? 192u + (f3 >> 10) : f2 ? 128u + (f2 >> 10) : (unsigned int)key >> 25;
        };
        constexpr int U = 9;
        if (one) count_digit(s_hist[buf], first_digit(mine.key), have && my_hi == thr_hi);
        for (unsigned int i0 = one ? hi_end : lo; i0 < hi_end; i0 += SELECT_THREADS * U) {
            unsigned long long h[U], key[U];
#pragma unroll
            for (int e = 0; e < U; ++e) {
                const unsigned int i = i0 + e * SELECT_THREADS + threadIdx.x;
                h[e] = i < hi_end ? __ldcg(L.r_hi + i) : ~thr_hi;
            }
#pragma unroll
            for (int e = 0; e < U; ++e) {
                key[e] = 0ull;
                if (h[e] == thr_hi) key[e] = __ldcg(L.r_key + i0 + e * SELECT_THREADS + threadIdx.x);
            }
            unsigned int mine = 0;
#pragma unroll
            for (int e = 0; e < U; ++e) mine += h[e] == thr_hi ? 1u : 0u;
            // one append per warp, its lanes in order
            unsigned int inc = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                if (lane >= (unsigned)off) inc += v;
            }
            unsigned int at = 0;
            if (lane == 31 && inc) at = atomicAdd(&s_n, inc);
            at = __shfl_sync(0xFFFFFFFFu, at, 31) + inc - mine;
#pragma unroll
            for (int e = 0; e < U; ++e)
                if (h[e] == thr_hi) { if (at < room) s_keys[at] = key[e]; ++at; }
#pragma unroll
            for (int e = 0; e < U; ++e) count_digit(s_hist[buf], first_digit(key[e]), h[e] == thr_hi);
        }
        __syncthreads();
        const bool held = s_n <= room;                      // else the slice is read again (a table trimmed late)
        const unsigned int c_end = one ? 0u : held ? s_n : hi_end - lo;
        const unsigned int d = settle();
        int undecided;                                      // the lowest so many bits
        if (d >= 192u) { least = 1ull << 48; undecided = 58; thr_lo = (unsigned long long)(d - 192u) << 58; }
        else if (d >= 128u) { least = 1ull << 32; undecided = 42; thr_lo = (unsigned long long)(d - 128u) << 42; }
        else { undecided = 25; thr_lo = (unsigned long long)d << 25; }
        decided = ~0ull << undecided;
        while (undecided > 0 && n_match > k_rem) {
            const int w = min(8, undecided);
            undecided -= w;
            if (one) count_digit(s_hist[buf], (unsigned int)(mine.key >> undecided) & ((1u << w) - 1u),
                                 have && my_hi == thr_hi && mine.key >= least && (mine.key & decided) == thr_lo);
            for (unsigned int i0 = 0; i0 < c_end; i0 += SELECT_THREADS) {
                const unsigned int i = i0 + threadIdx.x;
                bool ok = i < c_end;
                unsigned long long key = 0ull;
                if (ok) {
                    key = held ? s_keys[i] : __ldcg(L.r_key + lo + i);
                    ok = key >= least && (key & decided) == thr_lo && (held || __ldcg(L.r_hi + lo + i) == thr_hi);
                }
                count_digit(s_hist[buf], (unsigned int)(key >> undecided) & ((1u << w) - 1u), ok);
            }
            const unsigned int d = settle();
            thr_lo |= (unsigned long long)d << undecided;
            decided |= (unsigned long long)((1u << w) - 1u) << undecided;
        }
    }
    thr_lo |= ~decided;                                     // every candidate left is among the k
    od_cluster_arrive();                                    // (waited for below: nobody leaves while its histogram may still be read)
    if (have && (my_hi > thr_hi || (my_hi == thr_hi && mine.key > thr_lo))) place_entry(to, cap, mine);
    if (place && !one)
        for (unsigned int i = lo + threadIdx.x; i < hi_end; i += SELECT_THREADS) {
            const unsigned long long hi = __ldcg(L.r_hi + i), key = __ldcg(L.r_key + i);
            const Entry en = from.load(__ldcg(L.r_slot + i));   // (though some are dropped: one round trip less)
            if (hi > thr_hi || (hi == thr_hi && key > thr_lo)) place_entry(to, cap, en);
        }
    od_cluster_wait();
    if (rank == 0 && threadIdx.x == 0) { st->thr_hi = thr_hi; st->thr_lo = thr_lo; st->oldest = (unsigned int)thr_hi; }
}

// ---- the same as a chain of launches, for tables too large for one cluster -----------------

// Is digit `pass` the same in every listed entry? Only asked for the five bytes of (new?, score).
__device__ __forceinline__ bool digit_is_constant(int pass, unsigned long long hi_and, unsigned long long hi_or)
{
    return pass < 5 && (((hi_or & ~hi_and) >> (8 * (4 - pass))) & 0xFFull) == 0ull;
}

// The state at the start of pass `pass` (0..PASSES), worked out from the state at the start of
// the pass before it and that pass's histogram: by every block alike, the same arithmetic on the
// same numbers. All threads of the block call; s_hist (256 words) and s_sel are its scratch.
__device__ __forceinline__ SelState select_state(int pass, const TrimState *st, unsigned int *s_hist, SelState *s_sel)
{
    if (pass == 0) {
        SelState z = {};
        z.k_rem = __ldcg(&st->k_rem);
        z.n_in = z.n_match = __ldcg(&st->n_list);
        return z;
    }
    const int q = pass - 1;                                  // the digit to settle
    s_hist[threadIdx.x] = __ldcg(&st->hist[q][threadIdx.x]);
    if (threadIdx.x == 0) {
        SelState t;
        const SelState *g = &st->sel[q];
        t.pre_hi = __ldcg(&g->pre_hi); t.pre_lo = __ldcg(&g->pre_lo);
        t.mask_hi = __ldcg(&g->mask_hi); t.mask_lo = __ldcg(&g->mask_lo);
        t.k_rem = __ldcg(&g->k_rem); t.n_in = __ldcg(&g->n_in);
        t.n_match = __ldcg(&g->n_match); t.cur = __ldcg(&g->cur);
        *s_sel = t;
    }
    const unsigned long long hi_and = __ldcg(&st->hi_and), hi_or = __ldcg(&st->hi_or);
    const unsigned int n_out = __ldcg(&st->n_out[q]);
    __syncthreads();
    if (threadIdx.x < 32) {
        SelState t = *s_sel;
        const int lane = threadIdx.x;
        unsigned int d, run = 0, in_bin = t.n_match;
        if (digit_is_constant(q, hi_and, hi_or)) {
            d = (unsigned int)(hi_or >> (8 * (4 - q))) & 0xFFu;   // every candidate has it: nothing else changes
        } else {
            // lane l owns bins 8l .. 8l+7; the first bin at which the running count reaches k_rem
            unsigned int mine = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) mine += s_hist[lane * 8 + i];
            unsigned int inc = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                if (lane >= off) inc += v;
            }
            const unsigned int reach = __ballot_sync(0xFFFFFFFFu, inc >= t.k_rem);
            const int owner = reach ? __ffs(reach) - 1 : 31;
            run = inc - mine; d = 255;
            if (lane == owner) {
                for (int i = 0; i < 8; ++i) {
                    if (run + s_hist[lane * 8 + i] >= t.k_rem) { d = lane * 8 + i; break; }
                    run += s_hist[lane * 8 + i];
                }
                if (d == 255u && !reach) run = inc;          // counts fell short: everything below the last bin
                in_bin = s_hist[d];
            }
            d = __shfl_sync(0xFFFFFFFFu, d, owner);
            run = __shfl_sync(0xFFFFFFFFu, run, owner);
            in_bin = __shfl_sync(0xFFFFFFFFu, in_bin, owner);
            // the pass copied its matching candidates if that at least halved a list worth copying
            if (2u * t.n_match <= t.n_in && t.n_in > 1024u) { t.cur = t.cur == 1u ? 2u : 1u; t.n_in = n_out; }
        }
        if (lane == 0) {
            t.k_rem -= run;
            t.n_match = in_bin;
            if (q < 5) {
                t.pre_hi |= (unsigned long long)d << (8 * (4 - q));
                t.mask_hi |= 0xFFull << (8 * (4 - q));
            } else {
                t.pre_lo |= (unsigned long long)d << (8 * (12 - q));
                t.mask_lo |= 0xFFull << (8 * (12 - q));
            }
            *s_sel = t;
        }
    }
    __syncthreads();
    return *s_sel;
}

// Pass `pass` of the radix select over the current candidate list: histogram of digit `pass`
// over the candidates that match the digits decided so far. If those are at most half of the
// list, they are copied into the other scratch list on the way (the next pass reads that one).
__global__ void trim_hist_kernel(int pass, int64_t cap, void *lists, TrimState *st)
{
    __shared__ unsigned int s_hist[256];
    __shared__ unsigned int s_warp[32];
    __shared__ unsigned int s_base;
    __shared__ SelState s_sel;
    chain_wait();
    if (__ldcg(&st->n_list) == 0u) return;                   // nothing to find out: every block leaves
    const SelState S = select_state(pass, st, s_hist, &s_sel);
    if (blockIdx.x == 0 && threadIdx.x == 0) st->sel[pass] = S;
    if (digit_is_constant(pass, __ldcg(&st->hi_and), __ldcg(&st->hi_or))) return;   // the next pass fills it in
    __syncthreads();
    s_hist[threadIdx.x] = 0u;
    __syncthreads();
    const TrimLists L = trim_lists(lists, cap);
    const bool copy = 2u * S.n_match <= S.n_in && S.n_in > 1024u;   // short lists are not worth the copy
    const unsigned long long *in_hi = S.cur == 0u ? L.r_hi : L.l_hi[S.cur - 1u];
    const unsigned long long *in_lo = S.cur == 0u ? L.r_key : L.l_lo[S.cur - 1u];
    const unsigned int dst = S.cur == 1u ? 1u : 0u;          // scratch list 2 if list 1 is the input, else list 1
    unsigned long long *out_hi = L.l_hi[dst], *out_lo = L.l_lo[dst];
    // two entries per thread and iteration, both loads issued before the first use
    const unsigned int per_iter = gridDim.x * blockDim.x * 2u;
    for (unsigned int i0 = blockIdx.x * blockDim.x * 2u; i0 < S.n_in; i0 += per_iter) {
        const unsigned int i = i0 + threadIdx.x;
        const unsigned int j = i + blockDim.x;
        unsigned long long hi[2] = {0ull, 0ull}, lo[2] = {0ull, 0ull};
        bool ok[2] = {i < S.n_in, j < S.n_in};
        if (ok[0]) { hi[0] = __ldcg(in_hi + i); lo[0] = __ldcg(in_lo + i); }
        if (ok[1]) { hi[1] = __ldcg(in_hi + j); lo[1] = __ldcg(in_lo + j); }
        unsigned int n = 0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            ok[e] = ok[e] && (hi[e] & S.mask_hi) == S.pre_hi && (lo[e] & S.mask_lo) == S.pre_lo;
            if (ok[e]) {
                // scores are heavily tied (most digits are equal across the table): one
                // shared-memory add per distinct digit of the warp, not one per entry
                const unsigned int d = digit_of(pass, hi[e], lo[e]);
                const unsigned int peers = __match_any_sync(__activemask(), d);
                if ((int)(__ffs(peers) - 1) == (int)(threadIdx.x & 31)) atomicAdd(&s_hist[d], (unsigned int)__popc(peers));
                ++n;
            }
        }
        if (copy) {                                          // the same for every thread of the grid
            unsigned int total;
            unsigned int at = block_offsets(n, s_warp, total);
            if (threadIdx.x == 0) s_base = total ? atomicAdd(&st->n_out[pass], total) : 0u;
            __syncthreads();
            at += s_base;
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (ok[e]) { out_hi[at] = hi[e]; out_lo[at] = lo[e]; ++at; }
        }
    }
    __syncthreads();
    if (s_hist[threadIdx.x]) atomicAdd(&st->hist[pass][threadIdx.x], s_hist[threadIdx.x]);
}

// The listed entries that stay, and the survivors that were not in the group their run hashes to, go into the new table;
// which slot of its group an entry gets depends on timing, the set of entries does not. `held`: behind trim_select_kernel,
// which has placed lists of at most so many entries itself (then one block waits for it, so that what waits for this launch
// waits for it too); 0: behind the chain of histograms.
__global__ void __launch_bounds__(TRIM_THREADS)
trim_place_kernel(const Table from, const Table to, int64_t cap, void *lists, TrimState *st, unsigned int held)
{
    __shared__ unsigned int s_hist[256];
    __shared__ SelState s_sel;
    asm volatile("griddepcontrol.launch_dependents;");
    const TrimLists L = trim_lists(lists, cap);
    const unsigned int i0 = blockIdx.x * TRIM_THREADS + threadIdx.x, stride = gridDim.x * TRIM_THREADS;
    unsigned int n = 0u;
    unsigned long long hi = 0ull;
    Entry en = {};
    const auto load = [&](unsigned int i) { hi = __ldcg(L.r_hi + i); en = from.load(__ldcg(L.r_slot + i)); };
    if (held) {                                             // the list was complete when trim_select_kernel let this kernel start
        n = __ldcg(&st->n_list);
        if (n <= held) {
            if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
            return;
        }
        if (i0 < n) load(i0);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!held && blockIdx.x == 0) st->bins[threadIdx.x] = 0u;   // for the next trim
    unsigned long long thr_hi, thr_lo;
    if (held) {
        thr_hi = __ldcg(&st->thr_hi); thr_lo = __ldcg(&st->thr_lo);
    } else {
        n = __ldcg(&st->n_list);
        if (n > 0u) {                                       // block-uniform
            const SelState S = select_state(PASSES, st, s_hist, &s_sel);
            thr_hi = S.pre_hi; thr_lo = S.pre_lo;
            if (i0 < n) load(i0);
            if (i0 == 0) st->next_oldest = (unsigned int)thr_hi;
        }
    }
    for (unsigned int i = i0; i < n; i += stride) {
        if (i != i0) load(i);
        if (hi > thr_hi || (hi == thr_hi && en.key > thr_lo)) place_entry(to, cap, en);   // the others are among the k first: dropped
    }
    const unsigned int late = __ldcg(&st->n_late);
    for (unsigned int i = i0; i < late; i += stride) place_entry(to, cap, from.load(__ldcg(L.r_slot + (cap - 1 - (int64_t)i))));
}

__global__ void trim_end_kernel(TrimState *st)
{
    chain_wait();
    st->size -= st->k; st->k = 0u; st->oldest = st->next_oldest;
}

#define OD_CUDA(call)                                  \
    do {                                               \
        cudaError_t e__ = (call);                      \
        if (e__ != cudaSuccess) return OD_ERR_CUDA;    \
    } while (0)

struct Guard {
    int prev; bool ok;
    explicit Guard(int dev) : prev(-1), ok(false) { if (cudaGetDevice(&prev) == cudaSuccess) ok = cudaSetDevice(dev) == cudaSuccess; }
    ~Guard() { if (prev >= 0) cudaSetDevice(prev); }
};

template <typename T>
int32_t alloc_zero(T **p, size_t n)
{
    *p = nullptr;
    cudaError_t e = cudaMalloc((void **)p, (n ? n : 1) * sizeof(T));
    if (e == cudaErrorMemoryAllocation) return OD_ERR_NOMEM;
    if (e != cudaSuccess) return OD_ERR_CUDA;
    return cudaMemset(*p, 0, (n ? n : 1) * sizeof(T)) == cudaSuccess ? OD_OK : OD_ERR_CUDA;
}

// Room for the tying keys in a block's shared memory: a slice of the entries that one insertion
// leaves over the bound.
unsigned int select_room(const od_ctx *c, int blocks)
{
    return (unsigned int)((c->dyn_max + c->dyn_max_insert + blocks - 1) / blocks);
}
constexpr unsigned int SELECT_ROOM_MAX = 24 * 1024;         // 192 KB

void select_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, const od_ctx *c, int blocks)
{
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3(SELECT_THREADS);
    cfg.dynamicSmemBytes = (size_t)select_room(c, blocks) * 8;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
}

// Groups of a half-warp at a time in the two passes over the table: as few as leave two blocks to a multiprocessor at one,
// four at two (an insertion and a trim with 1, 2 and 4: 4096 entries and 512 new ones 16.0, 16.6 and 18.4 us, 16000 and 256 by LFU
// 28.8, 29.6 and 32.4, 32768 and 4096 19.7, 20.2 and 22.0, 65536 and 2048 19.9, 18.7 and 20.3, 262144 and 16384 41.6, 38.8 and 37.4).
int trim_quad(const od_ctx *c)
{
    const int64_t blocks = (c->cap / OD_GROUP + TRIM_HALVES - 1) / TRIM_HALVES;   // with one
    return blocks <= c->sm_count * 2 ? 1 : blocks <= c->sm_count * 8 ? 2 : 4;
}

// Blocks of the one-launch select, 0 = the table is too large for it: the keys of a list of all its entries have to fit in
// the blocks' shared memory (16 blocks: 393216 entries; 196608 where clusters of 16 are not to be had). As few as give every
// entry of the table a thread of its own: by LFU the list is most of the table as a rule (16000 entries, 256 new ones, an
// insertion and a trim: 35.4 us with two entries a thread, 32.4 so).
int select_blocks(const od_ctx *c)
{
    if (cudaFuncSetAttribute(trim_select_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(trim_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SELECT_ROOM_MAX * 8) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int64_t entries = c->dyn_max + c->dyn_max_insert;
    const int64_t want = (entries + SELECT_THREADS - 1) / SELECT_THREADS;
    int blocks = 1, best = 0;
    for (; blocks <= SELECT_MAX_BLOCKS; blocks *= 2) {
        if (select_room(c, blocks) > SELECT_ROOM_MAX) continue;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        select_config(cfg, attr, c, blocks);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, trim_select_kernel, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            continue;
        }
        best = blocks;
        if (blocks >= want) break;
    }
    return best;
}

}  // namespace

void od_cache_free_dynamic(od_ctx *c)
{
    void *ptrs[] = {c->d_stamp, c->d_freq, c->d_born, c->d_keys2, c->d_vals2, c->d_stamp2, c->d_freq2,
                    c->d_born2, c->d_fill, c->d_fill2, c->d_owner, c->d_cand_slot, c->d_trim, c->d_trim_lists};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    c->d_stamp = c->d_freq = c->d_born = c->d_stamp2 = c->d_freq2 = c->d_born2 = c->d_owner = nullptr;
    c->d_fill = c->d_fill2 = nullptr;
    c->d_keys2 = nullptr; c->d_vals2 = nullptr; c->d_cand_slot = nullptr; c->d_trim = nullptr;
    c->d_trim_lists = nullptr;
    c->dyn = false;
}

extern "C" {

int32_t od_cache_configure(od_ctx *c, int64_t max_entries, int32_t policy, int32_t max_insert)
{
    if (!c || max_entries < 1 || max_entries > ((int64_t)1 << 28) || max_insert < 1 ||
        max_insert > (1 << 24) || (policy != 0 && policy != 1))
        return OD_ERR_INVALID_ARG;
    if (c->v_q > 65535) return OD_ERR_UNSUPPORTED;           // a run packs 16 bits per id
    Guard g(c->device);
    if (!g.ok) return OD_ERR_CUDA;
    OD_CUDA(cudaDeviceSynchronize());
    od_cache_free_dynamic(c);
    if (c->d_keys) { cudaFree(c->d_keys); c->d_keys = nullptr; }
    if (c->d_vals) { cudaFree(c->d_vals); c->d_vals = nullptr; }
    c->cap = 0;
    int64_t cap = 64;
    while (cap < 2 * (max_entries + max_insert)) cap <<= 1;  // load stays under 1/2 even before a trim
    int32_t st = alloc_zero(&c->d_keys, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_vals, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_stamp, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_freq, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_born, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_keys2, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_vals2, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_stamp2, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_freq2, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_born2, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_fill, fill_words(cap));
    if (st == OD_OK) st = alloc_zero(&c->d_fill2, fill_words(cap));
    if (st == OD_OK) st = alloc_zero(&c->d_owner, (size_t)cap);
    if (st == OD_OK) st = alloc_zero(&c->d_cand_slot, (size_t)max_insert);
    TrimState *ts = nullptr;
    if (st == OD_OK) st = alloc_zero(&ts, 1);
    c->d_trim = ts;
    unsigned char *tl = nullptr;
    if (st == OD_OK) st = alloc_zero(&tl, (size_t)cap * TRIM_LIST_BYTES_PER_SLOT);
    c->d_trim_lists = tl;
    if (st != OD_OK) { od_cache_free_dynamic(c); return st; }
    OD_CUDA(cudaMemset(c->d_vals, 0xFF, (size_t)cap * sizeof(int32_t)));    // -1: no value
    OD_CUDA(cudaMemset(c->d_vals2, 0xFF, (size_t)cap * sizeof(int32_t)));
    OD_CUDA(cudaMemset(c->d_owner, 0xFF, (size_t)cap * sizeof(uint32_t)));
    c->cap = cap;
    c->table_written = true;
    c->dyn = true; c->dyn_policy = policy; c->dyn_max = max_entries; c->dyn_max_insert = max_insert;
    c->clock = 0;
    c->trim_blocks = select_blocks(c);
    return OD_OK;
}

int32_t od_cache_set_clock(od_ctx *c, uint32_t clock)
{
    if (!c) return OD_ERR_INVALID_ARG;
    if (!c->dyn) return OD_ERR_STATE;
    c->clock = clock;
    return OD_OK;
}

int32_t od_cache_insert(od_ctx *c, int32_t N, const int32_t *runs, const int32_t *len,
                        const int32_t *target, void *stream)
{
    if (!c || N < 0) return OD_ERR_INVALID_ARG;
    if (!c->dyn) return OD_ERR_STATE;
    if (N > c->dyn_max_insert) return OD_ERR_INVALID_ARG;
    if (N == 0) return OD_OK;
    if (!runs || !len || !target) return OD_ERR_INVALID_ARG;
    Guard g(c->device);
    if (!g.ok) return OD_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    c->table_written = true;
    const int threads = 128, blocks = (N + threads - 1) / threads;
    const bool pdl = c->opt_pdl != 0;
    OD_CUDA(chain_launch(insert_claim_kernel, (unsigned)blocks, (unsigned)threads, s, pdl, N, c->v_q, c->v_p, runs, len,
                         target, (unsigned long long *)c->d_keys, (const int32_t *)c->d_vals, c->cap,
                         c->d_owner, c->d_cand_slot, c->d_fill, (TrimState *)c->d_trim));
    OD_CUDA(chain_launch(insert_commit_kernel, (unsigned)blocks, (unsigned)threads, s, pdl, N, target, c->d_vals,
                         c->d_stamp, c->d_freq, c->d_born, c->d_owner, (const int32_t *)c->d_cand_slot,
                         c->clock, (TrimState *)c->d_trim));
    OD_CUDA(cudaGetLastError());
    return OD_OK;
}

int32_t od_cache_trim(od_ctx *c, void *stream)
{
    if (!c) return OD_ERR_INVALID_ARG;
    if (!c->dyn) return OD_ERR_STATE;
    Guard g(c->device);
    if (!g.ok) return OD_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    c->table_written = true;
    TrimState *st = (TrimState *)c->d_trim;
    // one resident wave at most, and no more blocks than have anything to do
    const int64_t most = c->sm_count * 4;
    const int quad = trim_quad(c);
    const unsigned passes = (unsigned)std::min<int64_t>(most, (c->cap / OD_GROUP + quad * TRIM_HALVES - 1) / (quad * TRIM_HALVES));
    const bool pdl = c->opt_pdl != 0;
    const int blocks = c->trim_blocks;                      // 0: the select is a chain of launches
    // whether the list may be longer than what the select's cluster places by itself
    const int64_t entries = c->dyn_max + c->dyn_max_insert;
    const bool follow = !blocks || entries > (int64_t)blocks * SELECT_THREADS;
    // (without a long list that launch costs a trim 0.9 us with four blocks to a multiprocessor, 0.7 with two, 0.5 with one; with
    // 262144 entries to place four and two take the same, one 2.5 us more)
    const unsigned place = (unsigned)std::min<int64_t>(blocks ? c->sm_count * 2 : most, (entries + TRIM_THREADS - 1) / TRIM_THREADS);
    const Table from = {(unsigned long long *)c->d_keys, c->d_vals, c->d_stamp, c->d_freq, c->d_born, c->d_fill};
    const Table to = {(unsigned long long *)c->d_keys2, c->d_vals2, c->d_stamp2, c->d_freq2, c->d_born2, c->d_fill2};
    if (!blocks) OD_CUDA(chain_launch(trim_begin_kernel, 1u, 256u, s, pdl, st));
    const auto count = quad == 4 ? trim_count_kernel<4> : quad == 2 ? trim_count_kernel<2> : trim_count_kernel<1>;
    const auto split = quad == 4 ? trim_split_kernel<4> : quad == 2 ? trim_split_kernel<2> : trim_split_kernel<1>;
    OD_CUDA(chain_launch(count, passes, (unsigned)TRIM_THREADS, s, pdl, c->dyn_policy, c->clock, from.vals,
                         c->dyn_policy == 0 ? from.stamp : from.freq, from.born, c->cap, st));
    OD_CUDA(chain_launch(split, passes, (unsigned)TRIM_THREADS, s, pdl, c->dyn_policy, c->clock,
                         (unsigned int)c->dyn_max, from, to, c->cap, c->d_trim_lists, st));
    if (blocks) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        select_config(cfg, attr, c, blocks);
        cfg.stream = s;
        cfg.numAttrs = pdl ? 2 : 1;
        OD_CUDA(cudaLaunchKernelEx(&cfg, trim_select_kernel, select_room(c, blocks), from, to, c->cap, c->d_trim_lists, st,
                                   follow ? 1 : 0));
    } else {
        for (int pass = 0; pass < PASSES; ++pass)
            OD_CUDA(chain_launch(trim_hist_kernel, (unsigned)c->sm_count, 256u, s, pdl, pass, c->cap,
                                 c->d_trim_lists, st));
    }
    if (follow)
        OD_CUDA(chain_launch(trim_place_kernel, place, (unsigned)TRIM_THREADS, s, pdl, from, to, c->cap, c->d_trim_lists,
                             st, (unsigned)blocks * SELECT_THREADS));
    if (!blocks) OD_CUDA(chain_launch(trim_end_kernel, 1u, 1u, s, pdl, st));
    // the rebuilt table is the table for every call enqueued from now on
    std::swap(c->d_keys, c->d_keys2); std::swap(c->d_vals, c->d_vals2);
    std::swap(c->d_stamp, c->d_stamp2); std::swap(c->d_freq, c->d_freq2); std::swap(c->d_born, c->d_born2);
    std::swap(c->d_fill, c->d_fill2);
    return OD_OK;
}

int32_t od_cache_stats(od_ctx *c, int64_t *entries, int64_t *invalid, int64_t *dropped)
{
    if (!c) return OD_ERR_INVALID_ARG;
    if (!c->dyn) return OD_ERR_STATE;
    Guard g(c->device);
    if (!g.ok) return OD_ERR_CUDA;
    OD_CUDA(cudaDeviceSynchronize());
    unsigned int size = 0, inv = 0, drop = 0;
    const char *st = (const char *)c->d_trim;
    OD_CUDA(cudaMemcpy(&size, st + offsetof(TrimState, size), sizeof(size), cudaMemcpyDeviceToHost));
    OD_CUDA(cudaMemcpy(&inv, st + offsetof(TrimState, invalid), sizeof(inv), cudaMemcpyDeviceToHost));
    OD_CUDA(cudaMemcpy(&drop, st + offsetof(TrimState, dropped), sizeof(drop), cudaMemcpyDeviceToHost));
    if (entries) *entries = size;
    if (invalid) *invalid = inv;
    if (dropped) *dropped = drop;
    return OD_OK;
}

int32_t od_cache_dump(od_ctx *c, int64_t max_out, int32_t *runs, int32_t *len, int32_t *target,
                      uint32_t *stamp, uint32_t *freq, int64_t *n_out)
{
    if (!c || !n_out || max_out < 0) return OD_ERR_INVALID_ARG;
    if (!c->dyn) return OD_ERR_STATE;
    Guard g(c->device);
    if (!g.ok) return OD_ERR_CUDA;
    OD_CUDA(cudaDeviceSynchronize());
    const size_t cap = (size_t)c->cap;
    std::vector<uint64_t> keys(cap);
    std::vector<int32_t> vals(cap);
    std::vector<uint32_t> st(cap), fr(cap);
    OD_CUDA(cudaMemcpy(keys.data(), c->d_keys, cap * 8, cudaMemcpyDeviceToHost));
    OD_CUDA(cudaMemcpy(vals.data(), c->d_vals, cap * 4, cudaMemcpyDeviceToHost));
    OD_CUDA(cudaMemcpy(st.data(), c->d_stamp, cap * 4, cudaMemcpyDeviceToHost));
    OD_CUDA(cudaMemcpy(fr.data(), c->d_freq, cap * 4, cudaMemcpyDeviceToHost));
    int64_t n = 0;
    for (size_t s = 0; s < cap; ++s) {
        if (keys[s] == 0 || vals[s] < 0) continue;
        if (n < max_out && runs && len && target) {
            int L = 0;
            for (int j = 0; j < OD_NGRAM_MAX; ++j) {
                const uint32_t f = (uint32_t)(keys[s] >> (16 * j)) & 0xFFFFu;
                runs[n * OD_NGRAM_MAX + j] = f ? (int32_t)f - 1 : -1;
                if (f) L = j + 1;
            }
            len[n] = L; target[n] = vals[s];
            if (stamp) stamp[n] = st[s];
            if (freq) freq[n] = fr[s];
        }
        ++n;
    }
    *n_out = n;
    return OD_OK;
}

}  // extern "C"
