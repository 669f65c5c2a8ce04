// Shared declarations of the CUDA library: the context, device helpers
// (Philox4x32-10, logit decoding, (max, sum) pair algebra) and the kernel
// launchers implemented in od_map.cu / od_verify.cu / od_sample.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "omnidraft.h"

#define OD_WARP 32
#define OD_GROUP 32                 // slots of one hash-table probe group
#define OD_SAMPLE_TILE 256          // elements of one residual-sampler tile (8 per lane of a warp)
#define OD_SAMPLE_THREADS 256       // of the vocabulary shards' sampler; a shard's mass by blocks of 256, 512 or 1024
#define OD_SHARD_SIZES 3
#define OD_SHARD_MAX_THREADS (OD_SAMPLE_THREADS << (OD_SHARD_SIZES - 1))
#define OD_SAMPLE_LEVELS 8          // 1, 2, 3, 4, 5, 6, 8 or 16 blocks draw for one sequence
#define OD_SAMPLE_MAX_PARTS 16      // (over 8: a non-portable cluster)
#define OD_SAMPLE_MAX_SLOTS 53248   // mapped ids of a part: 208 KB of shared memory
#define OD_SAMPLE_SMEM_MAX (200 * 1024)  // dynamic shared memory the sampler may ask for: 8 bytes per tile
#define OD_VERIFY_SEG_MAX 64        // most segments (partials) one logit row is cut into
#define OD_VERIFY_MAX_B 2048        // sequences per od_verify launch (longer batches go in slices)

#define OD_DISTILL_LEVELS 4         // the distillation kernel cuts the draft ids into 1, 2, 4 or 8 chunks
#define OD_DISTILL_MAX_CHUNKS 8     // (a portable cluster)
#define OD_DISTILL_MAX_CHUNK_IDS 56320   // 220 KB of shared memory

struct od_ctx {
    int device;
    int32_t v_q, v_p, max_batch, max_k;
    int sm_count;

    // vocabulary map (device)
    int32_t *d_vocab_map;           // [v_q]
    int32_t *d_inv_map;             // [v_p], -1 outside the image
    void *d_distill_lists;          // gather lists of the distillation kernel (od_distill_lists)
    void *d_sample_lists;           // and of the sampler (od_sample_lists)
    int32_t sample_slots[OD_SAMPLE_LEVELS];   // most mapped ids of a part
    int32_t sample_clusters[OD_SAMPLE_LEVELS];   // clusters of the sampler that are resident at a time
    int32_t step_clusters[OD_SAMPLE_LEVELS];     // of the whole step in one launch: a multiprocessor to each block
    int32_t shard_clusters[OD_SHARD_SIZES][OD_SAMPLE_MAX_PARTS + 1];   // of a shard's mass, by threads and blocks
    int32_t distill_few_clusters[OD_DISTILL_LEVELS];   // of the distillation loss with two blocks to a multiprocessor
    bool have_map;
    bool distill_lists;             // some map had gather lists: every later one has the distillation kernel's
    // The map's serial number. A launch is laid out for the map of its time (where ids are shared, how many
    // are staged); a kernel that finds another number on the device was replayed from a CUDA graph
    // captured before od_set_vocab_map, and looks every id up in the maps instead.
    int32_t map_serial, *d_map_serial;
    int64_t n_mapped;               // draft ids with a direct map
    bool map_same_ids;              // every draft id is mapped to the target id of the same number

    // n-gram cache: open addressing over groups of 32 slots
    uint64_t *d_keys;               // [cap], 0 = empty
    int32_t *d_vals;                // [cap]
    int64_t cap;                    // power of two, multiple of 32, or 0

    // online cache (od_cache_configure): per-slot access data of the current table, a
    // second table that od_cache_trim rebuilds into, and the scratch of insert and trim
    bool dyn;
    int32_t dyn_policy;             // 0 = LRU, 1 = LFU
    int64_t dyn_max;                // entries kept by a trim
    int32_t dyn_max_insert;         // largest batch of od_cache_insert
    uint32_t clock;                 // stamp of accesses and insertions
    uint32_t *d_stamp, *d_freq, *d_born;            // [cap]
    uint64_t *d_keys2; int32_t *d_vals2;            // [cap] spare table
    uint32_t *d_stamp2, *d_freq2, *d_born2;
    uint32_t *d_fill, *d_fill2;     // [cap / 32] slots taken in each group, of the table and of the spare one
    uint32_t *d_owner;              // [cap] first-wins claims of a batch (0xFFFFFFFF = none)
    int32_t *d_cand_slot;           // [dyn_max_insert]
    void *d_trim;                   // trim / size state (device)
    int32_t trim_blocks;            // blocks of the one-launch select, 0 = the table is too large for it
    void *d_trim_lists;             // trim scratch: the listed entries and two candidate lists, 52 bytes per slot

    // od_verify scratch
    float4 *d_partials;             // [rows][OD_VERIFY_SEG_MAX] (c, sum, max, -), rows of one launch

    // od_sample_residual scratch
    double *d_tile_sums;            // [max_batch * tiles_per_row] value of each tile
    int32_t tiles_per_row;

    // options
    int64_t opt_verify_grid;        // blocks of the stream kernel (0 = one per multiprocessor)
    int64_t opt_early_inputs;       // the caller promises complete inputs: od_verify reads logits and temperatures, the
                                    // translation kernel the proposal, before griddepcontrol.wait
    int64_t opt_sample_tiles_per_warp;
    int64_t opt_pdl;                // launch with programmatic stream serialization

    // set by the entry points for the verify launch that follows: space A may be streamed early
    bool verify_early;
    bool table_written;             // a kernel that writes the n-gram table was launched since the last translation kernel

    // The last launch on this context that a draw's inputs depend on was a verification's, which let the next kernel
    // start only after the translation was complete: the draw behind it may read the translation's outputs before
    // griddepcontrol.wait. Not behind a translation, nor behind a fetch of rows that the draw reads, nor behind
    // anything the library did not launch itself for this step.
    bool translation_complete;

    // last launch info
    int64_t info[4];

    // od_step_host staging (device)
    bool host_reserved;
    int32_t host_dtype;
    void *s_logits;
    float *s_q_rows, *s_q_sel, *s_temperature;
    int32_t *s_draft_ids, *s_draft_len;
    uint64_t *s_seed;
    int32_t *s_tgt_ids, *s_span_start, *s_span_len, *s_m, *s_n_acc, *s_n_draft, *s_token;
    float *s_q_prime, *s_row_max, *s_row_sum, *s_p_sel, *s_ratio, *s_mass;
    uint8_t *s_tail;
    uint32_t *s_vflags, *s_sflags;
};

// ---- launchers ------------------------------------------------------------
cudaError_t od_launch_map(od_ctx *c, int32_t B, int32_t K_max, const int32_t *draft_ids,
                          const int32_t *draft_len, const float *q_sel, int32_t *tgt_ids,
                          float *q_prime, int32_t *span_start, int32_t *span_len, int32_t *m,
                          uint8_t *tail_kind, uint32_t *counters, bool early, bool release_early, cudaStream_t s);

cudaError_t od_launch_verify(od_ctx *c, int32_t B, int32_t K_max, const void *logits,
                             int32_t dtype, int64_t row_stride, int64_t seq_stride,
                             const int32_t *tgt_ids, const float *q_prime,
                             const int32_t *span_len, const int32_t *m,
                             const float *temperature, const uint64_t *seed, uint64_t step,
                             float *row_max, float *row_sum, float *p_sel, float *ratio,
                             int32_t *n_accepted, int32_t *n_draft_accepted,
                             uint32_t *flags, cudaStream_t s);


// od_step: the streaming pass of step 2 alone (no decide kernel), and what the sampler then needs
// to take step 2's decisions itself: the split of the pass and where step 2's outputs go.
struct od_fused_verify {
    int32_t W, n_chunks, span_min, span_a, seg_warps;
    float *row_max, *row_sum, *p_sel, *ratio;
    int32_t *n_accepted, *n_draft_accepted;
    uint32_t *flags;
};
// od_step and od_verify in one launch (od_step.cu), where a batch's clusters are all resident at a time
bool od_step_one_launch(const od_ctx *c, int32_t B, int32_t K_max, int32_t dtype);
bool od_verify_one_launch(const od_ctx *c, int32_t B, int32_t K_max, int32_t v_len, int32_t dtype);
cudaError_t od_step_prepare_device(int32_t *clusters);
cudaError_t od_launch_step(od_ctx *c, int32_t B, int32_t K_max, const int32_t *draft_ids, const int32_t *draft_len,
                           const float *q_sel, const float *q_rows, const void *logits, int32_t dtype, int64_t row_stride,
                           int64_t seq_stride, const float *temperature, const uint64_t *seed, uint64_t step, int32_t *tgt_ids,
                           float *q_prime, int32_t *span_start, int32_t *span_len, int32_t *m, uint8_t *tail_kind,
                           uint32_t *counters, const od_fused_verify *fuse, int32_t *out_token, float *resid_mass, uint32_t *flags,
                           bool early, cudaStream_t s);
cudaError_t od_launch_verify_rows(od_ctx *c, int32_t B, int32_t K_max, const void *logits, int32_t dtype, int64_t row_stride,
                                  int64_t seq_stride, const int32_t *tgt_ids, const float *q_prime, const int32_t *span_len,
                                  const int32_t *m, const float *temperature, const uint64_t *seed, uint64_t step,
                                  const od_fused_verify *out, bool early, cudaStream_t s);
cudaError_t od_launch_shard_rows(od_ctx *c, int32_t B, int32_t K_max, int32_t shard_lo, int32_t shard_len, const void *logits,
                                 int32_t dtype, int64_t row_stride, int64_t seq_stride, const int32_t *tgt_ids, const int32_t *m,
                                 const float *temperature, float *stats, bool early, cudaStream_t s);
// od_step_host (od_host.cu): page-locked buffers that the device reads itself, where that is not slower than copies
bool od_host_better_copied(const od_ctx *c, int32_t B, int32_t K_max, const int32_t *draft_len, size_t lrow, size_t qrow);
bool od_host_rows_readable(const void *logits, size_t logits_bytes, const void *q_rows, size_t q_bytes, const char **d_logits,
                           const char **d_q_rows);
cudaError_t od_launch_fetch_logits(od_ctx *c, int32_t B, int32_t K_max, const char *src, size_t row_bytes, cudaStream_t s);
cudaError_t od_launch_fetch_drafter(od_ctx *c, int32_t B, int32_t K_max, const char *src, cudaStream_t s);
int32_t od_verify_slice(int32_t K_max, int32_t v_len, int32_t dtype);   // sequences one stream launch takes
cudaError_t od_launch_verify_stream(od_ctx *c, int32_t B, int32_t K_max, const void *logits, int32_t dtype,
                                    int64_t row_stride, int64_t seq_stride, const int32_t *m,
                                    const float *temperature, od_fused_verify *plan, cudaStream_t s);

cudaError_t od_launch_sample(od_ctx *c, int32_t B, int32_t K_max, const void *logits,
                             int32_t dtype, int64_t row_stride, int64_t seq_stride,
                             const float *row_max, const float *row_sum, const float *q_rows,
                             const int32_t *draft_ids, const int32_t *tgt_ids,
                             const float *q_prime, const int32_t *span_start,
                             const int32_t *span_len, const int32_t *m,
                             const uint8_t *tail_kind, const int32_t *n_accepted,
                             const float *temperature, const uint64_t *seed, uint64_t step,
                             int32_t *out_token, float *resid_mass, uint32_t *flags,
                             cudaStream_t s, const od_fused_verify *fuse = nullptr);

size_t od_sample_smem_bytes(int32_t ntiles);            // dynamic shared memory of the shard sampler's kernel
// opt in to the dynamic shared memory and the cluster size that the sampler's kernels may ask for
cudaError_t od_sample_prepare_device(int32_t *clusters, int32_t (*shard_clusters)[OD_SAMPLE_MAX_PARTS + 1]);   // resident at a time

// The pairs of a vocabulary map in target-id order (host).
struct OdMappedIds {
    std::vector<int32_t> target, draft;
};

// The lists below: pads the open group of 32 words at `next` and gives the groups from `end` on their base.
inline void od_end_group(uint32_t *words, uint32_t *&next, int32_t *bases, int32_t base, int32_t &end)
{
    while ((next - words) % 32) *next++ = 0xFFFFu;
    for (; end < (next - words) / 32; ++end) bases[end] = base;
}

// What the sampler knows about the vocabulary map, one block of memory. The mapped target ids in
// order have ranks 0, 1, ...; a row's tiles are cut into 1, 2, 3, ... parts (the levels), and a
// part's mapped ids, in draft-id order, are a list in groups of 32: an entry is (draft id - the
// group's base) << 16 | (rank - the part's first rank), or 0xFFFF in the low half where the
// group has no more.
struct OdSampleLists {
    int64_t groups;                 // room for this many groups in each level
    uint32_t *word;                 // [levels][groups][32]
    int32_t *base;                  // [levels][groups]
    int32_t *part;                  // [levels][max parts][4] a part's groups within its level (the first, one past the last), first rank, the map's serial number
    uint32_t *octet;                // [ceil(v_p / 8)] of target ids 8i .. 8i+7: rank of the first mapped one << 8 | which are mapped
};
inline OdSampleLists od_sample_lists(void *base, int32_t v_q, int32_t v_p)
{
    OdSampleLists l;
    // a group ends full, or with 65536 draft ids, or with its part
    l.groups = ((int64_t)(v_q < v_p ? v_q : v_p) + 31) / 32 + OD_SAMPLE_MAX_PARTS * ((int64_t)v_q / 65536 + 2);
    l.word = (uint32_t *)base;
    l.part = (int32_t *)(l.word + OD_SAMPLE_LEVELS * l.groups * 32);
    l.base = l.part + OD_SAMPLE_LEVELS * OD_SAMPLE_MAX_PARTS * 4;
    l.octet = (uint32_t *)(l.base + OD_SAMPLE_LEVELS * l.groups);
    return l;
}
inline size_t od_sample_lists_bytes(int32_t v_q, int32_t v_p)
{
    const OdSampleLists l = od_sample_lists(nullptr, v_q, v_p);
    return (size_t)((uintptr_t)(l.octet + (v_p + 7) / 8) - (uintptr_t)nullptr);
}
// parts of a level, and the tiles of one
inline int32_t od_sample_parts(int level)
{
    const int32_t parts[OD_SAMPLE_LEVELS] = {1, 2, 3, 4, 5, 6, 8, 16};
    return parts[level];
}
inline int32_t od_sample_part_tiles(int32_t v_p, int level)
{
    const int32_t n = od_sample_parts(level);
    return ((v_p + OD_SAMPLE_TILE - 1) / OD_SAMPLE_TILE + n - 1) / n;
}
// host; slots: [levels] most mapped ids of a part
void od_sample_plan(int32_t v_q, int32_t v_p, const OdMappedIds &mapped, int32_t serial, void *out, int32_t *slots);

// vocabulary shards (columns [shard_lo, shard_lo + shard_len) of the rows on this GPU)
cudaError_t od_launch_verify_shard_stats(od_ctx *c, int32_t B, int32_t K_max, int32_t shard_lo,
                                         int32_t shard_len, const void *logits, int32_t dtype,
                                         int64_t row_stride, int64_t seq_stride, const int32_t *tgt_ids,
                                         const int32_t *m, const float *temperature, float *stats,
                                         cudaStream_t s);
cudaError_t od_launch_verify_shard_finish(od_ctx *c, int32_t B, int32_t K_max, int32_t n_shards,
                                          const float *stats_all, const int32_t *tgt_ids,
                                          const float *q_prime, const int32_t *span_len, const int32_t *m,
                                          const float *temperature, const uint64_t *seed, uint64_t step,
                                          float *row_max, float *row_sum, float *p_sel, float *ratio,
                                          int32_t *n_accepted, int32_t *n_draft_accepted, uint32_t *flags,
                                          cudaStream_t s);
cudaError_t od_launch_sample_shard_mass(od_ctx *c, int32_t B, int32_t K_max, int32_t shard_lo,
                                        int32_t shard_len, const void *logits, int32_t dtype,
                                        int64_t row_stride, int64_t seq_stride, const float *row_max,
                                        const float *row_sum, const float *q_rows, const int32_t *draft_ids,
                                        const int32_t *tgt_ids, const float *q_prime,
                                        const int32_t *span_start, const int32_t *span_len, const int32_t *m,
                                        const uint8_t *tail_kind, const int32_t *n_accepted,
                                        const float *temperature, double *mass, cudaStream_t s);
cudaError_t od_launch_sample_shard_pick(od_ctx *c, int32_t B, int32_t K_max, int32_t n_shards,
                                        int32_t shard_index, int32_t shard_lo, int32_t shard_len,
                                        const double *mass_all, const void *logits, int32_t dtype,
                                        int64_t row_stride, int64_t seq_stride, const float *row_max,
                                        const float *row_sum, const float *q_rows, const int32_t *draft_ids,
                                        const int32_t *tgt_ids, const float *q_prime,
                                        const int32_t *span_start, const int32_t *span_len, const int32_t *m,
                                        const uint8_t *tail_kind, const int32_t *n_accepted,
                                        const float *temperature, const uint64_t *seed, uint64_t step,
                                        int32_t *out_token, float *resid_mass, uint32_t *flags, cudaStream_t s);

cudaError_t od_launch_distill(od_ctx *c, int32_t B, int32_t K_max, const float *q_rows,
                              const int32_t *draft_ids, const int32_t *tgt_ids, const int32_t *span_start,
                              const int32_t *span_len, const int32_t *m, const void *logits, int32_t dtype,
                              int64_t row_stride, int64_t seq_stride, const float *row_max,
                              const float *row_sum, const float *p_sel, const float *temperature,
                              float lambda, int32_t lambda_mode, float *loss, float *grad, cudaStream_t s);

// The gather lists of the distillation kernel, one block of memory: per level (1, 2, 4, 8 chunks
// of the draft ids) the mapped ids chunk by chunk, in target-id order inside a chunk, in groups
// of 32: an entry is (target id - the group's base) << 16 | (draft id - the chunk's first), or
// 0xFFFF in the low half where the group has no more.
struct OdDistillLists {
    int64_t groups;                 // room for this many groups in each level, a multiple of the chunks
    uint32_t *word;                 // [levels][groups][32]
    int32_t *base;                  // [levels][groups]
    int32_t *ofs;                   // [levels][max chunks][2] a chunk's groups within its level: the first, one past the last
    uint32_t *bits;                 // [ceil(v_q / 32)] bit d: draft id d is mapped
};
inline OdDistillLists od_distill_lists(void *base, int32_t v_q, int32_t v_p)
{
    OdDistillLists l;
    // a group ends full, or with 65536 target ids, or with its chunk; a chunk is whole
    // multiples of 32 ids
    l.groups = OD_DISTILL_MAX_CHUNKS * (((int64_t)v_q + 255) / 256 + (int64_t)v_p / 65536 + 1);
    l.word = (uint32_t *)base;
    l.base = (int32_t *)(l.word + OD_DISTILL_LEVELS * l.groups * 32);
    l.ofs = l.base + OD_DISTILL_LEVELS * l.groups;
    l.bits = (uint32_t *)(l.ofs + OD_DISTILL_LEVELS * OD_DISTILL_MAX_CHUNKS * 2);
    return l;
}
inline size_t od_distill_lists_bytes(int32_t v_q, int32_t v_p)
{
    const OdDistillLists l = od_distill_lists(nullptr, v_q, v_p);
    return (size_t)((uintptr_t)(l.bits + (v_q + 31) / 32) - (uintptr_t)nullptr);
}
void od_distill_plan(int32_t v_q, int32_t v_p, const OdMappedIds &mapped, void *out);   // host
cudaError_t od_distill_prepare_device(int32_t v_q);
void od_distill_resident(int32_t *clusters);             // [levels]

void od_cache_free_dynamic(od_ctx *c);   // frees what od_cache_configure allocated beyond keys / vals

cudaError_t od_launch_exit(int32_t B, int32_t K_max, const float *head_logits, const int32_t *avail_len,
                           float gamma, int32_t *draft_len, float *reject_prob, uint32_t *flags, bool pdl,
                           cudaStream_t s);

// 64-bit key of a run of draft ids: (id + 1) in 16 bits per position, first id
// in the low bits. Never 0 for a non-empty run.
__host__ __device__ inline uint64_t od_pack_run(const int32_t *ids, int len)
{
    uint64_t k = 0;
    for (int j = 0; j < len; ++j) k |= (uint64_t)(uint32_t)(ids[j] + 1) << (16 * j);
    return k;
}

// 64-bit finaliser of MurmurHash3 (Appleby, public domain): spreads the packed
// key over the table's groups.
__host__ __device__ inline uint64_t od_hash64(uint64_t h)
{
    h ^= h >> 33; h *= 0xff51afd7ed558ccdULL;
    h ^= h >> 33; h *= 0xc4ceb9fe1a85ec53ULL;
    h ^= h >> 33;
    return h;
}

#ifdef __CUDACC__
// ---- Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) ----------------------
__device__ __forceinline__ uint32_t od_philox_word0(uint32_t c0, uint32_t c1, uint32_t c2,
                                                    uint32_t c3, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        uint32_t n0 = hi1 ^ c1 ^ k0;
        uint32_t n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return c0;
}

// uniform in [0,1) on the 24-bit grid for (seed, step, position, tag)
__device__ __forceinline__ float od_uniform(uint64_t seed, uint64_t step, uint32_t position,
                                            uint32_t tag)
{
    uint32_t w = od_philox_word0((uint32_t)step, (uint32_t)(step >> 32), position, tag,
                                 (uint32_t)seed, (uint32_t)(seed >> 32));
    return (float)(w >> 8) * (1.0f / 16777216.0f);
}

__device__ __forceinline__ float od_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Thread-block clusters: the barrier in its two halves, and a word of block `rank`'s shared memory, at the
// address of `p` in this block.
__device__ __forceinline__ void od_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void od_cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void od_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t od_cluster_address(const void *p, uint32_t rank)
{
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return at;
}
__device__ __forceinline__ void od_cluster_store(double *p, uint32_t rank, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(od_cluster_address(p, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ unsigned int od_cluster_load(const unsigned int *p, uint32_t rank)
{
    unsigned int v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(od_cluster_address(p, rank)) : "memory");
    return v;
}

// Packed fp32 pairs (one instruction for two lanes of arithmetic on sm_100).
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// acc += (exp2(lo*scale - c), exp2(hi*scale - c))
__device__ __forceinline__ uint64_t f2_exp_acc(uint64_t acc, float lo, float hi, uint64_t scale2, uint64_t nc2)
{
    float e0, e1;
    f2_unpack(f2_fma(f2_pack(lo, hi), scale2, nc2), e0, e1);
    return f2_add(acc, f2_pack(od_ex2(e0), od_ex2(e1)));
}

// (max, sum) of exp2((x - max) * scale): merge two partial pairs
__device__ __forceinline__ void od_pair_merge(float &m, float &s, float m2, float s2, float scale)
{
    float nm = fmaxf(m, m2);
    s = s * od_ex2((m - nm) * scale) + s2 * od_ex2((m2 - nm) * scale);
    m = nm;
}

__device__ __forceinline__ float od_bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float od_bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

template <int DTYPE>
__device__ __forceinline__ float od_load_logit(const void *row, int64_t t)
{
    if (DTYPE == OD_F32) return __ldg((const float *)row + t);
    uint16_t h = __ldg((const unsigned short *)row + t);
    return __uint_as_float((uint32_t)h << 16);
}
#endif  // __CUDACC__
