// A step, or its step 2, in ONE launch, for batches whose sequences' clusters are all resident at a time.
//
// Grid (P, B), clusters of P blocks of 16 warps, one to a multiprocessor; a cluster takes one sequence
// through everything and waits for no other. A block owns a slice of the target vocabulary (the same tiles
// that it draws from in step 3):
//   translation  by every block alike (warp s looks up the runs at offset s, then every warp walks the
//                proposal with shuffles); block 0 writes the outputs;
//   statistics   the block's slice of row 0, requested before the lookups, then of rows 1..m_b laid end to
//                end: a warp takes one contiguous run of units. Per row the warps' partials are merged
//                in shared memory, sent to every block of the cluster, and merged again behind one
//                cluster barrier: the reduction order depends on the slice alone;
//   decisions    by every warp alike (decide), block 0 writes them;
//   the draw     as in od_sample.cu.
// What it takes the place of is three launches (translation, streaming pass, sampler), each of which waits
// for the slowest block of the one before it, and writes and reads partials through L2. Bound by the chain of
// round trips: one sequence of 128256 bf16 ids, six tokens, 14.5 -> 12.4 us a step; of 32000 fp32 ids (stamps): 1.0 us to
// the proposal and the map, 0.9 to the pieces, 1.6 the rows, 1.5 the exchange, 0.6 the decisions, 1.6 the tiles, 0.9 the
// exchange of their sums, 1.5 the tile and the id.
#include <float.h>

#include "od_common.cuh"
#include "od_decide.cuh"
#include "od_draw.cuh"
#include "od_lookup.cuh"
#include "od_stream.cuh"

namespace {

struct StepArgs : SampleArgs {
    int32_t part_units, W;              // 512-byte units of a block's slice, of a row
    // translation
    const int32_t *draft_len;
    const float *q_sel;
    const uint64_t *keys;
    const int32_t *vals;
    int64_t cap;
    MapOut out;
    float4 *stats;                      // vocabulary shards: [row slot] (c, sum, max, x[t_i] or -inf)
    int32_t inputs_early, table_early;  // the inputs (the table) may be read before griddepcontrol.wait
};

constexpr int REC = (OD_MAX_K + 1) * CWARPS;                // partials: [row][warp], [row][block]
constexpr size_t REC_BYTES = 2 * REC * sizeof(float4);
static_assert(OD_SAMPLE_MAX_PARTS <= CWARPS, "one lane per block of the cluster");

__device__ __forceinline__ void cluster_store4(float4 *p, uint32_t rank, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};"
                 ::"r"(od_cluster_address(p, rank)), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// A block's slice [u0, u1) of a row, in units
struct Slice {
    int u0, u1, full;                   // full: units of a row that are whole
    uint32_t inv;                       // ceil(2^32 / units): f / units for f < 2^32 / units, without a division behind the walk
    __device__ __forceinline__ int units() const { return u1 - u0; }
    __device__ __forceinline__ int rows_before(int f) const { return units() > 1 ? (int)__umulhi((uint32_t)f, inv) : f; }
};
template <int DTYPE>
__device__ __forceinline__ Slice slice_of(const StepArgs &a, int part)
{
    Slice s;
    s.u0 = min(part * a.part_units, a.W);
    s.u1 = min(s.u0 + a.part_units, a.W);
    s.full = full_units_of<DTYPE>(a.v_p);
    s.inv = s.u1 > s.u0 ? 0xFFFFFFFFu / (uint32_t)(s.u1 - s.u0) + 1u : 0u;
    return s;
}
template <int DTYPE>
__device__ __forceinline__ const char *row_of(const StepArgs &a, int b, int r)
{
    return (const char *)a.logits + ((size_t)b * a.seq_stride + (size_t)r * a.row_stride) * (DTYPE == OD_BF16 ? 2 : 4);
}

// Units a warp requests at a time. fp32 rows have twice the bytes to each exponential: twice the loads in flight make
// a step faster where the rows come from HBM (inputs that change from pass to pass, sequences x K_max: 9 x 3, 152064 ids
// 18.4 -> 16.8 us; 24 x 4, 50001 17.9 -> 17.2; 15 x 4 14.3 -> 14.0; 1 x 4, 32000 9.2 -> 9.3), and 1 to 2 % slower where they
// are in L2 (13.8 -> 13.9, 13.4 -> 13.7, 11.1 -> 11.2, 8.1 -> 8.3). bf16 steps are slower by the code and the registers
// that this costs (one sequence of 128256 ids, from L2, 12.0 -> 12.3).
template <int DTYPE>
constexpr int GROUP = DTYPE == OD_BF16 ? U : 2 * U;

// One warp's units [v0, v1) of a row; the first group of `run` has been requested.
template <int DTYPE>
__device__ __forceinline__ void warp_segment(UnitRun<DTYPE, 1, GROUP<DTYPE>> &run, const char *row, int v1, int full, int v_p, int lane, float scale,
                                             float4 *rec)
{
    Lane<DTYPE> L;
    L.reset();
    run.finish(L, scale);
    if (v1 > full) absorb_ragged<DTYPE>(L, row, v_p, lane, scale);
    float c = L.c, s = L.s, mx = L.max_seen();
    warp_merge(c, s, mx);
    if (lane == 0) *rec = make_float4(c, s, mx, 0.f);
}

// Row 0: the warps take equal runs of the slice.
template <int DTYPE>
struct RowZero {
    UnitRun<DTYPE, 1, GROUP<DTYPE>> run;
    int v0, v1;
    __device__ __forceinline__ void begin(const StepArgs &a, const Slice &s, int b, int warp, int lane)
    {
        const int per = (s.units() + CWARPS - 1) / CWARPS;
        v0 = min(s.u0 + warp * per, s.u1);
        v1 = min(v0 + per, s.u1);
        run.begin(row_of<DTYPE>(a, b, 0), v0, min(v1, s.full), lane);
    }
    __device__ __forceinline__ void finish(const StepArgs &a, const Slice &s, int b, int warp, int lane, float scale, float4 *s_rec)
    {
        if (v0 < v1) warp_segment<DTYPE>(run, row_of<DTYPE>(a, b, 0), v1, s.full, a.v_p, lane, scale, s_rec + warp);
    }
};

// Rows 1..mb: the slices laid end to end, one contiguous run per warp. (Asynchronous copies into a ring of
// shared memory, 96 KB of them in flight per block, in place of two groups of register loads: 24 sequences of
// 128256 bf16 ids 30.7 us, this 24.6; 64 31.8 and 25.1.)
template <int DTYPE>
__device__ __forceinline__ void rows_from_one(const StepArgs &a, const Slice &s, int b, int mb, int warp, int lane, float scale,
                                              float4 *s_rec)
{
    const int n = s.units(), total = mb * n, per = (total + CWARPS - 1) / CWARPS;
    int f = warp * per;
    const int f_hi = min(f + per, total);
    if (f >= f_hi) return;
    int r = 1 + s.rows_before(f), v = f - (r - 1) * n;  // (f < OD_MAX_K * n, and a block has at most 320 KB of rows)
    while (f < f_hi) {
        const int cnt = min(n - v, f_hi - f), v0 = s.u0 + v, v1 = v0 + cnt;
        const char *row = row_of<DTYPE>(a, b, r);
        UnitRun<DTYPE, 1, GROUP<DTYPE>> run;
        run.begin(row, v0, min(v1, s.full), lane);
        warp_segment<DTYPE>(run, row, v1, s.full, a.v_p, lane, scale, s_rec + r * CWARPS + warp);
        f += cnt; v = 0; ++r;
    }
}

// 2^d for d <= 0, to fp32's last place or so (Taylor's series of e^(f ln 2), |f| <= 1/2, to f^7: 5e-9), 0 below 2^-125.
// Every level of the merge multiplies whole sums by it, ever fewer and larger ones, and ex2.approx (2^-22) errs on one side:
// mean error of 600 row sums against 64 bits, 15 sequences of 50001 bf16 ids: -5.6e-8 with ex2.approx, -0.3e-8 so; 60 of
// 8000 fp32 ids -4.5e-8, -0.4e-8 (root mean square 9.5e-8, 8.0e-8; the streaming pass, one such level: -4.1e-8, 8.8e-8).
__device__ __forceinline__ float exp2_to_last_place(float d)
{
    const float m = d + 12582912.f, f = d - (m - 12582912.f);   // 1.5 * 2^23: the nearest whole number n in m's low bits
    float p = 1.5252733804e-5f;
    p = fmaf(p, f, 1.5403530394e-4f); p = fmaf(p, f, 1.3333558147e-3f); p = fmaf(p, f, 9.6181291076e-3f);
    p = fmaf(p, f, 5.5504108665e-2f); p = fmaf(p, f, 2.4022650696e-1f); p = fmaf(p, f, 6.9314718056e-1f); p = fmaf(p, f, 1.f);
    return d < -125.f ? 0.f : p * __int_as_float((__float_as_int(m) + 127) << 23);
}
// warp_merge with it
__device__ __forceinline__ void merge_to_last_place(float &c, float &s, float &mx)
{
    const float cm = warp_max(c);
    mx = warp_max(mx);
    s *= exp2_to_last_place(c - cm);
    c = cm;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
}

// The rows' statistics from the warps' partials: merged per row, exchanged over the cluster, merged again by
// every block alike; row(r, c, sum, mx) is called by every lane of the warp that merged row r. The caller
// has arrived (relaxed) at the cluster's first barrier. All threads call.
template <typename Row>
__device__ __forceinline__ void exchange_rows(const Slice &s, int mb, unsigned part, unsigned nparts, int warp, int lane,
                                              float4 *s_rec, float4 *s_all, Row row)
{
    const int n = s.units(), per0 = (n + CWARPS - 1) / CWARPS, per = (mb * n + CWARPS - 1) / CWARPS;
    __syncthreads();
    od_cluster_wait();                                      // every block runs
    for (int r = warp; r <= mb; r += CWARPS) {
        // the warps that had units of the row: from unit lane * per on, per of them
        const bool held = r == 0 ? lane * per0 < n : lane * per < r * n && (lane + 1) * per > (r - 1) * n;
        float c = -FLT_MAX, sum = 0.f, mx = -INFINITY;
        if (held) {
            const float4 v = s_rec[r * CWARPS + lane];
            c = v.x; sum = v.y; mx = v.z;
        }
        merge_to_last_place(c, sum, mx);
        if (lane < (int)nparts) cluster_store4(s_all + r * CWARPS + part, (uint32_t)lane, make_float4(c, sum, mx, 0.f));
    }
    __syncwarp();
    od_cluster_arrive();
    od_cluster_wait();
    for (int r = warp; r <= mb; r += CWARPS) {
        float c = -FLT_MAX, sum = 0.f, mx = -INFINITY;
        if (lane < (int)nparts) {
            const float4 v = s_all[r * CWARPS + lane];
            c = v.x; sum = v.y; mx = v.z;
        }
        merge_to_last_place(c, sum, mx);
        row(r, c, sum, mx);
    }
}
// ... as lane k's maximum and sum of row k, in every warp; s_bad: not 0 if a sum is not a positive number
__device__ __forceinline__ void exchange_rows(const Slice &s, int mb, unsigned part, unsigned nparts, int warp, int lane, float scale,
                                              float4 *s_rec, float4 *s_all, float *s_M, float *s_S, unsigned int *s_bad, float &rm,
                                              float &rs)
{
    exchange_rows(s, mb, part, nparts, warp, lane, s_rec, s_all, [&](int r, float c, float sum, float mx) {
        if (lane != 0) return;
        const float S = row_sum_of(c, sum, mx, scale);      // sum of exp2((x - M)*scale)
        s_M[r] = mx; s_S[r] = S;
        if (!(S > 0.f) || !(S <= FLT_MAX)) atomicOr(s_bad, 1u);
    });
    __syncthreads();
    rm = 0.f; rs = 0.f;
    if (lane <= mb) { rm = s_M[lane]; rs = s_S[lane]; }
}

__device__ __forceinline__ void wait_for_earlier() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_next() { asm volatile("griddepcontrol.launch_dependents;"); }

template <int DTYPE, int SOURCE>
__global__ void __launch_bounds__(CTHREADS, 1)
od_step_kernel(const __grid_constant__ StepArgs a)
{
    __shared__ float s_M[OD_MAX_K + 1], s_S[OD_MAX_K + 1];
    __shared__ int4 s_piece[OD_MAX_K];                      // piece that begins at an offset: length (0: none), target, table slot, q'
    __shared__ unsigned int s_bad;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    float4 *s_rec = (float4 *)s_dyn, *s_all = s_rec + REC;
    const unsigned part = blockIdx.x, nparts = gridDim.x;
    const int b = blockIdx.y, K = a.K_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *s_q = (float *)s_dyn, *s_val = s_q + (SOURCE == STAGED ? a.slots : 0) + warp * a.tiles_per_warp;

    // Under the caller's promise (inputs_early) everything but the writes runs before the wait (the table's lookups
    // where no writer of it may be at work). The next launch is released behind the wait all the same: it may be a
    // step that reads its own inputs early, and the promise is that what is two launches back is complete.
    const bool all_early = a.inputs_early && a.table_early;
    const int32_t map_serial = SOURCE == FROM_ROW ? __ldg(a.map_serial_now) : a.map_serial;
    if (threadIdx.x == 0) s_bad = 0;
    od_cluster_arrive_relaxed();                            // this block runs: the others may store to it
    if (!a.inputs_early) { wait_for_earlier(); release_next(); }

    // ---- the proposal: lane k of every warp holds position k's id and probability
    int Kb = a.draft_len[b];
    int32_t id = -1;
    float qs = 0.f;
    if (lane < K) {
        id = a.draft_ids[(size_t)b * K + lane];
        qs = a.q_sel[(size_t)b * K + lane];
    }
    Ahead h;
    h.T = a.temperature[b];
    const uint64_t seed = a.seed[b];
    const Slice slice = slice_of<DTYPE>(a, (int)part);
    RowZero<DTYPE> zero;
    zero.begin(a, slice, b, warp, lane);
    if (a.inputs_early && !all_early) { wait_for_earlier(); release_next(); }
    Kb = Kb < 0 ? 0 : (Kb > K ? K : Kb);
    const float u = od_uniform(seed, a.step, (uint32_t)lane, 0u);
    h.u_draw = od_uniform(seed, a.step, (uint32_t)lane, 1u);
    // ---- the piece that begins at offset `warp`: the longest cached run, else the direct map
    if (warp < Kb) {
        const int4 piece = look_up_piece(id, qs, warp, Kb, a.v_q, a.vocab_map, a.keys, a.vals, a.cap, lane);
        if (lane == 0) s_piece[warp] = piece;
    }
    h.scale = 1.4426950408889634f / h.T;
    const float scale = h.T > 0.f ? h.scale : 0.f;
    zero.finish(a, slice, b, warp, lane, scale, s_rec);
    __syncthreads();

    // ---- the walk, by every warp
    const Walk w = walk_proposal(lane < Kb ? s_piece[lane] : make_int4(0, -1, -1, 0), id, Kb, lane);
    const int mb = w.m;
    h.mb = mb;
    h.stop = w.stopped;
    h.l_len = w.len; h.l_tgt = w.tgt; h.l_qp = w.q;
    float x_t = 0.f;
    const bool t_ok = lane < mb && h.l_tgt >= 0 && h.l_tgt < a.v_p;
    if (t_ok) x_t = od_load_logit<DTYPE>(row_of<DTYPE>(a, b, lane), h.l_tgt);

    // ---- step 2
    rows_from_one<DTYPE>(a, slice, b, mb, warp, lane, scale, s_rec);
    // (what the draw starts with travels during the exchange)
    prepare_positions(a, h, b, lane, w.start, w.first_id);
    load_first_probability(a, h, b);
    Part<SOURCE> mine;
    mine.prepare(a, (int)part, warp, lane);
    float rm, rs;
    exchange_rows(slice, mb, part, nparts, warp, lane, scale, s_rec, s_all, s_M, s_S, &s_bad, rm, rs);
    if (all_early) { wait_for_earlier(); release_next(); }  // nothing has been written yet
    const bool writes = part == 0 && warp == 0;
    if (writes) {
        store_walk(a.out, w, b, K, a.v_q, lane);
        if (lane <= mb) {
            const size_t row_slot = (size_t)b * (K + 1) + lane;
            a.w_row_max[row_slot] = rm; a.w_row_sum[row_slot] = rs;
        }
    }
    const int j = decide(a, h, b, lane, rm, rs, t_ok, x_t, u, s_bad, writes);
    if (!(h.T > 0.f)) {                                     // every block of the sequence leaves here
        if (part == 0 && threadIdx.x == 0) { a.out_token[b] = -1; a.resid_mass[b] = 0.f; a.flags[b] = OD_SF_BAD_TEMPERATURE; }
        return;
    }
    draw<DTYPE, SOURCE, true, true>(a, h, mine, b, part, nparts, warp, lane, j, rm, rs, map_serial == a.map_serial, s_q, s_val);
}

// Step 2 alone, with the same slices and the same order of reduction. SHARD: the rows are the columns [col0,
// col0 + v_p) of the full rows; a row's merged statistics are stored as this shard's record.
template <int DTYPE, bool SHARD>
__global__ void __launch_bounds__(CTHREADS, 1)
od_verify_rows_kernel(const __grid_constant__ StepArgs a)
{
    __shared__ float s_M[OD_MAX_K + 1], s_S[OD_MAX_K + 1];
    __shared__ unsigned int s_bad;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    float4 *s_rec = (float4 *)s_dyn, *s_all = s_rec + REC;
    const unsigned part = blockIdx.x, nparts = gridDim.x;
    const int b = blockIdx.y, K = a.K_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_bad = 0;
    od_cluster_arrive_relaxed();
    if (!a.inputs_early) { wait_for_earlier(); release_next(); }
    Ahead h = {};
    h.T = a.temperature[b];
    h.scale = 1.4426950408889634f / h.T;
    const float scale = h.T > 0.f ? h.scale : 0.f;
    const Slice slice = slice_of<DTYPE>(a, (int)part);
    RowZero<DTYPE> zero;
    zero.begin(a, slice, b, warp, lane);
    if (a.inputs_early) {
        zero.finish(a, slice, b, warp, lane, scale, s_rec);
        wait_for_earlier(); release_next();
    }
    // what the translation kernel wrote
    h.mb = clamp_m(a.m[b], K);
    const uint64_t seed = SHARD ? 0ull : a.seed[b];
    h.l_tgt = -1;
    if (lane < K) {
        const size_t o = (size_t)b * K + lane;
        h.l_tgt = a.tgt_ids[o];
        if (!SHARD) { h.l_len = a.span_len[o]; h.l_qp = a.q_prime[o]; }
    }
    if (!a.inputs_early) zero.finish(a, slice, b, warp, lane, scale, s_rec);
    float x_t = 0.f, u = 0.f;
    if (SHARD) h.l_tgt -= a.col0;
    const bool t_ok = lane < h.mb && h.l_tgt >= 0 && h.l_tgt < a.v_p;
    if (t_ok) x_t = od_load_logit<DTYPE>(row_of<DTYPE>(a, b, lane), h.l_tgt);
    if (!SHARD && lane < h.mb) u = od_uniform(seed, a.step, (uint32_t)lane, 0u);
    rows_from_one<DTYPE>(a, slice, b, h.mb, warp, lane, scale, s_rec);
    if (SHARD) {
        if (!t_ok) x_t = -INFINITY;
        exchange_rows(slice, h.mb, part, nparts, warp, lane, s_rec, s_all, [&](int r, float c, float sum, float mx) {
            const float x = __shfl_sync(0xFFFFFFFFu, x_t, r < h.mb ? r : 31);
            if (part == 0 && lane == 0) a.stats[b * (K + 1) + r] = make_float4(c, sum, mx, x);
        });
        return;
    }
    float rm, rs;
    exchange_rows(slice, h.mb, part, nparts, warp, lane, scale, s_rec, s_all, s_M, s_S, &s_bad, rm, rs);
    if (part != 0 || warp != 0) return;
    if (lane <= h.mb) {
        const size_t row_slot = (size_t)b * (K + 1) + lane;
        a.w_row_max[row_slot] = rm; a.w_row_sum[row_slot] = rs;
    }
    decide(a, h, b, lane, rm, rs, t_ok, x_t, u, s_bad, true);
}

template <typename K>
cudaError_t allow(K kernel, size_t bytes)
{
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}
template <int DTYPE>
cudaError_t allow_all()
{
    const size_t staged = (size_t)(OD_SAMPLE_MAX_SLOTS + 1) * 4 + 8 * 1024;
    cudaError_t e = allow(od_step_kernel<DTYPE, FROM_MAP>, OD_SAMPLE_SMEM_MAX);
    if (e == cudaSuccess) e = allow(od_step_kernel<DTYPE, FROM_ROW>, OD_SAMPLE_SMEM_MAX);
    if (e == cudaSuccess) e = allow(od_step_kernel<DTYPE, STAGED>, staged);
    if (e == cudaSuccess) e = allow(od_verify_rows_kernel<DTYPE, false>, REC_BYTES);
    if (e == cudaSuccess) e = allow(od_verify_rows_kernel<DTYPE, true>, REC_BYTES);
    return e;
}

template <typename Kern>
cudaError_t launch_clusters(Kern kern, int parts, int32_t B, size_t smem, cudaStream_t s, bool pdl, const StepArgs &a)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)parts, (unsigned)B); cfg.blockDim = dim3(CTHREADS);
    // the partials, and in their place the draw's probabilities and tile values
    cfg.dynamicSmemBytes = smem > REC_BYTES ? smem : REC_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)parts; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// Blocks per sequence (a level of od_sample_parts) for rows of v_len elements in one launch of which a block may
// stream `most` bytes, or -1: more launches are better. The most blocks whose clusters all have a multiprocessor to
// every block (two blocks to one leave 64 registers a thread, and what is then spilled costs 1 to 2.5 us; a second wave
// costs a whole step), and a tile for half the warps (8000 ids, one sequence: 8.2 us with 16 blocks, 7.9 with 4 to 8).
int level_within(const od_ctx *c, int32_t B, int32_t K_max, int32_t v_len, int32_t dtype, int parts, int64_t most)
{
    if (c->opt_verify_grid > 0 || c->opt_sample_tiles_per_warp > 0 || B < 1) return -1;
    int level = -1;
    for (int next = 0; next < OD_SAMPLE_LEVELS; ++next)
        if (B <= c->step_clusters[next] && (next == 0 || od_sample_part_tiles(v_len, next) >= CWARPS / 2)) level = next;
    if (level < 0 || (od_sample_parts(level) < parts && od_sample_part_tiles(v_len, level) > CWARPS)) return -1;
    const int64_t bytes = (int64_t)od_sample_part_tiles(v_len, level) * OD_SAMPLE_TILE * (dtype == OD_BF16 ? 2 : 4);
    return bytes * (K_max + 1) <= most ? level : -1;
}
// A cluster streams its sequence's rows by itself, at most 60 GB/s a block (the special-function unit's rate; 40 from
// HBM with what it has in flight), however few rows others have; three launches spread all rows over all
// multiprocessors. The line lies where a block may have 320 KB to stream (device time of a step, three launches -> one;
// sequences x K_max, target ids, blocks: KB; in brackets with inputs that change from pass to pass, from HBM):
//   1 x 6, 128256 bf16, 16: 112 KB  14.5 -> 12.4 (14.9 -> 13.1)     15 x 6, 8: 221 KB  18.6 -> 15.4 (19.7 -> 16.7)
//   22 x 6, 6: 294 KB  20.0 -> 18.0 (20.9 -> 19.6)                  24 x 6, 5: 354 KB  20.3 -> 19.8 (21.3 -> 21.5)
//   15 x 12, 8: 410 KB  19.8 -> 19.3                  28 x 6, 4: 441 KB  21.5 -> 21.7     22 x 12, 6: 546 KB  23.2 -> 23.4
//   7 x 3, 152064 bf16, 16: 76 KB  16.4 -> 12.4      24 x 4, 50001 fp32, 6: 165 KB  16.5 -> 13.7 (19.5 -> 17.2)
// One line for both types, though fp32 rows have half the exponentials to a byte: 36 x 4, 50001 fp32, 3: 330 KB, just
// beyond it, would be 20.4 -> 17.6 from L2 (three launches there now 18.5). Batches of two blocks a sequence gain little (60 x 8, 32000: 16.0 -> 15.3; 60 x 6, 128256: 30.0 -> 34.8).
int step_level(const od_ctx *c, int32_t B, int32_t K_max, int32_t v_len, int32_t dtype)
{
    return level_within(c, B, K_max, v_len, dtype, 3, 320 * 1024);
}
// Step 2 alone takes the place of two launches, not three, and its blocks leave no room for those of the next call:
// 200 KB (the three calls: 20 x 4, 50001 fp32, 6: 167 KB  18.3 -> 18.2; 44 x 4, 40000, 3: 133 KB  20.7 -> 20.0; 15 x 6,
// 128256, 8: 224 KB  19.9 -> 21.1). Of a vocabulary shard 240 KB, with any number of blocks (a rank's
// five calls: 64 x 6, 32064 columns, 2: 224 KB  27.6 -> 27.1; 100 x 6, 16000, 1: 224 KB  28.1 -> 26.9).
int rows_level(const od_ctx *c, int32_t B, int32_t K_max, int32_t v_len, int32_t dtype)
{
    return v_len == c->v_p ? level_within(c, B, K_max, v_len, dtype, 3, 200 * 1024)
                           : level_within(c, B, K_max, v_len, dtype, 1, 240 * 1024);
}

void cut_rows(int level, int32_t dtype, StepArgs &a)
{
    const int64_t esz = dtype == OD_BF16 ? 2 : 4;
    a.W = (int32_t)(((int64_t)a.v_p * esz + 511) / 512);
    a.part_units = od_sample_part_tiles(a.v_p, level) * (int32_t)(OD_SAMPLE_TILE * esz / 512);
}

template <int DTYPE>
cudaError_t launch_step(int source, int parts, size_t smem, cudaStream_t s, bool pdl, const StepArgs &a)
{
    if (source == STAGED) return launch_clusters(od_step_kernel<DTYPE, STAGED>, parts, a.B, smem, s, pdl, a);
    if (source == FROM_ROW) return launch_clusters(od_step_kernel<DTYPE, FROM_ROW>, parts, a.B, smem, s, pdl, a);
    return launch_clusters(od_step_kernel<DTYPE, FROM_MAP>, parts, a.B, smem, s, pdl, a);
}

}  // namespace

// clusters: [levels] resident at a time with a multiprocessor to every block
cudaError_t od_step_prepare_device(int32_t *clusters)
{
    cudaError_t e = allow_all<OD_BF16>();
    if (e == cudaSuccess) e = allow_all<OD_F32>();
    if (e != cudaSuccess) return e;
    for (int level = 0; level < OD_SAMPLE_LEVELS; ++level)
        clusters[level] = resident_clusters(od_step_kernel<OD_BF16, STAGED>, od_sample_parts(level), 64 * 1024);
    return cudaSuccess;
}

bool od_step_one_launch(const od_ctx *c, int32_t B, int32_t K_max, int32_t dtype)
{
    return step_level(c, B, K_max, c->v_p, dtype) >= 0;
}
bool od_verify_one_launch(const od_ctx *c, int32_t B, int32_t K_max, int32_t v_len, int32_t dtype)
{
    return rows_level(c, B, K_max, v_len, dtype) >= 0;
}

// od_step in one launch (od_step_one_launch). fuse: where step 2's outputs go.
cudaError_t od_launch_step(od_ctx *c, int32_t B, int32_t K_max, const int32_t *draft_ids, const int32_t *draft_len,
                           const float *q_sel, const float *q_rows, const void *logits, int32_t dtype, int64_t row_stride,
                           int64_t seq_stride, const float *temperature, const uint64_t *seed, uint64_t step, int32_t *tgt_ids,
                           float *q_prime, int32_t *span_start, int32_t *span_len, int32_t *m, uint8_t *tail_kind,
                           uint32_t *counters, const od_fused_verify *fuse, int32_t *out_token, float *resid_mass, uint32_t *flags,
                           bool early, cudaStream_t s)
{
    const int level = step_level(c, B, K_max, c->v_p, dtype);
    const bool pdl = c->opt_pdl != 0;
    StepArgs a = {};
    a.logits = logits; a.row_stride = row_stride; a.seq_stride = seq_stride;
    a.B = B; a.K_max = K_max; a.v_p = c->v_p; a.q_rows = q_rows;
    a.draft_ids = draft_ids; a.temperature = temperature; a.seed = seed; a.step = step;
    a.out_token = out_token; a.resid_mass = resid_mass; a.flags = flags;
    a.w_row_max = fuse->row_max; a.w_row_sum = fuse->row_sum; a.w_p_sel = fuse->p_sel; a.w_ratio = fuse->ratio;
    a.w_n_accepted = fuse->n_accepted; a.w_n_draft = fuse->n_draft_accepted; a.w_vflags = fuse->flags;
    a.draft_len = draft_len; a.q_sel = q_sel;
    a.keys = c->d_keys; a.vals = c->d_vals; a.cap = c->cap;
    a.out = map_out(c, tgt_ids, q_prime, span_start, span_len, m, tail_kind, counters);
    a.inputs_early = early && pdl; a.table_early = !c->table_written;
    context_args(c, a);
    const DrawPlan plan = plan_draw(c, level, a);
    cut_rows(level, dtype, a);
    c->table_written = false;
    c->translation_complete = false;                        // (it releases the next launch before it has written anything)
    const int parts = od_sample_parts(level);
    c->info[0] = (int64_t)parts * B; c->info[1] = a.part_units;
    c->info[2] = (int64_t)parts * B; c->info[3] = a.tiles_per_warp;
    return dtype == OD_BF16 ? launch_step<OD_BF16>(plan.source, parts, plan.smem, s, pdl, a)
                            : launch_step<OD_F32>(plan.source, parts, plan.smem, s, pdl, a);
}

// od_verify in one launch (od_verify_one_launch)
cudaError_t od_launch_verify_rows(od_ctx *c, int32_t B, int32_t K_max, const void *logits, int32_t dtype, int64_t row_stride,
                                  int64_t seq_stride, const int32_t *tgt_ids, const float *q_prime, const int32_t *span_len,
                                  const int32_t *m, const float *temperature, const uint64_t *seed, uint64_t step,
                                  const od_fused_verify *out, bool early, cudaStream_t s)
{
    const int level = rows_level(c, B, K_max, c->v_p, dtype);
    StepArgs a = {};
    a.logits = logits; a.row_stride = row_stride; a.seq_stride = seq_stride;
    a.B = B; a.K_max = K_max; a.v_p = c->v_p;
    a.tgt_ids = tgt_ids; a.q_prime = q_prime; a.span_len = span_len; a.m = m;
    a.temperature = temperature; a.seed = seed; a.step = step;
    a.w_row_max = out->row_max; a.w_row_sum = out->row_sum; a.w_p_sel = out->p_sel; a.w_ratio = out->ratio;
    a.w_n_accepted = out->n_accepted; a.w_n_draft = out->n_draft_accepted; a.w_vflags = out->flags;
    a.inputs_early = early && c->opt_pdl != 0;
    cut_rows(level, dtype, a);
    c->translation_complete = true;
    const int parts = od_sample_parts(level);
    c->info[0] = (int64_t)parts * B; c->info[1] = a.part_units;
    const bool pdl = c->opt_pdl != 0;
    return dtype == OD_BF16 ? launch_clusters(od_verify_rows_kernel<OD_BF16, false>, parts, B, 0, s, pdl, a)
                            : launch_clusters(od_verify_rows_kernel<OD_F32, false>, parts, B, 0, s, pdl, a);
}

// od_verify_shard_stats in one launch (od_verify_one_launch for shard_len columns)
cudaError_t od_launch_shard_rows(od_ctx *c, int32_t B, int32_t K_max, int32_t shard_lo, int32_t shard_len, const void *logits,
                                 int32_t dtype, int64_t row_stride, int64_t seq_stride, const int32_t *tgt_ids, const int32_t *m,
                                 const float *temperature, float *stats, bool early, cudaStream_t s)
{
    const int level = rows_level(c, B, K_max, shard_len, dtype);
    StepArgs a = {};
    a.logits = logits; a.row_stride = row_stride; a.seq_stride = seq_stride;
    a.B = B; a.K_max = K_max; a.v_p = shard_len; a.col0 = shard_lo;
    a.tgt_ids = tgt_ids; a.m = m; a.temperature = temperature;
    a.stats = (float4 *)stats;
    a.inputs_early = early && c->opt_pdl != 0;
    cut_rows(level, dtype, a);
    c->translation_complete = true;
    const int parts = od_sample_parts(level);
    c->info[0] = (int64_t)parts * B; c->info[1] = a.part_units;
    const bool pdl = c->opt_pdl != 0;
    return dtype == OD_BF16 ? launch_clusters(od_verify_rows_kernel<OD_BF16, true>, parts, B, 0, s, pdl, a)
                            : launch_clusters(od_verify_rows_kernel<OD_F32, true>, parts, B, 0, s, pdl, a);
}
