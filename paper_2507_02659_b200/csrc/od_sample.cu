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
//   mode 1  pass 1 over the window by a cluster of blocks, whose sums meet in the first
//           one: the shard's share of the residual mass (and, when that is zero, of the
//           mass of p_j, for the fallback);
//   mode 2  after the shares of all shards were exchanged: every shard forms the
//           same total and target = u * total, finds the shard in which the running
//           sum over shards crosses the target, and that shard alone scans its
//           window (offset by the shares before it) as in pass 2.
#include <float.h>

#include <vector>

#include "od_common.cuh"
#include "od_decide.cuh"
#include "od_draw.cuh"

namespace {

constexpr int WARPS = OD_SAMPLE_THREADS / 32;

template <int DTYPE, bool FUSED, int SOURCE>
__global__ void __launch_bounds__(CTHREADS, 2)
od_sample_kernel(const SampleArgs a)
{
    __shared__ float s_M[FUSED ? OD_MAX_K + 1 : 1], s_S[FUSED ? OD_MAX_K + 1 : 1];
    __shared__ int s_red[2][CWARPS];
    __shared__ unsigned int s_vbits;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const unsigned part = blockIdx.x, nparts = gridDim.x;
    const int b = blockIdx.y;
    const int K = a.K_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the staged probabilities, then the warps' tile values
    float *s_q = (float *)s_dyn, *s_val = s_q + (SOURCE == STAGED ? a.slots : 0) + warp * a.tiles_per_warp;

    // Under programmatic dependent launch this grid is resident while the verification
    // kernels still run. What the translation kernel wrote (it finished before them) is
    // read now. (a.early = 0: no verification is in front of this launch; everything waits.)
    // Inside od_step the next launch is released at once (the streaming pass in front has waited). A call of its own
    // releases behind its wait: the launch in front may be anything, and what is behind may read its inputs early.
    if (FUSED) asm volatile("griddepcontrol.launch_dependents;");
    if (!a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int32_t map_serial = SOURCE == FROM_ROW ? __ldg(a.map_serial_now) : a.map_serial;
    Ahead h = load_ahead(a, b, lane);
    if (FUSED) load_first_probability(a, h, b);             // (the step's inputs were complete before its translation)
    else request_first_probability(a, h, b);
    const int mb = h.mb;

    // FUSED, still before the wait: where the rows' partials will be (sums of m), and position
    // k's inputs of the acceptance test in lane k
    int before = 0, total = 0, segments = 0;
    float d_xt = 0.f, d_u = 0.f;
    bool d_tok = false;
    if (threadIdx.x == 0) s_vbits = 0;
    if (FUSED) {
        for (int i = threadIdx.x; i < a.B; i += CTHREADS) {
            const int v = clamp_m(a.m[i], K);
            total += v;
            if (i < b) before += v;
        }
        before = __reduce_add_sync(0xFFFFFFFFu, before);
        total = __reduce_add_sync(0xFFFFFFFFu, total);
        if (lane == 0) { s_red[0][warp] = before; s_red[1][warp] = total; }
        if (lane < mb) {
            d_tok = h.l_tgt >= 0 && h.l_tgt < a.v_p;
            const char *row_k = (const char *)a.logits +
                                ((size_t)b * a.seq_stride + (size_t)lane * a.row_stride) * (DTYPE == OD_BF16 ? 2 : 4);
            if (d_tok) d_xt = od_load_logit<DTYPE>(row_k, h.l_tgt);
        }
        const uint64_t seed = a.seed[b];
        d_u = od_uniform(seed, a.step, (uint32_t)lane, 0u);
        h.u_draw = od_uniform(seed, a.step, (uint32_t)lane, 1u);
        __syncthreads();
        before = __reduce_add_sync(0xFFFFFFFFu, lane < CWARPS ? s_red[0][lane] : 0);
        total = __reduce_add_sync(0xFFFFFFFFu, lane < CWARPS ? s_red[1][lane] : 0);
        segments = row_partial_segments(a.plan, b, warp, before, total);   // (of the row this warp merges first)
    }

    Part<SOURCE> mine;
    mine.prepare(a, (int)part, warp, lane);

    // n_accepted and the row statistics come from the verification kernels
    if (a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!FUSED) asm volatile("griddepcontrol.launch_dependents;");
    if (!FUSED) load_first_probability(a, h, b);

    int j = 0;
    float rm = 0.f, rs = 0.f;                      // lane k: statistics of row k
    if (FUSED) {
        // ---- step 2's decisions (what od_verify_decide_kernel does, same arithmetic, same order)
        const bool bad_T = !(h.T > 0.f);
        const float dscale = bad_T ? 0.f : h.scale;
        for (int r = warp; r <= mb; r += CWARPS) {
            const int row_slot = b * (K + 1) + r;
            float c, sum, mx;
            merge_row_partials(a.plan, row_slot, r == warp ? segments : row_partial_segments(a.plan, b, r, before, total), lane, c, sum, mx);
            if (lane == 0) {
                const float S = row_sum_of(c, sum, mx, dscale);
                s_M[r] = mx; s_S[r] = S;
                if (part == 0) { a.w_row_max[row_slot] = mx; a.w_row_sum[row_slot] = S; }
                if (!(S > 0.f) || !(S <= FLT_MAX)) atomicOr(&s_vbits, 1u);
            }
        }
        __syncthreads();
        if (lane <= mb) { rm = s_M[lane]; rs = s_S[lane]; }
        j = decide(a, h, b, lane, rm, rs, d_tok, d_xt, d_u, s_vbits, part == 0 && warp == 0);
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
    if (SOURCE != FROM_ROW || nparts > 1) od_cluster_arrive_relaxed();   // this block runs: the others may store to it (waited for below)
    draw<DTYPE, SOURCE, false, FUSED>(a, h, mine, b, part, nparts, warp, lane, j, rm, rs, planned, s_q, s_val);
}

// ---- vocabulary shards: MODE 1, a shard's mass shares; MODE 2, a shard's pick ---------------
// 64 registers in both: four blocks of 256 threads to a multiprocessor; MODE 1 may have blocks of up to 1024.
template <int DTYPE, int MODE>
__global__ void __launch_bounds__(MODE == 1 ? OD_SHARD_MAX_THREADS : OD_SAMPLE_THREADS, MODE == 1 ? 1 : 4)
od_sample_shard_kernel(const SampleArgs a)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];   // ntiles x 8 bytes
    double *s_val = (double *)s_dyn;                         // pass 2: tile values
    __shared__ double s_warp[MODE == 1 ? OD_SHARD_MAX_THREADS / 32 : WARPS];
    __shared__ double s_sums[MODE == 1 && DTYPE != OD_BF16 ? OD_SHARD_MAX_THREADS / 32 * 2 : 1];
    const int warps = MODE == 1 ? (int)(blockDim.x >> 5) : WARPS;
    __shared__ double s_part[OD_SAMPLE_MAX_PARTS];          // MODE 1: the cluster's blocks' sums, in its first block
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

    if (!a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    Ahead h = load_ahead(a, b, lane);
    const int mb = h.mb;
    const float T = h.T;
    const bool planned = __ldg(a.map_serial_now) == a.map_serial;   // (as in od_sample_kernel)

    // a shard's tiles and ids keep their numbers of the full row
    const int tile_lo = a.tile_lo, tile_hi = a.tile_hi;
    // pass 1's whole tiles of this warp, and the inverse-map entries of their first pair
    const int p_lo = tile_lo + ((int)part * warps + warp) * a.tiles_per_warp;
    int p_hi = p_lo + a.tiles_per_warp;
    if (p_hi > tile_hi) p_hi = tile_hi;
    const int p_hi_w = p_hi < a.v_p / OD_SAMPLE_TILE ? p_hi : a.v_p / OD_SAMPLE_TILE;
    int4 ni[2][2] = {};
    if (MODE == 1 && !a.same_ids && p_lo < p_hi_w) first_pair_entries(a, p_lo, p_hi_w, lane, ni);

    // n_accepted and the row statistics come from the verification kernels
    if (a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");      // (behind the wait, as in od_sample_kernel)
    load_first_probability(a, h, b);
    // MODE 2: all it needs from memory is requested here, in one trip: the first 1024 tile values, the seed, lane k the
    // shares of shard k
    const int ntiles = a.ntiles;
    double *tile_val = a.tile_val + (size_t)b * ntiles;
    double first_val[4], share_r = 0.0, share_e = 0.0;
    uint64_t seed_b = 0;
    if (MODE == 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = tile_lo + (int)threadIdx.x + i * OD_SAMPLE_THREADS;
            first_val[i] = t < tile_hi ? __ldcg(tile_val + t) : 0.0;
        }
        seed_b = a.seed[b];
        if (lane < a.n_shards) {
            share_r = a.mass_all[((size_t)lane * a.B + b) * 2];
            share_e = a.mass_all[((size_t)lane * a.B + b) * 2 + 1];
        }
    }

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
    if (MODE == 1) od_cluster_arrive_relaxed();    // this block runs: the first one may be stored to (waited for below)
    float rm = 0.f, rs = 0.f;                      // lane k: statistics of row k
    if (lane <= mb) {
        rm = a.row_max[b * (K + 1) + lane];
        rs = a.row_sum[b * (K + 1) + lane];
    }
    int j = a.n_accepted[b];
    j = j < 0 ? 0 : (j > mb ? mb : j);
    const SeqState q = seq_state<DTYPE>(a, h, b, j, rm, rs, a.col0, planned);
    if (MODE == 1 && q.residual && threadIdx.x == 0) prefetch_q_row(a, q, part, nparts);

    if (MODE == 1) {
        SummedTiles<DTYPE> out = {tile_val, s_sums + (DTYPE == OD_BF16 ? 0 : 2 * warp), lane, 0.0};
        out.clear();
        // ---- pass 1: the value of every tile ----
        const int hi_w = planned || !a.same_ids ? p_hi_w : p_lo;
        if (a.same_ids) warp_run<DTYPE, FROM_ROW, false>(q, a, p_lo, p_hi, hi_w, lane, out, ni);
        else warp_run<DTYPE, FROM_MAP, false>(q, a, p_lo, p_hi, hi_w, lane, out, ni);
        // ---- the window's sum: the blocks' sums meet in the first block of the cluster
        const double run_sum = out.sum();
        if (lane == 0) s_warp[warp] = run_sum;
        __syncthreads();
        od_cluster_wait();
        if (threadIdx.x == 0) {
            double sum = 0.0;
            for (int w = 0; w < warps; ++w) sum += s_warp[w];
            od_cluster_store(&s_part[part], 0u, sum);
        }
        od_cluster_arrive();
        od_cluster_wait();
        if (part != 0) return;
        double mass_r = 0.0, mass_e = 0.0;
        for (unsigned int i = 0; i < nparts; ++i) mass_r += s_part[i];
        if (q.residual && !(mass_r > 0.0)) {
            // no residual mass here: should no shard have any, the draw is from p_j
            out.clear();
            for (int t_lo = tile_lo + warp * 2; t_lo < tile_hi; t_lo += warps * 2)
                warp_tiles_dense<DTYPE, 2>(q, a, false, t_lo, t_lo + 2 < tile_hi ? t_lo + 2 : tile_hi, lane, out);
            const double e_sum = out.sum();
            if (lane == 0) s_warp[warp] = e_sum;
            __syncthreads();
            for (int w = 0; w < warps; ++w) mass_e += s_warp[w];
        }
        if (threadIdx.x == 0) { a.mass_out[2 * b] = mass_r; a.mass_out[2 * b + 1] = mass_e; }
        return;
    }

    // ---- pass 2 (one block per sequence) ----
    bool residual = q.residual;
    uint32_t flags = residual ? 0u : OD_SF_BONUS;
    const int per = (tile_hi - tile_lo + OD_SAMPLE_THREADS - 1) / OD_SAMPLE_THREADS;
    const int my_lo = tile_lo + threadIdx.x * per < tile_hi ? tile_lo + threadIdx.x * per : tile_hi;
    const int my_hi = my_lo + per < tile_hi ? my_lo + per : tile_hi;
    // tile values (rounding can leave a tile without residual mass slightly negative)
    const float u = od_uniform(seed_b, a.step, (uint32_t)j, 1u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = tile_lo + (int)threadIdx.x + i * OD_SAMPLE_THREADS;
        if (t < tile_hi) s_val[t] = fmax(0.0, first_val[i]);
    }
    for (int t = tile_lo + (int)threadIdx.x + 4 * OD_SAMPLE_THREADS; t < tile_hi; t += OD_SAMPLE_THREADS) s_val[t] = fmax(0.0, __ldcg(tile_val + t));
    __syncthreads();

    double shard_before = 0.0, shard_total = 0.0;      // sums over the shards before this one / all
    const auto share = [&](int s, bool e) -> double {
        if (s < 32) return __shfl_sync(0xFFFFFFFFu, e ? share_e : share_r, s);
        return a.mass_all[((size_t)s * a.B + b) * 2 + (e ? 1 : 0)];
    };
    double tot_r = 0.0, tot_e = 0.0;
    for (int s = 0; s < a.n_shards; ++s) { tot_r += share(s, false); tot_e += share(s, true); }
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
            const double v = share(s, use_e);
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
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_sample_shard_kernel<DTYPE, 1>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = allow_smem(od_sample_shard_kernel<DTYPE, 2>, bytes);
    return e;
}

// Rows beyond 6144 tiles (and the staged probabilities) need more dynamic shared memory than a
// kernel gets by default, and clusters of 16 blocks are not portable: opt in, to the same limit in every
// context (it is the kernel's: a smaller one would take it from a context made earlier), and ask how many
// clusters of each size are resident at a time (0: the device has no room for one; the device must be
// current; allocates nothing).
cudaError_t od_sample_prepare_device(int32_t *clusters, int32_t (*shard_clusters)[OD_SAMPLE_MAX_PARTS + 1])
{
    cudaError_t e = prepare_kernels<OD_BF16>();
    if (e == cudaSuccess) e = prepare_kernels<OD_F32>();
    if (e != cudaSuccess) return e;
    for (int level = 0; level < OD_SAMPLE_LEVELS; ++level)
        clusters[level] = resident_clusters(od_sample_kernel<OD_BF16, true, STAGED>, od_sample_parts(level), 64 * 1024);
    for (int size = 0; size < OD_SHARD_SIZES; ++size) {
        shard_clusters[size][0] = 0;
        for (int parts = 1; parts <= OD_SAMPLE_MAX_PARTS; ++parts)
            shard_clusters[size][parts] = resident_clusters(od_sample_shard_kernel<OD_F32, 1>, parts, 0, OD_SAMPLE_THREADS << size);
    }
    return cudaSuccess;
}

// How a shard's window of `tiles` tiles is cut for B sequences (MODE 1): blocks of a cluster, their threads, tiles of a warp
struct ShardCut {
    int blocks, threads;
    int64_t tiles_per_warp;
};
// As few tiles a warp as give every sequence a cluster that is resident at once, which is asked of the device for every size:
// a cluster is placed as a whole, and those that find no place wait for a whole round (45 sequences, half of 152064 bf16 ids, a
// rank's five calls: 28.0 us with 13 blocks of 256 threads, of which 38 clusters are resident, 24.7 with 10 and 56). A sixteenth of
// the room is left free, or the last ones are placed late (70 sequences, a quarter of 128256 ids: 8 blocks with 71 places
// 23.8, 2 of 1024 threads 22.6). An even number of tiles, since warps work on pairs. Larger blocks where they give each warp
// fewer tiles: in windows that 16 blocks of 256 threads cannot share so finely (one sequence, half of a million ids: 24.1
// and 20.8 with 1024) and for numbers of sequences between theirs (145, half of 152064: 43.5 with 3 of 256, 40.4 with 2 of 512).
static ShardCut shard_cut(const od_ctx *c, int32_t B, int64_t tiles)
{
    const int64_t asked = c->opt_sample_tiles_per_warp;
    for (int64_t tpw = asked > 0 ? asked : 2;; tpw += asked > 0 ? 1 : 2)
        for (int size = 0; size < OD_SHARD_SIZES; ++size) {
            const int threads = OD_SAMPLE_THREADS << size, warps = threads / 32;
            const int64_t blocks = (tiles + tpw * warps - 1) / (tpw * warps);
            if (blocks > OD_SAMPLE_MAX_PARTS) continue;
            const int32_t room = c->shard_clusters[size][blocks];
            const bool fits = asked > 0 ? room > 0 : B <= (blocks > 2 ? room - room / 16 : room);
            if (!fits && (size > 0 || blocks > 1)) continue;    // (single blocks, whatever their number)
            return {(int)blocks, threads, asked > 0 ? tpw : (tiles + blocks * warps - 1) / (blocks * warps)};
        }
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
    ShardCut cut = {1, OD_SAMPLE_THREADS, 1};
    int level = 0;
    if (mode == 0) {
        level = draw_level(c, B);
        cut.blocks = od_sample_parts(level);
    } else if (mode == 1) {
        cut = shard_cut(c, B, tile_hi - tile_lo);
    }
    SampleArgs a = {};
    a.logits = logits; a.row_stride = row_stride; a.seq_stride = seq_stride;
    a.B = B; a.K_max = K_max; a.v_p = mode == 0 ? c->v_p : shard_lo + shard_len;
    a.tiles_per_warp = (int32_t)cut.tiles_per_warp;
    a.row_max = row_max; a.row_sum = row_sum; a.q_rows = q_rows;
    a.draft_ids = draft_ids; a.tgt_ids = tgt_ids; a.q_prime = q_prime;
    a.span_start = span_start; a.span_len = span_len; a.m = m; a.tail_kind = tail_kind;
    a.n_accepted = n_accepted; a.temperature = temperature; a.seed = seed; a.step = step;
    a.out_token = out_token; a.resid_mass = resid_mass; a.flags = flags;
    context_args(c, a);
    a.tile_lo = tile_lo; a.tile_hi = tile_hi; a.col0 = mode == 0 ? 0 : shard_lo;
    a.n_shards = n_shards; a.shard_index = shard_index; a.mass_all = mass_all; a.mass_out = mass_out;
    a.early = c->translation_complete ? 1 : 0;
    if (fuse) {
        a.plan.W = fuse->W; a.plan.n_chunks = fuse->n_chunks; a.plan.span_min = fuse->span_min;
        a.plan.span_a = fuse->span_a; a.plan.seg_warps = fuse->seg_warps; a.plan.partials = c->d_partials;
        a.w_row_max = fuse->row_max; a.w_row_sum = fuse->row_sum; a.w_p_sel = fuse->p_sel; a.w_ratio = fuse->ratio;
        a.w_n_accepted = fuse->n_accepted; a.w_n_draft = fuse->n_draft_accepted; a.w_vflags = fuse->flags;
    }
    if (mode != 1) c->translation_complete = false;         // of this step; the next one has its own
    const DrawPlan plan = mode == 0 ? plan_draw(c, level, a) : DrawPlan{};
    if (mode != 2) {
        c->info[2] = (int64_t)cut.blocks * B;
        c->info[3] = a.tiles_per_warp;
    }

    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = c->opt_pdl ? attr : attr + 1;
    const bool bf = dtype == OD_BF16;
    if (mode == 0) {
        cfg.gridDim = dim3((unsigned)cut.blocks, (unsigned)B);
        cfg.blockDim = dim3(CTHREADS);
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)cut.blocks; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = c->opt_pdl ? 2 : 1;
        cfg.dynamicSmemBytes = plan.smem;
        return bf ? launch_step<OD_BF16>(cfg, a, fuse != nullptr, plan.source) : launch_step<OD_F32>(cfg, a, fuse != nullptr, plan.source);
    }
    cfg.gridDim = dim3((unsigned)B, (unsigned)cut.blocks);
    cfg.blockDim = dim3((unsigned)cut.threads);
    cfg.dynamicSmemBytes = mode == 1 ? 0 : od_sample_smem_bytes(ntiles);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = (unsigned)cut.blocks; attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = (c->opt_pdl ? 1 : 0) + (mode == 1 ? 1 : 0);
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
