// Step 1: translation of the draft proposal into the target vocabulary
// (Section 3.1, Eq. (1); Algorithm 1, translation line).
//
// One thread block per sequence, one warp per proposal offset. Warp s probes
// the n-gram cache for the runs of length 4, 3, 2 that start at offset s: the
// cache is an open-addressing table of 32-slot groups, a probe reads one group
// with one coalesced 256-byte load (lane <-> slot) and resolves it with two
// ballots (key match / empty slot). The first probes of the three lengths are
// issued together, each with the values of its group, so their latencies overlap
// and a hit in the first group costs one memory round trip, and the warp keeps the piece that
// begins at its offset: the longest hit, else the direct map. After a block barrier one warp
// walks the proposal left to right with a shuffle a piece (lane k holds the piece at offset k), and
// its lanes write a piece each. Integer work throughout, except the product
// of at most four fp32 draft probabilities. Bound by latency: the proposal, then the table's groups.
#include "od_common.cuh"
#include "od_lookup.cuh"

namespace {

__global__ void __launch_bounds__(OD_MAX_K *OD_WARP)
od_map_kernel(int32_t B, int32_t K_max, int32_t v_q, const int32_t *__restrict__ draft_ids,
              const int32_t *__restrict__ draft_len, const float *__restrict__ q_sel,
              const int32_t *__restrict__ vocab_map, const uint64_t *__restrict__ keys,
              const int32_t *__restrict__ vals, int64_t cap, const MapOut out, int32_t early)
{
    __shared__ int4 s_piece[OD_MAX_K];                      // the piece that begins at each offset

    const int b = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // The proposal itself (ids, length, probabilities) is the caller's input. Where the
    // caller has promised that it was complete before the launch in front of this one was
    // enqueued (early bit 0), it is requested before the wait. The n-gram table and the
    // vocabulary map belong to the context: unless a kernel that writes the table was
    // launched on this context since the last translation kernel (early bit 1 clear), the
    // probes run before the wait as well, and only the serial walk, which writes, is left
    // for after it. Inside od_step (early bit 2) the next kernel is the streaming pass, which
    // starts on logit rows 0 before its own wait (inputs under the same promise) and releases
    // ITS successor only after that wait: it is released at once, so that rows 0 stream under
    // the tail of the step in front.
    int K = 0;
    int32_t id = -1;                                        // lane k of every warp: position k's id and probability
    float q = 0.f;
    const bool early_proposal = (early & 1) != 0, early_table = (early & 2) != 0, early_release = (early & 4) != 0;
    auto load_proposal = [&]() {
        K = draft_len[b];
        if (lane < K_max) {
            id = draft_ids[(size_t)b * K_max + lane];
            q = q_sel[(size_t)b * K_max + lane];
        }
        K = K < 0 ? 0 : (K > K_max ? K_max : K);
    };
    auto probe = [&]() {
        if (warp >= K) return;
        const int4 piece = look_up_piece(id, q, warp, K, v_q, vocab_map, keys, vals, cap, lane);
        if (lane == 0) s_piece[warp] = piece;
    };
    if (early_release) asm volatile("griddepcontrol.launch_dependents;");
    if (early_proposal && b < B) {
        load_proposal();
        if (early_table) probe();
    }

    // under programmatic dependent launch: wait for everything earlier in the
    // stream first, only then (no promise) let the verification kernel start its prefetch
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!early_release) asm volatile("griddepcontrol.launch_dependents;");

    if (b >= B) return;
    if (!early_proposal) load_proposal();
    if (!(early_proposal && early_table)) probe();
    __syncthreads();
    if (warp == 0) store_walk(out, walk_proposal(lane < K ? s_piece[lane] : make_int4(0, -1, -1, 0), id, K, lane), b, K_max, v_q, lane);
}

}  // namespace

cudaError_t od_launch_map(od_ctx *c, int32_t B, int32_t K_max, const int32_t *draft_ids,
                          const int32_t *draft_len, const float *q_sel, int32_t *tgt_ids,
                          float *q_prime, int32_t *span_start, int32_t *span_len, int32_t *m,
                          uint8_t *tail_kind, uint32_t *counters, bool early, bool release_early,
                          cudaStream_t s)
{
    if (B == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)B);
    cfg.blockDim = dim3((unsigned)(K_max * OD_WARP));
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c->opt_pdl ? 1 : 0;
    c->translation_complete = false;
    // A kernel that writes the table (insert, trim) may be the launch in front of this one: then
    // the probes stay behind the wait. A translation kernel releases its successor after its
    // wait, or (inside od_step) that successor is the streaming pass, which does: either way
    // every later translation kernel starts after those writers are done.
    const int32_t early_bits = early && c->opt_pdl ? (c->table_written ? 1 : 3) | (release_early ? 4 : 0) : 0;
    c->table_written = false;
    return cudaLaunchKernelEx(&cfg, od_map_kernel, B, K_max, c->v_q, draft_ids, draft_len, q_sel,
                              (const int32_t *)c->d_vocab_map, (const uint64_t *)c->d_keys,
                              (const int32_t *)c->d_vals, c->cap,
                              map_out(c, tgt_ids, q_prime, span_start, span_len, m, tail_kind, counters), early_bits);
}
