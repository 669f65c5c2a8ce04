// Hybrid cross-vocabulary distillation loss (Section 3.2, Eq. (3)) and its gradient
// with respect to the drafter's logits, per proposed draft position:
//   directly mapped token (its piece of the translated proposal has one sub-token,
//   target position i):   L = KL(q' || p_i) = sum over mapped draft ids d of
//                             q(d) * (ln q(d) - ln p_i(map[d]))
//   sub-token of a cached n-gram:   L = -lambda * ln q(d_j)   (lambda constant, or the
//                             verified target probability of the n-gram)
//   not translated:       L = 0.
// With q = softmax(z):  KL:  dL/dz(d) = q(d) * (g(d) - sum_e q(e) g(e)),
//                            g(d) = [d mapped] * (ln q(d) - ln p(map[d]) + 1)
//                       NLL: dL/dz(d) = lambda * (q(d) - [d == d_j]).
// ln p_i(t) = (x_t - M_i)/T - ln S_i reuses the row statistics od_verify produced, so
// the target row is only gathered at the mapped ids, never streamed again.
//
// Bound by HBM: the drafter's row and the target row in, the gradient row out. What has to be
// kept from adding to that is the gather, one logit per mapped id, scattered over the target
// row: in draft-id order each takes a line and a 32-byte sector of its own, and the load/store
// units and L2 bound the kernel. So the logits are gathered in TARGET-id order, from lists that
// belong to the context (od_distill_plan): the 32 lanes of a load then sit within 7 lines or so;
// they are put down in shared memory at their draft ids, and everything after that is
// coalesced.
//
// A position is cut into `C` chunks of draft ids, one block of a thread-block cluster each, so
// that three blocks share a multiprocessor and a few positions still fill the chip. Three
// passes: the gather; over the chunk, loss and sum_e q(e) g(e), whose block sums are exchanged over
// distributed shared memory; over the chunk again, the gradient (q from L2, g worked out again).
//
// Measured on 64 x 6 positions of v_q = 32000, v_p = 128256 bf16, 0.6 of them translated: 47.4 ->
// 32.9 us (the bytes alone: 20.7); 5 x 10 positions with v_p = 152064 fp32: 22.7 -> 12.3 us. Per
// block on the former (stamps): 1.1 us to find the piece, 11 the gather (HBM at its rate), 4 the
// sums, 2.3 the exchange, 2 the gradient. The blocks go through these passes together, which
// is what is left. Not kept: probabilities instead of logits in shared memory (two random
// accesses per id instead of one: 38 us), q(d) parked there and four to five blocks of fewer
// threads (39 to 59 us), bulk prefetches of the rows into L2 (no change), one chunk at 64 KB (45 us).
#include <float.h>

#include <vector>

#include "od_common.cuh"

namespace {

constexpr int THREADS = 512;                     // three blocks to a multiprocessor at 40 registers
constexpr int WARPS = THREADS / 32;
constexpr int FEW_EB = 6, FEW_PQ = 4;             // two blocks to a multiprocessor, 64 registers: more in flight (see the launcher)
constexpr int FEW_CHUNK = FEW_PQ * THREADS * 4;

struct DistillArgs {
    int32_t B, K_max, v_q, v_p;
    const float *q_rows;
    const int32_t *draft_ids, *tgt_ids, *span_start, *span_len, *m;
    const void *logits;
    int64_t row_stride, seq_stride;
    const float *row_max, *row_sum, *p_sel, *temperature;
    const int32_t *vocab_map;
    // the context's lists for this launch's number of chunks (od_distill_plan); chunk = draft ids per block
    const int32_t *list_base, *list_ofs;
    const uint32_t *list_word, *mapped_bits;
    int32_t chunk;
    int32_t map_serial;                                      // of the map this launch was laid out for
    const int32_t *map_serial_now;
    float lambda;
    int32_t lambda_mode;
    float *loss, *grad;
};

// log2 on the special-function unit (relative error about 2^-22; the terms it enters are
// weighted by q, so the loss and the gradient see it far below their fp32 rounding)
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// the terms of one mapped id with probability qd and target logit x: loss += q f, qg += q (f + 1);
// returns g = f + 1 (0 for an id without (normal) mass)
struct KlRow {
    float M, scale, lg2_S;
};
__device__ __forceinline__ float kl_term(const KlRow &r, float qd, float x, float &loss, float &qg)
{
    // in base 2: ln q - ln p(t) = ln 2 * (lg2 q - ((x_t - M) * log2(e)/T - lg2 S))
    const bool ok = qd >= FLT_MIN;
    const float f = ok ? 0.6931471805599453f * (lg2_approx(qd) - fmaf(x - r.M, r.scale, -r.lg2_S)) : 0.f;
    const float g = ok ? f + 1.f : 0.f;
    loss += qd * f;
    qg += qd * g;
    return g;
}

// What a block finds out about its position (b, j) first: the piece of the translated proposal
// that covers it, if any. Thread i looks at piece i, whether or not there is one (i < K_max keeps the address inside the
// arrays): one round trip, not one for m and another for the pieces.
__device__ __forceinline__ void find_piece(const DistillArgs &a, int b, int j, int *s_piece, int &piece, int &plen)
{
    if (threadIdx.x < 32) {
        const int i = (int)threadIdx.x;
        int s0 = 0, L = 0;
        if (i < a.K_max) {
            const size_t o = (size_t)b * a.K_max + i;
            s0 = a.span_start[o]; L = a.span_len[o];
        }
        const unsigned covers = __ballot_sync(0xFFFFFFFFu, i < a.m[b] && i < a.K_max && j >= s0 && j < s0 + L);
        const int p = covers ? 31 - __clz(covers) : -1;
        L = __shfl_sync(0xFFFFFFFFu, L, p & 31);
        if (i == 0) { s_piece[0] = p; s_piece[1] = p < 0 ? 0 : L; }
    }
    __syncthreads();
    piece = s_piece[0]; plen = s_piece[1];
}

// Positions without a Kullback-Leibler term, ids [lo, hi) of the gradient row: nothing translated
// there (loss 0), or a sub-token of a cached n-gram (-w ln q(d_j)). `first`: this block writes the loss.
template <bool VEC4>
__device__ __forceinline__ void write_grad_plain(float *grad, const float *q, int lo, int hi, float w, int dj)
{
    if (VEC4) {
        for (int d = lo + (int)threadIdx.x * 4; d < hi; d += THREADS * 4) {
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q) {
                const float4 v = __ldg((const float4 *)(q + d));
                o.x = w * (v.x - (d == dj ? 1.f : 0.f)); o.y = w * (v.y - (d + 1 == dj ? 1.f : 0.f));
                o.z = w * (v.z - (d + 2 == dj ? 1.f : 0.f)); o.w = w * (v.w - (d + 3 == dj ? 1.f : 0.f));
            }
            __stcs((float4 *)(grad + d), o);
        }
    } else {
        for (int d = lo + (int)threadIdx.x; d < hi; d += THREADS) grad[d] = q ? w * (__ldg(q + d) - (d == dj ? 1.f : 0.f)) : 0.f;
    }
}
template <bool VEC4>
__device__ __forceinline__ void plain_position(const DistillArgs &a, int b, int j, int piece, bool ngram, const float *q,
                                               float *grad, int lo, int hi, bool first)
{
    const size_t o = (size_t)b * a.K_max + j;
    if (!ngram) {                                            // not translated: no loss, no gradient
        if (first && threadIdx.x == 0) a.loss[o] = 0.f;
        if (grad) write_grad_plain<VEC4>(grad, nullptr, lo, hi, 0.f, -1);
        return;
    }
    const int32_t dj = a.draft_ids[o];
    const float w = a.lambda_mode == 0 ? a.lambda : a.p_sel[(size_t)b * a.K_max + piece];
    if (first && threadIdx.x == 0) a.loss[o] = (dj >= 0 && dj < a.v_q) ? -w * logf(q[dj]) : 0.f;
    if (grad) write_grad_plain<VEC4>(grad, q, lo, hi, w, dj);
}

__device__ __forceinline__ double block_sum(double v, double *s_red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < THREADS / 32; ++w) t += s_red[w];   // the same order in every thread
    return t;
}

// A logit as it is stored
template <int DTYPE>
struct Logit {
    typedef float raw;
    static __device__ __forceinline__ float load(const float *p) { return *p; }
    static __device__ __forceinline__ float4 load4(const float *p) { return *(const float4 *)p; }
    static __device__ __forceinline__ float4 load4_global(const float *p) { return __ldg((const float4 *)p); }
    static __device__ __forceinline__ void store4(float *p, float4 v) { *(float4 *)p = v; }
};
template <>
struct Logit<OD_BF16> {
    typedef unsigned short raw;
    static __device__ __forceinline__ float load(const raw *p) { return __uint_as_float((uint32_t)*p << 16); }
    static __device__ __forceinline__ float4 load4(const raw *p)
    {
        const uint2 v = *(const uint2 *)p;
        return make_float4(od_bf16_lo(v.x), od_bf16_hi(v.x), od_bf16_lo(v.y), od_bf16_hi(v.y));
    }
    static __device__ __forceinline__ float4 load4_global(const raw *p)
    {
        const uint2 v = __ldg((const uint2 *)p);
        return make_float4(od_bf16_lo(v.x), od_bf16_hi(v.x), od_bf16_lo(v.y), od_bf16_hi(v.y));
    }
    static __device__ __forceinline__ void store4(raw *p, float4 v)   // (exact: the values are bf16)
    {
        *(uint2 *)p = make_uint2(__float_as_uint(v.x) >> 16 | (__float_as_uint(v.y) & 0xFFFF0000u),
                                 __float_as_uint(v.z) >> 16 | (__float_as_uint(v.w) & 0xFFFF0000u));
    }
};

// One position by one block, every id looked up in the map: a launch for shared ids under another map (the
// other kernels read lists that are the present map's whenever they were laid out). Out of line: loops in the
// kernel below, in all its forms, cost 0.15 us of 5 to 13 although they are not run.
template <int DTYPE>
__device__ __noinline__ void looked_up_position(const DistillArgs &a, int b, int j, int *s_piece, double *s_red)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int piece, plen;
    find_piece(a, b, j, s_piece, piece, plen);
    const float T = a.temperature[b];
    const bool translated = piece >= 0 && T > 0.f;
    const size_t o = (size_t)b * a.K_max + j, row_of = (size_t)b * (a.K_max + 1) + piece;
    const char *row = (const char *)a.logits + ((size_t)b * a.seq_stride + (size_t)piece * a.row_stride) * (DTYPE == OD_BF16 ? 2 : 4);
    const float *q = a.q_rows + o * a.v_q;
    float *grad = a.grad ? a.grad + o * a.v_q : nullptr;
    if (!translated || plen >= 2) {
        plain_position<false>(a, b, j, piece, translated, q, grad, 0, a.v_q, true);
        return;
    }
    KlRow kl;
    kl.M = a.row_max[row_of];
    kl.scale = 1.4426950408889634f / T;
    kl.lg2_S = lg2_approx(a.row_sum[row_of]);
    float loss_t = 0.f, qg_t = 0.f;
    const auto g_of = [&](int d, float v) {
        const int32_t t = __ldg(a.vocab_map + d);
        return kl_term(kl, t >= 0 ? v : 0.f, od_load_logit<DTYPE>(row, t >= 0 ? t : 0), loss_t, qg_t);
    };
    for (int d = threadIdx.x; d < a.v_q; d += THREADS) g_of(d, __ldg(q + d));
    const double l = block_sum((double)loss_t, s_red), qg = block_sum((double)qg_t, s_red);
    if (threadIdx.x == 0) a.loss[o] = (float)l;
    if (!grad) return;
    for (int d = threadIdx.x; d < a.v_q; d += THREADS) {
        const float v = __ldg(q + d);
        grad[d] = fmaf(-v, (float)qg, v * g_of(d, v));
    }
}

// Grid (C, K, B), clusters of C blocks. VEC4: the draft vocabulary is a multiple of 4 and the
// rows are 16-byte aligned, so the coalesced accesses (q, gradient) move four ids per
// instruction; chunks are multiples of 32 ids. SAME: target ids are draft ids, nothing is
// gathered; the logits wait in shared memory for the gradient.
template <int DTYPE, bool VEC4, bool SAME, int RESIDENT>
__global__ void __launch_bounds__(THREADS, RESIDENT)
od_distill_kernel(const __grid_constant__ DistillArgs a)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];   // [chunk] the logit of each mapped id, at its draft id
    typedef typename Logit<DTYPE>::raw raw_t;
    raw_t *s_x = (raw_t *)s_dyn;
    __shared__ double s_red[2][WARPS], s_all[OD_DISTILL_MAX_CHUNKS][2];
    __shared__ int s_piece[2];
    const int rank = blockIdx.x, C = gridDim.x, j = blockIdx.y, b = blockIdx.z;
    const int lo = rank * a.chunk < a.v_q ? rank * a.chunk : a.v_q;
    const int hi = lo + a.chunk < a.v_q ? lo + a.chunk : a.v_q;
    const float *q = a.q_rows + ((size_t)b * a.K_max + j) * a.v_q;
    float *grad = a.grad ? a.grad + ((size_t)b * a.K_max + j) * a.v_q : nullptr;
    // The chunk's list: groups of 32 entries, one per lane (od_distill_lists). It belongs to the
    // context: the first entries are requested before the wait, the others a batch ahead.
    // groups per warp and batch (five in 40 registers: one chunk of 8000 bf16 ids 2 to 7 % slower, 32000 in four 2 to 4 %,
    // 64 x 6 of 32000 and 128256 1 % faster)
    constexpr int EB = RESIDENT == 2 ? FEW_EB : 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2 groups = SAME ? make_int2(0, 0) : __ldg((const int2 *)a.list_ofs + rank);
    const int g_hi = groups.y;
    int g_at = groups.x + warp;                          // this warp's next group to request
    uint32_t word[EB];
    int32_t base[EB];
    auto load_words = [&]() {
#pragma unroll
        for (int e = 0; e < EB; ++e) {
            const bool in = g_at + e * WARPS < g_hi;
            word[e] = in ? __ldg(a.list_word + (size_t)(g_at + e * WARPS) * 32 + lane) : 0xFFFFu;
            base[e] = in ? __ldg(a.list_base + g_at + e * WARPS) : 0;
        }
        g_at += EB * WARPS;
    };
    if (!SAME) load_words();
    const int32_t map_serial = SAME ? __ldg(a.map_serial_now) : a.map_serial;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float T = a.temperature[b];
    int piece, plen;
    find_piece(a, b, j, s_piece, piece, plen);
    const bool translated = piece >= 0 && T > 0.f;
    if (SAME && map_serial != a.map_serial) {                // ids are not shared any more (asked here, where the answer has arrived)
        if (rank == 0) looked_up_position<DTYPE>(a, b, j, s_piece, s_red[0]);
        return;
    }
    if (!translated || plen >= 2) {                          // the same for every block of the cluster
        plain_position<VEC4>(a, b, j, piece, translated, q, grad, lo, hi, rank == 0);
        return;
    }
    od_cluster_arrive();                                     // this block runs: the others may store to it (waited for below)
    // ---- a directly mapped token: KL(q' || p_i) over the mapped ids
    const char *row = (const char *)a.logits + ((size_t)b * a.seq_stride + (size_t)piece * a.row_stride) * sizeof(raw_t);
    const float M = a.row_max[b * (a.K_max + 1) + piece], S = a.row_sum[b * (a.K_max + 1) + piece];
    KlRow kl;
    kl.M = M;
    kl.scale = 1.4426950408889634f / T;
    float loss_t = 0.f, qg_t = 0.f;
    // four ids from d: their probabilities with 0 for the ids without a map
    auto mapped4 = [&](int d, float4 v) {
        if (SAME) return v;
        const uint32_t w = __ldg(a.mapped_bits + (d >> 5)) >> (d & 31);
        return make_float4(w & 1u ? v.x : 0.f, w & 2u ? v.y : 0.f, w & 4u ? v.z : 0.f, w & 8u ? v.w : 0.f);
    };
    auto mapped1 = [&](int d, float v) {
        return SAME || (__ldg(a.mapped_bits + (d >> 5)) >> (d & 31) & 1u) ? v : 0.f;
    };
    // four ids' terms before they meet the running sums
    auto sum4 = [&](float4 v, float4 x) {
        float l = 0.f, g = 0.f;
        kl_term(kl, v.x, x.x, l, g); kl_term(kl, v.y, x.y, l, g);
        kl_term(kl, v.z, x.z, l, g); kl_term(kl, v.w, x.w, l, g);
        loss_t += l; qg_t += g;
    };
    const raw_t *xrow = (const raw_t *)row;
    constexpr bool KEEP = RESIDENT == 2;                     // the chunk's probabilities stay in registers
    float4 kept[KEEP ? FEW_PQ : 1];
    if (!SAME) {
        // (the first probabilities travel meanwhile)
        constexpr int PQ = 2;                                // vectors of four probabilities in flight per thread
        float4 qv[PQ];
        if (KEEP) {
#pragma unroll
            for (int i = 0; i < FEW_PQ; ++i) {
                const int d = lo + (int)threadIdx.x * 4 + i * THREADS * 4;
                if (d < hi) kept[KEEP ? i : 0] = __ldg((const float4 *)(q + d));
            }
        } else if (VEC4) {
#pragma unroll
            for (int i = 0; i < PQ; ++i) {
                const int d = lo + (int)threadIdx.x * 4 + i * THREADS * 4;
                if (d < hi) qv[i] = __ldg((const float4 *)(q + d));
            }
        }
        // ---- the chunk's logits, gathered in target-id order, to their draft ids in shared memory
        for (;;) {
            raw_t x[EB];
            uint32_t at[EB];
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                at[e] = word[e] & 0xFFFFu;
                if (at[e] != 0xFFFFu) x[e] = __ldg((const raw_t *)row + base[e] + (int)(word[e] >> 16));
            }
            const bool more = g_at < g_hi;                   // the same for every lane of a warp
            if (more) load_words();
#pragma unroll
            for (int e = 0; e < EB; ++e)
                if (at[e] != 0xFFFFu) s_x[at[e]] = x[e];
            if (!more) break;
        }
        kl.lg2_S = lg2_approx(S);
        __syncthreads();
        // ---- the loss and sum_e q(e) g(e)
        if (KEEP) {
#pragma unroll
            for (int i = 0; i < FEW_PQ; ++i) {
                const int d = lo + (int)threadIdx.x * 4 + i * THREADS * 4;
                if (d < hi) sum4(mapped4(d, kept[KEEP ? i : 0]), Logit<DTYPE>::load4(s_x + (d - lo)));
            }
        } else if (VEC4) {
            const int d0 = lo + (int)threadIdx.x * 4;
            for (int d1 = d0; d1 < hi; d1 += PQ * THREADS * 4) {
                float4 nx[PQ];
#pragma unroll
                for (int i = 0; i < PQ; ++i) {
                    const int d = d1 + (i + PQ) * THREADS * 4;
                    if (d < hi) nx[i] = __ldg((const float4 *)(q + d));
                }
#pragma unroll
                for (int i = 0; i < PQ; ++i) {
                    const int d = d1 + i * THREADS * 4;
                    if (d < hi) sum4(mapped4(d, qv[i]), Logit<DTYPE>::load4(s_x + (d - lo)));
                }
#pragma unroll
                for (int i = 0; i < PQ; ++i) qv[i] = nx[i];
            }
        } else {
#pragma unroll 4
            for (int d = lo + (int)threadIdx.x; d < hi; d += THREADS)
                kl_term(kl, mapped1(d, __ldg(q + d)), Logit<DTYPE>::load(s_x + (d - lo)), loss_t, qg_t);
        }
    } else {
        kl.lg2_S = lg2_approx(S);
        if (VEC4) {
            constexpr int EV = 2;                            // vectors of four ids in flight per thread
            for (int d1 = lo + (int)threadIdx.x * 4; d1 < hi; d1 += EV * THREADS * 4) {
                float4 v[EV], x[EV];
#pragma unroll
                for (int i = 0; i < EV; ++i) {
                    const int d = d1 + i * THREADS * 4;
                    if (d < hi) { v[i] = __ldg((const float4 *)(q + d)); x[i] = Logit<DTYPE>::load4_global(xrow + d); }
                }
#pragma unroll
                for (int i = 0; i < EV; ++i) {
                    const int d = d1 + i * THREADS * 4;
                    if (d >= hi) continue;
                    if (grad) Logit<DTYPE>::store4(s_x + (d - lo), x[i]);
                    sum4(v[i], x[i]);
                }
            }
        } else {
#pragma unroll 4
            for (int d = lo + (int)threadIdx.x; d < hi; d += THREADS) {
                const raw_t x = __ldg(xrow + d);
                if (grad) s_x[d - lo] = x;
                kl_term(kl, __ldg(q + d), Logit<DTYPE>::load(&x), loss_t, qg_t);
            }
        }
    }
    // the block's two sums, to every block of the cluster
    {
        double l = loss_t, g = qg_t;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            l += __shfl_xor_sync(0xFFFFFFFFu, l, off);
            g += __shfl_xor_sync(0xFFFFFFFFu, g, off);
        }
        if (lane == 0) { s_red[0][warp] = l; s_red[1][warp] = g; }
        od_cluster_wait();
        __syncthreads();
        if (warp == 0) {
            const int which = lane >> 4, w = lane & 15;
            static_assert(WARPS <= 16, "one lane per warp and sum");
            double v = w < WARPS ? s_red[which][w] : 0.0;
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
            // lanes 0.. store the loss, lanes 16.. the other sum, one block of the cluster each
            if (w < C) od_cluster_store(&s_all[rank][which], (uint32_t)w, v);
        }
        od_cluster_arrive();
        od_cluster_wait();
    }
    double loss = 0.0, qg = 0.0;
    for (int r = 0; r < C; ++r) { loss += s_all[r][0]; qg += s_all[r][1]; }   // the same order in every block
    if (rank == 0 && threadIdx.x == 0) a.loss[(size_t)b * a.K_max + j] = (float)loss;
    if (!grad) return;
    // ---- the gradient: q(d) (g(d) - sum_e q(e) g(e))
    const float gbar = (float)qg;
    if (KEEP) {
#pragma unroll
        for (int i = 0; i < FEW_PQ; ++i) {
            const int d = lo + (int)threadIdx.x * 4 + i * THREADS * 4;
            if (d >= hi) continue;
            const float4 v = kept[KEEP ? i : 0], u = mapped4(d, v);
            const float4 x = Logit<DTYPE>::load4(s_x + (d - lo));
            float4 o;
            o.x = fmaf(-v.x, gbar, v.x * kl_term(kl, u.x, x.x, loss_t, qg_t));
            o.y = fmaf(-v.y, gbar, v.y * kl_term(kl, u.y, x.y, loss_t, qg_t));
            o.z = fmaf(-v.z, gbar, v.z * kl_term(kl, u.z, x.z, loss_t, qg_t));
            o.w = fmaf(-v.w, gbar, v.w * kl_term(kl, u.w, x.w, loss_t, qg_t));
            __stcs((float4 *)(grad + d), o);
        }
    } else if (VEC4) {
#pragma unroll 4
        for (int d = lo + (int)threadIdx.x * 4; d < hi; d += THREADS * 4) {
            const float4 v = __ldg((const float4 *)(q + d)), u = mapped4(d, v);
            const float4 x = Logit<DTYPE>::load4(s_x + (d - lo));
            float4 o;
            o.x = fmaf(-v.x, gbar, v.x * kl_term(kl, u.x, x.x, loss_t, qg_t));
            o.y = fmaf(-v.y, gbar, v.y * kl_term(kl, u.y, x.y, loss_t, qg_t));
            o.z = fmaf(-v.z, gbar, v.z * kl_term(kl, u.z, x.z, loss_t, qg_t));
            o.w = fmaf(-v.w, gbar, v.w * kl_term(kl, u.w, x.w, loss_t, qg_t));
            __stcs((float4 *)(grad + d), o);
        }
    } else {
#pragma unroll 4
        for (int d = lo + (int)threadIdx.x; d < hi; d += THREADS) {
            const float v = __ldg(q + d), x = Logit<DTYPE>::load(s_x + (d - lo));
            grad[d] = fmaf(-v, gbar, v * kl_term(kl, mapped1(d, v), x, loss_t, qg_t));
        }
    }
}

// One block per position, the ids in draft order, each gathering its logit; q(d) g(d) waits in
// the gradient row for the second sweep.
template <int DTYPE, bool VEC4>
__global__ void __launch_bounds__(THREADS, 2)
od_distill_position_kernel(const DistillArgs a)
{
    __shared__ double s_red[THREADS / 32];
    __shared__ int s_piece[2];
    const int j = blockIdx.x, b = blockIdx.y;
    const float *q = a.q_rows + ((size_t)b * a.K_max + j) * a.v_q;
    float *grad = a.grad ? a.grad + ((size_t)b * a.K_max + j) * a.v_q : nullptr;
    int piece, plen;
    find_piece(a, b, j, s_piece, piece, plen);
    const float T = a.temperature[b];
    const bool translated = piece >= 0 && T > 0.f;
    if (!translated || plen >= 2) {
        plain_position<VEC4>(a, b, j, piece, translated, q, grad, 0, a.v_q, true);
        return;
    }
    const size_t esz = DTYPE == OD_BF16 ? 2 : 4;
    const char *row = (const char *)a.logits + ((size_t)b * a.seq_stride + (size_t)piece * a.row_stride) * esz;
    // the gathers touch practically every sector of the row in no particular order: the copy
    // engine brings it into L2 as one sequential transfer
    if (threadIdx.x == 0) {
        const uint32_t bytes = (uint32_t)((size_t)a.v_p * esz / 16 * 16);
        if (bytes) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row), "r"(bytes) : "memory");
    }
    KlRow kl;
    kl.M = a.row_max[b * (a.K_max + 1) + piece];
    kl.lg2_S = lg2_approx(a.row_sum[b * (a.K_max + 1) + piece]);
    kl.scale = 1.4426950408889634f / T;
    float loss_t = 0.f, qg_t = 0.f;
    // one id: q (negative = no map) and its gathered logit; returns q(d) g(d)
    auto term = [&](float qs, float x) -> float {
        const bool ok = qs >= FLT_MIN;
        const float qa = fabsf(qs);
        const float f = ok ? 0.6931471805599453f * (lg2_approx(qa) - fmaf(x - kl.M, kl.scale, -kl.lg2_S)) : 0.f;
        const float g = ok ? f + 1.f : 0.f;
        loss_t += qa * f;
        qg_t += qa * g;
        return qa * g;
    };
    if (VEC4) {
        constexpr int EV = 4;                                // vectors of 4 ids in flight per thread
        for (int base = threadIdx.x * 4; base < a.v_q; base += THREADS * 4 * EV) {
            int4 t[EV];
            float4 qv[EV];
#pragma unroll
            for (int e = 0; e < EV; ++e) {
                const int d = base + e * THREADS * 4;
                t[e] = d < a.v_q ? __ldg((const int4 *)(a.vocab_map + d)) : make_int4(-1, -1, -1, -1);
                qv[e] = d < a.v_q ? __ldg((const float4 *)(q + d)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float x[EV][4];
#pragma unroll
            for (int e = 0; e < EV; ++e) {
                x[e][0] = od_load_logit<DTYPE>(row, t[e].x >= 0 ? t[e].x : 0);
                x[e][1] = od_load_logit<DTYPE>(row, t[e].y >= 0 ? t[e].y : 0);
                x[e][2] = od_load_logit<DTYPE>(row, t[e].z >= 0 ? t[e].z : 0);
                x[e][3] = od_load_logit<DTYPE>(row, t[e].w >= 0 ? t[e].w : 0);
            }
#pragma unroll
            for (int e = 0; e < EV; ++e) {
                const int d = base + e * THREADS * 4;
                float4 o;
                o.x = term(t[e].x < 0 ? -qv[e].x : qv[e].x, x[e][0]);
                o.y = term(t[e].y < 0 ? -qv[e].y : qv[e].y, x[e][1]);
                o.z = term(t[e].z < 0 ? -qv[e].z : qv[e].z, x[e][2]);
                o.w = term(t[e].w < 0 ? -qv[e].w : qv[e].w, x[e][3]);
                if (grad && d < a.v_q) *(float4 *)(grad + d) = o;
            }
        }
    } else {
        constexpr int EB = 16;
        for (int base = threadIdx.x; base < a.v_q; base += THREADS * EB) {
            float qd[EB], x[EB];
            {
                int32_t t[EB];
#pragma unroll
                for (int e = 0; e < EB; ++e) {
                    const int d = base + e * THREADS;
                    t[e] = d < a.v_q ? __ldg(a.vocab_map + d) : -1;
                    qd[e] = d < a.v_q ? __ldg(q + d) : 0.f;
                }
#pragma unroll
                for (int e = 0; e < EB; ++e)
                    if (t[e] < 0) qd[e] = -qd[e];
#pragma unroll
                for (int e = 0; e < EB; ++e) x[e] = od_load_logit<DTYPE>(row, t[e] >= 0 ? t[e] : 0);
            }
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                const int d = base + e * THREADS;
                const float v = term(qd[e], x[e]);
                if (grad && d < a.v_q) grad[d] = v;
            }
        }
    }
    const double loss = block_sum((double)loss_t, s_red), qg = block_sum((double)qg_t, s_red);
    if (threadIdx.x == 0) a.loss[(size_t)b * a.K_max + j] = (float)loss;
    if (!grad) return;
    // every thread revisits the ids it wrote itself: no barrier for the parked values
    const float gbar = (float)qg;
    if (VEC4) {
#pragma unroll 4
        for (int d = threadIdx.x * 4; d < a.v_q; d += THREADS * 4) {
            const float4 v = __ldg((const float4 *)(q + d));
            float4 g = *(float4 *)(grad + d);
            g.x = fmaf(-v.x, gbar, g.x); g.y = fmaf(-v.y, gbar, g.y); g.z = fmaf(-v.z, gbar, g.z); g.w = fmaf(-v.w, gbar, g.w);
            *(float4 *)(grad + d) = g;
        }
    } else {
#pragma unroll 4
        for (int d = threadIdx.x; d < a.v_q; d += THREADS) grad[d] = fmaf(-__ldg(q + d), gbar, grad[d]);
    }
}

template <int DTYPE, bool VEC4, bool SAME, int RESIDENT>
cudaError_t launch_chunks(const DistillArgs &a, int C, bool pdl, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C, (unsigned)a.K_max, (unsigned)a.B);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SAME && !a.grad ? 0 : (size_t)a.chunk * (DTYPE == OD_BF16 ? 2 : 4);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, od_distill_kernel<DTYPE, VEC4, SAME, RESIDENT>, a);
}
template <int DTYPE, bool VEC4>
cudaError_t launch(const DistillArgs &a, int C, bool same, bool few, bool pdl, cudaStream_t s)
{
    if (C == 0) {
        od_distill_position_kernel<DTYPE, VEC4><<<dim3((unsigned)a.K_max, (unsigned)a.B), THREADS, 0, s>>>(a);
        return cudaGetLastError();
    }
    if (same) return launch_chunks<DTYPE, VEC4, true, 3>(a, C, pdl, s);
    if constexpr (VEC4)
        if (few) return launch_chunks<DTYPE, true, false, 2>(a, C, pdl, s);
    return launch_chunks<DTYPE, VEC4, false, 3>(a, C, pdl, s);
}

// draft ids per chunk for a vocabulary cut into C = 1 << level chunks: whole words of the mapped
// bits, and each a run of the same eighths
int32_t fine_ids(int32_t v_q) { return ((v_q + 7) / 8 + 31) / 32 * 32; }
int32_t chunk_ids(int32_t v_q, int level) { return fine_ids(v_q) << (OD_DISTILL_LEVELS - 1 - level); }
constexpr int CHUNK_BYTES = 36 * 1024;
static_assert(1 << (OD_DISTILL_LEVELS - 1) == OD_DISTILL_MAX_CHUNKS && OD_DISTILL_MAX_CHUNKS == 8, "the finest level");

}  // namespace

cudaError_t od_launch_distill(od_ctx *c, int32_t B, int32_t K_max, const float *q_rows,
                              const int32_t *draft_ids, const int32_t *tgt_ids, const int32_t *span_start,
                              const int32_t *span_len, const int32_t *m, const void *logits, int32_t dtype,
                              int64_t row_stride, int64_t seq_stride, const float *row_max,
                              const float *row_sum, const float *p_sel, const float *temperature,
                              float lambda, int32_t lambda_mode, float *loss, float *grad, cudaStream_t s)
{
    if (B == 0) return cudaSuccess;
    DistillArgs a = {};
    a.B = B; a.K_max = K_max; a.v_q = c->v_q; a.v_p = c->v_p;
    a.q_rows = q_rows; a.draft_ids = draft_ids; a.tgt_ids = tgt_ids; a.span_start = span_start;
    a.span_len = span_len; a.m = m; a.logits = logits; a.row_stride = row_stride; a.seq_stride = seq_stride;
    a.row_max = row_max; a.row_sum = row_sum; a.p_sel = p_sel; a.temperature = temperature;
    a.vocab_map = c->d_vocab_map; a.map_serial = c->map_serial; a.map_serial_now = c->d_map_serial; a.lambda = lambda; a.lambda_mode = lambda_mode; a.loss = loss; a.grad = grad;
    const bool bf = dtype == OD_BF16, same = c->map_same_ids, pdl = c->opt_pdl != 0;
    const bool vec4 = c->v_q % 4 == 0 && ((uintptr_t)q_rows & 15u) == 0 && (!grad || ((uintptr_t)grad & 15u) == 0);
    // The number of chunks: the fewest with which a chunk's logits take 36 KB or less (what is left of
    // a multiprocessor's memory is the L1 that the gather lives on: 32000 bf16 ids in two chunks of
    // 32 KB 34.9 us, in one of 64 KB 44.7, in four 38), more while all blocks still fit one resident
    // wave (a few positions: 5 x 10 at v_q = 32000 takes 8 chunks).
    int level = 0;
    const auto more = [&](int l) { return l + 1 < OD_DISTILL_LEVELS; };
    const int64_t positions = (int64_t)B * K_max, wave = (int64_t)c->sm_count * 3;
    while (more(level) && !(same && !grad) && chunk_ids(c->v_q, level) * (bf ? 2 : 4) > (same ? 2 : 1) * CHUNK_BYTES) ++level;
    while (more(level) && positions * 2 << level <= wave) ++level;
    a.chunk = chunk_ids(c->v_q, level);
    // Where two blocks to a multiprocessor hold them all, they have 64 registers instead of 40: six groups of the list in
    // flight, and a thread's probabilities stay in registers from the sums to the gradient (128256 bf16 / 152064 fp32 ids, 1 x 4
    // 6.55 -> 6.05 us / 6.6 -> 6.3, 5 x 5 8.3 -> 7.6 / 8.6 -> 8.1, 12 x 6 11.8 -> 10.3 / 12.2 -> 11.1; 8 or 10 groups spill).
    // The device says how many clusters it holds (33 of 8 blocks, where 296 blocks would be 37: 6 x 6 positions of 128256 bf16 ids
    // 8.3 us with 40 registers, 9.4 with 64). One in 32 too many is no loss: positions without a translation leave at once (71 of
    // 4 blocks: 12 x 6 are faster by 3 to 17 % in eleven of twelve forms).
    const int64_t room = c->distill_few_clusters[level];
    const bool few = !same && vec4 && a.chunk <= FEW_CHUNK && positions << level <= (int64_t)c->sm_count * 2 && positions <= room + room / 32;
    // One block per position instead where the chunks would not fit, or where the target row is so
    // short that the gather in draft order finds its lines in L1 and there are positions enough
    // (128 x 10, v_q = 32000, 22400 ids mapped, v_p = 34330 / 45000 / 64000 / 128000: without a gradient
    // 43 / 32 / 34 / 45 us against 55 / 36 / 36 / 40, with one 80 / 59 / 65 us against 81 / 53 / 54),
    // or where target ids are draft ids, so that the gather is coalesced as it stands (64 x 6 at 32000:
    // 27.8 us against 28.2, without a gradient 16.6 against 19.0; 5 x 6: 12.4 against 5.5).
    const int64_t short_row = c->n_mapped * (grad ? 9 : 16) / 5;
    int C = 1 << level;
    if ((a.chunk > OD_DISTILL_MAX_CHUNK_IDS && !(same && !grad)) ||
        (!same && c->v_p < short_row && positions >= wave) || (same && vec4 && positions >= c->sm_count * 2)) C = 0;
    const OdDistillLists l = od_distill_lists(c->d_distill_lists, c->v_q, c->v_p);
    a.list_word = l.word + (size_t)level * l.groups * 32; a.list_base = l.base + (size_t)level * l.groups;
    a.list_ofs = l.ofs + level * OD_DISTILL_MAX_CHUNKS * 2; a.mapped_bits = l.bits;
    if (vec4) return bf ? launch<OD_BF16, true>(a, C, same, few, pdl, s) : launch<OD_F32, true>(a, C, same, few, pdl, s);
    return bf ? launch<OD_BF16, false>(a, C, same, few, pdl, s) : launch<OD_F32, false>(a, C, same, few, pdl, s);
}

// Clusters of each number of chunks that are resident with two blocks to a multiprocessor
void od_distill_resident(int32_t *clusters)
{
    for (int level = 0; level < OD_DISTILL_LEVELS; ++level) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1u << level); cfg.blockDim = dim3(THREADS); cfg.dynamicSmemBytes = FEW_CHUNK * 4;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1u << level; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, od_distill_kernel<OD_F32, true, false, 2>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        clusters[level] = n;
    }
}

// The kernels' dynamic shared memory (a chunk of a draft vocabulary of v_q ids): opt in where it
// exceeds the default (the device must be current; allocates nothing).
cudaError_t od_distill_prepare_device(int32_t v_q)
{
    const int n = OD_DISTILL_MAX_CHUNK_IDS * 4;
    if (chunk_ids(v_q, 0) * 4 <= 48 * 1024) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(od_distill_kernel<OD_BF16, true, false, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_F32, true, false, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_BF16, false, false, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_F32, false, false, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_BF16, true, true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_F32, true, true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_BF16, false, true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(od_distill_kernel<OD_F32, false, true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    return e;
}

// The gather lists of the distillation kernel, on the host, in the layout of od_distill_lists.
void od_distill_plan(int32_t v_q, int32_t v_p, const OdMappedIds &mapped, void *out)
{
    const OdDistillLists l = od_distill_lists(out, v_q, v_p);
    for (int w = 0; w < (v_q + 31) / 32; ++w) l.bits[w] = 0u;
    for (int32_t d : mapped.draft) l.bits[d >> 5] |= 1u << (d & 31);
    const int32_t fine = fine_ids(v_q);
    std::vector<uint8_t> eighth((size_t)(v_q + 31) / 32);    // of 32 ids
    for (size_t w = 0; w < eighth.size(); ++w) eighth[w] = (uint8_t)((int32_t)w * 32 / fine);
    int first = OD_DISTILL_LEVELS - 1;                       // the coarsest level that a launch can ask for
    while (first > 0 && chunk_ids(v_q, first - 1) * 2 <= CHUNK_BYTES) --first;
    for (int level = 0; level < OD_DISTILL_LEVELS; ++level) {
        uint32_t *words = l.word + (size_t)level * l.groups * 32, *next[OD_DISTILL_MAX_CHUNKS];   // a chunk's next entry
        int32_t *bases = l.base + (size_t)level * l.groups, *ofs = l.ofs + level * OD_DISTILL_MAX_CHUNKS * 2;
        for (int k = 0; k < OD_DISTILL_MAX_CHUNKS; ++k) {
            ofs[k * 2] = ofs[k * 2 + 1] = (int32_t)(k * (l.groups >> level));
            next[k] = words + (size_t)ofs[k * 2] * 32;
        }
        if (level < first) continue;
        const int32_t shift = OD_DISTILL_LEVELS - 1 - level;
        // a chunk's entries in target-id order; groups end with 65536 target ids, of which the first is their base
        size_t i = 0;
        for (int32_t page = 0; page < v_p; page += 65536) {
            // (a chunk of more than OD_DISTILL_MAX_CHUNK_IDS ids is not asked for: the cut does not matter)
            for (; i < mapped.target.size() && mapped.target[i] - page < 65536; ++i) {
                const int32_t d = mapped.draft[i], k = eighth[d >> 5] >> shift;
                *next[k]++ = (uint32_t)(mapped.target[i] - page) << 16 | (uint32_t)((d - (k << shift) * fine) & 0xFFFF);
            }
            for (int k = 0; k < 1 << level; ++k) od_end_group(words, next[k], bases, page, ofs[k * 2 + 1]);
        }
    }
}
