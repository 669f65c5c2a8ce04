// Adaptive-drafting exit rule (Section 3.3, Eq. (4)-(6)): from the acceptance head's
// outputs f_phi(e_i) of the proposed tokens, the probability that some token up to
// k is rejected, 1 - prod_{i<=k} sigmoid(f_i), and the draft length: the first k at
// which that probability exceeds gamma (all available tokens if it never does).
// The result is the ragged draft_len that od_map_proposals takes.
//
// A few dozen flops per sequence, bound by latency: sixteen lanes per sequence, a token each, so that the loads
// and the sigmoids of all tokens run at once; the product is taken in token order exactly as the definition
// reads, a shuffle a token, in fp32. (One thread per sequence loaded a token at a time: the rule and a step for one
// sequence, 10 tokens, 16.5 us, so 14.2.) Launched with programmatic stream serialization: it waits at once.
#include "od_common.cuh"

namespace {

__device__ __forceinline__ float sigmoid_f32(float x)
{
    // the two branches avoid overflow of exp for large |x|
    if (x >= 0.f) return 1.f / (1.f + expf(-x));
    const float e = expf(x);
    return e / (1.f + e);
}

constexpr int LANES = 16;                                  // of a sequence
static_assert(OD_MAX_K <= LANES, "a lane per token");

__global__ void od_exit_kernel(int32_t B, int32_t K_max, const float *__restrict__ head_logits,
                               const int32_t *__restrict__ avail_len, float gamma,
                               int32_t *__restrict__ draft_len, float *__restrict__ reject_prob,
                               uint32_t *__restrict__ flags)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const unsigned b = blockIdx.x * (blockDim.x / LANES) + threadIdx.x / LANES;
    const int i = threadIdx.x % LANES, shift = threadIdx.x & 31 & ~(LANES - 1);
    const bool live = b < (unsigned)B;
    int n = 0;
    float x = 0.f;
    if (live) {
        n = avail_len ? avail_len[b] : K_max;
        if (i < K_max) x = head_logits[(size_t)b * K_max + i];
    }
    n = n < 0 ? 0 : (n > K_max ? K_max : n);
    const float sig = sigmoid_f32(x);
    float keep = 1.f, mine = 1.f;                          // running product of Eq. (5)
#pragma unroll
    for (int k = 0; k < LANES; ++k) {
        const float s = __shfl_sync(0xFFFFFFFFu, sig, k, LANES);
        if (k < n) keep *= s;
        if (k == i) mine = keep;
    }
    const float rej = i < n ? 1.f - mine : 0.f;
    const unsigned over = __ballot_sync(0xFFFFFFFFu, i < n && rej > gamma) >> shift & 0xFFFFu;
    const unsigned near = __ballot_sync(0xFFFFFFFFu, i < n && fabsf(rej - gamma) <= OD_TAU_EXIT) >> shift & 0xFFFFu;
    if (!live) return;
    if (reject_prob && i < K_max) reject_prob[(size_t)b * K_max + i] = rej;
    if (i == 0) {
        const int first = over ? __ffs(over) - 1 : LANES - 1;
        draft_len[b] = over ? first + 1 : n;
        // fp32 may land on the other side: at the token whose test fires, or before it
        if (flags) flags[b] = near & ((2u << first) - 1u);
    }
}

}  // namespace

cudaError_t od_launch_exit(int32_t B, int32_t K_max, const float *head_logits, const int32_t *avail_len,
                           float gamma, int32_t *draft_len, float *reject_prob, uint32_t *flags, bool pdl,
                           cudaStream_t s)
{
    if (B == 0) return cudaSuccess;
    const int threads = 128, per = threads / LANES;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((B - 1) / per + 1)); cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, od_exit_kernel, B, K_max, head_logits, avail_len, gamma, draft_len, reject_prob, flags);
}
