// The whole step on host buffers (od_step_host): what of them crosses the bus, and how.
//
// The bus is the bound (51 GB/s for device reads, whatever the grid), so what counts is how many bytes cross it.
// From page-locked buffers the device fetches the rows itself: the logit rows 0..m_b once the
// translation has found m_b, and the ONE drafter row that the draw needs once step 2 has decided where it is,
// not the K_b rows that the step might have needed. (32 sequences x up to 6 tokens, 128256 bf16 ids: 51 MB in 59
// copies of about 1 MB, which themselves run at 45 GB/s where one large copy reaches 55; fetched 41 MB: 1220 -> 826 us.)
// Buffers that the device cannot read, and those of which all is likely needed (od_host_better_copied), are copied, rows
// 0..K_b and 0..K_b-1 of every sequence.
#include "od_common.cuh"

namespace {

constexpr int FETCH_THREADS = 256, FETCH_VECS = 4;
constexpr int FETCH_BYTES = FETCH_THREADS * FETCH_VECS * 16;    // of a row, by one block

// Bytes [from, from + FETCH_BYTES) of a row of `bytes`: 16-byte loads (all requested before the first store)
// where source and destination are 16-byte aligned alike, single words for what is left at either end.
__device__ __forceinline__ void fetch_piece(char *dst, const char *src, int64_t bytes, int64_t from)
{
    const int64_t head = (16 - (int64_t)((uintptr_t)src & 15u)) & 15, vecs = bytes > head ? (bytes - head) / 16 : 0;
    const int64_t v0 = from / 16 + threadIdx.x;
    const uint4 *s = (const uint4 *)(src + head);
    uint4 *d = (uint4 *)(dst + head);
    uint4 x[FETCH_VECS];
#pragma unroll
    for (int i = 0; i < FETCH_VECS; ++i)
        if (v0 + i * FETCH_THREADS < vecs) x[i] = s[v0 + i * FETCH_THREADS];
#pragma unroll
    for (int i = 0; i < FETCH_VECS; ++i)
        if (v0 + i * FETCH_THREADS < vecs) d[v0 + i * FETCH_THREADS] = x[i];
    if (from == 0) {
        // (rows are whole 4-byte words, or whole vectors: at most 3 words at the head and 3 behind the vectors)
        const int64_t w = (int64_t)threadIdx.x * 4, tail = head + vecs * 16;
        if (w < head && w < bytes) *(uint32_t *)(dst + w) = *(const uint32_t *)(src + w);
        if (tail + w < bytes) *(uint32_t *)(dst + tail + w) = *(const uint32_t *)(src + tail + w);
    }
}

// Grid (pieces of a row, rows 0..K_max, sequences): the logit rows 0..m_b. The buffers are laid out alike.
__global__ void __launch_bounds__(FETCH_THREADS)
fetch_logits_kernel(char *dst, const char *src, int64_t row_bytes, int32_t K_max, const int32_t *m)
{
    const int b = blockIdx.z, r = blockIdx.y;
    if (r > m[b]) return;
    const size_t at = ((size_t)b * (K_max + 1) + r) * row_bytes;
    fetch_piece(dst + at, src + at, row_bytes, (int64_t)blockIdx.x * FETCH_BYTES);
}

// Grid (pieces of a row, sequences): the drafter's row at the position of the draw, if it is a residual one.
__global__ void __launch_bounds__(FETCH_THREADS)
fetch_drafter_kernel(char *dst, const char *src, int64_t row_bytes, int32_t K_max, const int32_t *m, const uint8_t *tail_kind,
                     const int32_t *n_accepted, const int32_t *span_start)
{
    const int b = blockIdx.y;
    const int mb = m[b], j = n_accepted[b];
    if (j >= mb && tail_kind[b] != OD_TAIL_UNMAPPED_STOP) return;      // the free token is drawn from p itself
    const size_t at = ((size_t)b * K_max + span_start[(size_t)b * K_max + j]) * row_bytes;
    fetch_piece(dst + at, src + at, row_bytes, (int64_t)blockIdx.x * FETCH_BYTES);
}

// Where the device finds [p, p + bytes) of page-locked host memory, or null (pageable, or not all of it one
// page-locked range, or not 16-byte aligned).
const char *device_view(const void *p, size_t bytes)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (at.type != cudaMemoryTypeHost || !at.devicePointer || ((uintptr_t)at.devicePointer & 15u)) return nullptr;
    // (the runtime does not say how far the range goes; the driver does)
    typedef int (*GetAttribute)(void *, int, unsigned long long);
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess || !fn) {
        cudaGetLastError();
        return nullptr;
    }
    constexpr int RANGE_START = 11, RANGE_SIZE = 12;        // CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, _SIZE
    unsigned long long start = 0;
    size_t size = 0;
    const unsigned long long d = (unsigned long long)(uintptr_t)at.devicePointer;
    if (((GetAttribute)fn)(&start, RANGE_START, d) != 0 || ((GetAttribute)fn)(&size, RANGE_SIZE, d) != 0) return nullptr;
    return d >= start && d - start <= size && bytes <= size - (d - start) ? (const char *)at.devicePointer : nullptr;
}

}  // namespace

// One token from every sequence, of another vocabulary and with rows no longer than the target's: all of both buffers is
// likely needed, and two large copies bring it at 55 GB/s. (128256 bf16 ids, sequences: copied, fetched us: 4: 138, 139;
// 8: 182, 189; 32: 472, 486; 128: 1595, 1675. fp32 4: 175, 178; 64: 1437, 1527. 64000 bf16 8: 147, 144; 32: 316, 326. With
// one vocabulary the accepted sequences' drafter rows are not fetched: 32000 fp32 32: 315, 274. Two tokens each: 32
// sequences of 128256 bf16 ids 690, 638, fp32 1137, 1110.)
bool od_host_better_copied(const od_ctx *c, int32_t B, int32_t K_max, const int32_t *draft_len, size_t lrow, size_t qrow)
{
    if (K_max != 1 || c->map_same_ids || qrow > lrow || (size_t)B * (2 * lrow + qrow) < (size_t)4 << 20) return false;
    for (int32_t b = 0; b < B; ++b)
        if (draft_len[b] < 1) return false;
    return true;
}

bool od_host_rows_readable(const void *logits, size_t logits_bytes, const void *q_rows, size_t q_bytes, const char **d_logits,
                           const char **d_q_rows)
{
    *d_logits = device_view(logits, logits_bytes);
    *d_q_rows = *d_logits ? device_view(q_rows, q_bytes) : nullptr;
    return *d_q_rows != nullptr;
}

cudaError_t od_launch_fetch_logits(od_ctx *c, int32_t B, int32_t K_max, const char *src, size_t row_bytes, cudaStream_t s)
{
    const unsigned pieces = (unsigned)((row_bytes + FETCH_BYTES - 1) / FETCH_BYTES);
    fetch_logits_kernel<<<dim3(pieces, (unsigned)K_max + 1, (unsigned)B), FETCH_THREADS, 0, s>>>((char *)c->s_logits, src, (int64_t)row_bytes,
                                                                                         K_max, c->s_m);
    return cudaGetLastError();
}

cudaError_t od_launch_fetch_drafter(od_ctx *c, int32_t B, int32_t K_max, const char *src, cudaStream_t s)
{
    c->translation_complete = false;                        // the draw behind this launch waits for it before it reads anything
    const int64_t row_bytes = (int64_t)c->v_q * 4;
    const unsigned pieces = (unsigned)((row_bytes + FETCH_BYTES - 1) / FETCH_BYTES);
    fetch_drafter_kernel<<<dim3(pieces, (unsigned)B), FETCH_THREADS, 0, s>>>((char *)c->s_q_rows, src, row_bytes, K_max, c->s_m, c->s_tail,
                                                                             c->s_n_acc, c->s_span_start);
    return cudaGetLastError();
}
