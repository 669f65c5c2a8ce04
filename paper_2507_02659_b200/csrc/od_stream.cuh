// The streaming pass over a logit row, by warps: units of 512 contiguous bytes, 16 per lane, folded into
// a running (reference exponent, sum of exp2, maximum) per lane.
#pragma once

#include <float.h>

#include "od_common.cuh"
#include "od_decide.cuh"

namespace {

constexpr int U = 4;                            // 16-byte loads in flight per thread

__device__ __forceinline__ uint4 ld_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Running state of one thread inside a segment.
template <int DTYPE>
struct Lane {
    float c, s;             // reference exponent (scaled domain), sum of exp2(x*scale - c)
    float mx;               // fp32 rows: running maximum
    uint32_t pm;            // bf16 rows: packed running maxima (exact)
    __device__ __forceinline__ void reset()
    {
        c = -FLT_MAX; s = 0.f; mx = -INFINITY; pm = 0xFF80FF80u;
    }
    // make c >= gm*scale (branch-free: one rescale per group of vectors)
    __device__ __forceinline__ void raise(float gm, float scale)
    {
        const float cn = fmaxf(fmaxf(gm * scale, -FLT_MAX), c);
        s *= od_ex2(c - cn);
        c = cn;
    }
    __device__ __forceinline__ float max_seen() const
    {
        if (DTYPE == OD_BF16) return fmaxf(od_bf16_lo(pm), od_bf16_hi(pm));
        return mx;
    }
};

// absorb N 16-byte vectors held in registers
template <int DTYPE, int N>
__device__ __forceinline__ void absorb(Lane<DTYPE> &L, const uint4 *v, float scale)
{
    if (DTYPE == OD_BF16) {
        uint32_t g = L.pm;
#pragma unroll
        for (int u = 0; u < N; ++u) {
            g = bf16x2_max(g, v[u].x); g = bf16x2_max(g, v[u].y);
            g = bf16x2_max(g, v[u].z); g = bf16x2_max(g, v[u].w);
        }
        L.pm = g;
        L.raise(fmaxf(od_bf16_lo(g), od_bf16_hi(g)), scale);
    } else {
        float gm = -INFINITY;
#pragma unroll
        for (int u = 0; u < N; ++u) {
            gm = fmaxf(gm, fmaxf(fmaxf(__uint_as_float(v[u].x), __uint_as_float(v[u].y)),
                                 fmaxf(__uint_as_float(v[u].z), __uint_as_float(v[u].w))));
        }
        L.mx = fmaxf(L.mx, gm);
        L.raise(gm, scale);
    }
    const uint64_t scale2 = f2_pack(scale, scale), nc2 = f2_pack(-L.c, -L.c);
    uint64_t a0 = 0ull, a1 = 0ull;                          // two pairs of zeros
#pragma unroll
    for (int u = 0; u < N; ++u) {
        if (DTYPE == OD_BF16) {
            a0 = f2_exp_acc(a0, od_bf16_lo(v[u].x), od_bf16_hi(v[u].x), scale2, nc2);
            a1 = f2_exp_acc(a1, od_bf16_lo(v[u].y), od_bf16_hi(v[u].y), scale2, nc2);
            a0 = f2_exp_acc(a0, od_bf16_lo(v[u].z), od_bf16_hi(v[u].z), scale2, nc2);
            a1 = f2_exp_acc(a1, od_bf16_lo(v[u].w), od_bf16_hi(v[u].w), scale2, nc2);
        } else {
            a0 = f2_exp_acc(a0, __uint_as_float(v[u].x), __uint_as_float(v[u].y), scale2, nc2);
            a1 = f2_exp_acc(a1, __uint_as_float(v[u].z), __uint_as_float(v[u].w), scale2, nc2);
        }
    }
    float s0, s1;
    f2_unpack(f2_add(a0, a1), s0, s1);
    L.s += s0 + s1;
}

template <int DTYPE>
__device__ __forceinline__ void absorb_one(Lane<DTYPE> &L, float x, float scale)
{
    if (DTYPE == OD_BF16) {
        // x is a bf16 value: keep the packed maximum exact
        L.pm = bf16x2_max(L.pm, __float_as_uint(x) >> 16 | 0xFF800000u);
    } else {
        L.mx = fmaxf(L.mx, x);
    }
    L.raise(x, scale);
    L.s += od_ex2(fmaf(x, scale, -L.c));
}

// the first n (1..G, the same for the whole warp) loads of a group
template <int TW, int G>
__device__ __forceinline__ void load_group(uint4 (&x)[G], const uint4 *p, int n)
{
#pragma unroll
    for (int u = 0; u < G; ++u)
        if (u < n) x[u] = ld_stream(p + u * TW * 32);
}

template <int DTYPE>
__device__ __forceinline__ void absorb_group(Lane<DTYPE> &L, const uint4 *x, int n, float scale)
{
    static_assert(U == 4, "one case per group size");
    if (n == 4) absorb<DTYPE, 4>(L, x, scale);
    else if (n == 3) absorb<DTYPE, 3>(L, x, scale);
    else if (n == 2) absorb<DTYPE, 2>(L, x, scale);
    else absorb<DTYPE, 1>(L, x, scale);
}

template <int DTYPE>
__device__ __forceinline__ void absorb_up_to(Lane<DTYPE> &L, const uint4 (&x)[U], int n, float scale) { absorb_group<DTYPE>(L, x, n, scale); }
template <int DTYPE>
__device__ __forceinline__ void absorb_up_to(Lane<DTYPE> &L, const uint4 (&x)[2 * U], int n, float scale)
{
    if (n == 2 * U) { absorb<DTYPE, 2 * U>(L, x, scale); return; }
    if (n < U) { absorb_group<DTYPE>(L, x, n, scale); return; }
    absorb<DTYPE, U>(L, x, scale);
    if (n > U) absorb_group<DTYPE>(L, x + U, n - U, scale);
}

// A warp's run of whole units of a row, v, v + TW, ... (in front of v1f): begin() requests the first group,
// finish() folds all of them in.
// Software pipeline over groups of U units: the loads of the next group are
// issued before the current group is folded in, so a warp always has loads in
// flight while it keeps the exp pipe busy (warps of a block move in lockstep,
// they cannot hide one another's latency). The last group holds what is left
// (1..U units) and is requested like any other, one group ahead; no lane ever
// computes on padding.
template <int DTYPE, int TW, int G = U>
struct UnitRun {
    const uint4 *p;
    int cnt, na;
    uint4 xa[G];
    __device__ __forceinline__ void begin(const char *row, int v, int v1f, int lane)
    {
        p = (const uint4 *)row + (size_t)v * 32 + lane;
        cnt = v < v1f ? (v1f - v + TW - 1) / TW : 0;
        na = cnt < G ? cnt : G;
        load_group<TW>(xa, p, na);
        cnt -= na; p += G * TW * 32;
    }
    __device__ __forceinline__ void finish(Lane<DTYPE> &L, float scale)
    {
        if (na == 0) return;
        uint4 xb[G];
        for (;;) {
            if (cnt == 0) { absorb_up_to<DTYPE>(L, xa, na, scale); break; }
            const int nb = cnt < G ? cnt : G;
            load_group<TW>(xb, p, nb);
            cnt -= nb; p += G * TW * 32;
            absorb<DTYPE, G>(L, xa, scale);
            if (cnt == 0) { absorb_up_to<DTYPE>(L, xb, nb, scale); break; }
            na = cnt < G ? cnt : G;
            load_group<TW>(xa, p, na);
            cnt -= na; p += G * TW * 32;
            absorb<DTYPE, G>(L, xb, scale);
        }
    }
};

// Units of a row of v_p elements whose 32 lanes are all inside it; behind them at most one ragged unit:
// lanes past the end of the row, or a final piece under 16 bytes.
template <int DTYPE>
__device__ __forceinline__ int full_units_of(int v_p) { return v_p / (DTYPE == OD_BF16 ? 8 : 4) >> 5; }

// the ragged unit, by one warp: whole vectors, then single elements
template <int DTYPE>
__device__ __forceinline__ void absorb_ragged(Lane<DTYPE> &L, const char *row, int v_p, int lane, float scale)
{
    constexpr int VEC = DTYPE == OD_BF16 ? 8 : 4;          // elements per 16 bytes
    const int full_vecs = v_p / VEC, i = (full_vecs >> 5) * 32 + lane;
    if (i < full_vecs) {
        uint4 x[1];
        x[0] = ld_stream((const uint4 *)row + i);
        absorb<DTYPE, 1>(L, x, scale);
    }
    const int e = full_vecs * VEC + lane;
    if (e < v_p) absorb_one<DTYPE>(L, od_load_logit<DTYPE>(row, e), scale);
}

}  // namespace
