// Device helpers shared by the pair kernels (nf_force.cu, nf_sym.cu) and, for the
// packed arithmetic, the far field (nf_far.cu): FP32x2 arithmetic, asynchronous copies of the source stages, cell lookups.
#pragma once

#include <cuda_runtime.h>

#include "nf_internal.cuh"

namespace nf {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr float kTiny = 1e-25f;     // r^2 floor: coincident pairs stay finite (r^-3 < FLT_MAX)
constexpr float kFarSrc = 1e18f;    // padding source coordinate: adds exactly 0
constexpr float kFarSink = -1e18f;  // padding sink coordinate
constexpr float kBig = 3.0e38f;

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int wrap(int a, int K)
{
    a %= K;
    return a < 0 ? a + K : a;
}

__device__ __forceinline__ int find_box_by_cell(const BoxDev* boxes, int nboxes, int g)
{
    int lo = 0, hi = nboxes - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (boxes[mid].cell_base <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int cell_count(const int* off, int cid, int* start)
{
    int s = off[cid];
    *start = s;
    return off[cid + 1] - s;
}

__device__ __forceinline__ int cost_bucket(unsigned long long cost)
{
    if (cost == 0) return kBuckets - 1;
    int h = (int)floorf(2.0f * log2f((float)cost));
    int b = (kBuckets - 2) - h;
    return b < 0 ? 0 : (b > kBuckets - 2 ? kBuckets - 2 : b);
}

// Source cells of a unit, (b, d): the centre, then the half rings 1 .. 4
// (b > 0, or b = 0 and d > 0).  The first 1 + ((2R+1)^2 - 1)/2 entries are
// the half plane of radius R.
constexpr int kHalfMax = 41;
__constant__ signed char c_half[kHalfMax][2] = {
    {0, 0}, {0, 1}, {1, -1}, {1, 0}, {1, 1}, {0, 2}, {1, -2}, {1, 2}, {2, -2}, {2, -1}, {2, 0}, {2, 1}, {2, 2},
    {0, 3}, {1, -3}, {1, 3}, {2, -3}, {2, 3}, {3, -3}, {3, -2}, {3, -1}, {3, 0}, {3, 1}, {3, 2}, {3, 3},
    {0, 4}, {1, -4}, {1, 4}, {2, -4}, {2, 4}, {3, -4}, {3, 4}, {4, -4}, {4, -3}, {4, -2}, {4, -1}, {4, 0},
    {4, 1}, {4, 2}, {4, 3}, {4, 4}};
static_assert(NF_MAX_R <= 4, "the half-ring table covers R <= 4");

// Pipe cycles of a unit: 28 per group and step (14 packed instructions), and
// what a step costs beside them.
__device__ __forceinline__ unsigned long long sym_cost(int n_sink, int n_src, int GM)
{
    const unsigned long long tiles = (unsigned)(n_src + 31) >> 5;
    const unsigned ng = (unsigned)(n_sink + 63) >> 6, nch = (ng + GM - 1) / GM;
    return tiles * 32ull * (unsigned long long)(28u * ng + 10u * nch);
}

struct Coef {
    float c0, c1, c2;  // Eq. (spline) polynomial in cell units: c0 + r^2 (c2 + c1/r)
    float e0, e1;      // f'(r)/r inside the softening: e1 + e0/r
    float eps2;
    int dens_defer;    // top hat only in stages where some lane met r < b
};

// Packed FP32x2 arithmetic (sm_100+ `add/mul/fma.rn.f32x2`): one instruction
// works on the two halves of a 64-bit register pair.  The pair loops put two
// sources side by side in each pair, so every instruction computes two
// interactions of one sink; this halves the issue slots of the FP32 work.
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
// one half of a packed pair (the unpack names both halves; one is unused)
#pragma nv_diag_suppress 550
__device__ __forceinline__ float lo(f2 v)
{
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a;
}
__device__ __forceinline__ float hi(f2 v)
{
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return b;
}
#pragma nv_diag_default 550
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ f2 rsqrt2(f2 v) { return pk(rsqrt_approx(lo(v)), rsqrt_approx(hi(v))); }
// Smallest r^2 met so far, updated with both halves of a packed r^2: one
// three-input min (sm_100 and later) instead of two.
#ifndef NF_MIN3
#define NF_MIN3 1
#endif
__device__ __forceinline__ float track_min(float t, f2 r2)
{
#if NF_MIN3
    float m;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(t), "f"(lo(r2)), "f"(hi(r2)));
    return m;
#else
    return fminf(t, fminf(lo(r2), hi(r2)));
#endif
}
// r^-2 from the MUFU reciprocal: keeps the FMA pipe (the bottleneck) for the sums
__device__ __forceinline__ f2 rcp2(f2 v) { return pk(rcp_approx(lo(v)), rcp_approx(hi(v))); }

// Top-hat density term of one packed pair (Sec. "Force Kernel"): b^2 - r^2 where positive.
__device__ __forceinline__ f2 tophat2(f2 r2, f2 b2)
{
    const f2 t = fma2(r2, pk(-1.0f, -1.0f), b2);
    return pk(fmaxf(lo(t), 0.0f), fmaxf(hi(t), 0.0f));
}

// Error-free sum of two floats: s + e == a + b exactly (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc)
{
    unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

}  // namespace

}  // namespace nf
