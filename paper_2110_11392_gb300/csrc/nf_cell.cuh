// The short form of the binning's cell rule, for the device (nf_bin.cu) and, compiled
// without fused contraction, for the host, so that a CPU can compare it with the rule.
#pragma once

#include <cmath>

namespace nf {

#if defined(__CUDACC__)
#define NF_HD __host__ __device__ __forceinline__
#else
#define NF_HD inline
#endif

namespace rn {
#if defined(__CUDA_ARCH__)
NF_HD float mul(float a, float b) { return __fmul_rn(a, b); }
NF_HD float add(float a, float b) { return __fadd_rn(a, b); }
NF_HD float sub(float a, float b) { return __fsub_rn(a, b); }
NF_HD float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
NF_HD float mul(float a, float b) { return a * b; }
NF_HD float add(float a, float b) { return a + b; }
NF_HD float sub(float a, float b) { return a - b; }
NF_HD float fma(float a, float b, float c) { return fmaf(a, b, c); }
#endif
}  // namespace rn

// Cell and offset of a coordinate x > 0 for any K / box: t = x K/box as a float pair p + e,
// within err of the FP64 product (kl_hi + kl_lo is K / box to 2^-48).  False where this form
// does not decide; the integer path (nf_bin.cu) then does.
//   The product's rounding moves p by at most 2^-24 p and leaving out x kl_lo by another
// 2^-24 p, so |e| <= 2^-23 p, which can be 1.5 units in the last place of p: next to a face
// p can lie on the wrong side of it (K = 32, box = 3.7: x = 0.115625001 is in cell 1, and its
// p in cell 0).  So values within 2^-22 p of a face are left to the integer path, for which
// every other c = floor(p) is the rule's floor(t).
//   The counting form (OFF false) and the sorting form (OFF true) take a cell from here under
// this one condition, so they cannot disagree about a particle.  The sorting form also needs
// the offset's rounding decided: the sum rounded to 24 bits, taken where no value within err
// rounds otherwise (not near a rounding boundary or a cell centre).
//   A third of the integer path's instructions (see cell_coord_general).
template <bool OFF>
NF_HD bool cell_short(float x, float kl_hi, float kl_lo, int* cell, float* off)
{
    const float p = rn::mul(x, kl_hi);
    if (!(p >= 0.000244140625f && p < 1048576.0f)) return false;  // NaN, and any x when kl_hi is 0
    const float c = floorf(p), f = rn::sub(p, c);
    const float face = rn::mul(p, 2.384185791015625e-07f);  // 2^-22 p
    if (!(f >= face && rn::sub(1.0f, f) >= face)) return false;
    *cell = (int)c;
    if constexpr (OFF) {
        const float e = rn::fma(x, kl_lo, rn::fma(x, kl_hi, -p));
        const float a = rn::sub(f, 0.5f);
        // f - 1/2 - a, exact: |f| <= 1/2 wherever a is rounded
        const float tail = rn::add(rn::sub(f, rn::add(a, 0.5f)), e);
        const float o = rn::add(a, tail);
        const float r = rn::sub(tail, rn::sub(o, a));
        const float err = rn::fma(p, 1.4210854715202004e-14f, 8.8817841970012523e-16f);  // 2^-46 p + 2^-50
        *off = o;
        return fabsf(a) >= 0.000244140625f && rn::add(o, rn::add(r, err)) == o && rn::add(o, rn::sub(r, err)) == o;
    }
    return true;
}

}  // namespace nf
