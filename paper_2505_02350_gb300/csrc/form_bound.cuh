// The bound by which the fused adjoint leaves a kernel out of an item.  Plain
// C++ as well (with a float4 of the includer's), so that the host can compile
// it and hold it against 64-bit moments.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define SERBF_BOTH __host__ __device__ __forceinline__
#else
#define SERBF_BOTH inline
#endif

namespace serbf {

// Biased exponent of a float of either sign bit 0: v < 2^(e - 126).
SERBF_BOTH int biased_exponent(float v) {
#ifdef __CUDA_ARCH__
    return (int)(__float_as_uint(v) >> 23);
#else
    uint32_t b;
    memcpy(&b, &v, sizeof(b));
    return (int)(b >> 23);
#endif
}

// Bits that a positive count takes: cnt < 2^bits.
SERBF_BOTH int count_bits(int cnt) {
#ifdef __CUDA_ARCH__
    return 32 - __clz(cnt);
#else
    int n = 0;
    for (; cnt > 0; cnt >>= 1) ++n;
    return n;
#endif
}

// Lower bound of a kernel's quadratic form (log2 units) over a box with
// centre b and half diagonal hd, less ceil(log2(max(1, r2))): by the triangle
// inequality sqrt(q) falls by at most sqrt(largest eigenvalue of Q) hd on the
// way from the centre, and k2.w holds that root.  A box that may hold the
// kernel's centre (s <= 0) has the form's least value 0, and still the factor
// of r2: moments of a support wider than 1 grow by it.  The float error of q,
// here and in the pair loop, is a few units of 2^-24 of the largest eigenvalue
// times |Delta|^2, and |Delta|^2 < r2 for a support pair: eps covers both many
// times over.  Not finite in, NaN out (which culls nothing).
SERBF_BOTH float form_floor(float4 k0, float4 k1, float4 k2, float4 b, float hd) {
    const float dx = b.x - k0.x, dy = b.y - k0.y, dz = b.z - k0.z;
    const float ra = fmaf(k2.y, dz, fmaf(k2.x, dy, k1.x * dx)), rb = fmaf(k2.z, dz, k1.y * dy);
    const float q = fmaf(k1.z, dz * dz, fmaf(dy, rb, dx * ra));
    const float eps = 1.6e-5f * k2.w * k2.w * k0.w;
    const float s = fmaf(-1.0001f * k2.w, hd, sqrtf(q - eps));
    const float lg = fmaxf((float)(biased_exponent(k0.w) - 126), 0.f);
    return s > 0.f ? fmaf(s, s, -eps) - lg : (s == s ? -lg : s);
}

// Power of two above which a kernel's form makes all its moments over the
// item's cnt residual points round to zero: |moment| <= cnt max|E| 2^-q
// max(1, r2) (phi <= 2^-q, and |Delta| <= sqrt(r2) in the support) is below
// 2^-38 for q - log2(max(1, r2)) > this.  Infinite when a residual is not
// finite (emax is the largest of the residuals' absolute bits, where a NaN
// lies above everything).
SERBF_BOTH float form_limit(float emax, int cnt) {
    const int e = biased_exponent(emax);  // emax < 2^(e - 126)
    return e >= 255 ? INFINITY : (float)(38 + (e - 126) + count_bits(cnt));
}

}  // namespace serbf
