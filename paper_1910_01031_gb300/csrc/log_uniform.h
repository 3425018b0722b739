// Logarithm of a uniform number u = (a + 1/2) 2^-32 to more than float
// precision, in float operations: FP64 has a 64th of their rate on this GPU.
// Every operation is IEEE (no approximations, no contraction), so host and
// device give the same bits.
#pragma once
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define IEWPF_HD __host__ __device__ __forceinline__
#else
#define IEWPF_HD inline
#endif

namespace iewpf {

// log u = hi + lo, |lo| below half an ulp or so of hi, relative error below
// 2^-28 (a double's logarithm rounded to float has 2^-25).
//
// u = m 2^e with m in [sqrt(1/2), sqrt(2)), f = m - 1 formed exactly in
// integers (so also next to u = 1) and kept as two floats; log m = 2 artanh z =
// 2 z + 2/3 z^3 + 2/5 z^5 + ..., z = f / (2 + f), |z| <= 0.172, with z as a
// quotient and its remainder's quotient (Dekker 1971) and the series, a hundredth
// of 2 z, to z^11 in float; e log 2 with log 2 split so that the first product
// is exact (Cody and Waite 1980).
IEWPF_HD void log_uniform(uint32_t a, float& hi, float& lo)
{
#ifdef __CUDA_ARCH__
    const int lz = __clz((int)a);
    const uint32_t F = __funnelshift_lc(0x80000000u, a, lz);
#else
    const int lz = a ? __builtin_clz(a) : 32;
    const uint32_t F = (uint32_t)(((((uint64_t)a << 32) | 0x80000000u) << lz) >> 32);
#endif
    // u = (F + half) 2^(-32 - lz), F >= 2^31
    const float half = lz == 0 ? 0.5f : 0.0f;
    const bool up = F >= 0xB504F334u;                 // sqrt(1/2) 2^32
    const uint32_t k = up ? ~F : F & 0x7fffffffu;     // f = -(k + 1 - half) 2^-32 or (k + half) 2^-31
    const float scale = up ? -0x1p-32f : 0x1p-31f;
    const float kh = (float)(k & ~255u), kl = (float)(k & 255u) + (up ? 1.0f - half : half);
    float fh = kh + kl, fl = (kh - fh) + kl;
    fh *= scale;
    fl *= scale;
    const float e = (float)(up ? -lz : -lz - 1);
    const float dh = 2.0f + fh, dl = ((2.0f - dh) + fh) + fl;
#ifdef __CUDA_ARCH__
    const float r = __frcp_rn(dh);
#else
    const float r = 1.0f / dh;
#endif
    const float zh = fh * r;
    const float z2 = 2.0f * ((fmaf(-zh, dh, fh) + fmaf(-zh, dl, fl)) * r);
    const float w = zh * zh;
    float p = fmaf(w, 2.0f / 11, 2.0f / 9);
    p = fmaf(w, p, 2.0f / 7);
    p = fmaf(w, p, 2.0f / 5);
    p = fmaf(w, p, 2.0f / 3);
    p = w * p;
    const float eh = e * 0x1.62e4p-1f;                // log 2 = 0x1.62e4p-1 + 0x1.7f7d1cp-20 + ...
    const float s = eh + 2.0f * zh;
    const float t = fmaf(e, 0x1.7f7d1cp-20f, fmaf(zh, p, fmaf(w, z2, z2))) + ((eh - s) + 2.0f * zh);
    hi = s + t;
    lo = (s - hi) + t;
}

}  // namespace iewpf
