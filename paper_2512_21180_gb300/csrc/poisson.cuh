// Poisson counts of the data simulation: the FP64 definition (poisson_draw) and a sampler in
// FP32 that gives the same counts. The GPU has 1/64 of its FP32 rate in FP64, and one FP64 draw
// takes an exponential, a square root, a logarithm and several divisions; but a count depends on
// its mean only through comparisons and one floor. poisson_fast evaluates each of them in FP32
// with a bound on its error and gives up (-1) where the bound does not decide it — about one draw
// in 10^4 at a mean of 100 — and the caller then makes the FP64 draw. The counts are those of
// the FP64 definition in every case.
#pragma once

#include <stdint.h>

#include "common.cuh"

namespace cbct {

__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

__device__ __forceinline__ double u01(uint32_t x) { return ((double)x + 0.5) * (1.0 / 4294967296.0); }

// One Poisson(lam) draw for element e: key (seed lo, seed hi), counter
// (e lo, e hi, block, 0x50303031); block 0 word 0 for inversion (lam < 10); blocks
// 0, 1, ... two words per attempt for PTRS (lam >= 10).
__device__ __noinline__ int32_t poisson_draw(double lam, unsigned long long e, unsigned long long seed) {
    if (!(lam > 0.0)) return 0;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    uint4 ctr = make_uint4((uint32_t)e, (uint32_t)(e >> 32), 0u, 0x50303031u);
    // every step rounded as written (no FMA contraction), as in the definition
    if (lam < 10.0) {
        const uint4 r = philox(ctr, k0, k1);
        const double u = u01(r.x);
        double p = exp(-lam), F = p;
        int32_t k = 0;
        while (u > F && k < 1000) {
            k++;
            p = __dmul_rn(p, __ddiv_rn(lam, (double)k));
            F = __dadd_rn(F, p);
        }
        return k;
    }
    const double slam = sqrt(lam), loglam = log(lam);
    const double b = __dadd_rn(0.931, __dmul_rn(2.53, slam));
    const double a = __dadd_rn(-0.059, __dmul_rn(0.02483, b));
    const double inv_alpha = __dadd_rn(1.1239, __ddiv_rn(1.1328, __dsub_rn(b, 3.4)));
    const double vr = __dsub_rn(0.9277, __ddiv_rn(3.6224, __dsub_rn(b, 2.0)));
    const double twoa = __dmul_rn(2.0, a);
    for (uint32_t j = 0; j < 4096u; ++j) {
        ctr.z = j;
        const uint4 r = philox(ctr, k0, k1);
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const double U = __dsub_rn(u01(w[2 * h]), 0.5), V = u01(w[2 * h + 1]);
            const double us = __dsub_rn(0.5, fabs(U));
            const double kf = floor(__dadd_rn(__dadd_rn(__dmul_rn(__dadd_rn(__ddiv_rn(twoa, us), b), U), lam), 0.43));
            if (us >= 0.07 && V <= vr) return (int32_t)kf;
            if (kf < 0.0 || (us < 0.013 && V > us)) continue;
            const double lhs = log(__ddiv_rn(__dmul_rn(V, inv_alpha), __dadd_rn(__ddiv_rn(a, __dmul_rn(us, us)), b)));
            const double rhs = __dsub_rn(__dadd_rn(-lam, __dmul_rn(kf, loglam)), lgamma(__dadd_rn(kf, 1.0)));
            if (lhs <= rhs) return (int32_t)kf;
        }
    }
    return (int32_t)floor(lam + 0.5);
}

// A mean as hi + lo (FP32 each), off by at most err.
struct Mean32 {
    float hi, lo, err;
};

// i0 exp(-(a + alo)) with i0 = ih + il. Cody-Waite reduction a = -n ln2 - r with ln2 in two
// parts (the first 16 bits long, so that its product with n is exact), Taylor polynomial of
// exp(r) - 1 to r^8 on |r| <= 0.35, kept as 1 + tail so that the sum loses nothing. Relative
// error in units of |r|: two roundings of r (1.2e-7), one of the tail (0.7e-7) and the
// polynomial's (0.4e-7), over 1 + tail >= 0.7: at most 3.3e-7 |r| (and 1e-9 of truncation and lo).
// Means of 2^22 and more and non-finite ones come back as NaN, those below 1e-15 as 0 (either
// way the definition draws 0 from a u below 1).
__device__ __forceinline__ Mean32 mean32(float ih, float il, float a, float alo) {
    const float n = rintf(a * -1.44269504f);
    float r = fmaf(n, -0.693145751953125f, -a);  // ln2 to 16 bits; exact
    r = fmaf(n, -1.4286068e-6f, r) - alo;         // the next bits
    float t = fmaf(r, 2.4801587e-5f, 1.9841270e-4f);
    t = fmaf(t, r, 1.3888889e-3f);
    t = fmaf(t, r, 8.3333333e-3f);
    t = fmaf(t, r, 4.1666667e-2f);
    t = fmaf(t, r, 0.16666667f);
    t = fmaf(t, r, 0.5f);
    const float tail = fmaf(t * r, r, r);
    const float s = __int_as_float((127 + (int)fminf(fmaxf(n, -100.f), 100.f)) << 23);
    const float x = ih * s;
    Mean32 m;
    m.hi = fmaf(x, tail, x);
    m.lo = fmaf(x, tail, x - m.hi) + il * s * (1.f + tail);
    m.err = m.hi * fmaf(fabsf(r), 3.3e-7f, 1e-9f);
    if (!(fabsf(n) < 90.f && m.hi < 4194304.f && x > 1e-30f))
        m.hi = m.lo = m.err = n <= -90.f && a < 3e38f && ih >= 0.f && ih < 1e12f ? 0.f : NAN;
    return m;
}

// log k! for k < 16
__constant__ const float kLogFactorial[16] = {0.f, 0.f, 0.6931472f, 1.7917595f, 3.1780538f, 4.787492f, 6.579251f, 8.525161f,
                                              10.604603f, 12.801827f, 15.104413f, 17.502308f, 19.987214f, 22.552164f,
                                              25.191221f, 27.899271f};

// The count of poisson_draw(lam, e, seed) for lam = m, or -1 where FP32 does not decide it (checked
// against the FP64 definition over 1.5e9 draws at means of 1e-22 to 3e6, with the divisions off by
// up to two units in the last place: no count differs; undecided 1e-4 at means around 100, 1e-3
// at 1e5, 0.1 above 1e6).
__device__ __forceinline__ int32_t poisson_fast(Mean32 m, unsigned long long e, unsigned long long seed) {
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    uint4 ctr = make_uint4((uint32_t)e, (uint32_t)(e >> 32), 0u, 0x50303031u);
    const uint4 r0 = philox(ctr, k0, k1);
    const float lam = m.hi;
    constexpr float kTwo32 = 1.f / 4294967296.f;
    if (lam < 9.9999f) {
        // inversion: u against the running sum of k + 1 terms. Each term is off by less than (3 k + 6)
        // 2^-24 of itself and each addition by 2^-24, so up to k = 30 the sum is within 1e-5
        const float u = fmaf((float)r0.x, kTwo32, 0.5f * kTwo32);
        float p = mean32(1.f, 0.f, lam, m.lo).hi, F = p;
        int32_t k = 0;
        while (u > F + 1e-5f && k < 30) {
            k++;
            p *= __fdividef(lam, (float)k);
            F += p;
        }
        return u < F - 1e-5f ? k : -1;  // (a NaN mean decides nothing)
    }
    if (!(lam > 10.0001f)) return -1;
    const float slam = sqrtf(lam);
    const float b = fmaf(2.53f, slam, 0.931f), a = fmaf(0.02483f, b, -0.059f);
    const float vr = 0.9277f - __fdividef(3.6224f, b - 2.0f);
    // lam = li + lf, li whole
    const float li = floorf(lam), lf = (lam - li) + m.lo;
    uint4 r = r0;
    for (uint32_t j = 0;;) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t wu = h ? r.z : r.x, wv = h ? r.w : r.y;
            // us = (q + 1/2) 2^-32 and V = (wv + 1/2) 2^-32 exactly: the comparisons of us with 0.07
            // and 0.013 and of V with us are integer ones
            const bool neg = wu < 0x80000000u;
            const uint32_t q = neg ? wu : ~wu;
            const float us = fmaf((float)q, kTwo32, 0.5f * kTwo32), V = fmaf((float)wv, kTwo32, 0.5f * kTwo32);
            const bool wide = q >= 300647711u;  // us >= 0.07
            if (!wide && q < 55834575u && wv > q) continue;  // us < 0.013 and V > us
            if (wide && fabsf(V - vr) < 2e-6f) return -1;
            const bool quick = wide && V < vr;
            // k = floor((2 a / us + b) U + lam + 0.43): relative error of the first term within 1e-6
            const float c = __fdividef(2.0f * a, us) + b;
            const float t = neg ? c * (us - 0.5f) : c * (0.5f - us);
            const float y = lf + t + 0.43f, ky = floorf(y), fr = y - ky;
            const float tol = m.err + fmaf(fabsf(t), 1.2e-6f, 2e-6f);
            if (!(fr > tol && fr < 1.0f - tol)) return -1;
            const float kf = li + ky;
            if (quick) return (int32_t)kf;
            if (kf < 0.f) continue;
            // log(V inv_alpha / (a / us^2 + b)) <= k log lam - lam - log k!. With d = k - lam and Stirling's
            // series the right side is -(k log1p(d / lam) - d) - log(2 pi k) / 2 - 1 / (12 k) + ...
            // (the series' next term is below 1e-9 for k >= 16)
            const float inv_alpha = 1.1239f + __fdividef(1.1328f, b - 3.4f);
            const float lhs = logf(__fdividef(V * inv_alpha, __fdividef(a, us * us) + b));
            float rhs, err;
            if (kf >= 16.f) {
                const float d = (kf - lam) - m.lo, ik = __fdividef(1.0f, kf);
                const float g = kf * log1pf(__fdividef(d, lam)) - d;
                rhs = -g - 0.5f * logf(6.2831853f * kf) - ik * (0.083333333f - 0.0027777778f * ik * ik);
                err = fmaf(fabsf(d), 3e-6f, 2e-5f);
            } else {
                const float l = kf * logf(lam);
                rhs = (l - lam) - kLogFactorial[(int)kf];
                err = fmaf(l + lam, 1e-6f, 2e-5f);
            }
            if (!(fabsf(lhs - rhs) > err)) return -1;
            if (lhs < rhs) return (int32_t)kf;
        }
        if (++j > 8u) return -1;
        ctr.z = j;
        r = philox(ctr, k0, k1);
    }
}

}  // namespace cbct
