// Classical reconstructions: the learned method's start and the baseline it is compared with:
//  - FDK with redundancy weighting (paper Algorithm 1 initialisation "FDK_w",
//    Sec. 2.6; Feldkamp, Davis, Kress 1984): cosine and redundancy weights, Ram-Lak
//    ramp filter along detector rows at the isocentre pitch, distance-weighted
//    voxel backprojection. An offset panel's rows are zero-padded on the short side
//    to the mirror image of the long edge before filtering.
//  - PDHG (Chambolle-Pock 2011) for 1/2 ||P x - y||^2 + lam TV(x), x >= 0, isotropic
//    TV by forward differences (the paper's TV baseline, Sec. 2.5), on K = [P; gamma grad]
//    with the TV ball radius lam / gamma.
//  - Landweber iterations x <- x - tau P^T (P x - y) (the gradient term of Algorithm 1).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "geom_impl.h"

namespace cbct {

static int grid1(long long n) {
    long long b = (n + 255) / 256;
    return (int)std::max<long long>(1, std::min<long long>(b, 32LL * sm_count()));
}

// Floats of a scratch array rounded up so that the next one starts on 256 bytes: the projector
// reads and writes whole 16-byte groups where its buffers allow it.
static long long padded(long long n) { return (n + 63) & ~63LL; }

// ---- FDK ---------------------------------------------------------------------------

// q0[b][k][v][e] = proj * w(u) * sdd / sqrt(sdd^2 + u^2 + v^2) on the extended row
// (e = iu + lo), zero in the padding.
__global__ void k_fdk_weight(const float *__restrict__ proj, const float *__restrict__ w, float *__restrict__ q0,
                             int nu, int nv, int nue, int lo, int rows, float du, float dv, float uoff,
                             float voff, float sdd) {
    const int ie = blockIdx.x * blockDim.x + threadIdx.x, iu = ie - lo;
    if (ie >= nue) return;
    const float u = ((float)iu - 0.5f * (float)(nu - 1)) * du + uoff;
    const float wu = (iu >= 0 && iu < nu) ? w[iu] * sdd : 0.f;
    for (int row = blockIdx.y; row < rows; row += gridDim.y) {
        const int iv = row % nv;
        const float v = ((float)iv - 0.5f * (float)(nv - 1)) * dv + voff;
        q0[(long long)row * nue + ie] =
            wu != 0.f ? proj[(long long)row * nu + iu] * wu * rsqrtf(sdd * sdd + u * u + v * v) : 0.f;
    }
}

// Ram-Lak filter of each extended row: q[e] = h(0) q0[e] + sum over m of the other
// parity of h(e - m) q0[m], h(d) = -1 / (pi^2 tau d^2) for odd d (zero for even d != 0).
// Per parity the sum is a Toeplitz product on the compact arrays x_j = q0[2 j + p_m]:
// out_i = sum_j g[i - j + c] x_j with g[t] = h(2 t + 1). A thread computes kRampB
// consecutive outputs of one parity and slides a window of kRampB filter taps held in
// registers along j: two shared loads per kRampB multiply-adds. The lanes of a warp read taps
// kRampB apart: one word of padding per 32 puts them into different banks (without it the loads were
// 8-way conflicts and the shared-memory pipe the limit). For short rows; long ones take the
// transform below.
constexpr int kRampB = 8;
__host__ __device__ constexpr int tap_at(int i) { return i + (i >> 5); }
__global__ void __launch_bounds__(128) k_fdk_ramp(const float *__restrict__ q0, float *__restrict__ q, int nue, int nv,
                                                  float tau) {
    extern __shared__ float sm[];
    const int half = (nue + 1) / 2;                         // compact length bound, both parities
    const int npad = (half + kRampB - 1) / kRampB * kRampB;  // compact arrays padded to a block multiple
    float *xs = sm;                                          // [2][npad]: x of parity 0, then parity 1
    float *gs = xs + 2 * npad;                               // g[t] at gs[t + goff], t = -goff .. goff + ...
    float *os = gs + tap_at(2 * npad + 2 * kRampB + 2) + 1;              // [nue] filtered row
    const int goff = npad + kRampB;
    const long long r = blockIdx.x;
    const float *src = q0 + r * nue;
    const float c1 = -1.0f / (3.14159265358979f * 3.14159265358979f * tau), h0 = 1.0f / (4.0f * tau);
    for (int i = threadIdx.x; i < 2 * npad; i += blockDim.x) {
        const int p = i >= npad, j = i - p * npad, e = 2 * j + p;
        xs[i] = e < nue ? src[e] : 0.f;
    }
    for (int k = threadIdx.x; k < 2 * npad + 2 * kRampB + 2; k += blockDim.x) {
        const float d = (float)(2 * (k - goff) + 1);
        gs[tap_at(k)] = c1 / (d * d);
    }
    __syncthreads();
    const int nb = npad / kRampB;  // output blocks per parity
    for (int wk = threadIdx.x; wk < 2 * nb; wk += blockDim.x) {
        const int pe = wk >= nb, i0 = (wk - pe * nb) * kRampB, pm = 1 - pe;
        const int c = pe - 1;  // e - m = 2 (i - j + c) + 1
        const float *x = xs + pm * npad;
        const float *xe = xs + pe * npad;
        float acc[kRampB], R[kRampB];
#pragma unroll
        for (int b = 0; b < kRampB; ++b) {
            acc[b] = h0 * xe[i0 + b];
            R[b] = gs[tap_at(goff + i0 + b + c)];  // window at j = 0: win_b = g[i0 + b + c]
        }
        for (int j = 0; j < npad; j += kRampB) {
#pragma unroll
            for (int jj = 0; jj < kRampB; ++jj) {
                const float xv = x[j + jj];
#pragma unroll
                for (int b = 0; b < kRampB; ++b) acc[b] = fmaf(R[(b - jj + kRampB) % kRampB], xv, acc[b]);
                // slide: the tap that fell off becomes g[i0 + c - (j + jj) - 1]
                R[(kRampB - 1 - jj) % kRampB] = gs[tap_at(goff + i0 + c - (j + jj) - 1)];
            }
        }
#pragma unroll
        for (int b = 0; b < kRampB; ++b) {
            const int e = 2 * (i0 + b) + pe;
            if (e < nue) os[e] = acc[b];
        }
    }
    __syncthreads();
    // output row of the zero-padded layout [na][nv + 2][nue + 2] (one zero row and column each side)
    const long long kk = r / nv, iv = r - kk * nv;
    float *dst = q + (kk * (nv + 2) + iv + 1) * (nue + 2) + 1;
    for (int e = threadIdx.x; e < nue; e += blockDim.x) dst[e] = os[e];
}

// ---- Ram-Lak by transforms ---------------------------------------------------------
//
// The filter of an extended row of nue columns is a linear convolution with lags below nue: a
// circular one of length N >= 2 nue - 1 whose kernel is h(d) on |d| < N / 2 (the lags beyond nue - 1
// meet only zeros). h is real and even, so its transform H is real, and two rows packed as real and
// imaginary part of one complex row are filtered by one transform pair.
//
// Transform: N = 512 R points, N / 8 threads with 8 points each; decimation in frequency by 8, 8, 8
// and R forward, the mirror image back, so that the frequencies stay in digit-reversed order and
// nothing is reordered (H is stored in that order). The first and last pass take their points
// from and to global memory, both middle passes meet in registers around the multiplication by
// H: six exchanges through shared memory per pair of rows. The cosine and redundancy weights are
// applied at the load, the zero border that the backprojection relies on is written with the rows.
// A row with a non-finite value stays out of the transform and is summed tap by tap; rows of unequal
// size are brought to one (exactly, by powers of two), so that a row's rounding is relative to its own
// largest value (unscaled, a partner 10^3 times larger left 2.7e-5 of the row's). Clinical scan
// (153,600 rows of 912): 1.15 ms, against 7.65 ms for weighting, clearing and the direct filter of
// k_fdk_ramp with its bank conflicts.

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a (forward: -i a, inverse: i a)
template <bool INV>
__device__ __forceinline__ float2 crot(float2 a) { return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x); }

template <bool INV>
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d) {
    const float2 s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = crot<INV>(csub(b, d));
    a = cadd(s0, s2);
    b = cadd(s1, s3);
    c = csub(s0, s2);
    d = csub(s1, s3);
}

// v[m] <- sum_n v[n] exp(-+ 2 pi i n m / 8), from the transforms of the even and the odd points
template <bool INV>
__device__ __forceinline__ void dft8(float2 v[8]) {
    dft4<INV>(v[0], v[2], v[4], v[6]);
    dft4<INV>(v[1], v[3], v[5], v[7]);
    const float r = 0.70710678f;
    const float2 o1 = INV ? make_float2(r * (v[3].x - v[3].y), r * (v[3].x + v[3].y))
                          : make_float2(r * (v[3].x + v[3].y), r * (v[3].y - v[3].x));
    const float2 o2 = crot<INV>(v[5]);
    const float2 o3 = INV ? make_float2(-r * (v[7].x + v[7].y), r * (v[7].x - v[7].y))
                          : make_float2(r * (v[7].y - v[7].x), -r * (v[7].x + v[7].y));
    const float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// transforms of R consecutive points, 8 / R of them
template <int R, bool INV>
__device__ __forceinline__ void dft_tail(float2 v[8]) {
    if constexpr (R == 8) dft8<INV>(v);
    else if constexpr (R == 4) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
        dft4<INV>(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const float2 a = v[i], b = v[i + 1];
            v[i] = cadd(a, b);
            v[i + 1] = csub(a, b);
        }
    }
}

// v[m] *= w^m (the inverse takes the conjugate)
template <bool INV>
__device__ __forceinline__ void twiddle(float2 v[8], float2 w) {
    const float2 w1 = INV ? make_float2(w.x, -w.y) : w, w2 = cmul(w1, w1), w3 = cmul(w2, w1), w4 = cmul(w2, w2);
    v[1] = cmul(v[1], w1);
    v[2] = cmul(v[2], w2);
    v[3] = cmul(v[3], w3);
    v[4] = cmul(v[4], w4);
    v[5] = cmul(v[5], cmul(w4, w1));
    v[6] = cmul(v[6], cmul(w3, w3));
    v[7] = cmul(v[7], cmul(w4, w3));
}

// one element of padding per 8: conflict-free at every stride of the passes
__host__ __device__ constexpr int fft_at(int i) { return i + (i >> 3); }

// H / N in the order of the forward transform's output: position m0 N / 8 + m1 N / 64 + m2 R + m3
// holds frequency m0 + 8 m1 + 64 m2 + 512 m3. H(f) = h(0) + 2 sum over odd d < N / 2 of h(d)
// cos(2 pi f d / N) with the taps of k_fdk_ramp (rounded to FP32 as there: their common rounding sets
// the filter's gain at f = 0, which the backprojection adds up over all angles), summed in FP64;
// 16 threads per frequency.
__global__ void __launch_bounds__(256) k_fdk_response(int n, float tau, float *__restrict__ H) {
    extern __shared__ float ct[];  // cos(2 pi m / n), m = 0 .. n / 4
    for (int m = threadIdx.x; m <= n / 4; m += 256) ct[m] = cospif(2.0f * (float)m / (float)n);
    __syncthreads();
    const float c1 = -1.0f / (3.14159265358979f * 3.14159265358979f * tau), h0 = 1.0f / (4.0f * tau);
    const int f = blockIdx.x * 16 + (threadIdx.x >> 4), l = threadIdx.x & 15;
    double s = 0.0;
    for (int d = 2 * l + 1; d < n / 2; d += 32) {
        int m = (int)((long long)f * d & (n - 1));
        if (m > n / 2) m = n - m;
        s = fma((double)(c1 / ((float)d * (float)d)), (double)(m <= n / 4 ? ct[m] : -ct[n / 2 - m]), s);
    }
    for (int o = 8; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, 16);
    if (l == 0) {
        const int R = n / 512, pos = (f & 7) * (n / 8) + ((f >> 3) & 7) * (n / 64) + ((f >> 6) & 7) * R + (f >> 9);
        H[pos] = (float)(((double)h0 + 2.0 * s) / n);
    }
}

template <int N>
__global__ void __launch_bounds__(N / 8, N <= 1024 ? 8 : N == 2048 ? 4 : 2)
    k_fdk_filter(const float *__restrict__ proj, const float *__restrict__ w, const float *__restrict__ H,
                 float *__restrict__ q, int nu, int nv, int nue, int lo, long long frames, float du, float dv, float uoff,
                 float voff, float sdd, float tau) {
    constexpr int T = N / 8, R = N / 512;
    __shared__ float2 sm[fft_at(N)];
    __shared__ uint2 rowmax[2][T / 32];  // (two: a warp may be a pair ahead of the one that still reads)
    int odd = 0;
    const int t = threadIdx.x;
    float2 tw[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int S = N >> (3 * (p + 1)), j = t % S;
        float sn, cs;
        sincospif(2.f * (float)j / (float)(8 * S), &sn, &cs);
        tw[p] = make_float2(cs, -sn);
    }
    float h[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) h[m] = H[8 * t + m];
    const int pitch = nue + 2;
    // weighted value of column e (extended) of a row
    auto weighted = [&](const float *row, int e, float v) {
        const int iu = e - lo;
        if (iu < 0 || iu >= nu) return 0.f;
        const float u = ((float)iu - 0.5f * (float)(nu - 1)) * du + uoff, wu = w[iu] * sdd;
        return wu != 0.f ? row[iu] * wu * rsqrtf(sdd * sdd + u * u + v * v) : 0.f;
    };
    const int pairs = (nv + 1) / 2;  // of one frame: rows of different frames do not share a transform
    for (long long pr = blockIdx.x; pr < frames * pairs; pr += gridDim.x) {
        const long long frame = pr / pairs;
        const int iv0 = 2 * (int)(pr - frame * pairs);
        const bool two = iv0 + 1 < nv;
        const float v0 = ((float)iv0 - 0.5f * (float)(nv - 1)) * dv + voff;
        const float v1 = ((float)(iv0 + 1) - 0.5f * (float)(nv - 1)) * dv + voff;
        const float *p0 = proj + (frame * nv + iv0) * nu;
        float2 v[8];
        unsigned a0 = 0u, a1 = 0u;  // bits of the rows' largest magnitudes (above 0x7f7fffff: not finite)
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            v[m] = make_float2(weighted(p0, t + m * T, v0), two ? weighted(p0 + nu, t + m * T, v1) : 0.f);
            a0 = max(a0, __float_as_uint(v[m].x) & 0x7fffffffu);
            a1 = max(a1, __float_as_uint(v[m].y) & 0x7fffffffu);
        }
        a0 = __reduce_max_sync(0xffffffffu, a0);
        a1 = __reduce_max_sync(0xffffffffu, a1);
        if ((t & 31) == 0) rowmax[odd][t >> 5] = make_uint2(a0, a1);
        __syncthreads();  // (also: the previous pair's last reads are done)
#pragma unroll
        for (int i = 0; i < T / 32; ++i) {
            const uint2 a = rowmax[odd][i];
            a0 = max(a0, a.x);
            a1 = max(a1, a.y);
        }
        odd ^= 1;
        // a row with a non-finite value stays out of the transform, which would spread it over both rows
        const int bad = (a0 >= 0x7f800000u ? 1 : 0) | (a1 >= 0x7f800000u ? 2 : 0);
        if (bad) {
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                if (bad & 1) v[m].x = 0.f;
                if (bad & 2) v[m].y = 0.f;
            }
        }
        // the transform rounds to the larger of the two rows: rows of different size (more than a factor
        // of 4 to 8) go through it scaled to about 1 by powers of two, and come back by back0, back1 (an
        // empty row by 0)
        unsigned back0 = a0 ? 127u : 0u, back1 = a1 ? 127u : 0u;  // exponents
        const int e0 = (int)(a0 >> 23), e1 = (int)(a1 >> 23);
        if (a0 && a1 && !bad && abs(e0 - e1) > 2) {
            back0 = (unsigned)min(max(e0, 1), 253);
            back1 = (unsigned)min(max(e1, 1), 253);
            const float s0 = __uint_as_float((254u - back0) << 23), s1 = __uint_as_float((254u - back1) << 23);
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = make_float2(v[m].x * s0, v[m].y * s1);
        }
        const unsigned backs = back0 | back1 << 8;
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const int S = N >> (3 * (p + 1)), base = (t / S) * (8 * S) + t % S;
            if (p > 0) {
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = sm[fft_at(base + m * S)];
            }
            dft8<false>(v);
            twiddle<false>(v, tw[p]);
#pragma unroll
            for (int m = 0; m < 8; ++m) sm[fft_at(base + m * S)] = v[m];
            __syncthreads();
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = sm[fft_at(8 * t + m)];
        dft_tail<R, false>(v);
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = make_float2(v[m].x * h[m], v[m].y * h[m]);
        dft_tail<R, true>(v);
#pragma unroll
        for (int m = 0; m < 8; ++m) sm[fft_at(8 * t + m)] = v[m];
        __syncthreads();
#pragma unroll
        for (int p = 2; p >= 0; --p) {
            const int S = N >> (3 * (p + 1)), base = (t / S) * (8 * S) + t % S;
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = sm[fft_at(base + m * S)];
            twiddle<true>(v, tw[p]);
            dft8<true>(v);
            if (p > 0) {
#pragma unroll
                for (int m = 0; m < 8; ++m) sm[fft_at(base + m * S)] = v[m];
                __syncthreads();
            }
        }
        // rows of the zero-bordered layout [na][nv + 2][nue + 2]; where the transform gave no finite
        // value (a row kept out of it, or an overflow) the taps are summed one by one
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (i && !two) break;
            const int iv = iv0 + i;
            float *dst = q + (frame * (nv + 2) + iv + 1) * pitch + 1;
            const float back = __uint_as_float((i ? backs >> 8 : backs & 0xffu) << 23);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int e = t + m * T;
                float f = i ? v[m].y : v[m].x;
                if (e < nue && (((bad >> i) & 1) || !(fabsf(f) < INFINITY))) {
                    const float *row = p0 + i * nu;
                    const float vv = i ? v1 : v0, c1 = -1.0f / (3.14159265358979f * 3.14159265358979f * tau);
                    f = weighted(row, e, vv) / (4.0f * tau);
                    for (int o = (e + 1) & 1; o < nue; o += 2) {
                        const float d = (float)(e - o);
                        f = fmaf(c1 / (d * d), weighted(row, o, vv), f);
                    }
                } else {
                    f *= back;
                }
                if (e < nue) dst[e] = f;
            }
            if (t == 0) dst[-1] = dst[nue] = 0.f;
            if (iv == 0)
                for (int e = t; e < pitch; e += T) dst[e - 1 - pitch] = 0.f;
            if (iv == nv - 1)
                for (int e = t; e < pitch; e += T) dst[e - 1 + pitch] = 0.f;
        }
    }
}

// vol(P) (+)= (2 pi / n_angles) sum_k (sid / U)^2 bilinear(q_k, u(P), v(P)). A thread
// owns a run of kFdkZ voxels along z: the source distance U, the magnification, the
// detector column and the weight depend only on (x, y, angle) and are computed once
// per angle; the detector row is linear in z. A warp covers 8 x 4 voxels in (x, y): neighbours
// are about four columns apart, so a 32 x 1 row would spread every load over 120 columns (half
// the L1 sectors). Bounded by instruction issue and load latency, hence the packed pairs, the early
// end of runs off the panel, and runs that lie inside it without tests (their loads overlap).
// Clinical scan: 5.57 -> 3.1 ms (tests on every voxel 3.6). 4 CTAs per SM of 64 registers: the whole
// call 4.28 ms, with 3 / 5 / 6 of them 4.49 / 4.46 / 4.61 (before the filter's row scaling, 0.05 ms).
constexpr int kFdkZ = 8;
__global__ void __launch_bounds__(256, 4) k_fdk_backproject(const float *__restrict__ q, const float2 *__restrict__ cs,
                                                         float *__restrict__ vol, int nx, int ny, int nz, int na, int nue,
                                                         int nv, int lo, int nu, float vx, float vy, float vz, float cx,
                                                         float cy, float cz, float sid, float sdd, float rdu, float rdv,
                                                         float uoff, float voff, int accumulate, int nparts) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ix = blockIdx.x * 32 + (warp & 3) * 8 + (lane & 7), iy = blockIdx.y * 8 + (warp >> 2) * 4 + (lane >> 3);
    const int nzr = (nz + kFdkZ - 1) / kFdkZ;
    const int part = blockIdx.z % nparts, zb = blockIdx.z / nparts;
    const int iz0 = (zb % nzr) * kFdkZ, b = zb / nzr;
    if (ix >= nx || iy >= ny) return;
    const int k0 = (int)((long long)na * part / nparts), k1 = (int)((long long)na * (part + 1) / nparts);
    // a part of the angles goes to its own volumes
    vol += (long long)part * (gridDim.z / nparts / nzr) * nz * ny * nx;
    const float px = (ix - 0.5f * (nx - 1)) * vx + cx;
    const float py = (iy - 0.5f * (ny - 1)) * vy + cy;
    const float pz0 = (iz0 - 0.5f * (nz - 1)) * vz + cz;
    const float hu = 0.5f * (nu - 1) + lo, hv = 0.5f * (nv - 1);
    const int pitch = nue + 2;  // zero-padded rows: every bilinear neighbour is in bounds
    const int pitch4 = pitch * 4;
    const float *qb = q + (long long)b * na * (nv + 2) * pitch;
    float acc[kFdkZ];
#pragma unroll
    for (int j = 0; j < kFdkZ; ++j) acc[j] = 0.f;
    for (int k = k0; k < k1; ++k) {
        const float2 t = __ldg(cs + k);
        const float c = t.x, s = t.y;
        const float U = sid - (px * c + py * s);
        if (!(U > 0.f)) continue;
        const float rU = __frcp_rn(U), m = sdd * rU;
        const float fu = (m * (-px * s + py * c) - uoff) * rdu + hu;
        const float u0 = floorf(fu), au = fu - u0;
        const int ju = (int)u0;
        if (ju < -1 || ju >= nue) continue;
        const float r = sid * rU, w = r * r;
        // the detector row coordinate is affine along the z-run; a run whose first and last row lie
        // off the same edge of the panel has no sample
        const float fv0 = (m * pz0 - voff) * rdv + hv, dfv = m * vz * rdv;
        const float fv7 = fmaf((float)(kFdkZ - 1), dfv, fv0);
        if (fmaxf(fv0, fv7) < -1.f || fminf(fv0, fv7) >= (float)nv) continue;
        const float *qk = qb + ((long long)k * (nv + 2) + 1) * pitch + 1 + ju, *qk1 = qk + pitch;  // (row 0, column ju)
        const float2 mone = make_float2(-1.f, -1.f), au2 = make_float2(au, au), w2 = make_float2(w, w);
        // two voxels at a time as packed FP32 pairs (each half rounds like the scalar operation)
        auto at = [&](const float *p, int row) {
            return reinterpret_cast<const float *>(reinterpret_cast<const char *>(p) + (long long)row * pitch4);
        };
        auto pairs = [&](auto all) {  // all: every voxel of the run has its sample
#pragma unroll
            for (int j = 0; j < kFdkZ; j += 2) {
                const float2 fv = __ffma2_rn(make_float2((float)j, (float)(j + 1)), make_float2(dfv, dfv), make_float2(fv0, fv0));
                const float2 v0 = make_float2(floorf(fv.x), floorf(fv.y)), av = __ffma2_rn(v0, mone, fv);
                const int jx = (int)v0.x, jy = (int)v0.y;
                const bool okx = all.value || (unsigned)(jx + 1) <= (unsigned)nv;  // in [-1, nv)
                const bool oky = all.value || (unsigned)(jy + 1) <= (unsigned)nv;
                if (!okx && !oky) continue;
                const int rx = okx ? jx : jy, ry = oky ? jy : jx;
                const float *rx0 = at(qk, rx), *rx1 = at(qk1, rx), *ry0 = at(qk, ry), *ry1 = at(qk1, ry);
                const float2 q00 = make_float2(__ldg(rx0), __ldg(ry0)), q10 = make_float2(__ldg(rx0 + 1), __ldg(ry0 + 1));
                const float2 q01 = make_float2(__ldg(rx1), __ldg(ry1)), q11 = make_float2(__ldg(rx1 + 1), __ldg(ry1 + 1));
                const float2 a0 = __ffma2_rn(au2, __ffma2_rn(q00, mone, q10), q00);
                const float2 a1 = __ffma2_rn(au2, __ffma2_rn(q01, mone, q11), q01);
                const float2 val = __ffma2_rn(av, __ffma2_rn(a0, mone, a1), a0);
                const float2 sum = __ffma2_rn(w2, val, make_float2(acc[j], acc[j + 1]));
                if (okx) acc[j] = sum.x;
                if (oky) acc[j + 1] = sum.y;
            }
        };
        if (fminf(fv0, fv7) >= -1.f && fmaxf(fv0, fv7) < (float)nv) pairs(std::true_type());
        else pairs(std::false_type());
    }
    const float sc = 6.28318530717958647f / na;
#pragma unroll
    for (int j = 0; j < kFdkZ; ++j) {
        if (iz0 + j < nz) {
            float *o = vol + (((long long)b * nz + iz0 + j) * ny + iy) * nx + ix;
            *o = accumulate ? *o + acc[j] * sc : acc[j] * sc;
        }
    }
}

// ---- PDHG-TV pieces -------------------------------------------------------------------

// z1 <- (z1 + sigma (p - y)) / (1 + sigma)
__global__ void k_pdhg_dual1(float *__restrict__ z1, const float *__restrict__ p, const float *__restrict__ y,
                             long long n, float sigma) {
    const float inv = 1.0f / (1.0f + sigma);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        z1[e] = (z1[e] + sigma * (p[e] - y[e])) * inv;
}

// z2 <- project_{|.| <= rad}(z2 + sigma gamma grad xbar), grad = forward differences
// (zero on the last index of each axis); z2 layout [3][B][nz][ny][nx]
__global__ void k_pdhg_dual2(float *__restrict__ z2, const float *__restrict__ xb, int nx, int ny, int nz, int batch,
                             float sg, float rad) {
    const long long N = (long long)batch * nx * ny * nz;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < N; e += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(e % nx), iy = (int)((e / nx) % ny), iz = (int)((e / ((long long)nx * ny)) % nz);
        const float x = xb[e];
        const float gx = ix < nx - 1 ? xb[e + 1] - x : 0.f;
        const float gy = iy < ny - 1 ? xb[e + nx] - x : 0.f;
        const float gz = iz < nz - 1 ? xb[e + (long long)nx * ny] - x : 0.f;
        const float a0 = z2[e] + sg * gx, a1 = z2[N + e] + sg * gy, a2 = z2[2 * N + e] + sg * gz;
        const float nrm = sqrtf(a0 * a0 + a1 * a1 + a2 * a2);
        const float sc = nrm > rad ? rad / nrm : 1.0f;
        z2[e] = a0 * sc;
        z2[N + e] = a1 * sc;
        z2[2 * N + e] = a2 * sc;
    }
}

// x+ = max(0, x - tau (bt - gamma div z2)); xbar = 2 x+ - x; x = x+
__global__ void k_pdhg_primal(float *__restrict__ x, float *__restrict__ xb, const float *__restrict__ bt,
                              const float *__restrict__ z2, int nx, int ny, int nz, int batch, float tau, float gamma,
                              int nonneg) {
    const long long N = (long long)batch * nx * ny * nz;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < N; e += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(e % nx), iy = (int)((e / nx) % ny), iz = (int)((e / ((long long)nx * ny)) % nz);
        const long long sxy = (long long)nx * ny;
        float dv = 0.f;
        dv += (ix < nx - 1 ? z2[e] : 0.f) - (ix > 0 ? z2[e - 1] : 0.f);
        dv += (iy < ny - 1 ? z2[N + e] : 0.f) - (iy > 0 ? z2[N + e - nx] : 0.f);
        dv += (iz < nz - 1 ? z2[2 * N + e] : 0.f) - (iz > 0 ? z2[2 * N + e - sxy] : 0.f);
        const float xo = x[e];
        float xn = xo - tau * (bt[e] - gamma * dv);
        if (nonneg && xn < 0.f) xn = 0.f;
        xb[e] = 2.f * xn - xo;
        x[e] = xn;
    }
}

// r = p - y
// r = p - y elementwise; r may alias p (in-place residual), so no restrict on those two
__global__ void k_sub(const float *p, const float *__restrict__ y, float *r, long long n) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        r[e] = p[e] - y[e];
}

// x <- x - tau g  (optionally clamped at 0)
__global__ void k_axpy_clamp(float *__restrict__ x, const float *__restrict__ gr, long long n, float tau, int nonneg) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        float v = x[e] - tau * gr[e];
        if (nonneg && v < 0.f) v = 0.f;
        x[e] = v;
    }
}

// out = P^T P x - gamma^2 div grad x  (operator of the power iteration for ||K||)
__global__ void k_tv_normal(const float *__restrict__ x, float *__restrict__ out, int nx, int ny, int nz, int batch,
                            float g2) {
    const long long N = (long long)batch * nx * ny * nz, sxy = (long long)nx * ny;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < N; e += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(e % nx), iy = (int)((e / nx) % ny), iz = (int)((e / sxy) % nz);
        const float c = x[e];
        // -div grad x = sum over axes of (x - x_prev) contributions, Neumann
        float l = 0.f;
        if (ix < nx - 1) l += c - x[e + 1];
        if (ix > 0) l += c - x[e - 1];
        if (iy < ny - 1) l += c - x[e + nx];
        if (iy > 0) l += c - x[e - nx];
        if (iz < nz - 1) l += c - x[e + sxy];
        if (iz > 0) l += c - x[e - sxy];
        out[e] += g2 * l;
    }
}

__global__ void k_sumsq_d(const float *__restrict__ x, long long n, double *out) {
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double v = x[i];
        s += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, s);
}

__global__ void k_scale_inv_sqrt(float *x, long long n, const double *sumsq) {
    const float s = (float)(1.0 / sqrt(*sumsq));
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] *= s;
}

__global__ void k_fill1(float *x, long long n, float v) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] = v;
}

}  // namespace cbct

using namespace cbct;

extern "C" int cbct_fdk_pad(const cbct_geom *g) {
    if (!g) return fail(CBCT_EINVAL, "cbct_fdk_pad: NULL geometry");
    return (int)ceil(2.0 * fabs(g->desc.u_offset) / g->desc.du - 1e-9);
}

extern "C" int cbct_fdk(const cbct_geom *g, const float *proj, float *vol, int batch, int accumulate, void *stream) {
    if (!g || !proj || !vol || batch < 1 || (accumulate != 0 && accumulate != 1))
        return fail(CBCT_EINVAL, "cbct_fdk: invalid argument");
    cudaStream_t st = (cudaStream_t)stream;
    const cbct_geom_desc &d = g->desc;
    const int npad = cbct_fdk_pad(g), nue = d.nu + npad, lo = d.u_offset > 0 ? npad : 0;
    const long long rows = (long long)batch * d.n_angles * d.nv;
    if (rows > 0x7fffffffLL) return fail(CBCT_EINVAL, "cbct_fdk: too many detector rows");
    const int ramp_pad = ((nue + 1) / 2 + kRampB - 1) / kRampB * kRampB;
    const size_t smem = sizeof(float) * (2 * (size_t)ramp_pad + tap_at(2 * ramp_pad + 2 * kRampB + 2) + 1 + nue);
    if (sizeof(float) * (4 * (size_t)ramp_pad + 2 * kRampB + 2 + nue) > 200 * 1024)
        return fail(CBCT_EINVAL, "cbct_fdk: extended detector row too long");
    // rows of more than 256 columns by transforms, except a few of them, which do not pay for the
    // response kernel (12 us). Whole call on a 16^3 volume, direct / transform: 19,200 rows of 300 329 /
    // 271 us, of 512 304 / 186, of 1000 744 / 312; 2000 rows of 1000 110 / 66; 1024 rows of 300 54 / 55
    const int nfft = nue <= 256 || nue > 2048 || rows < 1024 ? 0 : nue <= 512 ? 1024 : nue <= 1024 ? 2048 : 4096;
    // small volumes split the angles over CTAs (at least 8 angles each), towards 8 CTAs per SM: a thread's
    // angles are a serial chain of loads (whole call, 1 / up to 16 parts: 23^3 / 17 angles of a batch of 4
    // 316 / 45 us, 64^3 / 64 angles 144 / 46 us, 128^3 / 200 angles 607 / 472 us)
    const int nzr = (d.nz + kFdkZ - 1) / kFdkZ;
    const long long ctas = (long long)((d.nx + 31) / 32) * ((d.ny + 7) / 8) * nzr * batch;
    int nparts = (int)std::max<long long>(1, std::min<long long>({16, d.n_angles / 8, 8LL * sm_count() / ctas}));
    while (nparts > 1 && (long long)nzr * batch * nparts > 65535) --nparts;
    const long long nvol = (long long)batch * d.nx * d.ny * d.nz;
    // q: filtered rows, zero-bordered [batch na][nv + 2][nue + 2]; q0: weighted extended rows [rows][nue] for
    // the direct filter
    const long long nq0 = nfft ? 0 : padded(rows * nue), nq = padded((long long)batch * d.n_angles * (d.nv + 2) * (nue + 2));
    float *q0 = nullptr, *q = nullptr, *w = nullptr;
    const long long fixed = nq0 + nq + padded(d.nu) + nfft;
    cudaError_t ea = scratch_alloc((void **)&q0, sizeof(float) * (fixed + (nparts > 1 ? nparts * nvol : 0)), st);
    if (ea == cudaErrorMemoryAllocation && nparts > 1) {  // without the parts' volumes
        cudaGetLastError();
        nparts = 1;
        ea = scratch_alloc((void **)&q0, sizeof(float) * fixed, st);
    }
    CBCT_CUDA_TRY(ea);
    q = q0 + nq0;
    w = q + nq;
    float *H = w + padded(d.nu), *partial = H + nfft;
    cudaError_t e = nfft ? cudaSuccess : cudaMemsetAsync(q, 0, sizeof(float) * nq, st);
    int rc = 0;
    if (e == cudaSuccess) rc = cbct_redundancy_weight(g, w, stream);
    if (e == cudaSuccess && rc == 0) {
        const float tau = (float)(d.du * d.sid / d.sdd);
        if (nfft) {
            k_fdk_response<<<nfft / 16, 256, sizeof(float) * (nfft / 4 + 1), st>>>(nfft, tau, H);
            auto filter = nfft == 1024 ? k_fdk_filter<1024> : nfft == 2048 ? k_fdk_filter<2048> : k_fdk_filter<4096>;
            const int per_sm = nfft == 1024 ? 8 : nfft == 2048 ? 4 : 2;
            const long long frames = (long long)batch * d.n_angles;
            const int grid = (int)std::min<long long>(frames * ((d.nv + 1) / 2), (long long)per_sm * sm_count());
            filter<<<grid, nfft / 8, 0, st>>>(proj, w, H, q, d.nu, d.nv, nue, lo, frames, (float)d.du, (float)d.dv,
                                              (float)d.u_offset, (float)d.v_offset, (float)d.sdd, tau);
        } else {
            dim3 gw((nue + 127) / 128, (unsigned)std::min<long long>(rows, 65535));
            k_fdk_weight<<<gw, 128, 0, st>>>(proj, w, q0, d.nu, d.nv, nue, lo, (int)rows, (float)d.du, (float)d.dv,
                                             (float)d.u_offset, (float)d.v_offset, (float)d.sdd);
            if (smem > 48 * 1024) cudaFuncSetAttribute(k_fdk_ramp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            k_fdk_ramp<<<(unsigned)rows, 128, smem, st>>>(q0, q, nue, d.nv, tau);
        }
        dim3 grd((d.nx + 31) / 32, (d.ny + 7) / 8, nzr * batch * nparts);
        k_fdk_backproject<<<grd, 256, 0, st>>>(
            q, g->cs32, nparts > 1 ? partial : vol, d.nx, d.ny, d.nz, d.n_angles, nue, d.nv, lo, d.nu, (float)d.vox[0], (float)d.vox[1],
            (float)d.vox[2], (float)d.center[0], (float)d.center[1], (float)d.center[2], (float)d.sid, (float)d.sdd,
            (float)(1.0 / d.du), (float)(1.0 / d.dv), (float)d.u_offset, (float)d.v_offset, nparts > 1 ? 0 : accumulate,
            nparts);
        if (nparts > 1) sum_parts(partial, nparts, nvol, vol, accumulate, st);
        e = cudaGetLastError();
    }
    cudaFreeAsync(q0, st);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "cbct_fdk");
    return 0;
}

extern "C" int cbct_opnorm(const cbct_geom *g, double gamma, int iters, double *out, void *stream) {
    if (!g || !out || iters < 1) return fail(CBCT_EINVAL, "cbct_opnorm: invalid argument");
    cudaStream_t st = (cudaStream_t)stream;
    const GeomDev &d = g->dev;
    const long long nvox = (long long)d.n[0] * d.n[1] * d.n[2], nproj = (long long)d.na * d.nv * d.nu;
    float *x = nullptr, *p = nullptr, *y = nullptr;
    double *acc = nullptr;
    CBCT_CUDA_TRY(scratch_alloc((void **)&x, sizeof(float) * (2 * padded(nvox) + padded(nproj)) + 16, st));
    y = x + padded(nvox);
    p = y + padded(nvox);
    acc = reinterpret_cast<double *>(p + padded(nproj));
    int rc = 0;
    k_fill1<<<grid1(nvox), 256, 0, st>>>(x, nvox, 1.0f);
    double nrm2 = 0.0;
    for (int it = 0; it < iters && rc == 0; ++it) {
        cudaMemsetAsync(acc, 0, sizeof(double), st);
        k_sumsq_d<<<grid1(nvox), 256, 0, st>>>(x, nvox, acc);
        k_scale_inv_sqrt<<<grid1(nvox), 256, 0, st>>>(x, nvox, acc);
        rc = forward_project(g, x, p, 1, 0, stream);
        if (rc == 0) rc = back_project(g, p, y, 1, 0, stream);
        if (rc == 0 && gamma != 0.0)
            k_tv_normal<<<grid1(nvox), 256, 0, st>>>(x, y, d.n[0], d.n[1], d.n[2], 1, (float)(gamma * gamma));
        std::swap(x, y);
    }
    cudaError_t e = cudaSuccess;
    if (rc == 0) {
        cudaMemsetAsync(acc, 0, sizeof(double), st);
        k_sumsq_d<<<grid1(nvox), 256, 0, st>>>(x, nvox, acc);
        e = cudaMemcpyAsync(&nrm2, acc, sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    cudaFreeAsync(std::min(x, y), st);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "cbct_opnorm");
    *out = sqrt(sqrt(nrm2));
    return 0;
}

extern "C" int cbct_pdhg(const cbct_geom *g, const float *y, const float *x0, float *x, int batch, int niter,
                         double lam, double gamma, double sigma, double tau, int nonneg, void *stream) {
    if (!g || !y || !x0 || !x || batch < 1 || niter < 0 || !(gamma > 0) || !(sigma > 0) || !(tau > 0) || lam < 0)
        return fail(CBCT_EINVAL, "cbct_pdhg: invalid argument");
    cudaStream_t st = (cudaStream_t)stream;
    const GeomDev &d = g->dev;
    const long long N = (long long)batch * d.n[0] * d.n[1] * d.n[2], M = (long long)batch * d.na * d.nv * d.nu;
    float *buf = nullptr;
    // xbar, bt (N each), z2 (3N), z1, p (M each)
    const long long Np = padded(N), Mp = padded(M), N3 = padded(3 * N);
    CBCT_CUDA_TRY(scratch_alloc((void **)&buf, sizeof(float) * (2 * Np + N3 + 2 * Mp), st));
    float *xb = buf, *bt = xb + Np, *z2 = bt + Np, *z1 = z2 + N3, *p = z1 + Mp;
    if (x != x0) cudaMemcpyAsync(x, x0, sizeof(float) * N, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(xb, x0, sizeof(float) * N, cudaMemcpyDeviceToDevice, st);
    cudaMemsetAsync(z2, 0, sizeof(float) * (N3 + M), st);
    int rc = 0;
    const float rad = (float)(lam / gamma);
    for (int it = 0; it < niter && rc == 0; ++it) {
        rc = forward_project(g, xb, p, batch, 0, stream);
        if (rc) break;
        k_pdhg_dual1<<<grid1(M), 256, 0, st>>>(z1, p, y, M, (float)sigma);
        k_pdhg_dual2<<<grid1(N), 256, 0, st>>>(z2, xb, d.n[0], d.n[1], d.n[2], batch, (float)(sigma * gamma), rad);
        rc = back_project(g, z1, bt, batch, 0, stream);
        if (rc) break;
        k_pdhg_primal<<<grid1(N), 256, 0, st>>>(x, xb, bt, z2, d.n[0], d.n[1], d.n[2], batch, (float)tau,
                                                 (float)gamma, nonneg);
    }
    cudaError_t e = cudaGetLastError();
    cudaFreeAsync(buf, st);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "cbct_pdhg");
    return 0;
}

extern "C" int cbct_landweber(const cbct_geom *g, const float *y, float *x, int batch, int niter, double tau,
                              int nonneg, void *stream) {
    if (!g || !y || !x || batch < 1 || niter < 0) return fail(CBCT_EINVAL, "cbct_landweber: invalid argument");
    cudaStream_t st = (cudaStream_t)stream;
    const GeomDev &d = g->dev;
    const long long N = (long long)batch * d.n[0] * d.n[1] * d.n[2], M = (long long)batch * d.na * d.nv * d.nu;
    float *buf = nullptr;
    CBCT_CUDA_TRY(scratch_alloc((void **)&buf, sizeof(float) * (padded(N) + M), st));
    float *gr = buf, *r = buf + padded(N);
    int rc = 0;
    for (int it = 0; it < niter && rc == 0; ++it) {
        rc = forward_project(g, x, r, batch, 0, stream);
        if (rc) break;
        k_sub<<<grid1(M), 256, 0, st>>>(r, y, r, M);
        rc = back_project(g, r, gr, batch, 0, stream);
        if (rc) break;
        k_axpy_clamp<<<grid1(N), 256, 0, st>>>(x, gr, N, (float)tau, nonneg);
    }
    cudaError_t e = cudaGetLastError();
    cudaFreeAsync(buf, st);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "cbct_landweber");
    return 0;
}
