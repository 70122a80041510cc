// Cone-beam projector pair (a2, a3): Joseph-style forward projection P and its
// exact transpose P* as an atomic-free voxel-driven gather (paper Sec. 2.2,
// projection operator and its adjoint, the backprojection).
//
// Forward (k_forward): one thread per ray; the ray visits every voxel-centre plane
// of its principal axis between source and pixel and accumulates the bilinear
// sample of that plane (zero outside the grid) times the step length.
//
// Backward (k_backproject): one thread per voxel run along z. For each angle and
// each principal axis it finds the detector columns whose rays cross the voxel's
// own plane within one voxel of it (a closed-form interval), then the rows, and
// gathers step * bilinear weight * projection over exactly the (ray, plane,
// neighbour) triples the forward visits. The per-ray step is folded into the
// projection beforehand (k_weight_rays) so the gather needs no square root.
// This kernel serves the FP64 instantiation and geometries whose principal-axis
// columns do not form intervals; FP32 calls otherwise use the segment gather
// k_backproject_seg further down, which visits the same triples.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "common.cuh"
#include "geom_impl.h"
#include "tma.cuh"

namespace cbct {

// Conservative plane interval for q0 + i dq in (L, H); intersects [lo, hi].
template <typename T>
__device__ __forceinline__ void lin_range(T q0, T dq, T L, T H, T &lo, T &hi) {
    if (dq == T(0)) {
        if (!(q0 > L && q0 < H)) { lo = T(1); hi = T(0); }
        return;
    }
    T i1 = (L - q0) / dq, i2 = (H - q0) / dq;
    lo = fmax(lo, fmin(i1, i2));
    hi = fmin(hi, fmax(i1, i2));
}

// ---- forward projection -------------------------------------------------------

template <typename T>
__global__ void __launch_bounds__(256) k_forward(GeomDev g, const T *__restrict__ vol, T *__restrict__ proj,
                                                 int accumulate) {
    const int iu = blockIdx.x * 32 + threadIdx.x;
    const int iv = blockIdx.y * 8 + threadIdx.y;
    const int k = blockIdx.z % g.na, b = blockIdx.z / g.na;
    if (iu >= g.nu || iv >= g.nv) return;
    const int a = principal_axis(g.f32[k], iu);
    const ColT<T> c = col_of<T>(g, k, iu);
    const T rz = rz_of<T>(g, iv);
    T dqz, qcz;
    ray_row(g, c, rz, dqz, qcz);
    const int na = g.n[a], nb = g.n[1 - a], nz = g.n[2];
    const T ca = T(0.5) * T(na - 1);
    const long long nx = g.n[0], nxy = (long long)g.n[0] * g.n[1];
    const long long sa = a == 0 ? 1 : nx, sb = a == 0 ? nx : 1;
    const T *V = vol + (long long)b * nxy * nz;

    // planes with t in (0, 1) and the in-plane point in (-1, n): conservative range
    // in di = i - ca, the exact tests are repeated per sample
    T lo = -ca, hi = ca;
    lin_range(c.tc, c.inv, T(0), T(1), lo, hi);
    lin_range(c.qcb, c.dqb, T(-1), T(nb), lo, hi);
    lin_range(qcz, dqz, T(-1), T(nz), lo, hi);
    const int ilo = max(0, (int)floor(lo + ca) - 1), ihi = min(na - 1, (int)ceil(hi + ca) + 1);

    T acc = T(0);
    for (int i = ilo; i <= ihi; ++i) {
        const T di = T(i) - ca;
        const T t = fma_rn(di, c.inv, c.tc);
        if (!(t > T(0) && t < T(1))) continue;
        const T qb = fma_rn(di, c.dqb, c.qcb);
        const T qz = fma_rn(di, dqz, qcz);
        if (!(qb > T(-1) && qb < T(nb) && qz > T(-1) && qz < T(nz))) continue;
        const T fb0 = floor(qb), fz0 = floor(qz);
        const int jb = (int)fb0, jz = (int)fz0;
        const T fb = qb - fb0, fz = qz - fz0;
        const T *P = V + i * sa;
        const bool b0 = jb >= 0, b1 = jb + 1 < nb, z0 = jz >= 0, z1 = jz + 1 < nz;
        const long long o = (long long)jb * sb + (long long)jz * nxy;
        const T v00 = (b0 && z0) ? __ldg(P + o) : T(0);
        const T v10 = (b1 && z0) ? __ldg(P + o + sb) : T(0);
        const T v01 = (b0 && z1) ? __ldg(P + o + nxy) : T(0);
        const T v11 = (b1 && z1) ? __ldg(P + o + sb + nxy) : T(0);
        acc += (T(1) - fz) * ((T(1) - fb) * v00 + fb * v10) + fz * ((T(1) - fb) * v01 + fb * v11);
    }
    T scale;
    if constexpr (sizeof(T) == 4) scale = g.scale; else scale = g.scaled;
    acc *= ray_step<T>(g, a, c.dqb, dqz) * scale;
    T *out = proj + (((long long)b * g.na + k) * g.nv + iv) * g.nu + iu;
    *out = accumulate ? *out + acc : acc;
}

// ---- backprojection -------------------------------------------------------------

// pw = proj * step(ray) * scale (* colw[column] when colw is given)
template <typename T>
__global__ void k_weight_rays(GeomDev g, const T *__restrict__ proj, T *__restrict__ pw, const T *__restrict__ colw) {
    const int iu = blockIdx.x * 32 + threadIdx.x;
    const int iv = blockIdx.y * 8 + threadIdx.y;
    const int k = blockIdx.z % g.na, b = blockIdx.z / g.na;
    if (iu >= g.nu || iv >= g.nv) return;
    const int a = principal_axis(g.f32[k], iu);
    const ColT<T> c = col_of<T>(g, k, iu);
    T dqz, qcz;
    ray_row(g, c, rz_of<T>(g, iv), dqz, qcz);
    T scale;
    if constexpr (sizeof(T) == 4) scale = g.scale; else scale = g.scaled;
    const long long o = (((long long)b * g.na + k) * g.nv + iv) * g.nu + iu;
    const T v = proj[o] * ray_step<T>(g, a, c.dqb, dqz) * scale;
    pw[o] = colw ? v * colw[iu] : v;
}

// The same for the segment gather's padded rows (pitch a multiple of 4 floats): a thread keeps four
// neighbouring columns and walks nrows rows, so a ray costs one read, one write and its square root
// (one thread per ray, reloading its column, took 300 us for the clinical scan, three times the
// DRAM time; now 118 us). vec: proj's rows start on 16 bytes.
__global__ void __launch_bounds__(256) k_weight_rows(GeomDev g, const float *__restrict__ proj, float *__restrict__ pw,
                                                     const float *__restrict__ colw, int pitch, int vec, int nrows) {
    const int u0 = (blockIdx.x * 32 + threadIdx.x) * 4, v0 = (blockIdx.y * 8 + threadIdx.y) * nrows;
    const int k = blockIdx.z % g.na;
    if (u0 >= g.nu) return;
    const Frame32 &F = g.f32[k];
    ColT<float> c[4];
    int a[4];
    float w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int u = min(u0 + i, g.nu - 1);
        a[i] = principal_axis(F, u);
        c[i] = col_of<float>(g, k, u);
        w[i] = colw ? colw[u] : 1.f;
    }
    const long long frame = blockIdx.z;  // batch item and angle
#pragma unroll 2
    for (int r = 0; r < nrows; ++r) {
        const int v = v0 + r;
        if (v >= g.nv) break;
        const float *src = proj + (frame * g.nv + v) * g.nu + u0;
        float p[4];
        if (vec) {
            const float4 q = *reinterpret_cast<const float4 *>(src);
            p[0] = q.x; p[1] = q.y; p[2] = q.z; p[3] = q.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = u0 + i < g.nu ? src[i] : 0.f;
        }
        const float rz = rz_of<float>(g, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float dqz, qcz;
            ray_row(g, c[i], rz, dqz, qcz);
            p[i] = p[i] * ray_step<float>(g, a[i], c[i].dqb, dqz) * g.scale;
            if (colw) p[i] *= w[i];
        }
        *reinterpret_cast<float4 *>(pw + (frame * g.nv + v) * pitch + u0) = make_float4(p[0], p[1], p[2], p[3]);
    }
}

// Detector column (continuous) hit by the ray from the source through the xy
// index-space point (px, py): D0S + u EU parallel to P - S.
__device__ __forceinline__ float column_of(const Frame32 &F, float px, float py) {
    const float dx = px - F.S[0], dy = py - F.S[1];
    const float num = F.D0S[0] * dy - F.D0S[1] * dx;
    const float den = F.EU[0] * dy - F.EU[1] * dx;
    return -num / den;
}

// column_of with the approximate division: for candidate ranges that carry a margin of a
// column or more (relative error a few ulp; non-finite where column_of is)
__device__ __forceinline__ float column_of_approx(const Frame32 &F, float px, float py) {
    const float dx = px - F.S[0], dy = py - F.S[1];
    const float num = F.D0S[0] * dy - F.D0S[1] * dx;
    const float den = F.EU[0] * dy - F.EU[1] * dx;
    return -__fdividef(num, den);
}

template <typename T, int ZS>
__global__ void __launch_bounds__(256) k_backproject(GeomDev g, const T *__restrict__ pw, T *__restrict__ vol,
                                                     int accumulate) {
    const int ix = blockIdx.x * 32 + threadIdx.x;
    const int iy = blockIdx.y * 8 + threadIdx.y;
    const int nzs = (g.n[2] + ZS - 1) / ZS;
    const int z0 = (blockIdx.z % nzs) * ZS, b = blockIdx.z / nzs;
    if (ix >= g.n[0] || iy >= g.n[1]) return;
    const int nz = g.n[2];
    T acc[ZS];
#pragma unroll
    for (int j = 0; j < ZS; ++j) acc[j] = T(0);
    const T *PB = pw + (long long)b * g.na * g.nv * g.nu;
    const T Sz = sz_of<T>(g);
    // rows: q_z = Sz + t rz(v) and rz(v) = rz0 + v drz
    const float rz0 = g.rz32[0], drz = g.nv > 1 ? g.rz32[1] - g.rz32[0] : 1.0f;

    for (int k = 0; k < g.na; ++k) {
        const Frame32 &F = g.f32[k];
        const T *Pk = PB + (long long)k * g.nv * g.nu;
        for (int a = 0; a < 2; ++a) {
            const int alo = a == 0 ? F.ux_lo : F.uy_lo, ahi = a == 0 ? F.ux_hi : F.uy_hi;
            if (alo > ahi) continue;
            const int i = a == 0 ? ix : iy;   // the voxel's plane on axis a
            const int j = a == 0 ? iy : ix;   // its in-plane coordinate along b
            const T di = T(i) - T(0.5) * T(g.n[a] - 1);
            // columns whose rays meet plane i inside (j - 1, j + 1)
            float u1, u2;
            if (a == 0) { u1 = column_of(F, (float)ix, (float)(iy - 1)); u2 = column_of(F, (float)ix, (float)(iy + 1)); }
            else { u1 = column_of(F, (float)(ix - 1), (float)iy); u2 = column_of(F, (float)(ix + 1), (float)iy); }
            int ulo = alo, uhi = ahi;
            if (isfinite(u1) && isfinite(u2)) {
                const float lo_f = fmaxf(fminf(u1, u2), -1.0e6f), hi_f = fminf(fmaxf(u1, u2), 1.0e6f);
                ulo = max(ulo, (int)floorf(lo_f) - 1);
                uhi = min(uhi, (int)ceilf(hi_f) + 1);
            }
            for (int u = ulo; u <= uhi; ++u) {
                if (principal_axis(F, u) != a) continue;
                const ColT<T> c = col_of<T>(g, k, u);
                const T t = fma_rn(di, c.inv, c.tc);
                if (!(t > T(0) && t < T(1))) continue;
                const T qb = fma_rn(di, c.dqb, c.qcb);
                const T wb = T(1) - fabs(qb - T(j));
                if (!(wb > T(0))) continue;
                // rows whose sample on plane i lies within one voxel of [z0, z0+ZS-1]
                const float tf = (float)t;
                float v1 = ((float)(z0 - 1) - (float)Sz) / tf, v2 = ((float)(z0 + ZS) - (float)Sz) / tf;
                v1 = (v1 - rz0) / drz;
                v2 = (v2 - rz0) / drz;
                if (!(v1 == v1) || !(v2 == v2)) continue;
                const float vmin = fmaxf(fminf(v1, v2), -1.0e6f), vmax = fminf(fmaxf(v1, v2), 1.0e6f);
                const int vlo = max(0, (int)floorf(vmin) - 1);
                const int vhi = min(g.nv - 1, (int)ceilf(vmax) + 1);
                for (int v = vlo; v <= vhi; ++v) {
                    T dqz, qcz;
                    ray_row(g, c, rz_of<T>(g, v), dqz, qcz);
                    const T qz = fma_rn(di, dqz, qcz);
                    const T p = wb * __ldg(Pk + (long long)v * g.nu + u);
#pragma unroll
                    for (int jj = 0; jj < ZS; ++jj) {
                        const T wz = T(1) - fabs(qz - T(z0 + jj));
                        if (wz > T(0)) acc[jj] += wz * p;
                    }
                }
            }
        }
    }
    const long long nxy = (long long)g.n[0] * g.n[1];
    T *out = vol + (long long)b * nxy * nz + ((long long)z0 * g.n[1] + iy) * g.n[0] + ix;
#pragma unroll
    for (int jj = 0; jj < ZS; ++jj) {
        if (z0 + jj < nz) {
            T *o = out + (long long)jj * nxy;
            *o = accumulate ? *o + acc[jj] : acc[jj];
        }
    }
}

// Segment gather (FP32, geometries whose x- and y-principal columns form intervals).
// CTA = brick of 16 x 16 voxel columns x 8 voxels in z, 288 threads. For the rays of
// principal axis a at angle k, plane i of the brick is crossed at q_b(u) =
// fma(di, dqb(u), qcb(u)), monotone in the detector column u. The columns with
// floor(q_b) = s form segment s of the plane; their samples lie between voxels s and
// s + 1 with weights 1 - frac(q_b) and frac(q_b). Thread (segment, plane) accumulates
// SA[z] for voxel s and SB[z] for voxel s + 1 in registers over all angles of one
// principal axis; after each sweep every voxel takes the SA of its own segment, then
// (after a barrier) the SB of the segment below — a fixed order, so the result does not
// depend on scheduling.
//
// Along a column the samples of plane i have q_z affine in the row, and a row in the unit
// interval (L, L + 1] weighs L + 1 - q_z on voxel L and q_z - L on voxel L + 1: each interval
// needs only sum p and sum p row over its rows. Neighbouring planes and segments of a
// brick ask for overlapping rows of the same columns (about 60 requests per loaded value),
// so the tile of the projection that the brick sees at one angle is loaded once (TMA, the
// next tile in flight while this one is summed), turned into prefix sums (sum p,
// sum (row - h) p) down each column, and every interval is the difference of two entries:
// 10 instructions instead of a run of predicated row loads (3 to 5 rows per interval at
// these magnifications); boundaries, shares and sums of two voxels go through packed FP32
// instructions (12, one voxel at a time, with the same results: clinical 9.02 against 8.82 ms). The
// sums start at the tile's middle row h and run outwards, so
// they span at most half a tile (26 rows) of one column: FP32 rounding stays that of a
// short sum, and the measured error against 64 bits is the row-by-row kernel's (clinical
// 3.3e-7 against 3.5e-7). Bounded by instruction issue (68 % of the issue slots; the rest
// mostly the two barriers of a tile, 27 % of the stalls): about 3/4 of the instructions are the
// intervals, 1/6 the prefix sums. Back projection by CUDA events, row by row -> now:
// clinical 17.4 -> 9.56 ms, 2 x 128^3 / 200 angles 3.79 -> 1.68 ms, 64^3 / 64 angles 126 -> 54 us.
//
// A prefix sum keeps the rounding of every row on its way, so a column half that is not finite or
// spans too wide a range (kWideLog2) is summed row by row instead, over the same intervals: a large,
// infinite or NaN pixel reaches the voxels its ray touches and no others. Below the factor the
// differences round to little more than what the positions do (largest error of a voxel that pixels 10^3 times
// their background do not touch, 100 angles: 8.6e-6 of its value against 3.7e-6 without them; with prefix
// sums everywhere 8e-5 at 10^4 and 6e-3 at 10^6). Such columns lie
// at the edges of the body, where a tile's middle is inside it: 0.1 % of the column halves of a phantom's
// projections, which cost the clinical adjoint 6 %. They are read from the landing box, so the next one is sent for after them. A brick
// whose footprint exceeds the tile takes several tiles per angle: the intervals are linear in
// the rows, so a tile that holds part of an interval adds its part.
//
// Tile 112 x 52: the largest that lets three CTAs share an SM (clinical, one voxel at a time, 9.3 ms; 96 x 60 9.7,
// 120 x 48 9.8, 128 x 46 10.0, 80 x 64 11.0 with more tiles split in columns; 112 x 56 at two
// CTAs per SM 10.9; without the TMA stage, reading the rows from L2, 10.6 at three and 12.5
// at four CTAs of 56 registers).
constexpr int kB3 = 16, kZ3 = 8, kThreads3 = 288, kWarps3 = kThreads3 / 32;
constexpr int kBC = 112, kBR = 52;       // tile: detector columns x rows
constexpr int kEP = kBC + 1;            // pitch of the prefix sums (entries), odd: rows fall into different banks
constexpr int kChunk3 = 128;            // angles listed at a time
constexpr size_t kE3Bytes = (((size_t)(kBR + 1) * kEP * 8) + 127) & ~(size_t)127;
constexpr size_t kRaw3Bytes = (size_t)kBC * kBR * 4;
static_assert(kBC <= 32 * (kWarps3 / 2), "two warps per 32 columns");
static_assert(kRaw3Bytes % 128 == 0 && (size_t)kZ3 * kB3 * (kB3 + 1) * 4 <= kE3Bytes, "tile layout");
constexpr size_t kSmem3 = 128 + kRaw3Bytes + kE3Bytes;

// A column half in which a window of rows is smaller (and not zero) by more than 2^kWideLog2 than one
// nearer to the middle row, where the sums start, is summed row by row. Window: the |p| of four rows
// (the outermost: up to seven), of one row on panels with fewer than two rows per voxel, so that it is
// hardly longer than what a voxel sees, and in halves of fewer than eight rows. Clinical adjoint with 2^8 / 2^9 / 2^10 / 2^11,
// before the groups' loads were batched: projections of a phantom 10.04 / 9.95 / 9.85 / 9.73 ms, with counting
// noise 10.35 / 10.1 / 9.88 / 9.69, even data 9.3; now with 2^10 9.75, 9.79 and 9.22.
constexpr int kWideLog2 = 10;

// Columns [u0, u1] and rows [v0, v1] of one angle that reach a brick.
struct AngleSpan {
    int k, u0, u1, v0, v1;
};

__device__ __forceinline__ bool all_finite(float a, float b) { return fabsf(a) < INFINITY && fabsf(b) < INFINITY; }

// Sends for a tile's box. (Out of line: the two places it is called from cost the gather 1 % in line.)
__device__ __noinline__ void issue_box(float *raw, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *full) {
    mbar_arrive_expect_tx(full, (uint32_t)kRaw3Bytes);
    tma_load_3d(raw, map, c0, c1, c2, full);
}

template <int WIN>
__global__ void __launch_bounds__(kThreads3, 3)
    k_backproject_seg(const __grid_constant__ CUtensorMap pmap, GeomDev g, const float *__restrict__ pw, int pitch,
                      float *__restrict__ vol, int accumulate, int nparts, float *__restrict__ partial, int *status) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float *raw = reinterpret_cast<float *>(sm);
    float2 *E = reinterpret_cast<float2 *>(sm + kRaw3Bytes);
    float *vacc = reinterpret_cast<float *>(E);  // between the sweeps
    __shared__ AngleSpan list[kChunk3];
    __shared__ int wcount[kWarps3];
    __shared__ unsigned char wide[2][kBC];  // column halves to be summed row by row
    __shared__ uint64_t full;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int il = tid & 15, seg = tid >> 4;  // plane il of the brick; segment j0 - 1 + seg
    const bool item = seg <= kB3;             // 17 segments x 16 planes
    const int x0 = blockIdx.x * kB3, y0 = blockIdx.y * kB3;
    const int nzb = (g.n[2] + kZ3 - 1) / kZ3;
    const int part = blockIdx.z % nparts, zb = blockIdx.z / nparts;
    const int z0 = (zb % nzb) * kZ3, b = zb / nzb;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nv = g.nv;
    const int k_begin = (int)((long long)g.na * part / nparts);
    const int k_end = (int)((long long)g.na * (part + 1) / nparts);
    const float Sz = g.Sz;
    const float rz0 = g.rz32[0], drz = g.f32[0].EV[2], inv_drz = 1.0f / drz;
    if (tid == 0) {
        mbar_init(&full, 1);
        fence_mbar_init();
        prefetch_tmap(&pmap);
    }
    uint32_t phase = 0;
    bool ok = true;
    constexpr int kKeep = (kZ3 * kB3 * kB3 + kThreads3 - 1) / kThreads3;
    float keep[kKeep];
#pragma unroll
    for (int j = 0; j < kKeep; ++j) keep[j] = 0.f;

#pragma unroll 1
    for (int a = 0; a < 2; ++a) {
        const int i0 = a == 0 ? x0 : y0, j0 = a == 0 ? y0 : x0;
        const int i = i0 + il, s = j0 - 1 + seg;
        const bool mine = item && i < g.n[a] && s < g.n[1 - a];
        const float di = (float)i - 0.5f * (float)(g.n[a] - 1);
        float2 SA[kZ3 / 2], SB[kZ3 / 2];  // two voxels each
#pragma unroll
        for (int q = 0; q < kZ3 / 2; ++q) SA[q] = SB[q] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int kc = k_begin; kc < k_end; kc += kChunk3) {
            // list the angles of this chunk that reach the brick, in order
            __syncthreads();
            AngleSpan sp{0, 0, -1, 0, -1};
            if (tid < kChunk3 && kc + tid < k_end) {
                const Frame32 &F = g.f32[kc + tid];
                const int alo = a == 0 ? F.ux_lo : F.uy_lo, ahi = a == 0 ? F.ux_hi : F.uy_hi;
                if (alo <= ahi) {
                    // the support (planes i0 .. i0 + 15, in-plane j0 - 1 .. j0 + 16) seen from the source
                    const float den = F.EU[0] * F.D0S[1] - F.EU[1] * F.D0S[0];
                    float tmin = INFINITY, tmax = -INFINITY, umin = INFINITY, umax = -INFINITY;
                    bool fin = true;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float ci = (float)(i0 + (c & 1) * (kB3 - 1)), cj = (float)(j0 - 1 + (c >> 1) * (kB3 + 1));
                        const float px = a == 0 ? ci : cj, py = a == 0 ? cj : ci;
                        const float t = __fdividef(F.EU[0] * (py - F.S[1]) - F.EU[1] * (px - F.S[0]), den);
                        const float u = column_of_approx(F, px, py);
                        fin = fin && all_finite(t, u);
                        tmin = fminf(tmin, t);
                        tmax = fmaxf(tmax, t);
                        umin = fminf(umin, u);
                        umax = fmaxf(umax, u);
                    }
                    int ulo = alo, uhi = ahi, vlo = 0, vhi = nv - 1;
                    // a support that reaches the source's own plane has no such bounds: whole panel
                    if (fin && tmin > 1e-3f) {
                        ulo = max(alo, (int)floorf(fmaxf(umin, -1.0e6f)) - 1);
                        uhi = min(ahi, (int)ceilf(fminf(umax, 1.0e6f)) + 1);
                        const float zlo = (float)(z0 - 1) - Sz, zhi = (float)(z0 + kZ3) - Sz;
                        const float rlo = fminf(__fdividef(zlo, tmin), __fdividef(zlo, tmax));
                        const float rhi = fmaxf(__fdividef(zhi, tmin), __fdividef(zhi, tmax));
                        const float va = (rlo - rz0) * inv_drz, vb = (rhi - rz0) * inv_drz;
                        vlo = max(0, (int)floorf(fmaxf(fminf(va, vb), -1.0e6f)) - 1);
                        vhi = min(nv - 1, (int)ceilf(fminf(fmaxf(va, vb), 1.0e6f)) + 1);
                    } else if (fin && tmax <= 0.f) {
                        uhi = ulo - 1;  // behind the source
                    }
                    if (ulo <= uhi && vlo <= vhi)
                        sp = AngleSpan{kc + tid, ulo & ~3, uhi, vlo, vhi};
                }
            }
            const bool has = sp.u0 <= sp.u1 && sp.v0 <= sp.v1;
            const unsigned bal = __ballot_sync(0xffffffffu, has);
            if (lane == 0) wcount[warp] = __popc(bal);
            __syncthreads();
            int at = __popc(bal & ((1u << lane) - 1u)), nlist = 0;
            for (int w = 0; w < kWarps3; ++w) {
                if (w < warp) at += wcount[w];
                nlist += wcount[w];
            }
            if (has) list[at] = sp;
            __syncthreads();
            if (nlist == 0) continue;

            // tiles of the listed angles: (angle n, columns tu .., rows tv ..); the box of the next
            // tile is on its way while the current one is summed
            int n = 0, tu = list[0].u0, tv = list[0].v0;
            if (tid == 0) {
                mbar_arrive_expect_tx(&full, (uint32_t)kRaw3Bytes);
                tma_load_3d(raw, &pmap, tu, tv, b * g.na + list[0].k, &full);
            }
            while (n < nlist) {
                const AngleSpan cur = list[n];
                const int k = cur.k, nc = min(kBC, cur.u1 - tu + 1), nr = min(kBR, cur.v1 - tv + 1);
                const int u0 = tu, v0 = tv;
                // next tile
                tv += kBR;
                if (tv > cur.v1) {
                    tv = cur.v0;
                    tu += kBC;
                    if (tu > cur.u1) {
                        ++n;
                        if (n < nlist) {
                            tu = list[n].u0;
                            tv = list[n].v0;
                        }
                    }
                }
                ok = mbar_wait(&full, phase, status);
                if (!ok) mbar_wait(&full, phase, status);  // a copy still in flight lands before the CTA leaves
                phase ^= 1u;
                const int h = (nr - 1) >> 1;
                bool odd = false;
                if (ok) {
                    // prefix sums of each column, from the middle row h outwards: E[r][c] = sum
                    // over rows h .. r - 1 (minus rows r .. h - 1) of (p, (row - h) p). A warp takes 32
                    // columns of one half.
                    const int c = (warp >> 1) * 32 + lane;
                    if (c < nc) {
                        float s0 = 0.f, s1 = 0.f, rr;
                        // the bits of the largest window so far over 2^kWideLog2, and of the smallest one
                        // that is not zero, less 1
                        int small = 0;
                        unsigned least = 0xffffffffu;
                        auto close = [&](float w) {
                            const unsigned bits = __float_as_uint(w);
                            odd |= bits - 1u < (unsigned)small;
                            small = __viaddmax_s32((int)bits, -(kWideLog2 << 23), small);
                            least = __viaddmin_u32(bits, 0xffffffffu, least);
                        };
                        // groups of four rows: loads first (the sums' stores could alias them), then the sums;
                        // the rows left over join the last window (fewer would be small by chance)
                        auto windows = [&](int rows, auto load, auto row) {
                            float w = 0.f;
                            int r = 0;
                            if (WIN != 1 && rows < 8) {  // one window would be all there is: row by row
#pragma unroll 1
                                for (; r < rows; ++r) {
                                    const float p = load(r);
                                    row(r, p);
                                    close(fabsf(p));
                                }
                                return;
                            }
#pragma unroll 1
                            for (; r + 4 <= rows; r += 4) {
                                float p[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) p[j] = load(r + j);
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    row(r + j, p[j]);
                                    if (WIN == 1) close(fabsf(p[j]));
                                    else w = j ? w + fabsf(p[j]) : fabsf(p[j]);
                                }
                                if (WIN != 1) close(w);
                            }
#pragma unroll 1
                            for (; r < rows; ++r) {
                                const float p = load(r);
                                row(r, p);
                                if (WIN == 1) close(fabsf(p));
                                else w += fabsf(p);
                            }
                            if (WIN != 1) close(w);
                        };
                        if (warp & 1) {
                            const float *src = raw + c + (h - 1) * kBC;
                            float2 *dst = E + c + (h - 1) * kEP;
                            rr = 1.f;
                            windows(h, [&](int r) { return src[-r * kBC]; }, [&](int r, float p) {
                                s0 -= p;
                                s1 = fmaf(rr, p, s1);
                                rr += 1.f;
                                dst[-r * kEP] = make_float2(s0, s1);
                            });
                        } else {
                            const float *src = raw + c + h * kBC;
                            float2 *dst = E + c + h * kEP;
                            rr = 0.f;
                            dst[0] = make_float2(0.f, 0.f);
                            windows(nr - h, [&](int r) { return src[r * kBC]; }, [&](int r, float p) {
                                s0 += p;
                                s1 = fmaf(rr, p, s1);
                                rr += 1.f;
                                dst[(r + 1) * kEP] = make_float2(s0, s1);
                            });
                        }
                        // where the panel or the tile cuts the brick's rows, a large last window may have
                        // small rows behind its pixel that no window shows: there its order does not matter
                        const bool cut = warp & 1 ? v0 > cur.v0 || v0 == 0 : v0 + nr <= cur.v1 || v0 + nr == nv;
                        odd = odd || !all_finite(s0, s1) || (cut && least < (unsigned)small);
                        wide[warp & 1][c] = odd;
                    }
                }
                // a wait that gave up ends the sweep for every thread; columns whose sums are not
                // finite or span too wide a range are taken row by row
                const CtaVote vote = cta_vote(!ok, odd);
                if (vote.gave_up) {
                    ok = false;
                    break;
                }
                // (columns taken row by row still need this box)
                if (!vote.odd && tid == 0 && n < nlist) issue_box(raw, &pmap, tu, tv, b * g.na + list[n].k, &full);
                if (mine) {
                    const Frame32 &F = g.f32[k];
                    const float rzh = rz_of<float>(g, v0 + h), Szb = Sz - (float)(z0 - 1);
                    const int tlo = max(u0, a == 0 ? F.ux_lo : F.uy_lo);
                    const int thi = min(u0 + nc - 1, a == 0 ? F.ux_hi : F.uy_hi);
                    auto column = [&](int u, float &t, float &qb) {
                        const ColT<float> c = col_of<float>(g, k, u);
                        t = fma_rn(di, c.inv, c.tc);
                        qb = fma_rn(di, c.dqb, c.qcb);
                        return t > 0.f && t < 1.f && floorf(qb) == (float)s;
                    };
                    // columns of the segment: q_b crosses s and s + 1 at u1 and u2; the exact test
                    // settles the column nearest to each
                    float u1, u2;
                    if (a == 0) { u1 = column_of_approx(F, (float)i, (float)s); u2 = column_of_approx(F, (float)i, (float)(s + 1)); }
                    else { u1 = column_of_approx(F, (float)s, (float)i); u2 = column_of_approx(F, (float)(s + 1), (float)i); }
                    int ua = tlo, ub = thi;
                    if (all_finite(u1, u2)) {
                        ua = max(tlo, (int)rintf(fmaxf(fminf(u1, u2), -1.0e6f)));
                        ub = min(thi, (int)rintf(fminf(fmaxf(u1, u2), 1.0e6f)));
                        float t, qb;
                        if (ua <= ub && !column(ua, t, qb)) ++ua;
                        if (ua < ub && !column(ub, t, qb)) --ub;
                    }
#pragma unroll 1
                    for (int u = ua; u <= ub; ++u) {
                        float t, qb;
                        if (!column(u, t, qb)) continue;
                        const float wu = qb - floorf(qb), wl = 1.0f - wu;
                        const float step = t * drz, irs = __fdividef(1.0f, step);
                        // z of the tile's middle row relative to z0 - 1
                        const float qh = fmaf(t, rzh, Szb);
                        const float h1 = (float)(h + 1), vb = fmaf(-qh, irs, h1);
                        if (!(vote.odd && (wide[0][u - u0] | wide[1][u - u0]))) {
                            // x(m): tile row coordinate of z0 - 1 + m, plus one; the first row above
                            // is floor(x). In units of step, the rows of interval m weigh
                            // S1 = T - (x - 1 - h) S0 on the upper voxel and irs S0 - S1 on the lower.
                            const float2 irs2 = make_float2(irs, irs), vb2 = make_float2(vb, vb), h12 = make_float2(h1, h1);
                            const float2 sl2 = make_float2(wl * step, wl * step), su2 = make_float2(wu * step, wu * step);
                            const float2 *Eu = E + (u - u0);
                            auto rows = [&](float2 &e, float x) {  // sums between the last boundary and x
                                const float2 f = Eu[min(__float2uint_rd(x), (unsigned)nr) * (unsigned)kEP];
                                const float2 d = __fadd2_rn(f, make_float2(-e.x, -e.y));
                                e = f;
                                return d;
                            };
                            // boundary m's x and h + 1 - x, two at a time
                            auto ends = [&](float m, float2 &x, float2 &y) {
                                x = __ffma2_rn(make_float2(m, m + 1.f), irs2, vb2);
                                y = __fadd2_rn(h12, make_float2(-x.x, -x.y));
                            };
                            float2 x, y, e = make_float2(0.f, 0.f);
                            ends(0.f, x, y);
                            rows(e, x.x);
                            float2 d = rows(e, x.y);
                            float carry = fmaf(y.x, d.x, d.y);  // upper-voxel share of the previous interval
#pragma unroll
                            for (int q = 0; q < kZ3 / 2; ++q) {
                                // voxels z0 + 2 q and z0 + 2 q + 1: upper share of interval m - 1, lower share of m
                                float2 xn, yn;
                                ends(2.f * q + 2.f, xn, yn);
                                const float2 d1 = rows(e, xn.x), d2 = rows(e, xn.y);
                                const float s1 = fmaf(y.y, d1.x, d1.y), s2 = fmaf(yn.x, d2.x, d2.y);
                                const float2 R = __fadd2_rn(make_float2(carry, s1), make_float2(fmaf(irs, d1.x, -s1),
                                                                                                fmaf(irs, d2.x, -s2)));
                                SA[q] = __ffma2_rn(sl2, R, SA[q]);
                                SB[q] = __ffma2_rn(su2, R, SB[q]);
                                carry = s2;
                                y = yn;
                            }
                        } else {
                            // the same intervals, each over its own rows
                            const float *Pu = raw + (u - u0);
                            int r = (int)min(__float2uint_rd(vb), (unsigned)nr);
                            float carry = 0.f;  // upper-voxel share of the previous interval
#pragma unroll
                            for (int m = 0; m <= kZ3; ++m) {
                                const int end = (int)min(__float2uint_rd(fmaf((float)(m + 1), irs, vb)), (unsigned)nr);
                                float up = 0.f, low = 0.f;
#pragma unroll 1
                                for (; r < end; ++r) {
                                    const float p = Pu[r * kBC];
                                    const float f = fmaf((float)(r - h), step, qh - (float)m);
                                    if (f > 0.f) up = fmaf(f, p, up);
                                    if (f < 1.f) low = fmaf(1.f - f, p, low);
                                }
                                if (m > 0) {
                                    const float R = carry + low;
                                    float &sa = m & 1 ? SA[(m - 1) / 2].x : SA[(m - 1) / 2].y;
                                    float &sb = m & 1 ? SB[(m - 1) / 2].x : SB[(m - 1) / 2].y;
                                    sa = fmaf(wl, R, sa);
                                    sb = fmaf(wu, R, sb);
                                }
                                carry = up;
                            }
                        }
                    }
                }
                __syncthreads();
                if (vote.odd && tid == 0 && n < nlist) issue_box(raw, &pmap, tu, tv, b * g.na + list[n].k, &full);
            }
            if (!ok) break;
        }
        // onto the sum so far (a voxel per thread and step), every voxel (plane il, local index
        // seg - 1) adds its own segment's lower shares, then the upper shares of the segment
        // below it
        auto kept = [&](int j) -> float & {
            const int e = tid + j * kThreads3;
            return vacc[(e / (kB3 * kB3)) * kB3 * (kB3 + 1) + ((e / kB3) & (kB3 - 1)) * (kB3 + 1) + (e & (kB3 - 1))];
        };
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kKeep; ++j)
            if (tid + j * kThreads3 < kZ3 * kB3 * kB3) kept(j) = keep[j];
        __syncthreads();
        if (mine && seg >= 1) {
            const int vl = seg - 1;
            float *v = vacc + (a == 0 ? vl * (kB3 + 1) + il : il * (kB3 + 1) + vl);
#pragma unroll
            for (int m = 0; m < kZ3; ++m) v[m * kB3 * (kB3 + 1)] += m & 1 ? SA[m / 2].y : SA[m / 2].x;
        }
        __syncthreads();
        if (mine && seg < kB3) {
            float *v = vacc + (a == 0 ? seg * (kB3 + 1) + il : il * (kB3 + 1) + seg);
#pragma unroll
            for (int m = 0; m < kZ3; ++m) v[m * kB3 * (kB3 + 1)] += m & 1 ? SB[m / 2].y : SB[m / 2].x;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kKeep; ++j)
            if (tid + j * kThreads3 < kZ3 * kB3 * kB3) keep[j] = kept(j);
        if (!ok) break;  // outputs stay unwritten
    }
    if (!ok) return;
    const long long nxy = (long long)nx * ny;
    const int nbatch = (int)(gridDim.z / nparts / nzb);
    float *out = nparts > 1 ? partial + ((long long)part * nbatch + b) * nxy * nz : vol + (long long)b * nxy * nz;
    const int acc_mode = nparts > 1 ? 0 : accumulate;
#pragma unroll
    for (int j = 0; j < kKeep; ++j) {
        const int e = tid + j * kThreads3;
        const int xl = e & (kB3 - 1), yl = (e / kB3) & (kB3 - 1), zl = e / (kB3 * kB3);
        const int ix = x0 + xl, iy = y0 + yl, iz = z0 + zl;
        if (e < kZ3 * kB3 * kB3 && ix < nx && iy < ny && iz < nz) {
            float *o = out + ((long long)iz * ny + iy) * nx + ix;
            *o = acc_mode ? *o + keep[j] : keep[j];
        }
    }
}

// vol (+)= sum over parts of partial[part], in part order (deterministic)
__global__ void k_sum_parts(const float *__restrict__ partial, int nparts, long long n, float *__restrict__ vol,
                            int accumulate) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        float s = accumulate ? vol[e] : 0.f;
        for (int p = 0; p < nparts; ++p) s += partial[(long long)p * n + e];
        vol[e] = s;
    }
}

void sum_parts(const float *partial, int nparts, long long n, float *vol, int accumulate, cudaStream_t st) {
    const int gs = (int)std::min<long long>(8LL * sm_count(), (n + 255) / 256);
    k_sum_parts<<<gs, 256, 0, st>>>(partial, nparts, n, vol, accumulate);
}

// ---- sample count -----------------------------------------------------------------

__global__ void __launch_bounds__(256) k_count(GeomDev g, unsigned long long *total) {
    const int iu = blockIdx.x * 32 + threadIdx.x;
    const int iv = blockIdx.y * 8 + threadIdx.y;
    const int k = blockIdx.z;
    unsigned long long cnt = 0;
    if (iu < g.nu && iv < g.nv) {
        const int a = principal_axis(g.f32[k], iu);
        const ColT<float> c = col_of<float>(g, k, iu);
        float dqz, qcz;
        ray_row(g, c, rz_of<float>(g, iv), dqz, qcz);
        const int na = g.n[a], nb = g.n[1 - a], nz = g.n[2];
        const float ca = 0.5f * (float)(na - 1);
        for (int i = 0; i < na; ++i) {
            const float di = (float)i - ca;
            const float t = fma_rn(di, c.inv, c.tc);
            if (!(t > 0.0f && t < 1.0f)) continue;
            const float qb = fma_rn(di, c.dqb, c.qcb);
            const float qz = fma_rn(di, dqz, qcz);
            if (qb > -1.0f && qb < float(nb) && qz > -1.0f && qz < float(nz)) cnt++;
        }
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(total, cnt);
}

// ---- FP64 norms for the power iteration ------------------------------------------

__global__ void k_sumsq(const float *__restrict__ x, long long n, double *out) {
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double v = x[i];
        s += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, s);
}

__global__ void k_scale_by(float *x, long long n, const double *sumsq) {
    const float s = (float)(1.0 / sqrt(*sumsq));
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] *= s;
}

__global__ void k_fill(float *x, long long n, float v) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] = v;
}

// ---- launchers ------------------------------------------------------------------------

static int check_common(const cbct_geom *g, const void *a, const void *b, int batch, int accumulate) {
    if (!g || !a || !b) return fail(CBCT_EINVAL, "NULL geometry or buffer");
    if (batch < 1) return fail(CBCT_EINVAL, "batch must be >= 1");
    if (accumulate != 0 && accumulate != 1) return fail(CBCT_EINVAL, "accumulate must be 0 or 1");
    if ((long long)batch * g->dev.na > 65535) return fail(CBCT_EINVAL, "batch * n_angles must be <= 65535");
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != g->device) return fail(CBCT_EINVAL, "current device differs from the geometry's device");
    return 0;
}

template <typename T>
static int forward_impl(const cbct_geom *g, const T *vol, T *proj, int batch, int accumulate, cudaStream_t st) {
    int rc = check_common(g, vol, proj, batch, accumulate);
    if (rc) return rc;
    if constexpr (sizeof(T) == 4) {
        rc = forward_staged(g, vol, proj, batch, accumulate, st);
        if (rc < 0) return rc;
        if (rc == 1) return 0;
    }
    const GeomDev &d = g->dev;
    dim3 blk(32, 8), grd((d.nu + 31) / 32, (d.nv + 7) / 8, d.na * batch);
    k_forward<T><<<grd, blk, 0, st>>>(d, vol, proj, accumulate);
    CBCT_LAUNCH_CHECK("forward_project launch");
    return 0;
}

constexpr int kZS = 4;

// Segment gather (FP32). Scratch, one allocation: the weighted projections and the parts' volumes.
static int backward_segments(const cbct_geom *g, const float *proj, float *vol, int batch, int accumulate, cudaStream_t st,
                             const float *colw) {
    const GeomDev &d = g->dev;
    const int pitch = (d.nu + 3) & ~3;  // rows on 16 bytes, for TMA
    const int nzb = (d.n[2] + kZ3 - 1) / kZ3, bx = (d.n[0] + kB3 - 1) / kB3, by = (d.n[1] + kB3 - 1) / kB3;
    // split the angles so that about 24 CTAs per SM (8 per resident slot) are available: bricks
    // differ in how many angles see them, and the last ones must not leave SMs idle
    // (2 x 128^3: 12 / 24 / 48 per SM 1800 / 1680 / 1640 us; one 128^3 930 / 868 / 875; the
    // clinical volume has 40 per SM unsplit)
    const long long base = (long long)bx * by * nzb * batch, want = 24LL * sm_count();
    int nparts = (int)std::min<long long>(16, std::max<long long>(1, (want + base - 1) / base));
    // parts of at least 8 angles, as long as that leaves two waves of 3 CTAs per SM: a CTA's set-up
    // and its write and re-read of a partial volume cost about as much as two angles (64^3 at 4 mm:
    // 64 angles 58.5 -> 54.0 us, two volumes 107.7 -> 92.3, 32 angles 43.7 -> 36.3; 100^3, 40 angles
    // 80.1 -> 76.7; with one wave 40.7 and 16 angles 68 at 64 and 32 angles, with four no change)
    nparts = (int)std::min<long long>(nparts, std::max<long long>((d.na + 7) / 8, (6LL * sm_count() + base - 1) / base));
    nparts = std::min(nparts, d.na);
    while (nparts > 1 && (long long)nzb * batch * nparts > 65535) --nparts;
    if ((long long)nzb * batch * nparts > 65535) return cuda_fail(cudaErrorInvalidConfiguration, "back_project launch");
    const long long nvol = (long long)batch * d.n[0] * d.n[1] * d.n[2];
    const long long npw = ((long long)batch * d.na * d.nv * pitch + 63) & ~63LL;
    float *pw = nullptr;
    CBCT_CUDA_TRY(scratch_alloc((void **)&pw, sizeof(float) * (npw + (nparts > 1 ? nparts * nvol : 0)), st));
    float *partial = nparts > 1 ? pw + npw : nullptr;
    const int vec = (d.nu & 3) == 0 && (reinterpret_cast<uintptr_t>(proj) & 15) == 0;
    // 8 rows per thread, fewer when that leaves SMs without a CTA
    const long long frames = (long long)d.na * batch;
    const int nrows = (int)std::max<long long>(1, std::min<long long>(8, frames * d.nv * ((d.nu + 127) / 128) / (32LL * sm_count())));
    dim3 gw((d.nu + 127) / 128, (d.nv + 8 * nrows - 1) / (8 * nrows), (unsigned)frames);
    k_weight_rows<<<gw, dim3(32, 8), 0, st>>>(d, proj, pw, colw, pitch, vec, nrows);
    cudaError_t e = cudaGetLastError();
    CUtensorMap pmap;
    const uint64_t dims[3] = {(uint64_t)d.nu, (uint64_t)d.nv, (uint64_t)d.na * batch};
    const uint64_t str[2] = {(uint64_t)pitch * 4, (uint64_t)pitch * d.nv * 4};
    const uint32_t box[3] = {kBC, kBR, 1};
    const int rc = encode_tmap(&pmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, pw, dims, str, box);
    if (e == cudaSuccess && rc == 0) {
        // rows per voxel at the centre of rotation (f32[0].EV[2] voxels from row to row on the panel)
        const double rows = g->desc.sdd / (g->desc.sid * (double)g->h32[0].EV[2]);
        const auto kern = rows < 2.0 ? k_backproject_seg<1> : k_backproject_seg<4>;
        kern<<<dim3(bx, by, nzb * batch * nparts), kThreads3, kSmem3, st>>>(pmap, d, pw, pitch, vol, accumulate, nparts, partial,
                                                                           g->status);
        e = cudaGetLastError();
        if (e == cudaSuccess && nparts > 1) {
            sum_parts(partial, nparts, nvol, vol, accumulate, st);
            e = cudaGetLastError();
        }
    }
    cudaFreeAsync(pw, st);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "back_project launch");
    return 0;
}

template <typename T>
static int backward_impl(const cbct_geom *g, const T *proj, T *vol, int batch, int accumulate, cudaStream_t st,
                         const T *colw = nullptr) {
    int rc = check_common(g, proj, vol, batch, accumulate);
    if (rc) return rc;
    const GeomDev &d = g->dev;
    const long long nproj = (long long)batch * d.na * d.nv * d.nu;
    const int nzs = (d.n[2] + kZS - 1) / kZS;
    if ((long long)nzs * batch > 65535) return fail(CBCT_EINVAL, "back_project: batch too large");
    if constexpr (sizeof(T) == 4)
        if (g->axis_contiguous) return backward_segments(g, proj, vol, batch, accumulate, st, colw);
    T *pw = nullptr;
    CBCT_CUDA_TRY(scratch_alloc((void **)&pw, sizeof(T) * nproj, st));
    dim3 blk(32, 8), gw((d.nu + 31) / 32, (d.nv + 7) / 8, d.na * batch);
    k_weight_rays<T><<<gw, blk, 0, st>>>(d, proj, pw, colw);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        dim3 gb((d.n[0] + 31) / 32, (d.n[1] + 7) / 8, nzs * batch);
        k_backproject<T, kZS><<<gb, blk, 0, st>>>(d, pw, vol, accumulate);
        e = cudaGetLastError();
    }
    cudaFreeAsync(pw, st);
    if (e != cudaSuccess) return cuda_fail(e, "back_project launch");
    return 0;
}

// P^T (colw x proj): the adjoint of a projection scaled per detector column (the
// redundancy weight of the learned primal block), the scaling folded into the
// per-ray weighting pass.
int back_project_colw(const cbct_geom *g, const float *proj, const float *colw, float *vol, int batch, int accumulate,
                      cudaStream_t st) {
    return backward_impl<float>(g, proj, vol, batch, accumulate, st, colw);
}

int operator_norm(cbct_geom *g, int iters, double *out) {
    const GeomDev &d = g->dev;
    const long long nvox = (long long)d.n[0] * d.n[1] * d.n[2], nproj = (long long)d.na * d.nv * d.nu;
    float *x = nullptr, *p = nullptr;
    double *acc = nullptr;
    cudaError_t e = cudaMalloc(&x, sizeof(float) * nvox);
    if (e == cudaSuccess) e = cudaMalloc(&p, sizeof(float) * nproj);
    if (e == cudaSuccess) e = cudaMalloc(&acc, sizeof(double));
    double nrm2 = 0.0;
    int rc = 0;
    if (e == cudaSuccess) {
        k_fill<<<1024, 256>>>(x, nvox, 1.0f);
        for (int it = 0; it < iters && rc == 0; ++it) {
            cudaMemset(acc, 0, sizeof(double));
            k_sumsq<<<1024, 256>>>(x, nvox, acc);
            k_scale_by<<<1024, 256>>>(x, nvox, acc);
            rc = forward_impl<float>(g, x, p, 1, 0, 0);
            if (rc == 0) rc = backward_impl<float>(g, p, x, 1, 0, 0);
        }
        if (rc == 0) {
            cudaMemset(acc, 0, sizeof(double));
            k_sumsq<<<1024, 256>>>(x, nvox, acc);
            e = cudaMemcpy(&nrm2, acc, sizeof(double), cudaMemcpyDeviceToHost);
        }
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(x);
    cudaFree(p);
    cudaFree(acc);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "operator norm");
    *out = sqrt(sqrt(nrm2));  // ||P^T P x|| with ||x|| = 1 -> ||P||^2
    return 0;
}

}  // namespace cbct

using namespace cbct;

extern "C" int forward_project(const cbct_geom *g, const float *vol, float *proj, int batch, int accumulate,
                               void *stream) {
    return forward_impl<float>(g, vol, proj, batch, accumulate, (cudaStream_t)stream);
}

extern "C" int back_project(const cbct_geom *g, const float *proj, float *vol, int batch, int accumulate,
                            void *stream) {
    return backward_impl<float>(g, proj, vol, batch, accumulate, (cudaStream_t)stream);
}

extern "C" int forward_project_f64(const cbct_geom *g, const double *vol, double *proj, int batch, int accumulate,
                                   void *stream) {
    return forward_impl<double>(g, vol, proj, batch, accumulate, (cudaStream_t)stream);
}

extern "C" int back_project_f64(const cbct_geom *g, const double *proj, double *vol, int batch, int accumulate,
                                void *stream) {
    return backward_impl<double>(g, proj, vol, batch, accumulate, (cudaStream_t)stream);
}

extern "C" int cbct_count_samples(const cbct_geom *g, long long *out, void *stream) {
    if (!g || !out) return fail(CBCT_EINVAL, "cbct_count_samples: NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned long long *d = nullptr, h = 0;
    CBCT_CUDA_TRY(scratch_alloc((void **)&d, sizeof(unsigned long long), st));
    cudaMemsetAsync(d, 0, sizeof(unsigned long long), st);
    const GeomDev &v = g->dev;
    dim3 blk(32, 8), grd((v.nu + 31) / 32, (v.nv + 7) / 8, v.na);
    k_count<<<grd, blk, 0, st>>>(v, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(d, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "cbct_count_samples");
    *out = (long long)h;
    return 0;
}

// ---- backprojection without allocation --------------------------------------------
//
// back_project needs a scratch copy of the projections with the per-ray step
// length folded in, which it takes from the stream-ordered pool. Some callers
// cannot allocate device memory at call time: a host framework that owns the
// whole device memory budget through its own allocator, or a latency-critical
// loop that must not enter the CUDA allocator (which may take locks or wait on
// the device). back_project_noalloc serves them: its scratch is the fixed
// device array below, and it processes the angles in chunks that fit it.

namespace cbct {

// 8 Mi floats (32 MiB). The CUDA runtime places it on every GPU that loads this
// library, for the lifetime of the process.
constexpr long long kNoAllocScratchFloats = 8ll * 1024 * 1024;
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchFloats];

static std::mutex g_noalloc_mu;
constexpr int kMaxDevices = 256;
static float *g_noalloc_ptr[kMaxDevices] = {};

// Device address of the scratch array on `dev` (the current device). Looked up
// once per device: in host code the array's name is only a host-side stand-in.
static int noalloc_scratch(int dev, float **out) {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (dev < 0 || dev >= kMaxDevices) return fail(CBCT_EINVAL, "back_project_noalloc: device index out of range");
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "back_project_noalloc: cudaGetSymbolAddress");
        g_noalloc_ptr[dev] = static_cast<float *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return 0;
}

int projector_prime(int dev) {
    float *p = nullptr;
    for (auto kern : {k_backproject_seg<1>, k_backproject_seg<4>})
        CBCT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem3));
    const int rc = forward_prime();
    return rc ? rc : noalloc_scratch(dev, &p);
}

}  // namespace cbct

extern "C" int back_project_noalloc(const cbct_geom *g, const float *proj, float *vol, int batch, int accumulate,
                                    void *stream) {
    int rc = check_common(g, proj, vol, batch, accumulate);
    if (rc) return rc;
    const GeomDev &d = g->dev;
    const long long per_angle = (long long)d.nv * d.nu;
    if (per_angle > kNoAllocScratchFloats)
        return fail(CBCT_EINVAL, "back_project_noalloc: one projection (nu * nv = " + std::to_string(per_angle) +
                                     " floats) exceeds the fixed scratch of " +
                                     std::to_string(kNoAllocScratchFloats) + " floats");
    float *scratch = nullptr;
    rc = noalloc_scratch(g->device, &scratch);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const int chunk = (int)std::min<long long>(d.na, kNoAllocScratchFloats / per_angle);
    const int nzs = (d.n[2] + kZS - 1) / kZS;
    const long long nvox = (long long)d.n[0] * d.n[1] * d.n[2];
    dim3 blk(32, 8);
    for (int b = 0; b < batch; ++b) {
        for (int k0 = 0; k0 < d.na; k0 += chunk) {
            const int kc = std::min(chunk, d.na - k0);
            // the same kernels on the angle sub-range [k0, k0 + kc)
            GeomDev v = d;
            v.na = kc;
            v.f32 = d.f32 + k0;
            v.f64 = d.f64 + k0;
            v.col32 = d.col32 + (long long)k0 * d.nu;
            v.col64 = d.col64 + (long long)k0 * d.nu;
            const float *pb = proj + ((long long)b * d.na + k0) * per_angle;
            dim3 gw((d.nu + 31) / 32, (d.nv + 7) / 8, kc);
            k_weight_rays<float><<<gw, blk, 0, st>>>(v, pb, scratch, nullptr);
            dim3 gb((d.n[0] + 31) / 32, (d.n[1] + 7) / 8, nzs);
            k_backproject<float, kZS><<<gb, blk, 0, st>>>(v, scratch, vol + b * nvox, k0 == 0 ? accumulate : 1);
            CBCT_LAUNCH_CHECK("back_project_noalloc launch");
        }
    }
    return 0;
}
