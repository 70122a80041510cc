// Forward projector with TMA-staged volume tiles (a2, paper Sec. 2.2 projection
// operator; Joseph-style ray sums as in projector.cu).
//
// Layout: a plane of constant x or y is read as rows of its in-plane coordinate b that varies
// along a detector row, so a warp's bilinear reads hit distinct shared-memory banks. Planes of
// constant y are rows of the volume itself (x fastest; a padded copy when its rows do not start
// on 16 bytes, the TMA stride); for planes of constant x the volume is first copied as
// T_x[x][z][y], rows padded to a multiple of 4 floats.
//
// CTA = one angle x a 32 (u) x 16 (v) ray tile: 4 consumer warps and one producer warp. The
// planes are processed in chunks; for each chunk the producer computes the box of voxels the
// tile's rays can touch (from the four corner rays at the chunk's end planes: the sample
// position is monotone in column, row and plane) and TMA-loads it (box BW x ZH x planes) into a
// 2-stage shared-memory ring. TMA fills voxels outside the volume with zeros, so the consumers
// sample without bounds checks. A chunk whose footprint exceeds the box, or that the source or the
// pixel cuts, falls back to bounds-checked global loads; a chunk whose box misses the volume is
// skipped (all its samples are zero). Tiles that contain rays of both principal axes (near 45
// degrees) make one pass per axis. Every mbarrier wait is bounded in time (tma.cuh).
//
// A consumer thread carries four consecutive rows of its column. They share the column's
// in-plane coordinate q_b on every plane, and their q_z lie within 3 t drz voxels (0.8 at
// the clinical isocentre), so they fall into two z-cells (a third or more where the rows are
// coarser, decided per chunk): the thread interpolates the levels L_j they share once along b,
// and a row at x cells above the lowest one is L_1 + sat(1 - x) (L_0 - L_1) + sat(x - 1) (L_2 - L_1) — six
// shared loads and about 40 instructions for four samples, against sixteen loads and 90 for
// four separate bilinear samples. Both cells end at L_1, so that a level outside a row's own cell enters it
// with an exact zero and leaves no rounding there, however large it is (started from L_0, a row two levels
// away was off by 1e-7 of L_0: 4e-4 of its own value where L_0 is 10^4 times larger). With three cells and
// more no level belongs to all of them, and each level gets its weight. The planes of a chunk are unrolled for two, for three and for
// any number of cells: a test and a loop in every plane cost 8 % (clinical 7.87 -> 7.23 ms). L_1 is summed once for the four rows. Where a result is not
// finite (a NaN or infinite voxel in a level that only some of the rows use) every ray is
// summed again from its own samples. Sums run per chunk and then over chunks, which keeps the
// rounding of a ray well below one long sum's: error against 64 bits 1.5e-7 at the clinical size
// (7.4e-7 with one running sum). Bounded by instruction issue (80 % of issue slots). Forward
// projection by CUDA events, two rays per thread -> four: clinical 14.9 -> 7.42 ms, 2 x 128^3 /
// 200 angles 2.07 -> 1.06 ms, 181 x 167 x 93 / 150 angles 2.10 -> 0.92 ms, 64^3 / 64 angles 48 -> 31 us (started
// from L_0: clinical 7.32 ms).
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "geom_impl.h"
#include "tma.cuh"

namespace cbct {

constexpr int kTU = 32, kTV = kForwardTileRows, kStages = 2;
constexpr int kRows = 4;  // consecutive rows per thread
constexpr int kConsumerWarps = kTV / kRows;
constexpr int kThreads = 32 * (kConsumerWarps + 1);

// CTAs per SM that the two stages of a box leave room for (at most six: more would cap the
// registers below the 64 the kernel needs)
constexpr int forward_ctas(int bw, int zh, int np) {
    const int n = 220 * 1024 / (kStages * np * zh * bw * 4 + 2048);
    return n > 6 ? 6 : n;
}

// The volume seen plane by plane along one axis: element (item, plane i, z, b) at base + item
// item + plane i + row z + b.
struct PlaneView {
    const float *base;
    long long item, plane, row;
};

struct ChunkInfo {
    int b0, z0, flag;  // flag: 0 skip (box outside the volume), 1 TMA box, 2 global fallback
    int cells;         // z-cells that a thread's rows can span on a plane of the chunk
};

// ---- tensor maps -------------------------------------------------------------------

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

int encode_tmap(CUtensorMap *map, CUtensorMapDataType dt, int rank, const void *base, const uint64_t *dims,
                const uint64_t *strides, const uint32_t *box) {
    auto fn = encode_fn();
    if (!fn) return fail(CBCT_ECUDA, "cuTensorMapEncodeTiled unavailable");
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, dt, (cuuint32_t)rank, const_cast<void *>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(CBCT_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return 0;
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

// ---- plane-major copies ----------------------------------------------------------------

// (both: slices z of all items go round the grid, whose z and y extents end at 65535)
// T_y[b][y][z][x] = V[b][z][y][x]   (row pitch py >= nx)
__global__ void k_planes_y(const float *__restrict__ V, float *__restrict__ T, int nx, int ny, int nz, long long slices,
                           int py) {
    const int y = blockIdx.x;
    for (long long s = blockIdx.y; s < slices; s += gridDim.y) {
        const long long b = s / nz, z = s - b * nz;
        const float *src = V + (s * ny + y) * nx;
        float *dst = T + ((b * ny + y) * nz + z) * py;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) dst[x] = src[x];
    }
}

// T_x[b][x][z][y] = V[b][z][y][x]   (row pitch px >= ny), 32x32 tiles through smem
__global__ void k_planes_x(const float *__restrict__ V, float *__restrict__ T, int nx, int ny, int nz, long long slices,
                           int px) {
    __shared__ float tile[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (long long s = blockIdx.z; s < slices; s += gridDim.z) {
        const long long b = s / nz, z = s - b * nz;
        const float *src = V + s * ny * (long long)nx;
        for (int j = threadIdx.y; j < 32; j += blockDim.y) {
            const int y = y0 + j, x = x0 + threadIdx.x;
            tile[j][threadIdx.x] = (y < ny && x < nx) ? src[(long long)y * nx + x] : 0.0f;
        }
        __syncthreads();
        for (int j = threadIdx.y; j < 32; j += blockDim.y) {
            const int x = x0 + j, y = y0 + threadIdx.x;
            if (x < nx && y < ny) T[((b * nx + x) * nz + z) * px + y] = tile[threadIdx.x][j];
        }
        __syncthreads();
    }
}

// ---- the staged forward kernel -----------------------------------------------------------

__device__ __forceinline__ int floor_i(float v) { return (int)floorf(fminf(fmaxf(v, -1.0e8f), 1.0e8f)); }

// Sum of the bilinear samples of one ray on planes [i0, i1) by bounds-checked loads from one
// item T of a plane view.
__device__ __noinline__ float direct_samples(const float *__restrict__ T, long long plane, long long pitch, int nb, int nz,
                                             float ca, float tc, float inv, float qcb, float dqb, float qcz, float dqz,
                                             int i0, int i1) {
    float acc = 0.f;
    for (int i = i0; i < i1; ++i) {
        const float di = (float)i - ca;
        const float t = fma_rn(di, inv, tc);
        if (!(t > 0.f && t < 1.f)) continue;
        const float qb = fma_rn(di, dqb, qcb), qz = fma_rn(di, dqz, qcz);
        if (!(qb > -1.f && qb < (float)nb && qz > -1.f && qz < (float)nz)) continue;
        const float fb0 = floorf(qb), fb = qb - fb0, fz0 = floorf(qz), fz = qz - fz0;
        const int jb = (int)fb0, jz = (int)fz0;
        const bool b0 = jb >= 0, b1 = jb + 1 < nb, z0 = jz >= 0, z1 = jz + 1 < nz;
        const float *P = T + i * plane + jz * pitch + jb;
        const float v00 = (b0 && z0) ? __ldg(P) : 0.f, v10 = (b1 && z0) ? __ldg(P + 1) : 0.f;
        const float v01 = (b0 && z1) ? __ldg(P + pitch) : 0.f, v11 = (b1 && z1) ? __ldg(P + pitch + 1) : 0.f;
        const float a0 = fmaf(fb, v10 - v00, v00), a1 = fmaf(fb, v11 - v01, v01);
        acc += fmaf(fz, a1 - a0, a0);
    }
    return acc;
}

template <int BW, int ZH, int kP>
__global__ void __launch_bounds__(kThreads, forward_ctas(BW, ZH, kP))
    k_forward_tma(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_y, GeomDev g,
                  PlaneView vx, PlaneView vy, float *__restrict__ proj, int accumulate, int *status) {
    constexpr int SE = kP * ZH * BW;  // floats per stage
    constexpr uint32_t kBytes = SE * 4;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // TMA destinations: 128-byte aligned (the launch reserves 128 bytes of slack)
    float *stages = reinterpret_cast<float *>(smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u));
    uint64_t *full = reinterpret_cast<uint64_t *>(stages + kStages * SE);
    uint64_t *empty = full + kStages;
    ChunkInfo *info = reinterpret_cast<ChunkInfo *>(empty + kStages);
    int &abort_flag = *reinterpret_cast<int *>(info + (max(g.n[0], g.n[1]) + kP - 1) / kP);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = blockIdx.z % g.na, b = blockIdx.z / g.na;
    const int u0 = blockIdx.x * kTU, v0 = blockIdx.y * kTV;
    const Frame32 &F = g.f32[k];

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], kConsumerWarps);
        }
        abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&map_x);
        prefetch_tmap(&map_y);
    }
    __syncthreads();

    // consumer ray set-up (the canonical per-ray quantities of common.cuh): column terms once,
    // row terms for the thread's rows (a row past the panel repeats the last row and is dropped
    // at the store)
    const bool consumer = warp < kConsumerWarps;
    const int iu = u0 + lane, iv0 = v0 + kRows * warp;
    const bool col_ok = consumer && iu < g.nu;
    const int my_a = col_ok ? principal_axis(F, iu) : -1;
    ColT<float> c{0.f, 0.f, 0.f, 0.f};
    float2 dqz[2], qcz[2];
    dqz[0] = dqz[1] = qcz[0] = qcz[1] = make_float2(0.f, 0.f);
    if (col_ok) {
        c = col_of<float>(g, k, iu);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            ray_row(g, c, rz_of<float>(g, min(iv0 + 2 * j, g.nv - 1)), dqz[j].x, qcz[j].x);
            ray_row(g, c, rz_of<float>(g, min(iv0 + 2 * j + 1, g.nv - 1)), dqz[j].y, qcz[j].y);
        }
    }
    float2 acc[2];
    acc[0] = acc[1] = make_float2(0.f, 0.f);
    int gc = 0;  // chunks issued so far (both passes): stage = gc % kStages, use = gc / kStages

    for (int a = 0; a < 2; ++a) {
        const int lo = a == 0 ? F.ux_lo : F.uy_lo, hi = a == 0 ? F.ux_hi : F.uy_hi;
        const int ua = max(u0, lo), ub = min(min(u0 + kTU, g.nu) - 1, hi);
        if (ua > ub) continue;  // block-uniform
        const int na = g.n[a], nb = g.n[1 - a], nz = g.n[2];
        const int nch = (na + kP - 1) / kP;
        const float ca = 0.5f * (float)(na - 1);

        if (warp == kConsumerWarps) {
            // chunk boxes from the tile's corner rays at the chunk's end planes
            const ColT<float> cA = col_of<float>(g, k, ua), cB = col_of<float>(g, k, ub);
            const float rzA = rz_of<float>(g, v0), rzB = rz_of<float>(g, min(v0 + kTV, g.nv) - 1);
            const float drz = F.EV[2];
            for (int ch = lane; ch < nch; ch += 32) {
                const int i0 = ch * kP, i1 = min(i0 + kP, na) - 1;
                const float d0 = (float)i0 - ca, d1 = (float)i1 - ca;
                float bmin = INFINITY, bmax = -INFINITY, zmin = INFINITY, zmax = -INFINITY, tmax = 0.f;
                const ColT<float> cc[2] = {cA, cB};
                const float rr[2] = {rzA, rzB};
                const float dd[2] = {d0, d1};
#pragma unroll
                for (int iu2 = 0; iu2 < 2; ++iu2)
#pragma unroll
                    for (int id = 0; id < 2; ++id) {
                        const float qb = fma_rn(dd[id], cc[iu2].dqb, cc[iu2].qcb);
                        bmin = fminf(bmin, qb);
                        bmax = fmaxf(bmax, qb);
                        tmax = fmaxf(tmax, fabsf(fma_rn(dd[id], cc[iu2].inv, cc[iu2].tc)));
#pragma unroll
                        for (int ir = 0; ir < 2; ++ir) {
                            float dz, qz0;
                            ray_row(g, cc[iu2], rr[ir], dz, qz0);
                            const float qz = fma_rn(dd[id], dz, qz0);
                            zmin = fminf(zmin, qz);
                            zmax = fmaxf(zmax, qz);
                        }
                    }
                ChunkInfo ci;
                const bool finite = isfinite(bmin) && isfinite(bmax) && isfinite(zmin) && isfinite(zmax);
                // rows a voxel apart in q_z by tmax drz: the floors of kRows rows differ by at most
                // ceil((kRows - 1) tmax drz)
                ci.cells = 1 + (int)ceilf(fminf((kRows - 1) * tmax * drz * 1.0001f + 1e-4f, 1.0e6f));
                const int jb0 = floor_i(bmin) - 1, jb1 = floor_i(bmax) + 2;
                // every thread reads levels up to its lowest row's cell + cells
                const int jz0 = floor_i(zmin) - 1, jz1 = floor_i(zmax) + 1 + ci.cells;
                ci.b0 = jb0 & ~3;
                ci.z0 = jz0;
                if (!finite || jb1 > ci.b0 + BW - 1 || jz1 > ci.z0 + ZH - 1) ci.flag = 2;
                else if (ci.b0 + BW <= 0 || ci.b0 >= nb || ci.z0 + ZH <= 0 || ci.z0 >= nz) ci.flag = 0;
                else ci.flag = 1;
                info[ch] = ci;
            }
        }
        __syncthreads();
        if (abort_flag) break;

        if (warp == kConsumerWarps) {
            if (lane == 0) {
                const CUtensorMap *map = a == 0 ? &map_x : &map_y;
                for (int ch = 0; ch < nch; ++ch) {
                    const int q = gc + ch, s = q % kStages, use = q / kStages;
                    if (use > 0 && !mbar_wait(&empty[s], (use - 1) & 1, status)) {
                        abort_flag = 1;
                        // let the copies already issued land before leaving
                        for (int r = 1; r <= kStages && q - r >= 0; ++r) {
                            const int qq = q - r;
                            mbar_wait(&full[qq % kStages], (qq / kStages) & 1, status);
                        }
                        break;
                    }
                    const ChunkInfo ci = info[ch];
                    if (ci.flag == 1) {
                        mbar_arrive_expect_tx(&full[s], kBytes);
                        tma_load_4d(stages + s * SE, map, ci.b0, ci.z0, ch * kP, b, &full[s]);
                    } else {
                        mbar_arrive(&full[s]);
                    }
                }
            }
        } else {
            const bool mine = my_a == a;
            const PlaneView &pv = a == 0 ? vx : vy;
            const float *T = pv.base + b * pv.item;
            auto direct = [&](float qz0, float dz, int i0, int i1) {
                return direct_samples(T, pv.plane, pv.row, nb, nz, ca, c.tc, c.inv, c.qcb, c.dqb, qz0, dz, i0, i1);
            };
            for (int ch = 0; ch < nch; ++ch) {
                const int q = gc + ch, s = q % kStages, use = q / kStages;
                if (!mbar_wait(&full[s], use & 1, status)) {
                    // (by vote or by staying, as in the convolutions, cost 3 % of the kernel)
                    abort_flag = 1;
                    leave_warp_loop(nch - ch);
                    break;
                }
                const ChunkInfo ci = info[ch];
                const float d0 = (float)(ch * kP) - ca;
                // a chunk that the source or the pixel cuts is summed sample by sample
                const float ta = fma_rn(d0, c.inv, c.tc), tb = fma_rn(d0 + (float)(kP - 1), c.inv, c.tc);
                const bool inside = ta > 0.f && ta < 1.f && tb > 0.f && tb < 1.f;
                if (mine && ci.flag == 1 && inside) {
                    const float *st = stages + s * SE;
                    const int base = -(ci.z0 * BW + ci.b0), cells = ci.cells;
                    const unsigned top = (unsigned)((ZH - cells) * BW - 2);
                    // sums over the chunk of the level that all rows use, and of what each row adds to it
                    // (short partial sums: less rounding than one run over all planes)
                    float low = 0.f;
                    float2 part[2];
                    part[0] = part[1] = make_float2(0.f, 0.f);
                    auto plane = [&](int p, auto known) {  // known: cells, or 0
                        const float di = d0 + (float)p;
                        const float qb = fma_rn(di, c.dqb, c.qcb);
                        const float fb0 = floorf(qb), fb = qb - fb0;
                        const float2 di2 = make_float2(di, di);
                        const float2 q0 = __ffma2_rn(di2, dqz[0], qcz[0]), q1 = __ffma2_rn(di2, dqz[1], qcz[1]);
                        const float jz = floorf(q0.x);
                        // jz BW + fb0 is an exact small integer in FP32: one conversion
                        const unsigned o = __viaddmin_u32((unsigned)(int)fmaf(jz, (float)BW, fb0), (unsigned)base, top);
                        const float *r = st + p * ZH * BW + o;
                        const float2 va = make_float2(r[0], r[BW]), vb = make_float2(r[1], r[BW + 1]);
                        const float2 l01 = __ffma2_rn(make_float2(fb, fb), __ffma2_rn(va, make_float2(-1.f, -1.f), vb), va);
                        const float l2 = fmaf(fb, r[2 * BW + 1] - r[2 * BW], r[2 * BW]);
                        const float j1 = jz + 1.f;
                        if constexpr (known.value == 2) {
                            // every row lies in a cell that has L_1 as one end
                            const float e0 = l01.x - l01.y, e2 = l2 - l01.y;
                            const float2 e00 = make_float2(e0, e0), e22 = make_float2(e2, e2);
                            low += l01.y;
                            part[0] = __ffma2_rn(make_float2(__saturatef(j1 - q0.x), __saturatef(j1 - q0.y)), e00, part[0]);
                            part[1] = __ffma2_rn(make_float2(__saturatef(j1 - q1.x), __saturatef(j1 - q1.y)), e00, part[1]);
                            part[0].y = fmaf(__saturatef(q0.y - j1), e2, part[0].y);
                            part[1] = __ffma2_rn(make_float2(__saturatef(q1.x - j1), __saturatef(q1.y - j1)), e22, part[1]);
                        } else {
                            // level j weighs sat(x - j + 1) - sat(x - j): zero outside the row's own cell
                            const float2 one = make_float2(1.f, 1.f), neg = make_float2(-1.f, -1.f);
                            float2 s0 = make_float2(__saturatef(q0.x - jz), __saturatef(q0.y - jz));
                            float2 s1 = make_float2(__saturatef(q1.x - jz), __saturatef(q1.y - jz));
                            part[0] = __ffma2_rn(__ffma2_rn(s0, neg, one), make_float2(l01.x, l01.x), part[0]);
                            part[1] = __ffma2_rn(__ffma2_rn(s1, neg, one), make_float2(l01.x, l01.x), part[1]);
                            auto level = [&](float l, float j) {  // (the lowest row lies in the lowest cell)
                                const float2 t0 = make_float2(0.f, __saturatef(q0.y - j));
                                const float2 t1 = make_float2(__saturatef(q1.x - j), __saturatef(q1.y - j));
                                part[0] = __ffma2_rn(__ffma2_rn(t0, neg, s0), make_float2(l, l), part[0]);
                                part[1] = __ffma2_rn(__ffma2_rn(t1, neg, s1), make_float2(l, l), part[1]);
                                s0 = t0;
                                s1 = t1;
                            };
                            auto load = [&](int m) {
                                const float *rm = r + m * BW;
                                return fmaf(fb, rm[1] - rm[0], rm[0]);
                            };
                            level(l01.y, j1);
                            level(l2, jz + 2.f);
                            int m = 3;
                            if constexpr (known.value == 0) {
#pragma unroll 1
                                for (; m < cells; ++m) level(load(m), jz + (float)m);
                            }
                            const float l = load(m);
                            part[0].y = fmaf(s0.y, l, part[0].y);
                            part[1] = __ffma2_rn(s1, make_float2(l, l), part[1]);
                        }
                    };
                    // (planes past the volume are zero in the box)
                    auto planes = [&](auto known) {
#pragma unroll
                        for (int p = 0; p < kP; ++p) plane(p, known);
                    };
                    if (cells == 2) planes(std::integral_constant<int, 2>());
                    else if (cells == 3) planes(std::integral_constant<int, 3>());
                    else planes(std::integral_constant<int, 0>());
                    acc[0] = __fadd2_rn(acc[0], __fadd2_rn(part[0], make_float2(low, low)));
                    acc[1] = __fadd2_rn(acc[1], __fadd2_rn(part[1], make_float2(low, low)));
                } else if (mine && ci.flag != 0) {
                    const int i0 = ch * kP, i1 = min(i0 + kP, na);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        acc[j].x += direct(qcz[j].x, dqz[j].x, i0, i1);
                        acc[j].y += direct(qcz[j].y, dqz[j].y, i0, i1);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
            }
            if (mine) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    // the rows share the levels they load: where a result is not finite (an infinite or
                    // NaN voxel, or an overflow), each ray is summed from its own samples
                    if (!(fabsf(acc[j].x) < INFINITY)) acc[j].x = direct(qcz[j].x, dqz[j].x, 0, na);
                    if (!(fabsf(acc[j].y) < INFINITY)) acc[j].y = direct(qcz[j].y, dqz[j].y, 0, na);
                }
            }
        }
        gc += nch;
        __syncthreads();
        if (abort_flag) break;
    }
    if (consumer && !abort_flag) {
        // per row: when the row's 32 columns lie inside the panel and start on a 16-byte
        // boundary, every fourth lane stores its own and its three neighbours' rays as one
        // float4 (eight vector stores per warp and row); otherwise one float per ray
#pragma unroll
        for (int rr = 0; rr < kRows; ++rr) {
            const int iv = iv0 + rr;
            const bool ray_ok = col_ok && iv < g.nv;
            const float sum = rr & 1 ? acc[rr >> 1].y : acc[rr >> 1].x, dz = rr & 1 ? dqz[rr >> 1].y : dqz[rr >> 1].x;
            const float r = ray_ok ? sum * ray_step<float>(g, my_a, c.dqb, dz) * g.scale : 0.f;
            float *out = proj + (((long long)b * g.na + k) * g.nv + iv) * g.nu + iu;
            if ((g.nu & 3) == 0 && (reinterpret_cast<uintptr_t>(proj) & 15) == 0 && u0 + kTU <= g.nu &&
                iv < g.nv) {  // uniform over the warp
                const float r1 = __shfl_down_sync(0xffffffffu, r, 1);
                const float r2 = __shfl_down_sync(0xffffffffu, r, 2);
                const float r3 = __shfl_down_sync(0xffffffffu, r, 3);
                if ((lane & 3) == 0) {
                    float4 v = make_float4(r, r1, r2, r3);
                    if (accumulate) {
                        const float4 q = *reinterpret_cast<const float4 *>(out);
                        v.x += q.x; v.y += q.y; v.z += q.z; v.w += q.w;
                    }
                    *reinterpret_cast<float4 *>(out) = v;
                }
            } else if (ray_ok) {
                *out = accumulate ? *out + r : r;
            }
        }
    }
}

// ---- launcher ----------------------------------------------------------------------

// Boxes (columns, z, planes per chunk), smallest first. Coarse panels spread a tile over more
// voxels: fewer planes per chunk keep several CTAs per SM, and any box beats the direct kernel
// (226 x 221 x 211 voxels, 256 x 257 panel, 48 x 28 x 4 box: 4.1 ms against 10.2 direct).
struct FwdCfg {
    int bw, zh, np;
};
static const FwdCfg kCfgs[] = {{28, 14, 8}, {32, 16, 8}, {36, 18, 8}, {40, 24, 4}, {48, 28, 4}, {64, 36, 4}, {96, 48, 2}};

// Shared memory of the staged kernel: two boxes, their barriers, the chunk list, the abort flag.
static size_t staged_smem(const GeomDev &d, const FwdCfg &c) {
    const size_t chunks = (std::max(d.n[0], d.n[1]) + c.np - 1) / c.np;
    return 128 + (size_t)kStages * c.np * c.zh * c.bw * 4 + 2 * kStages * 8 + chunks * sizeof(ChunkInfo) + sizeof(int);
}
constexpr size_t kStagedSmemMax = 227 * 1024;

template <int BW, int ZH, int NP>
static int launch_cfg(const cbct_geom *g, const CUtensorMap &mx, const CUtensorMap &my, const PlaneView &vx,
                      const PlaneView &vy, float *proj, int batch, int accumulate, cudaStream_t st) {
    static_assert(BW % 4 == 0 && BW <= 256 && ZH <= 256, "TMA box");
    const GeomDev &d = g->dev;
    auto kern = k_forward_tma<BW, ZH, NP>;
    const size_t smem = staged_smem(d, FwdCfg{BW, ZH, NP});
    dim3 grd((d.nu + kTU - 1) / kTU, (d.nv + kTV - 1) / kTV, d.na * batch);
    kern<<<grd, kThreads, smem, st>>>(mx, my, d, vx, vy, proj, accumulate, g->status);
    CBCT_LAUNCH_CHECK("forward_project (staged) launch");
    return 0;
}

// Rays times planes below which one launch of the direct kernel is faster than the plane copy
// and the staged kernel: 16^3 / 8 angles (2^16) 16 us direct against 33 staged, 64^3 / 64 angles
// (2^24.6) 88 against 38.
constexpr long long kDirectSamples = 1 << 20;

// Returns 1 if the staged kernel handled the call, 0 if the caller should use the direct kernel
// (small calls, boxes or chunk lists that do not fit, no memory for the plane copies: the direct kernel
// needs none), negative on error.
int forward_staged(const cbct_geom *g, const float *vol, float *proj, int batch, int accumulate, cudaStream_t st) {
    const GeomDev &d = g->dev;
    const int nx = d.n[0], ny = d.n[1], nz = d.n[2];
    if (g->fwd_cfg < 0 || (long long)batch * d.na * d.nv * d.nu * std::max(nx, ny) <= kDirectSamples) return 0;
    const FwdCfg cf = kCfgs[g->fwd_cfg];
    if (staged_smem(d, cf) > kStagedSmemMax) return 0;
    const long long nvox = (long long)nx * ny * nz, slices = (long long)nz * batch;
    // y planes are read from the volume itself when its rows start on 16 bytes (a TMA stride)
    const bool copy_y = (nx & 3) != 0 || (reinterpret_cast<uintptr_t>(vol) & 15) != 0;
    const int px = (ny + 3) & ~3, py = (nx + 3) & ~3;
    const long long ex = (long long)batch * nx * nz * px, ey = copy_y ? (long long)batch * ny * nz * py : 0;
    float *buf = nullptr;
    const cudaError_t ea = scratch_alloc((void **)&buf, sizeof(float) * (ex + ey), st);
    if (ea == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return 0;
    }
    CBCT_CUDA_TRY(ea);
    float *tx = buf, *ty = buf + ex;
    const PlaneView vx{tx, (long long)nx * nz * px, (long long)nz * px, px};
    const PlaneView vy = copy_y ? PlaneView{ty, (long long)ny * nz * py, (long long)nz * py, py}
                                : PlaneView{vol, nvox, nx, (long long)nx * ny};
    int rc = 0;
    {
        const unsigned gz = (unsigned)std::min<long long>(slices, 65535);
        dim3 gx((nx + 31) / 32, (ny + 31) / 32, gz);
        k_planes_x<<<gx, dim3(32, 8), 0, st>>>(vol, tx, nx, ny, nz, slices, px);
        if (copy_y) k_planes_y<<<dim3(ny, gz), 128, 0, st>>>(vol, ty, nx, ny, nz, slices, py);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "forward_project: plane copies");
    }
    CUtensorMap mx, my;
    if (rc == 0) {
        auto encode = [&](CUtensorMap *m, const PlaneView &v, int nb, int np) {
            const uint64_t dims[4] = {(uint64_t)nb, (uint64_t)nz, (uint64_t)np, (uint64_t)batch};
            const uint64_t str[3] = {(uint64_t)v.row * 4, (uint64_t)v.plane * 4, (uint64_t)v.item * 4};
            const uint32_t box[4] = {(uint32_t)cf.bw, (uint32_t)cf.zh, (uint32_t)cf.np, 1};
            return encode_tmap(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, v.base, dims, str, box);
        };
        rc = encode(&mx, vx, ny, nx);
        if (rc == 0) rc = encode(&my, vy, nx, ny);
    }
    if (rc == 0) {
        switch (g->fwd_cfg) {
            case 0: rc = launch_cfg<28, 14, 8>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
            case 1: rc = launch_cfg<32, 16, 8>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
            case 2: rc = launch_cfg<36, 18, 8>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
            case 3: rc = launch_cfg<40, 24, 4>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
            case 4: rc = launch_cfg<48, 28, 4>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
            case 5: rc = launch_cfg<64, 36, 4>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
            default: rc = launch_cfg<96, 48, 2>(g, mx, my, vx, vy, proj, batch, accumulate, st); break;
        }
    }
    cudaFreeAsync(buf, st);
    return rc == 0 ? 1 : rc;
}

// Shared-memory limits of the staged kernels on the current device (once per geometry: a limit set by
// each call for its own volume could be lowered by another thread's call before the launch).
int forward_prime() {
    for (auto kern : {k_forward_tma<28, 14, 8>, k_forward_tma<32, 16, 8>, k_forward_tma<36, 18, 8>, k_forward_tma<40, 24, 4>,
                      k_forward_tma<48, 28, 4>, k_forward_tma<64, 36, 4>, k_forward_tma<96, 48, 2>})
        CBCT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmemMax));
    return 0;
}

// Pick the smallest box that holds a tile's footprint over one chunk of np planes (need + (np -
// 1) slope voxels, host bounds of geometry_create), or -1 for the direct kernel.
int choose_forward_cfg(double need_b, double need_z, double slope_b, double slope_z) {
    for (int i = 0; i < (int)(sizeof(kCfgs) / sizeof(kCfgs[0])); ++i) {
        const FwdCfg &c = kCfgs[i];
        if (need_b + (c.np - 1) * slope_b <= c.bw && need_z + (c.np - 1) * slope_z <= c.zh) return i;
    }
    return -1;
}

}  // namespace cbct
