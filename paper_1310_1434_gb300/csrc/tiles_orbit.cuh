// Tile functions of the projector pair over orbits of rays (orbit.h): the
// integer walk of one canonical ray serves the four or eight rays that the
// symmetries of the pixel grid and of the scan take into one another.
#pragma once

#include "air_internal.cuh"
#include "packed.cuh"

namespace air {

// Physical pixel of the canonical pixel (k, r) in a frame.
__device__ __forceinline__ void orb_pixel(int code, int n, int k, int r, int &ix, int &iy) {
    const int a = code & ORB_FX ? n - 1 - k : k, b = code & ORB_FY ? n - 1 - r : r;
    ix = code & ORB_T ? b : a;
    iy = code & ORB_T ? a : b;
}

// ======================================================================
// Stack of frames: stack[plane][k][r + ORB_PAD] = the four pixels that the
// plane's frames put at the canonical pixel (k, r), one float4.  The pad rows
// are zeroed with the plan.  One 32 x 32 canonical tile of one plane per block.
// Frames without ORB_T read along k and are turned in shared memory.
// ======================================================================
__device__ __forceinline__ void tile_orb_pack(const SliceDesc &s, int arg, int tile, float *sm) {
    const bool swap = (arg & ARG_SWAP) != 0;
    arg &= ARG_MASK;
    const bool cg = arg == SRC_P || arg == SRC_P_NEXT, next = arg == SRC_P_NEXT;
    const int stop = cg ? s.cg->stop : 0;
    // SRC_P_NEXT: p = r + beta p on the way, from the image that held it to the
    // other one; plane 0 writes what it reads for its first frame, every pixel
    // once.  (Folded into the general path's copies it gained nothing.)
    const float *src = arg == SRC_X ? s.x : (!cg ? s.ext_in : (swap != next ? s.q : s.p));
    float *to = swap ? s.q : s.p;
    const float bt = next ? (float)s.cg->beta : 0.f;
    const int n = s.n, tpr = (n + 31) / 32, nt = tpr * tpr;
    const int plane = tile / nt, t = tile - plane * nt;
    const int k0 = (t % tpr) * 32, r0 = (t / tpr) * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float(*f)[32][33] = reinterpret_cast<float(*)[32][33]>(sm);   // [frame][k][r]
    constexpr int STEP = AIR_THREADS / 32, ROWS = 32 / STEP;
    float in[4][ROWS], res[4][ROWS];                     // on their way together, and with stop
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int code = s.orb_frame[4 * plane + q];
        const bool tr = (code & ORB_T) != 0;
#pragma unroll
        for (int m = 0; m < ROWS; ++m) {
            const int kk = tr ? w + m * STEP : lane, rr = tr ? lane : w + m * STEP;
            in[q][m] = res[q][m] = 0.f;
            if (k0 + kk < n && r0 + rr < n) {
                int ix, iy;
                orb_pixel(code, n, k0 + kk, r0 + rr, ix, iy);
                const size_t i = (size_t)iy * n + ix;
                in[q][m] = ld_data(src + i);
                if (next) res[q][m] = ld_data(s.r + i);
            }
        }
    }
    if (stop) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int code = s.orb_frame[4 * plane + q];
        const bool tr = (code & ORB_T) != 0;
#pragma unroll
        for (int m = 0; m < ROWS; ++m) {
            const int kk = tr ? w + m * STEP : lane, rr = tr ? lane : w + m * STEP;
            const float v = next ? fmaf(bt, in[q][m], res[q][m]) : in[q][m];
            if (next && plane == 0 && q == 0 && k0 + kk < n && r0 + rr < n) {
                int ix, iy;
                orb_pixel(code, n, k0 + kk, r0 + rr, ix, iy);
                to[(size_t)iy * n + ix] = v;
            }
            f[q][kk][rr] = v;
        }
    }
    __syncthreads();
    const int ld = orb_ld(n);
    float4 *out = s.orb_stack + (size_t)plane * n * ld;
#pragma unroll
    for (int m = 0; m < 32; m += AIR_THREADS / 32) {
        const int kk = w + m;
        if (k0 + kk < n && r0 + lane < n)
            out[(size_t)(k0 + kk) * ld + r0 + lane + ORB_PAD] =
                make_float4(f[0][kk][lane], f[1][kk][lane], f[2][kk][lane], f[3][kk][lane]);
    }
    __syncthreads();
}
constexpr int ORB_PACK_FLOATS = 4 * 32 * 33;

// ======================================================================
// Projector over orbits.  One thread walks one canonical ray for the rays of
// its orbit (NP planes of four): per column one evaluation of the overlaps
// (orb_overlap), and for each plane one 16-byte load of the four pixels of
// row r0, one of row r0 + 1 where the span reaches it, and two packed FMAs
// for each.  The lanes of a warp hold neighbouring rays and walk the same
// columns in step, so that a load's 32 addresses are neighbouring pixels of
// one stack column; outside a ray's own walk range its row is clamped into
// the zero pads.  The columns of a warp's rays are split over orb_ks warps,
// whose sums are added in a fixed order: at 512^2 / 800 views eight parts a
// ray took 89 us, four 98, two 99, one 155 (the image copies included, and
// before the loads of four columns were issued together: 78.5 us now).
// Bound: bytes into registers (8 for each ray and column; 18 M L1 data-pipe
// wavefronts, 72 % of their rate) and L2 latency (a third of the sectors hit
// L1).  The general pair's projector takes 137 us there, 36 M wavefronts.
// ======================================================================

// Overlaps of the span [p, p + Ma] (2^-32 px) with row p >> 32 and the next
// one.  np = ~p: the first row takes min(Ma, ~(p mod 2^32)), a row boundary
// 2^-32 px early, and the next the rest; both kernels use this form.
__device__ __forceinline__ void orb_overlap(unsigned nlo, unsigned Ma, unsigned &ov0, unsigned &ov1) {
    ov0 = min(Ma, nlo);
    ov1 = Ma - ov0;
}

// Four pixels, or zeros where `want` is 0 (the load is not issued).  In PTX so
// that the loads of several steps are issued ahead of their FMAs: as plain
// loads the 512^2 / 800 views projection took 98 us instead of 86.
__device__ __forceinline__ ulonglong2 ld_pixels(const ulonglong2 *p) {
    ulonglong2 v;
    asm volatile("ld.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ ulonglong2 ld_pixels_if(const ulonglong2 *p, unsigned want) {
    ulonglong2 v;
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n mov.b64 %0, 0;\n mov.b64 %1, 0;\n"
        " @q ld.global.v2.u64 {%0, %1}, [%2];\n}"
        : "=&l"(v.x), "=&l"(v.y)
        : "l"(p), "r"(want));
    return v;
}

constexpr int ORB_U = 4;                                          // columns whose loads are in flight together
template <int NP>
struct OrbAcc {
    unsigned long long v[2 * NP];   // frames {0, 1}, {2, 3} of each plane
};

// U columns of the walk: every load is issued before the first FMA, so that a
// warp has 4 U of them (two planes) in flight.
template <int NP, int U>
__device__ __forceinline__ void orb_steps(unsigned long long &np, const ulonglong2 *col, int ld, size_t plane, unsigned Ma,
                                          int n, OrbAcc<NP> &a, OrbAcc<NP> &b) {
    ulonglong2 x0[U][NP], x1[U][NP];
    unsigned ov0[U], ov1[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        orb_overlap((unsigned)np, Ma, ov0[u], ov1[u]);
        const int nr = min(max((int)(np >> 32), -1 - n), ORB_PAD - 1);   // ~row, the row clamped to [-2, n]
        const ulonglong2 *c = col + u * ld - nr;                         // col is one row past the column's row 0
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            x0[u][q] = ld_pixels(c + q * plane - 1);
            x1[u][q] = ld_pixels_if(c + q * plane, ov1[u]);
        }
        np -= Ma;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const float f0 = __uint2float_rn(ov0[u]), f1 = __uint2float_rn(ov1[u]);
        const unsigned long long w0 = pair2(f0, f0), w1 = pair2(f1, f1);
        OrbAcc<NP> &s = u & 1 ? b : a;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            s.v[2 * q] = fma2(w0, x0[u][q].x, s.v[2 * q]);
            s.v[2 * q + 1] = fma2(w0, x0[u][q].y, s.v[2 * q + 1]);
            s.v[2 * q] = fma2(w1, x1[u][q].x, s.v[2 * q]);
            s.v[2 * q + 1] = fma2(w1, x1[u][q].y, s.v[2 * q + 1]);
        }
    }
}

template <int NP>
__device__ __forceinline__ void tile_orb_fwd_np(const SliceDesc &s, int arg, int tile, float *sm) {
    float *__restrict__ dst = arg == SRC_EXT ? s.ext_out : s.z;
    const int n = s.n, KS = s.orb_ks, W = AIR_THREADS / 32 / KS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rw = warp % W, kp = warp / W;
    const int t = tile * W + rw;
    const bool live = t < s.orb_ntask;
    float sum[4 * NP] = {};
    uint2 info = make_uint2(0u, 0u);
    float c = 0.f;
    int i = 0;
    bool mine = false;
    if (live) {
        const unsigned word = __ldg(s.orb_task + t);
        const int first = (int)(word & 0x3ffffffu), cnt = (int)(word >> 26) + 1;
        mine = lane < cnt;
        i = first + min(lane, cnt - 1);
        const RayFx r = s.orb_ray[i];
        c = r.cs;
        info = __ldg(s.orb_info + i);
        const int k0 = walk_k0(info.x), k1 = walk_k1(info.x);
        const int ka = __reduce_min_sync(0xffffffffu, k0 < k1 ? k0 : n);
        const int kb = max(ka, (int)__reduce_max_sync(0xffffffffu, k0 < k1 ? k1 : 0));
        const int q0 = ka + (kb - ka) * kp / KS, q1 = ka + (kb - ka) * (kp + 1) / KS;
        const int ld = orb_ld(n);
        const size_t plane = (size_t)n * ld;
        const ulonglong2 *col = reinterpret_cast<const ulonglong2 *>(s.orb_stack) + (size_t)q0 * ld + ORB_PAD;
        if (NP == 1) col += plane * s.orb_seg[info.y].cls;
        const unsigned Ma = r.Mlo;
        unsigned long long np = ~((unsigned long long)r.L0 + (unsigned long long)q0 * Ma);
        OrbAcc<NP> a{}, b{};
        int k = q0;
#pragma unroll 1
        for (; k + ORB_U <= q1; k += ORB_U) {
            orb_steps<NP, ORB_U>(np, col, ld, plane, Ma, n, a, b);
            col += ORB_U * ld;
        }
#pragma unroll 1
        for (; k + 2 <= q1; k += 2) {
            orb_steps<NP, 2>(np, col, ld, plane, Ma, n, a, b);
            col += 2 * ld;
        }
        if (k < q1) orb_steps<NP, 1>(np, col, ld, plane, Ma, n, a, b);
#pragma unroll
        for (int q = 0; q < 2 * NP; ++q) {
            const float2 x = unpair2(a.v[q]), y = unpair2(b.v[q]);
            sum[2 * q] = x.x + y.x;
            sum[2 * q + 1] = x.y + y.y;
        }
    }
    if (KS > 1) {
        float4 *part = reinterpret_cast<float4 *>(sm);            // [plane][kp][rw][lane]
#pragma unroll
        for (int q = 0; q < NP; ++q)
            part[q * AIR_THREADS + threadIdx.x] = make_float4(sum[4 * q], sum[4 * q + 1], sum[4 * q + 2], sum[4 * q + 3]);
        __syncthreads();
        if (kp == 0) {
            for (int h = 1; h < KS; ++h)
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const float4 v = part[q * AIR_THREADS + h * W * 32 + threadIdx.x];
                    sum[4 * q] += v.x;
                    sum[4 * q + 1] += v.y;
                    sum[4 * q + 2] += v.z;
                    sum[4 * q + 3] += v.w;
                }
        }
        __syncthreads();
    }
    if (kp == 0 && live && mine) {
        const OrbSeg &g = s.orb_seg[info.y];
        const int j = i - g.ray0, down = g.down;
#pragma unroll
        for (int q = 0; q < 4 * NP; ++q) {
            const int z = g.zoff[q];
            if (z >= 0) dst[z + ((down >> q) & 1 ? -j : j)] = s.dx * (c * sum[q]);
        }
    }
}

__device__ __forceinline__ void tile_orb_fwd(const SliceDesc &s, int arg, int tile, float *sm) {
    if (arg == SRC_P && s.cg->stop) return;
    if (s.orb == 8) tile_orb_fwd_np<2>(s, arg, tile, sm);
    else tile_orb_fwd_np<1>(s, arg, tile, sm);
}

// ======================================================================
// Backprojector over orbits, gathered: a thread owns four pixels of a column
// in the canonical frame and sums, for each of the frames, what the rays of
// the tile's segments put there.  Per segment and pair of rows the first ray
// that can meet them follows from the fan angle of their lower right corner
// (rays ascend by angle; the angle is expanded to second order once per warp
// and segment), and the next few rays are tried with the integer overlaps of
// the projector's walk: a ray's span covers one or both rows, or misses with
// weight zero.  Trying a ray for two rows at a time loads it and its samples
// 2.8 times per pair instead of twice 2.05 times.  The tile's rays are
// staged in shared memory four segments at a time by asynchronous copies:
// the rays, and the samples of their orbits, which OP_ORB_ZPACK put side by
// side, times the ray's c.  A segment's rays past the tile's last one, which
// no pixel of the tile meets, are staged as well: the candidates may run
// onto them.  The sums of each frame go to an image of their own, which
// OP_BWD_FIN adds in a fixed order.
// A sum of FP32 values that grows over all the views loses more by each
// addition the larger it gets: the accumulators are put aside every few rounds
// (`fold`) and start again from zero, about ORB_SUMS partial sums to a pixel
// and frame over all splits.  They lie in shared memory, where they take the
// place of a third stage of the ring, which brought nothing.  With the images
// summed as in bwd_fin the error of A^T against FP64, relative to the image, is
// 3.4e-8 at 512^2 / 800 views (one accumulator and a running sum 9.3e-8, the
// general pair 6.0e-8), 3.5e-8 at 350^2 / 200 (6.6e-8, 5.1e-8), 4.6e-8 at
// 1024^2 / 800 (9.0e-8, 5.6e-8).
// At 512^2 / 800 views a call with packing and sum takes 87 us (89 with one
// accumulator and three stages; general: 239): 55 M instead of 207 M warp
// instructions and 19 M instead of 55 M shared-memory wavefronts.
// Bound: the shared-memory data path (72 %) and instruction issue (63 % active).
// ======================================================================
// Weights of the rows 0 and 1 of a span that starts in row d: f0 belongs to row
// d and f1 to row d + 1.  In PTX because the compiler made branches of it.
__device__ __forceinline__ void orb_rows(int d, float f0, float f1, float &lo, float &hi) {
    asm("{\n .reg .pred a, b, c;\n .reg .f32 t, u;\n"
        " setp.eq.s32 a, %2, 0;\n setp.eq.s32 b, %2, -1;\n setp.eq.s32 c, %2, 1;\n"
        " selp.f32 t, %4, 0f00000000, b;\n selp.f32 u, %3, 0f00000000, c;\n"
        " selp.f32 %0, %3, t, a;\n selp.f32 %1, %4, u, a;\n}"
        : "=f"(lo), "=f"(hi)
        : "r"(d), "f"(f0), "f"(f1));
}

constexpr int ORB_SEGS = 4;                              // segments staged at a time
constexpr int ORB_STAGES = 2;
constexpr int ORB_ROWS = 4;                              // pixels of a thread, along r
constexpr int ORB_SUMS = 8;                              // partial sums a pixel and frame is made of, of at least two
constexpr int ORB_FOLD_MAX = 8;                          // and at most eight rounds
constexpr int ORB_EARLY = 152;                           // blocks of a launch that leaves SMs idle: one per SM
constexpr int ORB_ENT = ORB_RAYS + ORB_CAND;             // staged rays of a segment

constexpr int ORB_PATCH_K = 8, ORB_PATCH_R = 16;         // pixels of a warp
constexpr int ORB_PAR = 2 * AIR_THREADS / 32;            // float4s of a staged segment's parameters, two per warp

__host__ __device__ inline size_t orb_bwd_smem(int nf) {
    return ((size_t)ORB_STAGES * ORB_SEGS * (ORB_ENT * (1 + nf / 4) + ORB_PAR) + (size_t)AIR_THREADS * nf) * 16;
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Samples of the orbits' rays side by side: orb_z[plane][padded ray] = c times
// the four samples of the plane's frames, zero for the empty rays.
__device__ __forceinline__ void tile_orb_zpack(const SliceDesc &s, int mode, int tile) {
    const float *Z = mode == BWD_PLAIN ? s.ext_in : s.zc;
    const int nch = orb_zchunks(s), seg = tile / nch;
    const OrbSeg &g = s.orb_seg[seg];
    const int i = (tile - seg * nch) * ORB_ZPACK + (int)threadIdx.x;
    const float c = i < g.cnt ? __ldg(&s.orb_ray[g.ray0 + i].cs) : 0.f;
    const int down = g.down;
    grid_wait();
    if (i >= g.cnt + ORB_CAND || (mode == BWD_Q && s.cg->stop)) return;
    for (int p = 0; p < orb_planes(s); ++p) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int z = g.zoff[4 * p + q];
            v[q] = z < 0 || i >= g.cnt ? 0.f : c * ld_data(Z + z + ((down >> (4 * p + q)) & 1 ? -i : i));
        }
        s.orb_z[(size_t)p * s.orb_npad + g.pad0 + i] = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// arctan(u) for |u| <= 0.45 by its Maclaurin (Gregory) series through u^13;
// the alternating-series remainder is below 0.45^15/15 = 4.2e-7 rad.
__device__ __forceinline__ float atan_series(float u) {
    const float w = u * u;
    float p = 1.f / 13.f;
    p = fmaf(p, w, -1.f / 11.f);
    p = fmaf(p, w, 1.f / 9.f);
    p = fmaf(p, w, -1.f / 7.f);
    p = fmaf(p, w, 1.f / 5.f);
    p = fmaf(p, w, -1.f / 3.f);
    p = fmaf(p, w, 1.f);
    return u * p;
}
__device__ __forceinline__ float orb_atan(float u) { return fabsf(u) <= 0.45f ? atan_series(u) : atanf(u); }

// The four pixels of a thread once more, where a sample that is not finite has
// reached them: the sweep below gives it to every pixel whose candidates it was
// among, with a weight of zero where its ray misses.  Here a miss is left out.
// By itself, on the rays in memory; a function that is called, so that the
// sweep's code stays together (with a second sweep behind it 20 CG steps at
// 128^2 / 90 views took 685 us instead of 672).
template <int NF>
__device__ __noinline__ void orb_bwd_hits(const SliceDesc &s, int cls, int split, int txy, int k, int r) {
    const int S = s.orb_splits, t0 = cls * (tiles_bwd_xy(s) + 1) + txy;
    const int e0 = __ldg(s.orb_tile0 + t0), e1 = __ldg(s.orb_tile0 + t0 + 1);
#pragma unroll 1
    for (int y = 0; y < ORB_ROWS; ++y) {
        if (k >= s.n || r + y >= s.n) continue;
        float acc[NF] = {}, sum[NF] = {};
#pragma unroll 1
        for (int e = e0 + split, m = 1; e < e1; e += S, ++m) {
            const uint2 w = __ldg(s.orb_ent + e);
            const OrbSeg *__restrict__ g = s.orb_seg + (w.x & 0x1ffffu);
            // the first ray that can meet the pixel pair of the sweep
            const float X = (float)(k + 1) - g->sx, Y = (float)(r + (y & ~1)) - g->sy;
            const float cr = fmaf(g->cx, Y, -g->cy * X), dt = fmaf(g->cx, X, g->cy * Y);
            const int i = __float2int_ru(fmaf(orb_atan(cr / dt), s.inv_dg, g->ioff - (float)((int)w.y - g->pad0)));
            const int first = (int)w.y + min(max(i, 0), (int)((w.x >> 17) & 0x7fu)), nc = (int)(w.x >> 24);
#pragma unroll 1
            for (int c = first; c < first + nc; ++c) {
                const uint4 ray = __ldg(s.orb_bray + c);
                const unsigned long long p = (unsigned long long)(unsigned)k * ray.z + (((unsigned long long)ray.y << 32) | ray.x);
                unsigned ov0, ov1;
                orb_overlap(~(unsigned)p, ray.z, ov0, ov1);
                const int d = (int)(p >> 32) - (r + y);
                if (d != 0 && d != -1) continue;
                const float f = __uint2float_rn(d == 0 ? ov0 : ov1);
#pragma unroll
                for (int v = 0; v < NF / 4; ++v) {
                    const float4 z = ld_data(s.orb_z + (size_t)v * s.orb_npad + c);
                    acc[4 * v] = fmaf(f, z.x, acc[4 * v]);
                    acc[4 * v + 1] = fmaf(f, z.y, acc[4 * v + 1]);
                    acc[4 * v + 2] = fmaf(f, z.z, acc[4 * v + 2]);
                    acc[4 * v + 3] = fmaf(f, z.w, acc[4 * v + 3]);
                }
            }
            if (m % (2 * ORB_SEGS) == 0 || e + S >= e1) {
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    sum[f] += acc[f];
                    acc[f] = 0.f;
                }
            }
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            int ix, iy;
            orb_pixel(s.orb_frame[cls * 4 + f], s.n, k, r + y, ix, iy);
            s.bwd_part[((size_t)(split * 8 + cls * 4 + f) * s.n + iy) * s.n + ix] = sum[f];
        }
    }
}

template <int NF>
__device__ __forceinline__ void tile_orb_bwd_nf(const SliceDesc &s, int mode, int tile, float *sm) {
    constexpr int NV = NF / 4;                           // float4s of samples per ray
    constexpr int SEG = ORB_ENT * (1 + NV) + ORB_PAR;    // float4s of a staged segment
    const int n = s.n, ntxy = tiles_bwd_xy(s), S = s.orb_splits;
    const int cls = NF == 8 ? 0 : tile / (ntxy * S);
    const int ct = tile - cls * ntxy * S, split = ct / ntxy, txy = ct - split * ntxy;
    const int tpr = (n + BWD_T - 1) / BWD_T;
    const int K0 = (txy % tpr) * BWD_T, R0 = (txy / tpr) * BWD_T;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = K0 + (warp & 3) * ORB_PATCH_K + (lane & 7);
    const int r = R0 + (warp >> 2) * ORB_PATCH_R + (lane >> 3) * ORB_ROWS;
    const int e0 = __ldg(s.orb_tile0 + cls * (ntxy + 1) + txy), e1 = __ldg(s.orb_tile0 + cls * (ntxy + 1) + txy + 1);
    const int ne = e1 - e0 > split ? (e1 - e0 - split + S - 1) / S : 0;      // this split's entries
    const uint2 *__restrict__ ent = s.orb_ent + e0 + split;                  // every S-th
    float4 *buf = reinterpret_cast<float4 *>(sm);
    ulonglong2 *aside = reinterpret_cast<ulonglong2 *>(buf + ORB_STAGES * ORB_SEGS * SEG) + threadIdx.x;   // [NF][AIR_THREADS]

    // warps 2 q and 2 q + 1 stage the round's segment q; warp `round` mod 8
    // writes every warp's parameters of the four segments.  The rays and the
    // parameters come from the plan's tables: those of the first round
    // are asked for before the wait for the last kernel where a launch leaves
    // SMs idle (128^2 / 90 views: 734 -> 703 us for 20 CG steps; a launch of
    // more than a block per SM lost half a percent by it).
    auto stage = [&](int round, bool rays, bool samples) {
        const int e = round * ORB_SEGS + (warp >> 1);
        float4 *ring = buf + (round % ORB_STAGES) * ORB_SEGS * SEG;
        if (e < ne) {
            const uint2 w = __ldg(ent + (size_t)e * S);
            const int m = (int)((w.x >> 17) & 0x7fu) + ORB_CAND;
            float4 *st = ring + (warp >> 1) * SEG;
            for (int i = (warp & 1) * 32 + lane; i < m; i += 64) {
                if (rays) cp_async16(st + i, s.orb_bray + w.y + i);
#pragma unroll
                for (int v = 0; v < NV && samples; ++v) cp_async16(st + ORB_ENT * (1 + v) + i, s.orb_z + (size_t)v * s.orb_npad + w.y + i);
            }
        }
        if (rays && (round & 7) == warp) {
            const int q = lane >> 3, pw = lane & 7, eq = round * ORB_SEGS + q;   // segment, warp
            if (eq < ne) {
                // the ray index over warp pw's pixels, to second order about
                // the middle of their lower right corners
                const uint2 w = __ldg(ent + (size_t)eq * S);
                const OrbSeg *__restrict__ g = s.orb_seg + (w.x & 0x1ffffu);
                const float4 src = __ldg(reinterpret_cast<const float4 *>(g));      // source, central direction
                const float first = (float)((int)w.y - __ldg(&g->pad0));
                const float X = (float)(K0 + (pw & 3) * ORB_PATCH_K + 1) + 0.5f * (ORB_PATCH_K - 1) - src.x;
                const float Y = (float)(R0 + (pw >> 2) * ORB_PATCH_R) + 0.5f * (ORB_PATCH_R - 1) - src.y;
                const float cr = fmaf(src.z, Y, -src.w * X), dt = fmaf(src.z, X, src.w * Y);
                const float i2 = __fdividef(1.f, fmaf(cr, cr, dt * dt)), si = s.inv_dg * i2, sii = si * i2;
                float4 *par = ring + q * SEG + SEG - ORB_PAR + 2 * pw;
                par[0] = make_float4(fmaf(orb_atan(__fdividef(cr, dt)), s.inv_dg, __ldg(&g->ioff) - first), -Y * si, X * si,
                                     2.f * X * Y * sii);
                par[1] = make_float4(fmaf(Y, Y, -X * X) * sii, __uint_as_float(w.x >> 24),
                                     __uint_as_float((w.x >> 17) & 0x7fu), 0.f);
            }
        }
        if (samples) asm volatile("cp.async.commit_group;" ::: "memory");
    };

    unsigned long long acc[ORB_ROWS][NF / 2];
#pragma unroll
    for (int q = 0; q < ORB_ROWS; ++q)
#pragma unroll
        for (int f = 0; f < NF / 2; ++f) acc[q][f] = 0ull;

    const bool early = gridDim.x <= ORB_EARLY;
    if (early) stage(0, true, false);
    grid_wait();
    const int stop = mode == BWD_Q ? s.cg->stop : 0;     // on its way with the first round
    stage(0, !early, true);
    // the thread's column and first row from the middle of its warp's pixels
    const float u = (float)(lane & 7) - 0.5f * (ORB_PATCH_K - 1);
    const float v0 = (float)((lane >> 3) * ORB_ROWS) - 0.5f * (ORB_PATCH_R - 1);
    const int rounds = stop ? 0 : (ne + ORB_SEGS - 1) / ORB_SEGS;
    // rounds that are summed by themselves: see above
    const int fold = min(ORB_FOLD_MAX, max(2, (rounds * S + ORB_SUMS - 1) / ORB_SUMS));
#pragma unroll 1
    for (int round = 0; round < rounds;) {
        const int from = round, to = min(round + fold, rounds);
#pragma unroll 1
        for (; round < to; ++round) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();             // this round's rays are there; the last round's buffer is free
            stage(round + 1, true, true);
            const int m = min(ORB_SEGS, ne - round * ORB_SEGS);
#pragma unroll 1
            for (int q = 0; q < m; ++q) {
                const float4 *st = buf + ((round % ORB_STAGES) * ORB_SEGS + q) * SEG;
                const float4 ia = st[SEG - ORB_PAR + 2 * warp], ib = st[SEG - ORB_PAR + 2 * warp + 1];
                const int nc = __float_as_int(ib.y), cnt = __float_as_int(ib.z);
                const float4 *at[ORB_ROWS / 2];
#pragma unroll
                for (int y = 0; y < ORB_ROWS / 2; ++y) {
                    const float v = v0 + (float)(2 * y);
                    const int i = __float2int_ru(fmaf(ib.x, u * v, fmaf(ia.w, 0.5f * (u * u - v * v),
                                                                        fmaf(ia.z, v, fmaf(ia.y, u, ia.x)))));
                    at[y] = st + min(max(i, 0), cnt);
                }
#pragma unroll 1
                for (int c = 0; c < nc; ++c) {
#pragma unroll
                    for (int y = 0; y < ORB_ROWS / 2; ++y) {
                        const float4 ray = at[y][c];
                        const unsigned Ma = __float_as_uint(ray.z);
                        const unsigned long long p =
                            (unsigned long long)(unsigned)k * Ma +
                            (((unsigned long long)__float_as_uint(ray.y) << 32) | __float_as_uint(ray.x));
                        unsigned ov0, ov1;
                        orb_overlap(~(unsigned)p, Ma, ov0, ov1);
                        const int d = (int)(p >> 32) - (r + 2 * y);
                        const float f0 = __uint2float_rn(ov0), f1 = __uint2float_rn(ov1);
                        float lo, hi;
                        orb_rows(d, f0, f1, lo, hi);
                        const unsigned long long w0 = pair2(lo, lo), w1 = pair2(hi, hi);
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(at[y] + ORB_ENT * (1 + v) + c);
                            acc[2 * y][2 * v] = fma2(w0, z.x, acc[2 * y][2 * v]);
                            acc[2 * y][2 * v + 1] = fma2(w0, z.y, acc[2 * y][2 * v + 1]);
                            acc[2 * y + 1][2 * v] = fma2(w1, z.x, acc[2 * y + 1][2 * v]);
                            acc[2 * y + 1][2 * v + 1] = fma2(w1, z.y, acc[2 * y + 1][2 * v + 1]);
                        }
                    }
                }
            }
        }
        if (to == rounds) break;
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            unsigned long long *a = &acc[0][0] + 2 * i;
            ulonglong2 t = make_ulonglong2(a[0], a[1]);
            if (from) {
                const ulonglong2 f = aside[i * AIR_THREADS];
                t = make_ulonglong2(add2(f.x, t.x), add2(f.y, t.y));
            }
            aside[i * AIR_THREADS] = t;
            a[0] = a[1] = 0ull;
        }
    }
    if (rounds > fold) {
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            const ulonglong2 f = aside[i * AIR_THREADS];
            unsigned long long *a = &acc[0][0] + 2 * i;
            a[0] = add2(f.x, a[0]);
            a[1] = add2(f.y, a[1]);
        }
    }
    if (k < n && !stop) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            float *img = s.bwd_part + (size_t)(split * 8 + cls * 4 + f) * n * n;
            const int code = s.orb_frame[cls * 4 + f];
#pragma unroll
            for (int y = 0; y < ORB_ROWS; ++y) {
                if (r + y >= n) continue;
                int ix, iy;
                orb_pixel(code, n, k, r + y, ix, iy);
                const float2 v = unpair2(acc[y][f / 2]);
                img[(size_t)iy * n + ix] = f & 1 ? v.y : v.x;
            }
        }
    }
    unsigned long long zero = 0ull;                      // or NaN, with any sum that is not finite (which is stored again)
#pragma unroll
    for (int i = 0; i < 2 * NF; ++i) zero = fma2((&acc[0][0])[i], 0ull, zero);
    const float2 finite = unpair2(zero);
    if (!(finite.x + finite.y == 0.f)) orb_bwd_hits<NF>(s, cls, split, txy, k, r);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();   // shared memory is reused by the next tile of a persistent block
}

__device__ __forceinline__ void tile_orb_bwd(const SliceDesc &s, int mode, int tile, float *sm) {
    if (s.orb == 8) tile_orb_bwd_nf<8>(s, mode, tile, sm);
    else tile_orb_bwd_nf<4>(s, mode, tile, sm);
}

// ======================================================================
// Fan-beam FBP over orbits of views: the fan angle, bin position, weight and
// distance of a (pixel, base view) pair serve the four or eight pixels and
// views that the scan's symmetries take it to, whose samples lie side by side
// (orbit.h, FbpOrbits).  One thread per pixel and split of the base views; its
// sum for each symmetry goes to an image of its own.
// ======================================================================
__device__ __forceinline__ void tile_fbp_pack(const SliceDesc &s, int tile) {
    const int ld = s.nb + 4;
    const long long i = (long long)tile * AIR_THREADS + threadIdx.x;
    if (i >= (long long)s.fbp_nbase * ld) return;
    const int b = (int)(i / ld), j = (int)(i - (long long)b * ld) - 2;
    const int *__restrict__ view = s.fbp_view + 8 * b;
    const bool in = j >= 0 && j < s.nb;
    for (int p = 0; p < s.fbp_nf / 4; ++p) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int w = __ldg(view + 4 * p + q);
            v[q] = !in || w == FBP_NONE ? 0.f
                                        : ld_data(s.zc + (w < 0 ? (size_t)~w * s.nb + (s.nb - 1 - j) : (size_t)w * s.nb + j));
        }
        s.fbp_q[(size_t)i * (s.fbp_nf / 4) + p] = make_float4(v[0], v[1], v[2], v[3]);
    }
}

template <int NV>
__device__ __forceinline__ void tile_fbp_orb_nv(const SliceDesc &s, int tile) {
    const int n = s.n, nb = s.nb, tpr = (n + SHR_T - 1) / SHR_T, nt = tiles_shr(s);
    const int split = tile / nt, t = tile - split * nt, S = s.fbp_splits;
    // a warp takes 8 x 4 pixels
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ix = (t % tpr) * SHR_T + (w & 1) * 8 + (lane & 7), iy = (t / tpr) * SHR_T + (w >> 1) * 4 + (lane >> 3);
    const float x = (float)ix + 0.5f - s.half_n, y = (float)iy + 0.5f - s.half_n;
    const unsigned long long minus = pair2(-1.f, -1.f);
    unsigned long long acc[2 * NV];
#pragma unroll
    for (int f = 0; f < 2 * NV; ++f) acc[f] = 0ull;
    const ulonglong2 *Q = reinterpret_cast<const ulonglong2 *>(s.fbp_q) + 2 * NV;   // bin 0 of view 0
#pragma unroll 2
    for (int v = split; v < s.fbp_nbase; v += S) {
        const float2 c = __ldg(s.fbp_c + v);
        const float cr = fmaf(c.x, y, -c.y * x);                 // L sin(gamma')
        const float dt = fmaf(c.x, x, fmaf(c.y, y, s.dso_px));   // L cos(gamma') > 0
        const float u = cr / dt;
        const float gp = fabsf(u) <= 0.45f ? atan_series(u) : atan2f(cr, dt);
        // bin position as in tile_fbp
        const float tr = floorf(fmaf(gp, s.inv_dg, s.jmid));
        float wt = fmaf(gp, s.inv_dg, s.jmid - tr);
        wt = fmaf(gp, s.inv_dg_lo, wt);
        const int j0 = (int)tr + (wt < 0.f ? -1 : (wt >= 1.f ? 1 : 0));
        wt = wt < 0.f ? wt + 1.f : (wt >= 1.f ? wt - 1.f : wt);
        const float r2 = __fdividef(1.f, fmaf(cr, cr, dt * dt));
        const unsigned long long w2 = pair2(wt, wt), i2 = pair2(r2, r2);
        // off the detector: onto the zero bins at the row's ends
        const ulonglong2 *q = Q + ((size_t)v * (nb + 4) + min(max(j0, -2), nb)) * NV;
#pragma unroll
        for (int f = 0; f < NV; ++f) {
            const ulonglong2 a = ld_data(q + f), b = ld_data(q + NV + f);
            acc[2 * f] = fma2(i2, fma2(w2, fma2(a.x, minus, b.x), a.x), acc[2 * f]);
            acc[2 * f + 1] = fma2(i2, fma2(w2, fma2(a.y, minus, b.y), a.y), acc[2 * f + 1]);
        }
    }
    if (ix >= n || iy >= n) return;
#pragma unroll
    for (int f = 0; f < 4 * NV; ++f) {
        const int code = s.fbp_code[f];
        const int a = code & ORB_T ? iy : ix, b = code & ORB_T ? ix : iy;
        const int px = code & ORB_FX ? n - 1 - a : a, py = code & ORB_FY ? n - 1 - b : b;
        const float2 r = unpair2(acc[f / 2]);
        s.bwd_part[(size_t)(split * 4 * NV + f) * n * n + (size_t)py * n + px] = f & 1 ? r.y : r.x;
    }
}

__device__ __forceinline__ void tile_fbp_orb(const SliceDesc &s, int tile) {
    if (s.fbp_nf == 8) tile_fbp_orb_nv<2>(s, tile);
    else tile_fbp_orb_nv<1>(s, tile);
}

}  // namespace air
