// frame_kernels.cuh -- the whole path for one frame in one persistent, cooperatively launched
// kernel: Laplacian tiles -> grid barrier -> bilateral tiles (normals, filter, mask, groups,
// tile-local segments) -> grid barrier -> segment merge across tile borders -> grid barrier ->
// labels (and the tri_min filter). Each CTA loops over the tiles of a phase; the grid barrier
// (sync.cuh) orders the phases. Included once per (Laplacian radius, bilateral radius).
//
// Bilateral arithmetic (Eq. 3-6): centroids are stored pre-scaled by sqrt(log2(e) / (2 sigma_c^2))
// and, for unit normals, |n_i - n_j|^2 = 2 - 2 n_i . n_j, so W_c W_s for a pair is one base-2
// exponential of -(|c'_i - c'_j|^2 + a - a n_i . n_j), a = log2(e) / sigma_s^2; a triangle is
// filtered against both triangles of a neighbour quad at once with paired FP32 instructions.
//
// Tiles are staged from HBM with TMA: the input points and the displacements are both AoS
// [H][W][3] floats, seen as 2-D tensors of H rows x 3W floats, so one box per array covers a
// tile plus its halo (points outside the image read as NaN, displacements as 0). The box's x
// coordinate is rounded down to a 16-byte boundary; `delta` is the float offset of the tile's
// first point inside a box row. When TMA cannot be used (W not a multiple of 4, a misaligned
// pointer, or a phase split into several launches' worth of iterations), the same box is
// filled with plain loads, so everything after staging is identical.
#pragma once

#include <math.h>

#include "df32.cuh"
#include "f32x2.cuh"
#include "pl3d_internal.cuh"
#include "sync.cuh"
#include "uf.cuh"

namespace pl3d {
namespace frame {

constexpr int T = kTile;   // tile edge: points (Laplacian) or quads (bilateral)

struct V3 {
    float x, y, z;
};

__device__ __forceinline__ float dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

__device__ __forceinline__ V3 cross(V3 a, V3 b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// Hardware approximations from the PTX ISA: base-2 exponential (ex2(-inf) = +0, subnormal
// results flush to zero) and reciprocal square root (rsqrt(+inf) = 0), both within 2 ulp.
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Floor of x to a multiple of 4 (also for negative x).
__device__ __forceinline__ int floor4(int x) { return x & ~3; }

// ------------------------------------------------------------------------------------ staging

// Fills the box rows x cols (floats) whose top-left element is (x0, y0) of the AoS array
// `src` seen as H rows of 3W floats: TMA when `map` is given, else plain loads. Elements
// outside the array read as `fill`. `bar` completes when the TMA bytes have landed; plain loads have
// landed after cp_async_wait_all() and the caller's barrier.
__device__ __forceinline__ void stage_box(float* dst, const float* src, const CUtensorMap* map, const BoxGeom& b,
                                          int x0, int y0, int H, int W, float fill, uint64_t* bar, int n_tma_boxes,
                                          bool issue_tma) {
    if (map) {
        if (issue_tma && threadIdx.x == 0) {
            if (n_tma_boxes > 0) mbar_arrive_expect_tx(bar, (unsigned)(n_tma_boxes * b.rows * b.cols * 4));
            tma_load_2d(dst, map, x0, y0, bar);
        }
        return;
    }
    // A warp per box row, every copy in flight at once (4 bytes each: the rows of an odd width share
    // no 16-byte alignment with the box). What bounds it is the latency of L2: one load at a time per
    // thread took 9.7 us per bilateral tile of a 243x317 frame, these copies 2.8 us (the frame with all
    // options 53.2 -> 45.9 us). Displacements were
    // written earlier in this launch by other CTAs; the grid barrier's acquire orders these reads.
    const int row_floats = 3 * W, lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < b.rows; r += blockDim.x >> 5) {
        const int gy = y0 + r;
        const bool in = src && gy >= 0 && gy < H;
        const long long g0 = (long long)gy * row_floats + x0;   // (outside the array when x0 < 0: not formed)
        float* const d = dst + r * b.cols;
        for (int x = lane; x < b.cols; x += 32) {
            if (in && x0 + x >= 0 && x0 + x < row_floats) cp_async4(d + x, src + (g0 + x));
            else d[x] = fill;
        }
    }
}

// ------------------------------------------------------------------------------ Laplacian

// A Jacobi iteration of a 5 x 5 or 7 x 7 window updates strips of kLapStrip vertically adjacent
// points per thread (a 3 x 3 window walks, see lap_walk): the
// strip shares the loads of its (kLapStrip + 2R) x (2R + 1) window, and two strip points closer
// than the radius share one weight (w_ij = w_ji, opposite differences).
constexpr int kLapStrip = 4;

// A point as an iteration sees it: input position (invalid -> kInvalidCoord) and displacement.
struct LapPt {
    float x, y, z, dx, dy, dz;
};

// WITH_D = false: the displacement is zero everywhere (the first iteration of the first pass),
// so it is neither loaded nor summed -- the same values as adding zeros.
template <bool WITH_D>
__device__ __forceinline__ LapPt lap_load(const float* V0, const float* D, int o) {
    LapPt p;
    p.x = V0[o];
    p.y = V0[o + 1];
    p.z = V0[o + 2];
    if (WITH_D) {
        p.dx = D[o];
        p.dy = D[o + 1];
        p.dz = D[o + 2];
    } else {
        p.dx = p.dy = p.dz = 0.f;
    }
    return p;
}

struct LapAcc {
    LapPt c;                     // centre
    float sx, sy, sz, ws;        // weighted sums
};

// The Laplacian arithmetic below is written with explicit rounding intrinsics (no contraction
// left to the compiler), so that every kernel that evaluates Eq. 1-2 -- the fused tile passes and
// the single-iteration pass (lap1.cu) -- gives the same bits for the same point.

// Difference q - p of two smoothed points, input and displacement parts subtracted separately.
template <bool WITH_D>
__device__ __forceinline__ void lap_diff(const LapPt& p, const LapPt& q, float& ex, float& ey, float& ez) {
    if (WITH_D) {
        ex = __fadd_rn(__fsub_rn(q.x, p.x), __fsub_rn(q.dx, p.dx));
        ey = __fadd_rn(__fsub_rn(q.y, p.y), __fsub_rn(q.dy, p.dy));
        ez = __fadd_rn(__fsub_rn(q.z, p.z), __fsub_rn(q.dz, p.dz));
    } else {
        ex = __fsub_rn(q.x, p.x);
        ey = __fsub_rn(q.y, p.y);
        ez = __fsub_rn(q.z, p.z);
    }
}

// Eq. 2: w = 1 / |v_j - v|; a neighbour at distance 0 is skipped. An invalid point holds
// kInvalidCoord: the squared distance overflows to +inf and rsqrt(+inf) = 0. A difference and its
// negation give the same weight (w_ij = w_ji).
__device__ __forceinline__ float lap_weight(float ex, float ey, float ez) {
    const float d2 = fmaf(ez, ez, fmaf(ey, ey, __fmul_rn(ex, ex)));
    return d2 > 0.f ? rsqrt_approx(d2) : 0.f;
}

// s += w e for a neighbour difference e and its weight w (the centre's sums of Eq. 1).
__device__ __forceinline__ void lap_accumulate(float& sx, float& sy, float& sz, float& ws, float w, float ex, float ey,
                                               float ez) {
    sx = fmaf(w, ex, sx);
    sy = fmaf(w, ey, sy);
    sz = fmaf(w, ez, sz);
    ws = __fadd_rn(ws, w);
}

template <bool WITH_D>
__device__ __forceinline__ void lap_add(LapAcc& A, const LapPt& q) {
    float ex, ey, ez;
    lap_diff<WITH_D>(A.c, q, ex, ey, ez);
    lap_accumulate(A.sx, A.sy, A.sz, A.ws, lap_weight(ex, ey, ez), ex, ey, ez);
}

// Eq. 1 on the displacement of a centre point: d' = d + (lambda / W) s, or d unchanged (keep).
__device__ __forceinline__ float lap_scale(bool keep, float lambda, float ws) {
    return keep ? 0.f : __fdividef(lambda, ws);
}

// Top-left element (x0, u0) of a Laplacian tile's box in the AoS array seen as H rows of 3W
// floats, and the offset of the tile's first point inside its box row. Tiles are th points high
// (LapPhase::tile_h, 16 to 64) and T = 32 points wide.
struct LapOrigin {
    int u0, c0, x0, dlt;
};

__device__ __forceinline__ LapOrigin lap_origin(int W, int halo, int th, int tile) {
    const int tiles_x = div_up(W, T);
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    LapOrigin o;
    o.u0 = ty * th - halo;
    o.c0 = tx * T - halo;
    o.x0 = floor4(3 * o.c0);
    o.dlt = 3 * o.c0 - o.x0;
    return o;
}

// What a Laplacian tile needs, read from the frame's arguments once per tile: the batch kernel
// keeps them in global memory, where every barrier would make the compiler load them again.
struct LapJob {
    const float* points;
    const float* d_in;             // previous pass's displacement, or nullptr (first pass)
    float* d_out;
    float* export_points;
    int* error;
    int H, W, iters, halo, th;
    BoxGeom box;
    float lambda;
    LapOrigin og;
};

__device__ __forceinline__ LapJob lap_job(const FrameArgs& a, const LapPhase& ph, int tile) {
    LapJob j;
    j.points = a.points;
    j.d_in = ph.d_in;
    j.d_out = ph.d_out;
    j.export_points = ph.export_points;
    j.error = a.error;
    j.H = a.H;
    j.W = a.W;
    j.iters = ph.iters;
    j.halo = ph.halo;
    j.th = ph.tile_h;
    j.box = ph.box;
    j.lambda = a.lambda;
    j.og = lap_origin(j.W, j.halo, j.th, tile);
    return j;
}

// Issues the TMA load of a tile's box of input points into V0 (thread 0; completes on bar). The
// input points are never written inside the launch, so only the box's earlier shared-memory use
// needs ordering -- a global proxy fence would also wait for this thread's own pending stores.
__device__ __forceinline__ void lap_issue(const FrameArgs& a, const LapPhase& ph, const CUtensorMap* map, int tile,
                                          float* V0, uint64_t* bar) {
    if (threadIdx.x != 0) return;
    const LapOrigin o = lap_origin(a.W, ph.halo, ph.tile_h, tile);
    fence_proxy_async_shared();
    mbar_arrive_expect_tx(bar, (unsigned)(ph.box.rows * ph.box.cols * 4));
    tma_load_2d(V0, map, o.x0, o.u0, bar);
}
// One Jacobi iteration with a 3 x 3 window over the region [lo, RH - lo) x [lo, RW - lo) of the staged
// tile: from `cur` (displacements; unused when WITH_D = false) into `nxt`. Each thread walks down
// one column of a segment of rows with a three-row window in registers: a row costs the loads of
// three points, and its S edge is the next row's N edge. What bounds the pass is instruction issue
// and the barrier after each iteration; the segments are cut as evenly as whole rows allow (at most
// 7, 7, 6, 5, 4 rows a thread in five iterations of a 32 x 32 tile), where strips of four rows took
// two rounds of the CTA for four of the five: 256 mixed frames 5723 -> 5656 us, 720x1280 181.6 ->
// 179.8 us.
// Every point takes its window in row-major order, so its sum does not depend on where the segments
// fall (fused or split passes give the same bits).
template <bool WITH_D>
__device__ __forceinline__ void lap_walk(int H, int W, float lambda, int cols, const LapOrigin& og, int RH, int RW,
                                         int lo, const float* V0, const float* cur, float* nxt) {
    const int cw = RW - 2 * lo, nr = RH - 2 * lo;
    const int segs = kThreads / cw;                      // (cw <= 48)
    const int n = (nr + segs - 1) / segs;
    const int seg = (int)threadIdx.x / cw;
    const int c = lo + (int)threadIdx.x - seg * cw;
    int r = lo + seg * n;
    const int end = min(r + n, RH - lo);
    if (seg >= segs || r >= end) return;
    int o = r * cols + og.dlt + 3 * c;
    const int gv = og.c0 + c;
    const bool colpin = gv < 1 || gv >= W - 1;
    struct Row {
        LapPt l, c, r;
    };
    auto load = [&](Row& w, int at) {
        w.l = lap_load<WITH_D>(V0, cur, at - 3);
        w.c = lap_load<WITH_D>(V0, cur, at);
        w.r = lap_load<WITH_D>(V0, cur, at + 3);
    };
    Row A, B, C;
    load(A, o - cols);
    load(B, o);
    float ex, ey, ez;                                    // the edge from the point above to this one
    lap_diff<WITH_D>(A.c, B.c, ex, ey, ez);
    float w = lap_weight(ex, ey, ez);
    auto step = [&](const Row& u, const Row& m, Row& d) {
        load(d, o + cols);
        LapAcc S;
        S.c = m.c;
        S.sx = S.sy = S.sz = S.ws = 0.f;
        lap_add<WITH_D>(S, u.l);
        S.sx = fmaf(-w, ex, S.sx);                       // fma(-w, e) = fma(w, -e)
        S.sy = fmaf(-w, ey, S.sy);
        S.sz = fmaf(-w, ez, S.sz);
        S.ws = __fadd_rn(S.ws, w);
        lap_add<WITH_D>(S, u.r);
        lap_add<WITH_D>(S, m.l);
        lap_add<WITH_D>(S, m.r);
        lap_add<WITH_D>(S, d.l);
        lap_diff<WITH_D>(m.c, d.c, ex, ey, ez);
        w = lap_weight(ex, ey, ez);
        lap_accumulate(S.sx, S.sy, S.sz, S.ws, w, ex, ey, ez);
        lap_add<WITH_D>(S, d.r);
        // Eq. 1 on the displacement; the pinned border ring, invalid points and points without a
        // usable neighbour keep their displacement
        const int gu = og.u0 + r;
        const bool keep = colpin || gu < 1 || gu >= H - 1 || m.c.x == kInvalidCoord || !(S.ws > 0.f);
        const float s = lap_scale(keep, lambda, S.ws);
        nxt[o] = fmaf(s, S.sx, m.c.dx);
        nxt[o + 1] = fmaf(s, S.sy, m.c.dy);
        nxt[o + 2] = fmaf(s, S.sz, m.c.dz);
        o += cols;
        ++r;
    };
    while (true) {
        step(A, B, C);
        if (r == end) break;
        step(B, C, A);
        if (r == end) break;
        step(C, A, B);
        if (r == end) break;
    }
}

// One Jacobi iteration (Eq. 1-2) over the region [lo, RH - lo) x [lo, RW - lo) of the staged
// tile: from `cur` (displacements; unused when WITH_D = false) into `nxt`. A strip that runs
// past the region's last row computes its extra points from the box's spare rows and discards
// them; each kept point's window lies inside the region the previous iteration wrote.
template <int R, bool WITH_D>
__device__ __forceinline__ void lap_iteration(int H, int W, float lambda, int cols, const LapOrigin& og, int RH, int RW,
                                              int lo, const float* V0, const float* cur, float* nxt) {
    constexpr int S = kLapStrip;
    const int cw = RW - 2 * lo;
    const int strips = (RH - 2 * lo + S - 1) / S;
    // (strip, column) of item i = threadIdx.x + k blockDim.x, stepped without a division per item
    const int step_s = (int)blockDim.x / cw, step_c = (int)blockDim.x - step_s * cw;
    int sr = (int)threadIdx.x / cw, cc = (int)threadIdx.x - sr * cw;
    for (; sr < strips; sr += step_s, cc += step_c) {
        if (cc >= cw) {
            cc -= cw;
            ++sr;
            if (sr >= strips) break;
        }
        const int r = lo + S * sr, c = lo + cc;
        const int rows = min(S, RH - lo - r);
        const int o0 = r * cols + og.dlt + 3 * c;
        LapAcc A[S];
#pragma unroll
        for (int k = 0; k < S; ++k) {
            A[k].c = lap_load<WITH_D>(V0, cur, o0 + k * cols);
            A[k].sx = A[k].sy = A[k].sz = A[k].ws = 0.f;
        }
        // Each point takes its window in row-major order whatever its place in the strip, so a
        // point's sum does not depend on how the strips fall (fused or split passes give the
        // same bits). Strip points m < k within the radius share one weight: computed when the
        // traversal reaches row m (where k needs it), kept for row k (where m needs it).
        float pex[S][S], pey[S][S], pez[S][S], pw[S][S];
#pragma unroll
        for (int dr = -R; dr < S + R; ++dr) {
#pragma unroll
            for (int dc = -R; dc <= R; ++dc) {
                if (dc == 0 && dr >= 0 && dr < S) {
                    const int m = dr;   // a strip point
#pragma unroll
                    for (int k = 0; k < S; ++k) {
                        if (k > m && k <= m + R) {
                            lap_diff<WITH_D>(A[m].c, A[k].c, pex[m][k], pey[m][k], pez[m][k]);
                            const float w = lap_weight(pex[m][k], pey[m][k], pez[m][k]);
                            pw[m][k] = w;
                            // fma(-w, e) = fma(w, -e): the same bits as k's own term for m
                            A[k].sx = fmaf(-w, pex[m][k], A[k].sx);
                            A[k].sy = fmaf(-w, pey[m][k], A[k].sy);
                            A[k].sz = fmaf(-w, pez[m][k], A[k].sz);
                            A[k].ws = __fadd_rn(A[k].ws, w);
                        }
                        if (k < m && k >= m - R)
                            lap_accumulate(A[k].sx, A[k].sy, A[k].sz, A[k].ws, pw[k][m], pex[k][m], pey[k][m],
                                           pez[k][m]);
                    }
                    continue;
                }
                const LapPt q = lap_load<WITH_D>(V0, cur, o0 + dr * cols + 3 * dc);
#pragma unroll
                for (int k = 0; k < S; ++k)
                    if (dr - k >= -R && dr - k <= R) lap_add<WITH_D>(A[k], q);
            }
        }
        // Eq. 1 on the displacement; the pinned border ring, invalid points and points without
        // a usable neighbour keep their displacement
        const int gu = og.u0 + r, gv = og.c0 + c;
        const bool colpin = gv < R || gv >= W - R;
#pragma unroll
        for (int k = 0; k < S; ++k) {
            if (k >= rows) break;
            const bool keep = colpin || gu + k < R || gu + k >= H - R || A[k].c.x == kInvalidCoord || !(A[k].ws > 0.f);
            const float s = lap_scale(keep, lambda, A[k].ws);
            const int o = o0 + k * cols;
            nxt[o] = fmaf(s, A[k].sx, A[k].c.dx);
            nxt[o + 1] = fmaf(s, A[k].sy, A[k].c.dy);
            nxt[o + 2] = fmaf(s, A[k].sz, A[k].c.dz);
        }
    }
}

// One Laplacian tile: th x T output points, `iters` fused Jacobi iterations (Eq. 1-2). The input
// box is in V0, either already issued by TMA on `bar` (tma = true: wait for it) or to be loaded
// here with plain loads. Da, Db: the displacement ping-pong (a single-iteration first pass reads
// no displacement and writes only Db; then Da may alias Db). The box has kLapStrip - 1 spare rows
// below the tile's halo for the strips that run past the region.
template <int R>
__device__ void lap_tile(const LapJob& j, float* V0, float* Da, float* Db, bool tma, uint64_t* bar, unsigned parity) {
    const int H = j.H, W = j.W, h = j.halo, th = j.th;
    const int RH = th + 2 * h, RW = T + 2 * h;
    const BoxGeom b = j.box;                   // rows = RH + kLapStrip - 1, cols >= 3 RW + delta
    const LapOrigin og = j.og;
    const int u0 = og.u0, c0 = og.c0, dlt = og.dlt;
    const bool first = j.d_in == nullptr;

    if (!tma) stage_box(V0, j.points, nullptr, b, og.x0, u0, H, W, NAN, bar, 0, false);
    if (!first) stage_box(Da, j.d_in, nullptr, b, og.x0, u0, H, W, 0.f, bar, 0, false);
    if (!tma || !first) cp_async_wait_all();
    if (tma) mbar_wait_bounded(bar, parity, j.error);   // the caller flips its parity
    __syncthreads();
    // invalid points (non-finite or out of range, including outside the image) become the
    // finite sentinel with zero displacement; the first pass reads no displacement, and without
    // iterations (lap_iters = 0) its output is the zero displacement itself
    const bool zero_all = first && j.iters == 0;
    // (row, column) of item i = threadIdx.x + k blockDim.x, stepped without a division per item;
    // four items per round, their loads issued together
    {
        constexpr int U = 4;
        const int step_r = blockDim.x / RW, step_c = blockDim.x - step_r * RW;
        int r = threadIdx.x / RW, c = threadIdx.x - r * RW;
        for (int i0 = threadIdx.x; i0 < RH * RW; i0 += U * blockDim.x) {
            int o[U];
            float x[U], y[U], z[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                o[u] = r * b.cols + dlt + 3 * c;
                r += step_r;
                c += step_c;
                if (c >= RW) {
                    c -= RW;
                    ++r;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = i0 + u * (int)blockDim.x < RH * RW;
                x[u] = in ? V0[o[u]] : 0.f;
                y[u] = in ? V0[o[u] + 1] : 0.f;
                z[u] = in ? V0[o[u] + 2] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (i0 + u * (int)blockDim.x >= RH * RW) break;
                const bool bad = !point_valid(x[u], y[u], z[u]);
                if (bad) V0[o[u]] = V0[o[u] + 1] = V0[o[u] + 2] = kInvalidCoord;
                if ((bad && !first) || zero_all) Da[o[u]] = Da[o[u] + 1] = Da[o[u] + 2] = 0.f;
            }
        }
    }
    __syncthreads();

    float* cur = Da;
    float* nxt = Db;
    for (int t = 1; t <= j.iters; ++t) {
        if constexpr (R == 1) {
            if (first && t == 1) lap_walk<false>(H, W, j.lambda, b.cols, og, RH, RW, 1, V0, cur, nxt);
            else lap_walk<true>(H, W, j.lambda, b.cols, og, RH, RW, t, V0, cur, nxt);
        } else {
            if (first && t == 1) lap_iteration<R, false>(H, W, j.lambda, b.cols, og, RH, RW, R, V0, cur, nxt);
            else lap_iteration<R, true>(H, W, j.lambda, b.cols, og, RH, RW, t * R, V0, cur, nxt);
        }
        __syncthreads();
        float* tmp = cur;
        cur = nxt;
        nxt = tmp;
    }

    // The tile's own points: displacement out (AoS, row-contiguous), optional export. With
    // W % 4 == 0 a tile row (96 floats) starts 16-byte aligned both here (dlt + 3h = 0 mod 4, the
    // box width a multiple of 4) and in the array (3W and 96 tx multiples of 4): float4 stores.
    if ((W & 3) == 0) {
        // thread -> tile rows threadIdx.x / 8 + 32 k and float4 columns (threadIdx.x % 8) + 8 m
        static_assert(kThreads == 8 * T && (3 * T / 4) % 8 == 0, "one tile row per 8 threads");
        const int q = threadIdx.x & 7;
        const int gv3 = 3 * (c0 + h) + 4 * q;
        for (int rr = threadIdx.x >> 3; rr < th; rr += kThreads / 8) {
            const int gu = u0 + h + rr;
            if (gu >= H) break;
            const float* src = cur + (h + rr) * b.cols + dlt + 3 * h + 4 * q;
            float* dst = j.d_out + (size_t)gu * 3 * W + gv3;
#pragma unroll
            for (int m = 0; m < 3 * T / 32; ++m)
                if (gv3 + 32 * m < 3 * W)   // then gv3 + 32 m + 3 < 3W as well
                    *reinterpret_cast<float4*>(dst + 32 * m) = *reinterpret_cast<const float4*>(src + 32 * m);
        }
    }
    if ((W & 3) != 0 || j.export_points) {
        for (int e = threadIdx.x; e < th * 3 * T; e += blockDim.x) {
            const int r = e / (3 * T), f = e - r * (3 * T);
            const int gu = u0 + h + r, gv3 = 3 * (c0 + h) + f;
            if (gu >= H || gv3 >= 3 * W) continue;
            const int o = (h + r) * b.cols + dlt + 3 * h + f;
            const size_t g = (size_t)gu * 3 * W + gv3;
            const float d = cur[o];
            if ((W & 3) != 0) j.d_out[g] = d;
            if (j.export_points) {
                const int pt = o - (f % 3);
                j.export_points[g] = V0[pt] != kInvalidCoord ? __fadd_rn(V0[o], d) : NAN;
            }
        }
    }
    __syncthreads();
}
// ------------------------------------------------------------------------------ bilateral

// A staged point: input position and displacement.
struct SP {
    float x, y, z, dx, dy, dz;
};

__device__ __forceinline__ SP load_sp(const float* V0, const float* D, int o) {
    return {V0[o], V0[o + 1], V0[o + 2], D[o], D[o + 1], D[o + 2]};
}

struct PairEdge {
    F2 x, y, z;
};

__device__ __forceinline__ PairEdge pair_edge(const SP& a, const SP& b) {
    return {pair_diff(a.x, a.dx, b.x, b.dx), pair_diff(a.y, a.dy, b.y, b.dy), pair_diff(a.z, a.dz, b.z, b.dz)};
}

__device__ __forceinline__ V3 pair_cross(const PairEdge& e1, const PairEdge& e2) {
    return {pair_sub_round(pair_mul(e1.y, e2.z), pair_mul(e1.z, e2.y)),
            pair_sub_round(pair_mul(e1.z, e2.x), pair_mul(e1.x, e2.z)),
            pair_sub_round(pair_mul(e1.x, e2.y), pair_mul(e1.y, e2.x))};
}

// Edge b - a in FP32 and the size of what was summed to form it (for the error bound).
struct FastEdge {
    V3 e;
    float m;    // sum over coordinates of the differences |v0_b - v0_a|, |d_b - d_a| that were rounded
    float l1;   // sum over coordinates of |e|
};

// |q - p| where the difference q - p was rounded, 0 where it is exact: a computed difference
// below both operands in magnitude proves that q lies within a factor 2 of p (rounding is
// monotonic, so the exact difference is below them too), and then q - p is exact (Sterbenz).
__device__ __forceinline__ float rounded_part(float diff, float p, float q) {
    const float ad = fabsf(diff);
    return ad < fminf(fabsf(p), fabsf(q)) ? 0.f : ad;
}

// Edge b - a in FP32 (the same value as fast_edge(a, b).e).
__device__ __forceinline__ V3 edge_of(const SP& a, const SP& b) {
    return {(b.x - a.x) + (b.dx - a.dx), (b.y - a.y) + (b.dy - a.dy), (b.z - a.z) + (b.dz - a.dz)};
}

// Dominant normals up to this count are held in registers by the group assignment.
constexpr int kRegGroups = 4;

__device__ __forceinline__ FastEdge fast_edge(const SP& a, const SP& b) {
    const float ax = b.x - a.x, ay = b.y - a.y, az = b.z - a.z;
    const float dx = b.dx - a.dx, dy = b.dy - a.dy, dz = b.dz - a.dz;
    FastEdge f;
    f.e = {ax + dx, ay + dy, az + dz};
    // (the displacements' differences are counted as rounded: they are rarely within a factor 2)
    f.m = (rounded_part(ax, a.x, b.x) + fabsf(dx)) + (rounded_part(ay, a.y, b.y) + fabsf(dy)) +
          (rounded_part(az, a.z, b.z) + fabsf(dz));
    f.l1 = fabsf(f.e.x) + fabsf(f.e.y) + fabsf(f.e.z);
    return f;
}

// Error of the FP32 normal. Each edge coordinate is off by at most u (m_c + |e_c|), u = 2^-24,
// m_c the rounded differences summed into it; the cross product adds u per product and u for
// the difference. So |d cr|_1 <= u (m1 |e2|_1 + |e1|_1 m2 + 4 |e1|_1 |e2|_1), and the angle is
// off by at most sqrt(3) |d cr|_1 / |cr|_1. Accept the FP32 normal when that bound is below
// sqrt(3) 64 u = 6.6e-6 rad (15 times inside the 1e-4 rad tolerance), otherwise recompute it
// from exact pairs.
__device__ __forceinline__ bool fast_cross_ok(const FastEdge& e1, const FastEdge& e2, V3 cr) {
    const float crl1 = fabsf(cr.x) + fabsf(cr.y) + fabsf(cr.z);
    return e1.m * e2.l1 + e1.l1 * e2.m + 4.f * (e1.l1 * e2.l1) <= 64.f * crl1;
}

__device__ __forceinline__ V3 centroid3(const SP& a, const SP& b, const SP& c) {
    const float k = 1.f / 3.f;
    return {((a.x + b.x + c.x) + (a.dx + b.dx + c.dx)) * k, ((a.y + b.y + c.y) + (a.dy + b.dy + c.dy)) * k,
            ((a.z + b.z + c.z) + (a.dz + b.dz + c.dz)) * k};
}

// Per-quad records in shared memory: 6 floats interleaving the quad's two triangles,
// {x0, x1, y0, y1, z0, z1}, so that each 64-bit load yields one coordinate of both triangles as
// a packed pair (f32x2.cuh).
__device__ __forceinline__ void load_quad(const float* A, int q, V3& t0, V3& t1) {
    const float2* p = reinterpret_cast<const float2*>(A) + 3 * q;
    const float2 x = p[0], y = p[1], z = p[2];
    t0 = {x.x, y.x, z.x};
    t1 = {x.y, y.y, z.y};
}

__device__ __forceinline__ void load_quad2(const float* A, int q, f2& x, f2& y, f2& z) {
    const f2* p = reinterpret_cast<const f2*>(A) + 3 * q;
    x = p[0];
    y = p[1];
    z = p[2];
}

__device__ __forceinline__ void store_quad(float* A, int q, V3 t0, V3 t1) {
    float2* p = reinterpret_cast<float2*>(A) + 3 * q;
    p[0] = make_float2(t0.x, t1.x);
    p[1] = make_float2(t0.y, t1.y);
    p[2] = make_float2(t0.z, t1.z);
}

__device__ __forceinline__ bool has_normal(V3 n) { return n.x != 0.f || n.y != 0.f || n.z != 0.f; }

__device__ __forceinline__ V3 finish_normal(V3 s, V3 own) {
    const float l2 = dot(s, s);
    if (!has_normal(own) || !(l2 > 0.f)) return own;
    const float inv = rsqrtf(l2);
    return {s.x * inv, s.y * inv, s.z * inv};
}

// One own triangle i against the two triangles of a neighbour quad at once, in packed pairs:
//   W_j = ex2(-(|c'_i - c'_j|^2 + a - a n_i . n_j)),   s_i += W_j n_j   (j = both triangles)
// The state holds i's centroid and -a n_i broadcast to both halves, and the two halves of the
// running sum (added together at the end).
struct OwnTri {
    f2 cx, cy, cz;
    f2 px, py, pz;
    f2 sx, sy, sz;
};

__device__ __forceinline__ void own_begin(OwnTri& o, V3 c, V3 n, float a) {
    o.cx = bc(c.x);
    o.cy = bc(c.y);
    o.cz = bc(c.z);
    o.px = bc(-a * n.x);
    o.py = bc(-a * n.y);
    o.pz = bc(-a * n.z);
    o.sx = o.sy = o.sz = 0ull;
}

__device__ __forceinline__ f2 own_weights(const OwnTri& o, f2 a2, f2 cx, f2 cy, f2 cz, f2 nx, f2 ny, f2 nz) {
    const f2 dx = sub2(o.cx, cx), dy = sub2(o.cy, cy), dz = sub2(o.cz, cz);
    f2 ne = fma2(o.px, nx, a2);
    ne = fma2(o.py, ny, ne);
    ne = fma2(o.pz, nz, ne);
    ne = fma2(dz, dz, ne);
    ne = fma2(dy, dy, ne);
    ne = fma2(dx, dx, ne);
    float e0, e1;
    upk(ne, e0, e1);
    return pk(ex2(-e0), ex2(-e1));
}

__device__ __forceinline__ void own_add(OwnTri& o, f2 w, f2 nx, f2 ny, f2 nz) {
    o.sx = fma2(w, nx, o.sx);
    o.sy = fma2(w, ny, o.sy);
    o.sz = fma2(w, nz, o.sz);
}

__device__ __forceinline__ V3 own_sum(const OwnTri& o) {
    float a, b, c, d, e, f;
    upk(o.sx, a, b);
    upk(o.sy, c, d);
    upk(o.sz, e, f);
    return {a + b, c + d, e + f};
}

// A quad's two triangles: their own quad first. Each triangle's weight with itself is exactly 1, so what
// is left is one weight of each with the other, in scalar steps that share the difference of the
// centroids (the same roundings as a half of own_weights): 21 FP32 cycles instead of 48 of a quad's 432,
// a packed instruction taking two. 480x640 frame 64.4 -> 64.0 us. In the batch kernel the iterations' own
// CTA time rose with it (256 frames 383 -> 391 ms) while the bilateral phase took 3392 -> 3364 us.
struct QuadAcc {
    OwnTri t0, t1;
    V3 n0, n1;   // current normals (a triangle without a normal keeps n = 0)
};

__device__ __forceinline__ void quad_begin(QuadAcc& A, const float* Cq, const float* cur, int q, float a) {
    f2 cx, cy, cz, nx, ny, nz;
    load_quad2(Cq, q, cx, cy, cz);
    load_quad2(cur, q, nx, ny, nz);
    float c0x, c1x, c0y, c1y, c0z, c1z, n0x, n1x, n0y, n1y, n0z, n1z;
    upk(cx, c0x, c1x);
    upk(cy, c0y, c1y);
    upk(cz, c0z, c1z);
    upk(nx, n0x, n1x);
    upk(ny, n0y, n1y);
    upk(nz, n0z, n1z);
    A.n0 = {n0x, n0y, n0z};
    A.n1 = {n1x, n1y, n1z};
    own_begin(A.t0, {c0x, c0y, c0z}, A.n0, a);
    own_begin(A.t1, {c1x, c1y, c1z}, A.n1, a);
    const float dx = c0x - c1x, dy = c0y - c1y, dz = c0z - c1z;
    float e0 = fmaf(lo_of(A.t0.px), n1x, a), e1 = fmaf(lo_of(A.t1.px), n0x, a);
    e0 = fmaf(lo_of(A.t0.py), n1y, e0), e1 = fmaf(lo_of(A.t1.py), n0y, e1);
    e0 = fmaf(lo_of(A.t0.pz), n1z, e0), e1 = fmaf(lo_of(A.t1.pz), n0z, e1);
    e0 = fmaf(dz, dz, e0), e1 = fmaf(dz, dz, e1);
    e0 = fmaf(dy, dy, e0), e1 = fmaf(dy, dy, e1);
    e0 = fmaf(dx, dx, e0), e1 = fmaf(dx, dx, e1);
    const float w0 = ex2(-e0), w1 = ex2(-e1);
    A.t0.sx = pk(n0x, w0 * n1x), A.t0.sy = pk(n0y, w0 * n1y), A.t0.sz = pk(n0z, w0 * n1z);
    A.t1.sx = pk(w1 * n0x, n1x), A.t1.sy = pk(w1 * n0y, n1y), A.t1.sz = pk(w1 * n0z, n1z);
}

__device__ __forceinline__ void quad_neighbour(QuadAcc& A, f2 a2, f2 cx, f2 cy, f2 cz, f2 nx, f2 ny, f2 nz) {
    own_add(A.t0, own_weights(A.t0, a2, cx, cy, cz, nx, ny, nz), nx, ny, nz);
    own_add(A.t1, own_weights(A.t1, a2, cx, cy, cz, nx, ny, nz), nx, ny, nz);
}

// One bilateral tile: TH x T quads (TH = a.bil_th rows of T = 32, so that a warp spans a tile row);
// geometry, `ph.iters` fused iterations (Eq. 3-6), then either
// the carry for the next chunk or mask, normals, groups (Algorithm 4) and the tile-local
// segments (Algorithm 5); with JOIN (the single-frame kernel) also the joins across the tile's
// borders with finished neighbours.
// Shared-memory header of the persistent kernels (128 bytes before the tiles' buffers): the staging
// mbarriers from byte 0, the bilateral tile's deferred-normal count at byte 64, the grid barrier's
// generation at byte 68, and for the stage
// timing the last stamp at byte 72 and the stage totals' address (or nullptr) at byte 80.
constexpr int kHdrExact = 64, kHdrGen = 68, kHdrStamp = 72, kHdrStages = 80;

// The borders of a finished tile's segments with its neighbours' (defined with the merge phase).
__device__ __forceinline__ void join_tile_borders(const FrameArgs& a, int tile);

__device__ __forceinline__ void set_stage_timing(uint64_t* bar, unsigned long long* sns) {
    if (threadIdx.x == 0) *reinterpret_cast<unsigned long long**>(reinterpret_cast<unsigned char*>(bar) + kHdrStages) = sns;
}

// With stage timing on (set_stage_timing), thread 0 adds the tile's time in each stage -- staging,
// geometry, iterations, finish (groups and outputs, or the carry), tile labels -- to the totals
// (%globaltimer nanoseconds summed over tiles: CTA time, not wall time). The state lives in the
// shared-memory header, so that it holds no register across the tile.
__device__ __forceinline__ void stage_mark(uint64_t* bar, int k) {
    if (threadIdx.x == 0) {
        unsigned char* hdr = reinterpret_cast<unsigned char*>(bar);
        unsigned long long* sns = *reinterpret_cast<unsigned long long**>(hdr + kHdrStages);
        if (sns) {
            unsigned long long* last = reinterpret_cast<unsigned long long*>(hdr + kHdrStamp);
            const unsigned long long t = global_ns();
            if (k >= 0) atomicAdd(sns + k, t - *last);
            *last = t;
        }
    }
}

template <int R, bool JOIN>
__device__ void bil_tile(const FrameArgs& a, const BilPhase& ph, int tile, float* smem, uint64_t* bar,
                         unsigned& parity) {
    stage_mark(bar, -1);
    // the frame's arguments, read once (the batch kernel keeps them in global memory, where every
    // barrier and every global store would make the compiler load them again)
    const int H = a.H, W = a.W, Hq = H - 1, Wq = W - 1;
    const int h = ph.halo, iters = ph.iters;
    const bool first = ph.first != 0, last = ph.last != 0;
    const float* const carry_in = ph.carry_in;
    float* const carry_out = ph.carry_out;
    int* const error = a.error;
    const float max_edge2 = a.max_edge2;
    const int TH = a.bil_th;
    const int RQH = TH + 2 * h, RQW = T + 2 * h;         // staged quads
    const int nq = RQH * RQW;
    const int nqs = nq + RQW;                            // one spare row of quads
    const BoxGeom b = ph.box;                            // rows = RQH + 1 points, cols >= 3 (RQW + 1) + delta
    const int bsz = align_floats(b.rows * b.cols);
    float* Cq = smem;                                    // [nqs][6] scaled centroids
    float* Na = Cq + align_floats(6 * nqs);              // [nqs][6] normals
    float* X = Na + align_floats(6 * nqs);               // Nb, or the two staged boxes before the iterations
    float* Nb = X;
    float* V0 = X;
    float* Dp = X + bsz;
    const int xw = max(align_floats(6 * nqs), 2 * bsz);
    uint8_t* Mk = reinterpret_cast<uint8_t*>(X + xw);    // [TH*T*2] own masks (room for T*T*2)
    uint16_t* ex_list = reinterpret_cast<uint16_t*>(Mk + 2 * T * T);   // [nq] deferred exact normals: quad | which
    constexpr int kDefer0 = 1 << 12, kDefer1 = 1 << 13;
    static_assert((T + 2 * kBilMaxHalo) * (T + 2 * kBilMaxHalo) <= kDefer0, "staged quads in 12 bits");
    const int tiles_x = div_up(Wq, T);
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const int qu0 = ty * TH - h, qv0 = tx * T - h;
    const int x0 = floor4(3 * qv0);
    const int dlt = 3 * qv0 - x0;
    const float cs = a.c_scale;

    const CUtensorMap* mp = ph.use_tma ? &a.tm_pts_bil : nullptr;
    const CUtensorMap* md = ph.use_tma ? &a.tm_disp_bil : nullptr;
    if (mp && threadIdx.x == 0) fence_proxy_async_all();
    stage_box(V0, a.points, mp, b, x0, qu0, H, W, NAN, bar, 2, true);
    stage_box(Dp, a.disp, md, b, x0, qu0, H, W, 0.f, bar, 0, true);
    if (mp) {
        mbar_wait_bounded(bar, parity, error);
        parity ^= 1u;
    } else {
        cp_async_wait_all();
    }
    __syncthreads();
    int* n_exact = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(bar) + kHdrExact);   // in the smem header
    if (threadIdx.x == 0) *n_exact = 0;
    {
        // (row, column) of point i = threadIdx.x + k blockDim.x, stepped without a division; four
        // points per round, their loads issued together
        constexpr int U = 4;
        const int PW = RQW + 1, NP = (RQH + 1) * PW;
        const int step_r = blockDim.x / PW, step_c = blockDim.x - step_r * PW;
        int r = threadIdx.x / PW, c = threadIdx.x - r * PW;
        for (int i0 = threadIdx.x; i0 < NP; i0 += U * blockDim.x) {
            int o[U];
            float x[U], y[U], z[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                o[u] = r * b.cols + dlt + 3 * c;
                r += step_r;
                c += step_c;
                if (c >= PW) {
                    c -= PW;
                    ++r;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = i0 + u * (int)blockDim.x < NP;
                x[u] = in ? V0[o[u]] : 0.f;
                y[u] = in ? V0[o[u] + 1] : 0.f;
                z[u] = in ? V0[o[u] + 2] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (i0 + u * (int)blockDim.x >= NP) break;
                if (!point_valid(x[u], y[u], z[u])) {
                    V0[o[u]] = V0[o[u] + 1] = V0[o[u] + 2] = NAN;
                    Dp[o[u]] = Dp[o[u] + 1] = Dp[o[u] + 2] = 0.f;
                }
            }
        }
    }
    __syncthreads();
    stage_mark(bar, 0);

    // Centroids and normals of every staged triangle; masks of the tile's own quads. A normal
    // whose FP32 error bound fails is deferred: its quad goes on a list (with room for every staged
    // quad) that a second loop recomputes from exact pairs with every lane busy. On a LiDAR scan a fifth
    // of the quads are; a list of 256 with a divergent path past it took 33.4 us for a 64x1024 frame
    // and 868 us for 64 frames at one iteration, this one 33.1 and 863 us.
    auto exact_normals = [&](const SP& p1, const SP& p2, const SP& p3, const SP& p4, bool do0, bool do1, V3& n0,
                             V3& n1) {
        const PairEdge pd = pair_edge(p3, p1);
        if (do0) n0 = pair_cross(pair_edge(p3, p2), pd);
        if (do1) {
            const PairEdge pdn = {{-pd.x.h, -pd.x.l}, {-pd.y.h, -pd.y.l}, {-pd.z.h, -pd.z.l}};
            n1 = pair_cross(pair_edge(p1, p4), pdn);
        }
    };
    auto unit_or_none = [](V3 cr, bool valid) {
        const float len2 = dot(cr, cr);
        V3 n = {0.f, 0.f, 0.f};
        if (valid && len2 > kDegenerateLen2) {
            const float inv = rsqrtf(len2);
            n = {cr.x * inv, cr.y * inv, cr.z * inv};
        }
        return n;
    };
    auto scaled_centroid = [&](const SP& va, const SP& vb, const SP& vc, V3 n) {
        V3 c = {kAbsentCentroid, kAbsentCentroid, kAbsentCentroid};
        if (has_normal(n)) {
            const V3 m = centroid3(va, vb, vc);
            c = {m.x * cs, m.y * cs, m.z * cs};
        }
        return c;
    };
    // (row, column) of quad q = threadIdx.x + k blockDim.x, stepped without a division per quad
    const int gstep_r = blockDim.x / RQW, gstep_c = blockDim.x - gstep_r * RQW;
    int g_qr = threadIdx.x / RQW, g_qc = threadIdx.x - g_qr * RQW;
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
        const int qr = g_qr, qc = g_qc;
        g_qr += gstep_r;
        g_qc += gstep_c;
        if (g_qc >= RQW) {
            g_qc -= RQW;
            ++g_qr;
        }
        const int gu = qu0 + qr, gv = qv0 + qc;
        const bool exists = gu >= 0 && gu < Hq && gv >= 0 && gv < Wq;
        const int o1 = qr * b.cols + dlt + 3 * qc;
        const SP p1 = load_sp(V0, Dp, o1), p2 = load_sp(V0, Dp, o1 + 3);
        const SP p3 = load_sp(V0, Dp, o1 + b.cols + 3), p4 = load_sp(V0, Dp, o1 + b.cols);
        const bool own = last && qr >= h && qr < h + TH && qc >= h && qc < h + T;
        const bool v1 = p1.x == p1.x, v2 = p2.x == p2.x, v3 = p3.x == p3.x, v4 = p4.x == p4.x;
        const bool valid0 = exists && v1 && v2 && v3;                            // Algorithm 1
        const bool valid1 = exists && v1 && v3 && v4;
        V3 nn[2] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
        // first = {p3, p2, p1}: (p2 - p3) x (p1 - p3);  second = {p1, p4, p3}: (p4 - p1) x (p3 - p1)
        const FastEdge er = fast_edge(p3, p2), ed = fast_edge(p3, p1), el = fast_edge(p1, p4);
        if (first) {
            const FastEdge edn = {{-ed.e.x, -ed.e.y, -ed.e.z}, ed.m, ed.l1};
            V3 cr0 = cross(er.e, ed.e), cr1 = cross(el.e, edn.e);
            const bool exact0 = valid0 && !fast_cross_ok(er, ed, cr0);
            const bool exact1 = valid1 && !fast_cross_ok(el, edn, cr1);
            if (exact0 || exact1)
                ex_list[atomicAdd(n_exact, 1)] = (uint16_t)(q | (exact0 ? kDefer0 : 0) | (exact1 ? kDefer1 : 0));
            // a deferred quad's records are written again by the second loop
            nn[0] = unit_or_none(cr0, valid0 && !exact0);
            nn[1] = unit_or_none(cr1, valid1 && !exact1);
        } else {
            const bool vk[2] = {valid0, valid1};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!vk[k]) continue;
                const size_t gid = 2 * ((size_t)gu * Wq + gv) + k;
                const float nx = __ldcg(carry_in + 3 * gid);   // written by the previous pass
                if (nx == nx) nn[k] = {nx, __ldcg(carry_in + 3 * gid + 1), __ldcg(carry_in + 3 * gid + 2)};
            }
        }
        const V3 cc0 = scaled_centroid(p3, p2, p1, nn[0]), cc1 = scaled_centroid(p1, p4, p3, nn[1]);
        if (own) {                                                               // Algorithm 4, l_max
            // FP32 edges: ~1e-7 relative error, far inside the 1e-5 m band where FP32 and FP64
            // may disagree
            const V3 et = edge_of(p2, p1), eb = edge_of(p4, p3);
            const float d2 = dot(ed.e, ed.e);
            const float l0 = fmaxf(d2, fmaxf(dot(er.e, er.e), dot(et, et)));
            const float l1 = fmaxf(d2, fmaxf(dot(el.e, el.e), dot(eb, eb)));
            const int t = 2 * ((qr - h) * T + (qc - h));
            Mk[t] = (valid0 && l0 <= max_edge2) ? 1 : 0;
            Mk[t + 1] = (valid1 && l1 <= max_edge2) ? 1 : 0;
        }
        store_quad(Cq, q, cc0, cc1);
        store_quad(Na, q, nn[0], nn[1]);
    }
    __syncthreads();
    // the deferred normals (and their centroids), one quad per lane
    const int n_ex = *n_exact;
    for (int i = threadIdx.x; i < n_ex; i += blockDim.x) {
        const int e = ex_list[i];
        const int q = e & (kDefer0 - 1);
        const bool do0 = e & kDefer0, do1 = e & kDefer1;
        const int qr = q / RQW, qc = q - qr * RQW;
        const int o1 = qr * b.cols + dlt + 3 * qc;
        const SP p1 = load_sp(V0, Dp, o1), p2 = load_sp(V0, Dp, o1 + 3);
        const SP p3 = load_sp(V0, Dp, o1 + b.cols + 3), p4 = load_sp(V0, Dp, o1 + b.cols);
        V3 cr0 = {0.f, 0.f, 0.f}, cr1 = cr0;
        exact_normals(p1, p2, p3, p4, do0, do1, cr0, cr1);
        // the flagged triangles are valid (the flag requires it); write only their slots
        float* cq = Cq + 6 * q;
        float* na = Na + 6 * q;
        if (do0) {
            const V3 n = unit_or_none(cr0, true), c = scaled_centroid(p3, p2, p1, n);
            na[0] = n.x, na[2] = n.y, na[4] = n.z;
            cq[0] = c.x, cq[2] = c.y, cq[4] = c.z;
        }
        if (do1) {
            const V3 n = unit_or_none(cr1, true), c = scaled_centroid(p1, p4, p3, n);
            na[1] = n.x, na[3] = n.y, na[5] = n.z;
            cq[1] = c.x, cq[3] = c.y, cq[5] = c.z;
        }
    }
    __syncthreads();   // the staged boxes are dead from here on; Nb reuses their space
    stage_mark(bar, 1);

    // Fused bilateral iterations: each work item is a vertical pair of quads.
    float* cur = Na;
    float* nxt = Nb;
    const float an = a.a_norm;
    const f2 a2 = bc(an);
    for (int it = 1; it <= iters; ++it) {
        const int lo = it * R;
        const int ch = RQH - 2 * lo, cw = RQW - 2 * lo;
        const int strips = (ch + 1) >> 1;
        for (int i = threadIdx.x; i < strips * cw; i += blockDim.x) {
            const int sr = i / cw;
            const int qr = lo + 2 * sr, qc = lo + (i - sr * cw);
            const bool two = qr + 1 < RQH - lo;
            const int qA = qr * RQW + qc, qB = qA + RQW;
            QuadAcc A, B;
            quad_begin(A, Cq, cur, qA, an);
            quad_begin(B, Cq, cur, qB, an);
#pragma unroll
            for (int dr = -R; dr <= R + 1; ++dr) {
#pragma unroll
                for (int dc = -R; dc <= R; ++dc) {
                    const bool forA = dr <= R && !(dr == 0 && dc == 0);
                    const bool forB = dr >= 1 - R && !(dr == 1 && dc == 0);
                    const int qj = qA + dr * RQW + dc;
                    f2 cx, cy, cz, nx, ny, nz;
                    load_quad2(Cq, qj, cx, cy, cz);
                    load_quad2(cur, qj, nx, ny, nz);
                    if (forA) quad_neighbour(A, a2, cx, cy, cz, nx, ny, nz);
                    if (forB) quad_neighbour(B, a2, cx, cy, cz, nx, ny, nz);
                }
            }
            store_quad(nxt, qA, finish_normal(own_sum(A.t0), A.n0), finish_normal(own_sum(A.t1), A.n1));
            if (two) store_quad(nxt, qB, finish_normal(own_sum(B.t0), B.n0), finish_normal(own_sum(B.t1), B.n1));
        }
        __syncthreads();
        float* tmp = cur;
        cur = nxt;
        nxt = tmp;
    }
    stage_mark(bar, 2);

    if (!last) {
        for (int i = threadIdx.x; i < TH * T; i += blockDim.x) {
            const int r = i / T, c = i - r * T;
            const int gu = ty * TH + r, gv = tx * T + c;
            if (gu >= Hq || gv >= Wq) continue;
            V3 n[2];
            load_quad(cur, (r + h) * RQW + (c + h), n[0], n[1]);
            const size_t gid0 = 2 * ((size_t)gu * Wq + gv);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool has = has_normal(n[k]);
                float* o = carry_out + 3 * (gid0 + k);
                o[0] = has ? n[k].x : NAN;
                o[1] = has ? n[k].y : NAN;
                o[2] = has ? n[k].z : NAN;
            }
        }
        __syncthreads();
        stage_mark(bar, 3);
        return;
    }

    // Outputs and segments of the tile, TH / 8 consecutive quad rows per warp with lane = column, so
    // that a warp's groups, runs and links stay in its registers and shared memory holds only the
    // runs' parents. What bounds it is latency: short dependent steps on two CTAs per SM. The label
    // stage took 7.4 us of a tile's 26 us in a 256-frame batch with prefix-max shuffles for the
    // runs, a compare-and-swap union per linked pair of runs and a walk per run, and takes 5.5 us
    // with ballots and rounds over all links at once, 4.7 us with the links inside a warp made on the
    // way down its rows (batch 5869 -> 5716 us at the first; 64 frames at one
    // iteration 916 -> 882 us; a 480x640 frame 69.6 -> 68.1 us).
    //
    // free after the last iteration (>= 6 * nqs floats, nqs >= (TH + 1) T): parents of the run
    // representatives [2 TH T], and each warp's last row for the warp below it: the representative
    // (-1 without a group) and group of second(v), and the row's two link masks
    int32_t* Lp = reinterpret_cast<int32_t*>(nxt);
    int32_t* UpRep = Lp + 2 * TH * T;                    // [kThreads / 32][T]
    int32_t* UpGrp = UpRep + kThreads;                   // [kThreads / 32][T]
    unsigned* UpMask = reinterpret_cast<unsigned*>(UpGrp + kThreads);   // [kThreads / 32][2]
    constexpr int kRows = T / (kThreads / 32);           // most rows of a warp
    constexpr unsigned kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = TH / (kThreads / 32), r0 = warp * rows;
    uint8_t* const out_mask = a.out_mask;
    float* const out_normals = a.out_normals;
    uint8_t* const out_groups = a.groups;
    int32_t* const sizes = a.sizes;
    const float min_dot = a.min_dot;
    // up to kRegGroups dominant normals held in registers; more are read from the arguments
    const int K = a.nd.K;
    const float* const ndv = a.nd.v;
    float nd[3 * kRegGroups];
#pragma unroll
    for (int j = 0; j < 3 * kRegGroups; ++j) nd[j] = j < 3 * K ? ndv[j] : 0.f;
    // quads' outputs as 2-byte and 8-byte stores when the arrays allow (a quad starts at an even
    // GID; sizes, when present, are scratch of this library and 8-byte aligned)
    const bool vec_out = ((uintptr_t)out_mask & 1u) == 0 && ((uintptr_t)out_groups & 1u) == 0 &&
                         ((uintptr_t)out_normals & 7u) == 0;
    static_assert(kRows == 4, "a warp's groups: 16 bits per row in one word");
    unsigned long long grp = 0;                          // 16 bits per row: first(v)'s group, second(v)'s
    const int gv = tx * T + lane;
#pragma unroll 1   // (unrolled: 1,100 instructions more, 45 bytes spilled)
    for (int row = 0; row < rows; ++row) {
        const int r = r0 + row;
        const int gu = ty * TH + r;
        const bool exists = gu < Hq && gv < Wq;
        V3 n[2];
        load_quad(cur, (r + h) * RQW + (lane + h), n[0], n[1]);
        const size_t gid0 = exists ? 2 * ((size_t)gu * Wq + gv) : 0;
        const unsigned mk = *reinterpret_cast<const uint16_t*>(Mk + 2 * (r * T + lane));
        int gk[2];
        bool kk[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool kept = ((mk >> (8 * k)) & 255u) != 0;
            const bool has = has_normal(n[k]);
            int g = PL3D_NO_GROUP;
            if (exists && kept && has) {                                         // Algorithm 4, ang_min
                float best = -1.0f;
                if (K <= kRegGroups) {
#pragma unroll
                    for (int j = 0; j < kRegGroups; ++j) {
                        if (j >= K) break;
                        const float s = n[k].x * nd[3 * j] + n[k].y * nd[3 * j + 1] + n[k].z * nd[3 * j + 2];
                        if (s > best) {
                            best = s;
                            g = j;
                        }
                    }
                } else {
                    for (int j = 0; j < K; ++j) {
                        const float s = n[k].x * ndv[3 * j] + n[k].y * ndv[3 * j + 1] + n[k].z * ndv[3 * j + 2];
                        if (s > best) {
                            best = s;
                            g = j;
                        }
                    }
                }
                if (best < min_dot) g = PL3D_NO_GROUP;
            }
            gk[k] = g;
            kk[k] = kept;
            if (!has) n[k] = {NAN, NAN, NAN};
        }
        grp |= (unsigned long long)(unsigned)(gk[0] | (gk[1] << 8)) << (16 * row);
        if (exists) {
            // the quad's two triangles are consecutive GIDs: one store per array when aligned
            if (vec_out) {
                *reinterpret_cast<uint16_t*>(out_mask + gid0) = (uint16_t)((kk[0] ? 1 : 0) | (kk[1] ? 256 : 0));
                *reinterpret_cast<uint16_t*>(out_groups + gid0) = (uint16_t)(gk[0] | (gk[1] << 8));
                float2* o = reinterpret_cast<float2*>(out_normals + 3 * gid0);
                o[0] = make_float2(n[0].x, n[0].y);
                o[1] = make_float2(n[0].z, n[1].x);
                o[2] = make_float2(n[1].y, n[1].z);
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    out_mask[gid0 + k] = kk[k] ? 1 : 0;
                    out_groups[gid0 + k] = (uint8_t)gk[k];
                    float* o = out_normals + 3 * (gid0 + k);
                    o[0] = n[k].x;
                    o[1] = n[k].y;
                    o[2] = n[k].z;
                }
            }
            if (sizes) *reinterpret_cast<int2*>(sizes + gid0) = make_int2(0, 0);
        }
    }
    stage_mark(bar, 3);

    // Connected components inside the tile (twins of Algorithm 2 that stay in the tile).
    const bool offs = a.max_offset_scaled > 0.f;
    const float lim = a.max_offset_scaled;
    auto offset_ok = [&](int g, V3 ci, V3 cj) {
        const float* n = ndv + 3 * g;
        return !offs || fabsf(n[0] * (ci.x - cj.x) + n[1] * (ci.y - cj.y) + n[2] * (ci.z - cj.z)) <= lim;
    };
    auto group_of = [&](int k) { return (int)(grp >> (8 * k)) & 255; };   // 2 row + side
    // (1) Runs along each quad row. Chain position 2v is second(v), 2v+1 is first(v); a run breaks
    // at second(v) unless first(v-1) links to it (right), at first(v) unless the quad's diagonal
    // links (diag). The last break at or before a position comes from the two ballots. A run linked to
    // one of the warp's row above takes that run's root at its first link, so that what is left for
    // the rounds below is a forest of few roots and shallow chains.
    int rootF[kRows], rootS[kRows];                      // roots inside the warp's rows, -1 without a group
    unsigned bD[kRows] = {}, bR[kRows] = {};
    int x[kRows], y[kRows];                              // the ends of links still to make; equal: none
    bool own[2 * kRows];                                 // this triangle is a root
    const unsigned le = kFull >> (31 - lane), lt = le >> 1;
    // first(r, v) with second(r-1, v), of group g_up: the lanes that link, without those whose runs,
    // above and below, both reach from the link of their left neighbour
    auto links = [&](int row, int g_up, unsigned upD, unsigned upR, unsigned& all) {
        const int r = r0 + row, gf = group_of(2 * row);
        bool link = gf != PL3D_NO_GROUP && g_up == gf;
        if (offs && link) {
            V3 cf, c1, c0u, cu;
            load_quad(Cq, (r + h) * RQW + (lane + h), cf, c1);
            load_quad(Cq, (r - 1 + h) * RQW + (lane + h), c0u, cu);
            link = offset_ok(gf, cf, cu);
        }
        all = __ballot_sync(kFull, link);
        return all & ~((all << 1) & (bR[row] << 1) & bD[row] & (upD << 1) & (upR << 1));
    };
#pragma unroll
    for (int row = 0; row < kRows; ++row) {
        rootF[row] = rootS[row] = -1;
        x[row] = y[row] = 0;
        own[2 * row] = own[2 * row + 1] = false;
        if (row >= rows) continue;
        const int r = r0 + row;
        const int gf = group_of(2 * row), gs = group_of(2 * row + 1);
        const int gs_next = __shfl_down_sync(kFull, gs, 1);
        bool diag = gf != PL3D_NO_GROUP && gs == gf;
        bool right = lane < 31 && gf != PL3D_NO_GROUP && gs_next == gf;
        if (offs) {
            V3 cf, cs2;
            load_quad(Cq, (r + h) * RQW + (lane + h), cf, cs2);
            const V3 cs_next = {__shfl_down_sync(kFull, cs2.x, 1), __shfl_down_sync(kFull, cs2.y, 1),
                                __shfl_down_sync(kFull, cs2.z, 1)};
            diag = diag && offset_ok(gf, cf, cs2);
            right = right && offset_ok(gf, cf, cs_next);
        }
        bD[row] = __ballot_sync(kFull, diag);
        bR[row] = __ballot_sync(kFull, right);
        const unsigned brk_f = ~bD[row], brk_s = ~(bR[row] << 1);   // (bit 0 of brk_s: a row starts a run)
        const int ls = 31 - __clz((int)(brk_s & le));
        const int start_f = max(2 * (31 - __clz((int)(brk_f & le))) + 1, 2 * ls);
        const int start_s = max(2 * (31 - __clz((int)(brk_f & lt))) + 1, 2 * ls);
        // smallest GID of a run starting at chain position p: first(p/2), unless the run is
        // second(p/2) alone
        auto root_of = [&](int p) {
            const int l0 = p >> 1;
            return 2 * (r * T + l0) + (((p & 1) || !((brk_f >> l0) & 1u)) ? 0 : 1);
        };
        const int tf = 2 * (r * T + lane);
        if (gf != PL3D_NO_GROUP) rootF[row] = root_of(start_f);
        if (gs != PL3D_NO_GROUP) rootS[row] = root_of(start_s);
        if (row > 0) {
            unsigned all;
            const unsigned some = links(row, group_of(row > 0 ? 2 * row - 1 : 0), bD[row > 0 ? row - 1 : 0],
                                        bR[row > 0 ? row - 1 : 0], all);
            // the lanes whose first triangle is in this lane's run: from the run's start to its last
            const unsigned cont = bR[row] & (bD[row] >> 1);        // first(v) reaches first(v+1)
            const int last = lane + __ffs((int)~(cont >> lane)) - 1;
            const unsigned run = (kFull >> (31 - last)) & (kFull << (start_f >> 1));
            const int f = __ffs((int)(all & run)) - 1;             // the run's first link
            const int up = rootS[row > 0 ? row - 1 : 0];
            const int root = __shfl_sync(kFull, up, f & 31);
            if (gf != PL3D_NO_GROUP && f >= 0) rootF[row] = root;
            const int left = __shfl_up_sync(kFull, rootF[row], 1);
            if (diag) rootS[row] = rootF[row];
            else if (lane > 0 && ((bR[row] >> (lane - 1)) & 1u)) rootS[row] = left;
            if (((some >> lane) & 1u) && up != rootF[row]) {
                x[row] = rootF[row];
                y[row] = up;
            }
        }
        own[2 * row] = rootF[row] == tf;
        own[2 * row + 1] = rootS[row] == tf + 1;
        if (own[2 * row]) Lp[tf] = tf;
        if (own[2 * row + 1]) Lp[tf + 1] = tf + 1;
        if (row == rows - 1) {
            UpRep[threadIdx.x] = rootS[row];
            UpGrp[threadIdx.x] = gs;
            if (lane == 0) {
                UpMask[2 * warp] = bD[row];
                UpMask[2 * warp + 1] = bR[row];
            }
        }
    }
    __syncthreads();
    // (2) The links of the warp's first row with the row above, another warp's.
    if (warp > 0) {
        unsigned all;
        const unsigned some = links(0, UpGrp[threadIdx.x - 32], UpMask[2 * warp - 2], UpMask[2 * warp - 1], all);
        if ((some >> lane) & 1u) {
            x[0] = rootF[0];
            y[0] = UpRep[threadIdx.x - 32];
        }
    }
    // (3) Segments from the links, in rounds over all links at once. At the start of a round every
    // root of (1) points at its root so far. A link between two roots lowers the parent of the larger
    // to the smaller (the smallest wins; a link stays on the list until it finds its two ends under
    // one root, so one whose update lost is tried again). Then each root of (1) jumps to its root,
    // all at once, which takes the logarithm of a chain's length. A round that changes anything removes
    // a root; scans take two or three rounds.
    // A thread's loads are issued together in every step: what bounds a round is their latency.
    volatile int32_t* const vp = Lp;
    while (true) {
        int a0[kRows], b0[kRows];
        bool todo = false;
#pragma unroll
        for (int row = 0; row < kRows; ++row) {
            const bool on = x[row] != y[row];
            a0[row] = on ? vp[x[row]] : 0;
            b0[row] = on ? vp[y[row]] : 0;
        }
#pragma unroll
        for (int row = 0; row < kRows; ++row) {
            if (a0[row] != b0[row]) {
                atomicMin(Lp + max(a0[row], b0[row]), min(a0[row], b0[row]));
                todo = true;
            } else {
                x[row] = y[row];
            }
        }
        if (!__syncthreads_or(todo)) break;
        int up[2 * kRows];                               // current parent of each own root, -1: none
#pragma unroll
        for (int k = 0; k < 2 * kRows; ++k) up[k] = own[k] ? vp[2 * ((r0 + (k >> 1)) * T + lane) + (k & 1)] : -1;
        bool more;
        do {
            more = false;
            int g[2 * kRows];
#pragma unroll
            for (int k = 0; k < 2 * kRows; ++k) g[k] = up[k] >= 0 ? vp[up[k]] : -1;
#pragma unroll
            for (int k = 0; k < 2 * kRows; ++k)
                if (g[k] != up[k]) {
                    up[k] = g[k];
                    vp[2 * ((r0 + (k >> 1)) * T + lane) + (k & 1)] = g[k];
                    more = true;
                }
        } while (more);
        __syncthreads();
    }
    // (4) Each triangle leaves with the GID of its tile-local root (-1 without a group).
    int32_t* const labels = a.labels;
    const bool vec_lab = ((uintptr_t)labels & 7u) == 0;   // a quad's two labels in one 8-byte store
    const int base = 2 * (ty * TH * Wq + tx * T);         // GID of the tile's first triangle
#pragma unroll
    for (int row = 0; row < kRows; ++row) {
        if (row >= rows) break;
        const int gu = ty * TH + r0 + row;
        const int tF = rootF[row] >= 0 ? Lp[rootF[row]] : -1, tS = rootS[row] >= 0 ? Lp[rootS[row]] : -1;
        // tile-local index 2 (row T + column) + side -> GID
        const int labF = tF >= 0 ? base + (tF / (2 * T)) * (2 * Wq) + tF % (2 * T) : -1;
        const int labS = tS >= 0 ? base + (tS / (2 * T)) * (2 * Wq) + tS % (2 * T) : -1;
        if (gu >= Hq || gv >= Wq) continue;
        const size_t gid0 = 2 * ((size_t)gu * Wq + gv);
        if (vec_lab) {
            *reinterpret_cast<int2*>(labels + gid0) = make_int2(labF, labS);
        } else {
            labels[gid0] = labF;
            labels[gid0 + 1] = labS;
        }
    }
    __syncthreads();
    // (5) The borders with the neighbouring tiles, when this launch joins them here (the
    // single-frame kernel; the batch kernel joins them in its merge phase).
    if (JOIN && a.border) join_tile_borders(a, tile);
    stage_mark(bar, 4);
}

// ------------------------------------------------------------------------- segments (Alg. 5)

// Centroid of triangle k of quad (u, v) from the smoothed points v0 + d (offset test only).
__device__ __forceinline__ V3 centroid_global(const FrameArgs& a, int u, int v, int k) {
    const int W = a.W;
    const size_t p1 = (size_t)u * W + v, p2 = p1 + 1, p3 = p1 + W + 1, p4 = p1 + W;
    const size_t ia = 3 * (k == 0 ? p3 : p1), ib = 3 * (k == 0 ? p2 : p4), ic = 3 * (k == 0 ? p1 : p3);
    const float* P = a.points;
    const float* D = a.disp;   // written earlier in this launch: L2-coherent loads
    const float kk = 1.f / 3.f;
    return {((P[ia] + P[ib] + P[ic]) + (__ldcg(D + ia) + __ldcg(D + ib) + __ldcg(D + ic))) * kk,
            ((P[ia + 1] + P[ib + 1] + P[ic + 1]) + (__ldcg(D + ia + 1) + __ldcg(D + ib + 1) + __ldcg(D + ic + 1))) * kk,
            ((P[ia + 2] + P[ib + 2] + P[ic + 2]) + (__ldcg(D + ia + 2) + __ldcg(D + ib + 2) + __ldcg(D + ic + 2))) * kk};
}

// Twins that cross a tile border: the top edge of a tile's first quad row and the right edge of
// its last quad column (tiles of a.bil_th x T quads). Work items: (row borders) x Wq, then
// (column borders) x Hq. Returns
// whether item w joins two triangles, and then their current labels (each in its triangle's
// set: the tile root, or an ancestor of it once a union has linked that root).
__device__ __forceinline__ bool merge_pair(const FrameArgs& a, long long w, int& ra, int& rb) {
    const int Wq = a.W - 1, Hq = a.H - 1, TH = a.bil_th;
    const long long n_row_items = (long long)(div_up(Hq, TH) - 1) * Wq;
    int u, v, uj, vj;
    if (w < n_row_items) {
        u = (int)(w / Wq + 1) * TH;
        v = (int)(w % Wq);
        uj = u - 1;
        vj = v;
    } else {
        const long long x = w - n_row_items;
        v = (int)(x / Hq + 1) * T - 1;
        u = (int)(x % Hq);
        uj = u;
        vj = v + 1;
    }
    const int i = 2 * (u * Wq + v);
    const int j = 2 * (uj * Wq + vj) + 1;
    const int g = __ldcg(a.groups + i);   // written by the bilateral pass of this launch
    if (g == PL3D_NO_GROUP || __ldcg(a.groups + j) != g) return false;
    if (a.max_offset > 0.f) {
        const V3 ci = centroid_global(a, u, v, 0), cj = centroid_global(a, uj, vj, 1);
        const float* nd = a.nd.v + 3 * g;
        if (fabsf(nd[0] * (ci.x - cj.x) + nd[1] * (ci.y - cj.y) + nd[2] * (ci.z - cj.z)) > a.max_offset) return false;
    }
    ra = __ldcg(a.labels + i);
    rb = __ldcg(a.labels + j);
    return true;
}

// merge_pair with the item's two groups and two labels loaded together (one round trip to L2
// instead of two; the labels are read whether or not the item joins).
__device__ __forceinline__ bool merge_pair_eager(const FrameArgs& a, long long w, int& ra, int& rb) {
    const int Wq = a.W - 1, Hq = a.H - 1, TH = a.bil_th;
    const long long n_row_items = (long long)(div_up(Hq, TH) - 1) * Wq;
    int u, v, uj, vj;
    if (w < n_row_items) {
        u = (int)(w / Wq + 1) * TH;
        v = (int)(w % Wq);
        uj = u - 1;
        vj = v;
    } else {
        const long long x = w - n_row_items;
        v = (int)(x / Hq + 1) * T - 1;
        u = (int)(x % Hq);
        uj = u;
        vj = v + 1;
    }
    const int i = 2 * (u * Wq + v);
    const int j = 2 * (uj * Wq + vj) + 1;
    const int g = __ldcg(a.groups + i), gj = __ldcg(a.groups + j);
    ra = __ldcg(a.labels + i);
    rb = __ldcg(a.labels + j);
    if (g == PL3D_NO_GROUP || gj != g) return false;
    if (a.max_offset > 0.f) {
        const V3 ci = centroid_global(a, u, v, 0), cj = centroid_global(a, uj, vj, 1);
        const float* nd = a.nd.v + 3 * g;
        if (fabsf(nd[0] * (ci.x - cj.x) + nd[1] * (ci.y - cj.y) + nd[2] * (ci.z - cj.z)) > a.max_offset) return false;
    }
    return true;
}

// One union per distinct pair in a warp: consecutive lanes walk one border, where long runs
// of twins join the same two tile segments; a lane whose pair (and frame) equals its left
// neighbour's leaves the union to that lane. Called by whole warps.
__device__ __forceinline__ void merge_unite(int32_t* labels, bool link, int ra, int rb, int frame) {
    if (!link) ra = rb = -1;
    const int pa = __shfl_up_sync(0xffffffffu, ra, 1), pb = __shfl_up_sync(0xffffffffu, rb, 1);
    const int pf = __shfl_up_sync(0xffffffffu, frame, 1);
    const bool dup = (threadIdx.x & 31) > 0 && pa == ra && pb == rb && pf == frame;
    if (link && !dup) uf_unite(labels, ra, rb);
}

// Joins a finished tile's segments with its neighbours' across the tile's borders, in the
// bilateral pass instead of a merge phase of its own. Each border is joined by the second of its
// two tiles to finish: both add 1 to the border's counter (an acquire-release atomic, after the
// barrier that ends the tile's label stores), and the one that reads an odd count joins it, so
// that no tile waits for another. Every launch adds 2 to each counter, so the counters are even
// between launches. Counter 2t is tile t's top border, 2t + 1 its left border. Warp k of the CTA
// takes side k (top, left, bottom, right), its lanes along the border (merge_pair's items); the
// other warps go on. Each item's groups and labels are loaded together; the unions halve the
// paths they walk, which keeps the trees shallow for the flatten phase (without halving: 6 us slower per
// 480x640 frame, most of it in the flatten).
__device__ __forceinline__ void join_tile_borders(const FrameArgs& a, int tile) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= 4) return;
    const int Wq = a.W - 1, Hq = a.H - 1, TH = a.bil_th;
    const int tiles_x = div_up(Wq, T), tiles_y = div_up(Hq, TH);
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const bool has = warp == 0 ? ty > 0 : warp == 1 ? tx > 0 : warp == 2 ? ty + 1 < tiles_y : tx + 1 < tiles_x;
    if (!has) return;
    const int c = warp == 0 ? 2 * tile : warp == 1 ? 2 * tile + 1 : warp == 2 ? 2 * (tile + tiles_x) : 2 * (tile + 1) + 1;
    unsigned n = 0;
    if (lane == 0) n = atom_add_acq_rel_gpu(a.border + c, 1u);
    __syncwarp();   // the lanes' loads below ordered after lane 0's acquire
    if (!(__shfl_sync(0xffffffffu, n, 0) & 1u)) return;   // the neighbour joins it when it finishes
    // row borders first among the items, then columns
    const long long n_row_items = (long long)(tiles_y - 1) * Wq;
    const int len = (warp & 1) ? min(TH, Hq - ty * TH) : min(T, Wq - tx * T);
    const long long w0 = warp == 0   ? (long long)(ty - 1) * Wq + tx * T
                         : warp == 1 ? n_row_items + (long long)(tx - 1) * Hq + ty * TH
                         : warp == 2 ? (long long)ty * Wq + tx * T
                                     : n_row_items + (long long)tx * Hq + ty * TH;
    int32_t* const L = a.labels;
    for (int i0 = 0; i0 < len; i0 += 32) {   // the same trip count in every lane
        int ra = -1, rb = -1;
        const bool link = i0 + lane < len && merge_pair_eager(a, w0 + i0 + lane, ra, rb);
        if (!link) ra = rb = -1;
        const int pa = __shfl_up_sync(0xffffffffu, ra, 1), pb = __shfl_up_sync(0xffffffffu, rb, 1);
        const bool dup = lane > 0 && pa == ra && pb == rb;   // one union per distinct pair
        if (link && !dup) uf_unite(L, ra, rb);
    }
}

__device__ __forceinline__ void merge_phase(const FrameArgs& a) {
    const int Wq = a.W - 1, Hq = a.H - 1;
    const long long n = (long long)(div_up(Hq, a.bil_th) - 1) * Wq + (long long)(div_up(Wq, T) - 1) * Hq;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n_iter = (n + stride - 1) / stride;   // uniform: whole warps stay together
    const long long base = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (long long it = 0; it < n_iter; ++it) {
        const long long w = base + it * stride;
        int ra = -1, rb = -1;
        const bool link = w < n && merge_pair(a, w, ra, rb);
        merge_unite(a.labels, link, ra, rb, 0);
    }
}

// Flatten: every grouped triangle takes its root, in blocks of 128 VEC consecutive labels per
// warp, VEC 16-byte loads per lane. A triangle's label is the root of its tile's segment, whose
// parent chain (one or two hops, measured) ends at the segment's root.
//
// What bounds it: most of a frame's chains end at a few roots (the floor, a wall), so thousands of
// warps ask for the same words. Read past L1 those requests queue at one L2 slice: on a batch of 256
// mixed frames (73.9 M triangles) the mean warp took 0.6 ms and the last one 1.9 ms. The parents are
// therefore read through L1: the grid barrier before this phase acquires at GPU scope, so a line
// cached here is no older than the last union, and a word that another thread has meanwhile replaced
// by its root was and is an ancestor, either way. The labels themselves are read once, past L1, 16
// bytes per lane. With both, the phase took 0.38 ms and the batch 5.88 instead of 7.40 ms; a 480x640
// frame 69.6 instead of 73.7 us. After that a warp waits for one load after another, so a batch,
// whose warps take dozens of blocks each, has kFlatVecBatch loads per lane in flight (417 us at 2, 278 us
// at 4, 178 us at 8); a 480x640 frame has less than a block per warp, and 4 cost it 0.9 us (a 720x1280 frame
// has three, at 2 as well).
constexpr int kFlatVec = 2, kFlatVecBatch = 8;
template <int VEC>
constexpr int kFlatBlock = 32 * 4 * VEC;

// Blocks of a frame of n labels; blocks start at 16-byte boundaries, up to 3 labels before the first.
template <int VEC>
__device__ __forceinline__ long long flatten_blocks(long long n) { return (n + 3 + kFlatBlock<VEC> - 1) / kFlatBlock<VEC>; }

// Block b of the labels L[0 .. n): roots into L and, when given, into `copy`; with `sizes` the
// segment sizes are counted (an atomic per root and warp load, one per block when it has one root).
// Called by whole warps.
template <int VEC>
__device__ __forceinline__ void flatten_block(int32_t* L, long long n, int32_t* sizes, int32_t* copy, long long b) {
    const int lane = threadIdx.x & 31;
    const int shift = (int)(((uintptr_t)L >> 2) & 3u);
    const long long i0 = b * kFlatBlock<VEC> - shift + 4 * lane;
    int x[4 * VEC], p[4 * VEC];
    bool whole[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        const long long i = i0 + 128 * v;
        whole[v] = i >= 0 && i + 4 <= n;
        if (whole[v]) {
            const int4 q = __ldcg(reinterpret_cast<const int4*>(L + i));
            x[4 * v] = q.x, x[4 * v + 1] = q.y, x[4 * v + 2] = q.z, x[4 * v + 3] = q.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) x[4 * v + k] = i + k >= 0 && i + k < n ? __ldcg(L + i + k) : -1;
        }
    }
#pragma unroll
    for (int k = 0; k < 4 * VEC; ++k) p[k] = x[k] >= 0 ? __ldca(L + x[k]) : -1;
    // one hop of every unfinished walk per round, their loads together
    bool more;
    do {
        more = false;
#pragma unroll
        for (int k = 0; k < 4 * VEC; ++k)
            if (p[k] != x[k]) {
                x[k] = p[k];
                p[k] = __ldca(L + x[k]);
                more = true;
            }
    } while (more);
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        const long long i = i0 + 128 * v;
        if (whole[v]) {
            *reinterpret_cast<int4*>(L + i) = make_int4(x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i + k >= 0 && i + k < n) L[i + k] = x[4 * v + k];
        }
        if (copy) {
            // page-locked host memory as a rule: whole lines when it is aligned as L is (4-byte stores
            // of every fourth word cost a 240x320 host-buffer call 3 us)
            if (whole[v] && (((uintptr_t)copy ^ (uintptr_t)L) & 15u) == 0) {
                *reinterpret_cast<int4*>(copy + i) = make_int4(x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (i + k >= 0 && i + k < n) copy[i + k] = x[4 * v + k];
            }
        }
    }
    if (sizes) {
        __syncwarp();
        // the block's first root; a block that has no other needs one atomic
        int first = -1, mine = 0;
        bool one = true;
#pragma unroll
        for (int k = 0; k < 4 * VEC; ++k) {
            if (x[k] < 0) continue;
            if (first < 0) first = x[k];
            one &= x[k] == first;
            ++mine;
        }
        const unsigned have = __ballot_sync(0xffffffffu, mine > 0);
        if (!have) return;
        const int lead = __ffs(have) - 1;
        const int root = __shfl_sync(0xffffffffu, first, lead);
        if (__all_sync(0xffffffffu, mine == 0 || (one && first == root))) {
            const int count = __reduce_add_sync(0xffffffffu, mine);
            if (lane == lead) atomicAdd(sizes + root, count);
        } else {
#pragma unroll
            for (int k = 0; k < 4 * VEC; ++k) {
                const unsigned peers = __match_any_sync(0xffffffffu, x[k]);
                if (x[k] >= 0 && lane == __ffs(peers) - 1) atomicAdd(sizes + x[k], __popc(peers));
            }
        }
    }
}

__device__ __forceinline__ void flatten_phase(const FrameArgs& a) {
    const long long n = 2LL * (a.H - 1) * (a.W - 1);
    int32_t* const L = a.labels;
    int32_t* const sizes = a.sizes;
    int32_t* const copy = sizes ? nullptr : a.labels_copy;   // with tri_min the filter writes it
    const long long blocks = flatten_blocks<kFlatVec>(n);
    const int warps = gridDim.x * (kThreads / 32);
    // warp k of every CTA takes blocks k gridDim.x + the CTA's index: a frame of fewer blocks than
    // warps spreads over all SMs
    for (long long b = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; b < blocks; b += warps)
        flatten_block<kFlatVec>(L, n, sizes, copy, b);
}

// Algorithm 5 keeps a segment only when it has more than tri_min triangles.
__device__ __forceinline__ void filter_phase(const FrameArgs& a) {
    const long long n = 2LL * (a.H - 1) * (a.W - 1);
    int32_t* const labels = a.labels;
    int32_t* const copy = a.labels_copy;
    const int32_t* const sizes = a.sizes;
    const int min_triangles = a.min_triangles;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int l = __ldcg(labels + i);
        const bool drop = l >= 0 && __ldcg(sizes + l) <= min_triangles;   // sizes: other CTAs' atomics
        if (drop) labels[i] = -1;
        if (copy) copy[i] = drop ? -1 : l;
    }
}

__device__ __forceinline__ void phase_mark(const FrameArgs& a, int slot, uint64_t& t_prev) {
    if (a.phase_ns && blockIdx.x == 0 && threadIdx.x == 0) {
        const uint64_t t = global_ns();
        atomicAdd(a.phase_ns + slot, (unsigned long long)(t - t_prev));
        t_prev = t;
    }
}

}  // namespace frame

template <int RL, int RB>
__global__ void __launch_bounds__(kThreads, 2) frame_kernel(const __grid_constant__ FrameArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);   // [kLapMaxStages]: one per staging slot
    float* smem = reinterpret_cast<float*>(smem_raw + 128);
    unsigned* gen = reinterpret_cast<unsigned*>(smem_raw + frame::kHdrGen);
    grid_barrier_begin(a.barrier, gen);
    if (threadIdx.x == 0)
        for (int i = 0; i < kLapMaxStages; ++i) mbar_init(bar + i, 1);
    frame::set_stage_timing(bar, a.phase_ns ? a.phase_ns + kStageSlot : nullptr);
    __syncthreads();
    unsigned par = 0;   // mbarrier parities of the staging slots, one bit each
    uint64_t t_prev = 0;
    if (a.phase_ns && blockIdx.x == 0 && threadIdx.x == 0) t_prev = global_ns();

    // a launch may run part of the path (a.part): the smoothing and tile-local segments, or the
    // segments across tiles; the launch boundary then orders the two
    if (a.part != 2) {
        for (int c = 0; c < a.n_lap; ++c) {
            const LapPhase& ph = a.lap[c];
            const int tiles_lap = ph.tiles;
            const CUtensorMap* map = ph.use_tma ? &a.tm_pts_lap : nullptr;
            // buffers: [box 0 .. box ns-1][D a][D b] (one D buffer for a single-iteration first
            // pass); the box of this CTA's tile k is slot k mod ns, and the TMA loads of its next
            // ns - 1 tiles are in flight while tile k computes
            const int P = align_floats(ph.box.rows * ph.box.cols);
            const int ns = map ? ph.stages : 1;
            float* Da = smem + ns * P;
            float* Db = Da + (ph.dbufs - 1) * P;
            for (int k = 0; k + 1 < ns; ++k) {
                const int t = (int)blockIdx.x + k * (int)gridDim.x;
                if (t < tiles_lap) frame::lap_issue(a, ph, map, t, smem + k * P, bar + k);
            }
            int s = 0;
            for (int t = blockIdx.x; t < tiles_lap; t += gridDim.x) {
                if (map) {
                    const int ahead = t + (ns - 1) * (int)gridDim.x;
                    const int sa = s == 0 ? ns - 1 : s - 1;   // the slot of the previous tile, now free
                    if (ahead < tiles_lap) frame::lap_issue(a, ph, map, ahead, smem + sa * P, bar + sa);
                }
                const frame::LapJob j = frame::lap_job(a, ph, t);
                frame::lap_tile<RL>(j, smem + s * P, Da, Db, map != nullptr, bar + s, (par >> s) & 1u);
                if (map) par ^= 1u << s;
                s = s + 1 == ns ? 0 : s + 1;
            }
            grid_barrier(a.barrier, a.error, gen);
        }
        frame::phase_mark(a, 0, t_prev);
        const int tiles_bil = div_up(a.H - 1, a.bil_th) * div_up(a.W - 1, kTile);
        unsigned par0 = par & 1u;   // the bilateral stages through slot 0
        for (int c = 0; c < a.n_bil; ++c) {
            for (int t = blockIdx.x; t < tiles_bil; t += gridDim.x) frame::bil_tile<RB, true>(a, a.bil[c], t, smem, bar, par0);
            if (a.part == 0 || c + 1 < a.n_bil) grid_barrier(a.barrier, a.error, gen);
        }
        frame::phase_mark(a, 1, t_prev);
    }
    if (a.part == 1) {
        // one bilateral pass after a Laplacian in kernels of its own: no barrier, and with fewer tiles
        // than CTAs some CTAs come here at once
        grid_barrier_unused();
        return;
    }
    if (!a.border) {   // else the bilateral tiles joined their borders
        frame::merge_phase(a);
        grid_barrier(a.barrier, a.error, gen);
    }
    frame::phase_mark(a, 2, t_prev);
    frame::flatten_phase(a);
    if (a.min_triangles > 0) {
        grid_barrier(a.barrier, a.error, gen);
        frame::filter_phase(a);
    }
    frame::phase_mark(a, 3, t_prev);
}

namespace frame {

// Frame of work item t: the largest f < n with pre[f] <= t (pre[0] = 0 <= t < pre[n]).
__device__ __forceinline__ int find_frame(const int* pre, int n, int t) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(pre + mid) <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Tiles of a batch phase go to the CTAs one at a time, round-robin, so that no CTA gets more than one
// above the others: in runs of 4 consecutive tiles (closer halos, a tensor-map acquire per run) a CTA
// took 8 tiles of a batch that has 4.5 for each, 368 us for 8 mixed frames against 254 us, 1014 / 977 for
// 48, 5465 / 5352 for 256 of one mix (one iteration: 209 / 156, 576 / 557, 3109 / 3080).
__device__ __forceinline__ int next_tile(int t) { return t + (int)gridDim.x; }

// Advances f (never backwards) to the frame whose range of pre holds item i.
__device__ __forceinline__ int advance_frame(const long long* pre, int f, long long i) {
    while (__ldg(pre + f + 1) <= i) ++f;
    return f;
}

}  // namespace frame

// Many frames in one persistent launch: each phase runs over the concatenated work of all
// frames (tiles, tile-border twins, triangles), with one grid barrier between phases, so the
// small frames of a batch share the GPU instead of leaving most of it idle.
template <int RL, int RB>
__global__ void __launch_bounds__(kThreads, 2) batch_kernel(const __grid_constant__ BatchArgs b) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);   // [kLapMaxStages]: one per staging slot
    float* smem = reinterpret_cast<float*>(smem_raw + 128);
    unsigned* gen = reinterpret_cast<unsigned*>(smem_raw + frame::kHdrGen);
    grid_barrier_begin(b.barrier, gen);
    if (threadIdx.x == 0)
        for (int i = 0; i < kLapMaxStages; ++i) mbar_init(bar + i, 1);
    frame::set_stage_timing(bar, b.hdr->timing ? b.phase_ns + kStageSlot : nullptr);
    __syncthreads();
    unsigned par = 0;   // mbarrier parities of the staging slots, one bit each
    const int n = b.hdr->n, n_lap = b.hdr->n_lap, n_bil = b.hdr->n_bil;
    const bool any_filter = b.hdr->any_filter != 0;
    unsigned long long* pns = b.hdr->timing ? b.phase_ns : nullptr;
    uint64_t t_prev = 0;
    const bool stamp = pns && blockIdx.x == 0 && threadIdx.x == 0;
    auto mark = [&](int slot) {
        if (stamp) {
            const uint64_t t = global_ns();
            atomicAdd(pns + slot, (unsigned long long)(t - t_prev));
            t_prev = t;
        }
    };
    if (stamp) t_prev = global_ns();

    for (int c = 0; c < n_lap; ++c) {
        const int* pre = b.lap_tiles + c * b.stride;
        const int total = __ldg(pre + n);
        // buffers as in the frame kernel, sized for the largest box of this pass over the frames:
        // [box 0 .. box ns-1][D a][D b]; the box of this CTA's k-th tile is slot k mod ns
        const int P = b.hdr->lap_buf[c];
        const int ns = b.hdr->lap_stages[c];
        float* Da = smem + ns * P;
        float* Db = Da + (b.hdr->lap_dbufs[c] - 1) * P;
        // TMA-issues tile t (of frame f) into a slot when the frame stages by TMA. A CTA meets the
        // frames in increasing order, so it acquires each frame's tensor map once.
        int acquired = -1;
        auto issue = [&](int t, int f, int slot) {
            const FrameArgs& a = b.frames[f];
            if (!a.lap[c].use_tma) return;
            const CUtensorMap* map = &a.tm_pts_lap;
            if (f != acquired) {
                if (threadIdx.x == 0) tensormap_acquire(map);
                acquired = f;
            }
            frame::lap_issue(a, a.lap[c], map, t - __ldg(pre + f), smem + slot * P, bar + slot);
        };
        const int t_begin = (int)blockIdx.x;
        int f_cur = t_begin < total ? frame::find_frame(pre, n, t_begin) : 0;
        // the furthest tile of the sequence issued so far, and its frame (frames grow along it)
        int t_ahd = t_begin, f_ahd = f_cur;
        if (ns > 1 && t_begin < total) {
            issue(t_begin, f_cur, 0);
            for (int k = 1; k + 1 < ns; ++k) {
                t_ahd = frame::next_tile(t_ahd);
                if (t_ahd >= total) break;
                while (__ldg(pre + f_ahd + 1) <= t_ahd) ++f_ahd;
                issue(t_ahd, f_ahd, k);
            }
        }
        int s = 0;
        for (int t = t_begin; t < total; t = frame::next_tile(t)) {
            while (__ldg(pre + f_cur + 1) <= t) ++f_cur;
            if (ns > 1) {
                t_ahd = frame::next_tile(t_ahd);
                if (t_ahd < total) {
                    while (__ldg(pre + f_ahd + 1) <= t_ahd) ++f_ahd;
                    issue(t_ahd, f_ahd, s == 0 ? ns - 1 : s - 1);   // the previous tile's slot, now free
                }
            } else {
                issue(t, f_cur, 0);
            }
            const FrameArgs& a = b.frames[f_cur];
            const bool tma = a.lap[c].use_tma != 0;
            const frame::LapJob j = frame::lap_job(a, a.lap[c], t - __ldg(pre + f_cur));
            frame::lap_tile<RL>(j, smem + s * P, Da, Db, tma, bar + s, (par >> s) & 1u);
            if (tma) par ^= 1u << s;
            s = s + 1 == ns ? 0 : s + 1;
        }
        grid_barrier(b.barrier, b.error, gen);
    }
    mark(0);
    unsigned par0 = par & 1u;   // the bilateral stages through slot 0
    for (int c = 0; c < n_bil; ++c) {
        const int* pre = b.bil_tiles + c * b.stride;
        const int total = __ldg(pre + n);
        int acquired = -1;   // frames come in increasing order: each frame's maps acquired once
        const int t_begin = (int)blockIdx.x;
        int f = t_begin < total ? frame::find_frame(pre, n, t_begin) : 0;
        for (int t = t_begin; t < total; t = frame::next_tile(t)) {
            while (__ldg(pre + f + 1) <= t) ++f;
            const FrameArgs& a = b.frames[f];
            if (a.bil[c].use_tma && f != acquired) {
                if (threadIdx.x == 0) {
                    tensormap_acquire(&a.tm_pts_bil);
                    tensormap_acquire(&a.tm_disp_bil);
                }
                acquired = f;
            }
            frame::bil_tile<RB, false>(a, a.bil[c], t - __ldg(pre + f), smem, bar, par0);
        }
        grid_barrier(b.barrier, b.error, gen);
    }
    mark(1);
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long base = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    {
        const long long total = __ldg(b.merge_items + n);
        const long long n_iter = (total + stride - 1) / stride;   // uniform: whole warps stay together
        int f = 0;
        for (long long it = 0; it < n_iter; ++it) {
            const long long w = base + it * stride;
            int ra = -1, rb = -1;
            bool link = false;
            int32_t* labels = nullptr;
            if (w < total) {
                f = frame::advance_frame(b.merge_items, f, w);
                const FrameArgs& a = b.frames[f];
                labels = a.labels;
                link = frame::merge_pair(a, w - __ldg(b.merge_items + f), ra, rb);
            }
            frame::merge_unite(labels, link, ra, rb, f);
        }
    }
    grid_barrier(b.barrier, b.error, gen);
    mark(2);
    {
        // every grouped triangle takes its root, block by block. Frame f's blocks start at
        // tris[f] / B + 2 f: at least flatten_blocks() of them, the last ones empty
        constexpr int B = frame::kFlatBlock<frame::kFlatVecBatch>;
        const long long total = __ldg(b.tris + n) / B + 2LL * n;
        int f = 0;
        for (long long k = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; k < total;
             k += (long long)gridDim.x * (kThreads / 32)) {
            while (__ldg(b.tris + f + 1) / B + 2LL * (f + 1) <= k) ++f;
            const long long t0 = __ldg(b.tris + f);
            const FrameArgs& a = b.frames[f];
            frame::flatten_block<frame::kFlatVecBatch>(a.labels, __ldg(b.tris + f + 1) - t0, a.sizes, nullptr,
                                                       k - (t0 / B + 2LL * f));
        }
    }
    if (any_filter) {
        grid_barrier(b.barrier, b.error, gen);
        // Algorithm 5 keeps a segment only when it has more than tri_min triangles
        const long long total = __ldg(b.tris + n);
        int f = 0;
        for (long long i = base; i < total; i += stride) {
            f = frame::advance_frame(b.tris, f, i);
            const FrameArgs& a = b.frames[f];
            if (!a.sizes) continue;
            const int li = (int)(i - __ldg(b.tris + f));
            const int l = __ldcg(a.labels + li);
            if (l >= 0 && __ldcg(a.sizes + l) <= a.min_triangles) a.labels[li] = -1;
        }
    }
    mark(3);
}

}  // namespace pl3d
