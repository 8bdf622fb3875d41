// sl_gather2d.cuh -- the 2-D FP32 production step of the FSL scheme (arXiv:1410.2817) for up to four
// fields: one launch of two phases.
//
//   A. every node once: the jump flags of Sec. 2.3, written with the field values as records of up
//      to three fields and a flag word per node (16 bytes, or 8 for a single field);
//   B. every target: refined start, element walk with FP32 Newton inversion (Sec. 2.2, eq.
//      mapping1), order from the OR of the 16 taps' flag words, cubic and bilinear tensor sums (eq.
//      multiZ) -- all operands through L1: displacements as FP32 pairs, a tap of up to three fields
//      and its flags as one 128-bit load.
//
// A fused step integrates the next step's trajectories (eq. vel) between the phases: they depend on
// the velocity alone, so they fill the time phase B waits for phase A.
//
// What bounds it is instruction issue and load latency, not HBM (all of a 1024^2 x 3 step's operands
// fit L2): 16.4 M warp instructions for the remap (98 a node in phase A, ~390 a target in phase B),
// issue-active 46 % with 32 warps per SM.  Against the tiles staged in shared memory it tests each node
// once instead of 1.8 times (the tiles' windows overlap) and has no window boxes, staging or block
// barriers per tile.  Back to back with warm L2 (us a launch; TMA-staged tiles / per-element-copy
// tiles / this kernel), three fields of the swirl: remap 256^2 14.9 / 10.7 / 7.8, 1024^2 37.5 / 31.5 /
// 26.9, 2048^2 124 / 129 / 98.5; fused step 1024^2 50.3 / 44.3 / 38.7; Burgers 1024^2 33.9 (tiles) / 28.3.
// Where the tiles are better (two_phase_size has the rule) they stay.
#pragma once

#include "sl_tile2d.cuh"

namespace {

// CTAs per SM the registers are cut for (1024^2 x 3 remap: 3 / 4 / 5 / 6 measured 30.9 / 30.8 / 34.3 / 40.9 us)
constexpr int GMINB = 4;
constexpr int GNT = 256;       // threads per CTA: 8 warps, one row of 32 targets each
constexpr int GTX = 32, GTY = 8;
constexpr int GHOPS = 4;       // elements a target of the fast path tries (fewer under a lower hop limit)
// nodes of a warp in phase A (2 / 4 / 8 rows: 32.6 / 30.8 / 31.8 us)
constexpr int GCOLS = 30, GROWS = 4;

// Records: groups of up to three fields.  Group g holds in_rec(NF, g) fields from field 3 g; a group
// of one field takes 8 bytes per node (value, flags), larger ones 16 (values, flags in the last word).
__host__ __device__ constexpr int rec_groups(int nf) { return (nf + 2) / 3; }
__host__ __device__ constexpr int in_rec(int nf, int g) { return nf - 3 * g < 3 ? nf - 3 * g : 3; }

// The record planes carry the periodic images a stencil may reach: one node to the left and below, two
// to the right and above, in rows of n0 + 3 records.
constexpr int REC_LO = 1, REC_HI = 2;

struct GatherArgs {
    TileArgs t;
    void *rec[2];        // node (0, 0) of each group's plane (up to four fields: two groups)
    unsigned *sync;      // claims taken, claims done, CTAs that left
    unsigned long long *timeouts;
    int tiles_y, ntiles; // GTX x GTY tiles, numbered down the columns
    int step_x, step_y;  // what gridDim.x tiles on means: columns of nodes, tiles down
    float reach0, reach1;  // displacements of the fast path: n - 12
    int strips, nflag;   // phase A: strips of GCOLS columns, warp items
    int nclaim;          // claims of one item per warp of a CTA
    int hops;            // the smaller of GHOPS and the grid's walk_max
};

// ---- the order of the phases --------------------------------------------------------------------
// Phase A's work is claimed item by item from a counter by whichever CTAs run, and phase B waits until
// every item is done.  An item is always in the hands of a running CTA that waits for nothing before
// it is done, so the wait ends whether or not every CTA is resident: no cooperative launch is needed
// (it costs ~12 us a launch here) and launches on several streams may share the SMs.  Words: items
// claimed, items done, CTAs that left; the last CTA to leave clears them for the next launch.
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Thread 0 waits, for GWAITS looks at the counter (a quarter of a microsecond and more each: over 2 s;
// looks are counted instead of time because a clock runs on while another process has the GPU); the CTA
// learns the result.
constexpr int GWAITS = 1 << 23;
__device__ __forceinline__ bool wait_items(const unsigned *sync, unsigned n, int *s_ok)
{
    if (threadIdx.x == 0) {
        int left = GWAITS;
        while (ld_acquire(sync + 1) < n && left > 0) {
            __nanosleep(40);
            --left;
        }
        __threadfence();
        *s_ok = left > 0;
    }
    __syncthreads();
    return *s_ok != 0;
}
__device__ __forceinline__ void leave(unsigned *sync)
{
    if (threadIdx.x == 0 && atomicAdd(sync + 2, 1u) == gridDim.x - 1) {
        sync[0] = 0u;
        sync[1] = 0u;
        sync[2] = 0u;
    }
}

// ---- phase A -----------------------------------------------------------------------------------
// Sec. 2.3 jump test from the one-sided differences dp = h+ - h, dm = h - h-
__device__ __forceinline__ bool jump_pair(float dp, float dm, float thr)
{
    return fabsf(dp - dm) > thr * fmaxf(fabsf(dp), fabsf(dm));
}

__device__ __forceinline__ void store_rec(int nc, void *rec, int i, const float h[3], unsigned bits)
{
    if (nc == 1)
        reinterpret_cast<float2 *>(rec)[i] = make_float2(h[0], __uint_as_float(bits));
    else
        reinterpret_cast<float4 *>(rec)[i] = make_float4(h[0], h[1], nc > 2 ? h[2] : 0.f, __uint_as_float(bits));
}
// the periodic images of node (x, y) that lie within reach of the far side
__device__ __forceinline__ void store_images(int nc, void *rec, int n0, int n1, int x, int y, const float h[3],
                                             unsigned bits)
{
    const int pitch = n0 + REC_LO + REC_HI, i = y * pitch + x;
    const int wx = x < REC_HI ? n0 : (x >= n0 - REC_LO ? -n0 : 0), wy = y < REC_HI ? n1 : (y >= n1 - REC_LO ? -n1 : 0);
    if (wx != 0) store_rec(nc, rec, i + wx, h, bits);
    if (wy != 0) store_rec(nc, rec, i + wy * pitch, h, bits);
    if (wx != 0 && wy != 0) store_rec(nc, rec, i + wx + wy * pitch, h, bits);
}

// A warp takes GCOLS columns (its outer lanes hold the neighbours) and GROWS rows.  Its column values
// are all loaded up front; the differences along x come from a shuffle each (the forward difference
// of a lane is the backward one of the next), along y from the row before.  BORDER: the item touches
// the edge of the grid, where rows and columns wrap and nodes have images.
template <int NF, bool BORDER>
__device__ __forceinline__ void flag_item(const GatherArgs &A, int xs, int y0, bool limit)
{
    const TileArgs &a = A.t;
    const int n0 = a.n0, n1 = a.n1, lane = threadIdx.x & 31, x = xs - 1 + lane;
    const int pitch = n0 + REC_LO + REC_HI;
    const bool store = lane >= 1 && lane <= GCOLS && (!BORDER || x < n0);
    unsigned o[GROWS + 2];
    if (BORDER) {
        const unsigned xw = (unsigned)wrap_idx(x, n0);
#pragma unroll
        for (int k = 0; k < GROWS + 2; ++k) {
            const int y = min(y0 - 1 + k, n1);  // none past the first image row
            o[k] = (unsigned)(y < 0 ? n1 - 1 : (y >= n1 ? 0 : y)) * (unsigned)n0 + xw;
        }
    } else {
        o[0] = (unsigned)(y0 - 1) * (unsigned)n0 + (unsigned)x;
#pragma unroll
        for (int k = 1; k < GROWS + 2; ++k) o[k] = o[k - 1] + (unsigned)n0;
    }
#pragma unroll
    for (int q = 0; q < rec_groups(NF); ++q) {
        const int nc = in_rec(NF, q);
        float h[3][GROWS + 2];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < GROWS + 2; ++k) h[c][k] = c < nc ? __ldg(a.in[3 * q + (c < nc ? c : 0)] + o[k]) : 0.f;
        int i = y0 * pitch + x;
#pragma unroll
        for (int k = 1; k <= GROWS; ++k) {
            unsigned b = 0u;
            if (limit) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if (c >= nc) continue;
                    const float dp = __shfl_down_sync(0xffffffffu, h[c][k], 1) - h[c][k];
                    const float dm = __shfl_up_sync(0xffffffffu, dp, 1);
                    const bool hit =
                        jump_pair(dp, dm, a.thr) | jump_pair(h[c][k + 1] - h[c][k], h[c][k] - h[c][k - 1], a.thr);
                    b |= hit ? 1u << c : 0u;
                }
            }
            const float v[3] = {h[0][k], h[1][k], h[2][k]};
            if (store && (!BORDER || y0 + k - 1 < n1)) {
                store_rec(nc, A.rec[q], i, v, b);
                if (BORDER) store_images(nc, A.rec[q], n0, n1, x, y0 + k - 1, v, b);
            }
            i += pitch;
        }
    }
}

template <int NF>
__device__ __forceinline__ void flag_records(const GatherArgs &A, int item, bool limit)
{
    if (item >= A.nflag) return;
    const int chunk = item / A.strips;
    const int xs = (item - chunk * A.strips) * GCOLS, y0 = chunk * GROWS;
    // (the outer lanes' columns xs - 1 and xs + GCOLS and the rows y0 - 1 and y0 + GROWS are read too)
    const bool border = xs < REC_HI || xs + GCOLS >= A.t.n0 - REC_LO || y0 < REC_HI || y0 + GROWS >= A.t.n1 - REC_LO;
    if (border)
        flag_item<NF, true>(A, xs, y0, limit);
    else
        flag_item<NF, false>(A, xs, y0, limit);
}

// ---- phase B -----------------------------------------------------------------------------------
// (x, y) within a period of the grid, wrapped into it
__device__ __forceinline__ void wrap_cell(int x, int y, int n0, int n1, int &wx, int &wy)
{
    wx = x;
    wy = y;
    if ((unsigned)x >= (unsigned)n0 || (unsigned)y >= (unsigned)n1) {
        wx = wrap_near(x, n0);
        wy = wrap_near(y, n1);
    }
}

// displacements of the four vertices of the element with lower corner (x, y), wrapped into the grid
__device__ __forceinline__ void load_quad(const TileArgs &a, int x, int y, float2 d[4])
{
    const float2 *D = reinterpret_cast<const float2 *>(a.D);
    const unsigned i = (unsigned)y * (unsigned)a.n0 + (unsigned)x;
    if (x < a.n0 - 1 && y < a.n1 - 1) {
        const float2 *p = D + i, *q = D + (i + (unsigned)a.n0);
        d[0] = __ldg(p);
        d[1] = __ldg(p + 1);
        d[2] = __ldg(q);
        d[3] = __ldg(q + 1);
    } else {
        const unsigned xr = x == a.n0 - 1 ? 0u : (unsigned)x + 1u, yu = y == a.n1 - 1 ? 0u : ((unsigned)y + 1u) * (unsigned)a.n0;
        d[0] = __ldg(D + i);
        d[1] = __ldg(D + (i - (unsigned)x + xr));
        d[2] = __ldg(D + (yu + (unsigned)x));
        d[3] = __ldg(D + (yu + xr));
    }
}

// eq. (multiZ) for the NC fields of a group whose 4x4 taps start at record r: the cubic sums and the OR
// of the taps' flags; a flagged field takes the bilinear sum over the element's own vertices instead
// (Sec. 2.3; few targets, so it is formed only where a lane of the warp needs it).  Every product and
// sum is rounded in the order of the other 2-D kernels (rows, then the column): the same bits.
__device__ __forceinline__ float field_of(const float4 &t, int c) { return c == 0 ? t.x : (c == 1 ? t.y : t.z); }
__device__ __forceinline__ float field_of(const float2 &t, int) { return t.x; }
__device__ __forceinline__ unsigned rec_flags(const float4 &t) { return __float_as_uint(t.w); }
__device__ __forceinline__ unsigned rec_flags(const float2 &t) { return __float_as_uint(t.y); }

template <int NF, int G>
__device__ __forceinline__ void target_group(const GatherArgs &A, unsigned jj, int o, const float wc[2][4], float xi0,
                                             float xi1, bool limit, unsigned &nlin)
{
    constexpr int NC = in_rec(NF, G);
    using T = typename std::conditional<NC == 1, float2, float4>::type;
    const TileArgs &a = A.t;
    const int pitch = a.n0 + REC_LO + REC_HI;
    const T *r0 = reinterpret_cast<const T *>(A.rec[G]) + o, *r = r0;
    float v[NC];
    unsigned bits = 0u;
#pragma unroll
    for (int c = 0; c < NC; ++c) v[c] = 0.f;
#pragma unroll
    for (int ky = 0; ky < 4; ++ky) {
        const T t0 = r[0], t1 = r[1], t2 = r[2], t3 = r[3];
        bits |= rec_flags(t0) | rec_flags(t1) | rec_flags(t2) | rec_flags(t3);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            float q = __fmul_rn(wc[0][0], field_of(t0, c));
            q = __fmaf_rn(wc[0][1], field_of(t1, c), q);
            q = __fmaf_rn(wc[0][2], field_of(t2, c), q);
            q = __fmaf_rn(wc[0][3], field_of(t3, c), q);
            v[c] = __fmaf_rn(wc[1][ky], q, v[c]);
        }
        r += pitch;
    }
    const unsigned lin = (a.max_order == 0 ? 7u : (limit ? bits : 0u)) & ((1u << NC) - 1u);
    if (lin) {
        const T *q = r0 + pitch + 1;
        const T t0 = q[0], t1 = q[1], t2 = q[pitch], t3 = q[pitch + 1];
        const float u0 = 1.f - xi0, v0 = 1.f - xi1;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float a0 = __fmaf_rn(xi0, field_of(t1, c), __fmul_rn(u0, field_of(t0, c)));
            const float a1 = __fmaf_rn(xi0, field_of(t3, c), __fmul_rn(u0, field_of(t2, c)));
            const float l = __fmaf_rn(xi1, a1, __fmul_rn(v0, a0));
            v[c] = (lin >> c) & 1u ? l : v[c];
        }
        nlin += __popc(lin);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) a.out[3 * G + c][jj] = v[c];
}

// sums of a target in the element with lower corner (ex, ey), wrapped into the grid
template <int NF>
__device__ __forceinline__ unsigned target_sums(const GatherArgs &A, unsigned jj, int ex, int ey, float xi0, float xi1,
                                                bool limit)
{
    float wc[2][4];
    cubic_weights(xi0, wc[0]);
    cubic_weights(xi1, wc[1]);
    unsigned nlin = 0u;
    const int o = (ey - 1) * (A.t.n0 + REC_LO + REC_HI) + (ex - 1);
    target_group<NF, 0>(A, jj, o, wc, xi0, xi1, limit, nlin);
    if constexpr (rec_groups(NF) > 1) target_group<NF, 1>(A, jj, o, wc, xi0, xi1, limit, nlin);
    return nlin;
}

// refined start of a target from s = j - D_j in element (cx, cy) with vertex displacements d: one
// fixed-point step s <- j - D(s), D bilinear over the element
__device__ __forceinline__ void refine(int jx, int jy, float2 s, float fsx, float fsy, const float2 d[4], int &ex, int &ey)
{
    const float fx = s.x - fsx, fy = s.y - fsy;
    const float bx = fmaf(fx, d[1].x - d[0].x, d[0].x), by = fmaf(fx, d[1].y - d[0].y, d[0].y);
    const float dx = fmaf(fy, fmaf(fx, d[3].x - d[2].x, d[2].x) - bx, bx);
    const float dy = fmaf(fy, fmaf(fx, d[3].y - d[2].y, d[2].y) - by, by);
    const float rx = (float)jx - dx, ry = (float)jy - dy;
    if (fabsf(rx - s.x) < 4.f && fabsf(ry - s.y) < 4.f) {  // false for NaN
        ex = (int)floorf(rx);
        ey = (int)floorf(ry);
    }
}

// One FP32 inversion of element (ex, ey) with vertex displacements d (the arithmetic of the tile
// kernels' walk_window)
__device__ __forceinline__ int invert_element(const TileArgs &a, int jx, int jy, int ex, int ey, const float2 d[4],
                                              float xf[3], int &iters, bool &degen)
{
    const float rx0 = (float)(ex - jx), rx1 = rx0 + 1.f, ry0 = (float)(ey - jy), ry1 = ry0 + 1.f;  // exact
    float P[8][3];
    P[0][0] = rx0 + d[0].x;
    P[0][1] = ry0 + d[0].y;
    P[1][0] = rx1 + d[1].x;
    P[1][1] = ry0 + d[1].y;
    P[2][0] = rx0 + d[2].x;
    P[2][1] = ry1 + d[2].y;
    P[3][0] = rx1 + d[3].x;
    P[3][1] = ry1 + d[3].y;
    int it = 0;
    const int st = newton_solve2<float>(P, a.max_iter, SL_NEWTON_TOL_F32, xf, &it, &degen);
    iters += it;
    return st;
}

// The FP64 re-solve of a failed or nearly degenerate FP32 inversion, with its sums (that of slow_target)
template <int NF>
__device__ __noinline__ TargetOut resolve_target(const TileArgs &a, bool limit, unsigned jj, int jx, int jy, int ex, int ey)
{
    TargetOut r = {ST_OK, 0, 0, 1, 0};
    const Win none = {0, 0, 0, 0};
    double xd[3] = {0.0, 0.0, 0.0};
    bool degen = false;
    r.st = walk2<double>(a, none, nullptr, jx, jy, ex, ey, xd, r.hops, r.iters, degen);
    if (r.st != ST_OK) {
#pragma unroll
        for (int f = 0; f < NF; ++f) a.out[f][jj] = __ldg(a.in[f] + jj);
        return r;
    }
    unsigned lin_mask = a.max_order == 0 ? 0xffu : 0u;
    if (limit) lin_mask = box_flags_global(a, ex, ey);
    r.nlin = __popc(lin_mask & ((1u << NF) - 1u));
    interp_global(a, jj, ex, ey, (float)xd[0], (float)xd[1], lin_mask);
    return r;
}

// The general path of one target, out of line: walks of several hops, displacements of a period, and the
// FP64 re-solve.  The walk is walk2<float>'s, hop by hop, with the records' sums at its end, so that a
// target that fails goes on to its FP64 walk at once.  (Fields torn by a solid-body rotation, whose failing
// walks of 55 hops set the launch's length, 200^2 x 3 / 1024^2 x 3: 539 / 460 us; repeating the FP32 walk in
// slow_target 1125 / 966; tiles 704 / 621.)
template <int NF>
__device__ __forceinline__ TargetOut general_target(const GatherArgs &A, int jx, int jy, bool limit)
{
    const TileArgs &a = A.t;
    const unsigned jj = (unsigned)jy * (unsigned)a.n0 + (unsigned)jx;
    const float2 dj = __ldg(reinterpret_cast<const float2 *>(a.D) + jj);
    const float2 s = start_point(jx, jy, dj);
    const float fsx = floorf(s.x), fsy = floorf(s.y);
    const int cx = (int)fsx, cy = (int)fsy;
    int ex = cx, ey = cy;
    float2 d[4];
    // a displacement of a period or more starts from floor(s), as on the tiled kernel's global path
    if (fabsf(dj.x) < (float)a.n0 && fabsf(dj.y) < (float)a.n1) {
        load_quad(a, wrap_idx(cx, a.n0), wrap_idx(cy, a.n1), d);
        refine(jx, jy, s, fsx, fsy, d, ex, ey);
    }
    const float slack = SL_SLACK_F32;
    TargetOut r = {ST_OK, 0, 0, 0, 0};
    CycleCheck cyc;
    cyc.start(ex, ey, 0);
    int st = ST_LOCATE, wx = 0, wy = 0;
    bool degen = false;
    float xf[3];
#pragma unroll 1
    for (int hop = 0; hop < a.walk_max; ++hop) {
        wx = wrap_idx(ex, a.n0);
        wy = wrap_idx(ey, a.n1);
        load_quad(a, wx, wy, d);
        r.hops += 1;
        st = invert_element(a, jx, jy, ex, ey, d, xf, r.iters, degen);
        if (!(finite_t(xf[0]) && finite_t(xf[1]))) {
            if (st == ST_OK) st = ST_NEWTON;
            break;
        }
        const bool lo0 = xf[0] < -slack, hi0 = xf[0] > 1.f + slack;
        const bool lo1 = xf[1] < -slack, hi1 = xf[1] > 1.f + slack;
        if (!(lo0 || hi0 || lo1 || hi1)) break;
        st = ST_LOCATE;
        ex += lo0 ? -1 : (hi0 ? 1 : 0);
        ey += lo1 ? -1 : (hi1 ? 1 : 0);
        if (cyc.step(ex, ey, 0)) break;
    }
    if (st == ST_OK && !degen) {
        r.nlin = (int)target_sums<NF>(A, jj, wx, wy, xf[0], xf[1], limit);
        return r;
    }
    const bool lost = st == ST_LOCATE || st == ST_FOLD;
    TargetOut q = resolve_target<NF>(a, limit, jj, jx, jy, lost ? cx : ex, lost ? cy : ey);
    q.hops += r.hops;
    q.iters += r.iters;
    return q;
}

// ... and its counters, added one target at a time to the SM's copy, so that the loop over the targets
// carries none of them in registers
template <int NF>
__device__ __noinline__ void general_path(const GatherArgs &A, int jx, int jy, bool limit)
{
    const TargetOut r = general_target<NF>(A, jx, jy, limit);
    unsigned smid;
    asm("mov.u32 %0, %%smid;" : "=r"(smid));
    DevCounters *g = A.t.stripes + (smid % SL_COUNTER_STRIPES);
    atomicAdd(&g->targets, 1ull);
    atomicAdd(&g->hops_sum, (unsigned long long)r.hops);
    atomicMax(&g->hops_max, (unsigned long long)r.hops);
    atomicAdd(&g->iters_sum, (unsigned long long)r.iters);
    atomicMax(&g->iters_max, (unsigned long long)r.iters);
    if (r.f64) atomicAdd(&g->newton_f64, 1ull);
    if (r.st == ST_OK) {
        if (r.nlin > 0) atomicAdd(&g->order_hist[0], (unsigned long long)r.nlin);
        if (r.nlin < NF) atomicAdd(&g->order_hist[1], (unsigned long long)(NF - r.nlin));
    } else {
        atomicAdd(r.st == ST_LOCATE ? &g->fail_locate : r.st == ST_NEWTON ? &g->fail_newton : &g->fail_fold, 1ull);
    }
}

// Where one target's departure point lies: refined start, up to A.hops elements; false where the target
// needs the general path.  (wx, wy) is the element's lower corner wrapped into the grid.
struct Located {
    int wx, wy, hops, iters;
    float xi0, xi1;
};
__device__ __forceinline__ bool locate(const GatherArgs &A, int jx, int jy, unsigned jj, Located &r)
{
    const TileArgs &a = A.t;
    const float2 dj = __ldg(reinterpret_cast<const float2 *>(a.D) + jj);
    const float2 s = make_float2((float)jx - dj.x, (float)jy - dj.y);
    const float fsx = floorf(s.x), fsy = floorf(s.y);
    // less than a period away (false for NaN)
    if (!(fabsf(dj.x) < A.reach0 && fabsf(dj.y) < A.reach1)) return false;
    const int cx = (int)fsx, cy = (int)fsy;
    int ex = cx, ey = cy;
    float2 d[4];
    wrap_cell(ex, ey, a.n0, a.n1, r.wx, r.wy);
    load_quad(a, r.wx, r.wy, d);
    refine(jx, jy, s, fsx, fsy, d, ex, ey);
    // (a refined start lies within 4 cells of the first one, itself within n - 11 of the target; the
    // walk may step GHOPS - 1 more)
    if (ex != cx || ey != cy) {
        wrap_cell(ex, ey, a.n0, a.n1, r.wx, r.wy);
        load_quad(a, r.wx, r.wy, d);
    }
    const float slack = SL_SLACK_F32;
    r.iters = r.hops = 0;
    for (;;) {
        // Newton from the solution of the linear part: the arithmetic of newton_solve2<float> (whose
        // early exits become conditions tested at the end)
        const float rx0 = (float)(ex - jx), rx1 = rx0 + 1.f, ry0 = (float)(ey - jy), ry1 = ry0 + 1.f;  // exact
        const float p0x = rx0 + d[0].x, p0y = ry0 + d[0].y, p1x = rx1 + d[1].x, p1y = ry0 + d[1].y;
        const float p2x = rx0 + d[2].x, p2y = ry1 + d[2].y, p3x = rx1 + d[3].x, p3y = ry1 + d[3].y;
        const float ax = p1x - p0x, ay = p1y - p0y, bx = p2x - p0x, by = p2y - p0y;
        const float exx = p3x - p1x - p2x + p0x, eyy = p3y - p1y - p2y + p0y;
        float det = diff_prod(ax, by, bx, ay);
        bool good = det > 0.f;
        float inv = recip_t(det);
        float xs = __fmul_rn(-diff_prod(p0x, by, p0y, bx), inv);
        float xt = __fmul_rn(-diff_prod(ax, p0y, ay, p0x), inv);
        float j11, j21, j12, j22, step;
        int it = 0;
        do {
            j11 = __fmaf_rn(xt, exx, ax);
            j21 = __fmaf_rn(xt, eyy, ay);
            j12 = __fmaf_rn(xs, exx, bx);
            j22 = __fmaf_rn(xs, eyy, by);
            const float st = __fmul_rn(xs, xt);
            const float gx = __fmaf_rn(st, exx, __fmaf_rn(xt, bx, __fmaf_rn(xs, ax, p0x)));
            const float gy = __fmaf_rn(st, eyy, __fmaf_rn(xt, by, __fmaf_rn(xs, ay, p0y)));
            det = diff_prod(j11, j22, j12, j21);
            good = good && det > 0.f;
            inv = recip_t(det);
            const float d0 = __fmul_rn(diff_prod(gx, j22, gy, j12), inv);
            const float d1 = __fmul_rn(diff_prod(j11, gy, j21, gx), inv);
            xs -= d0;
            xt -= d1;
            step = fmaxf(fabsf(d0), fabsf(d1));
            ++it;
        } while (step > SL_NEWTON_TOL_F32 && it < a.max_iter);
        const bool degen =
            det < __fmul_rn(SL_DEGENERATE, __fmul_rn(fabsf(j11) + fabsf(j21), fabsf(j12) + fabsf(j22)));
        if (!good || degen || !(step <= SL_NEWTON_TOL_F32)) return false;
        r.iters += it;
        ++r.hops;
        r.xi0 = xs;
        r.xi1 = xt;
        if (xs >= -slack && xs <= 1.f + slack && xt >= -slack && xt <= 1.f + slack) return true;
        if (r.hops == A.hops) return false;
        ex += xs < -slack ? -1 : (xs > 1.f + slack ? 1 : 0);
        ey += xt < -slack ? -1 : (xt > 1.f + slack ? 1 : 0);
        wrap_cell(ex, ey, a.n0, a.n1, r.wx, r.wy);
        load_quad(a, r.wx, r.wy, d);
    }
}

// The tiles b, b + G, .. of CTA b of G in turn: this thread's node (tiles numbered down the columns)
struct TileWalk {
    int jx, jy, ty;
    __device__ __forceinline__ explicit TileWalk(const GatherArgs &A)
    {
        const int tx = (int)blockIdx.x / A.tiles_y;
        ty = (int)blockIdx.x - tx * A.tiles_y;
        jx = tx * GTX + (int)(threadIdx.x & 31);
    }
    __device__ __forceinline__ int y() const { return ty * GTY + (int)(threadIdx.x >> 5); }
    __device__ __forceinline__ bool valid(const GatherArgs &A) const { return jx < A.t.n0 && y() < A.t.n1; }
    __device__ __forceinline__ bool end(const GatherArgs &A) const
    {
        return jx - (int)(threadIdx.x & 31) >= A.t.n0;
    }
    __device__ __forceinline__ void next(const GatherArgs &A)
    {
        ty += A.step_y;
        jx += A.step_x;
        if (ty >= A.tiles_y) {
            ty -= A.tiles_y;
            jx += GTX;
        }
    }
};

// eq. (vel): the next step's trajectories of the CTA's nodes, the swirl's for two tiles' nodes at a time
// on packed FP32x2 arithmetic
__device__ __forceinline__ void integrate_tiles(const GatherArgs &A, const VelArgs<float> &vn)
{
    float2 *Dn = reinterpret_cast<float2 *>(A.t.D_next);
    const unsigned n0 = (unsigned)A.t.n0;
    TileWalk w(A);
    if (vn.kind == SL_VEL_SWIRL2D && vn.integrator == SL_RK4 && vn.substeps == 1) {
#pragma unroll 1
        while (!w.end(A)) {
            const int xa = w.jx, ya = w.y();
            const bool ina = w.valid(A);
            w.next(A);
            const int xb = w.jx, yb = w.y();
            const bool inb = w.valid(A);
            w.next(A);
            if (!ina && !inb) continue;
            const float2 X = make_float2(node_position(vn.lo[0], xa, vn.dx[0]), node_position(vn.lo[0], xb, vn.dx[0]));
            const float2 Y = make_float2(node_position(vn.lo[1], ya, vn.dx[1]), node_position(vn.lo[1], yb, vn.dx[1]));
            float2 Dx, Dy;
            rk4_swirl_pair(vn, X, Y, Dx, Dy);
            if (ina) Dn[(unsigned)ya * n0 + (unsigned)xa] = make_float2(Dx.x, Dy.x);
            if (inb) Dn[(unsigned)yb * n0 + (unsigned)xb] = make_float2(Dx.y, Dy.y);
        }
        return;
    }
#pragma unroll 1
    for (; !w.end(A); w.next(A)) {
        if (!w.valid(A)) continue;
        float X[3] = {node_position(vn.lo[0], w.jx, vn.dx[0]), node_position(vn.lo[1], w.y(), vn.dx[1]), 0.f}, d[3];
        trajectory_cells<float, 2>(vn, X, d);
        Dn[(unsigned)w.y() * n0 + (unsigned)w.jx] = make_float2(d[0], d[1]);
    }
}

// A CTA whose wait ran out: its targets from w on keep their old values.
template <int NF, bool FUSED>
__device__ __noinline__ void keep_old(const GatherArgs &A, TileWalk w)
{
    const TileArgs &a = A.t;
    if (threadIdx.x == 0) atomicAdd(A.timeouts, 1ull);
    for (; !w.end(A); w.next(A)) {
        if (!w.valid(A)) continue;
        const unsigned jj = (unsigned)w.y() * (unsigned)a.n0 + (unsigned)w.jx;
        for (int f = 0; f < NF; ++f) a.out[f][jj] = a.in[f][jj];
        if (FUSED && a.D_next != nullptr && a.carried)
            reinterpret_cast<float2 *>(a.D_next)[jj] =
                make_float2(a.csc[0] * a.in[a.vf[0]][jj], a.csc[1] * a.in[a.vf[1]][jj]);
    }
}

template <int NF, bool FUSED>
__global__ void __launch_bounds__(GNT, GMINB) gather2d_kernel(const __grid_constant__ GatherArgs A, const VelArgs<float> vn)
{
    __shared__ int s_item, s_ok;
    __shared__ unsigned s_cnt[GNT / 32][6];
    const TileArgs &a = A.t;
    const bool limit = a.max_order >= 1 && a.thr >= 0.f;
    // phase A: claim after claim (the next one is claimed while one is computed)
    unsigned done = 0u;
    int item = 0;
    if (threadIdx.x == 0) s_item = (int)atomicAdd(A.sync, 1u);
    __syncthreads();
    for (item = s_item; item < A.nclaim; ++done) {
        int nx = 0;
        if (threadIdx.x == 0) nx = (int)atomicAdd(A.sync, 1u);
        flag_records<NF>(A, item * (GNT / 32) + (int)(threadIdx.x >> 5), limit);
        __syncthreads();  // (every thread has read s_item)
        if (threadIdx.x == 0) s_item = nx;
        __syncthreads();
        item = s_item;
    }
    if (threadIdx.x == 0 && done) {
        __threadfence();
        atomicAdd(A.sync + 1, done);
    }
    if (FUSED && a.D_next != nullptr && !a.carried) integrate_tiles(A, vn);
    unsigned nfast = 0u, nlin = 0u;
    int hops = 0, hops_max = 0, iters = 0, iters_max = 0;
    bool waited = false;  // the records are first needed after the first target is located
#pragma unroll 1
    for (TileWalk w(A); !w.end(A); w.next(A)) {
        const bool valid = w.valid(A);
        const int jy = w.y();
        const unsigned jj = (unsigned)jy * (unsigned)a.n0 + (unsigned)w.jx;
        Located r;
        const bool ok = valid && locate(A, w.jx, jy, jj, r);
        if (!waited) {
            waited = true;
            if (!wait_items(A.sync, (unsigned)A.nclaim, &s_ok)) {
                keep_old<NF, FUSED>(A, w);
                break;
            }
        }
        if (ok) {
            nlin += target_sums<NF>(A, jj, r.wx, r.wy, r.xi0, r.xi1, limit);
            nfast += 1;
            hops += r.hops;
            hops_max = max(hops_max, r.hops);
            iters += r.iters;
            iters_max = max(iters_max, r.iters);
        } else if (valid) {
            general_path<NF>(A, w.jx, jy, limit);
        }
        if (FUSED && a.D_next != nullptr && a.carried && valid) {
            // Sec. 3.2: D = dt u / dx from the remapped velocity (this thread's own outputs)
            reinterpret_cast<float2 *>(a.D_next)[jj] =
                make_float2(a.csc[0] * a.out[a.vf[0]][jj], a.csc[1] * a.out[a.vf[1]][jj]);
        }
    }
    leave(A.sync);
    // the CTA's counters: summed over its warps in shared memory, one set of atomics per CTA (a set per
    // warp cost 3 us of a 34 us launch)
    const unsigned wn = warp_sum(nfast), wh = warp_sum((unsigned)hops), wi = warp_sum((unsigned)iters),
                   wl = warp_sum(nlin), wmh = warp_max((unsigned)hops_max), wmi = warp_max((unsigned)iters_max);
    if ((threadIdx.x & 31) == 0) {
        unsigned *c = s_cnt[threadIdx.x >> 5];
        c[0] = wn;
        c[1] = wh;
        c[2] = wi;
        c[3] = wl;
        c[4] = wmh;
        c[5] = wmi;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        unsigned v = 0u;
#pragma unroll
        for (int k = 0; k < GNT / 32; ++k) v = threadIdx.x < 4 ? v + s_cnt[k][threadIdx.x] : max(v, s_cnt[k][threadIdx.x]);
        unsigned smid;
        asm("mov.u32 %0, %%smid;" : "=r"(smid));
        DevCounters *g = a.stripes + (smid % SL_COUNTER_STRIPES);
        const unsigned long long u = v;
        const unsigned nf = __shfl_sync(0x3fu, v, 0);
        if (threadIdx.x == 0) atomicAdd(&g->targets, u);
        if (threadIdx.x == 1) atomicAdd(&g->hops_sum, u);
        if (threadIdx.x == 2) atomicAdd(&g->iters_sum, u);
        if (threadIdx.x == 3) {
            atomicAdd(&g->order_hist[0], u);
            atomicAdd(&g->order_hist[1], (unsigned long long)NF * nf - u);
        }
        if (threadIdx.x == 4) atomicMax(&g->hops_max, u);
        if (threadIdx.x == 5) atomicMax(&g->iters_max, u);
    }
}

}  // namespace
