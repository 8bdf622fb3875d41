// sl_kernels.cu -- the plain kernels of the FSL step (arXiv:1410.2817): one thread per node with
// gathers straight from global memory (read-only cache).  They serve every dtype and dimension;
// the FP64 instantiation is the single-grid FP64 path, and every kernel here can write per-target
// diagnostics for parity checks.
//
//   flags_kernel          Sec. 2.3 jump criterion (bit f of a byte per node)
//   advect_kernel         eq. (vel), one classical RK4 step per Lagrangian node
//   remap_generic_kernel  Sec. 2.2 element search + Newton inversion, Sec. 2.3 order reduction,
//                         eq. (multiZ) tensor Z-spline sum
//   moments_*             Sec. 3.1 discrete moments, FP64 accumulation in a fixed order
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "sl_internal.h"
#include "sl_newton64.cuh"

// ------------------------------------------------------------------------------------------------
// argument builders
// ------------------------------------------------------------------------------------------------
template <typename T>
GridArgs<T> make_grid_args(const sl_grid *g)
{
    GridArgs<T> a;
    for (int q = 0; q < 3; ++q) a.n[q] = (int)(q < g->dim ? g->n[q] : 1);
    a.N = (long long)g->N;
    a.nfields = g->nfields;
    a.max_order = g->desc.max_order;
    a.threshold = (T)g->desc.limiter_threshold;
    a.newton_max_iter = g->desc.newton_max_iter;
    a.walk_max = g->desc.walk_max;
    a.walk_start = g->desc.walk_start;
    a.tol = sizeof(T) == 8 ? (T)1e-14 : (T)SL_NEWTON_TOL_F32;
    a.slack = sizeof(T) == 8 ? (T)1e-12 : (T)SL_SLACK_F32;
    return a;
}

template <typename T>
VelArgs<T> make_vel_args(const sl_grid *g, double t, double dt)
{
    VelArgs<T> v;
    memset(&v, 0, sizeof(v));
    v.kind = g->desc.velocity_kind;
    v.nmodes = (v.kind == SL_VEL_FOURIER2D || v.kind == SL_VEL_FOURIER3D) ? (int)g->vel_params[0] : 0;
    v.integrator = g->desc.integrator;
    v.substeps = g->desc.trajectory_substeps > 0 ? g->desc.trajectory_substeps : 1;
    for (int q = 0; q < SL_MAX_VEL_PARAMS; ++q) v.p[q] = (T)g->vel_params[q];
    v.pairs = sizeof(T) == 4 && v.kind == SL_VEL_FOURIER2D && fourier2d_pairs(v.integrator, v.substeps, dt, g->vel_params);
    if (v.kind == SL_VEL_SWIRL2D || v.kind == SL_VEL_DEFORM3D) {
        stage_time_factors<T>(t, dt, v.substeps, v.integrator, g->vel_params[0], v.ct);
    }
    for (int q = 0; q < 3; ++q) {
        v.lo[q] = (T)g->desc.lo[q];
        v.dx[q] = (T)g->dx[q];
        v.inv_dx[q] = (T)(1.0 / g->dx[q]);
    }
    v.dt = (T)dt;
    if (g->trig != nullptr && sizeof(T) == g->tsize)
        for (int q = 0; q < g->dim; ++q) v.sc[q] = (const T *)g->trig + g->trig_off[q];
    return v;
}

// sin(pi x), cos(pi x) at every node coordinate of every axis, computed by the kernels' own
// node_position and sincospi_t (so a table entry has the bits the kernels compute)
template <typename T>
__global__ void __launch_bounds__(256) trig_table_kernel(VelArgs<T> v, int dim, int n0, int n1, int n2, T *tab)
{
    const int n[3] = {n0, n1, n2};
    long long base = 0;
    for (int a = 0; a < dim; ++a) {
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n[a]; k += gridDim.x * blockDim.x) {
            T sn, cs;
            sincospi_t(node_position(v.lo[a], k, v.dx[a]), &sn, &cs);
            tab[base + 2 * k] = sn;
            tab[base + 2 * k + 1] = cs;
        }
        base += 2LL * n[a];
    }
}

cudaError_t launch_trig_tables(const sl_grid *g, cudaStream_t s)
{
    if (g->trig == nullptr) return cudaSuccess;
    const int n1 = g->dim > 1 ? (int)g->n[1] : 0, n2 = g->dim > 2 ? (int)g->n[2] : 0;
    if (g->dtype == SL_F64)
        trig_table_kernel<double><<<64, 256, 0, s>>>(make_vel_args<double>(g, 0.0, 1.0), g->dim, (int)g->n[0], n1, n2,
                                                     (double *)g->trig);
    else
        trig_table_kernel<float><<<64, 256, 0, s>>>(make_vel_args<float>(g, 0.0, 1.0), g->dim, (int)g->n[0], n1, n2,
                                                    (float *)g->trig);
    return cudaGetLastError();
}

// One block per `threads` nodes (the kernels also loop grid-stride, so any count is correct).
// Short-lived blocks let the block scheduler interleave work of higher-priority streams; the cap
// only guards the grid-size limit.
int grid_stride_blocks(const sl_grid *g, long long work, int threads)
{
    (void)g;
    long long b = (work + threads - 1) / threads;
    if (b > (1LL << 30)) b = 1LL << 30;
    if (b < 1) b = 1;
    return (int)b;
}

template GridArgs<double> make_grid_args<double>(const sl_grid *);
template GridArgs<float> make_grid_args<float>(const sl_grid *);
template VelArgs<double> make_vel_args<double>(const sl_grid *, double, double);
template VelArgs<float> make_vel_args<float>(const sl_grid *, double, double);

// ------------------------------------------------------------------------------------------------
// node index helpers
// ------------------------------------------------------------------------------------------------
template <int DIM>
__device__ __forceinline__ void node_coords(long long i, const int n[3], int k[3])
{
    // a grid has fewer than 2^31 nodes: 32-bit divisions
    const unsigned u = (unsigned)i, r = u / (unsigned)n[0];
    k[0] = (int)(u - r * (unsigned)n[0]);
    if (DIM == 3) {
        k[2] = (int)(r / (unsigned)n[1]);
        k[1] = (int)(r - (unsigned)k[2] * (unsigned)n[1]);
    } else {
        k[1] = (int)r;
        k[2] = 0;
    }
}

template <int DIM>
__device__ __forceinline__ long long node_index(const int k[3], const int n[3])
{
    long long idx = wrap_idx(k[0], n[0]) + (long long)n[0] * wrap_idx(k[1], n[1]);
    if (DIM == 3) idx += (long long)n[0] * n[1] * wrap_idx(k[2], n[2]);
    return idx;
}

template <typename T>
struct FieldPtrs {
    const T *in[SL_MAX_FIELDS];
    T *out[SL_MAX_FIELDS];
};

// ------------------------------------------------------------------------------------------------
// Sec. 2.3: jump flags
// ------------------------------------------------------------------------------------------------
template <typename T, int DIM>
__global__ void __launch_bounds__(256) flags_kernel(GridArgs<T> g, FieldPtrs<T> f, uint8_t *__restrict__ flags)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N;
         i += (long long)gridDim.x * blockDim.x) {
        unsigned bits = 0;
        if (g.threshold >= T(0)) {
            int k[3];
            node_coords<DIM>(i, g.n, k);
            long long nb[3][2];
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                int kp[3] = {k[0], k[1], k[2]}, km[3] = {k[0], k[1], k[2]};
                kp[a] += 1;
                km[a] -= 1;
                nb[a][0] = node_index<DIM>(km, g.n);
                nb[a][1] = node_index<DIM>(kp, g.n);
            }
            for (int q = 0; q < g.nfields; ++q) {
                const T *h = f.in[q];
                const T h0 = __ldg(h + i);
                bool hit = false;
#pragma unroll
                for (int a = 0; a < DIM; ++a) hit |= jump_test<T>(__ldg(h + nb[a][0]), h0, __ldg(h + nb[a][1]), g.threshold);
                if (hit) bits |= 1u << q;
            }
        }
        flags[i] = (uint8_t)bits;
    }
}

// FP64 2-D flags.  A warp takes 31 columns (lane 0 is the left neighbour of lane 1, whose forward
// difference is lane 1's backward one) and walks `rows` rows up, the forward difference of a row
// being the backward one of the next: two FP64 subtractions per field and node where flags_kernel
// takes four, and the test itself in FP32 (jump_diffs).  1024^2 x 3 fields: 79.8 -> 23.5 us, bound by
// the FP64 pipe still (6.9 FP64 instructions a node).
constexpr int FLAG_COLS = 31, FLAG_ROWS = 8;

template <int NFM>
__global__ void __launch_bounds__(128)
    flags64_kernel(int n0, int n1, int nfields, JumpBounds b, FieldPtrs<double> f, uint8_t *__restrict__ flags,
                   unsigned strips, unsigned nwarps, int rows)
{
    const int lane = threadIdx.x & 31;
    const unsigned warp = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    if (warp >= nwarps) return;
    const unsigned chunk = warp / strips;
    const int x = (int)(warp - chunk * strips) * FLAG_COLS - 1 + lane;
    const int xw = wrap_idx(x, n0), xr = wrap_near(xw + 1, n0);
    const int y0 = (int)chunk * rows, y1 = min(y0 + rows, n1);
    double c[NFM], dy[NFM];
    float fy[NFM];
#pragma unroll
    for (int q = 0; q < NFM; ++q) {
        if (q < nfields) {
            c[q] = __ldg(f.in[q] + (long long)y0 * n0 + xw);
            dy[q] = c[q] - __ldg(f.in[q] + (long long)wrap_near(y0 - 1, n1) * n0 + xw);
            fy[q] = narrow(dy[q]);
        }
    }
    for (int y = y0; y < y1; ++y) {
        const long long row = (long long)y * n0, up = (long long)wrap_near(y + 1, n1) * n0;
        unsigned bits = 0;
#pragma unroll
        for (int q = 0; q < NFM; ++q) {
            if (q < nfields) {
                const double u = __ldg(f.in[q] + up + xw);
                const double dp = __ldg(f.in[q] + row + xr) - c[q], dn = u - c[q];
                const float fp = narrow(dp), fn = narrow(dn);
                const double dm = __shfl_up_sync(0xffffffffu, dp, 1);
                const float fm = __shfl_up_sync(0xffffffffu, fp, 1);
                if (lane > 0 && (jump_diffs(dm, dp, fm, fp, b) || jump_diffs(dy[q], dn, fy[q], fn, b)))
                    bits |= 1u << q;
                c[q] = u;
                dy[q] = dn;
                fy[q] = fn;
            }
        }
        if (lane > 0 && x < n0) flags[row + x] = (uint8_t)bits;
    }
}

// ------------------------------------------------------------------------------------------------
// eq. (vel): RK4 displacement of every Lagrangian node (cell units), stride ds values per node
// ------------------------------------------------------------------------------------------------
template <typename T, int DIM>
__global__ void __launch_bounds__(256) advect_kernel(GridArgs<T> g, VelArgs<T> v, T *__restrict__ D, int ds)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N;
         i += (long long)gridDim.x * blockDim.x) {
        int k[3];
        node_coords<DIM>(i, g.n, k);
        T X[3] = {T(0), T(0), T(0)}, d[3];
#pragma unroll
        for (int a = 0; a < DIM; ++a) X[a] = node_position(v.lo[a], k[a], v.dx[a]);
        trajectory_cells_node<T, DIM>(v, X, k, d);
#pragma unroll
        for (int a = 0; a < DIM; ++a) D[i * ds + a] = d[a];
        if (DIM == 3) D[i * ds + 3] = T(0);
    }
}

// The RK4 step of a 2-D Fourier velocity in FP32, two nodes a thread (rk4_fourier2d_pair): nodes i and
// i + half of the grid.  NT threads a block, G modes at a time.
template <int NT, int G>
__global__ void __launch_bounds__(NT, NT == 256 ? 3 : 1)
    advect_fourier2d_kernel(GridArgs<float> g, VelArgs<float> v, float2 *__restrict__ D, unsigned half)
{
    __shared__ FourierPairs sf;
    __shared__ float4 base[SL_PAIR_MODES][NT];
    sf.load(v, threadIdx.x);
    __syncthreads();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= half) return;
    const unsigned j = i + half < g.N ? i + half : i;
    int a[3], b[3];
    node_coords<2>(i, g.n, a);
    node_coords<2>(j, g.n, b);
    const float2 X = make_float2(node_position(v.lo[0], a[0], v.dx[0]), node_position(v.lo[0], b[0], v.dx[0]));
    const float2 Y = make_float2(node_position(v.lo[1], a[1], v.dx[1]), node_position(v.lo[1], b[1], v.dx[1]));
    float2 Dx, Dy;
    rk4_fourier2d_pair<G>(sf, &base[0][threadIdx.x], NT, X, Y, Dx, Dy);
    D[i] = make_float2(Dx.x, Dy.x);
    if (j != i) D[j] = make_float2(Dx.y, Dy.y);
}

// The swirl's RK4 step in FP64 with as few FP64 instructions as the digits allow (110 per node for
// offsets below 1/128 of the box, against 209 for rk4_trig_from; 1024^2: 410 -> 218 us, the FP64 pipe
// busy 86 % of the time in both).  With S = sin(pi x), C = cos(pi x)
// along each axis the velocity is u = 2 ct Sx^2 (Sy Cy), v = -2 ct Sy^2 (Sx Cx).  The stages work on
// q = (Sx^2 Sy Cy, Sy^2 Sx Cx); the factors 2 ct, the step and pi are folded into the constants that
// turn q into the next stage's angle (A) and into the displacement (B, cell units), prepared on the
// host.  Sines and cosines of the node positions come from the grid's table, those of a stage's
// position from the angle-addition formulas with the Taylor series of the small angle:
// |a| <= pi/128: sin through a^7, cos through a^6 [3e-18]; |a| <= pi/16: a^11, a^12 [1e-19]; larger
// angles take rk4_trig_from.  The comparisons are integer ones on the high words.  A warp with a node whose
// first q promises such an angle takes rk4_trig_from at once (32^2 nodes moved by up to 4 cells:
// rk4_trig_from alone 22.9 us, both in turn 34.0, this 20.1; 1024^2 moved by a fifth of the box 515 / 415).
struct Swirl64 {
    int far;         // high word of the |q| from which on a stage's angle may exceed pi/16
    double A[3];     // angle of stage 2, 3, 4 per q of the stage before
    double Bx[3], By[3];  // displacement per q1, q2 + q3, q4
};

__device__ __forceinline__ bool rotate64(double a, double S, double C, double &s, double &c)
{
    const int h = __double2hiint(a) & 0x7fffffff;
    const double u = a * a;
    double ps, pc;
    if (h < 0x3f9921fb) {  // pi / 128
        ps = fma(u, -1.0 / 5040.0, 1.0 / 120.0);
        pc = fma(u, -1.0 / 720.0, 1.0 / 24.0);
    } else {
        if (h >= 0x3fc921fb) return false;  // pi / 16
        ps = fma(u, -1.0 / 39916800.0, 1.0 / 362880.0);
        pc = fma(u, 1.0 / 479001600.0, -1.0 / 3628800.0);
        ps = fma(u, ps, -1.0 / 5040.0);
        pc = fma(u, pc, 1.0 / 40320.0);
        ps = fma(u, ps, 1.0 / 120.0);
        pc = fma(u, pc, -1.0 / 720.0);
        pc = fma(u, pc, 1.0 / 24.0);
    }
    const double sd = a * fma(u, fma(u, ps, -1.0 / 6.0), 1.0), cd = fma(u, fma(u, pc, -0.5), 1.0);
    s = fma(S, cd, C * sd);
    c = fma(C, cd, -(S * sd));
    return true;
}

__global__ void __launch_bounds__(256)
    advect_swirl64_kernel(GridArgs<double> g, VelArgs<double> v, Swirl64 w, double2 *__restrict__ D)
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, i = t < g.N ? t : (unsigned)g.N - 1u;
    int k[3];
    node_coords<2>(i, g.n, k);
    const double2 X = __ldg(reinterpret_cast<const double2 *>(v.sc[0]) + k[0]);
    const double2 Y = __ldg(reinterpret_cast<const double2 *>(v.sc[1]) + k[1]);
    double sx = X.x, cx = X.y, sy = Y.x, cy = Y.y;
    double qx[4], qy[4];
    bool ok = true;
#pragma unroll
    for (int st = 0; st < 4; ++st) {
        qx[st] = (sx * sx) * (sy * cy);
        qy[st] = (sy * sy) * (sx * cx);
        if (st == 0) {
            const int h = max(__double2hiint(qx[0]) & 0x7fffffff, __double2hiint(qy[0]) & 0x7fffffff);
            ok = !__any_sync(0xffffffffu, h >= w.far);
            if (!ok) break;
        }
        if (st < 3) {
            ok &= rotate64(w.A[st] * qx[st], X.x, X.y, sx, cx);
            ok &= rotate64(-(w.A[st] * qy[st]), Y.x, Y.y, sy, cy);
            if (!ok) break;
        }
    }
    double2 d;
    if (ok) {
        d.x = fma(w.Bx[0], qx[0], fma(w.Bx[1], qx[1] + qx[2], w.Bx[2] * qx[3]));
        d.y = fma(w.By[0], qy[0], fma(w.By[1], qy[1] + qy[2], w.By[2] * qy[3]));
    } else {
        const double P[3] = {node_position(v.lo[0], k[0], v.dx[0]), node_position(v.lo[1], k[1], v.dx[1]), 0.0};
        const double s0[3] = {X.x, Y.x, 0.0}, c0[3] = {X.y, Y.y, 1.0};
        double o[3];
        rk4_trig_from<double, 2>(v, P, s0, c0, o);
        d = make_double2(o[0], o[1]);
    }
    if (t < g.N) D[i] = d;
}

// ------------------------------------------------------------------------------------------------
// Sec. 3.2: the velocity carried by the nodes (Burgers, Du/Dt = 0) is constant along each
// trajectory, so every integrator moves node i by dt u_i: D_i = (dt / dx_a) u_a,i in cell units.
// ------------------------------------------------------------------------------------------------
template <typename T, int DIM>
__global__ void __launch_bounds__(256)
    advect_carried_kernel(long long N, const T *__restrict__ u0, const T *__restrict__ u1, const T *__restrict__ u2,
                          T s0, T s1, T s2, T *__restrict__ D)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        if (DIM == 2) {
            using T2 = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
            T2 d;
            d.x = s0 * __ldg(u0 + i);
            d.y = s1 * __ldg(u1 + i);
            reinterpret_cast<T2 *>(D)[i] = d;
        } else {
            D[i * 4 + 0] = s0 * __ldg(u0 + i);
            D[i * 4 + 1] = s1 * __ldg(u1 + i);
            D[i * 4 + 2] = s2 * __ldg(u2 + i);
            D[i * 4 + 3] = T(0);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.2 element search with Newton inversion; the same walk as the paper's: invert, and while a
// local coordinate is out of range step into the neighbour it points to.
// ------------------------------------------------------------------------------------------------
template <typename TN>
struct WalkParams {
    TN tol, slack;
    int max_iter, walk_max;
};

// Start element (Sec. 2.2): the paper's "opposite the velocity" (the element having Lagrangian node
// j as a vertex on the side opposite its own displacement), or the backward estimate floor(j - D_j).
template <typename T, int DIM>
__device__ __forceinline__ void walk_start_cell(int mode, const int j[3], const T Dj[3], int c[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) c[a] = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        if (mode == SL_START_PAPER) {
            c[a] = j[a] - (Dj[a] > T(0) ? 1 : 0);
        } else if (sizeof(T) == 8) {
            // the same in three FP64 instructions: the conversion saturates, the clamp is an
            // integer one, and only a NaN keeps j
            const unsigned long long b = (unsigned long long)__double_as_longlong((double)Dj[a]) << 1;
            const int s = __double2int_rd(small_int(j[a]) - (double)Dj[a]);
            c[a] = b > 0xffe0000000000000ull ? j[a] : min(max(s, j[a] - 65536), j[a] + 65536);
        } else {
            // clamped so that a garbage displacement cannot overflow the walk's integer steps
            const T s = min_t(max_t(T(j[a]) - Dj[a], T(j[a]) - T(65536)), T(j[a]) + T(65536));
            c[a] = finite_t(s) ? (int)floor_t<T>(s) : j[a];
        }
    }
}

// Sec. 2.2 element search from element c: invert (Newton in precision TN) and, while a local
// coordinate is out of range, step into the neighbour it points to.  On return c is the last
// element tried and xi its local coordinates; *hops and *iters are incremented.
template <typename T, typename TN, int DIM>
__device__ __forceinline__ int walk_global(const WalkParams<TN> &w, const int n[3], const T *__restrict__ D, int ds,
                                           const int j[3], int c[3], TN xi[3], int *hops, int *iters,
                                           bool *degenerate = nullptr)
{
    CycleCheck cyc;
    cyc.start(c[0], c[1], c[2]);
    for (int hop = 0; hop < w.walk_max; ++hop) {
        TN P[8][3];
#pragma unroll
        for (int v = 0; v < (1 << DIM); ++v) {
            int k[3] = {c[0], c[1], c[2]};
#pragma unroll
            for (int a = 0; a < DIM; ++a) k[a] += (v >> a) & 1;
            const long long idx = node_index<DIM>(k, n);
#pragma unroll
            for (int a = 0; a < DIM; ++a) P[v][a] = TN(k[a] - j[a]) + (TN)__ldg(D + idx * ds + a);
        }
        int it = 0;
        const int st = newton_solve<TN, DIM>(P, w.max_iter, w.tol, xi, &it, degenerate);
        *hops += 1;
        *iters += it;
        bool finite = true, inside = true;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            if (!finite_t(xi[a])) finite = false;
            if (!(xi[a] >= -w.slack && xi[a] <= TN(1) + w.slack)) inside = false;
        }
        if (!finite) return st == ST_OK ? ST_NEWTON : st;
        if (inside) return st;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            if (xi[a] < -w.slack)
                c[a] -= 1;
            else if (xi[a] > TN(1) + w.slack)
                c[a] += 1;
        }
        if (cyc.step(c[0], c[1], c[2])) return ST_LOCATE;
    }
    return ST_LOCATE;
}

template <typename T>
struct RemapDebug {
    long long *cell;
    double *xi;
    uint8_t *order;
    uint8_t *status;
};

// Targets of one block: 32 x (threads / 32) nodes in 2-D, 16 x 4 x (threads / 64) in 3-D, so that
// the stencils of a block's targets share L1 lines along every axis.  Blocks are numbered along x
// first (grid dimensions y and z would limit the sides to 65535 blocks).
template <int DIM>
struct BlockShape {
    static constexpr int X = DIM == 2 ? 32 : 16, Y3 = 4;
    unsigned nb[3];
    __host__ __device__ __forceinline__ BlockShape(const int n[3], unsigned threads)
    {
        const unsigned y = DIM == 2 ? threads / X : Y3, z = DIM == 2 ? 1 : threads / (X * Y3);
        nb[0] = ((unsigned)n[0] + X - 1) / X;
        nb[1] = ((unsigned)n[1] + y - 1) / y;
        nb[2] = DIM == 2 ? 1 : ((unsigned)n[2] + z - 1) / z;
    }
    // targets of the blocks, the places outside the grid counted in
    unsigned long long places(unsigned threads) const { return (unsigned long long)nb[0] * nb[1] * nb[2] * threads; }
    __device__ __forceinline__ void node(unsigned block, unsigned threads, unsigned t, int j[3]) const
    {
        const unsigned r = block / nb[0], bx = block - r * nb[0];
        j[0] = (int)(bx * X + t % X);
        if (DIM == 2) {
            j[1] = (int)(r * (threads / X) + t / X);
            j[2] = 0;
        } else {
            const unsigned bz = r / nb[1], by = r - bz * nb[1];
            j[1] = (int)(by * Y3 + (t / X) % Y3);
            j[2] = (int)(bz * (threads / (X * Y3)) + t / (X * Y3));
        }
    }
};

// NMODE: 0 = Newton in T; 1 = Newton in FP64 (FP32 data); 2 = FP32 Newton, FP64 re-solve of targets
// whose FP32 inversion failed or whose element is close to degenerate.  FP64 searches (NMODE 0 of a
// double grid, NMODE 1) run walk_seeded (sl_newton64.cuh).
// QUINTIC: the grid may take order 2 (without it the kernel carries none of its code: the compiler
// hoists the quintic weights out of the fields' loop, 34 FP64 instructions a target; 331 -> 264 us).
// (Two blocks per SM for the 3-D FP64 search: left alone the compiler takes 153 registers and halves the
// warps, 64^3 x 2 fields 176 -> 196 us.)
template <typename T, int DIM, int NMODE, bool QUINTIC>
__global__ void __launch_bounds__(256, DIM == 3 && NMODE <= 1 ? 2 : 0)
    remap_generic_kernel(GridArgs<T> g, const T *__restrict__ D, int ds, const uint8_t *__restrict__ flags,
                         FieldPtrs<T> f, RemapDebug<T> dbg, DevCounters *counters, bool consecutive)
{
    typedef typename std::conditional<NMODE == 1, double, T>::type TW;
    constexpr bool SEEDED = sizeof(TW) == 8;
    LocalCounters cnt;
    cnt.clear();
    WalkParams<TW> wp;
    wp.tol = NMODE == 1 ? TW(1e-14) : TW(g.tol);
    wp.slack = NMODE == 1 ? TW(1e-12) : TW(g.slack);
    wp.max_iter = g.newton_max_iter;
    wp.walk_max = g.walk_max;
    // The cubic weights of an FP64 target wait in shared memory for the fields' sums: kept in registers,
    // the compiler saves those by forming the weights again for every field (18 FP64 instructions of 38;
    // 1024^2 x 3 fields: 386 -> 331 us).
    __shared__ volatile double sw[sizeof(T) == 8 ? DIM * 4 : 1][sizeof(T) == 8 ? 256 : 1];
    int j[3], c[3];
    if (consecutive) {
        const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
        node_coords<DIM>(i, g.n, j);
        if (i >= g.N) j[0] = g.n[0];  // past the end
    } else {
        const BlockShape<DIM> shape(g.n, blockDim.x);
        shape.node(blockIdx.x, blockDim.x, threadIdx.x, j);
    }
    const long long jj = ((long long)j[2] * g.n[1] + j[1]) * g.n[0] + j[0];
    // one pass (the loop only gives `continue` its meaning)
    for (bool todo = j[0] < g.n[0] && j[1] < g.n[1] && (DIM == 2 || j[2] < g.n[2]); todo; todo = false) {
        T Dj[3] = {T(0), T(0), T(0)};
        TW xw[3] = {TW(0), TW(0), TW(0)};
#pragma unroll
        for (int a = 0; a < DIM; ++a) Dj[a] = __ldg(D + jj * ds + a);
        int hops = 0, iters = 0;
        walk_start_cell<T, DIM>(g.walk_start, j, Dj, c);
        bool degen = false;
        int st;
        if constexpr (SEEDED)
            st = walk_seeded<T, DIM>(D, g.n, j, wp.max_iter, wp.walk_max, wp.tol, wp.slack, c, xw, &hops, &iters);
        else
            st = walk_global<T, TW, DIM>(wp, g.n, D, ds, j, c, xw, &hops, &iters, &degen);
        T xi[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int a = 0; a < DIM; ++a) xi[a] = (T)xw[a];
        if (NMODE == 2) {
            const bool redo = st != ST_OK || degen;
            if (redo) {
                WalkParams<double> wd;
                wd.tol = 1e-14;
                wd.slack = 1e-12;
                wd.max_iter = g.newton_max_iter;
                wd.walk_max = g.walk_max;
                double xd[3] = {0.0, 0.0, 0.0};
                if (st == ST_LOCATE || st == ST_FOLD) walk_start_cell<T, DIM>(g.walk_start, j, Dj, c);
                st = walk_global<T, double, DIM>(wd, g.n, D, ds, j, c, xd, &hops, &iters);
#pragma unroll
                for (int a = 0; a < DIM; ++a) xi[a] = (T)xd[a];
                cnt.f64 += 1;
            }
        }
        cnt.targets += 1;
        cnt.hops += hops;
        cnt.hops_max = max(cnt.hops_max, (unsigned)hops);
        cnt.iters += iters;
        cnt.iters_max = max(cnt.iters_max, (unsigned)iters);
        if (dbg.status) dbg.status[jj] = (uint8_t)st;
        if (dbg.xi)
            for (int a = 0; a < DIM; ++a) dbg.xi[jj * DIM + a] = (double)xw[a];
        if (st != ST_OK) {
            cnt.fl += st == ST_LOCATE;
            cnt.fn += st == ST_NEWTON;
            cnt.ff += st == ST_FOLD;
            if (dbg.cell) dbg.cell[jj] = -1;
            for (int q = 0; q < g.nfields; ++q) {
                f.out[q][jj] = f.in[q][jj];
                if (dbg.order) dbg.order[(long long)q * g.N + jj] = 0xff;
            }
            continue;
        }
        if (dbg.cell) dbg.cell[jj] = node_index<DIM>(c, g.n);
        // wrapped node offsets of the cubic stencil c-1 .. c+2 along each axis (taps and flags)
        long long ox[4], oy[4], oz[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            ox[k] = wrap_idx(c[0] - 1 + k, g.n[0]);
            oy[k] = (long long)wrap_idx(c[1] - 1 + k, g.n[1]) * g.n[0];
            oz[k] = DIM == 3 ? (long long)wrap_idx(c[2] - 1 + k, g.n[2]) * g.n[0] * g.n[1] : 0;
        }
        constexpr int KZ = DIM == 3 ? 4 : 1;
        // Sec. 2.3: OR of the flag bytes over the stencils of order 2 ([c-2, c+3]) and 1 ([c-1, c+2])
        unsigned box2 = 0, box1 = 0;
        const int max_order = QUINTIC ? g.max_order : min(g.max_order, 1);
        if (max_order == 1) {
#pragma unroll
            for (int kz = 0; kz < KZ; ++kz)
#pragma unroll
                for (int ky = 0; ky < 4; ++ky)
#pragma unroll
                    for (int kx = 0; kx < 4; ++kx) box1 |= __ldg(flags + oz[kz] + oy[ky] + ox[kx]);
        } else if (QUINTIC && max_order >= 2) {
            const int r = 2, w = 6;
            const int cnt_box = DIM == 3 ? w * w * w : w * w;
            for (int q = 0; q < cnt_box; ++q) {
                int o[3] = {q % w - r, (q / w) % w - r, DIM == 3 ? q / (w * w) - r : 0};
                int k[3] = {c[0] + o[0], c[1] + o[1], c[2] + o[2]};
                const unsigned fb = __ldg(flags + node_index<DIM>(k, g.n));
                box2 |= fb;
                bool inner = true;
#pragma unroll
                for (int a = 0; a < DIM; ++a) inner &= (o[a] >= -1 && o[a] <= 2);
                if (inner) box1 |= fb;
            }
        }
        // eq. (multiZ) weights of orders 1 (Z~1 at taps c-1 .. c+2, Appendix) and 0 (hat at c, c+1),
        // once per target
        T wc[DIM][4], wl[DIM][2];
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const T x = xi[a], y = T(1) - x, x2 = x * x, y2 = y * y;
            if (sizeof(T) == 8) {
                // the same cubics in 8 FP64 operations instead of 12: with p = x (1 - x),
                // -x y^2 / 2 = -p y / 2, 1 - 5/2 x^2 + 3/2 x^3 = y + p (1 - 3/2 x) and their mirrors
                const T p = x * y, h = T(-0.5) * p;
                wc[a][0] = h * y;
                wc[a][1] = y + p * (T(1) - T(1.5) * x);
                wc[a][2] = x + p * (T(1) - T(1.5) * y);
                wc[a][3] = h * x;
            } else {
                wc[a][0] = T(-0.5) * x * y2;
                wc[a][1] = T(1) + x2 * (T(1.5) * x - T(2.5));
                wc[a][2] = T(1) + y2 * (T(1.5) * y - T(2.5));
                wc[a][3] = T(-0.5) * x2 * y;
            }
            wl[a][0] = y;
            wl[a][1] = x;
            if (sizeof(T) == 8) {
#pragma unroll
                for (int k = 0; k < 4; ++k) sw[a * 4 + k][threadIdx.x] = wc[a][k];
            }
        }
        auto weight = [&](int a, int k) -> T { return sizeof(T) == 8 ? (T)sw[a * 4 + k][threadIdx.x] : wc[a][k]; };
        for (int q = 0; q < g.nfields; ++q) {
            int m = max_order;
            if (QUINTIC && m == 2 && ((box2 >> q) & 1u)) m = 1;
            if (m >= 1 && ((box1 >> q) & 1u)) m = 0;
            cnt.oh0 += m == 0;
            cnt.oh1 += m == 1;
            cnt.oh2 += m == 2;
            if (dbg.order) dbg.order[(long long)q * g.N + jj] = (uint8_t)m;
            const T *h = f.in[q];
            T sum = T(0);
            if (m == 1) {
                // rows of four taps, rows into a plane, planes into the sum
                auto row = [&](int kz, int ky) {
                    const T *r = h + oz[kz] + oy[ky];
                    T v = mul_rn_t(weight(0, 0), __ldg(r + ox[0]));
                    v = fma_rn_t(weight(0, 1), __ldg(r + ox[1]), v);
                    v = fma_rn_t(weight(0, 2), __ldg(r + ox[2]), v);
                    return fma_rn_t(weight(0, 3), __ldg(r + ox[3]), v);
                };
                auto plane = [&](int kz) {
                    T v = mul_rn_t(weight(1, 0), row(kz, 0));
                    v = fma_rn_t(weight(1, 1), row(kz, 1), v);
                    v = fma_rn_t(weight(1, 2), row(kz, 2), v);
                    return fma_rn_t(weight(1, 3), row(kz, 3), v);
                };
                if constexpr (DIM == 2) {
                    sum = plane(0);
                } else {
                    sum = mul_rn_t(weight(2, 0), plane(0));
                    sum = fma_rn_t(weight(2, 1), plane(1), sum);
                    sum = fma_rn_t(weight(2, 2), plane(2), sum);
                    sum = fma_rn_t(weight(2, 3), plane(3), sum);
                }
            } else if (m == 0) {
                auto row = [&](int kz, int ky) {
                    const T *r = h + oz[kz] + oy[ky];
                    return fma_rn_t(wl[0][1], __ldg(r + ox[2]), mul_rn_t(wl[0][0], __ldg(r + ox[1])));
                };
                auto plane = [&](int kz) { return fma_rn_t(wl[1][1], row(kz, 2), mul_rn_t(wl[1][0], row(kz, 1))); };
                if constexpr (DIM == 2)
                    sum = plane(0);
                else
                    sum = fma_rn_t(wl[2][1], plane(2), mul_rn_t(wl[2][0], plane(1)));
            } else if (QUINTIC) {
                T w[3][6];
#pragma unroll
                for (int a = 0; a < DIM; ++a) zs_weights<T>(m, xi[a], w[a]);
                const int wn = 2 * m + 2;
                const int wz = DIM == 3 ? wn : 1;
                for (int kz = 0; kz < wz; ++kz) {
                    for (int ky = 0; ky < wn; ++ky) {
                        for (int kx = 0; kx < wn; ++kx) {
                            int k[3] = {c[0] - m + kx, c[1] - m + ky, DIM == 3 ? c[2] - m + kz : 0};
                            T wt = w[0][kx] * w[1][ky];
                            if (DIM == 3) wt *= w[2][kz];
                            sum += __ldg(h + node_index<DIM>(k, g.n)) * wt;
                        }
                    }
                }
            }
            f.out[q][jj] = sum;
        }
    }
    // each warp adds into its SM's copy of the counters (the launch passes the per-SM copies)
    unsigned smid;
    asm("mov.u32 %0, %%smid;" : "=r"(smid));
    flush_counters_warp(cnt, counters + (smid % SL_COUNTER_STRIPES));
}

// ------------------------------------------------------------------------------------------------
// Sec. 3.1 moments: per-block partial sums (fixed grid, fixed tree order), then one final block
// ------------------------------------------------------------------------------------------------
struct MomentGeom {
    double lo[3], dx[3], cen[3];
};

template <typename T, int DIM>
__global__ void __launch_bounds__(256)
    moments_partial_kernel(GridArgs<T> g, MomentGeom mg, const T *__restrict__ h, int pmax, double *partials)
{
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N;
         i += (long long)gridDim.x * blockDim.x) {
        int k[3];
        node_coords<DIM>(i, g.n, k);
        const double hv = (double)h[i];
        acc[0] += hv;
        double r[3];
#pragma unroll
        for (int a = 0; a < DIM; ++a) r[a] = mg.lo[a] + (double)k[a] * mg.dx[a] - mg.cen[a];
        double rp[3] = {1.0, 1.0, 1.0};
        for (int p = 1; p <= pmax; ++p) {
            double s = 0.0;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                rp[a] *= r[a];
                s += rp[a];
            }
            acc[p] += hv * s;
        }
    }
    __shared__ double red[8][256];
    for (int p = 0; p <= pmax; ++p) red[p][threadIdx.x] = acc[p];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int p = 0; p <= pmax; ++p) red[p][threadIdx.x] += red[p][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int p = 0; p <= pmax; ++p) partials[blockIdx.x * 8 + p] = red[p][0];
}

__global__ void moments_final_kernel(const double *partials, int nblocks, int pmax, double *out)
{
    const int p = threadIdx.x;
    if (p > pmax) return;
    double s = 0.0;
    for (int b = 0; b < nblocks; ++b) s += partials[b * 8 + p];
    out[p] = s;
}

// ------------------------------------------------------------------------------------------------
// strided copy of displacements (set / get)
// ------------------------------------------------------------------------------------------------
// every field plane in one launch: 16-byte vector copies when all planes are 16-byte aligned
template <typename T, bool VEC>
__global__ void __launch_bounds__(256) copy_planes_kernel(long long N, int nf, FieldPtrs<T> f)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (VEC) {
        // every plane's vector at once: nf independent 16-byte loads in flight per thread; the
        // source (the scratch planes) is not read again before it is overwritten
        const long long nv = N * (long long)sizeof(T) / 16;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nv; i += stride) {
            float4 v[SL_MAX_FIELDS];
#pragma unroll
            for (int q = 0; q < SL_MAX_FIELDS; ++q)
                if (q < nf) v[q] = __ldcs(reinterpret_cast<const float4 *>(f.in[q]) + i);
#pragma unroll
            for (int q = 0; q < SL_MAX_FIELDS; ++q)
                if (q < nf) reinterpret_cast<float4 *>(f.out[q])[i] = v[q];
        }
    } else {
        for (int q = 0; q < nf; ++q)
            for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += stride)
                f.out[q][i] = f.in[q][i];
    }
}

template <typename T>
__global__ void copy_disp_kernel(long long N, int dim, const T *__restrict__ src, long long ss, T *__restrict__ dst,
                                 long long dsd)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        for (int a = 0; a < dim; ++a) dst[i * dsd + a] = src[i * ss + a];
        for (int a = dim; a < dsd; ++a) dst[i * dsd + a] = T(0);
    }
}

// ------------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------------
template <typename T>
static FieldPtrs<T> field_ptrs(const sl_grid *g, const void *const *in, void *const *out)
{
    FieldPtrs<T> f;
    memset(&f, 0, sizeof(f));
    for (int q = 0; q < g->nfields; ++q) {
        f.in[q] = in ? (const T *)in[q] : nullptr;
        f.out[q] = out ? (T *)out[q] : nullptr;
    }
    return f;
}

template <typename T>
cudaError_t Launch<T>::advect(const sl_grid *g, void *D, double t, double dt, cudaStream_t s)
{
    const GridArgs<T> ga = make_grid_args<T>(g);
    const VelArgs<T> va = make_vel_args<T>(g, t, dt);
    const int blocks = grid_stride_blocks(g, g->N, 256);
    if constexpr (sizeof(T) == 8) {
        if (va.kind == SL_VEL_SWIRL2D && va.sc[0] != nullptr && va.integrator == SL_RK4 && va.substeps == 1) {
            const double pi = 3.141592653589793238462643;
            Swirl64 w;
            w.A[0] = pi * dt * va.ct[0];
            w.A[1] = pi * dt * va.ct[1];
            w.A[2] = 2.0 * pi * dt * va.ct[1];
            // (a quarter less for the growth of q over the step; each stage still checks its own angle)
            const double steep = std::max(std::max(fabs(w.A[0]), fabs(w.A[1])), fabs(w.A[2]));
            const double far = std::min(pi / 16.0 / 1.25 / steep, 1.0);  // |q| <= 1/2
            uint64_t bits;
            memcpy(&bits, &far, sizeof(bits));
            w.far = (int)(bits >> 32);
            for (int q = 0; q < 3; ++q) {
                const double b = dt / 3.0 * va.ct[q] * (q == 1 ? 2.0 : 1.0);
                w.Bx[q] = b / g->dx[0];
                w.By[q] = -b / g->dx[1];
            }
            advect_swirl64_kernel<<<blocks, 256, 0, s>>>(ga, va, w, (double2 *)D);
            return cudaGetLastError();
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (va.pairs) {
            // small launches last as long as one thread's chain: blocks of 64 spread it over more SMs, four
            // modes at a time shorten it (8 modes, 32^2 5.1 -> 3.7 us, 400^2 9.4 -> 8.0; 512^2 10.9 either way)
            const unsigned half = (unsigned)((g->N + 1) / 2);
            if (g->N >= (1LL << 18))
                advect_fourier2d_kernel<256, 2><<<(half + 255) / 256, 256, 0, s>>>(ga, va, (float2 *)D, half);
            else
                advect_fourier2d_kernel<64, 4><<<(half + 63) / 64, 64, 0, s>>>(ga, va, (float2 *)D, half);
            return cudaGetLastError();
        }
    }
    if (g->dim == 2)
        advect_kernel<T, 2><<<blocks, 256, 0, s>>>(ga, va, (T *)D, g->ds);
    else
        advect_kernel<T, 3><<<blocks, 256, 0, s>>>(ga, va, (T *)D, g->ds);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::advect_carried(const sl_grid *g, const void *const *fields, void *D, double dt, cudaStream_t s)
{
    const T *u[3] = {nullptr, nullptr, nullptr};
    T sc[3] = {T(0), T(0), T(0)};
    for (int a = 0; a < g->dim; ++a) {
        u[a] = (const T *)fields[g->vel_field[a]];
        sc[a] = (T)(dt / g->dx[a]);
    }
    const int blocks = grid_stride_blocks(g, g->N, 256);
    if (g->dim == 2)
        advect_carried_kernel<T, 2><<<blocks, 256, 0, s>>>(g->N, u[0], u[1], u[1], sc[0], sc[1], sc[2], (T *)D);
    else
        advect_carried_kernel<T, 3><<<blocks, 256, 0, s>>>(g->N, u[0], u[1], u[2], sc[0], sc[1], sc[2], (T *)D);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::flags(const sl_grid *g, const void *const *in, uint8_t *flags, cudaStream_t s)
{
    const GridArgs<T> ga = make_grid_args<T>(g);
    const FieldPtrs<T> f = field_ptrs<T>(g, in, nullptr);
    const int blocks = grid_stride_blocks(g, g->N, 256);
    if constexpr (sizeof(T) == 8) {
        // (below 8 columns a warp of flags64_kernel wastes three lanes in four and more: 4 x 65536 nodes of
        // 3 fields 33.2 us against 22.6, 8 x 8192 8.0 against 8.2)
        if (g->dim == 2 && g->n[0] >= 8 && g->desc.limiter_threshold >= 0.0) {
            const unsigned strips = (unsigned)((g->n[0] + FLAG_COLS - 1) / FLAG_COLS);
            // fewer rows a warp where the grid has too few warps to fill the SMs: a row takes ~1 us of
            // dependent FP64 latency, which only other warps can hide
            const int rows = strips * (g->n[1] / FLAG_ROWS) >= 8u * g->num_sms ? FLAG_ROWS : 1;
            const unsigned nwarps = strips * (unsigned)((g->n[1] + rows - 1) / rows);
            const JumpBounds b(g->desc.limiter_threshold);
            const int n0 = (int)g->n[0], n1 = (int)g->n[1], nf = g->nfields;
            const unsigned nb = (nwarps + 3) / 4;
            if (nf == 1)
                flags64_kernel<1><<<nb, 128, 0, s>>>(n0, n1, nf, b, f, flags, strips, nwarps, rows);
            else if (nf <= 4)
                flags64_kernel<4><<<nb, 128, 0, s>>>(n0, n1, nf, b, f, flags, strips, nwarps, rows);
            else
                flags64_kernel<8><<<nb, 128, 0, s>>>(n0, n1, nf, b, f, flags, strips, nwarps, rows);
            return cudaGetLastError();
        }
    }
    if (g->dim == 2)
        flags_kernel<T, 2><<<blocks, 256, 0, s>>>(ga, f, flags);
    else
        flags_kernel<T, 3><<<blocks, 256, 0, s>>>(ga, f, flags);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::remap_generic(const sl_grid *g, const void *D, const uint8_t *flags, const void *const *in,
                                     void *const *out, const sl_remap_debug *dbg, cudaStream_t s)
{
    const GridArgs<T> ga = make_grid_args<T>(g);
    const FieldPtrs<T> f = field_ptrs<T>(g, in, out);
    RemapDebug<T> d;
    d.cell = dbg ? (long long *)dbg->cell : nullptr;
    d.xi = dbg ? dbg->xi : nullptr;
    d.order = dbg ? dbg->order : nullptr;
    d.status = dbg ? dbg->status : nullptr;
    // FP64 targets keep a warp busy for microseconds: a small grid is cut into small blocks, so that
    // its warps spread over the SMs
    const int NT = sizeof(T) == 4 || g->N >= 256LL * 4 * g->num_sms ? 256 : 64;
    // Blocks of targets share L1 lines (1-3 % faster on 512^2, 64^3 and 79^3); consecutive nodes where
    // more than a tenth of the blocks' places lie outside the grid and would idle in warps that cost an
    // FP64 instruction the same.  FP64 remaps of one field, us, consecutive / blocks: 4 x 65536 (8 places
    // a node) 50 / 238, 33 x 8192 (1.9) 47 / 72, 48 x 8192 (1.3) 61 / 75, 28 x 16384 (1.14) 65 / 73,
    // 512 x 512 (1) 50.6 / 49.3; 4 x 4 x 65536 (4) 318 / 1100, 14 x 64 x 400 (1.14) 127 / 137, 79^3 (1.03)
    // 203 / 203.  FP32 on these kernels: 4 x 65536 23 / 78, 33 x 8192 25 / 31, 64^3 45 / 44.
    const unsigned long long places = g->dim == 2 ? BlockShape<2>(ga.n, NT).places(NT) : BlockShape<3>(ga.n, NT).places(NT);
    const bool lin = (double)places > 1.1 * (double)g->N;
    const unsigned blocks = (unsigned)(lin ? (g->N + NT - 1) / NT : (long long)(places / NT));
    const bool n64 = g->desc.newton_mode == SL_NEWTON_F64;
    const T *d0 = (const T *)D;
    if constexpr (sizeof(T) == 8) {
        const bool z2 = g->desc.max_order > 1;
        if (g->dim == 2 && z2)
            remap_generic_kernel<T, 2, 0, true><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
        else if (g->dim == 2)
            remap_generic_kernel<T, 2, 0, false><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
        else if (z2)
            remap_generic_kernel<T, 3, 0, true><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
        else
            remap_generic_kernel<T, 3, 0, false><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
    } else if (g->dim == 2) {
        if (n64)
            remap_generic_kernel<T, 2, 1, true><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
        else
            remap_generic_kernel<T, 2, 2, true><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
    } else {
        if (n64)
            remap_generic_kernel<T, 3, 1, true><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
        else
            remap_generic_kernel<T, 3, 2, true><<<blocks, NT, 0, s>>>(ga, d0, g->ds, flags, f, d, g->stripes, lin);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::moments(const sl_grid *g, const void *field, int pmax, cudaStream_t s)
{
    const GridArgs<T> ga = make_grid_args<T>(g);
    MomentGeom mg;
    for (int a = 0; a < 3; ++a) {
        mg.lo[a] = g->desc.lo[a];
        mg.dx[a] = g->dx[a];
        mg.cen[a] = 0.5 * (g->desc.lo[a] + g->desc.hi[a]);
    }
    if (g->dim == 2)
        moments_partial_kernel<T, 2><<<SL_MOMENT_BLOCKS, 256, 0, s>>>(ga, mg, (const T *)field, pmax, g->partials);
    else
        moments_partial_kernel<T, 3><<<SL_MOMENT_BLOCKS, 256, 0, s>>>(ga, mg, (const T *)field, pmax, g->partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    moments_final_kernel<<<1, 32, 0, s>>>(g->partials, SL_MOMENT_BLOCKS, pmax, g->moment_out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::copy_planes(const sl_grid *g, const void *const *src, void *const *dst, cudaStream_t s)
{
    FieldPtrs<T> f;
    memset(&f, 0, sizeof(f));
    bool vec = ((size_t)g->N * sizeof(T)) % 16 == 0;
    for (int q = 0; q < g->nfields; ++q) {
        f.in[q] = (const T *)src[q];
        f.out[q] = (T *)dst[q];
        vec = vec && ((uintptr_t)src[q] & 15u) == 0 && ((uintptr_t)dst[q] & 15u) == 0;
    }
    const long long work = vec ? (long long)g->N * (long long)sizeof(T) / 16 : (long long)g->N;
    const int blocks = (int)std::min<long long>(grid_stride_blocks(g, work, 256), (long long)g->num_sms * 8);
    if (vec)
        copy_planes_kernel<T, true><<<blocks, 256, 0, s>>>((long long)g->N, g->nfields, f);
    else
        copy_planes_kernel<T, false><<<blocks, 256, 0, s>>>((long long)g->N, g->nfields, f);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::copy_disp(const sl_grid *g, const void *src, int64_t src_stride, void *dst, int64_t dst_stride,
                                 cudaStream_t s)
{
    const int blocks = grid_stride_blocks(g, g->N, 256);
    copy_disp_kernel<T><<<blocks, 256, 0, s>>>((long long)g->N, g->dim, (const T *)src, (long long)src_stride,
                                               (T *)dst, (long long)dst_stride);
    return cudaGetLastError();
}

template struct Launch<double>;
template struct Launch<float>;
