// sl_newton64.cuh -- the FP64 element search of Sec. 2.2 with its Newton inversion (eq. mapping1)
// started in FP32, for the plain kernels.
//
// What bounds an FP64 remap on GB300 is the FP64 pipe: 2 results per SM and cycle against 128 for
// FP32, so one FP64 instruction costs as much as 64 FP32 ones, and a dependent one takes 63 cycles.
// The all-FP64 search spends ~150 (2-D) and ~450 (3-D) FP64 instructions per element tried: three
// Newton iterations with their Jacobians, cofactors and divisions.  Here each element is inverted
// in FP32 first; FP64 is used where its digits matter:
//
//   * an element the FP32 solution says is left by more than that solution's error needs no more
//     digits: the walk steps on;
//   * otherwise the coordinates are polished: x <- x - Ji F(x) with the residual F in FP64 and the
//     inverse Jacobian Ji in FP32, which gains ~6 digits per pass (two passes as a rule, 12 / 42
//     FP64 instructions in 2-D / 3-D), down to the rounding error of F, as the FP64 iteration does.
//
// Conversions between FP32, FP64 and integers take an FP64 slot too and are done by bit operations.
// A 1024^2 x 3 remap issues 113 FP64 instructions per warp where the all-FP64 search needed 263 a target:
// 480 -> 223 us; 64^3 x 2 fields 640 -> 145 us.
//
// Every decision of the FP64 search (fold, no convergence, inside, next element) is taken from the
// FP32 solution only under a certificate (seed_solve): at every iterate the columns of J exceed
// their own rounding error by SEED_CLEAR and det J stays away from zero by more than that error can
// move it; the steps shrink; the iteration converges with iterations to spare.  Then the FP64
// iteration runs through nearly the same points and converges to the same root.  Without it the
// element is inverted by the FP64 iteration (newton_solve).
// How far the FP32 root can be from the FP64 one depends on the displacement's size (stored with 24
// bits, a shift of 2000 cells leaves 2e-4 of a cell), on the element's shape (the inverse Jacobian
// amplifies) and on how far outside the root lies, so a bound is formed for each coordinate (seed_clear),
// and only coordinates beyond it decide a step.  (A fixed margin of 1e-3 lost 172 targets of a 1024^2 grid
// displaced by 2048 cells under a shear of slope 10; the bounds cost 64^2 x 16 steps of a solid-body
// rotation, a chain of 27 hops each, 491 -> 524 us, a 64^3 x 2 step 170 -> 176 us, 1024^2 nothing.)
#pragma once

#include <type_traits>

#include "sl_device.cuh"

namespace {

// |det J| relative to the product of the 1-norms of J's columns (1 for a square element)
constexpr float SEED_DET = 0.05f;
// Iterates must stay within this distance of the element.  (The failing walks at the seam of a
// solid-body rotation meet sheared elements at coordinates of 30 to 60; with 16 here a quarter of
// their hops took the FP64 iteration, 112 against 21 us per 64^2 step.)
constexpr float SEED_REACH = 128.f;
// Columns of J must exceed the error of their entries by this factor: with entries off by e, det J
// is off by at most DIM^2 e / column of the columns' product, 0.02 in 2-D and 0.045 in 3-D: less than
// SEED_DET, so its sign is certain.
constexpr float SEED_CLEAR = 200.f;
// distance from a face beyond which the FP32 coordinates decide the step, on top of their own bound:
// what the last Newton step (at most SL_NEWTON_TOL_F32, halved by each further one) leaves over, and
// the room that polishing needs
constexpr float SEED_MARGIN = 1e-3f;
// Largest amplification of FP64 rounding (by Ji, the shape functions and the vertex coordinates) of an
// element whose polished coordinates are a target's result.  Above it the FP64 iteration may not come
// down to its stop, a step of 1e-14, and end as ST_NEWTON; and Map64's coefficients, rounded at the size
// of the displacements' differences, would cost digits that the vertices of a strongly compressed element
// have.
constexpr float SEED_STOP = 40.f;
// iterations the FP64 solve needs beyond the FP32 one: 3e-4 -> 1e-7 -> 1e-14 -> below its 1e-14 stop
constexpr int SEED_SPARE = 3;

enum { SEED_NONE = 0, SEED_OK = 1, SEED_FOLD = 2 };

template <int DIM>
struct Seed {
    float x[DIM];       // local coordinates
    float C[DIM][DIM];  // cofactors of J there: the inverse is C / det
    float det, noise;   // noise: error of a vertex coordinate and of differences of two
    float peak[DIM];    // largest vertex coordinate along each axis
    int iters;
};

// Error of an entry of J at x, from the error `noise` of a vertex coordinate: a difference of two
// vertices, extrapolated along the other axes (bounded by the largest coordinate).
template <int DIM>
__device__ __forceinline__ float entry_error(float noise, const float x[DIM])
{
    float far = fabsf(x[0]);
#pragma unroll
    for (int a = 1; a < DIM; ++a) far = fmaxf(far, fabsf(x[a]));
    const float f = 1.f + 2.f * far;
    return 2.f * noise * (DIM == 3 ? f * f : f);
}

// The shape functions' magnitudes at x, summed: what extrapolation does to an error of the vertices.
template <int DIM>
__device__ __forceinline__ float shape_sum(const float x[DIM])
{
    float f = 1.f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) f *= fabsf(x[a]) + fabsf(1.f - x[a]);
    return f;
}

// Does every coordinate lie on the same side of 0 and of 1 in FP64?  The residual at x is off by `noise`
// times the shape sum for the vertices, and by no more than three times that for its own rounding (16
// roundings of terms up to that sum times the largest vertex coordinate, of which `noise` holds 4); the
// inverse Jacobian carries it into the coordinates.  (No division: this ends every hop.)
template <int DIM>
__device__ __forceinline__ bool seed_clear(const Seed<DIM> &s)
{
    const float e = 4.f * s.noise * shape_sum<DIM>(s.x);
    bool clear = true;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        float sum = 0.f;
#pragma unroll
        for (int b = 0; b < DIM; ++b) sum += fabsf(s.C[a][b]);
        clear &= (fminf(fabsf(s.x[a]), fabsf(s.x[a] - 1.f)) - SEED_MARGIN) * s.det > sum * e;
    }
    return clear;
}

// Are polished coordinates inside the element as good as the FP64 iteration's?
template <int DIM>
__device__ __forceinline__ bool seed_final(const Seed<DIM> &s)
{
    float round = 0.f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        float sum = 0.f;
#pragma unroll
        for (int b = 0; b < DIM; ++b) sum += fabsf(s.C[a][b]) * fmaxf(s.peak[b], 1.f);
        round = fmaxf(round, sum);
    }
    return round * shape_sum<DIM>(s.x) <= SEED_STOP * s.det;
}

// FP32 Newton inversion of the bilinear element with vertices P (relative to the target), the
// iteration of newton_solve2 under the certificate described above (r.noise and r.peak given).
__device__ __forceinline__ int seed_solve(const float P[4][2], int max_iter, Seed<2> &r)
{
    const float px = P[0][0], py = P[0][1];
    const float ax = P[1][0] - px, ay = P[1][1] - py, bx = P[2][0] - px, by = P[2][1] - py;
    const float ex = P[3][0] - P[1][0] - bx, ey = P[3][1] - P[1][1] - by;
    float det = ax * by - bx * ay;
    const float na = fabsf(ax) + fabsf(ay), nb = fabsf(bx) + fabsf(by);
    bool sure = fabsf(det) > SEED_DET * (na * nb) && fminf(na, nb) > SEED_CLEAR * 2.f * r.noise;
    if (!(det > 0.f)) return sure ? SEED_FOLD : SEED_NONE;
    float inv = recip_t(det);
    float x[2] = {-(px * by - py * bx) * inv, -(ax * py - ay * px) * inv}, step = 3e38f;
    for (int it = 0;; ++it) {
        const float j11 = ax + x[1] * ex, j21 = ay + x[1] * ey, j12 = bx + x[0] * ex, j22 = by + x[0] * ey;
        det = j11 * j22 - j12 * j21;
        const float n1 = fabsf(j11) + fabsf(j21), n2 = fabsf(j12) + fabsf(j22);
        sure &= det > SEED_DET * (n1 * n2) && fminf(n1, n2) > SEED_CLEAR * entry_error<2>(r.noise, x) &&
                fmaxf(fabsf(x[0]), fabsf(x[1])) <= SEED_REACH;
        if (step <= SL_NEWTON_TOL_F32) {
            if (!sure) return SEED_NONE;
            r.x[0] = x[0];
            r.x[1] = x[1];
            r.C[0][0] = j22;
            r.C[0][1] = -j12;
            r.C[1][0] = -j21;
            r.C[1][1] = j11;
            r.det = det;
            r.iters = it;
            return SEED_OK;
        }
        if (!sure || it + SEED_SPARE >= max_iter) return SEED_NONE;
        inv = recip_t(det);
        const float fx = px + x[0] * j11 + x[1] * bx, fy = py + x[0] * j21 + x[1] * by;
        const float d0 = (fx * j22 - fy * j12) * inv, d1 = (j11 * fy - j21 * fx) * inv, last = step;
        x[0] -= d0;
        x[1] -= d1;
        step = fmaxf(fabsf(d0), fabsf(d1));
        sure = step <= 0.5f * last;
    }
}

// the same for the trilinear element (vertex v = x + 2 y + 4 z)
__device__ __forceinline__ int seed_solve(const float P[8][3], int max_iter, Seed<3> &r)
{
    float A[3][3], E01[3], E02[3], E12[3], G[3], x[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float d10 = P[1][a] - P[0][a], d32 = P[3][a] - P[2][a], d54 = P[5][a] - P[4][a], d76 = P[7][a] - P[6][a];
        A[a][0] = d10;
        A[a][1] = P[2][a] - P[0][a];
        A[a][2] = P[4][a] - P[0][a];
        E01[a] = d32 - d10;
        E02[a] = d54 - d10;
        E12[a] = P[6][a] - P[4][a] - A[a][1];
        G[a] = d76 - d54 - E01[a];
    }
    // cofactors C of J (the inverse is C / det), det, the product of the columns' norms and the least of them
    auto cofactors = [](const float J[3][3], float C[3][3], float &det, float &norm, float &least) {
        C[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
        C[1][0] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
        C[2][0] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
        det = J[0][0] * C[0][0] + J[0][1] * C[1][0] + J[0][2] * C[2][0];
        const float n0 = fabsf(J[0][0]) + fabsf(J[1][0]) + fabsf(J[2][0]),
                    n1 = fabsf(J[0][1]) + fabsf(J[1][1]) + fabsf(J[2][1]),
                    n2 = fabsf(J[0][2]) + fabsf(J[1][2]) + fabsf(J[2][2]);
        norm = n0 * n1 * n2;
        least = fminf(fminf(n0, n1), n2);
        C[0][1] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
        C[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
        C[2][1] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
        C[0][2] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
        C[1][2] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
        C[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    };
    float C[3][3], det, norm, least;
    cofactors(A, C, det, norm, least);
    bool sure = fabsf(det) > SEED_DET * norm && least > SEED_CLEAR * 2.f * r.noise;
    if (!(det > 0.f)) return sure ? SEED_FOLD : SEED_NONE;
    float inv = recip_t(det), step = 3e38f;
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = -(C[a][0] * P[0][0] + C[a][1] * P[0][1] + C[a][2] * P[0][2]) * inv;
    for (int it = 0;; ++it) {
        const float s01 = x[0] * x[1], s02 = x[0] * x[2], s12 = x[1] * x[2];
        float J[3][3], F[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            J[a][0] = A[a][0] + x[1] * E01[a] + x[2] * E02[a] + s12 * G[a];
            J[a][1] = A[a][1] + x[0] * E01[a] + x[2] * E12[a] + s02 * G[a];
            J[a][2] = A[a][2] + x[0] * E02[a] + x[1] * E12[a] + s01 * G[a];
            F[a] = P[0][a] + x[0] * J[a][0] + x[1] * (A[a][1] + x[2] * E12[a]) + x[2] * A[a][2];
        }
        cofactors(J, C, det, norm, least);
        sure &= det > SEED_DET * norm && least > SEED_CLEAR * entry_error<3>(r.noise, x) &&
                fmaxf(fmaxf(fabsf(x[0]), fabsf(x[1])), fabsf(x[2])) <= SEED_REACH;
        if (step <= SL_NEWTON_TOL_F32) {
            if (!sure) return SEED_NONE;
#pragma unroll
            for (int a = 0; a < 3; ++a) r.x[a] = x[a];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) r.C[a][b] = C[a][b];
            r.det = det;
            r.iters = it;
            return SEED_OK;
        }
        if (!sure || it + SEED_SPARE >= max_iter) return SEED_NONE;
        inv = recip_t(det);
        const float last = step;
        step = 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float d = (C[a][0] * F[0] + C[a][1] * F[1] + C[a][2] * F[2]) * inv;
            x[a] -= d;
            step = fmaxf(step, fabsf(d));
        }
        sure = step <= 0.5f * last;
    }
}

// The FP64 coefficients of an element's multilinear map about its lower corner, from the vertex
// displacements V and the corner's offset k = c - j from the target (the map of newton_solve2/3).
template <int DIM>
struct Map64;
template <>
struct Map64<2> {
    double p[2], a[2], b[2], e[2];
    template <typename T>
    __device__ __forceinline__ Map64(const T V[4][2], const int k[3])
    {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const double v0 = (double)V[0][q], v1 = (double)V[1][q], d20 = (double)V[2][q] - v0;
            p[q] = small_int(k[q]) + v0;
            a[q] = v1 - v0;
            e[q] = ((double)V[3][q] - v1) - d20;
            b[q] = d20;
        }
        a[0] += 1.0;
        b[1] += 1.0;
    }
    __device__ __forceinline__ void residual(const double x[3], float F[2]) const
    {
#pragma unroll
        for (int q = 0; q < 2; ++q) F[q] = narrow(fma(x[1], fma(x[0], e[q], b[q]), fma(x[0], a[q], p[q])));
    }
};
template <>
struct Map64<3> {
    double p[3], a[3], b[3], c[3], e01[3], e02[3], e12[3], g[3];
    template <typename T>
    __device__ __forceinline__ Map64(const T V[8][3], const int k[3])
    {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double v0 = (double)V[0][q], v2 = (double)V[2][q], v4 = (double)V[4][q], v6 = (double)V[6][q];
            const double d10 = (double)V[1][q] - v0, d32 = (double)V[3][q] - v2, d54 = (double)V[5][q] - v4,
                         d76 = (double)V[7][q] - v6;
            p[q] = small_int(k[q]) + v0;
            a[q] = d10;
            b[q] = v2 - v0;
            c[q] = v4 - v0;
            e01[q] = d32 - d10;
            e02[q] = d54 - d10;
            e12[q] = (v6 - v4) - b[q];
            g[q] = (d76 - d54) - e01[q];
        }
        a[0] += 1.0;
        b[1] += 1.0;
        c[2] += 1.0;
    }
    __device__ __forceinline__ void residual(const double x[3], float F[3]) const
    {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double u = fma(x[1], fma(x[2], g[q], e01[q]), fma(x[2], e02[q], a[q]));
            F[q] = narrow(fma(x[0], u, fma(x[1], fma(x[2], e12[q], b[q]), fma(x[2], c[q], p[q]))));
        }
    }
};

// x <- x - Ji F(x), Ji the FP32 inverse Jacobian, until what a pass leaves -- its move times the bound
// on |1 - Ji J| -- is below FP64 rounding.  The passes move x by less than SEED_MARGIN in all.  False
// where it does not settle.
template <int DIM>
__device__ __forceinline__ bool polish(const Map64<DIM> &m, const Seed<DIM> &s, double x[3], int *iters)
{
    const float inv = recip_t(s.det);
    float Ji[DIM][DIM], most = 0.f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        float sum = 0.f;
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
            Ji[a][b] = s.C[a][b] * inv;
            sum += fabsf(Ji[a][b]);
        }
        most = fmaxf(most, sum);
        x[a] = widen(s.x[a]);
    }
    // (1e-5: the rounding of Ji itself, a few 6e-8 / SEED_DET)
    const float rate = 1e-5f + (float)DIM * most * entry_error<DIM>(s.noise, s.x);
    for (int it = 0; it < 4; ++it) {
        float F[DIM], big = 0.f;
        m.residual(x, F);
        *iters += 1;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            float d = 0.f;
#pragma unroll
            for (int b = 0; b < DIM; ++b) d += Ji[a][b] * F[b];
            if (!(fabsf(d) <= 0.2f * SEED_MARGIN)) return false;
            x[a] -= widen(d);
            big = fmaxf(big, fabsf(d));
        }
        if (big * rate <= 1e-16f) return true;
    }
    return false;
}

// Element by element: vertex displacements V of element c, as stored.
template <typename T, int DIM>
__device__ __forceinline__ void load_vertices(const T *__restrict__ D, const int n[3], const int c[3],
                                              T V[1 << DIM][DIM])
{
    // one wrap per axis and side; a node is 2 (2-D) or 4 (3-D) values
    using T2 = typename std::conditional<sizeof(T) == 8, double2, float2>::type;
    const T2 *d = reinterpret_cast<const T2 *>(D);
    unsigned o[3][2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        o[0][s] = (unsigned)wrap_idx(c[0] + s, n[0]);
        o[1][s] = (unsigned)wrap_idx(c[1] + s, n[1]) * (unsigned)n[0];
        o[2][s] = DIM == 3 ? (unsigned)wrap_idx(c[2] + s, n[2]) * ((unsigned)n[0] * (unsigned)n[1]) : 0u;
    }
#pragma unroll
    for (int v = 0; v < (1 << DIM); ++v) {
        const size_t i = o[0][v & 1] + o[1][(v >> 1) & 1] + o[2][v >> 2];
        const T2 q = __ldg(d + (DIM == 3 ? 2 * i : i));
        V[v][0] = q.x;
        V[v][1] = q.y;
        if (DIM == 3) V[v][DIM - 1] = __ldg(D + 4 * i + 2);
    }
}

struct Solved64 {
    int st, iters;
    double x0, x1, x2;
};

// the FP64 iteration for an element without a certificate (rare: out of line)
template <typename T, int DIM>
__device__ __noinline__ Solved64 solve_element64(const T *__restrict__ D, int n0, int n1, int n2, int c0, int c1, int c2,
                                                 int j0, int j1, int j2, int max_iter, double tol)
{
    const int n[3] = {n0, n1, n2}, c[3] = {c0, c1, c2}, j[3] = {j0, j1, j2};
    T V[1 << DIM][DIM];
    load_vertices<T, DIM>(D, n, c, V);
    double P[8][3], x[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int v = 0; v < (1 << DIM); ++v)
#pragma unroll
        for (int a = 0; a < DIM; ++a) P[v][a] = double(c[a] + ((v >> a) & 1) - j[a]) + (double)V[v][a];
    Solved64 r;
    r.iters = 0;
    r.st = newton_solve<double, DIM>(P, max_iter, tol, x, &r.iters);
    r.x0 = x[0];
    r.x1 = x[1];
    r.x2 = x[2];
    return r;
}

// Sec. 2.2 element search from element c with FP64 coordinates: the walk of the plain kernels
// (walk_global), each element inverted as described at the top of this file.  The FP32 hops run in
// a loop of their own, so that the targets of a warp, which take different numbers of hops, do
// their FP64 work together (polished inside the hop loop, every hop count had its own pass over
// the FP64 code: 223 against 150 FP64 instructions per warp on a 1024^2 x 3 remap).
template <typename T, int DIM>
__device__ __forceinline__ int walk_seeded(const T *__restrict__ D, const int n[3], const int j[3], int max_iter,
                                           int walk_max, double tol, double slack, int c[3], double xi[3], int *hops,
                                           int *iters)
{
    CycleCheck cyc;
    cyc.start(c[0], c[1], c[2]);
    int hop = 0;
    for (;;) {
        // elements that the FP32 solution says are left, up to the first it cannot rule out
        T V[1 << DIM][DIM];
        Seed<DIM> s;
        int seed = SEED_NONE;
        bool inner = false;  // inside the element by SEED_MARGIN and more (polishing moves x by less)
        for (;;) {
            if (hop >= walk_max) return ST_LOCATE;
            load_vertices<T, DIM>(D, n, c, V);
            float P[1 << DIM][DIM], big = 0.f, most = 0.f;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                s.peak[a] = 0.f;
#pragma unroll
                for (int v = 0; v < (1 << DIM); ++v) {
                    const float f = narrow(V[v][a]);
                    if (sizeof(T) == 8) big = fmaxf(big, fabsf(f));
                    P[v][a] = (float)(c[a] + ((v >> a) & 1) - j[a]) + f;
                    s.peak[a] = fmaxf(s.peak[a], fabsf(P[v][a]));
                }
                most = fmaxf(most, s.peak[a]);
            }
            // 1.2e-7: the bits that narrow cuts off a double; 2.4e-7: four roundings, of P and differences
            s.noise = 1.2e-7f * big + 2.4e-7f * most;
            seed = seed_solve(P, max_iter, s);
            ++hop;
            *hops += 1;
            if (seed != SEED_OK) break;
            *iters += s.iters;
            bool out = false;
#pragma unroll
            for (int a = 0; a < DIM; ++a) out |= s.x[a] < 0.f || s.x[a] > 1.f;
            const bool clear = seed_clear(s);
            inner = clear && !out;
            if (!clear || !out) break;  // inside, or an axis in doubt
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                c[a] += s.x[a] < 0.f ? -1 : (s.x[a] > 1.f ? 1 : 0);
                xi[a] = widen(s.x[a]);
            }
            if (cyc.step(c[0], c[1], c[2])) return ST_LOCATE;
        }
        // this element in FP64
        int st = ST_OK;
        if (seed == SEED_FOLD) {
#pragma unroll
            for (int a = 0; a < DIM; ++a) xi[a] = NAN;
            return ST_FOLD;
        }
        bool polished = false;
        const bool final = seed == SEED_OK && seed_final(s);
        if (seed == SEED_OK && (final || !inner)) {
            const int k[3] = {c[0] - j[0], c[1] - j[1], c[2] - j[2]};
            const Map64<DIM> m(V, k);
            polished = polish<DIM>(m, s, xi, iters);
            if (polished && inner) return ST_OK;
        }
        int dir[3] = {0, 0, 0};
        for (;;) {
            if (!polished) {
                const Solved64 r = solve_element64<T, DIM>(D, n[0], n[1], n[2], c[0], c[1], c[2], j[0], j[1], j[2],
                                                           max_iter, tol);
                const double x[3] = {r.x0, r.x1, r.x2};
                st = r.st;
                *iters += r.iters;
                bool finite = true;
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    xi[a] = x[a];
                    finite &= finite_t(x[a]);
                }
                if (!finite) return st == ST_OK ? ST_NEWTON : st;
            }
#pragma unroll
            for (int a = 0; a < DIM; ++a) dir[a] = xi[a] < -slack ? -1 : (xi[a] > 1.0 + slack ? 1 : 0);
            if ((dir[0] | dir[1] | dir[2]) != 0) break;
            if (!polished || final) return st;
            polished = false;
        }
#pragma unroll
        for (int a = 0; a < DIM; ++a) c[a] += dir[a];
        if (cyc.step(c[0], c[1], c[2])) return ST_LOCATE;
    }
}

}  // namespace
