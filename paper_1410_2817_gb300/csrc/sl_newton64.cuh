// sl_newton64.cuh -- the FP64 element search of Sec. 2.2 with its Newton inversion (eq. mapping1)
// started in FP32, for the plain kernels.
//
// What bounds an FP64 remap on GB300 is the FP64 pipe: 2 results per SM and cycle against 128 for
// FP32, so one FP64 instruction costs as much as 64 FP32 ones, and a dependent one takes 63 cycles.
// The all-FP64 search spends ~150 (2-D) and ~450 (3-D) FP64 instructions per element tried: three
// Newton iterations with their Jacobians, cofactors and divisions.  Here each element is inverted
// in FP32 first; FP64 is used where its digits matter:
//
//   * an element the FP32 solution says is left by more than SEED_MARGIN needs no more digits: the
//     walk steps on;
//   * otherwise the coordinates are polished: x <- x - Ji F(x) with the residual F in FP64 and the
//     inverse Jacobian Ji in FP32, which gains ~6 digits per pass (two passes as a rule, 12 / 42
//     FP64 instructions in 2-D / 3-D), down to the rounding error of F, as the FP64 iteration does.
//
// Conversions between FP32, FP64 and integers take an FP64 slot too and are done by bit operations.
// A 1024^2 x 3 remap issues 113 FP64 instructions per warp where the all-FP64 search needed 263 a target:
// 480 -> 223 us; 64^3 x 2 fields 640 -> 145 us.
//
// Every decision of the FP64 search (fold, no convergence, inside, next element) is taken from the
// FP32 solution only under a certificate (seed_solve): Jacobian determinants at every iterate well
// away from zero, iterates that stay near the element, convergence with iterations to spare.  Then
// the FP64 iteration runs through the same points to 1e-5 and converges to the same root.  Without
// it the element is inverted by the FP64 iteration (newton_solve), as before.
#pragma once

#include <type_traits>

#include "sl_device.cuh"

namespace {

// |det J| relative to the product of the 1-norms of J's columns (1 for a square element): above it
// the FP32 inverse Jacobian is good to ~1e-6.
constexpr float SEED_DET = 0.05f;
// Iterates must stay within this distance of the element: FP32 coordinates that far out are good to
// 128 x 6e-8 / SEED_DET ~ 2e-4, within SEED_MARGIN.  (The failing walks at the seam of a solid-body
// rotation meet sheared elements at coordinates of 30 to 60; with 16 here a quarter of their hops
// took the FP64 iteration, 112 against 21 us per 64^2 step.)
constexpr float SEED_REACH = 128.f;
// columns of J must exceed the FP32 rounding of the vertices by this factor
constexpr float SEED_CLEAR = 1e3f;
// distance from a face beyond which the FP32 coordinates (good to ~1e-5) decide the step
constexpr float SEED_MARGIN = 1e-3f;
// iterations the FP64 solve needs beyond the FP32 one: 3e-4 -> 1e-7 -> 1e-14 -> below its 1e-14 stop
constexpr int SEED_SPARE = 3;

enum { SEED_NONE = 0, SEED_OK = 1, SEED_FOLD = 2 };

template <int DIM>
struct Seed {
    float x[DIM];        // local coordinates
    float Ji[DIM][DIM];  // inverse Jacobian there
    int iters;
};

// FP32 Newton inversion of the bilinear element with vertices P (relative to the target, rounded to
// within `noise`), the iteration of newton_solve2 under the certificate described above.
__device__ __forceinline__ int seed_solve(const float P[4][2], float noise, int max_iter, Seed<2> &r)
{
    const float px = P[0][0], py = P[0][1];
    const float ax = P[1][0] - px, ay = P[1][1] - py, bx = P[2][0] - px, by = P[2][1] - py;
    const float ex = P[3][0] - P[1][0] - bx, ey = P[3][1] - P[1][1] - by;
    float det = ax * by - bx * ay;
    const float na = fabsf(ax) + fabsf(ay), nb = fabsf(bx) + fabsf(by);
    if (!(fabsf(det) > SEED_DET * (na * nb) && fminf(na, nb) > SEED_CLEAR * noise)) return SEED_NONE;
    if (det < 0.f) return SEED_FOLD;
    float inv = recip_t(det);
    float s = -(px * by - py * bx) * inv, t = -(ax * py - ay * px) * inv, step = 1.f;
    for (int it = 0;; ++it) {
        if (!(fabsf(s) <= SEED_REACH && fabsf(t) <= SEED_REACH)) return SEED_NONE;
        const float j11 = ax + t * ex, j21 = ay + t * ey, j12 = bx + s * ex, j22 = by + s * ey;
        det = j11 * j22 - j12 * j21;
        if (!(det > SEED_DET * ((fabsf(j11) + fabsf(j21)) * (fabsf(j12) + fabsf(j22))))) return SEED_NONE;
        inv = recip_t(det);
        if (step <= SL_NEWTON_TOL_F32) {
            r.x[0] = s;
            r.x[1] = t;
            r.Ji[0][0] = j22 * inv;
            r.Ji[0][1] = -j12 * inv;
            r.Ji[1][0] = -j21 * inv;
            r.Ji[1][1] = j11 * inv;
            r.iters = it;
            return SEED_OK;
        }
        if (it + SEED_SPARE >= max_iter) return SEED_NONE;
        const float fx = px + s * j11 + t * bx, fy = py + s * j21 + t * by;
        const float d0 = (fx * j22 - fy * j12) * inv, d1 = (j11 * fy - j21 * fx) * inv;
        s -= d0;
        t -= d1;
        step = fmaxf(fabsf(d0), fabsf(d1));
    }
}

// the same for the trilinear element (vertex v = x + 2 y + 4 z)
__device__ __forceinline__ int seed_solve(const float P[8][3], float noise, int max_iter, Seed<3> &r)
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
    // rows of the cofactor matrix of J give det and the inverse
    auto invert = [](const float J[3][3], float Ji[3][3], float &det, float &norm, float &least) {
        const float c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1], c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2],
                    c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
        det = J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02;
        const float n0 = fabsf(J[0][0]) + fabsf(J[1][0]) + fabsf(J[2][0]),
                    n1 = fabsf(J[0][1]) + fabsf(J[1][1]) + fabsf(J[2][1]),
                    n2 = fabsf(J[0][2]) + fabsf(J[1][2]) + fabsf(J[2][2]);
        norm = n0 * n1 * n2;
        least = fminf(fminf(n0, n1), n2);
        const float inv = recip_t(det);
        Ji[0][0] = c00 * inv;
        Ji[1][0] = c01 * inv;
        Ji[2][0] = c02 * inv;
        Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) * inv;
        Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) * inv;
        Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) * inv;
        Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) * inv;
        Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) * inv;
        Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) * inv;
    };
    float det, norm, least;
    invert(A, r.Ji, det, norm, least);
    if (!(fabsf(det) > SEED_DET * norm && least > SEED_CLEAR * noise)) return SEED_NONE;
    if (det < 0.f) return SEED_FOLD;
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = -(r.Ji[a][0] * P[0][0] + r.Ji[a][1] * P[0][1] + r.Ji[a][2] * P[0][2]);
    float step = 1.f;
    for (int it = 0;; ++it) {
        if (!(fabsf(x[0]) <= SEED_REACH && fabsf(x[1]) <= SEED_REACH && fabsf(x[2]) <= SEED_REACH)) return SEED_NONE;
        const float s01 = x[0] * x[1], s02 = x[0] * x[2], s12 = x[1] * x[2];
        float J[3][3], F[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            J[a][0] = A[a][0] + x[1] * E01[a] + x[2] * E02[a] + s12 * G[a];
            J[a][1] = A[a][1] + x[0] * E01[a] + x[2] * E12[a] + s02 * G[a];
            J[a][2] = A[a][2] + x[0] * E02[a] + x[1] * E12[a] + s01 * G[a];
            F[a] = P[0][a] + x[0] * J[a][0] + x[1] * (A[a][1] + x[2] * E12[a]) + x[2] * A[a][2];
        }
        invert(J, r.Ji, det, norm, least);
        if (!(det > SEED_DET * norm)) return SEED_NONE;
        if (step <= SL_NEWTON_TOL_F32) {
#pragma unroll
            for (int a = 0; a < 3; ++a) r.x[a] = x[a];
            r.iters = it;
            return SEED_OK;
        }
        if (it + SEED_SPARE >= max_iter) return SEED_NONE;
        step = 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float d = r.Ji[a][0] * F[0] + r.Ji[a][1] * F[1] + r.Ji[a][2] * F[2];
            x[a] -= d;
            step = fmaxf(step, fabsf(d));
        }
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

// x <- x - Ji F(x) until a pass moves x by no more than 3e-11: what is left is that times the error
// of Ji (~1e-6), below FP64 rounding.  False where it does not settle.
template <int DIM>
__device__ __forceinline__ bool polish(const Map64<DIM> &m, const Seed<DIM> &s, double x[3], int *iters)
{
#pragma unroll
    for (int a = 0; a < DIM; ++a) x[a] = widen(s.x[a]);
    for (int it = 0; it < 4; ++it) {
        float F[DIM], big = 0.f;
        m.residual(x, F);
        *iters += 1;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            float d = 0.f;
#pragma unroll
            for (int b = 0; b < DIM; ++b) d += s.Ji[a][b] * F[b];
            if (!(fabsf(d) <= 0.2f * SEED_MARGIN)) return false;
            x[a] -= widen(d);
            big = fmaxf(big, fabsf(d));
        }
        if (big <= 3e-11f) return true;
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
        bool inner = false;  // inside the element by SEED_MARGIN (polishing moves x by less)
        for (;;) {
            if (hop >= walk_max) return ST_LOCATE;
            load_vertices<T, DIM>(D, n, c, V);
            float P[1 << DIM][DIM], big = 1.f;
#pragma unroll
            for (int v = 0; v < (1 << DIM); ++v)
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    const float f = narrow(V[v][a]);
                    big = fmaxf(big, fabsf(f));
                    P[v][a] = (float)(c[a] + ((v >> a) & 1) - j[a]) + f;
                }
            seed = seed_solve(P, 2.4e-7f * big, max_iter, s);
            ++hop;
            *hops += 1;
            if (seed != SEED_OK) break;
            *iters += s.iters;
            bool clear = true, out = false;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                clear &= fabsf(s.x[a]) > SEED_MARGIN && fabsf(s.x[a] - 1.f) > SEED_MARGIN;
                out |= s.x[a] < 0.f || s.x[a] > 1.f;
            }
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
        if (seed == SEED_OK) {
            const int k[3] = {c[0] - j[0], c[1] - j[1], c[2] - j[2]};
            const Map64<DIM> m(V, k);
            if (!polish<DIM>(m, s, xi, iters))
                seed = SEED_NONE;
            else if (inner)
                return ST_OK;
        }
        if (seed == SEED_NONE) {
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
        int dir[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < DIM; ++a) dir[a] = xi[a] < -slack ? -1 : (xi[a] > 1.0 + slack ? 1 : 0);
        if ((dir[0] | dir[1] | dir[2]) == 0) return st;
#pragma unroll
        for (int a = 0; a < DIM; ++a) c[a] += dir[a];
        if (cyc.step(c[0], c[1], c[2])) return ST_LOCATE;
    }
}

}  // namespace
