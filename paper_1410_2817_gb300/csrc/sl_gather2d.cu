// sl_gather2d.cu -- launches of the two-phase 2-D FP32 step (sl_gather2d.cuh).
#include <atomic>

#include "sl_gather2d.cuh"

// records of a grid with n0 x n1 nodes: one plane per group, each on a 256-byte boundary
static size_t plane_bytes(long long n0, long long n1, int nc)
{
    const size_t b = (size_t)(n0 + REC_LO + REC_HI) * (size_t)(n1 + REC_LO + REC_HI) * (nc == 1 ? 8 : 16);
    return (b + 255) & ~(size_t)255;
}
size_t gather2d_record_bytes(long long n0, long long n1, int nfields)
{
    size_t b = 0;
    for (int q = 0; q < rec_groups(nfields); ++q) b += plane_bytes(n0, n1, in_rec(nfields, q));
    return b;
}

template <int NF, bool FUSED>
static cudaError_t launch_gather_nf(const sl_grid *g, GatherArgs &A, const VelArgs<float> &vn, cudaStream_t s)
{
    // CTAs per SM, looked up once per device (threads of several grids may meet here)
    static std::atomic<int> per_sm[64];
    int n = per_sm[g->device & 63].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, gather2d_kernel<NF, FUSED>, GNT, 0);
        if (e != cudaSuccess) return e;
        if (n < 1) return cudaErrorInvalidConfiguration;
        per_sm[g->device & 63].store(n, std::memory_order_relaxed);
    }
    const long long ctas = std::min<long long>(A.ntiles, (long long)g->num_sms * n);
    A.step_y = (int)(ctas % A.tiles_y);
    A.step_x = (int)(ctas / A.tiles_y) * GTX;
    gather2d_kernel<NF, FUSED><<<(unsigned)ctas, GNT, 0, s>>>(A, vn);
    return cudaGetLastError();
}

template <bool FUSED>
static cudaError_t launch_gather(const sl_grid *g, GatherArgs &A, const VelArgs<float> &vn, cudaStream_t s)
{
    switch (g->nfields) {
    case 1: return launch_gather_nf<1, FUSED>(g, A, vn, s);
    case 2: return launch_gather_nf<2, FUSED>(g, A, vn, s);
    case 3: return launch_gather_nf<3, FUSED>(g, A, vn, s);
    default: return launch_gather_nf<4, FUSED>(g, A, vn, s);
    }
}

cudaError_t launch_gather2d(const sl_grid *g, const void *D, void *D_next, double t_next, double dt, bool fused,
                            const void *const *in, void *const *out, cudaStream_t s)
{
    GatherArgs A;
    memset(&A, 0, sizeof(A));
    A.t = make_tile_args(g, D, D_next, in, out);
    char *rec = (char *)g->rec;
    for (int q = 0; q < rec_groups(g->nfields); ++q) {
        const int nc = in_rec(g->nfields, q);
        const size_t first = (size_t)REC_LO * (size_t)(g->n[0] + REC_LO + REC_HI) + REC_LO;
        A.rec[q] = rec + first * (nc == 1 ? 8 : 16);
        rec += plane_bytes(g->n[0], g->n[1], nc);
    }
    A.sync = g->sync;
    A.timeouts = &g->counters->timeouts;
    A.reach0 = (float)g->n[0] - 12.f;
    A.reach1 = (float)g->n[1] - 12.f;
    A.tiles_y = (int)((g->n[1] + GTY - 1) / GTY);
    A.ntiles = (int)((g->n[0] + GTX - 1) / GTX) * A.tiles_y;
    A.strips = (int)((g->n[0] + GCOLS - 1) / GCOLS);
    A.nflag = A.strips * (int)((g->n[1] + GROWS - 1) / GROWS);
    A.hops = std::min(GHOPS, A.t.walk_max);
    A.nclaim = (A.nflag + GNT / 32 - 1) / (GNT / 32);
    VelArgs<float> vn;
    memset(&vn, 0, sizeof(vn));
    if (!fused) return launch_gather<false>(g, A, vn, s);
    set_carried(g, dt, A.t);
    vn = make_vel_args<float>(g, t_next, dt);
    return launch_gather<true>(g, A, vn, s);
}
