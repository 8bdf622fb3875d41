// sl_tiled.cu -- dispatch of the FP32 production kernels: 2-D grids go to the two-phase kernel
// (sl_gather2d.cuh; tile configuration 0, where use_gather says), to the persistent kernel with
// TMA-staged windows (sl_remap2d.cuh; tile configurations 6 and 7, up to 3 fields, analytic
// velocities) or to the shared-memory tiled kernels (sl_tile2d.cuh, one translation unit per tile
// configuration; the quintic Z-spline to sl_tiled_z2.cu), 3-D grids to the staged or blocked
// kernels (sl_blocked3d.cu, cubic and linear only).
#include <string.h>

#include "sl_internal.h"

// 2-D: one tiled launch; 3-D: flags with the x-OR, the y/z-OR, one staged or blocked launch
int tiled_kernels_per_call(const sl_grid *g) { return g->dim == 2 ? 1 : 3; }

template <typename T>
bool Launch<T>::tiled_supported(const sl_grid *g)
{
    if (sizeof(T) != 4 || g->desc.walk_start != SL_START_BACKWARD) return false;
    // the 2-D tile bodies invert in FP32 (FP64 re-solves only for failed or degenerate targets):
    // an FP64 inversion of every target runs on the plain kernels
    if (g->dim == 2 && g->desc.newton_mode == SL_NEWTON_F64) return false;
    if (g->desc.max_order > 1) return g->dim == 2 && tiled2d_smem_bytes_z2(g->nfields) <= 200 * 1024;
    // the 3-D kernels form 32-bit node offsets; their blocks are at least 4 rows and planes deep
    if (g->dim == 3) return g->N < (1LL << 31) && (g->n[1] + 3) / 4 <= 65535 && (g->n[2] + 3) / 4 <= 65535;
    const int c = g->desc.tile_config;
    const size_t smem = c == 2   ? tiled2d_smem_bytes_cfgb(g->nfields)
                        : c == 3 ? tiled2d_smem_bytes_cfgc(g->nfields)
                        : c == 4 ? tiled2d_smem_bytes_cfgd(g->nfields)
                                 : tiled2d_smem_bytes_cfga(g->nfields);  // 5 falls back to 1 above 4 fields
    return smem <= 200 * 1024;
}

// Does the two-phase kernel serve this call?  Counted in 32 x 32 tiles of the tiled kernel, whose 3 CTAs
// per SM take up to 456 in one wave.  Measured with warm L2, us a launch, two-phase / tiled:
//   up to 3 fields  256^2 (64 tiles) 7.8 / 10.7, 400^2 (169) 11.2 / 10.8, 513^2 (289) 13.1 / 11.5,
//                   724^2 (529) 17.5 / 19.7, 1024^2 26.9 / 31.5, 2048^2 98.5 / 129: below a fifth of a
//                   wave and above a whole one, and always where the launch also integrates
//                   trajectories (which fill the two-phase kernel's wait: 400^2 13.8 / 15.2, 513^2
//                   16.3 / 16.6) or is a carried step (400^2 11.5 / 11.6, 513^2 13.1 / 13.7);
//   4 fields        (two records a tap) 256^2 9.5 / 11.3, 400^2 13.7 / 11.5, 1024^2 36.3 / 33.6,
//                   1449^2 (2116) 68.0 / 63.2, 2048^2 (4096) 129 / 139: small and large grids only.
static bool use_gather(const sl_grid *g, const void *D_next)
{
    if (g->rec == nullptr) return false;
    const long long tiles = ((g->n[0] + 31) / 32) * ((g->n[1] + 31) / 32), wave = 3LL * g->num_sms;
    if (g->nfields <= 3) return D_next != nullptr || tiles <= wave / 4 || tiles > wave;
    return tiles <= wave / 5 || tiles > 7 * wave;
}

static cudaError_t launch_tiled2d(const sl_grid *g, const void *D, void *D_next, double t_next, double dt, bool fused,
                                  const void *const *in, void *const *out, cudaStream_t s)
{
    if (g->desc.max_order > 1) return launch_tiled2d_z2(g, D, D_next, t_next, dt, fused, in, out, s);
    const int c = g->desc.tile_config;
    if (use_gather(g, D_next)) return launch_gather2d(g, D, D_next, t_next, dt, fused, in, out, s);
    if ((c == 6 || c == 7) && remap2d_tma_supported(g, in, out))
        return launch_remap2d_tma(g, c == 6 ? 6 : 7, D, D_next, t_next, dt, fused, in, out, s);
    switch (c) {
    case 5:
        if (g->nfields <= 4) return launch_tiled2d_cfgp(g, D, D_next, t_next, dt, fused, in, out, s);
        return launch_tiled2d_cfga(g, D, D_next, t_next, dt, fused, in, out, s);
    case 2: return launch_tiled2d_cfgb(g, D, D_next, t_next, dt, fused, in, out, s);
    case 3: return launch_tiled2d_cfgc(g, D, D_next, t_next, dt, fused, in, out, s);
    case 4: return launch_tiled2d_cfgd(g, D, D_next, t_next, dt, fused, in, out, s);
    default: return launch_tiled2d_cfga(g, D, D_next, t_next, dt, fused, in, out, s);
    }
}

template <typename T>
cudaError_t Launch<T>::remap_tiled(const sl_grid *g, const void *D, const void *const *in, void *const *out,
                                   cudaStream_t s)
{
    if (!tiled_supported(g)) return cudaErrorNotSupported;
    if (g->dim == 3) {
        cudaError_t e = launch_box_flags3d(g, in, g->flags, g->flags2, s);
        if (e != cudaSuccess) return e;
        return launch_blocked3d(g, D, nullptr, g->flags2, 0.0, 0.0, false, in, out, s);
    }
    return launch_tiled2d(g, D, nullptr, 0.0, 0.0, false, in, out, s);
}

template <typename T>
cudaError_t Launch<T>::step_fused(const sl_grid *g, const void *D, void *D_next, double t_next, double dt,
                                  const void *const *in, void *const *out, cudaStream_t s)
{
    if (!tiled_supported(g)) return cudaErrorNotSupported;
    if (g->dim == 3) {
        cudaError_t e = launch_box_flags3d(g, in, g->flags, g->flags2, s);
        if (e != cudaSuccess) return e;
        return launch_blocked3d(g, D, D_next, g->flags2, t_next, dt, true, in, out, s);
    }
    return launch_tiled2d(g, D, D_next, t_next, dt, true, in, out, s);
}

template bool Launch<double>::tiled_supported(const sl_grid *);
template bool Launch<float>::tiled_supported(const sl_grid *);
template cudaError_t Launch<double>::remap_tiled(const sl_grid *, const void *, const void *const *, void *const *,
                                                 cudaStream_t);
template cudaError_t Launch<float>::remap_tiled(const sl_grid *, const void *, const void *const *, void *const *,
                                                cudaStream_t);
template cudaError_t Launch<double>::step_fused(const sl_grid *, const void *, void *, double, double,
                                                const void *const *, void *const *, cudaStream_t);
template cudaError_t Launch<float>::step_fused(const sl_grid *, const void *, void *, double, double,
                                               const void *const *, void *const *, cudaStream_t);
