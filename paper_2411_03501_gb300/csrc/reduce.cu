// reduce.cu -- the once-per-grid reduction that yields the global-LF
// coefficients for state-only bounds (Listing 4: artificialDissipationGLF
// with partialFunc; alpha_k = max over the grid of the bound on |dH/dp_k|).
#include "launch.h"
#include "stage_generic.cuh"
#include "stage_march.cuh"
#include "stage_tiled.cuh"
#include "adjoint.cuh"

namespace lsp {

cudaError_t launch_alpha_state(int dyn, const GridGeom& g, unsigned long long* out, cudaStream_t s)
{
    long long b = (g.npts + 255) / 256;
    const long long cap = 8LL * sm_count();
    const int nb = (int)(b < cap ? (b < 1 ? 1 : b) : cap);
    switch (dyn) {
    case NORMAL_SPEED: alpha_state_kernel<NORMAL_SPEED><<<nb, 256, 0, s>>>(g, out); break;
    case TRANSLATE: alpha_state_kernel<TRANSLATE><<<nb, 256, 0, s>>>(g, out); break;
    case AIR3D: alpha_state_kernel<AIR3D><<<nb, 256, 0, s>>>(g, out); break;
    case CAR4D: alpha_state_kernel<CAR4D><<<nb, 256, 0, s>>>(g, out); break;
    case ROCKETS: alpha_state_kernel<ROCKETS><<<nb, 256, 0, s>>>(g, out); break;
    case DOUBLE_INT: alpha_state_kernel<DOUBLE_INT><<<nb, 256, 0, s>>>(g, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

bool tile_valid(int ndim, int scheme, const Tile& t, const int* n)
{
    if (ndim != 3 && ndim != 4) return false;
    const int G = ghost_width(scheme);
    if (t.tb < 1 || t.ta < 1 || t.ch < 1) return false;
    if (t.minb < 2 || t.minb > 4) return false;
    const int nS = n[ndim - 3];
    const long long nz = (long long)((nS + t.ch - 1) / t.ch) * (ndim == 4 ? n[0] : 1);
    if (t.pair == 6) return march_tile_ok(ndim, scheme, t, n);
    if (t.pair == 5) return fused_tile_ok(ndim, scheme, t, n);  // temporally blocked RK2
    if (t.pair == 3 || t.pair == 4) {  // face-shared ENO runs of 4 or 2 nodes
        return (scheme == ENO2 || scheme == ENO3) &&
               run_tile_ok(ndim, scheme, t.pair == 3 ? 4 : 2, t.tb, t.ta) && nz <= 65535;
    }
    if (t.tb * t.ta > 256) return false;
    // pair 1: paired planes (WENO5, ENO2, ENO3); pair 2: WENO5 shared faces
    if (t.pair < 0 || t.pair > 2) return false;
    if (t.pair == 1 && scheme != WENO5 && scheme != ENO2 && scheme != ENO3) return false;
    if (t.pair == 2 && scheme != WENO5) return false;
    // each thread stages at most 3 values of the haloed plane tile (MAXE of
    // the tiled bodies; every shape the autotuner tries qualifies)
    if ((t.ta + 2 * G) * (t.tb + 2 * G) > 3 * t.ta * t.tb) return false;
    return nz <= 65535;
}

bool march_tile_ok(int ndim, int scheme, const Tile& t, const int* n)
{
    if (scheme != ENO2 && scheme != ENO3) return false;
    const int G = ghost_width(scheme), ra = kMarchRows, r0 = march_slabs(ndim);
    const int nB = n[ndim - 1], nA = n[ndim - 2], nS = n[ndim - 3];
    // whole tiles inside the grid, whole blocks of rows
    if (t.tb < 1 || t.tb > kMarchMaxTB || t.tb > nB || t.ta < ra || t.ta % ra || t.ta > nA) return false;
    if (ndim == 4 && n[0] < r0) return false;
    const int threads = march_threads(t);
    if (threads > kMarchThreads) return false;
    // the tile's frame in kMarchSlots values per thread
    if (2 * G * (t.tb + t.ta) > kMarchSlots * threads) return false;
    if (2 * sizeof(float) * r0 * (size_t)(t.ta + 2 * G) * kMarchPitch > kRunMaxSmem) return false;
    long long npts = 1;  // 32-bit offsets inside a plane
    for (int k = 0; k < ndim; ++k) npts *= n[k];
    const long long nz = (long long)((nS + t.ch - 1) / t.ch) * (ndim == 4 ? (n[0] + r0 - 1) / r0 : 1);
    return npts < (1LL << 30) && nz <= 65535 && (nA + t.ta - 1) / t.ta <= 65535;
}

bool run_tile_ok(int ndim, int scheme, int run, int tb, int ta)
{
    if (tb != 16 && tb != 28 && tb != 32) return false;
    const int tbt = tb / run, G = ghost_width(scheme);
    const size_t floats = (size_t)(ta + 2 * G) * (tb + 8) +
                          (size_t)((ndim == 4 ? 2 * G : 0) + 3) * ta * tb;
    return ta >= 1 && tbt * ta <= 256 && 2 * sizeof(float) * floats <= kRunMaxSmem;
}

// One node per thread in the chunks of a run or march tile.  A march's blocks
// hold 2 slabs of axis 0 (4-D), these one: longer chunks where the launch
// would pass 65535 z-blocks; ch = 0 when no chunk avoids that.
static Tile local_tile(int ndim, const Tile& t, const int* n)
{
    Tile l{32, 8, t.ch, 3, 0};
    const int nS = n[ndim - 3], outer = ndim == 4 ? n[0] : 1;
    const int most = 65535 / outer;  // chunks
    if (most < 1 || (n[ndim - 2] + l.ta - 1) / l.ta > 65535) l.ch = 0;
    else if ((nS + l.ch - 1) / l.ch > most) l.ch = (nS + most - 1) / most;
    return l;
}

cudaError_t launch_stage_tiled(int ndim, int scheme, int dyn, const StageArgs<float>& a,
                               const Tile& t, cudaStream_t s)
{
    // local coefficients and the variational clip run the scalar local
    // bodies, except on the WENO5 shared-face tile with state-only bounds,
    // whose kernel has a local variant
    if ((a.local_alpha || a.varform) && !(scheme == WENO5 && t.pair == 2 && dyn != QUADRATIC)) {
        // the face-shared runs and marches have no local variant: a one-node-per-thread
        // tile of the same chunking runs the local body
        if (t.pair != 3 && t.pair != 4 && t.pair != 6)
            return launch_stage_tiled_local(ndim, scheme, dyn, a, Tile{t.tb, t.ta, t.ch, t.minb, 0}, s);
        const Tile tl = local_tile(ndim, t, a.n);
        return tl.ch > 0 ? launch_stage_tiled_local(ndim, scheme, dyn, a, tl, s)
                         : launch_stage<float>(ndim, scheme, dyn, a, s);
    }
    if (t.pair == 5) {  // a single stage on a fused-RK2 tile: the scalar body
        const Tile ts{t.tb, t.ta, t.ch, t.minb, 0};
        return launch_stage_tiled(ndim, scheme, dyn, a, ts, s);
    }
    if (t.pair == 6)
        return ndim == 3 ? launch_stage_march<3>(scheme, dyn, a, t, s)
                         : launch_stage_march<4>(scheme, dyn, a, t, s);
    if (t.pair == 3) return launch_stage_run_r<4>(ndim, scheme, dyn, a, t, s);
    if (t.pair == 4) return launch_stage_run_r<2>(ndim, scheme, dyn, a, t, s);
    switch (t.minb) {
    case 2: return launch_stage_tiled_m<2>(ndim, scheme, dyn, a, t, s);
    case 3: return launch_stage_tiled_m<3>(ndim, scheme, dyn, a, t, s);
    case 4: return launch_stage_tiled_m<4>(ndim, scheme, dyn, a, t, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_alpha_argmax(int dyn, const GridGeom& g, const double* alpha,
                                unsigned long long* out, cudaStream_t s)
{
    long long b = (g.npts + 255) / 256;
    const long long cap = 8LL * sm_count();
    const int nb = (int)(b < cap ? (b < 1 ? 1 : b) : cap);
    switch (dyn) {
    case NORMAL_SPEED: alpha_argmax_kernel<NORMAL_SPEED><<<nb, 256, 0, s>>>(g, alpha, out); break;
    case TRANSLATE: alpha_argmax_kernel<TRANSLATE><<<nb, 256, 0, s>>>(g, alpha, out); break;
    case AIR3D: alpha_argmax_kernel<AIR3D><<<nb, 256, 0, s>>>(g, alpha, out); break;
    case CAR4D: alpha_argmax_kernel<CAR4D><<<nb, 256, 0, s>>>(g, alpha, out); break;
    case ROCKETS: alpha_argmax_kernel<ROCKETS><<<nb, 256, 0, s>>>(g, alpha, out); break;
    case DOUBLE_INT: alpha_argmax_kernel<DOUBLE_INT><<<nb, 256, 0, s>>>(g, alpha, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

bool stage_supported(int ndim, int scheme, int dyn)
{
    if (ndim < 1 || ndim > LSP_MAXD || scheme < UPWIND1 || scheme > WENO5) return false;
    if (dyn == AIR3D) return ndim == 3;
    if (dyn == CAR4D) return ndim == 4;
    if (dyn == ROCKETS) return ndim == 3;
    if (dyn == DOUBLE_INT) return ndim == 2;
    return dyn >= NORMAL_SPEED && dyn <= QUADRATIC;
}

}  // namespace lsp
