// stage_march.inl -- instantiations and launcher of the register-marching
// ENO2/ENO3 stage kernel (stage_march.cuh), Tile.pair = 6, for one
// number of dimensions LSP_MARCH_NDIM (included by stage_march_3d.cu and
// stage_march_4d.cu).
#include "launch.h"
#include "stage_march.cuh"

namespace lsp {

namespace {

constexpr int ND = LSP_MARCH_NDIM;

template <int SCHEME, int DYN>
cudaError_t march_launch(const StageArgs<float>& a, const Tile& t, cudaStream_t s)
{
    constexpr int R0 = march_slabs(ND), G = ghost_width(SCHEME);
    const int nB = a.n[ND - 1], nA = a.n[ND - 2], nS = a.n[ND - 3];
    const int nchunks = (nS + t.ch - 1) / t.ch;
    dim3 grid((nB + t.tb - 1) / t.tb, (nA + t.ta - 1) / t.ta,
              nchunks * (ND == 4 ? (a.n[0] + R0 - 1) / R0 : 1));
    const size_t smem = 2 * sizeof(float) * R0 * (t.ta + 2 * G) * kMarchPitch;
    const int threads = march_threads(t);
    // In 4-D a launch of many waves is faster as an ordinary one (us per stage,
    // ordinary and dependent: car4d 81^4, 27 planes, 6 waves 425, 480; 33 x 41
    // x 37 x 29, one wave 23.2, 21.7).  In 3-D the dependent form is faster
    // there too (rockets 300^3 161, 157; 100^3 11.0, 8.9).
    if constexpr (ND == 4) {
        constexpr int kResident = 65536 / 128;  // threads of an SM
        const long long ctas = (long long)grid.x * grid.y * grid.z;
        if (ctas * threads > 4LL * kResident * sm_count()) {
            auto* fn = stage_march_kernel<ND, SCHEME, DYN, LSP_MARCH_MINB, false>;
            if (const cudaError_t e = allow_smem(fn, smem, kRunMaxSmem)) return e;
            fn<<<grid, threads, smem, s>>>(a, t.tb, t.ta, t.ch, nchunks);
            return cudaGetLastError();
        }
    }
    auto* fn = stage_march_kernel<ND, SCHEME, DYN, LSP_MARCH_MINB, true>;
    if (const cudaError_t e = allow_smem(fn, smem, kRunMaxSmem)) return e;
    return launch_dependent(fn, grid, threads, smem, s, a, t.tb, t.ta, t.ch, nchunks);
}

template <int SCHEME>
cudaError_t march_dyn(int dyn, const StageArgs<float>& a, const Tile& t, cudaStream_t s)
{
    switch (dyn) {
    case NORMAL_SPEED: return march_launch<SCHEME, NORMAL_SPEED>(a, t, s);
    case TRANSLATE: return march_launch<SCHEME, TRANSLATE>(a, t, s);
    case QUADRATIC: return march_launch<SCHEME, QUADRATIC>(a, t, s);
    case AIR3D:
        if constexpr (ND == 3) return march_launch<SCHEME, AIR3D>(a, t, s);
        break;
    case ROCKETS:
        if constexpr (ND == 3) return march_launch<SCHEME, ROCKETS>(a, t, s);
        break;
    case CAR4D:
        if constexpr (ND == 4) return march_launch<SCHEME, CAR4D>(a, t, s);
        break;
    }
    return cudaErrorInvalidValue;
}

}  // namespace

template <>
cudaError_t launch_stage_march<LSP_MARCH_NDIM>(int scheme, int dyn, const StageArgs<float>& a,
                                               const Tile& t, cudaStream_t s)
{
    if (scheme == ENO2) return march_dyn<ENO2>(dyn, a, t, s);
    if (scheme == ENO3) return march_dyn<ENO3>(dyn, a, t, s);
    return cudaErrorInvalidValue;
}

}  // namespace lsp
