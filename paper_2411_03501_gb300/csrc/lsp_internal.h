// lsp_internal.h -- structures shared by the host layer and the kernels of
// the level-set library.  Not part of the public ABI (see include/lsp.h).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#define LSP_MAXD 4
#define LSP_NPARAM 8

namespace lsp {

enum Scheme { UPWIND1 = 0, ENO2 = 1, ENO3 = 2, WENO5 = 3 };
enum Dyn { NORMAL_SPEED = 0, TRANSLATE = 1, QUADRATIC = 2, AIR3D = 3, CAR4D = 4, ROCKETS = 5,
           DOUBLE_INT = 6 };

__host__ __device__ constexpr int ghost_width(int scheme) { return scheme == UPWIND1 ? 1 : (scheme == ENO2 ? 2 : 3); }

// Streaming multiprocessors of the current device, queried once per device
// index (152 on a GB300), for sizing grids in waves of resident CTAs.
inline int sm_count()
{
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
            n = 1;
        cache[dev] = n;
    }
    return cache[dev];
}

// Device control block, the first 256 bytes of every workspace.
struct Ctl {
    unsigned long long alpha_bits[LSP_MAXD];  // p-dependent GLF alpha (bits of
                                              // a non-negative double; atomicMax)
    double dt;                                // step chosen on the device
    double t;                                 // time after that step
    unsigned int flags;                       // bit 0: non-finite value produced
    unsigned int ticket;                      // blocks done of the costate-range launch
    unsigned int stop_at;                     // steps of the solve once its last is chosen, else 0
    unsigned int pad0;
    unsigned long long acc[LSP_MAXD];         // costate maxima being collected
    unsigned long long steps;                 // steps chosen on the device so far
    double dt_min, dt_max;                    // over those steps
    unsigned long long reserved[8];
};
// flags .. acc are zero at the start of every call that uses the block
constexpr size_t kCtlResetBytes = 4 * sizeof(unsigned int) + LSP_MAXD * sizeof(unsigned long long);
static_assert(sizeof(Ctl) <= 256, "control block must fit 256 bytes");
constexpr size_t kCtlBytes = 256;
constexpr unsigned int kFlagNonFinite = 1u;
constexpr unsigned int kFlagTimeout = 2u;

// Arguments of one fused stage launch.  Every launch computes, at every node,
//   out = c_n * phi_n + c_s * phi_s + c_l * dt * L(phi_s)
// (then min with the target if tube), with L the LF rate.
template <typename R>
struct StageArgs {
    const R* phi_s;     // stage input, read with the stencil
    const R* phi_n;     // phi^n, read pointwise (NULL when c_n == 0)
    const R* target;    // read pointwise when tube != 0
    R* out;             // may alias phi_n (pointwise read before write)
    int n[LSP_MAXD];    // nodes per axis
    int stride[LSP_MAXD];
    int periodic[LSP_MAXD];
    R inv_dx[LSP_MAXD];
    R lo[LSP_MAXD];     // coordinates: lo + i * h
    R h[LSP_MAXD];
    R alpha[LSP_MAXD];  // GLF coefficients (state-only dynamics)
    R prm[LSP_NPARAM];  // dynamics parameters
    R dt, c_n, c_s, c_l;
    int tube;
    int npts;
    Ctl* ctl;            // flags; alpha/dt for p-dependent dynamics
    int alpha_from_ctl;  // 1: read alpha from ctl->alpha_bits
    int dt_from_ctl;     // 1: read dt from ctl->dt
    int local_alpha;     // 1: LLF/LLLF coefficients per node instead of alpha[]
    int varform;         // 1: variational form, rate clipped at zero
    int step;            // with dt_from_ctl: index of the step in the solve
};

// What the costate-range launch does with the maxima (dynamics whose alpha
// depends on the field): 0 alpha alone, 1 also choose the solve's next step,
// 2 its first step.
struct StepChoice {
    int mode;
    double cfl, t0, t_final, t_stop;
    double dx[LSP_MAXD];
};

// Steps to enqueue when `left` steps of the last one's length remain: those and
// 3 % more (the field's range, and with it the step, changes slowly), at most
// 256.  A step too few costs one more read-back, one too many a step's
// launches, and the copy of the field with one stage per step (two steps of
// 1001 nodes, RK3: 125 us with a read-back per step, 147 with one step more
// than `left` rounded up, 122 now).
inline int steps_ahead(double left)
{
    const double n = left * (33.0 / 32.0);
    return n >= 256.0 ? 256 : n > 1.0 ? (int)n + ((double)(int)n < n) : 1;
}

#ifdef __CUDACC__
// Steps are enqueued ahead of the device's choice of dt: those past the last
// one leave every field alone.
template <typename R>
__device__ __forceinline__ bool past_last_step(const StageArgs<R>& a)
{
    if (!a.dt_from_ctl) return false;
    const unsigned stop = a.ctl->stop_at;
    return stop != 0 && (unsigned)a.step >= stop;
}
#endif

#ifdef __CUDACC__
// Stage kernels are launched so that their CTAs start before the previous
// stage has finished (launch_dependent, launch.h): a stage on a small grid is
// a few microseconds, much of it the gap between two launches and the CTA's
// own set-up.  stage_wait returns when every earlier kernel of the stream has
// finished and its writes are visible; stage_release lets the next launch's
// CTAs start.  Nothing that an earlier stage may have written (fields, the
// control block) is touched before stage_wait, and fields are read with
// ordinary loads after it, never through the read-only path, which the wait
// does not order.  Release comes after the wait: released at the top, several
// stages queue up on the SMs and a 101 x 101 FP64 stage takes 6.0 us.  Whole
// solves, ordinary launches -> this: 101 x 101 FP64 graph 515 -> 488 us, 257 x
// 193 FP32 with device-chosen steps 594 -> 405, air3d 41^3 593 -> 385, car4d
// 33 x 41 x 37 x 29 551 -> 516, rockets 300^3 1977 -> 1921.
__device__ __forceinline__ void stage_release()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

}  // namespace lsp
