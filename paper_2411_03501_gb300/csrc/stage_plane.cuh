// stage_plane.cuh -- the fused Runge-Kutta stage (Sec. V-A) and the costate
// range on 2-D grids, one thread per node, both precisions, every scheme.
//
// Same computation as stage_generic_kernel (stage_generic.cuh).  What bounds
// it is latency on small grids and, in FP64, the FP64 pipe of GB300 (2
// operations per SM and cycle): a stage of the 101 x 101 front is 10^4 nodes
// of about 45 FP64 operations.  So
//  - the block size is chosen to spread the nodes evenly over every SM
//    (plane_block: 96 threads for 101 x 101, 107 SMs busy instead of 40);
//  - index arithmetic is 32-bit, and all loads are requested at once:
//    windows next to an edge load wrapped or clamped nodes and have their
//    ghosts (Sec. III-B) replaced in registers;
//  - FP64 maxima and the finiteness test run on the bits of the values in the
//    integer pipe, the launch's constants come from the host (PlaneConst),
//    and WENO5 divides once per side instead of four times.  Otherwise the
//    operations and their order are the generic kernel's (first order, ENO2
//    and ENO3 give its results to the rounding of products that the compiler
//    fuses into sums).
// Measured (GB300, us per stage of whole solves, generic kernel before):
// 101 x 101 FP64 ENO2 8.7, 5.0; 127 x 93 FP64 WENO5 31.8, 13.6; 513 x 401
// FP64 WENO5 176, 128 (the FP64 pipe); 301 x 177 FP32 WENO5 6.6, 3.9; 4096^2
// FP32 first order 179, 93, WENO5 436, 276; 4096^2 FP64 first order 1019,
// 1014, ENO2 1596, 1642, ENO3 2474, 2485, WENO5 11470, 9720 (84 % of the FP64
// pipe; ENO2 executes one FP64 instruction more per axis than the generic
// kernel, found in the counters and not explained).  The
// Jiang-Peng form of WENO5 (stage_tiled.cuh) with one division takes 10-15 %
// less in FP64, but its error against FP64 torch was 2-15 % above the
// generic kernel's on four cases and it was not kept.
#pragma once
#include "stage_generic.cuh"

namespace lsp {

// |a| <= |b| (false when either is NaN).
template <typename R>
__device__ __forceinline__ bool mag_le(R a, R b) { return rabs(a) <= rabs(b); }
__device__ __forceinline__ unsigned long long mag_bits(double a)
{
    return (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
}
// max(|a|, |b|) of finite values (a NaN operand gives NaN)
__device__ __forceinline__ float mag_max(float a, float b) { return fmaxf(fabsf(a), fabsf(b)); }
__device__ __forceinline__ double mag_max(double a, double b)
{
    const unsigned long long ia = mag_bits(a), ib = mag_bits(b);
    return __longlong_as_double((long long)(ia > ib ? ia : ib));
}
__device__ __forceinline__ bool is_finite_bits(float v) { return isfinite(v); }
__device__ __forceinline__ bool is_finite_bits(double v)
{
    return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}

// Power of two that scales q_k = s_k + eps of the WENO5 weights (plane_weno),
// from eps alone, which is known before the q_k.  Close to 1/eps: then 1 <= q_k
// <= 4e7, and the products of weights and stencil values reach 3e30 max|v|,
// which overflows FP32 on rough data from undivided differences of 1e8 on.  In
// FP32 q_k is therefore scaled 2^13 lower where eps >= 1 (differences from 1e3
// on): 1.2e-4 <= q_k <= 5e3, products up to 6e14 max|v|, finite up to
// differences of 1e18.
__device__ __forceinline__ float weight_scale(float eps)
{
    const unsigned drop = eps >= 1.0f ? 13u << 23 : 0u;
    return __uint_as_float(0x7f000000u - (__float_as_uint(eps) & 0x7f800000u) - drop);
}
__device__ __forceinline__ double weight_scale(double eps)
{
    return __longlong_as_double(0x7fe0000000000000ll -
                                (__double_as_longlong(eps) & 0x7ff0000000000000ll));
}

// weno5_combine (stencil.cuh) with one division instead of four: the weights
// alpha_k = c_k / q_k^2 are multiplied by (q_1 q_2 q_3)^2, after q_k has been
// scaled by a power of two (exact).  Finite wherever the form with four
// divisions is (in FP32 its squares overflow from differences of 1e9 on), up
// to differences of 1e18 in FP32 and 1e150 in FP64.
template <typename R>
__device__ __forceinline__ R plane_weno(R v1, R v2, R v3, R v4, R v5, R floor_)
{
    const R phi1 = v1 * R(1.0 / 3.0) - v2 * R(7.0 / 6.0) + v3 * R(11.0 / 6.0);
    const R phi2 = -v2 * R(1.0 / 6.0) + v3 * R(5.0 / 6.0) + v4 * R(1.0 / 3.0);
    const R phi3 = v3 * R(1.0 / 3.0) + v4 * R(5.0 / 6.0) - v5 * R(1.0 / 6.0);
    const R a1 = v1 - R(2) * v2 + v3, b1 = v1 - R(4) * v2 + R(3) * v3;
    const R a2 = v2 - R(2) * v3 + v4, b2 = v2 - v4;
    const R a3 = v3 - R(2) * v4 + v5, b3 = R(3) * v3 - R(4) * v4 + v5;
    const R s1 = R(13.0 / 12.0) * a1 * a1 + R(0.25) * b1 * b1;
    const R s2 = R(13.0 / 12.0) * a2 * a2 + R(0.25) * b2 * b2;
    const R s3 = R(13.0 / 12.0) * a3 * a3 + R(0.25) * b3 * b3;
    const R m = mag_max(mag_max(mag_max(v1, v2), mag_max(v3, v4)), v5);
    const R eps = R(1e-6) * (m * m) + floor_;
    const R sc = weight_scale(eps);
    const R q1 = (s1 + eps) * sc, q2 = (s2 + eps) * sc, q3 = (s3 + eps) * sc;
    const R Q1 = q1 * q1, Q2 = q2 * q2, Q3 = q3 * q3;
    const R al1 = R(0.1) * (Q2 * Q3), al2 = R(0.6) * (Q1 * Q3), al3 = R(0.3) * (Q1 * Q2);
    return (al1 * phi1 + al2 * phi2 + al3 * phi3) / (al1 + al2 + al3);
}

// dx p- and dx p+ from the window u[0..2G].
template <int SCHEME, typename R>
__device__ __forceinline__ void plane_derivs(const R* u, R floor_, R& am, R& ap)
{
    if constexpr (SCHEME == UPWIND1) {
        am = u[1] - u[0];
        ap = u[2] - u[1];
    } else if constexpr (SCHEME == ENO2) {
        const R dm2 = u[1] - u[0], dm1 = u[2] - u[1], d0 = u[3] - u[2], d1 = u[4] - u[3];
        const R Sm1 = dm1 - dm2, S0 = d0 - dm1, S1 = d1 - d0;
        am = rfma(R(0.5), mag_le(Sm1, S0) ? Sm1 : S0, dm1);
        ap = rfma(R(-0.5), mag_le(S0, S1) ? S0 : S1, d0);
    } else if constexpr (SCHEME == ENO3) {
        const R dm3 = u[1] - u[0], dm2 = u[2] - u[1], dm1 = u[3] - u[2];
        const R d0 = u[4] - u[3], d1 = u[5] - u[4], d2 = u[6] - u[5];
        const R Sm2 = dm2 - dm3, Sm1 = dm1 - dm2, S0 = d0 - dm1, S1 = d1 - d0, S2 = d2 - d1;
        const R Tm2 = Sm1 - Sm2, Tm1 = S0 - Sm1, T0 = S1 - S0, T1 = S2 - S1;
        // smaller third difference of each node's pair (deriv_eno3)
        const R Mm1 = mag_le(Tm2, Tm1) ? Tm2 : Tm1, M0 = mag_le(Tm1, T0) ? Tm1 : T0;
        const R M1 = mag_le(T0, T1) ? T0 : T1;
        const bool l = mag_le(Sm1, S0), r = mag_le(S0, S1);
        am = rfma(l ? Mm1 : M0, l ? R(1.0 / 3.0) : R(-1.0 / 6.0), rfma(R(0.5), l ? Sm1 : S0, dm1));
        ap = rfma(r ? M0 : M1, r ? R(-1.0 / 6.0) : R(1.0 / 3.0), rfma(R(-0.5), r ? S0 : S1, d0));
    } else {
        const R dm3 = u[1] - u[0], dm2 = u[2] - u[1], dm1 = u[3] - u[2];
        const R d0 = u[4] - u[3], d1 = u[5] - u[4], d2 = u[6] - u[5];
        am = plane_weno(dm3, dm2, dm1, d0, d1, floor_);
        ap = plane_weno(d2, d1, d0, dm1, dm2, floor_);
    }
}

// Window of node c of a line of n nodes with stride s through p (the node's
// own address), ghosts substituted.
template <int G, typename R>
__device__ __forceinline__ void plane_window(const R* p, int c, int n, int s,
                                             int periodic, R* u)
{
    const bool inside = c >= G && c + G < n;
#pragma unroll
    for (int o = -G; o <= G; ++o) {
        int off = o * s;
        if (!inside) off = (into_axis(c + o, n, periodic) - c) * s;
        u[o + G] = p[off];
    }
    if (!inside && !periodic) fix_extrapolated<1, G>(u, c, n);
}

// Constants of a launch.  FP64: formed on the host, since a thread has few
// nodes and what it forms once costs FP64 operations (101 x 101 FP64 ENO2 4.6
// -> 4.4 us per stage of a graph; 2048^2 FP64 first order 282 -> 264).  FP32:
// formed by each thread, 1 to 2 % faster than loading them (4096^2 ENO3 162.3,
// 160.1 us).
template <typename R>
struct PlaneConst;

template <>
struct PlaneConst<float> {
    explicit PlaneConst(const StageArgs<float>&) {}
    __device__ __forceinline__ float rate_factor(const StageArgs<float>& a) const  // c_l dt
    {
        return a.c_l * (a.dt_from_ctl ? float(a.ctl->dt) : a.dt);
    }
    __device__ __forceinline__ float half_alpha(const StageArgs<float>& a, int k) const
    {
        return (a.alpha_from_ctl ? float(__longlong_as_double((long long)a.ctl->alpha_bits[k])) : a.alpha[k]) *
               0.5f;
    }
    __device__ __forceinline__ float floor_(const StageArgs<float>& a, int k) const
    {
        return Num<float>::eps_floor(a.inv_dx[k]);
    }
};

template <>
struct PlaneConst<double> {
    double cl, half[2], fl[2];
    explicit PlaneConst(const StageArgs<double>& a)
    {
        cl = a.c_l * a.dt;
        for (int k = 0; k < 2; ++k) {
            half[k] = a.alpha[k] * 0.5;
            fl[k] = Num<double>::eps_floor(a.inv_dx[k]);
        }
    }
    __device__ __forceinline__ double rate_factor(const StageArgs<double>& a) const
    {
        return a.dt_from_ctl ? a.c_l * a.ctl->dt : cl;
    }
    __device__ __forceinline__ double half_alpha(const StageArgs<double>& a, int k) const
    {
        return a.alpha_from_ctl ? __longlong_as_double((long long)a.ctl->alpha_bits[k]) * 0.5 : half[k];
    }
    __device__ __forceinline__ double floor_(const StageArgs<double>&, int k) const { return fl[k]; }
};

// A thread takes one node (FP32) or the nodes of a grid-stride loop (FP64, at
// most 16 blocks per SM: 4096^2 first order 1038 us in one pass of blocks,
// 1014 in the loop).
template <int SCHEME, int DYN, typename R>
__global__ void __launch_bounds__(256) stage_plane_kernel(StageArgs<R> a, PlaneConst<R> pc)
{
    constexpr int G = ghost_width(SCHEME);
    unsigned idx = blockIdx.x * blockDim.x + threadIdx.x;
    int i = (int)(idx / (unsigned)a.n[1]), j = (int)(idx - (unsigned)i * (unsigned)a.n[1]);
    stage_wait();
    stage_release();
    if (idx >= (unsigned)a.npts || past_last_step(a)) return;
    for (;;) {
        R u[2][2 * G + 1];
        plane_window<G>(a.phi_s + idx, i, a.n[0], a.stride[0], a.periodic[0], u[0]);
        plane_window<G>(a.phi_s + idx, j, a.n[1], 1, a.periodic[1], u[1]);
        const R vn = a.phi_n ? a.phi_n[idx] : R(0);
        const R g = a.tube ? a.target[idx] : R(0);
        const R cl = pc.rate_factor(a);
        const R x[2] = {rfma(R(i), a.h[0], a.lo[0]), rfma(R(j), a.h[1], a.lo[1])};
        R pbar[2], diss = R(0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            R pm, pp;
            plane_derivs<SCHEME>(u[k], pc.floor_(a, k), pm, pp);
            pm *= a.inv_dx[k];
            pp *= a.inv_dx[k];
            R ha = pc.half_alpha(a, k);
            if (a.local_alpha) ha = local_alpha<DYN>(x, k, a.prm, R(0), R(1), pm, pp) * R(0.5);
            pbar[k] = R(0.5) * (pp + pm);
            diss += ha * (pp - pm);
        }
        const R H = hamiltonian<DYN, 2>(x, pbar, a.prm);
        R L = -(H - diss);
        if (a.varform) L = rmin(L, R(0));
        R v = a.c_s * u[1][G] + cl * L;
        if (a.phi_n) v += a.c_n * vn;
        if (a.tube) v = rmin(v, g);
        if (!is_finite_bits(v)) atomicOr(&a.ctl->flags, kFlagNonFinite);
        a.out[idx] = v;
        if constexpr (sizeof(R) == 4) return;
        idx += gridDim.x * blockDim.x;  // below 2^31 + 2^23
        if (idx >= (unsigned)a.npts) return;
        i = (int)(idx / (unsigned)a.n[1]);
        j = (int)(idx - (unsigned)i * (unsigned)a.n[1]);
    }
}

// prange_kernel (stage_generic.cuh) on 2-D grids.
template <int SCHEME, typename R>
__global__ void __launch_bounds__(256) prange_plane_kernel(StageArgs<R> a, PlaneConst<R> pc, StepChoice ch)
{
    stage_wait();
    stage_release();
    constexpr int G = ghost_width(SCHEME);
    if (past_last_step(a)) return;
    const unsigned idx = blockIdx.x * blockDim.x + threadIdx.x;
    R m[2] = {R(0), R(0)};
    if (idx < (unsigned)a.npts) {
        const int i = (int)(idx / (unsigned)a.n[1]), j = (int)(idx - (unsigned)i * (unsigned)a.n[1]);
        R u[2][2 * G + 1];
        plane_window<G>(a.phi_s + idx, i, a.n[0], a.stride[0], a.periodic[0], u[0]);
        plane_window<G>(a.phi_s + idx, j, a.n[1], 1, a.periodic[1], u[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            R am, ap;
            plane_derivs<SCHEME>(u[k], pc.floor_(a, k), am, ap);
            m[k] = rmax(rabs(am), rabs(ap)) * a.inv_dx[k];
        }
    }
    __shared__ R sm[2][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[k] = rmax(m[k], __shfl_xor_sync(0xffffffffu, m[k], o));
        if (lane == 0) sm[k][warp] = m[k];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        R v = R(0);
        if (threadIdx.x < 2)
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = rmax(v, sm[threadIdx.x][w]);
        finish_prange<2>(a.ctl, (double)v, a.step, ch);
    }
}

}  // namespace lsp
