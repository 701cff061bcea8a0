// stage_march.cuh -- the fused Runge-Kutta stage (Sec. V-A) for the ENO2 and
// ENO3 schemes (Sec. IV-B) on 3-D and 4-D FP32 grids, marching small blocks
// of nodes in registers.
//
// Same computation as tiled_stage_body<.., ENO2/ENO3, ..> (stage_tiled.cuh):
// ghost cells (Sec. III-B), one-sided ENO derivatives, the LF numerical
// Hamiltonian with global-LF dissipation (Sec. IV-D), the RK combination and
// the min with the target (Sec. VI-A); every ENO choice is made once per
// cell face where both of its nodes belong to the thread (stencil.cuh).  The
// operations on a node, their order and the order of the axes are the scalar
// body's, and so are the results, bit for bit.
//
// These schemes are bound by instruction issue on GB300, not by HBM, so the
// layout is chosen to spend few instructions beside the arithmetic:
//  - a thread owns RA = 2 consecutive nodes of the second-fastest axis A (in
//    4-D on R0 = 2 slabs of the slowest axis) at one node of the fastest
//    axis B and marches along S.  Lanes run along B: loads coalesce
//    and no address is computed per node.  The faces along S are carried in
//    registers, those along A and axis 0 are shared inside the block.
//  - own values reach the thread once, as the lead value of the march (one
//    load per node and plane, requested a plane ahead); the thread stores
//    its plane to shared memory for its neighbours along A and B, and only
//    the G-wide frame of the tile is loaded for it (kMarchSlots values per
//    thread and slab).  One barrier per plane.
//  - tiles are TB <= 64 nodes wide and any number of rows; the last tile of
//    an axis is moved back to end at the edge (its first nodes are computed
//    twice and stored once), so tiles are never partial, every load is in
//    the grid and ghost cells exist only in the frame.
// The shared-memory pitch is a constant, so every shared access has an
// immediate offset from one address per thread.
//
// Measured (GB300, us per stage of whole solves; default tile of the scalar
// body before, its autotuned tile or run kernel in brackets, this kernel's
// default tile now): rockets 300^3 ENO2 388 (182), 157; 100^3 20.8 (14.3),
// 8.9; car4d 81^4 ENO3 870 (650), 425; 33 x 41 x 37 x 29 48, 21.7.  What
// bounds it: instruction issue (65 % of the cycles on rockets 200^3, 165
// instructions per node in 3-D and 244 in 4-D, of which 45 and 125 are the
// scheme's arithmetic) and the latency of the loads between barriers.
// Measured and not kept: 4 rows per thread (128 registers, fewer warps: 10.1
// against 9.5 us at 100^3, 26.7 against 22.5 on the 4-D grid above); reading
// every neighbour through L1 without staging (250 us at 300^3, 1580 at 81^4);
// requesting the plane's loads after the march step instead of before it
// (550 us at 81^4).
#pragma once
#include "stage_tiled.cuh"

namespace lsp {

constexpr int kMarchPitch = 72;    // floats per staged row (TB + 2G <= 72)
constexpr int kMarchMaxTB = 64;
constexpr int kMarchSlots = 2;     // frame values per thread and slab
constexpr int kMarchThreads = 256;

// Rows per thread (along A) and, in 4-D, slabs per thread (along axis 0).
constexpr int kMarchRows = 2;
__host__ __device__ constexpr int march_slabs(int ndim) { return ndim == 4 ? 2 : 1; }

// Threads of a tile's CTA (whole warps).
inline int march_threads(const Tile& t) { return (t.tb * (t.ta / kMarchRows) + 31) / 32 * 32; }

// The march along S at one node column: before plane s, u[] = u_s ..
// u_{s+G-1}, S0 = S_s, S1 = S_{s+1}, T1 = T_{s+1/2}, M0 = M_s (ENO3) and
// pm = dx p-_s.
template <int SCHEME>
struct ColMarch {
    float u[ghost_width(SCHEME)], S0, S1, T1, M0, pm;
};

// From w[k] = u_{s-G+k}, k = 0..2G-1.
template <int SCHEME>
__device__ __forceinline__ void col_init(const float* w, ColMarch<SCHEME>& m)
{
    constexpr int G = ghost_width(SCHEME);
#pragma unroll
    for (int k = 0; k < G; ++k) m.u[k] = w[G + k];
    float unused;
    if constexpr (SCHEME == ENO2) {
        const float da = w[1] - w[0], db = w[2] - w[1], dc = w[3] - w[2];
        m.S0 = dc - db;
        eno2_face(db, db - da, m.S0, unused, m.pm);  // face s - 1/2
    } else {
        float d[5], S[4], T[3];
#pragma unroll
        for (int k = 0; k < 5; ++k) d[k] = w[k + 1] - w[k];
#pragma unroll
        for (int k = 0; k < 4; ++k) S[k] = d[k + 1] - d[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) T[k] = S[k + 1] - S[k];
        m.M0 = eno_smaller(T[1], T[2]);
        eno3_face(d[2], S[1], S[2], eno_smaller(T[0], T[1]), m.M0, unused, m.pm);
        m.S0 = S[2];
        m.S1 = S[3];
        m.T1 = T[2];
    }
}

// Plane s: take u_{s+G}, give dx p-_s and dx p+_s, advance to plane s+1.
template <int SCHEME>
__device__ __forceinline__ void col_step(ColMarch<SCHEME>& m, float lead, float& pm, float& pp)
{
    constexpr int G = ghost_width(SCHEME);
    pm = m.pm;
    const float dA = m.u[1] - m.u[0];  // d_{s+1/2}
    if constexpr (SCHEME == ENO2) {
        const float S1 = (lead - m.u[1]) - dA;  // S_{s+1}
        eno2_face(dA, m.S0, S1, pp, m.pm);      // face s + 1/2
        m.S0 = S1;
    } else {
        const float S2 = (lead - m.u[2]) - (m.u[2] - m.u[1]);  // S_{s+2}
        const float T2 = S2 - m.S1;                            // T_{s+3/2}
        const float M1 = eno_smaller(m.T1, T2);                // M_{s+1}
        eno3_face(dA, m.S0, m.S1, m.M0, M1, pp, m.pm);         // face s + 1/2
        m.S0 = m.S1;
        m.S1 = S2;
        m.T1 = T2;
        m.M0 = M1;
    }
#pragma unroll
    for (int k = 0; k + 1 < G; ++k) m.u[k] = m.u[k + 1];
    m.u[G - 1] = lead;
}

// gridDim = (tiles along B, tiles along A, chunks x blocks of axis 0);
// blockDim.x >= TB TA / RA threads, thread t at column t % TB of block
// t / TB.  Offsets inside a plane are 32-bit: fields below 2^30 nodes.
// DEP: launched by launch_dependent (stage_wait, ordinary loads); otherwise an
// ordinary launch reading the fields through the read-only path.
template <int NDIM, int SCHEME, int DYN, int MINB, bool DEP>
__global__ void __launch_bounds__(kMarchThreads, MINB)
    stage_march_kernel(StageArgs<float> a, int TB, int TA, int ch, int nchunks)
{
    constexpr int RA = kMarchRows, R0 = march_slabs(NDIM);
    constexpr int G = ghost_width(SCHEME), P = kMarchPitch, NS = kMarchSlots;
    constexpr int AS = NDIM - 3, AA = NDIM - 2, AB = NDIM - 1;
    extern __shared__ float march_smem[];  // [buffer][slab][TA + 2G][P]
    const int nB = a.n[AB], nA = a.n[AA], nS = a.n[AS];
    const int sA = a.stride[AA], sS = a.stride[AS];
    const int perA = a.periodic[AA], perB = a.periodic[AB], perS = a.periodic[AS];
    const int H = TA + 2 * G, slab_floats = H * P;

    // tile origin (moved back at the end of an axis) and first own node
    const int bown = blockIdx.x * TB, aown = blockIdx.y * TA;
    const int b0 = min(bown, nB - TB), a0 = min(aown, nA - TA);
    const int chunk = blockIdx.z % nchunks;
    const int oown = (blockIdx.z / nchunks) * R0;
    const int o0 = NDIM == 4 ? min(oown, a.n[0] - R0) : 0;
    const int s_begin = chunk * ch, s_end = min(s_begin + ch, nS);

    const int nthr = TB * (TA / RA);
    const bool live = (int)threadIdx.x < nthr;
    const int t = live ? threadIdx.x : nthr - 1;  // spare threads repeat the last one's
    const int col = t % TB, run = t / TB;         // reads and store nothing
    const int b = b0 + col, ar = a0 + run * RA;

    // Byte offsets inside a field (32-bit, see march_tile_ok) added to a
    // uniform base: no 64-bit address arithmetic per load.
    const unsigned rowb = 4u * (unsigned)sA;
    unsigned slab[R0 + 2 * G];  // the axis-0 window's slabs (block-uniform)
    bool edge0 = false;
#pragma unroll
    for (int k = 0; k < R0 + 2 * G; ++k) slab[k] = 0u;
    if constexpr (NDIM == 4) {
        edge0 = !a.periodic[0] && (o0 < G || o0 + R0 + G > a.n[0]);
#pragma unroll
        for (int k = 0; k < R0 + 2 * G; ++k)
            slab[k] = 4u * (unsigned)(into_axis(o0 - G + k, a.n[0], a.periodic[0]) * a.stride[0]);
    }
    const unsigned own = 4u * (unsigned)(ar * sA + b);
    auto at = [](const float* base, unsigned bytes) {
        return reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + bytes);
    };
    auto ld = [](const float* p) -> float {
        if constexpr (DEP) return *p;
        else return __ldg(p);
    };

    // This thread's share of the tile's frame: rows above and below (TB
    // values each), then columns left and right (TA values each); corners
    // are never read (position 0 takes the values of slots past the frame).
    // A ghost value of an extrapolated axis is formed from the two nodes at
    // the edge when it is staged: u1 + q (u1 - u2).
    unsigned f1[NS], f2[NS];
    float fq[NS];
    int fs[NS];  // position in the staged slab
    const bool ghosts = (!perA && (a0 < G || a0 + TA + G > nA)) || (!perB && (b0 < G || b0 + TB + G > nB));
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const int e = threadIdx.x + i * blockDim.x;
        int p1 = ar * sA + b, p2 = p1;
        fq[i] = 0.0f;
        fs[i] = 0;
        if (e < 2 * G * TB) {
            const int r = e / TB, c = e - r * TB;
            const int j = r < G ? a0 - G + r : a0 + TA + r - G;
            fs[i] = (r < G ? r : TA + r) * P + G + c;
            p1 = p2 = into_axis(j, nA, perA) * sA + b0 + c;
            if (!perA && (j < 0 || j >= nA)) {
                p2 = (j < 0 ? 1 : nA - 2) * sA + b0 + c;
                fq[i] = float(j < 0 ? -j : j - nA + 1);
            }
        } else if (e < 2 * G * (TB + TA)) {
            const int w = e - 2 * G * TB, r = w / (2 * G), c = w - r * 2 * G;
            const int j = c < G ? b0 - G + c : b0 + TB + c - G;
            fs[i] = (G + r) * P + (c < G ? c : TB + c);
            p1 = p2 = (a0 + r) * sA + into_axis(j, nB, perB);
            if (!perB && (j < 0 || j >= nB)) {
                p2 = (a0 + r) * sA + (j < 0 ? 1 : nB - 2);
                fq[i] = float(j < 0 ? -j : j - nB + 1);
            }
        }
        f1[i] = 4u * (unsigned)p1;
        f2[i] = 4u * (unsigned)p2;
    }

    // heading (axis 2): axis B in 3-D, axis A in 4-D
    constexpr bool kTrig = DYN == AIR3D || DYN == CAR4D || DYN == ROCKETS;
    constexpr int NT = NDIM == 4 ? RA : 1;
    const float xb = fmaf(float(b), a.h[AB], a.lo[AB]);
    float sth[NT], cth[NT];
#pragma unroll
    for (int r = 0; r < NT; ++r) {
        sth[r] = 0.0f;
        cth[r] = 1.0f;
        if constexpr (kTrig)
            sincosf(NDIM == 4 ? fmaf(float(ar + r), a.h[AA], a.lo[AA]) : xb, &sth[r], &cth[r]);
    }
    // nodes this thread stores (slabs before oown are block-uniform)
    bool st[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) st[r] = live && b >= bown && ar + r >= aown;
    const bool has_n = a.phi_n != nullptr, tube = a.tube != 0;

    if constexpr (DEP) {
        stage_wait();
        stage_release();
    }
    if (past_last_step(a)) return;
    const float dt = a.dt_from_ctl ? float(a.ctl->dt) : a.dt;
    const float cl = a.c_l * dt;
    float ha[NDIM];  // alpha_k / 2
#pragma unroll
    for (int k = 0; k < NDIM; ++k)
        ha[k] = (a.alpha_from_ctl ? float(__longlong_as_double((long long)a.ctl->alpha_bits[k]))
                                  : a.alpha[k]) *
                0.5f;
    // axis k's central costate and p+ - p- of a node from dx p-, dx p+,
    // rounded as the scalar body's (p+ + p-) / 2 and p+ - p- are compiled: the
    // product of p- fused into the sum and the difference
    auto axis = [&](int k, float am, float ap, float& pbar) -> float {
        const float pp = __fmul_rn(ap, a.inv_dx[k]);
        pbar = 0.5f * __fmaf_rn(am, a.inv_dx[k], pp);
        return __fmaf_rn(-am, a.inv_dx[k], pp);
    };

    // plane of the lead value j (beyond the end of an extrapolated axis the
    // march continues its last difference instead)
    auto plane_of = [&](int j) { return a.phi_s + (size_t)(j < nS ? j : (perS ? j - nS : nS - 1)) * sS; };
    ColMarch<SCHEME> m[R0][RA];
    float lead[R0][RA], fv[R0][NS], gv[R0][NS];
    // the frame of one plane: requested into fv (gv: the second edge node)
    auto frame = [&](const float* plane) {
#pragma unroll
        for (int q = 0; q < R0; ++q)
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                fv[q][i] = ld(at(plane, slab[G + q] + f1[i]));
                gv[q][i] = ghosts ? ld(at(plane, slab[G + q] + f2[i])) : 0.0f;
            }
    };
    // this thread's nodes and frame values into a buffer of the staged tile
    const int mine = (G + run * RA) * P + G + col;
    auto stage = [&](float* buf) {
#pragma unroll
        for (int q = 0; q < R0; ++q) {
#pragma unroll
            for (int r = 0; r < RA; ++r) buf[q * slab_floats + mine + r * P] = m[q][r].u[0];
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                float v = fv[q][i];
                if (ghosts) v = fq[i] != 0.0f ? fmaf(fq[i], v - gv[q][i], v) : v;
                buf[q * slab_floats + fs[i]] = v;
            }
        }
    };
    frame(a.phi_s + (size_t)s_begin * sS);
#pragma unroll
    for (int q = 0; q < R0; ++q)
#pragma unroll
        for (int r = 0; r < RA; ++r) {
            const unsigned off = slab[G + q] + own + r * rowb;
            float w[2 * G];
#pragma unroll
            for (int k = 0; k < 2 * G; ++k)
                w[k] = line_value<float, DEP>(at(a.phi_s, off), s_begin - G + k, nS, sS, perS);
            col_init<SCHEME>(w, m[q][r]);
            lead[q][r] = ld(at(plane_of(s_begin + G), off));
        }
    stage(march_smem);

    float chk = 0.0f;  // stays 0 while every stored value is finite
    // plane s from buffer cur; plane s+1 is staged into nxt
    auto plane_step = [&](int s, const float* cur, float* nxt) {
        __syncthreads();  // plane s staged; nxt is free
        const size_t splane = (size_t)s * sS;
        const float* plane = a.phi_s + splane;
        const float* nplane = a.phi_n + splane;
        const float* tplane = a.target + splane;
        const bool more = s + 1 < s_end;
        // every load of the iteration first (the out field may be phi^n)
        const float* lplane = plane_of(s + 1 + G);
        float nlead[R0][RA], pn[R0][RA], tg[R0][RA];
#pragma unroll
        for (int q = 0; q < R0; ++q)
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                const unsigned off = slab[G + q] + own + r * rowb;
                nlead[q][r] = ld(at(lplane, off));
                pn[q][r] = tg[q][r] = 0.0f;
                if (st[r] && (NDIM < 4 || o0 + q >= oown)) {
                    if (has_n) pn[q][r] = *at(nplane, off);
                    if (tube) tg[q][r] = ld(at(tplane, off));
                }
            }
        float wo[NDIM == 4 ? 2 * G : 1][RA];
        if constexpr (NDIM == 4) {
#pragma unroll
            for (int k = 0; k < 2 * G; ++k)
#pragma unroll
                for (int r = 0; r < RA; ++r)
                    wo[k][r] = ld(at(plane, slab[k < G ? k : k + R0] + own + r * rowb));
        }
        if (more) frame(plane + sS);
        if (!perS && s + G >= nS) {  // beyond the end of an extrapolated axis
            const float* last = a.phi_s + (size_t)(nS - 1) * sS;
#pragma unroll
            for (int q = 0; q < R0; ++q)
#pragma unroll
                for (int r = 0; r < RA; ++r) {
                    const unsigned off = slab[G + q] + own + r * rowb;
                    const float un = ld(at(last, off));
                    lead[q][r] = fmaf(float(s + G - nS + 1), un - ld(at(last - sS, off)), un);
                }
        }

        float pbar[R0][RA][NDIM], diss[R0][RA], center[R0][RA];
        // axis S
#pragma unroll
        for (int q = 0; q < R0; ++q)
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                center[q][r] = m[q][r].u[0];
                float pm, pp;
                col_step<SCHEME>(m[q][r], lead[q][r], pm, pp);
                diss[q][r] = ha[AS] * axis(AS, pm, pp, pbar[q][r][AS]);
                lead[q][r] = nlead[q][r];
            }
        // Axis B is evaluated before A in 3-D, its dissipation added after A's
        // (fewer live values: rockets 300^3 1921 against 2033 us for 6 steps),
        // and after it in 4-D (car4d 81^4 2626 against 2684 us for 2 steps).
        float bdiss[R0][RA];
        auto axis_b = [&]() {
#pragma unroll
            for (int q = 0; q < R0; ++q)
#pragma unroll
                for (int r = 0; r < RA; ++r) {
                    const float* p = cur + q * slab_floats + mine + r * P;
                    float w[2 * G + 1], pm, pp;
#pragma unroll
                    for (int k = 0; k <= 2 * G; ++k) w[k] = k == G ? center[q][r] : p[k - G];
                    eno_line<SCHEME, 1>(w, &pm, &pp);
                    const float e = axis(AB, pm, pp, pbar[q][r][AB]);
                    if constexpr (NDIM == 3) bdiss[q][r] = e;
                    else diss[q][r] = rfma(ha[AB], e, diss[q][r]);
                }
        };
        if constexpr (NDIM == 3) axis_b();
        // axis A
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const float* p = cur + q * slab_floats + mine - G * P;
            float w[RA + 2 * G], pm[RA], pp[RA];
#pragma unroll
            for (int k = 0; k < RA + 2 * G; ++k)
                w[k] = k < G || k >= G + RA ? p[k * P] : center[q][(k - G) & (RA - 1)];
            eno_line<SCHEME, RA>(w, pm, pp);
#pragma unroll
            for (int r = 0; r < RA; ++r)
                diss[q][r] = rfma(ha[AA], axis(AA, pm[r], pp[r], pbar[q][r][AA]), diss[q][r]);
        }
        if constexpr (NDIM == 4) {
            axis_b();
        } else {
#pragma unroll
            for (int r = 0; r < RA; ++r) diss[0][r] = rfma(ha[AB], bdiss[0][r], diss[0][r]);
        }
        // axis 0
        if constexpr (NDIM == 4) {
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                float w[R0 + 2 * G], pm[R0], pp[R0];
#pragma unroll
                for (int k = 0; k < R0 + 2 * G; ++k)
                    w[k] = k < G ? wo[k < G ? k : 0][r]
                                 : (k >= G + R0 ? wo[k >= G + R0 ? k - R0 : 0][r]
                                                : center[(k - G) & (R0 - 1)][r]);
                if (edge0) fix_extrapolated<R0, G>(w, o0, a.n[0]);
                eno_line<SCHEME, R0>(w, pm, pp);
#pragma unroll
                for (int q = 0; q < R0; ++q)
                    diss[q][r] = rfma(ha[0], axis(0, pm[q], pp[q], pbar[q][r][0]), diss[q][r]);
            }
        }
        // Hamiltonian, rate, RK combination, tube
        const float xs = fmaf(float(s), a.h[AS], a.lo[AS]);
        float* oplane = a.out + splane;
#pragma unroll
        for (int q = 0; q < R0; ++q)
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                float x[NDIM];
                if constexpr (NDIM == 4) x[0] = fmaf(float(o0 + q), a.h[0], a.lo[0]);
                x[AS] = xs;
                x[AA] = fmaf(float(ar + r), a.h[AA], a.lo[AA]);
                x[AB] = xb;
                constexpr int kT = NDIM == 4;
                const float Hv = hamiltonian_sc<DYN, NDIM>(x, pbar[q][r], a.prm, sth[kT * r], cth[kT * r]);
                const float L = -(Hv - diss[q][r]);
                float v = fmaf(cl, L, a.c_s * center[q][r]);
                if (has_n) v = fmaf(a.c_n, pn[q][r], v);
                if (tube) v = fminf(v, tg[q][r]);
                if (st[r] && (NDIM < 4 || o0 + q >= oown)) {
                    chk = fmaf(v, 0.0f, chk);
                    *const_cast<float*>(at(oplane, slab[G + q] + own + r * rowb)) = v;
                }
            }
        if (more) stage(nxt);
    };
    float* const buf0 = march_smem;
    float* const buf1 = march_smem + R0 * slab_floats;
    for (int s = s_begin; s < s_end; s += 2) {
        plane_step(s, buf0, buf1);
        if (s + 1 < s_end) plane_step(s + 1, buf1, buf0);
    }
    if (!(chk == 0.0f)) atomicOr(&a.ctl->flags, kFlagNonFinite);
}

}  // namespace lsp
