// shapes.cu -- implicit surfaces on the device (Sec. III-C: signed distance
// primitives; Sec. III-D: calculus on implicit functions), for building
// targets and initial fields without a host round trip.
//
// Coordinates lo + i * dx per axis as the stage kernels use them, in the field's precision (FP64 arithmetic for FP32
// fields would run on GB300's slow FP64 pipe; the shape and grid constants
// are converted once, on the host).  Primitives measure distance in the non-ignored
// dimensions only (ignoring dimensions turns a sphere into a cylinder, a box
// into a slab); periodic axes are not wrapped.
#include <cmath>

#include "../../include/lsp.h"
#include "launch.h"
#include "stencil.cuh"

namespace lsp {

// The kernel's copy of the shape and the grid, in the field precision, with
// the multipliers that divide a node index by each axis length.
template <typename R>
struct ShapeDev {
    R lo[LSP_MAXD], h[LSP_MAXD], c[LSP_MAXD], d[LSP_MAXD], r;
    unsigned n[LSP_MAXD], m[LSP_MAXD];
    int l[LSP_MAXD];
    unsigned ignore, npts;
};

// floor(x / n) for 0 <= x < 2^31 by a multiply-high and a shift (Granlund and
// Montgomery, "Division by invariant integers using multiplication", 1994:
// l = ceil(log2 n), m = floor(2^32 (2^l - n) / n) + 1, q = (mulhi(m, x) + x) >> l;
// mulhi(m, x) < x, so the sum stays below 2^32)
__device__ __forceinline__ unsigned div_invariant(unsigned x, unsigned m, int l)
{
    return (__umulhi(x, m) + x) >> l;
}

static void division_multiplier(unsigned n, unsigned* m, int* l)
{
    int s = 0;
    while ((1ull << s) < n) ++s;
    *l = s;
    *m = (unsigned)(((((unsigned long long)1 << s) - n) << 32) / n + 1);
}

// A primitive's distance is collected axis by axis, the fastest axis last, so
// that nodes of one row share what the other axes contribute: the sum (q) of
// sphere, quadric and half space, the outside sum (q) and the inside maximum
// (in) of the box.
template <typename R>
struct ShapePart {
    R q, in;
};

template <int KIND, typename R>
__device__ __forceinline__ void shape_axis(const ShapeDev<R>& s, int k, R x, ShapePart<R>& p)
{
    if ((s.ignore >> k) & 1u) return;
    if constexpr (KIND == SHAPE_SPHERE) {
        p.q += (x - s.c[k]) * (x - s.c[k]);
    } else if constexpr (KIND == SHAPE_BOX) {
        const R e = rmax(s.c[k] - x, x - s.d[k]);  // > 0 outside this slab
        if (e > R(0)) p.q += e * e;
        p.in = rmax(p.in, e);
    } else if constexpr (KIND == SHAPE_QUADRIC) {
        p.q += s.d[k] * (x - s.c[k]) * (x - s.c[k]);
    } else {
        p.q += s.d[k] * (x - s.c[k]);
    }
}

template <int KIND, typename R>
__device__ __forceinline__ R shape_finish(const ShapeDev<R>& s, const ShapePart<R>& p)
{
    if constexpr (KIND == SHAPE_SPHERE) return real_sqrt(p.q) - s.r;  // |x - c| - r
    // exact distance to [c, d]
    else if constexpr (KIND == SHAPE_BOX) return p.q > R(0) ? real_sqrt(p.q) : p.in;
    else if constexpr (KIND == SHAPE_QUADRIC) return p.q - s.r;  // sum_k w_k (x_k - c_k)^2 - offset
    else return p.q / s.r;  // half space {n . (x - p) <= 0}: n . (x - p) / |n|, r = |n|
}

// 16 bytes of consecutive values
template <typename R, int V>
struct alignas(V * sizeof(R)) Vec {
    R v[V];
};

// V consecutive nodes per thread and round (V values fill 16 bytes; 1 for a
// field that is not 16-byte aligned, or small: shape_vector_nodes): one index split
// by the axis lengths (the fastest axis last), one store and, within a row,
// one pass over the other axes per V nodes.  Coordinates lo + index * dx as
// the stage kernels compute them.  Dimensions and the primitive are template
// parameters, so everything stays in registers; the host checks npts < 2^31
// (32-bit index arithmetic).  Bound by the writes and the launches in FP32 and
// by the FP64 pipe in FP64.  A launch has at most 16 blocks per SM, in a
// grid-stride loop: a block for every 256 threads' nodes is bound by the rate
// at which blocks start.  us per call, back to back: one node per thread and
// round with the primitive chosen in the kernel; V nodes in one pass of blocks;
// this.  201^3 FP32 sphere 16.7, 16.5, 12.3; quadric 14.5, 18.6, 10.3; half
// space 18.7, 22.8, 12.2; unaligned sphere 16.6, 22.8, 14.7; 400 x 401 x 402
// half space 123, 148, 60; 201^3 FP64 half space (the norm from the host) 460,
// 436, 256.  Cylinder, box and their union at 201^3 FP32: 49.6, 41.1, 35.6.
template <int NDIM, int KIND, typename R, int V>
__global__ void __launch_bounds__(256) shape_kernel(ShapeDev<R> s, R* out)
{
    for (unsigned i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V; i0 < s.npts;
         i0 += gridDim.x * blockDim.x * V) {
        Vec<R, V> w;
        ShapePart<R> row;
        unsigned c = 0, end = 0;  // fastest index of the next node, end of its row
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (v == 0 || c == end) {  // first node, or first of the next row
                row.q = R(0);
                row.in = R(-INFINITY);
                unsigned r = i0 + v;
                unsigned idx[NDIM];
#pragma unroll
                for (int k = NDIM - 1; k > 0; --k) {
                    const unsigned q = div_invariant(r, s.m[k], s.l[k]);
                    idx[k] = r - q * s.n[k];
                    r = q;
                }
                idx[0] = r;
#pragma unroll
                for (int k = 0; k < NDIM - 1; ++k)
                    shape_axis<KIND>(s, k, rfma(R(idx[k]), s.h[k], s.lo[k]), row);
                c = idx[NDIM - 1];
                end = s.n[NDIM - 1];
            }
            ShapePart<R> p = row;
            shape_axis<KIND>(s, NDIM - 1, rfma(R(c), s.h[NDIM - 1], s.lo[NDIM - 1]), p);
            w.v[v] = shape_finish<KIND>(s, p);
            ++c;
        }
        if (i0 + V <= s.npts) {
            *reinterpret_cast<Vec<R, V>*>(out + i0) = w;
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (i0 + v < s.npts) out[i0 + v] = w.v[v];
        }
    }
}

// union min(a, b), intersection max(a, b), complement -a, difference
// max(a, -b) (Sec. III-D), V consecutive values per thread and round, blocks
// as for shape_kernel (union of two 201^3 FP32 fields, forms as above: 18.6,
// 12.5, 10.6 us; unaligned 14.5, 28.9, 14.5)
template <int OP, typename R>
__device__ __forceinline__ R shape_op_value(R u, R b)
{
    if constexpr (OP == LSP_SHAPE_UNION) return fmin(u, b);
    else if constexpr (OP == LSP_SHAPE_INTERSECT) return fmax(u, b);
    else if constexpr (OP == LSP_SHAPE_COMPLEMENT) return -u;
    else return fmax(u, -b);
}

template <int OP, typename R, int V>
__global__ void __launch_bounds__(256) shape_op_kernel(const R* a, const R* b, R* out, unsigned n)
{
    for (unsigned i = (blockIdx.x * blockDim.x + threadIdx.x) * V; i < n; i += gridDim.x * blockDim.x * V) {
        if (i + V <= n) {
            const Vec<R, V> u = *reinterpret_cast<const Vec<R, V>*>(a + i);
            Vec<R, V> w = u;
            if constexpr (OP != LSP_SHAPE_COMPLEMENT) w = *reinterpret_cast<const Vec<R, V>*>(b + i);
#pragma unroll
            for (int v = 0; v < V; ++v) w.v[v] = shape_op_value<OP>(u.v[v], w.v[v]);
            *reinterpret_cast<Vec<R, V>*>(out + i) = w;
        } else {
            for (unsigned j = i; j < n; ++j) {
                if constexpr (OP == LSP_SHAPE_COMPLEMENT) out[j] = shape_op_value<OP>(a[j], R(0));
                else out[j] = shape_op_value<OP>(a[j], b[j]);
            }
        }
    }
}

static unsigned shape_blocks(long long n, int v)
{
    const long long t = (n + v - 1) / v, b = (t + 255) / 256, cap = 16LL * sm_count();
    return (unsigned)(b < cap ? b : cap);
}
// Fewest nodes for V consecutive ones per thread: two blocks per SM.  Below,
// the chain of V nodes in one thread is longer than what it saves.
static unsigned shape_vector_nodes(int v) { return 512u * v * sm_count(); }
static bool vec_aligned(const void* p) { return ((uintptr_t)p & 15u) == 0; }

template <int KIND, typename R, int V>
static cudaError_t shape_launch(int ndim, const ShapeDev<R>& d, R* out, cudaStream_t st)
{
    const unsigned nb = shape_blocks(d.npts, V);
    switch (ndim) {
    case 1: shape_kernel<1, KIND, R, V><<<nb, 256, 0, st>>>(d, out); break;
    case 2: shape_kernel<2, KIND, R, V><<<nb, 256, 0, st>>>(d, out); break;
    case 3: shape_kernel<3, KIND, R, V><<<nb, 256, 0, st>>>(d, out); break;
    case 4: shape_kernel<4, KIND, R, V><<<nb, 256, 0, st>>>(d, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename R, int V>
static cudaError_t shape_kind(int kind, int ndim, const ShapeDev<R>& d, R* out, cudaStream_t st)
{
    switch (kind) {
    case SHAPE_SPHERE: return shape_launch<SHAPE_SPHERE, R, V>(ndim, d, out, st);
    case SHAPE_BOX: return shape_launch<SHAPE_BOX, R, V>(ndim, d, out, st);
    case SHAPE_QUADRIC: return shape_launch<SHAPE_QUADRIC, R, V>(ndim, d, out, st);
    default: return shape_launch<SHAPE_HALFSPACE, R, V>(ndim, d, out, st);
    }
}

template <typename R>
static cudaError_t launch_shape_t(const ShapeGeom& g, const ShapeArgs& s, R* out, cudaStream_t st)
{
    ShapeDev<R> d;
    R nn = R(0);  // |n|^2 of a half space
    for (int k = 0; k < LSP_MAXD; ++k) {
        const bool used = k < g.ndim;
        d.lo[k] = used ? R(g.lo[k]) : R(0);
        d.h[k] = used ? R(g.h[k]) : R(0);
        d.c[k] = used ? R(s.c[k]) : R(0);
        d.d[k] = used ? R(s.d[k]) : R(0);
        d.n[k] = used ? (unsigned)g.n[k] : 1u;
        division_multiplier(d.n[k], &d.m[k], &d.l[k]);
        if (used && !((s.ignore >> k) & 1u)) nn = std::fma(d.d[k], d.d[k], nn);
    }
    d.r = s.kind == SHAPE_HALFSPACE ? std::sqrt(nn) : R(s.r);
    d.ignore = s.ignore;
    d.npts = (unsigned)g.npts;
    constexpr int V = 16 / sizeof(R);
    return vec_aligned(out) && d.npts >= shape_vector_nodes(V) ? shape_kind<R, V>(s.kind, g.ndim, d, out, st)
                                                              : shape_kind<R, 1>(s.kind, g.ndim, d, out, st);
}

cudaError_t launch_shape(const ShapeGeom& g, const ShapeArgs& s, int dtype, void* out,
                         cudaStream_t st)
{
    if (dtype == LSP_F64) return launch_shape_t<double>(g, s, (double*)out, st);
    return launch_shape_t<float>(g, s, (float*)out, st);
}

template <int OP, typename R>
static cudaError_t op_launch(const R* a, const R* b, R* out, long long n, cudaStream_t st)
{
    constexpr int V = 16 / sizeof(R);
    if (n >= shape_vector_nodes(V) && vec_aligned(a) && (OP == LSP_SHAPE_COMPLEMENT || vec_aligned(b)) &&
        vec_aligned(out))
        shape_op_kernel<OP, R, V><<<shape_blocks(n, V), 256, 0, st>>>(a, b, out, (unsigned)n);
    else
        shape_op_kernel<OP, R, 1><<<shape_blocks(n, 1), 256, 0, st>>>(a, b, out, (unsigned)n);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_op_t(int op, const R* a, const R* b, R* out, long long n, cudaStream_t st)
{
    switch (op) {
    case LSP_SHAPE_UNION: return op_launch<LSP_SHAPE_UNION>(a, b, out, n, st);
    case LSP_SHAPE_INTERSECT: return op_launch<LSP_SHAPE_INTERSECT>(a, b, out, n, st);
    case LSP_SHAPE_COMPLEMENT: return op_launch<LSP_SHAPE_COMPLEMENT>(a, b, out, n, st);
    default: return op_launch<LSP_SHAPE_DIFFERENCE>(a, b, out, n, st);
    }
}

cudaError_t launch_shape_op(int op, int dtype, const void* a, const void* b, void* out, long long n,
                            cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    if (dtype == LSP_F64)
        return launch_op_t(op, (const double*)a, (const double*)b, (double*)out, n, st);
    return launch_op_t(op, (const float*)a, (const float*)b, (float*)out, n, st);
}

}  // namespace lsp
