// What the 2D kernels that take several steps in shared memory have in common:
// the collision with rho1 kept, box indices, and the samplers' points and boxes.
#pragma once
#include <cmath>

#include "wlb_handle.cuh"
#include "wlb_kernels.cuh"

namespace wlb {
namespace {

constexpr int kMaxGroup = 64;  // points of a sampler CTA (four lanes each)
// And the length of their arc in cells.  FP64 boxes of eight cells of arc take
// longer than a tile: 128^2, 64 points, us per sampled step with arcs of 8, 6, 4, 3
// cells 1.72, 1.58, 1.53, 1.49.  FP32: 8 or shorter alike (256^2, 200 points: 0.83
// with 8, 0.91 with 4, more boxes than SMs).
template <typename R>
constexpr float max_arc() { return sizeof(R) == 8 ? 3.0f : 8.0f; }

// The value a stored state holds for v (storage rounding).
template <typename S> __device__ __forceinline__ typename Store<S>::R as_stored(typename Store<S>::R v) { return v; }
template <> __device__ __forceinline__ float as_stored<__half>(float v) { return __half2float(__float2half_rn(v)); }

// Largest moment box of a sampler CTA, in cells: the arc's extent, one cell of
// stencil on either side and two of rounding.
template <typename R>
__host__ __device__ constexpr int sampler_box() { return (int)max_arc<R>() + 5; }

// i / w for 0 <= i < 2^16 and w >= 1 by the high half of a product with
// ceil(2^32 / w) (which does not fit 32 bits for w = 1: a box one cell wide).
__device__ __forceinline__ unsigned divide_magic(int w) { return w > 1 ? 0xffffffffu / (unsigned)w + 1u : 0u; }
__device__ __forceinline__ int divide(int i, int w, unsigned magic) {
    return w > 1 ? (int)__umulhi((unsigned)i, magic) : i;
}

// a + b and a - b.  In FP64 as fused multiply-adds with one = 1 (exact products,
// the same rounding): the FP64 pipe takes 2.0 of them per clock and SM but 1.68
// additions.  `one` must come from memory, or the compiler makes them additions.
template <typename R>
__device__ __forceinline__ R plus(R a, R b, R one) {
    if constexpr (sizeof(R) == 8) return fma_rn(a, one, b);
    else return add_rn(a, b);
}
template <typename R>
__device__ __forceinline__ R minus(R a, R b, R one) {
    if constexpr (sizeof(R) == 8) return fma_rn(b, -one, a);
    else return sub_rn(a, b);
}

// The collision of collide_half for D = 2, with rho1 returned.  2 eq and
// 2 (rho1 - 2 eq) are exact, so the two fused multiply-adds round exactly as
// the product and difference do; they save two of thirteen operations, which
// in FP64 are the kernel's bound.
template <typename R>
__device__ __forceinline__ R collide_2d(R c2, const R (&f)[5], R (&o)[5], R one = R(1)) {
    const R rho = plus(plus(plus(plus(f[0], f[1], one), f[2], one), f[3], one), f[4], one);
    const R eq = mul_rn(c2, rho);
    o[0] = fma_rn(R(2), fma_rn(R(-2), eq, rho), -f[0]);
    o[1] = minus(eq, f[2], one);
    o[2] = minus(eq, f[1], one);
    o[3] = minus(eq, f[4], one);
    o[4] = minus(eq, f[3], one);
    return rho;
}

// The circle of the surface points, on the host (in FP64: ten operations of every
// block's first warp took the batched sampler 0.8 % of an ensemble's run).
inline Circle circle_of(const Geometry &g) {
    const double x = std::floor(g.center[0]), y = std::floor(g.center[1]);
    return Circle{(int)x, (int)y, (float)(g.center[0] - x), (float)(g.center[1] - y), (float)g.surface_radius};
}

// Whether box coordinates and their differences fit 32 bits; sampled steps of
// other lattices go without boxes.
inline bool boxes_fit(const Geometry &g) {
    constexpr int kMost = 1 << 29;
    for (int a = 0; a < 2; ++a)
        if (g.n[a] > kMost || !(std::fabs(g.center[a]) <= kMost)) return false;
    return true;
}

// Extent of the cells that the stencils of points p0 .. p1 - 1 of the circle
// read, by one warp: b = first column, first row, last column, last row (not
// wrapped).
__device__ __forceinline__ void arc_box(int p0, int p1, int n_surface, const Circle &c, int lane, int *b) {
    float lox = 1e30f, hix = -1e30f, loy = 1e30f, hiy = -1e30f;
    for (int p = p0 + lane; p < p1; p += 32) {
        float sn, cs;
        sincospif((float)(2 * p + 1) / (float)n_surface, &sn, &cs);
        const float X = c.fx + c.radius * cs, Y = c.fy + c.radius * sn;
        lox = fminf(lox, X);
        hix = fmaxf(hix, X);
        loy = fminf(loy, Y);
        hiy = fmaxf(hiy, Y);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        lox = fminf(lox, __shfl_xor_sync(kFull, lox, o));
        hix = fmaxf(hix, __shfl_xor_sync(kFull, hix, o));
        loy = fminf(loy, __shfl_xor_sync(kFull, loy, o));
        hiy = fmaxf(hiy, __shfl_xor_sync(kFull, hiy, o));
    }
    // centre cells floor(X + 1/2), one cell of stencil; 0.25 covers the FP32 error:
    // 2^-24 radius (2 pi for the angle, 3 for the sine, its product and the sum),
    // and twice 2 pi more beyond 2^23 points, is below 0.1 for radii up to 2^16
    // (the lattice of a larger circle takes over 400 GB)
    if (lane == 0) {
        b[0] = c.x + (int)floorf(lox + 0.25f) - 1;
        b[1] = c.y + (int)floorf(loy + 0.25f) - 1;
        b[2] = c.x + (int)floorf(hix + 0.75f) + 1;
        b[3] = c.y + (int)floorf(hiy + 0.75f) + 1;
    }
}

// A surface point on four neighbouring lanes, comp = lane & 3: rho, Jx, Jy (the
// fourth repeats rho).  add() takes the moments of one step from shared memory
// (rho, Jx, Jy, `area` cells each).
// comp 0: acc0 += p^2; comp 1: acc1 += u.u; comps 2, 3: acc2, acc3 += u_a (u.n),
// the nine terms in the order of sample_point_2d_thread; acc4 stays zero (the
// terms of the third component are exact zeros).
template <typename R>
struct PointQuad {
    R w[9], n0, n1, acc;
    int pc, comp;
    // p: the point; (x0, y0), tw x th: its moment box, inside rows of w0 cells
    // with a halo of H cells on either side
    __device__ __forceinline__ void load(int p, int component, const int4 *st_xyz, const R *st_w, const R *nrm,
                                         const R *sums, int x0, int y0, int tw, int th, int nx, int ny, int H,
                                         int w0) {
        comp = component;
        const int4 ctr = st_xyz[(long long)p * 9 + 4];
        int lx = (ctr.x - x0) % nx, ly = (ctr.y - y0) % ny;  // the box is no larger than the lattice
        lx += lx < 0 ? nx : 0;
        ly += ly < 0 ? ny : 0;
        pc = (min(max(ly, 1), th - 2) + H) * w0 + min(max(lx, 1), tw - 2) + H;  // in range by construction
#pragma unroll
        for (int l = 0; l < 9; ++l) w[l] = st_w[2 * ((long long)p * 9 + l) + (comp == 1 || comp == 2 ? 1 : 0)];
        n0 = nrm[4 * (long long)p];
        n1 = nrm[4 * (long long)p + 1];
        acc = sums[5 * (long long)p + comp];
    }
    __device__ __forceinline__ void add(const R *mom, int area, int w0, R one = R(1)) {
        const R *m = mom + (size_t)(comp < 3 ? comp : 0) * area + pc;
        R v[9];
#pragma unroll
        for (int l = 0; l < 9; ++l) v[l] = mul_rn(w[l], m[(l / 3 - 1) * w0 + l % 3 - 1]);
        R sum = plus(plus(v[0], v[8], one), v[4], one);
        sum = plus(sum, plus(v[2], v[6], one), one);
        sum = plus(sum, plus(plus(v[1], v[5], one), plus(v[3], v[7], one), one), one);
        const int base = (threadIdx.x & 31) & ~3;
        const R pr = __shfl_sync(kFull, sum, base), u0 = __shfl_sync(kFull, sum, base + 1),
                u1 = __shfl_sync(kFull, sum, base + 2);
        const R a = mul_rn(u0, comp == 1 ? u0 : n0);
        const R b = fma_rn(u1, comp == 1 ? u1 : n1, a);
        const R x = comp == 0 ? pr : (comp == 1 ? R(1) : (comp == 2 ? u0 : u1));
        acc = fma_rn(x, comp == 0 ? pr : b, acc);
    }
};

// Points per sampler CTA: an arc of at most max_arc cells, and no more points
// than take about as long as a tile (FP64: the pipe needs 60 cycles per point
// and step).
template <typename S>
inline int sampler_group(const Geometry &g) {
    const double spacing = 6.283185307179586 * g.surface_radius / g.n_surface;
    const int most = sizeof(typename Store<S>::R) == 8 ? 16 : kMaxGroup;
    const int n = (int)std::fmin((double)most, (double)max_arc<typename Store<S>::R>() / spacing + 1.0);
    return n < 1 ? 1 : n;
}

}  // namespace
}  // namespace wlb
