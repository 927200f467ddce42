// Two steps per launch for 3D lattices that the slab kernel (wlb_two_step.cu)
// does not take: the driven cavity, and rows of whole 16-byte vectors that are
// no multiple of 16 cells.
//
// One step per launch reads and writes every population from L2 or HBM for
// every step.  Here a CTA takes a tile of tx x ty x tz cells through two steps.
// Step 1 runs on the tile and on the cells that share a face with it and leaves
// in shared memory the populations that arrive at the tile's cells: a vector of
// W cells along x per thread and plane, its results stored whole at the cell
// they move to (+-x: at the cell they leave, shifted when step 2 reads them),
// side faces along y as vectors, along x one cell per row.  Step 2 reads its own
// cells' arrivals and writes the tile.  No plane of step 1 waits for another, so
// all of a CTA's warps have loads in flight; no CTA waits for another; the face
// cells are computed by both tiles.  The arithmetic per cell and step is that of
// the one-step kernels and the t+1 values are rounded to the storage type: the
// same bits.  A tile that spans an axis wraps around it instead of having faces.
//
// (One cell per thread, with or without a thread per column, issued 100 to 250
// instructions per cell and had too few bytes in flight: 64 x 64 x 203 driven FP32
// 9 and 6.2 us per step that way, 4.8 with vectors.)
//
// Sampled launches run `sample_boxes` beside the update: the points' centre cells
// are grouped into boxes of kBox^3 cells, and a CTA computes rho1 and J1 of a
// box's stencil cells once, at t and at t+1 (step 1 pushed into the box as
// above), in shared memory, from where a warp per point adds the sums.  (A warp
// per point reading global memory computes every cell's moments once per
// stencil that holds it, about 27 N / 4 pi R^2 times.)
#include <cmath>

#include "wlb_handle.cuh"
#include "wlb_kernels.cuh"

namespace wlb {
namespace {

constexpr int kMaxThreads = 512;
constexpr size_t kMaxSmem = 164 * 1024;     // of a tile
constexpr int kBox = 6;                     // edge of a box of centre cells
constexpr int kMom = kBox + 2;              // and of its stencils' cells
constexpr int kMomCells = kMom * kMom * kMom;
constexpr int kBoxAxis = 16;                // boxes per axis at most
constexpr int kSampleThreads = 1024;        // a stencil cell each, a warp per point

// The value a stored state holds for v (storage rounding).
template <typename S> __device__ __forceinline__ typename Store<S>::R as_stored(typename Store<S>::R v) { return v; }
template <> __device__ __forceinline__ float as_stored<__half>(float v) { return __half2float(__float2half_rn(v)); }

__device__ __forceinline__ int down(int v, int n) { return v == 0 ? n - 1 : v - 1; }
__device__ __forceinline__ int up(int v, int n) { return v == n - 1 ? 0 : v + 1; }

// The seven populations that arrive at (x, y, z) from the stored state A.
template <typename S>
__device__ __forceinline__ void pull(const S *__restrict__ A, long long nc, int nx, int ny, int nz, int x, int y, int z,
                                     typename Store<S>::R (&f)[7]) {
    const long long row = ((long long)z * ny + y) * nx;
    f[0] = Store<S>::get(A + row + x);
    f[1] = Store<S>::get(A + nc + row + down(x, nx));
    f[2] = Store<S>::get(A + 2 * nc + row + up(x, nx));
    f[3] = Store<S>::get(A + 3 * nc + ((long long)z * ny + down(y, ny)) * nx + x);
    f[4] = Store<S>::get(A + 4 * nc + ((long long)z * ny + up(y, ny)) * nx + x);
    f[5] = Store<S>::get(A + 5 * nc + ((long long)down(z, nz) * ny + y) * nx + x);
    f[6] = Store<S>::get(A + 6 * nc + ((long long)up(z, nz) * ny + y) * nx + x);
}

template <typename S>
struct Tile3D {
    using R = typename Store<S>::R;
    const S *A;  // state t
    S *B;        // state t + 2
    const uint8_t *cls;
    const R *c2f;
    int nx, ny, nz;
    long long ncell;
    int tx, ty, tz, tiles_x, tiles_y;
    int plane_threads, face_begin;  // threads per plane: vectors, then (from face_begin) cells of the x faces
    R c0sq, cpsq;
    Drive<R> drv[2];  // driven cavity, both steps
};

template <typename S>
inline size_t tile_smem(int tx, int ty, int tz) {  // seven arriving populations, padded rows for +-x
    return ((size_t)5 * tx + 2 * (tx + 2 * Store<S>::W)) * ty * tz * sizeof(typename Store<S>::R);
}

template <typename S, bool DRIVEN>
__global__ void __launch_bounds__(kMaxThreads, 1) tile_two_steps_3d(Tile3D<S> P) {
    using R = typename Store<S>::R;
    constexpr int W = Store<S>::W;
    extern __shared__ __align__(16) unsigned char tile_raw[];
    asm volatile("griddepcontrol.launch_dependents;");
    const int nx = P.nx, ny = P.ny, nz = P.nz, tid = threadIdx.x;
    const int bx = (int)(blockIdx.x % P.tiles_x), by = (int)(blockIdx.x / P.tiles_x) % P.tiles_y,
              bz = (int)(blockIdx.x / P.tiles_x) / P.tiles_y;
    const int x0 = bx * P.tx, y0 = by * P.ty, z0 = bz * P.tz;
    const int tw = min(P.tx, nx - x0), th = min(P.ty, ny - y0), td = min(P.tz, nz - z0);
    const bool wx = tw == nx, wy = th == ny, wz = td == nz;  // the tile spans the axis
    const int sheet = tw * th, cells = sheet * td;
    const int pad = tw + 2 * W, psheet = pad * th;           // +-x arrays: W cells beside every row
    R *a0 = reinterpret_cast<R *>(tile_raw), *a3 = a0 + cells, *a4 = a3 + cells, *a5 = a4 + cells, *a6 = a5 + cells;
    R *a1 = a6 + cells, *a2 = a1 + psheet * td;              // cell lx of a row at W + lx
    // this thread's vector (or face cell) of a plane: planes group, group + groups, ..
    const int nv = tw / W, vecs = nv * (th + (wy ? 0 : 2)), per = P.plane_threads;
    const int group = tid / per, groups = blockDim.x / per, t = tid - group * per;
    const bool vec = t < vecs, face = !vec && !wx && t >= P.face_begin && t - P.face_begin < 2 * th;
    int lx, ly;
    if (vec) {
        ly = t / nv;
        lx = (t - ly * nv) * W;
        ly -= wy ? 0 : 1;  // -1 and th: the side faces
    } else {
        const int q = t - P.face_begin, hi = q >= th;
        ly = q - (hi ? th : 0);
        lx = hi ? tw : -1;
    }
    const bool inner = vec && ly >= 0 && ly < th;
    int x = x0 + lx, y = y0 + ly;
    x = x < 0 ? nx - 1 : (x >= nx ? 0 : x);
    y = y < 0 ? ny - 1 : (y >= ny ? 0 : y);
    // 32-bit element indices (7 ncell < 2^32, see the planner): a plane's part is
    // uniform, a thread adds its own
    const unsigned c = (unsigned)(y * nx + x), cym = (unsigned)(down(y, ny) * nx + x), cyp = (unsigned)(up(y, ny) * nx + x);
    const unsigned cxm = (unsigned)(y * nx + down(x, nx)),
                   cxp = (unsigned)(y * nx + (x + (vec ? W : 1) >= nx ? 0 : x + (vec ? W : 1)));
    const unsigned plane = (unsigned)nx * (unsigned)ny, nc = (unsigned)P.ncell;
    asm volatile("griddepcontrol.wait;" ::: "memory");

    auto sound = [&](unsigned kc, unsigned id) {  // the c^2 the one-step kernels use for the class
        return kc == CELL_FLUID ? P.c0sq : (kc == CELL_OBJECT ? P.cpsq : P.c2f[id]);
    };
    auto collide = [&](int step, const R (&f)[7], R c2, unsigned kc, R (&o)[7]) {
        collide_half<R, 3>(c2, f, o);
        if (DRIVEN && kc >= CELL_WALL_LO) boundary_cell<R, 7>(kc, f, c2, P.drv[step], o);
    };
    // a vector's cells; most are fluid throughout: one test instead of one per cell
    auto collide_vec = [&](int step, const R (&f0)[W], const R (&f1)[W], const R (&f2)[W], const R (&f3)[W],
                           const R (&f4)[W], const R (&f5)[W], const R (&f6)[W], R left, R right,
                           unsigned long long cl, unsigned id, R (&o)[7][W]) {
        const bool fluid = cl == 0;
        R c2[W];
#pragma unroll
        for (int e = 0; e < W; ++e) c2[e] = P.c0sq;
        if (!fluid) {
#pragma unroll
            for (int e = 0; e < W; ++e) c2[e] = sound((unsigned)(cl >> (8 * e)) & 0xffu, id + e);
        }
#pragma unroll
        for (int e = 0; e < W; ++e) {
            const R f[7] = {f0[e], e > 0 ? f1[e > 0 ? e - 1 : 0] : left, e < W - 1 ? f2[e < W - 1 ? e + 1 : 0] : right,
                            f3[e], f4[e], f5[e], f6[e]};
            R q[7];
            collide_half<R, 3>(c2[e], f, q);
#pragma unroll
            for (int i = 0; i < 7; ++i) o[i][e] = q[i];
        }
        if (DRIVEN && !fluid) {
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const unsigned kc = (unsigned)(cl >> (8 * e)) & 0xffu;
                if (kc >= CELL_WALL_LO) {
                    const R f[7] = {f0[e], e > 0 ? f1[e > 0 ? e - 1 : 0] : left,
                                    e < W - 1 ? f2[e < W - 1 ? e + 1 : 0] : right, f3[e], f4[e], f5[e], f6[e]};
                    R q[7];
                    boundary_cell<R, 7>(kc, f, c2[e], P.drv[step], q);
#pragma unroll
                    for (int i = 0; i < 7; ++i) o[i][e] = q[i];
                }
            }
        }
    };
    auto vput = [](R *p, const R (&v)[W]) {
#pragma unroll
        for (int e = 0; e < W; e += 4) {
            *reinterpret_cast<float4 *>(p + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
    };
    auto vget = [](const R *p, R (&v)[W]) {
#pragma unroll
        for (int e = 0; e < W; e += 4) {
            const float4 q = *reinterpret_cast<const float4 *>(p + e);
            v[e] = q.x;
            v[e + 1] = q.y;
            v[e + 2] = q.z;
            v[e + 3] = q.w;
        }
    };
    // step 1
    if (vec) {
        const int lo = inner && !wz ? -1 : 0, hi = inner && !wz ? td + 1 : td;
        for (int lz = lo + group; lz < hi; lz += groups) {
            int z = z0 + lz;
            z = z < 0 ? nz - 1 : (z >= nz ? 0 : z);
            const unsigned pz = (unsigned)z * plane;
            R f0[W], f1[W], f2[W], f3[W], f4[W], f5[W], f6[W];
            Store<S>::load_cg(P.A + (pz + c), f0);
            Store<S>::load_cg(P.A + (nc + pz + c), f1);
            Store<S>::load_cg(P.A + (2 * nc + pz + c), f2);
            const R left = Store<S>::get(P.A + (nc + pz + cxm)), right = Store<S>::get(P.A + (2 * nc + pz + cxp));
            Store<S>::load_cg(P.A + (3 * nc + pz + cym), f3);
            Store<S>::load_cg(P.A + (4 * nc + pz + cyp), f4);
            Store<S>::load_cg(P.A + (5 * nc + (unsigned)down(z, nz) * plane + c), f5);
            Store<S>::load_cg(P.A + (6 * nc + (unsigned)up(z, nz) * plane + c), f6);
            const unsigned long long cl = load_classes<W>(P.cls + (pz + c));
            R o[7][W];
            collide_vec(0, f0, f1, f2, f3, f4, f5, f6, left, right, cl, pz + c, o);
#pragma unroll
            for (int i = 0; i < 7; ++i)
#pragma unroll
                for (int e = 0; e < W; ++e) o[i][e] = as_stored<S>(o[i][e]);
            const int b = lz * sheet + ly * tw + lx;
            if (!inner) {
                if (ly < 0) vput(a3 + b + tw, o[3]);
                else vput(a4 + b - tw, o[4]);
            } else if (lz < 0) {
                vput(a5 + b + sheet, o[5]);
            } else if (lz >= td) {
                vput(a6 + b - sheet, o[6]);
            } else {
                vput(a0 + b, o[0]);
                const int pb = lz * psheet + ly * pad + W + lx;
                vput(a1 + pb, o[1]);
                vput(a2 + pb, o[2]);
                if (ly + 1 < th || wy) vput(a3 + (ly + 1 < th ? b + tw : b + tw - sheet), o[3]);
                if (ly > 0 || wy) vput(a4 + (ly > 0 ? b - tw : b - tw + sheet), o[4]);
                if (lz + 1 < td || wz) vput(a5 + (lz + 1 < td ? b + sheet : b + sheet - cells), o[5]);
                if (lz > 0 || wz) vput(a6 + (lz > 0 ? b - sheet : b - sheet + cells), o[6]);
            }
        }
    } else if (face) {
        for (int lz = group; lz < td; lz += groups) {
            const int z = z0 + lz;
            const unsigned pz = (unsigned)z * plane;
            R f[7], o[7];
            f[0] = Store<S>::get(P.A + (pz + c));
            f[1] = Store<S>::get(P.A + (nc + pz + cxm));
            f[2] = Store<S>::get(P.A + (2 * nc + pz + cxp));
            f[3] = Store<S>::get(P.A + (3 * nc + pz + cym));
            f[4] = Store<S>::get(P.A + (4 * nc + pz + cyp));
            f[5] = Store<S>::get(P.A + (5 * nc + (unsigned)down(z, nz) * plane + c));
            f[6] = Store<S>::get(P.A + (6 * nc + (unsigned)up(z, nz) * plane + c));
            const unsigned kc = P.cls[pz + c];
            collide(0, f, sound(kc, pz + c), kc, o);
            const int pb = lz * psheet + ly * pad + W + lx;
            if (lx < 0) a1[pb] = as_stored<S>(o[1]);
            else a2[pb] = as_stored<S>(o[2]);
        }
    }
    __syncthreads();
    if (!inner) return;
    // step 2 on the tile
    for (int lz = group; lz < td; lz += groups) {
        const unsigned pz = (unsigned)(z0 + lz) * plane;
        const int b = lz * sheet + ly * tw + lx, pb = lz * psheet + ly * pad + W + lx;
        const unsigned long long cl = load_classes<W>(P.cls + (pz + c));
        R f0[W], f1[W], f2[W], f3[W], f4[W], f5[W], f6[W];
        vget(a0 + b, f0);
        vget(a1 + pb, f1);
        vget(a2 + pb, f2);
        const R left = a1[wx && lx == 0 ? pb + tw - 1 : pb - 1], right = a2[wx && lx + W == tw ? pb + W - tw : pb + W];
        vget(a3 + b, f3);
        vget(a4 + b, f4);
        vget(a5 + b, f5);
        vget(a6 + b, f6);
        R o[7][W];
        collide_vec(1, f0, f1, f2, f3, f4, f5, f6, left, right, cl, pz + c, o);
#pragma unroll
        for (int i = 0; i < 7; ++i) Store<S>::store_keep(P.B + (i * nc + pz + c), o[i]);
    }
}

// ---------------------------------------------------------------- sampling
// The grouping of the points lives in the unused fourth component of the
// stencil coordinates: entry 0 the number of boxes, 1 + 5 b .. of box b its first
// centre cell (x, y, z, not wrapped), its first place in the list and its point
// count; the list (points by box) in the last N entries.
__device__ __forceinline__ int &aux(int4 *st, long long i) { return st[i].w; }
__device__ __forceinline__ int aux(const int4 *__restrict__ st, long long i) { return st[i].w; }

// One block: centre cells (as the setup rounds them) into boxes, counted,
// scanned, listed.
__global__ void __launch_bounds__(1024) group_points(Geometry g, const double *__restrict__ pts, int4 *st) {
    constexpr int kBoxes = kBoxAxis * kBoxAxis * kBoxAxis;
    __shared__ int cnt[kBoxes];
    __shared__ int sums[32], kept[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, N = g.n_surface;
    int origin[3];
    for (int a = 0; a < 3; ++a) origin[a] = (int)floor(g.center[a] - g.surface_radius) - 1;
    for (int i = tid; i < kBoxes; i += 1024) cnt[i] = 0;
    __syncthreads();
    auto box_of = [&](int k) {
        int b = 0;
        for (int a = 2; a >= 0; --a) {
            const int c = ((int)floor(pts[7 * (long long)k + a] + 0.5) - origin[a]) / kBox;
            b = b * kBoxAxis + min(max(c, 0), kBoxAxis - 1);
        }
        return b;
    };
    for (int k = tid; k < N; k += 1024) atomicAdd(&cnt[box_of(k)], 1);
    __syncthreads();
    // exclusive scan of the counts, and of the number of boxes in use, 4 per thread
    constexpr int kPer = kBoxes / 1024;
    int c[kPer], s = 0, used = 0;
    for (int j = 0; j < kPer; ++j) {
        c[j] = cnt[tid * kPer + j];
        s += c[j];
        used += c[j] > 0;
    }
    int is = s, iu = used;
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(kFull, is, o), b = __shfl_up_sync(kFull, iu, o);
        if (lane >= o) {
            is += a;
            iu += b;
        }
    }
    if (lane == 31) {
        sums[warp] = is;
        kept[warp] = iu;
    }
    __syncthreads();
    int start = is - s, slot = iu - used;
    for (int w = 0; w < warp; ++w) {
        start += sums[w];
        slot += kept[w];
    }
    for (int j = 0; j < kPer; ++j) {
        const int b = tid * kPer + j;
        cnt[b] = start;
        if (c[j] > 0) {
            const long long e = 1 + 5 * (long long)slot++;
            aux(st, e) = origin[0] + kBox * (b % kBoxAxis);
            aux(st, e + 1) = origin[1] + kBox * (b / kBoxAxis % kBoxAxis);
            aux(st, e + 2) = origin[2] + kBox * (b / (kBoxAxis * kBoxAxis));
            aux(st, e + 3) = start;
            aux(st, e + 4) = c[j];
        }
        start += c[j];
    }
    if (tid == 1023) aux(st, 0) = slot;
    __syncthreads();
    const long long list = 27LL * N - N;
    for (int k = tid; k < N; k += 1024) aux(st, list + atomicAdd(&cnt[box_of(k)], 1)) = k;
}

// Surface sums of steps t and t+1 from the state A of time t, in the order two
// single steps add them: one box per block.
template <typename S>
__global__ void __launch_bounds__(kSampleThreads) sample_boxes(SampleArgs<S> a, const S *__restrict__ A,
                                                               const typename Store<S>::R *__restrict__ c2f) {
    using R = typename Store<S>::R;
    extern __shared__ __align__(16) unsigned char box_raw[];
    R(*arr)[kMomCells] = reinterpret_cast<R(*)[kMomCells]>(box_raw);                         // [7]: arriving at t+1
    R(*mom)[4][kMomCells] = reinterpret_cast<R(*)[4][kMomCells]>(box_raw + sizeof(R) * 7 * kMomCells);  // rho, J at t, t+1
    const Geometry &g = a.g;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], tid = threadIdx.x;
    // the grid is an upper bound of the boxes, but holds no more blocks than points
    // (count_boxes), so a block's entries lie in the list (5 N < 27 N): loaded beside
    // the number of boxes, not after it (18.4 ms against 18.3 for the driven cavity)
    const long long e = 1 + 5 * (long long)blockIdx.x;
    const int boxes = aux(a.st_xyz, 0), bx = aux(a.st_xyz, e), by = aux(a.st_xyz, e + 1), bz = aux(a.st_xyz, e + 2),
              first = aux(a.st_xyz, e + 3), count = aux(a.st_xyz, e + 4);
    if ((int)blockIdx.x >= boxes) return;  // block-uniform
    auto wrap = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    const int ox = wrap(bx - 1, nx), oy = wrap(by - 1, ny), oz = wrap(bz - 1, nz);
    // the warp's first point, its stencil and sums: loaded beside the populations
    const long long list = 27LL * g.n_surface - g.n_surface;
    const int lane = tid & 31, warp = tid >> 5, cell = lane < 27 ? lane : 26;
    struct Point {
        int k;
        int4 at;
        R wp, wu, n[3], acc[5];
    };
    auto fetch = [&](int j) {
        Point q;
        q.k = aux(a.st_xyz, list + first + j);
        const long long o = 27LL * q.k + cell;
        q.at = a.st_xyz[o];
        q.wp = a.st_w[2 * o];
        q.wu = a.st_w[2 * o + 1];
#pragma unroll
        for (int i = 0; i < 3; ++i) q.n[i] = a.nrm[4LL * q.k + i];
#pragma unroll
        for (int i = 0; i < 5; ++i) q.acc[i] = a.acc[5LL * q.k + i];
        return q;
    };
    Point pt = fetch(warp < count ? warp : 0);
    auto at = [](int o, int l, int n) {  // box coordinate -1 .. kMom to lattice coordinate
        int v = o + l;
        while (v >= n) v -= n;
        return v < 0 ? v + n : v;
    };
    constexpr int kSheet = kMom * kMom;
    for (int i = tid; i < kMomCells + 6 * kSheet; i += kSampleThreads) {
        int lx, ly, lz, dir = 0, dst = 0;
        if (i < kMomCells) {
            lz = i / kSheet;
            ly = i / kMom % kMom;
            lx = i % kMom;
        } else {
            const int q = i - kMomCells, face = q / kSheet, u = q % kMom, v = q / kMom % kMom;
            const int end = face & 1 ? kMom : -1, in = face & 1 ? kMom - 1 : 0;
            lx = face < 2 ? end : u;
            ly = face < 2 ? u : (face < 4 ? end : v);
            lz = face < 4 ? v : end;
            dir = face < 2 ? 1 + (face & 1) : (face < 4 ? 3 + (face & 1) : 5 + (face & 1));
            dst = face < 2 ? (v * kMom + u) * kMom + in : (face < 4 ? (v * kMom + in) * kMom + u : (in * kMom + v) * kMom + u);
        }
        const int x = at(ox, lx, nx), y = at(oy, ly, ny), z = at(oz, lz, nz);
        R f[7], o[7];
        pull<S>(A, g.ncell, nx, ny, nz, x, y, z, f);
        collide_half<R, 3>(c2f[((long long)z * ny + y) * nx + x], f, o);  // stencils lie clear of walls and sheet
        if (i < kMomCells) {
            R rho = add_rn(add_rn(add_rn(add_rn(f[0], f[1]), f[2]), f[3]), f[4]);
            mom[0][0][i] = add_rn(rho, add_rn(f[5], f[6]));
            mom[0][1][i] = sub_rn(f[1], f[2]);
            mom[0][2][i] = sub_rn(f[3], f[4]);
            mom[0][3][i] = sub_rn(f[5], f[6]);
            arr[0][i] = as_stored<S>(o[0]);
            if (lx + 1 < kMom) arr[1][i + 1] = as_stored<S>(o[1]);
            if (lx > 0) arr[2][i - 1] = as_stored<S>(o[2]);
            if (ly + 1 < kMom) arr[3][i + kMom] = as_stored<S>(o[3]);
            if (ly > 0) arr[4][i - kMom] = as_stored<S>(o[4]);
            if (lz + 1 < kMom) arr[5][i + kSheet] = as_stored<S>(o[5]);
            if (lz > 0) arr[6][i - kSheet] = as_stored<S>(o[6]);
        } else {
            R v = o[1];
#pragma unroll
            for (int d = 2; d < 7; ++d) v = dir == d ? o[d] : v;
            arr[dir][dst] = as_stored<S>(v);
        }
    }
    __syncthreads();
    for (int i = tid; i < kMomCells; i += kSampleThreads) {
        const R rho = add_rn(add_rn(add_rn(add_rn(arr[0][i], arr[1][i]), arr[2][i]), arr[3][i]), arr[4][i]);
        mom[1][0][i] = add_rn(rho, add_rn(arr[5][i], arr[6][i]));
        mom[1][1][i] = sub_rn(arr[1][i], arr[2][i]);
        mom[1][2][i] = sub_rn(arr[3][i], arr[4][i]);
        mom[1][3][i] = sub_rn(arr[5][i], arr[6][i]);
    }
    __syncthreads();
    // a warp per point: the sums of sample_point_with from shared memory
    for (int j = warp; j < count; j += kSampleThreads / 32) {
        int lx = pt.at.x - ox, ly = pt.at.y - oy, lz = pt.at.z - oz;
        lx += lx < 0 ? nx : 0;
        ly += ly < 0 ? ny : 0;
        lz += lz < 0 ? nz : 0;
        const int c = (min(lz, kMom - 1) * kMom + min(ly, kMom - 1)) * kMom + min(lx, kMom - 1);
        const int k = pt.k;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            R p = R(0), u[3] = {R(0), R(0), R(0)};
            if (lane < 27) {
                p = mul_rn(pt.wp, mom[s][0][c]);
#pragma unroll
                for (int i = 0; i < 3; ++i) u[i] = mul_rn(pt.wu, mom[s][1 + i][c]);
            }
#pragma unroll
            for (int m = 16; m >= 1; m >>= 1) {
                p = add_rn(p, __shfl_xor_sync(kFull, p, m));
#pragma unroll
                for (int i = 0; i < 3; ++i) u[i] = add_rn(u[i], __shfl_xor_sync(kFull, u[i], m));
            }
            accumulate_point(pt.acc, p, u, pt.n);
        }
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < 5; ++i) a.acc[5LL * k + i] = pt.acc[i];
        }
        if (j + kSampleThreads / 32 < count) pt = fetch(j + kSampleThreads / 32);
    }
}

// ---------------------------------------------------------------- host side: plans and launches

// Boxes that can hold a centre cell: those the sphere's surface, one cell thick
// on either side, passes through, and no more than there are points (sample_boxes
// relies on that bound).
int count_boxes(const Geometry &g) {
    const double R = g.surface_radius;
    int n = 0;
    double lo[3];
    for (int a = 0; a < 3; ++a) lo[a] = std::floor(g.center[a] - R) - 1 - g.center[a];
    const int per = (int)((2 * R + 4) / kBox) + 1;
    for (int z = 0; z < per; ++z)
        for (int y = 0; y < per; ++y)
            for (int x = 0; x < per; ++x) {
                const int b[3] = {x, y, z};
                double near = 0, far = 0;
                for (int a = 0; a < 3; ++a) {
                    const double l = lo[a] + kBox * b[a] - 1.0, h = l + kBox + 1.0;
                    const double d = l > 0 ? l : (h < 0 ? -h : 0.0), f = std::fmax(std::fabs(l), std::fabs(h));
                    near += d * d;
                    far += f * f;
                }
                n += near <= R * R && far >= R * R;
            }
    return n < g.n_surface ? n : g.n_surface;
}

template <typename S>
constexpr size_t box_smem() {
    return sizeof(typename Store<S>::R) * 15 * kMomCells;
}

template <typename S, bool DRIVEN>
cudaError_t allow_smem() {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tile_two_steps_3d<S, DRIVEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(sample_boxes<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)box_smem<S>());
    return e;
}

// Threads for one plane of a tile: its vectors and those of the y faces, then
// the cells of the x faces, both in whole warps.
template <typename S>
int plane_threads(const Geometry &g, int tx, int ty, int *face_begin) {
    const int v = tx / Store<S>::W * (ty + (ty == g.n[1] ? 0 : 2)), f = tx == g.n[0] ? 0 : 2 * ty;
    *face_begin = (v + 31) / 32 * 32;
    return *face_begin + (f + 31) / 32 * 32;
}

// Tile by estimated time of a launch, in SM cycles: 2500, and per wave of
// resident CTAs 800 and the rounds over the planes, each bound by the latency of
// its loads: 2000 in step 1, 1400 in step 2; at least what the bytes take at the
// HBM rate.  Rows the one-step kernel takes as whole warps of vectors stay there
// (256 x 64 x 103 driven FP16: 6.9 us per step, in tiles 11).  Measured (GB300, us
// per step unsampled, sampled; one step per launch as it was -> tiles):
//   64 x 64 x 203 driven FP32    7.5 -> 4.8    10.2 -> 6.6   (1000 points)
//   40 x 40 x 64 FP32            2.2 -> 1.5     4.7 -> 3.0   (500)
//   36 x 120 x 150 FP32          5.9 -> 3.5     9.7 -> 6.3   (1500)
//   200 x 201 x 128 FP32        44.5 -> 34.6   48.0 -> 35.8
//   200 x 256 x 252 FP32         109 -> 81      112 -> 82
//   200 x 200 x 100 FP16        31.2 -> 20.6   34.8 -> 21.3
template <typename S>
cudaError_t plan_for(const Geometry &g, int sms, size_t smem_max, TilePlan3D *out) {
    constexpr int W = Store<S>::W;
    if (update_is_vectorised(g, sizeof(S) == 2 ? Prec::F16 : Prec::F32)) return cudaSuccess;  // its row kernel is as fast
    if (g.n[0] % W != 0 || g.ncell > (1LL << 32) / 7 - 1) return cudaSuccess;
    // Loads in flight are held by the L1 cache, which gets what shared memory
    // leaves: 228 KB tiles ran at half the speed of 150 KB ones.
    if (smem_max > kMaxSmem) smem_max = kMaxSmem;
    TilePlan3D best;
    double best_cost = 0;
    int last_x = 0;
    for (int m = 1; m <= g.n[0]; ++m) {
        const int tx = ((g.n[0] + m - 1) / m + W - 1) / W * W;
        if (tx == last_x || tx > 512) continue;
        if (tx < 4 * W && m > 1) break;
        if (m > 1 && g.n[0] <= 80 * W) break;  // x faces are one cell per 32-byte sector: only for long rows
        last_x = tx;
        int last_y = 0;
        for (int n = 1; n <= g.n[1]; ++n) {
            const int ty = (g.n[1] + n - 1) / n;
            if (ty == last_y) continue;
            if (ty < 2 && n > 1) break;
            last_y = ty;
            int fb;
            const int pt = plane_threads<S>(g, tx, ty, &fb);
            if (pt > kMaxThreads || tile_smem<S>(tx, ty, 1) > smem_max) continue;
            const long long xy = (long long)((g.n[0] + tx - 1) / tx) * ((g.n[1] + ty - 1) / ty);
            int last_z = 0;
            for (long long r = 1; r <= 4096; r = r < 8 ? r + 1 : r + r / 4) {
                long long p = r * sms / xy;
                p = p < 1 ? 1 : (p > g.n[2] ? g.n[2] : p);
                const int tz = (int)((g.n[2] + p - 1) / p);
                if (tz == last_z) continue;
                last_z = tz;
                const size_t smem = tile_smem<S>(tx, ty, tz);
                if (smem > smem_max) continue;
                const int threads = pt * (kMaxThreads / pt < tz + 2 ? kMaxThreads / pt : tz + 2);
                const int groups = threads / pt;
                int res = (int)(smem_max / smem);  // resident CTAs, by shared memory and 112 registers a thread
                if (res > 65536 / (threads * 112)) res = 65536 / (threads * 112);
                if (res < 1) res = 1;
                const int planes1 = tz + (tz == g.n[2] ? 0 : 2);
                const double rounds = 2000.0 * ((planes1 + groups - 1) / groups) + 1400.0 * ((tz + groups - 1) / groups);
                const long long tiles = xy * ((g.n[2] + tz - 1) / tz);
                const double waves = std::ceil((double)tiles / ((double)sms * res));
                const double ratio = (double)pt * W / ((double)tx * ty) * planes1 / tz;
                const double bytes = (double)g.ncell * (7 * sizeof(S) * (ratio + 1.0) + 1);
                const double cost = std::fmax(2500.0 + waves * (800.0 + rounds * (1.0 + 0.3 * (res - 1))),
                                              2500.0 + 1.15 * bytes / (23.3 * sms));
                if (best.tx == 0 || cost < best_cost) {
                    best_cost = cost;
                    best.tx = tx;
                    best.ty = ty;
                    best.tz = tz;
                    best.smem = smem;
                    best.threads = threads;
                }
                if (p == g.n[2]) break;
            }
        }
    }
    if (best.tx == 0) return cudaSuccess;
    cudaError_t e = g.driven ? allow_smem<S, true>() : allow_smem<S, false>();
    if (e != cudaSuccess) return e;
    if (g.n_surface > 0 && 2 * g.surface_radius + 4 < kBox * kBoxAxis) best.boxes = count_boxes(g);
    *out = best;
    return cudaSuccess;
}

template <typename S>
cudaError_t launch_for(const Geometry &g, const Buffers &b, const TilePlan3D &pl, int src, bool sample, long long t_mod,
                       cudaStream_t s, const SideStream &side) {
    using R = typename Store<S>::R;
    cudaError_t e;
    const bool fork = sample && side.stream != nullptr;
    if (sample) {
        cudaStream_t ss = s;
        if (fork) {
            if ((e = cudaEventRecord(side.fork, s)) != cudaSuccess ||
                (e = cudaStreamWaitEvent(side.stream, side.fork, 0)) != cudaSuccess)
                return e;
            ss = side.stream;
        }
        sample_boxes<S><<<pl.boxes, kSampleThreads, box_smem<S>(), ss>>>(sample_args<S>(g, b), (const S *)b.pop[src], (const R *)b.c2);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    Tile3D<S> a;
    a.A = (const S *)b.pop[src];
    a.B = (S *)b.pop[src ^ 1];
    a.cls = b.cls;
    a.c2f = (const R *)b.c2;
    a.nx = g.n[0];
    a.ny = g.n[1];
    a.nz = g.n[2];
    a.ncell = g.ncell;
    a.tx = pl.tx;
    a.ty = pl.ty;
    a.tz = pl.tz;
    a.tiles_x = (g.n[0] + pl.tx - 1) / pl.tx;
    a.tiles_y = (g.n[1] + pl.ty - 1) / pl.ty;
    a.plane_threads = plane_threads<S>(g, pl.tx, pl.ty, &a.face_begin);
    a.c0sq = (R)(g.c0 * g.c0);
    a.cpsq = (R)(g.cp * g.cp);
    for (int i = 0; i < 2; ++i) {
        a.drv[i].rho_src = (R)(g.driven ? source_density(g, (t_mod + i) % g.period) : 0.0);
        a.drv[i].phi = (R)g.wall_damping;
        a.drv[i].axis = g.wave_axis;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((long long)a.tiles_x * a.tiles_y * ((g.n[2] + pl.tz - 1) / pl.tz)));
    cfg.blockDim = dim3(pl.threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = sample ? 0 : 1;  // beside a forked sampling kernel: plain stream order
    e = g.driven ? cudaLaunchKernelEx(&cfg, tile_two_steps_3d<S, true>, a)
                 : cudaLaunchKernelEx(&cfg, tile_two_steps_3d<S, false>, a);
    if (e != cudaSuccess || !fork) return e;
    if ((e = cudaEventRecord(side.join, side.stream)) != cudaSuccess) return e;
    return cudaStreamWaitEvent(s, side.join, 0);
}

}  // namespace

cudaError_t plan_tile_3d(const Geometry &g, Prec p, TilePlan3D *out) {
    *out = TilePlan3D{};
    if (g.dim != 3) return cudaSuccess;
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    switch (p) {
        case Prec::F64: return cudaSuccess;  // bound by the FP64 pipe: the face cells only add to it
        case Prec::F16: return plan_for<__half>(g, sms, (size_t)optin, out);
        default: return plan_for<float>(g, sms, (size_t)optin, out);
    }
}

cudaError_t launch_tile_3d(const Geometry &g, const Buffers &b, Prec p, const TilePlan3D &pl, int src, bool sample,
                           long long t_mod, cudaStream_t s, const SideStream &side) {
    switch (p) {
        case Prec::F64: return cudaErrorInvalidValue;
        case Prec::F16: return launch_for<__half>(g, b, pl, src, sample, t_mod, s, side);
        default: return launch_for<float>(g, b, pl, src, sample, t_mod, s, side);
    }
}

cudaError_t launch_group_points(const Geometry &g, const Buffers &b, cudaStream_t s) {
    group_points<<<1, 1024, 0, s>>>(g, b.pts, b.st_xyz);
    return cudaGetLastError();
}

}  // namespace wlb
