// Setup kernels: cell classes and sound-speed field (Sec. VI, Eq. 79), the
// standing-wave initial condition imposed through the equilibrium (Sec. V,
// Eqs. 71-72), surface elements (Sec. VI) and the interpolation stencils with
// the three-point kernel of Eq. (82).
//
// Everything is defined in FP64 (classes and points are bit-exact), and FP64
// is what bounds a direct evaluation: the chip retires about two FP64
// instructions per clock and SM.  So the FP64 work is done once where it is
// the same for many cells: the initial populations of fluid and object cells
// depend only on the coordinate along the wave (tables), and a cell whose
// distance from the surface is far outside the interface band is classified
// from an FP32 distance with an error margin; only the cells near the band
// evaluate |x - r0|^2, the tanh profile and their own equilibrium in FP64.
// Surface elements are spread over a thread per stencil cell.  A batch sets
// up all its lattices in the same three launches.  Measured (GB300): evaluated
// directly, one thread per cell and per point, 256^3 took 3.26 ms (cells) and
// 0.167 ms (2000 points), 512^3 25.9 ms, and a batch of 512 2D lattices set up
// one after another 37 ms; whole runs are now 3.1, 24.9 and 50 ms shorter (the
// last with the batch's forces in one launch).
#include <cuda_fp16.h>

#include <cstring>
#include <type_traits>

#include "wlb_internal.cuh"

namespace wlb {
namespace {

constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double kHalfPi = 1.5707963267948966192313216916398;
constexpr double kGoldenTurn = 0.3819660112501051517954131656;  // (3 - sqrt 5) / 2

__device__ __forceinline__ int wrap_index(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

// Minimum-image displacement along a periodic axis of length n.
__device__ __forceinline__ double min_image(double d, int n) {
    if (d >= 0.5 * n) return d - n;
    if (d < -0.5 * n) return d + n;
    return d;
}

// |x - r0|^2 - R^2, exact for centres on a 2^-10 grid.
__device__ double excess_r2(const Geometry &g, int x, int y, int z) {
    const int c[3] = {x, y, z};
    double s = 0.0;
    for (int a = 0; a < g.dim; ++a) {
        double d = min_image(__dadd_rn((double)c[a], -g.center[a]), g.n[a]);
        s = __dadd_rn(s, __dmul_rn(d, d));
    }
    return __dadd_rn(s, -__dmul_rn(g.radius, g.radius));
}

__device__ uint8_t cell_class(const Geometry &g, double q) {
    if (q >= g.band_half) return CELL_FLUID;
    if (q <= -g.band_half) return CELL_OBJECT;
    return CELL_BAND;
}

// Sound speed squared as the update kernel uses it: c0^2 for fluid cells,
// cp^2 for object cells, Eq. (79) (c0 outside, cp inside) in the band.
__device__ double sound_speed_sq(const Geometry &g, int x, int y, int z) {
    double q = excess_r2(g, x, y, z);
    uint8_t k = cell_class(g, q);
    if (k == CELL_FLUID) return g.c0 * g.c0;
    if (k == CELL_OBJECT) return g.cp * g.cp;
    double c = g.cp + 0.5 * (g.c0 - g.cp) * (1.0 + tanh(q / g.interface_d));
    return c * c;
}

// Standing-wave pressure at t = 0 (Eq. 38, s measured from an antinode) at
// coordinate s along the wave axis.
__device__ __forceinline__ double incident(const Geometry &g, int s) {
    return g.p_a * cos(2.0 * kPi * ((double)s - g.antinode) / g.wavelength);
}

// Conversion of an FP64 value to the storage type (round to nearest).
template <typename S> __device__ __forceinline__ S to_store(double v) { return (S)v; }
template <> __device__ __forceinline__ __half to_store<__half>(double v) { return __double2half(v); }

// f_0^eq = rho1 (1 - D c^2) of Eq. (71) with rho1 = p / c^2, times the storage
// scale; f_i^eq = c^2 rho1 / 2 for i > 0.
__device__ __forceinline__ double rest_population(const Geometry &g, double p, double c2) {
    return (p / c2) * (1.0 - g.dim * c2) * g.pop_scale;
}

// Tables along the wave axis for the cells kernel, in the read-back staging
// buffer (nothing else uses it during the setup): f_0^eq of fluid cells, of
// object cells, and f_i^eq.  They fit whenever the axis is no longer than the
// staged cells; otherwise every cell evaluates its own.
__host__ __device__ inline bool tables_fit(const Geometry &g, const Buffers &b) {
    return g.n[g.wave_axis] <= b.stage_cells;
}

// Launch 1: the tables and the incident pressure, and every buffer that must
// start at zero.
template <typename S, typename T>
__device__ void prepare_lattice(const Geometry &g, const Buffers &b, long long i0, long long stride) {
    const int ns = g.n[g.wave_axis];
    S *tab = reinterpret_cast<S *>(b.stage);
    for (long long s = i0; s < ns; s += stride) {
        const double p = g.driven ? 0.0 : incident(g, (int)s);  // the driven cavity starts from rest
        b.ptab[s] = p;
        if (tables_fit(g, b)) {
            tab[s] = to_store<S>(rest_population(g, p, g.c0 * g.c0));
            tab[ns + s] = to_store<S>(rest_population(g, p, g.cp * g.cp));
            tab[2 * (long long)ns + s] = to_store<S>(0.5 * p * g.pop_scale);
        }
    }
    auto zero = [&](void *ptr, size_t bytes) {  // buffers are padded to 256 bytes
        uint4 *v = reinterpret_cast<uint4 *>(ptr);
        for (long long i = i0; i < (long long)((bytes + 15) / 16); i += stride) v[i] = make_uint4(0, 0, 0, 0);
    };
    zero(b.band_rows, (size_t)g.n[1] * g.n[2]);
    if (g.n_surface > 0) {
        zero(b.acc, sizeof(T) * 5 * (size_t)g.n_surface);
        zero(b.acc64, sizeof(double) * 5 * (size_t)g.n_surface);
    }
    zero(b.force, 4 * sizeof(double));
    if (i0 == 0) *b.err = 0;
}

// Launch 2: the cells of a lattice row, W consecutive cells per thread.
// Populations are stored post-collision and pulled by the next update, so the
// stored value of direction i at cell x is the value that arrives at x + v_i:
// the equilibrium (Eq. 71 with rho1 = p1/c^2, J1 = 0) of the cell x + v_i,
// times the storage scale.
template <typename S, typename T, int W>
__device__ void setup_row(const Geometry &g, const Buffers &b, long long row, int lane) {
    const int nx = g.n[0], ny = g.n[1], ax = g.wave_axis, ns = g.n[ax];
    const int z = (int)(row < (1LL << 31) ? (unsigned)row / (unsigned)ny : row / ny);
    const int y = (int)(row - (long long)z * ny);
    const bool tables = tables_fit(g, b);
    const S *tab = reinterpret_cast<const S *>(b.stage);
    const double c0sq = g.c0 * g.c0, cpsq = g.cp * g.cp;
    const T c0t = (T)c0sq, cpt = (T)cpsq;
    // populations of fluid and object cells at coordinate s along the wave: rest,
    // +-i off the wave axis, and along it (+: arriving at s + 1, -: at s - 1)
    struct Column {
        S fluid, object, here, next, prev;
    };
    auto column = [&](int s) {
        const int sp = s == ns - 1 ? 0 : s + 1, sm = s == 0 ? ns - 1 : s - 1;
        Column c;
        if (tables) {
            const S *h = tab + 2 * (long long)ns;
            c.fluid = tab[s];
            c.object = tab[ns + s];
            c.here = h[s];
            c.next = h[sp];
            c.prev = h[sm];
        } else {
            c.fluid = to_store<S>(rest_population(g, b.ptab[s], c0sq));
            c.object = to_store<S>(rest_population(g, b.ptab[s], cpsq));
            c.here = to_store<S>(0.5 * b.ptab[s] * g.pop_scale);
            c.next = to_store<S>(0.5 * b.ptab[sp] * g.pop_scale);
            c.prev = to_store<S>(0.5 * b.ptab[sm] * g.pop_scale);
        }
        return c;
    };
    // FP32 distance from the centre: whole cells and a fraction apart, so that
    // its relative error stays a few 2^-24 on any axis length
    struct Centre {
        long long whole;
        float part;
    };
    auto centre = [&](int a) {
        const double f = floor(g.center[a]);
        return Centre{(long long)fmin(fmax(f, -1e15), 1e15), (float)(g.center[a] - f)};
    };
    auto offset = [](int c, const Centre &o, int n) {
        long long d = c - o.whole;
        if (2 * d >= n) d -= n;
        if (2 * d < -n) d += n;
        return (float)d - o.part;
    };
    const Centre ox = centre(0);
    const float dy = offset(y, centre(1), ny), dz = g.dim == 3 ? offset(z, centre(2), g.n[2]) : 0.0f;
    const float yz = dy * dy + dz * dz, r2 = (float)(g.radius * g.radius), half_band = (float)g.band_half;
    const int s_row = ax == 1 ? y : z;  // the row's coordinate along the wave (waves along x: per cell)
    Column col{};
    if (ax != 0) col = column(s_row);
    for (int x0 = lane * W; x0 < nx; x0 += 32 * W) {
        const long long id = row * nx + x0;
        uint8_t cls[W];
        T c2[W];
        S f0[W], fi[6][W];
        bool band = false;
#pragma unroll
        for (int e = 0; e < W; ++e) {
            const int x = x0 + e, s = ax == 0 ? x : s_row;
            if (ax == 0) col = column(x);
            const float dx = offset(x, ox, nx);
            const float r = dx * dx + yz, q = r - r2, margin = 0.5f + 1e-5f * (r + r2);
            uint8_t k = q > half_band + margin ? CELL_FLUID
                                               : (q < -half_band - margin ? CELL_OBJECT : (uint8_t)CELL_BAND);
            if (k == CELL_BAND) k = cell_class(g, excess_r2(g, x, y, z));  // near the band: exact
            if (k == CELL_BAND) {
                band = true;
                const double v = sound_speed_sq(g, x, y, z);
                c2[e] = (T)v;
                f0[e] = to_store<S>(rest_population(g, b.ptab[s], v));
            } else {
                c2[e] = k == CELL_FLUID ? c0t : cpt;
                f0[e] = k == CELL_FLUID ? col.fluid : col.object;
            }
            if (g.driven) {  // walls and source sheet lie in the fluid
                if (s == 0) k = CELL_WALL_LO;
                else if (s == ns - 1) k = CELL_WALL_HI;
                else if (s == 1) k = CELL_SOURCE;
            }
            cls[e] = k;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                fi[2 * a][e] = a == ax ? col.next : col.here;
                fi[2 * a + 1][e] = a == ax ? col.prev : col.here;
            }
        }
        if (band) b.band_rows[row] = 1;  // every writer stores the same value
        S *pop = reinterpret_cast<S *>(b.pop[0]);
        auto put = [](auto *dst, const auto (&v)[W]) {
            using V = typename std::remove_reference<decltype(v[0])>::type;
            constexpr int kBytes = (int)(W * sizeof(V));
            if constexpr (kBytes % 16 == 0) {
#pragma unroll
                for (int j = 0; j < kBytes / 16; ++j) {
                    uint4 t;
                    memcpy(&t, reinterpret_cast<const char *>(v) + 16 * j, 16);
                    reinterpret_cast<uint4 *>(dst)[j] = t;
                }
            } else if constexpr (kBytes == 8) {
                uint2 t;
                memcpy(&t, v, 8);
                *reinterpret_cast<uint2 *>(dst) = t;
            } else if constexpr (kBytes == 4 && W > 1) {
                unsigned t;
                memcpy(&t, v, 4);
                *reinterpret_cast<unsigned *>(dst) = t;
            } else {
#pragma unroll
                for (int e = 0; e < W; ++e) dst[e] = v[e];
            }
        };
        put(b.cls + id, cls);
        put(reinterpret_cast<T *>(b.c2) + id, c2);
        put(pop + id, f0);
#pragma unroll
        for (int i = 1; i < 7; ++i)
            if (i < g.q) put(pop + (long long)i * g.ncell + id, fi[i - 1]);
    }
}

// 1 / n! for n < 22, each the correctly rounded quotient of the exact
// factorial (all are below 2^66 with at most 53 significant bits).
struct InverseFactorials {
    double v[22];
    constexpr InverseFactorials() : v{} {
        double f = 1.0;
        v[0] = 1.0;
        for (int i = 1; i < 22; ++i) {
            f *= (double)i;
            v[i] = 1.0 / f;
        }
    }
};

// sin and cos of 2 pi t, t in [0, 1): exact quadrant reduction, then the Taylor
// series to x^21 (Horner in x^2, coefficients 1/n! from exact factorials) on
// [-pi/4, pi/4].  Only correctly rounded operations, no contraction, so the
// sequence of IEEE operations is fixed.
__device__ void sincos_turns(double t, double *s, double *c) {
    double u = __dmul_rn(t, 4.0);
    int q = (int)floor(u);
    double r = __dadd_rn(u, -(double)q);
    if (r > 0.5) { r = __dadd_rn(r, -1.0); q += 1; }
    double th = __dmul_rn(r, kHalfPi);
    double th2 = __dmul_rn(th, th);
    double ps = 0.0, pc = 0.0;
#pragma unroll
    for (int m = 10; m >= 0; --m) {
        constexpr InverseFactorials inv{};
        const double cs = m & 1 ? -inv.v[2 * m + 1] : inv.v[2 * m + 1];
        const double cc = m & 1 ? -inv.v[2 * m] : inv.v[2 * m];
        ps = __dadd_rn(__dmul_rn(ps, th2), cs);
        pc = __dadd_rn(__dmul_rn(pc, th2), cc);
    }
    double sv = __dmul_rn(th, ps), cv = pc;
    switch (q & 3) {
        case 0: *s = sv; *c = cv; break;
        case 1: *s = cv; *c = -sv; break;
        case 2: *s = -sv; *c = -cv; break;
        default: *s = -cv; *c = sv; break;
    }
}

// Eq. (82): three-point kernel, one axis.
__device__ double kernel3(double r) {
    double a = fabs(r);
    if (a <= 0.5) return (1.0 + sqrt(1.0 - 3.0 * r * r)) / 3.0;
    if (a <= 1.5) return (5.0 - 3.0 * a - sqrt(1.0 - 3.0 * (1.0 - a) * (1.0 - a))) / 6.0;
    return 0.0;
}

// Launch 3: surface elements, centre, normal and size (Sec. VI), then the
// 3^dim stencil of Eqs. (80)-(81) with tensor-product weights.  A block takes
// kSurfPoints elements of a lattice: a thread per element for the normals, per
// element and axis offset for the kernel values, and per stencil cell for the
// weights (the tanh of Eq. 79 in each is the long part).
constexpr int kSurfThreads = 224;
__host__ __device__ constexpr int surf_points(int dim) { return dim == 3 ? 8 : 24; }  // 216 stencil cells either way

template <typename T>
__device__ void setup_surface_block(const Geometry &g, const Buffers &b, int block) {
    __shared__ double sX[24][3], sW[24][3][3];
    __shared__ int sBase[24][3];
    const int P = surf_points(g.dim), k0 = block * P, tid = threadIdx.x;
    const int N = g.n_surface, np = N - k0 < P ? N - k0 : P;
    double *pts = b.pts;
    T *nrm = reinterpret_cast<T *>(b.nrm), *st_w = reinterpret_cast<T *>(b.st_w);
    if (tid < np) {
        const int k = k0 + tid;
        const double Rs = g.surface_radius;
        double n[3] = {0.0, 0.0, 0.0};
        double dS;
        if (g.dim == 2) {
            double t = __ddiv_rn((double)(2 * k + 1), (double)(2 * N));
            sincos_turns(t, &n[1], &n[0]);
            dS = __ddiv_rn(__dmul_rn(__dmul_rn(2.0, kPi), Rs), (double)N);
        } else {
            double zk = __dadd_rn(1.0, -__ddiv_rn((double)(2 * k + 1), (double)N));
            double rho = __dsqrt_rn(__dadd_rn(1.0, -__dmul_rn(zk, zk)));
            double a = __dmul_rn((double)k, kGoldenTurn);
            double t = __dadd_rn(a, -floor(a));
            double sp, cp;
            sincos_turns(t, &sp, &cp);
            n[0] = __dmul_rn(rho, cp);
            n[1] = __dmul_rn(rho, sp);
            n[2] = zk;
            dS = __ddiv_rn(__dmul_rn(__dmul_rn(4.0, kPi), __dmul_rn(Rs, Rs)), (double)N);
        }
        for (int a = 0; a < 3; ++a) {
            const double X = (a < g.dim) ? __dadd_rn(g.center[a], __dmul_rn(Rs, n[a])) : 0.0;
            pts[7 * (long long)k + a] = X;
            pts[7 * (long long)k + 3 + a] = n[a];
            nrm[4 * (long long)k + a] = (T)n[a];
            sX[tid][a] = X;
            sBase[tid][a] = a < g.dim ? (int)floor(X + 0.5) : 0;
        }
        nrm[4 * (long long)k + 3] = (T)0;
        pts[7 * (long long)k + 6] = dS;
    }
    __syncthreads();
    for (int i = tid; i < np * 9; i += kSurfThreads) {
        const int p = i / 9, a = (i / 3) % 3, d = i % 3;
        if (a < g.dim) sW[p][a][d] = kernel3((double)(sBase[p][a] + d - 1) - sX[p][a]);
    }
    __syncthreads();
    for (int i = tid; i < np * g.stencil; i += kSurfThreads) {
        const int p = i / g.stencil, slot = i % g.stencil;  // slot: dz outermost, dx innermost
        const int ix = slot % 3, iy = (slot / 3) % 3, iz = slot / 9;
        double w = sW[p][0][ix] * sW[p][1][iy];
        if (g.dim == 3) w *= sW[p][2][iz];
        const int cx = wrap_index(sBase[p][0] + ix - 1, g.n[0]);
        const int cy = wrap_index(sBase[p][1] + iy - 1, g.n[1]);
        const int cz = g.dim == 3 ? wrap_index(sBase[p][2] + iz - 1, g.n[2]) : 0;
        const long long o = (long long)(k0 + p) * g.stencil + slot;
        b.st_xyz[o] = make_int4(cx, cy, cz, 0);
        st_w[2 * o] = (T)(w * sound_speed_sq(g, cx, cy, cz));
        st_w[2 * o + 1] = (T)(w / g.rho0);
    }
}

// The three launches for one lattice and for a batch (blockIdx.y: lattice).
constexpr int kRowsPerBlock = 8;  // warps, one row each

template <typename S, typename T>
__global__ void __launch_bounds__(256) prepare_one(Geometry g, Buffers b) {
    prepare_lattice<S, T>(g, b, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}
template <typename S, typename T>
__global__ void __launch_bounds__(256) prepare_batch(const BatchLat *__restrict__ lats) {
    const BatchLat &L = lats[blockIdx.y];
    prepare_lattice<S, T>(L.g, L.b, (long long)blockIdx.x * blockDim.x + threadIdx.x,
                          (long long)gridDim.x * blockDim.x);
}
template <typename S, typename T, int W>
__global__ void __launch_bounds__(32 * kRowsPerBlock) cells_one(Geometry g, Buffers b) {
    const long long row = (long long)blockIdx.x * kRowsPerBlock + (threadIdx.x >> 5);
    if (row < (long long)g.n[1] * g.n[2]) setup_row<S, T, W>(g, b, row, threadIdx.x & 31);
}
template <typename S, typename T, int W>
__global__ void __launch_bounds__(32 * kRowsPerBlock) cells_batch(const BatchLat *__restrict__ lats) {
    const BatchLat &L = lats[blockIdx.y];
    const long long row = (long long)blockIdx.x * kRowsPerBlock + (threadIdx.x >> 5);
    if (row < (long long)L.g.n[1] * L.g.n[2]) setup_row<S, T, W>(L.g, L.b, row, threadIdx.x & 31);
}
template <typename T>
__global__ void __launch_bounds__(kSurfThreads) surface_one(Geometry g, Buffers b) {
    setup_surface_block<T>(g, b, blockIdx.x);
}
template <typename T>
__global__ void __launch_bounds__(kSurfThreads) surface_batch(const BatchLat *__restrict__ lats) {
    const BatchLat &L = lats[blockIdx.y];
    if ((int)blockIdx.x * surf_points(L.g.dim) < L.g.n_surface) setup_surface_block<T>(L.g, L.b, blockIdx.x);
}

template <typename S, typename T>
cudaError_t setup_impl(const Geometry &g, const Buffers &b, cudaStream_t s) {
    constexpr int W = 16 / (int)sizeof(S);
    const long long rows = (long long)g.n[1] * g.n[2];
    prepare_one<S, T><<<64, 256, 0, s>>>(g, b);
    const unsigned blocks = (unsigned)((rows + kRowsPerBlock - 1) / kRowsPerBlock);
    // W cells per thread (16-byte stores) where rows are whole vectors
    if (g.n[0] % W == 0)
        cells_one<S, T, W><<<blocks, 32 * kRowsPerBlock, 0, s>>>(g, b);
    else
        cells_one<S, T, 1><<<blocks, 32 * kRowsPerBlock, 0, s>>>(g, b);
    if (g.n_surface > 0)
        surface_one<T><<<(g.n_surface + surf_points(g.dim) - 1) / surf_points(g.dim), kSurfThreads, 0, s>>>(g, b);
    return cudaGetLastError();
}

template <typename S, typename T>
cudaError_t batch_setup_impl(const BatchLat *lats, const BatchLat *d_lats, int count, cudaStream_t s) {
    constexpr int W = 16 / (int)sizeof(S);  // batches hold only rows of whole 16-byte vectors
    long long rows = 0;
    int points = 0;
    for (int i = 0; i < count; ++i) {
        const long long r = (long long)lats[i].g.n[1] * lats[i].g.n[2];
        rows = r > rows ? r : rows;
        points = lats[i].g.n_surface > points ? lats[i].g.n_surface : points;
    }
    constexpr int kMaxY = 32768;  // lattices per launch (grid y limit 65535)
    for (int i = 0; i < count; i += kMaxY) {
        const unsigned n = (unsigned)(count - i < kMaxY ? count - i : kMaxY);
        prepare_batch<S, T><<<dim3(4, n), 256, 0, s>>>(d_lats + i);
        cells_batch<S, T, W><<<dim3((unsigned)((rows + kRowsPerBlock - 1) / kRowsPerBlock), n), 32 * kRowsPerBlock, 0, s>>>(
            d_lats + i);
        if (points > 0) {
            const int P = surf_points(lats[0].g.dim);
            surface_batch<T><<<dim3((unsigned)((points + P - 1) / P), n), kSurfThreads, 0, s>>>(d_lats + i);
        }
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_setup(const Geometry &g, const Buffers &b, Prec p, cudaStream_t s) {
    switch (p) {
        case Prec::F64: return setup_impl<double, double>(g, b, s);
        case Prec::F16: return setup_impl<__half, float>(g, b, s);
        default: return setup_impl<float, float>(g, b, s);
    }
}

cudaError_t launch_batch_setup(Prec p, const BatchLat *lats, const BatchLat *d_lats, int count, cudaStream_t s) {
    switch (p) {
        case Prec::F64: return batch_setup_impl<double, double>(lats, d_lats, count, s);
        case Prec::F16: return batch_setup_impl<__half, float>(lats, d_lats, count, s);
        default: return batch_setup_impl<float, float>(lats, d_lats, count, s);
    }
}

}  // namespace wlb
