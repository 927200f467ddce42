// Several steps per launch for a single 2D lattice: overlapped tiles.
//
// A 2D lattice of 128^2 .. 600^2 cells stays in L2 and a step of it is a
// microsecond of work at most, so one launch per step is bound by launch
// latency and, with rows as the unit of work, by the few SMs that get a row
// block.  Here a CTA takes one tile of the lattice through k steps: step 1 reads
// the populations of the tile and of a halo of k - 1 cells (plus the cells they
// pull from) from global memory, the later steps ping-pong in shared memory
// over a box that shrinks by one cell per side and step, and step k writes the
// tile.  The halo is recomputed by every tile that needs it, so no CTA waits
// for another, and the arithmetic per cell and step is that of the one-step
// kernels: the same bits for any tiling.
//
// Sampled launches add sampler CTAs: each takes a run of consecutive surface
// points, i.e. a short arc of the circle, through the same k steps on the small
// box its stencils need, keeps rho1 and J1 of every step in shared memory and
// adds the points' sums, four lanes per point, in the order the one-step
// kernels add them.  They recompute the box and write only the sums, so the
// points of a small object spread over many SMs and no tile waits for them.
//
// FP64 lattices are bound by the FP64 pipe (about two instructions per clock
// and SM): tiles spread the lattice over all SMs and box cells are numbered
// linearly so that warps are full.  Figures beside the planner below.
#include "wlb_box_2d.cuh"

namespace wlb {
namespace {

constexpr int kThreads = 512;   // a box cell each, so that latency is paid about once per step

template <typename S>
struct TileArgs {
    using R = typename Store<S>::R;
    const S *A;  // state t
    S *B;        // state t + k
    const uint8_t *cls;
    const R *c2f;
    int nx, ny;
    long long ncell;
    int tx, ty, tiles_x, tiles, k;
    int n_surface, group, samplers;  // points, points per sampler CTA, sampler CTAs (the first blocks)
    Circle circle;                  // of the surface points
    const int4 *st_xyz;
    const R *st_w, *nrm;
    R *acc;
    R one;                          // 1 (collide_2d)
    R phi;                          // driven cavity: wall damping,
    int axis;                       // wave axis
    R rho_src[kMaxTileSteps];       // and the source sheet's rho1 at every step
};

// Dynamic shared memory of a box of w x h cells (the halo included): two states
// of five populations, c^2, the driven cavity's classes and, for samplers, the
// moments of two steps; plus the wrapped columns and rows.
template <typename R>
__host__ __device__ inline size_t box_smem(int w, int h, bool sampler, bool driven) {
    const size_t area = (size_t)w * h;
    return (sampler ? 17 : 11) * area * sizeof(R) + (size_t)(w + h) * sizeof(int) + (driven ? area : 0);
}

template <typename S, bool DRIVEN, bool SAMPLE>
__global__ void __launch_bounds__(kThreads) tile_steps_2d(TileArgs<S> P) {
    using R = typename Store<S>::R;
    extern __shared__ __align__(16) unsigned char tile_raw[];
    __shared__ int s_box[4];
    const int tid = threadIdx.x, nx = P.nx, ny = P.ny, k = P.k, H = k - 1;
    const bool sampler = SAMPLE && (int)blockIdx.x < P.samplers;
    const int tile = (int)blockIdx.x - (SAMPLE ? P.samplers : 0);
    // the cells this CTA needs after the last step: the tile, or the stencils of
    // the sampler's points
    int x0, y0, tw, th;
    if (sampler) {
        if (tid < 32) {
            const int p0 = (int)blockIdx.x * P.group;
            arc_box(p0, min(P.n_surface, p0 + P.group), P.n_surface, P.circle, tid, s_box);
        }
        __syncthreads();
        x0 = s_box[0];
        y0 = s_box[1];
        tw = s_box[2] - x0 + 1;
        th = s_box[3] - y0 + 1;
    } else {
        x0 = (tile % P.tiles_x) * P.tx;
        y0 = (tile / P.tiles_x) * P.ty;
        tw = min(P.tx, nx - x0);
        th = min(P.ty, ny - y0);
    }
    const int w0 = tw + 2 * H, h0 = th + 2 * H, area = w0 * h0;
    R *buf = reinterpret_cast<R *>(tile_raw);  // [2][5][area]
    R *c2s = buf + 10 * (size_t)area;          // [area]
    R *mom = c2s + area;                       // [2][rho, Jx, Jy][area], samplers
    int *xs = reinterpret_cast<int *>(mom + (sampler ? 6 * (size_t)area : 0));  // wrapped columns of the box
    int *ys = xs + w0;                                                         // and rows
    uint8_t *kcl = reinterpret_cast<uint8_t *>(ys + h0);                       // [area], driven
    for (int i = tid; i < w0 + h0; i += kThreads) {
        const bool col = i < w0;
        const int n = col ? nx : ny;
        int v = (col ? x0 + i : y0 + i - w0) - H;
        v %= n;
        xs[i] = v < 0 ? v + n : v;
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    Drive<R> drv;
    drv.phi = P.phi;
    drv.axis = P.axis;
    // one cell of step s: collide, leave the moments (samplers) and the result
    // in shared memory, or in global memory after the last step
    auto cell = [&](int s, int lx, int ly, const R (&f)[5], R c2, unsigned kc) {
        const int c = ly * w0 + lx;
        if (SAMPLE && sampler) {
            R *m = mom + (size_t)(s & 1) * 3 * area + c;
            m[area] = minus(f[1], f[2], P.one);
            m[2 * (size_t)area] = minus(f[3], f[4], P.one);
        }
        R o[5];
        const R rho = collide_2d<R>(c2, f, o, P.one);
        if (SAMPLE && sampler) mom[(size_t)(s & 1) * 3 * area + c] = rho;
        if (DRIVEN && kc >= CELL_WALL_LO) {
            drv.rho_src = P.rho_src[s];
            boundary_cell<R, 5>(kc, f, c2, drv, o);
        }
        if (s == k - 1) {
            if (!SAMPLE || !sampler) {
                const long long id = (long long)ys[ly] * nx + xs[lx];
#pragma unroll
                for (int i = 0; i < 5; ++i) Store<S>::put(P.B + i * P.ncell + id, o[i]);
            }
        } else {
            R *d = buf + (size_t)(s & 1) * 5 * area + c;
#pragma unroll
            for (int i = 0; i < 5; ++i) d[i * (size_t)area] = as_stored<S>(o[i]);
        }
    };
    // step 1 from global memory
    {
        const unsigned magic = divide_magic(w0);
#pragma unroll 1  // about one round; the registers of more keep the next launch's CTAs off the SM (0.78 -> 0.70 us)
        for (int i = tid; i < area; i += kThreads) {
            const int ly = divide(i, w0, magic), lx = i - ly * w0;
            const int x = xs[lx], y = ys[ly];
            const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
            const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
            const long long row = (long long)y * nx;
            R f[5];
            f[0] = Store<S>::get(P.A + row + x);
            f[1] = Store<S>::get(P.A + P.ncell + row + xm);
            f[2] = Store<S>::get(P.A + 2 * P.ncell + row + xp);
            f[3] = Store<S>::get(P.A + 3 * P.ncell + (long long)ym * nx + x);
            f[4] = Store<S>::get(P.A + 4 * P.ncell + (long long)yp * nx + x);
            const R c2 = P.c2f[row + x];
            unsigned kc = 0;
            if (DRIVEN) {
                kc = P.cls[row + x];
                kcl[i] = (uint8_t)kc;
            }
            c2s[i] = c2;
            cell(0, lx, ly, f, c2, kc);
        }
    }
    // Not before this grid has its input: a grid that waits behind a waiting one
    // takes SMs' slots early and lands unevenly, two CTAs on SMs that have few
    // (192^2 FP32 0.73 -> 0.60 us per step, sampled 1.06 -> 0.79).
    asm volatile("griddepcontrol.launch_dependents;");
    // A sampler's points, in the last warps: the box's cells keep the first ones busy.
    const int rt = kThreads - 1 - tid, p0 = (int)blockIdx.x * P.group;
    const int n = sampler ? min(P.group, P.n_surface - p0) : 0;
    const bool warp_on = (rt >> 5) * 8 < n;  // whole warps sample (the shuffles)
    const bool own = (rt >> 2) < n;
    PointQuad<R> pt;
    if (SAMPLE && warp_on)
        pt.load(p0 + (own ? rt >> 2 : 0), 3 - (rt & 3), P.st_xyz, P.st_w, P.nrm, P.acc, x0, y0, tw, th, nx, ny, H, w0);
    auto sample = [&](int s) { pt.add(mom + (size_t)(s & 1) * 3 * area, area, w0, P.one); };
    __syncthreads();
    for (int s = 1; s < k; ++s) {
        if (SAMPLE && warp_on) sample(s - 1);
        const R *cur = buf + (size_t)((s - 1) & 1) * 5 * area;
        const int ws = w0 - 2 * s, nc = ws * (h0 - 2 * s);
        const unsigned magic = divide_magic(ws);
#pragma unroll 1  // one or two rounds: unrolled code only costs registers and branches
        for (int i = tid; i < nc; i += kThreads) {
            const int q = divide(i, ws, magic), lx = i - q * ws + s, ly = q + s;
            const int c = ly * w0 + lx;
            R f[5];
            f[0] = cur[c];
            f[1] = cur[(size_t)area + c - 1];
            f[2] = cur[2 * (size_t)area + c + 1];
            f[3] = cur[3 * (size_t)area + c - w0];
            f[4] = cur[4 * (size_t)area + c + w0];
            cell(s, lx, ly, f, c2s[c], DRIVEN ? kcl[c] : 0u);
        }
        if (SAMPLE || s < k - 1) __syncthreads();
    }
    if (SAMPLE && warp_on) {
        sample(k - 1);
        if (own) P.acc[5 * (long long)(p0 + (rt >> 2)) + pt.comp] = pt.acc;
    }
}

// ---------------------------------------------------------------- host side: plans and launches

// The shared-memory limit belongs to the kernel and is shared by every handle:
// set to the device's opt-in maximum.
template <typename S, bool DRIVEN, bool SAMPLE>
cudaError_t allow_smem() {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, tile_steps_2d<S, DRIVEN, SAMPLE>);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tile_steps_2d<S, DRIVEN, SAMPLE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes);
    return e;
}

// What a step of the one-step kernels takes, in SM cycles (from measured steps
// of 128^2 .. 4096^2 lattices): a launch, and the cells at the rate of HBM / L2 or
// of the FP64 pipe, which row blocks of 8 rows (256 cells without whole-row
// warps) spread over few SMs on small lattices; sampled steps add their points.
template <typename S>
double one_step_cost(const Geometry &g, Prec p, bool sample, int sms) {
    const bool rows = update_is_vectorised(g, p);
    const double cells = (double)g.ncell;
    double c;
    if (p == Prec::F64) {
        const double block = rows ? 8.0 * g.n[0] : 256.0;
        c = 1500.0 + std::fmax(0.05 * cells, std::ceil(cells / block / sms) * block * 9.3);
        return c + (sample ? 2300.0 + 6.0 * g.n_surface : 0.0);
    }
    c = 1500.0 + std::fmax((p == Prec::F16 && rows ? 0.0071 : 0.0123) * cells, 1300.0);
    return c + (sample ? 3500.0 : 0.0);
}

// Tile and steps per launch by estimated time per step, in SM cycles: per launch
// 400, per wave of resident CTAs 2200 (first loads) and 260 per step (a barrier
// and a dependent chain), and the box cells of all steps at the rate of the
// arithmetic (FP64: 11 operations at about 1.4 per clock and SM) or of shared
// memory (FP32, FP16); sampler CTAs count as tiles of their own box and points.
// Candidates: m x n tiles for every m and about one, two, three ... tiles per SM.
// k = 0 where one step per launch is estimated faster (large FP64 lattices, which
// the FP64 pipe bounds either way, and large FP16 ones).  Measured (us per step,
// one step per launch -> tiles; unsampled, sampled with N points):
//   128^2 FP64, N = 64      5.4 -> 1.17    6.6 -> 1.49    (3 steps, 16 x 7 cells)
//   64 x 203 driven FP64    7.7 -> 1.79    9.1 -> 1.91    (4 steps, 8 x 11)
//   192^2 FP32, N = 1000    1.5 -> 0.60    3.5 -> 0.79    (8 steps, 16 x 16)
//   256^2 FP16, N = 200     2.1 -> 0.68    2.6 -> 0.84
//   600^2 FP32, N = 500     3.3 -> 1.62    5.4 -> 1.92
//   4096^2 FP32             111 -> 75-81                  (4 steps, 70 x 57)
template <typename S>
TilePlan2D plan_for(const Geometry &g, Prec p, bool sample, int sms, size_t smem_max) {
    using R = typename Store<S>::R;
    constexpr bool kDouble = sizeof(R) == 8;
    const double per_cell = kDouble ? 8.0 : (sizeof(S) == 2 ? 1.1 : 0.95);
    const double per_point = kDouble ? 60.0 : 6.0;
    const int nx = g.n[0], ny = g.n[1];
    if (sample && !boxes_fit(g)) return TilePlan2D{};
    const int group = sample ? sampler_group<S>(g) : 0;
    const int samplers = sample ? (g.n_surface + group - 1) / group : 0;
    auto box_cells = [](int w, int h, int k) {
        double c = 0;
        for (int s = 0; s < k; ++s) c += (double)(w + 2 * s) * (h + 2 * s);
        return c;
    };
    TilePlan2D best;
    double best_cost = 0.0;
    int last_tx = 0;
    for (int m = 1; m <= nx; ++m) {
        const int tx = (nx + m - 1) / m;
        if (tx == last_tx || tx > 128) continue;
        if (tx < 8 && m > 1) break;
        last_tx = tx;
        int last_ty = 0;
        for (long long r = 1; r <= 4096; r = r < 4 ? r + 1 : r + r / 2) {
            // samplers take SMs of their own while they are few
            const long long spare = samplers < sms / 2 ? sms - samplers : sms;
            long long n = ((r - 1) * sms + spare) / m;
            n = n < 1 ? 1 : (n > ny ? ny : n);
            const int ty = (int)((ny + n - 1) / n);
            if (ty == last_ty || ty > 128) continue;
            if (ty < 4 && n > 1) break;
            last_ty = ty;
            const long long tiles = (long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
            for (int k = 1; k <= kMaxTileSteps; k = k < 4 ? k + 1 : k + 2) {
                const int H = k - 1;
                size_t smem = box_smem<R>(tx + 2 * H, ty + 2 * H, false, g.driven != 0);
                if (sample) {
                    const int b = sampler_box<R>() + 2 * H;
                    const size_t sb = box_smem<R>(b, b, true, g.driven != 0);
                    smem = sb > smem ? sb : smem;
                }
                if (smem > smem_max || (long long)(tx + 2 * H) * (ty + 2 * H) > 65535) break;  // box index division
                const double tile_c = box_cells(tx, ty, k) * per_cell;
                const double arc = sample ? std::fmin((double)max_arc<R>(), group * 6.283 * g.surface_radius / g.n_surface) : 0;
                const int bx = (int)arc + 4;
                const double samp_c = sample ? box_cells(bx, bx, k) * per_cell * 1.2 + k * (350.0 + group * per_point) : 0;
                const double work = (double)tiles + samplers * (samp_c > tile_c ? samp_c / tile_c : 1.0);
                const double per_sm = std::ceil(work / sms);
                int res = (int)(smem_max / smem);
                if (res > 4) res = 4;
                const double waves = std::ceil((double)(tiles + samplers) / ((double)sms * res));
                const double busy = std::fmax(per_sm * tile_c, samp_c);
                const double cost = (400.0 + waves * (2200.0 + 260.0 * k) + busy) / k;
                if (best.k == 0 || cost < best_cost) {
                    best_cost = cost;
                    best.k = k;
                    best.tx = tx;
                    best.ty = ty;
                    best.smem = smem;
                    best.group = group;
                }
            }
            if (n == ny) break;
        }
    }
    if (best_cost > one_step_cost<S>(g, p, sample, sms)) best.k = 0;
    // sampled FP64 steps of large lattices: no better than one step per launch
    // (600^2, N = 500: 15.7 us per step against 14.5 to 17.4 for tiles)
    if (kDouble && sample && g.ncell > 200000) best.k = 0;
    return best;
}

template <typename S>
cudaError_t launch_for(const Geometry &g, const Buffers &b, const TilePlan2D &pl, int src, bool sample, int k,
                       const double *rho_src, cudaStream_t s) {
    using R = typename Store<S>::R;
    TileArgs<S> a;
    a.A = (const S *)b.pop[src];
    a.B = (S *)b.pop[src ^ 1];
    a.cls = b.cls;
    a.c2f = (const R *)b.c2;
    a.nx = g.n[0];
    a.ny = g.n[1];
    a.ncell = g.ncell;
    a.tx = pl.tx;
    a.ty = pl.ty;
    a.tiles_x = (g.n[0] + pl.tx - 1) / pl.tx;
    a.tiles = a.tiles_x * ((g.n[1] + pl.ty - 1) / pl.ty);
    a.k = k;
    a.n_surface = g.n_surface;
    a.group = pl.group;
    a.samplers = sample ? tile_samplers(g, pl) : 0;
    a.circle = circle_of(g);
    a.st_xyz = b.st_xyz;
    a.st_w = (const R *)b.st_w;
    a.nrm = (const R *)b.nrm;
    a.acc = (R *)b.acc;
    a.one = R(1);
    a.phi = (R)g.wall_damping;
    a.axis = g.wave_axis;
    for (int i = 0; i < kMaxTileSteps; ++i) a.rho_src[i] = i < k ? (R)rho_src[i] : R(0);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.tiles + a.samplers));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = pl.smem;  // of the plan's k: enough for any fewer
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (g.driven)
        return sample ? cudaLaunchKernelEx(&cfg, tile_steps_2d<S, true, true>, a)
                      : cudaLaunchKernelEx(&cfg, tile_steps_2d<S, true, false>, a);
    return sample ? cudaLaunchKernelEx(&cfg, tile_steps_2d<S, false, true>, a)
                  : cudaLaunchKernelEx(&cfg, tile_steps_2d<S, false, false>, a);
}

template <typename S>
cudaError_t plan_both(const Geometry &g, Prec p, int sms, size_t smem_max, TilePlan2D *out) {
    for (int sample = 0; sample < 2; ++sample) {
        if (sample && g.n_surface == 0) continue;
        out[sample] = plan_for<S>(g, p, sample != 0, sms, smem_max);
        if (out[sample].k == 0) continue;
        cudaError_t e = g.driven ? (sample ? allow_smem<S, true, true>() : allow_smem<S, true, false>())
                                 : (sample ? allow_smem<S, false, true>() : allow_smem<S, false, false>());
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t plan_tile_2d(const Geometry &g, Prec p, TilePlan2D out[2]) {
    out[0] = out[1] = TilePlan2D{};
    if (g.dim != 2) return cudaSuccess;
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const size_t smem_max = (size_t)optin - 1024;
    switch (p) {
        case Prec::F64: return plan_both<double>(g, p, sms, smem_max, out);
        case Prec::F16: return plan_both<__half>(g, p, sms, smem_max, out);
        default: return plan_both<float>(g, p, sms, smem_max, out);
    }
}

cudaError_t launch_tile_2d(const Geometry &g, const Buffers &b, Prec p, const TilePlan2D &pl, int src, bool sample,
                           int k, long long t_mod, cudaStream_t s) {
    double rho_src[kMaxTileSteps];
    for (int i = 0; i < k; ++i) rho_src[i] = source_density(g, (t_mod + i) % g.period);
    switch (p) {
        case Prec::F64: return launch_for<double>(g, b, pl, src, sample, k, rho_src, s);
        case Prec::F16: return launch_for<__half>(g, b, pl, src, sample, k, rho_src, s);
        default: return launch_for<float>(g, b, pl, src, sample, k, rho_src, s);
    }
}

}  // namespace wlb
