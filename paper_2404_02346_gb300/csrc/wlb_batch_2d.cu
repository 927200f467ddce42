// Several steps per launch for batches of 2D lattices (D2Q5, periodic, FP32 or
// FP16): row sweeps of four to eight steps, and box samplers.
//
// Many lattices together are far larger than L2, so every launch streams all
// populations through HBM and the bound is bytes per step: K steps per launch
// cost 40 / K bytes per cell and step (FP32: five populations read and written;
// c^2 near the object comes on top).  A warp owns a chunk of whole rows of one lattice and sweeps it
// once with K time levels in flight: when row p of step 1 is computed from the
// staged populations, step l is computed on row p - l + 1 from the registers
// that hold the previous rows of step l - 1.  Per level and cell that is five
// values (rest, +x and -x of row p - l, +y of rows p - l and p - l - 1); -y comes
// straight from the level above.  The K - 1 rows on either side of a chunk are
// recomputed by the neighbour's warp, so no warp waits for another.
//
// A lane owns C consecutive cells of the row, so that one shuffle per direction
// and level moves a row by one cell; rows of C V cells wrap around by the
// shuffle's lane, others are staged with a halo of at least K columns on either
// side, for every step spoils one more column from the ends of the staged row, and
// their results are dropped.  Rows travel through shared memory: 16-byte
// asynchronous copies in (kDepth rows ahead, c^2 kept for all levels), 16-byte
// streaming stores out.
//
// Every step rounds its result to the storage type as a stored state would be
// and the arithmetic per cell is that of the one-step kernels: the same bits.
//
// 512 lattices of 192 x 192 cells, FP32, six steps per launch: 132 us per launch,
// 0.76 GB of HBM traffic (0.84 of the copy rate), against 3 x 155 us for two steps
// per launch; the samplers of 1000 points per lattice 107 us per launch against
// 3 x 100 us for one thread per point with the steps recomputed per stencil cell.
#include <algorithm>
#include <map>
#include <type_traits>

#include "wlb_box_2d.cuh"

namespace wlb {
namespace {

constexpr int kDepth = 2;       // rows of populations staged ahead
constexpr int kMaxSteps = 8;
constexpr int kMaxRows = 128;   // rows per warp chunk
constexpr int kMinRows = 8;
constexpr long long kMaxLaunches = 1ll << 28;  // of a run: launch and step-in-period numbers fit 32 bits
constexpr int kBoxThreads = 256;

// Steps per launch of rows with C cells per lane: about as many as 255 registers
// hold (5 C values per level), an even number.  Batches, ms per run with 4, 6, 8
// steps: 300 x 128^2 (C = 4) 15.0, 10.6, 8.8; 512 x 192^2 (6) 86, 61, 129 (spills);
// 200 x 208^2 (7) 29.8, 20.6, 53; FP16 40 x 224^2 (8) 8.3, 11.9, 43.
__host__ __device__ constexpr int steps_for(int c) { return c <= 4 ? 8 : (c <= 7 ? 6 : 4); }
// Rows of c^2 kept: kDepth ahead, steps - 1 behind.
__host__ __device__ constexpr int c2_rows(int c) { return c <= 4 ? 16 : 8; }
// Halo columns staged on either side of a row that its lanes do not cover exactly:
// at least a column per step, a whole number of 16-byte pieces.
__host__ __device__ constexpr int halo_for(int c, int w) { return (steps_for(c) + w - 1) / w * w; }

// Step t of a lattice at launch n and the steps of that launch: whole periods of
// launches of plan.nseg steps, the last one of a period shorter, so that a period's
// fold falls on a launch's end.
struct Turn {
    long long t;
    int pos, k;
};
__host__ __device__ inline long long launches_per_period(const BatchLat &L) {
    return (L.period + L.plan.nseg - 1) / L.plan.nseg;
}
__device__ __forceinline__ Turn turn_of(const BatchLat &L, int n) {
    const int per = (int)launches_per_period(L);
    const int p = n / per, pos = (n - p * per) * L.plan.nseg;
    Turn r;
    r.pos = pos;
    r.t = (long long)p * L.period + pos;
    r.k = (int)min((long long)L.plan.nseg, L.period - pos);
    return r;
}

// C consecutive values per lane, from and to shared memory, in the widest
// pieces their alignment allows (an odd stride of words has no bank conflicts).
template <int C>
__device__ __forceinline__ void ld_cells(const float *p, float (&v)[C]) {
    if constexpr (C % 4 == 0) {
#pragma unroll
        for (int e = 0; e < C; e += 4) {
            const float4 t = *reinterpret_cast<const float4 *>(p + e);
            v[e] = t.x; v[e + 1] = t.y; v[e + 2] = t.z; v[e + 3] = t.w;
        }
    } else if constexpr (C % 2 == 0) {
#pragma unroll
        for (int e = 0; e < C; e += 2) {
            const float2 t = *reinterpret_cast<const float2 *>(p + e);
            v[e] = t.x; v[e + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < C; ++e) v[e] = p[e];
    }
}
template <int C>
__device__ __forceinline__ void ld_cells(const __half *p, float (&v)[C]) {
#pragma unroll
    for (int e = 0; e < C; e += 2) {
        const float2 t = __half22float2(*reinterpret_cast<const __half2 *>(p + e));
        v[e] = t.x; v[e + 1] = t.y;
    }
}
template <int C>
__device__ __forceinline__ void st_cells(float *p, const float (&v)[C]) {
    if constexpr (C % 4 == 0) {
#pragma unroll
        for (int e = 0; e < C; e += 4) *reinterpret_cast<float4 *>(p + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    } else if constexpr (C % 2 == 0) {
#pragma unroll
        for (int e = 0; e < C; e += 2) *reinterpret_cast<float2 *>(p + e) = make_float2(v[e], v[e + 1]);
    } else {
#pragma unroll
        for (int e = 0; e < C; ++e) p[e] = v[e];
    }
}
template <int C>
__device__ __forceinline__ void st_cells(__half *p, const float (&v)[C]) {
#pragma unroll
    for (int e = 0; e < C; e += 2) *reinterpret_cast<__half2 *>(p + e) = __floats2half2_rn(v[e], v[e + 1]);
}

__device__ __forceinline__ void copy_in(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(__cvta_generic_to_global(src))
                 : "memory");
}
// Shared memory of a warp, in rows of 32 C cells.
template <typename S, int C>
struct RowBuf {
    S in[kDepth][5][32 * C];
    S out[5][32 * C];
    float c2[c2_rows(C)][32 * C];
};

// Of `rows` rows from row y0 on (periodic in ny): the range [n0, n1) outside which
// no row comes within `reach` rows of row c.
__device__ __forceinline__ void near_rows(int c, int reach, int ny, int y0, int rows, int &n0, int &n1) {
    n0 = 0;
    n1 = rows;
    if (rows > ny || 2 * reach + 1 >= ny) return;
    const int d = ((c - y0) % ny + ny) % ny;  // the first image at or above y0, the one below it and above it
    const bool below = d - ny + reach >= 0, own = d - reach < rows, above = d + ny - reach < rows;
    n0 = below ? 0 : (own ? max(0, d - reach) : (above ? d + ny - reach : rows));
    n1 = above ? rows : (own ? min(rows, d + reach + 1) : (below ? min(rows, d - ny + reach + 1) : 0));
}

// k = K steps of chunk rows [ya, yb) by one warp (warp-uniform flow).
template <typename S, int C, int K>
__device__ __forceinline__ void sweep(const BatchLat &L, int src, int chunk, int lane, RowBuf<S, C> &sm) {
    constexpr int W = 16 / (int)sizeof(S), CR = c2_rows(C);
    static_assert(K % 2 == 0 && CR >= K + kDepth && (CR & (CR - 1)) == 0, "rings");
    const int nx = L.g.n[0], ny = L.g.n[1], nc = (int)L.g.ncell;
    const int ya = chunk * L.plan.zc, yb = min(ny, ya + L.plan.zc);
    const bool exact = nx % C == 0 && nx / C <= 32;
    const int H = exact ? 0 : halo_for(C, W);  // halo columns staged on either side
    const int wl = nx + 2 * H;                 // staged row: at most 32 C cells
    const int V = exact ? nx / C : 32;
    const int left = lane == 0 ? V - 1 : lane - 1, right = lane == V - 1 ? 0 : (lane + 1) & 31;
    const S *__restrict__ A = (const S *)L.b.pop[src];
    S *__restrict__ B = (S *)L.b.pop[src ^ 1];
    const float *__restrict__ c2f = (const float *)L.b.c2;
    // this lane's 16-byte pieces of a staged row: wrapped column of each
    constexpr int PP = (32 * C / W + 31) / 32, PC = (8 * C + 31) / 32;  // per row of populations, of c^2
    int xp[PP], xc[PC];
#pragma unroll
    for (int j = 0; j < PP; ++j) {
        const int x = (j * 32 + lane) * W;
        xp[j] = x < wl ? ((x - H) % nx + nx) % nx : -1;
    }
#pragma unroll
    for (int j = 0; j < PC; ++j) {
        const int x = (j * 32 + lane) * 4;
        xc[j] = x < wl ? ((x - H) % nx + nx) % nx : -1;
    }
    // stage what step 1 of the it-th row reads: one commit group per row
    const int rows = yb - ya + 2 * (K - 1);
    // Rows farther from the centre than the interface band hold fluid cells only
    // and their c^2 is not read: FP32, 44 -> about 41 bytes per cell (512 x 192^2,
    // 1000 points: 60.7 -> 58.5 ms).  FP16 is bound by instructions (57.8 -> 59.4
    // ms), short rows by latency, and six levels of seven cells leave no registers.
    constexpr bool kSkip = sizeof(S) == 4 && C >= 4 && C * steps_for(C) < 40;
    const float c0sq = (float)(L.g.c0 * L.g.c0);
    int near0 = 0, near1 = rows;
    if (kSkip) near_rows(L.plan.ntile, L.plan.tx, ny, ya - (K - 1), rows, near0, near1);
    int ys = ((ya - (K - 1)) % ny + ny) % ny;  // row staged next
    auto stage = [&](int it) {
        if (it < rows) {
            const int r0 = ys * nx, rm = (ys == 0 ? ny - 1 : ys - 1) * nx, rp = (ys == ny - 1 ? 0 : ys + 1) * nx;
            S(*dst)[32 * C] = sm.in[it % kDepth];
#pragma unroll
            for (int j = 0; j < PP; ++j) {
                if (xp[j] < 0) continue;
                const int x = (j * 32 + lane) * W;
                copy_in(dst[0] + x, A + (r0 + xp[j]));
                copy_in(dst[1] + x, A + ((size_t)nc + r0 + xp[j]));
                copy_in(dst[2] + x, A + (2 * (size_t)nc + r0 + xp[j]));
                copy_in(dst[3] + x, A + (3 * (size_t)nc + rm + xp[j]));
                copy_in(dst[4] + x, A + (4 * (size_t)nc + rp + xp[j]));
            }
            float *c2 = sm.c2[it & (CR - 1)] + lane * 4;
            if (!kSkip || (it >= near0 && it < near1)) {
#pragma unroll
                for (int j = 0; j < PC; ++j)
                    if (xc[j] >= 0) copy_in(c2 + j * 128, c2f + (r0 + xc[j]));
            } else {
#pragma unroll
                for (int j = 0; j < PC; ++j)
                    if ((j * 32 + lane) * 4 < 32 * C)
                        *reinterpret_cast<float4 *>(c2 + j * 128) = make_float4(c0sq, c0sq, c0sq, c0sq);
            }
            ys = ys == ny - 1 ? 0 : ys + 1;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int d = 0; d < kDepth; ++d) stage(d);
    // level l (step l + 1) holds of step l + 1's input row: rest, +x, -x, and +y of
    // that row and the one before
    float h[K - 1][5][C];
#pragma unroll
    for (int l = 0; l < K - 1; ++l)
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int e = 0; e < C; ++e) h[l][i][e] = 0.0f;
    for (int it = 0; it < rows; ++it) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
        __syncwarp();
        float f[5][C];
        const S(*in)[32 * C] = sm.in[it % kDepth];
#pragma unroll
        for (int i = 0; i < 5; ++i) ld_cells<C>(in[i] + lane * C, f[i]);
        __syncwarp();
        stage(it + kDepth);  // the slot just read
#pragma unroll
        for (int l = 0; l < K; ++l) {
            float c2[C];
            ld_cells<C>(sm.c2[(it - l) & (CR - 1)] + lane * C, c2);
            const float fl = __shfl_sync(kFull, f[1][C - 1], left), fr = __shfl_sync(kFull, f[2][0], right);
            float o[5][C];
#pragma unroll
            for (int e = 0; e < C; ++e) {
                const float fin[5] = {f[0][e], e == 0 ? fl : f[1][e - 1], e == C - 1 ? fr : f[2][e + 1], f[3][e],
                                      f[4][e]};
                float t[5];
                collide_2d<float>(c2[e], fin, t);
#pragma unroll
                for (int i = 0; i < 5; ++i) o[i][e] = t[i];
            }
            if (l < K - 1) {
#pragma unroll
                for (int e = 0; e < C; ++e) {
                    f[0][e] = h[l][0][e];
                    f[1][e] = h[l][1][e];
                    f[2][e] = h[l][2][e];
                    f[3][e] = h[l][4][e];
                    f[4][e] = as_stored<S>(o[4][e]);
                    h[l][0][e] = as_stored<S>(o[0][e]);
                    h[l][1][e] = as_stored<S>(o[1][e]);
                    h[l][2][e] = as_stored<S>(o[2][e]);
                    h[l][4][e] = h[l][3][e];
                    h[l][3][e] = as_stored<S>(o[3][e]);
                }
            } else if (it >= 2 * (K - 1)) {  // row ya + it - 2 (K - 1) after the last step
                __syncwarp();  // the row before has been read
#pragma unroll
                for (int i = 0; i < 5; ++i) st_cells<C>(sm.out[i] + lane * C, o[i]);
                __syncwarp();
                S *row = B + (size_t)(ya + it - 2 * (K - 1)) * nx;
#pragma unroll
                for (int j = 0; j < PP; ++j) {
                    const int x = (j * 32 + lane) * W;
                    if (x >= nx) continue;
#pragma unroll
                    for (int i = 0; i < 5; ++i)
                        __stcs(reinterpret_cast<uint4 *>(row + (i * (size_t)nc + x)),
                               *reinterpret_cast<const uint4 *>(sm.out[i] + H + x));
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Block w (one warp: small blocks fill the SM's registers) sweeps chunk
// task0 + w - task_first[i] of lattice i.
template <typename S, int C>
__global__ void __launch_bounds__(32) batch_rows_2d(const BatchLat *__restrict__ lats,
                                                    const int *__restrict__ task_lat,
                                                    const int *__restrict__ task_first, int task0, int n) {
    extern __shared__ __align__(16) unsigned char raw[];
    constexpr int K = steps_for(C);
    const int task = task0 + (int)blockIdx.x, i = task_lat[task], lane = threadIdx.x;
    const BatchLat &L = lats[i];
    const Turn r = turn_of(L, n);
    if (r.t >= L.n_steps) return;
    RowBuf<S, C> &sm = *reinterpret_cast<RowBuf<S, C> *>(raw);
    const int chunk = task - task_first[i], src = n & 1;
    // a period's last launch takes the 2, 4 .. K steps that are left of it
    if (r.k == K) sweep<S, C, K>(L, src, chunk, lane, sm);
    else if (K > 6 && r.k == 6) sweep<S, C, (K > 6 ? 6 : 2)>(L, src, chunk, lane, sm);
    else if (K > 4 && r.k == 4) sweep<S, C, (K > 4 ? 4 : 2)>(L, src, chunk, lane, sm);
    else sweep<S, C, 2>(L, src, chunk, lane, sm);
}

// Shared memory of a sampler's largest box (the halo of k steps included): two
// states of five populations, c^2, the moments of two steps, wrapped columns and
// rows.
constexpr size_t box_bytes(int k) {
    const size_t b = sampler_box<float>() + 2 * (k - 1);
    return 17 * b * b * sizeof(float) + 2 * b * sizeof(int);
}

// Block groups i + j adds the sums of the launch's steps for the j-th group of points
// of lattice i: the steps on the small box the points' stencils need, as the
// sampler blocks of tile_steps_2d do, and the period's fold at its end.
template <typename S>
__global__ void __launch_bounds__(kBoxThreads) batch_sample_boxes_2d(const BatchLat *__restrict__ lats, int groups,
                                                                     int n) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ int s_box[4];
    const int lat = (int)blockIdx.x / groups;
    const BatchLat &L = lats[lat];
    const Turn r = turn_of(L, n);
    const int group = L.plan.H, np = L.g.n_surface, p0 = ((int)blockIdx.x - lat * groups) * group;
    if (r.t < L.window_begin || r.t >= L.n_steps || p0 >= np) return;
    const int tid = threadIdx.x, nx = L.g.n[0], ny = L.g.n[1], k = r.k, H = k - 1;
    const size_t nc = (size_t)L.g.ncell;
    const S *__restrict__ A = (const S *)L.b.pop[n & 1];
    const float *__restrict__ c2f = (const float *)L.b.c2;
    if (tid < 32) arc_box(p0, min(np, p0 + group), np, L.circle, tid, s_box);
    __syncthreads();
    const int x0 = s_box[0], y0 = s_box[1], tw = s_box[2] - x0 + 1, th = s_box[3] - y0 + 1;
    const int w0 = tw + 2 * H, h0 = th + 2 * H, area = w0 * h0;
    float *buf = reinterpret_cast<float *>(raw);  // [2][5][area]
    float *c2s = buf + 10 * area;                 // [area]
    float *mom = c2s + area;                      // [2][rho, Jx, Jy][area]
    int *xs = reinterpret_cast<int *>(mom + 6 * area), *ys = xs + w0;
    for (int i = tid; i < w0 + h0; i += kBoxThreads) {
        const bool col = i < w0;
        const int m = col ? nx : ny;
        int v = (col ? x0 + i : y0 + i - w0) - H;
        v %= m;
        xs[i] = v < 0 ? v + m : v;
    }
    __syncthreads();
    auto cell = [&](int s, int c, const float (&f)[5], float c2) {
        float *m = mom + (s & 1) * 3 * area + c, o[5];
        m[area] = sub_rn(f[1], f[2]);
        m[2 * area] = sub_rn(f[3], f[4]);
        m[0] = collide_2d<float>(c2, f, o);
        if (s < k - 1) {
            float *d = buf + (s & 1) * 5 * area + c;
#pragma unroll
            for (int i = 0; i < 5; ++i) d[i * area] = as_stored<S>(o[i]);
        }
    };
    {
        const unsigned magic = divide_magic(w0);
        for (int i = tid; i < area; i += kBoxThreads) {
            const int ly = divide(i, w0, magic), lx = i - ly * w0, x = xs[lx], y = ys[ly];
            const int xm = x == 0 ? nx - 1 : x - 1, xq = x == nx - 1 ? 0 : x + 1;
            const int ym = y == 0 ? ny - 1 : y - 1, yq = y == ny - 1 ? 0 : y + 1;
            const int row = y * nx;
            float f[5];
            f[0] = Store<S>::get(A + row + x);
            f[1] = Store<S>::get(A + nc + row + xm);
            f[2] = Store<S>::get(A + 2 * nc + row + xq);
            f[3] = Store<S>::get(A + 3 * nc + ym * nx + x);
            f[4] = Store<S>::get(A + 4 * nc + yq * nx + x);
            const float c2 = c2f[row + x];
            c2s[i] = c2;
            cell(0, i, f, c2);
        }
    }
    const int rt = kBoxThreads - 1 - tid, m = min(group, np - p0);
    const bool warp_on = (rt >> 5) * 8 < m;  // whole warps sample (the shuffles)
    const int p = p0 + ((rt >> 2) < m ? rt >> 2 : 0);
    PointQuad<float> pt;
    if (warp_on)
        pt.load(p, 3 - (rt & 3), L.b.st_xyz, (const float *)L.b.st_w, (const float *)L.b.nrm, (const float *)L.b.acc,
                x0, y0, tw, th, nx, ny, H, w0);
    __syncthreads();
    for (int s = 1; s < k; ++s) {
        if (warp_on) pt.add(mom + ((s - 1) & 1) * 3 * area, area, w0);
        const float *cur = buf + ((s - 1) & 1) * 5 * area;
        const int ws = w0 - 2 * s, cells = ws * (h0 - 2 * s);
        const unsigned magic = divide_magic(ws);
        for (int i = tid; i < cells; i += kBoxThreads) {
            const int q = divide(i, ws, magic), c = (q + s) * w0 + i - q * ws + s;
            const float f[5] = {cur[c], cur[area + c - 1], cur[2 * area + c + 1], cur[3 * area + c - w0],
                                cur[4 * area + c + w0]};
            cell(s, c, f, c2s[c]);
        }
        __syncthreads();
    }
    if (!warp_on) return;
    pt.add(mom + ((k - 1) & 1) * 3 * area, area, w0);
    if ((rt >> 2) >= m) return;
    float *a = (float *)L.b.acc + 5 * (size_t)p + pt.comp;
    if (r.pos + k < L.period) {
        *a = pt.acc;
    } else {  // the fold of batch_sample
        double *a64 = L.b.acc64 + 5 * (size_t)p + pt.comp;
        const double v = fold_value(*a64, (double)pt.acc, 1.0 / (L.g.pop_scale * L.g.pop_scale));
        *a64 = v;
        *a = 0.0f;
        if (!isfinite(v)) atomicExch(L.b.err, 1);
    }
}

// ---------------------------------------------------------------- host side: plans and launches

// Cells per lane for rows of nx cells: the fewest that cover the row exactly or
// with its halo (FP16: whole half2 pairs); 0 if more than eight are needed.
template <typename S>
int cells_per_lane(int nx) {
    constexpr int W = 16 / (int)sizeof(S), step = sizeof(S) == 2 ? 2 : 1;
    if (nx % W) return 0;
    for (int c = 2; c <= 8; c += step)
        if ((nx % c == 0 && nx / c <= 32) || nx + 2 * halo_for(c, W) <= 32 * c) return c;
    return 0;
}

// f(integral constant C) for the C of a group.
template <typename S, typename F>
cudaError_t with_cells(int c, F f) {
    switch (c) {
        case 2: return f(std::integral_constant<int, 2>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 8: return f(std::integral_constant<int, 8>{});
        default: break;
    }
    if constexpr (sizeof(S) == 4) {
        switch (c) {
            case 3: return f(std::integral_constant<int, 3>{});
            case 5: return f(std::integral_constant<int, 5>{});
            case 7: return f(std::integral_constant<int, 7>{});
            default: break;
        }
    }
    return cudaErrorInvalidValue;
}

// Sampler blocks of a planned lattice.
int box_groups(const BatchLat &L) { return (L.g.n_surface + L.plan.H - 1) / L.plan.H; }

template <typename S>
bool plan_for(BatchLat *lats, int count, int rows_fixed) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    double slots[9] = {0};  // warps of the launch that the device holds
    std::map<int, long long> heights[9];  // lattices by height: an ensemble has few (512 of one: 0.2 ms less to create)
    for (int i = 0; i < count; ++i) {
        const Geometry &g = lats[i].g;
        if (g.dim != 2 || g.driven || g.ncell > (1ll << 28) || !boxes_fit(g)) return false;
        const int c = cells_per_lane<S>(g.n[0]);
        if (c == 0) return false;
        ++heights[c][g.n[1]];
        lats[i].plan = TwoStepPlan{};
        lats[i].plan.chunks_per_lane = c;
        lats[i].plan.threads = 32;
        lats[i].plan.nslab = 1;
        lats[i].plan.nseg = steps_for(c);
        if (lats[i].n_steps / lats[i].period > kMaxLaunches / launches_per_period(lats[i])) return false;
        lats[i].plan.H = sampler_group<S>(g);
        lats[i].circle = circle_of(g);
        // the object's centre row and the rows to either side that it and its
        // interface band can reach (two more for rounding)
        const double cy = g.center[1] - g.n[1] * std::floor(g.center[1] / g.n[1]);
        lats[i].plan.ntile = cy >= 0.0 && cy < g.n[1] ? (int)cy : 0;
        const double reach = std::sqrt(g.radius * g.radius + g.band_half) + 2.0;
        lats[i].plan.tx = std::fabs(g.center[1]) < 1e9 && reach < g.n[1] ? (int)reach + 1 : g.n[1];
        if ((long long)count * box_groups(lats[i]) > 0x7fffffffll) return false;  // blocks of the sampler launch
    }
    int zc[9] = {0};
    for (int c = 2; c <= 8; ++c) {
        if (heights[c].empty()) continue;
        int bps = 0;
        cudaError_t e = with_cells<S>(c, [&](auto cc) {
            constexpr int C = decltype(cc)::value;
            const size_t smem = sizeof(RowBuf<S, C>);
            cudaError_t e2 = cudaFuncSetAttribute(batch_rows_2d<S, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  (int)smem);
            return e2 != cudaSuccess ? e2 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, batch_rows_2d<S, C>,
                                                                                          32, smem);
        });
        if (e != cudaSuccess || bps == 0) return false;
        slots[c] = (double)sms * bps;
        int rows = rows_fixed;
        if (rows <= 0) {
            double best = 0;
            for (int z = kMaxRows; z >= kMinRows; --z) {
                long long t = 0;
                int tall = 0;  // rows of the longest chunk
                for (const auto &[ny, lattices] : heights[c]) {
                    const int n = (ny + z - 1) / z;
                    t += n * lattices;
                    tall = std::max(tall, (ny + n - 1) / n);
                }
                const double cost = std::ceil((double)t / slots[c]) * (tall + 2 * (steps_for(c) - 1) + 2);
                if (rows <= 0 || cost < best) {
                    best = cost;
                    rows = z;
                }
            }
        }
        zc[c] = rows;
    }
    if (cudaFuncSetAttribute(batch_sample_boxes_2d<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)box_bytes(kMaxSteps)) != cudaSuccess)
        return false;
    for (int i = 0; i < count; ++i) {
        TwoStepPlan &pl = lats[i].plan;
        const int ny = lats[i].g.n[1], z = zc[pl.chunks_per_lane];
        pl.chunks = (ny + z - 1) / z;
        pl.zc = (ny + pl.chunks - 1) / pl.chunks;
        pl.chunks = (ny + pl.zc - 1) / pl.zc;
    }
    return true;
}

template <typename S>
cudaError_t launch_for(const BatchTwoGroup *groups, int ngroups, const BatchLat *lats, const int *task_lat,
                       const int *task_first, int count, int sample_groups, int sample_steps, int n, cudaStream_t s) {
    if (sample_groups > 0) {
        const size_t smem = box_bytes(sample_steps);
        batch_sample_boxes_2d<S><<<(unsigned)count * (unsigned)sample_groups, kBoxThreads, smem, s>>>(
            lats, sample_groups, n);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < ngroups; ++k) {
        const BatchTwoGroup &g = groups[k];
        cudaError_t e = with_cells<S>(g.ch, [&](auto cc) {
            constexpr int C = decltype(cc)::value;
            batch_rows_2d<S, C><<<g.ctas, 32, sizeof(RowBuf<S, C>), s>>>(lats, task_lat, task_first, g.cta_begin, n);
            return cudaGetLastError();
        });
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

bool plan_batch2d_rows(Prec p, BatchLat *lats, int count, int rows, BatchTwoGroup *groups, int *ngroups) {
    if (p == Prec::F64) return false;
    if (!(p == Prec::F16 ? plan_for<__half>(lats, count, rows) : plan_for<float>(lats, count, rows))) return false;
    int used = 0;
    for (int c = 2; c <= 8; ++c)
        for (int i = 0; i < count; ++i)
            if (lats[i].plan.chunks_per_lane == c) {
                groups[used] = BatchTwoGroup{};
                groups[used++].ch = c;
                break;
            }
    *ngroups = used;
    return true;
}

BatchTurns batch2d_turns(const BatchLat *lats, int count) {
    BatchTurns r;
    r.first_sampled = 0x7fffffff;
    for (int i = 0; i < count; ++i) {
        const BatchLat &L = lats[i];
        const long long per = launches_per_period(L);
        r.launches = std::max(r.launches, (int)(L.n_steps / L.period * per));
        if (L.window_begin < L.n_steps && L.g.n_surface > 0) {
            r.first_sampled = std::min(r.first_sampled, (int)(L.window_begin / L.period * per));
            r.groups = std::max(r.groups, box_groups(L));
            r.steps = std::max(r.steps, L.plan.nseg);
        }
    }
    return r;
}

long long batch2d_steps_taken(const BatchLat &L, int n) {
    const long long per = launches_per_period(L);
    const long long t = n / per * L.period + std::min(L.period, n % per * L.plan.nseg);
    return std::min(L.n_steps, t);
}

cudaError_t launch_batch2d_rows(Prec p, const BatchTwoGroup *groups, int ngroups, const BatchLat *lats,
                                const int *task_lat, const int *task_first, int count, const BatchTurns &turns, int n,
                                cudaStream_t s) {
    const int sample = n >= turns.first_sampled ? turns.groups : 0;
    return p == Prec::F16 ? launch_for<__half>(groups, ngroups, lats, task_lat, task_first, count, sample, turns.steps, n, s)
                          : launch_for<float>(groups, ngroups, lats, task_lat, task_first, count, sample, turns.steps,
                                              n, s);
}

}  // namespace wlb
