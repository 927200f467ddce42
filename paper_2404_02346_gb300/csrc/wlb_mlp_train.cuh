// One training step of the surrogate network in two launches (included by
// wlb_mlp.cu, inside its anonymous namespace).
//
//   train_tiles    one CTA per NB samples: forward, loss and the activation
//                  gradients of all layers on the chip;
//   train_weights  one CTA per 128 x 16 tile of a weight gradient, which then
//                  applies Adam to its tile and writes the tile's BF16 copy.
//
// A batch of 512 is 0.4 GFLOP: what bounds a step is the chain of layers and
// launches, not the tensor cores.  One GEMM launch per product on B / 128
// CTAs, each thread writing whole rows of strided activations, took 690 us
// per step of 512 samples (28-85 us per launch, 4 CTAs busy); these two
// launches take the products of the same operands in the same K order (the
// weight gradients keep their bits) in 19.7 us.  Of that (one CTA's clock),
// train_tiles takes 12 us: per layer about 1.1 us of products (65 cycles per
// M = 128, N = 16 instruction: reading the weights from shared memory bounds
// it) and 0.7 us until the next operand is ready; train_weights takes 5 us,
// 3.5 of them loading the operands and 1.5 Adam.
//
// Transposed products.  train_tiles computes D^T = W . H^T: M = 256 features
// (two tcgen05.mma of M = 128), N = NB samples, so a batch of 512 spreads over
// 32 CTAs.  TMEM lane f of half h is feature 128 h + f, so a thread owns one
// feature of every layer for its NB samples: it keeps GELU' of its own
// pre-activations in registers for the way back (no Z goes to memory;
// GELU' is evaluated while the next layer's product runs), and its NB
// consecutive samples are 16-byte pieces both of the next product's B operand
// in shared memory (MN-major core matrices) and of the batch-contiguous copies
// that the weight and bias gradients read.
//
// Weights are kept packed in 8 x 8 core matrices, element (o, i) of a 256 x
// 256 layer at (o / 8) 4096 + (i / 8) 128 + (o % 8) 16 + (i % 8) 2: read
// K-major (K = i) it is W for the forward product, read MN-major (M = i, K =
// o) it is W^T for the backward one, so there is one copy.  Three 64 KB
// regions of shared memory hold halves of it, each loaded by one bulk copy:
//   region 0: W2[0:128], then W3[128:256];   region 1: W2[128:256];
//   region 2: W3[0:128], then W2[0:128] again.
//
// Activations and their gradients go to memory as the weight gradients read
// them: for every 64 samples a contiguous block of core matrices (8 features
// x 8 samples), element (f, b) at (b / 64) 32768 + (f / 8) 1024 + (b % 64 / 8)
// 128 + (f % 8) 16 + (b % 8) 2, so that a 128 x 64 operand tile is one 16 KB
// bulk copy into the K-major layout that tcgen05.mma takes.
//
// Both kernels are launched with programmatic dependent launch; every wait is
// bounded (WLB_ERR_TIMEOUT).
//
// Small predictions (forward_small) are the forward half of train_tiles: for up to
// a few thousand queries the persistent kernel's 128-query tiles keep a few CTAs
// busy with 34 weight slices each, one after the other.  The same products and
// roundings give the same bits.

constexpr int kRegionBytes = 65536, kSmallBytes = 8192;
constexpr int kTrainEpi = 256, kTrainThreads = 288;  // warps 0-7 epilogues, warp 8 copies and products
constexpr int kChunkB = 64;                          // samples per block of the stored activations
constexpr int kWeightThreads = 160;                  // warps 0-3 epilogue, warp 4 copies and products
constexpr int kWSlots = 8, kWTileN = 16;
constexpr int kWSlotBytes = kTileM * kChunkB * 2 + kWTileN * kChunkB * 2;
constexpr int kWeightSmem = kWSlots * kWSlotBytes + 1024;
constexpr int kTilesNarrow = 152;  // CTAs of 16 samples up to one per SM; larger batches take 32 samples per CTA

struct TrainBuffers {
    uint8_t *W1p, *W2p, *W3p, *W4p;  // packed BF16 weights
    uint8_t *X0, *H[3], *dZ[3];      // inputs, activations and their gradients in blocks of 64 samples
    uint8_t *dz4;                    // dL/dy: per 64 samples 1 KB, row 0 of 8-row core matrices (rows 1-7 zero)
    float *sq;                       // every sample's share of the mean loss
};

struct TrainTiles {
    const float *x, *t;
    const int *perm;  // optional
    long long first;
    int n;            // real samples; the rest of the last tile is zero
    const float *lo, *hi, *w;
    TrainBuffers b;
    float *y;               // forward only: outputs
    unsigned char *inside;  // and whether the query lies in the box (optional)
    int *err;
};

// gelu'(z) v, rounded to BF16 as the gradients are stored.
__device__ __forceinline__ __nv_bfloat16 grad_bf16(float v, float gp) { return __float2bfloat16_rn(v * gp); }

template <int NB>
constexpr int train_tile_smem() {
    return kHid * NB * 2 + 2 * kSmallBytes + 3 * kRegionBytes + 128;
}

template <int NB, bool TRAIN>
__device__ __forceinline__ void tile_body(const TrainTiles &a) {
    extern __shared__ uint8_t train_raw[];
    // act first: the output product reads 16 groups of 8 rows from it (rows
    // at or beyond NB are other shared memory and give rows nobody reads)
    uint8_t *act = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(train_raw) + 127) & ~(uintptr_t)127);
    uint8_t *sW1 = act + kHid * NB * 2, *sW4 = sW1 + kSmallBytes;
    uint8_t *region[3] = {sW4 + kSmallBytes, sW4 + kSmallBytes + kRegionBytes, sW4 + kSmallBytes + 2 * kRegionBytes};
    constexpr uint32_t kCols = NB == 16 ? 64 : 128;  // accumulators: 2 x NB, output: 16
    constexpr int kGroups = NB / 8;
    __shared__ uint64_t full[4], accum, act_ready, region_free[2], drain;  // full[0..2] regions, [3] W1 and W4
    __shared__ uint32_t tmem_slot;
    __shared__ float s_dz4[NB];
    __shared__ int s_abort_store;
    volatile int *s_abort = &s_abort_store;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b0 = blockIdx.x * NB;
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                     "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full[i])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&accum)));
        for (int i = 0; i < 2; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&region_free[i])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&drain)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&act_ready)), "r"(kTrainEpi));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *s_abort = 0;
    }
    // normalised inputs, K = 16 rows of which 4 are real: read before the wait
    // (they do not change during training); the stored copy follows it
    constexpr int kPer = (kInPad * NB + kTrainEpi - 1) / kTrainEpi;
    __nv_bfloat16 xin[kPer];
    if (tid < kTrainEpi) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int e = tid + j * kTrainEpi, k = e / NB, i = e % NB;
            float v = 0.0f;
            if (k < kIn && b0 + i < a.n) {
                const long long src = a.perm ? a.perm[a.first + b0 + i] : a.first + b0 + i;
                v = normalise_input(a.x[src * kIn + k], a.lo[k], a.hi[k]);
            }
            xin[j] = __float2bfloat16_rn(v);
            *reinterpret_cast<__nv_bfloat16 *>(act + (i >> 3) * 4096 + (k >> 3) * 128 + (k & 7) * 16 + (i & 7) * 2) =
                xin[j];
        }
    }
    float target = 0.0f;  // of sample b0 + lane, in warp 0
    if (TRAIN && warp == 0 && lane < NB && b0 + lane < a.n)
        target = a.t[a.perm ? a.perm[a.first + b0 + lane] : a.first + b0 + lane];
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");

    if (warp == 8) {
        if (lane == 0) {
            asm volatile("fence.proxy.async;" ::: "memory");  // the packed weights were written by ordinary stores
            int issued[4] = {0, 0, 0, 0};
            auto load = [&](int r, void *dst, const uint8_t *src, uint32_t bytes) {
                mbar_expect(&full[r], bytes);
                bulk_load(dst, src, bytes, &full[r]);
                ++issued[r];
            };
            mbar_expect(&full[3], 2 * kSmallBytes);
            bulk_load(sW1, a.b.W1p, kSmallBytes, &full[3]);
            bulk_load(sW4, a.b.W4p, kSmallBytes, &full[3]);
            issued[3] = 1;
            load(0, region[0], a.b.W2p, kRegionBytes);
            load(1, region[1], a.b.W2p + kRegionBytes, kRegionBytes);
            load(2, region[2], a.b.W3p, kRegionBytes);
            bool ok = true;
            uint32_t ready = 0;
            auto wait = [&](uint64_t *bar, uint32_t phase) { ok = ok && mbar_wait_or_abort(bar, phase, s_abort); };
            auto operands = [&]() {  // the epilogue warps have written the next B operand
                wait(&act_ready, ready);
                ready ^= 1;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            };
            const uint32_t act0 = smem_addr(act);
            constexpr uint32_t kTransA = 1u << 15, kTransB = 1u << 16;  // MN-major operands
            const uint32_t id_fwd = mma_idesc(kTileM, NB) | kTransB;
            const uint32_t id_bwd = mma_idesc(kTileM, NB) | kTransA | kTransB;
            const uint32_t id_out = mma_idesc(kTileM, kOutPad) | kTransA;
            auto half_forward = [&](int h, const uint8_t *w) {  // rows 128 h .. 128 h + 127 of the layer
                for (int k = 0; k < kHid / 16; ++k)
                    mma_bf16(tmem + (uint32_t)(h * NB), smem_desc(smem_addr(w) + k * 256, 128, 4096),
                             smem_desc(act0 + k * 256, 128, 4096), id_fwd, k > 0);
            };
            auto half_backward = [&](int h, const uint8_t *w) {  // K = features 128 h .. of the upper layer
                for (int k = 0; k < kHid / 32; ++k)
                    for (int m = 0; m < 2; ++m)
                        mma_bf16(tmem + (uint32_t)(m * NB), smem_desc(smem_addr(w) + k * 8192 + m * 2048, 4096, 128),
                                 smem_desc(act0 + (h * (kHid / 32) + k) * 256, 128, 4096), id_bwd, h > 0 || k > 0);
            };
            // layer 1
            wait(&full[3], 0);
            operands();
            if (ok) {
                for (int h = 0; h < 2; ++h)
                    mma_bf16(tmem + (uint32_t)(h * NB), smem_desc(smem_addr(sW1) + h * 4096, 128, 256),
                             smem_desc(act0, 128, 4096), id_fwd, 0);
                mma_commit(&accum);
            }
            // layer 2
            wait(&full[0], 0);
            operands();
            if (ok) {
                half_forward(0, region[0]);
                mma_commit(&region_free[0]);
            }
            wait(&full[1], 0);
            if (ok) {
                half_forward(1, region[1]);
                mma_commit(&accum);
            }
            wait(&region_free[0], 0);
            if (ok) load(0, region[0], a.b.W3p + kRegionBytes, kRegionBytes);
            // layer 3
            wait(&full[2], 0);
            operands();
            if (ok) half_forward(0, region[2]);
            wait(&full[0], 1);
            if (ok) {
                half_forward(1, region[0]);
                mma_commit(&accum);
            }
            // output: rows are samples here (A = H3, 16 columns of which one is real)
            operands();
            if (ok) {
                for (int k = 0; k < kHid / 16; ++k)
                    mma_bf16(tmem + 2 * NB, smem_desc(act0 + k * 256, 128, 4096),
                             smem_desc(smem_addr(sW4) + k * 256, 128, 4096), id_out, k > 0);
                mma_commit(&accum);
            }
            if constexpr (TRAIN) {
                // gradient of H2 = W3^T dZ3
                operands();
                if (ok) {
                    half_backward(0, region[2]);
                    mma_commit(&region_free[1]);
                    half_backward(1, region[0]);
                    mma_commit(&accum);
                }
                wait(&region_free[1], 0);
                if (ok) load(2, region[2], a.b.W2p, kRegionBytes);
                // gradient of H1 = W2^T dZ2
                operands();
                wait(&full[2], 1);
                if (ok) {
                    half_backward(0, region[2]);
                    half_backward(1, region[1]);
                    mma_commit(&accum);
                }
            }
            if (!ok) {
                if (!*s_abort) {
                    *s_abort = 1;
                    raise(a.err);
                }
                // copies in flight land before the CTA exits
                for (int r = 0; r < 4; ++r)
                    if (issued[r] > 0) mbar_wait(&full[r], (uint32_t)((issued[r] - 1) & 1));
            }
            mma_commit(&drain);  // no product may still run when the tensor memory is freed
            mbar_wait(&drain, 0);
        }
        __syncwarp();
    } else {
        const int q = warp & 3, h = warp >> 2;
        const int f = h * kTileM + q * 32 + lane;  // this thread's feature
        const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(h * NB);
        uint8_t *my_act = act + (f >> 3) * 128 + (f & 7) * 16;  // sample group g at + 4096 g
        const size_t my_out = (size_t)(b0 / kChunkB) * (kHid * kChunkB * 2) + (size_t)(f >> 3) * 1024 +
                              (size_t)((b0 % kChunkB) / 8) * 128 + (size_t)(f & 7) * 16;  // group g at + 128 g
#pragma unroll
        for (int j = 0; j < (TRAIN ? kPer : 0); ++j) {
            const int e = tid + j * kTrainEpi, k = e / NB, b = b0 + e % NB;
            *reinterpret_cast<__nv_bfloat16 *>(a.b.X0 + (size_t)(b / kChunkB) * (kInPad * kChunkB * 2) +
                                               (k >> 3) * 1024 + ((b % kChunkB) >> 3) * 128 + (k & 7) * 16 +
                                               (b & 7) * 2) = xin[j];
        }
        const float bias[3] = {a.w[ob1 + f], a.w[ob2 + f], a.w[ob3 + f]};
        const float b4 = a.w[ob4];
        auto publish = [&]() {  // the operand in `act` is complete, the accumulator has been read
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(&act_ready);
        };
        // 16-byte pieces of this feature's samples: next operand (optional) and the stored copy
        auto store = [&](const uint32_t (&pk)[NB / 2], uint8_t *out, bool operand) {
#pragma unroll
            for (int g = 0; g < kGroups; ++g) {
                const uint4 v = make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
                if (operand) *reinterpret_cast<uint4 *>(my_act + g * 4096) = v;
                if (TRAIN) *reinterpret_cast<uint4 *>(out + my_out + g * 128) = v;
            }
        };
        uint32_t phase = 0;
        bool ok = true;
        auto accumulator = [&](float (&v)[NB]) {
            ok = ok && mbar_wait_or_abort(&accum, phase, s_abort);
            phase ^= 1;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (ok) {
#pragma unroll
                for (int c = 0; c < NB / 16; ++c) {
                    float u[16];
                    tmem_ld16(trow + (uint32_t)(16 * c), u);
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[16 * c + e] = u[e];
                }
            }
        };
        float gp[3][TRAIN ? NB : 1];
        publish();
        // no early exit from here: every warp reaches the block barriers and the
        // named barrier below; a failed wait skips the work
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            float v[NB];
            accumulator(v);
            if (ok) {
                uint32_t pk[NB / 2];
#pragma unroll
                for (int e = 0; e < NB; e += 2) {
                    v[e] = __fadd_rn(v[e], bias[l]);
                    v[e + 1] = __fadd_rn(v[e + 1], bias[l]);
                    float g0, g1;
                    gelu2(v[e], v[e + 1], g0, g1);
                    const __nv_bfloat162 p = __floats2bfloat162_rn(g0, g1);
                    pk[e / 2] = *reinterpret_cast<const uint32_t *>(&p);
                }
                store(pk, a.b.H[l], true);
                publish();
                // GELU' only now, while the next product runs: behind a branch on a
                // load that follows the hand-over, or the assembler evaluates it
                // ahead of it and holds every layer back by up to 2.7k cycles
                if (*s_abort) {
                    ok = false;
                } else if constexpr (TRAIN) {
#pragma unroll
                    for (int e = 0; e < NB; ++e) gp[l][e] = gelu_grad(v[e]);
                }
            }
        }
        if constexpr (!TRAIN) {
            if (warp == 1 && lane < NB && b0 + lane < a.n && a.inside) {
                bool in = true;
                for (int e = 0; e < kIn; ++e) {
                    const float xv = a.x[(size_t)(b0 + lane) * kIn + e];
                    in &= xv >= a.lo[e] && xv <= a.hi[e];
                }
                a.inside[b0 + lane] = in ? 1 : 0;
            }
        }
        // output, loss and dL/dy: one lane of warp 0 per sample
        ok = ok && mbar_wait_or_abort(&accum, phase, s_abort);
        phase ^= 1;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (warp == 0) {
            if (ok) {
                float v[16];
                tmem_ld16(tmem + 2 * NB, v);
                const int b = b0 + lane;
                float g = 0.0f, l = 0.0f;
                if (!TRAIN && lane < NB && b < a.n) a.y[b] = v[0] + b4;
                if (TRAIN && lane < NB && b < a.n) {
                    const float d = v[0] + b4 - target;
                    l = d * d / (float)a.n;
                    g = 2.0f * d / (float)a.n;
                }
                if (TRAIN && lane < NB) {
                    const __nv_bfloat16 gb = __float2bfloat16_rn(g);
                    s_dz4[lane] = __bfloat162float(gb);
                    *reinterpret_cast<__nv_bfloat16 *>(a.b.dz4 + (size_t)(b / kChunkB) * 1024 +
                                                       ((b % kChunkB) >> 3) * 128 + (b & 7) * 2) = gb;
                    a.b.sq[b] = l;
                }
            }
        }
        if constexpr (TRAIN) {
            asm volatile("bar.sync 1, %0;" ::"n"(kTrainEpi) : "memory");
            const float w4 = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(sW4 + (f >> 3) * 128 + (f & 7) * 2));
#pragma unroll
            for (int l = 2; l >= 0; --l) {
                float v[NB];
                if (l == 2) {
                    // dH3 = dL/dy W4: the product of two BF16 values is exact
#pragma unroll
                    for (int e = 0; e < NB; ++e) v[e] = s_dz4[e] * w4;
                } else {
                    accumulator(v);
                }
                if (ok) {
                    uint32_t pk[NB / 2];
#pragma unroll
                    for (int e = 0; e < NB; e += 2) {
                        __nv_bfloat162 p;
                        p.x = grad_bf16(v[e], gp[l][e]);
                        p.y = grad_bf16(v[e + 1], gp[l][e + 1]);
                        pk[e / 2] = *reinterpret_cast<const uint32_t *>(&p);
                    }
                    store(pk, a.b.dZ[l], l > 0);
                    if (l > 0) publish();
                }
            }
        }
        if (!ok && !*s_abort) {
            *s_abort = 1;
            raise(a.err);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 8) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
    }
}

template <int NB>
__global__ void __launch_bounds__(kTrainThreads, 1) train_tiles(TrainTiles a) {
    tile_body<NB, true>(a);
}
template <int NB>
__global__ void __launch_bounds__(kTrainThreads, 1) forward_small(TrainTiles a) {
    tile_body<NB, false>(a);
}

struct TrainWeights {
    TrainBuffers b;
    int blocks;       // 64-sample blocks
    float *w, *m1, *m2;
    float *g;         // non-null: write the gradient and leave the weights alone
    float *loss;      // += this batch's mean loss
    float lr, c1, c2;
    int *err;
};

// Adam (bias-corrected) on one FP32 master; the BF16 copy is the caller's.
__device__ __forceinline__ float adam_step(const TrainWeights &a, float w, float g, float &m1, float &m2) {
    m1 = 0.9f * m1 + 0.1f * g;
    m2 = 0.999f * m2 + 0.001f * g * g;
    return w - a.lr * (m1 * a.c1) / (sqrtf(m2 * a.c2) + 1e-8f);
}

// One scalar parameter: its gradient, or its update.  Returns the new value.
__device__ __forceinline__ float update_param(const TrainWeights &a, int p, float g) {
    if (a.g) {
        a.g[p] = g;
        return a.w[p];
    }
    float m1 = a.m1[p], m2 = a.m2[p];
    const float w = adam_step(a, a.w[p], g, m1, m2);
    a.m1[p] = m1;
    a.m2[p] = m2;
    a.w[p] = w;
    return w;
}

// Jobs of train_weights, by block: the 128 x 16 tiles of dW2, dW3 and dW1, the
// 1 x 16 tiles of dW4 (one real row of 128), the bias gradients in groups of
// 32 features, and the output bias with the loss.  16 columns per tile rather
// than 32: each thread's Adam updates are the longest phase after the
// products, and the chip has the SMs for it.
constexpr int kColTiles = kHid / kWTileN;
constexpr int kJobW3 = 2 * kColTiles, kJobW1 = 2 * kJobW3, kJobW4 = kJobW1 + 2, kJobBias = kJobW4 + kColTiles,
              kJobOut = kJobBias + 24, kWeightJobs = kJobOut + 1;
constexpr int kBiasRound = 64;  // groups of 32 samples per round of the bias jobs

__global__ void __launch_bounds__(kWeightThreads, 1) train_weights(TrainWeights a) {
    extern __shared__ uint8_t weights_raw[];
    uint8_t *slots =
        reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(weights_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[kWSlots], empty[kWSlots], accum, drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort_store;
    volatile int *s_abort = &s_abort_store;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, job = blockIdx.x;
    asm volatile("griddepcontrol.launch_dependents;");
    if (job >= kJobBias) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (job < kJobOut) {
            // sums over the samples of dZ as stored: every 32 samples as a tree,
            // the trees in sample order (the same bits for any grid)
            const int l = (job - kJobBias) >> 3, f = ((job - kJobBias) & 7) * 32 + lane;
            const uint8_t *src = a.b.dZ[l] + (size_t)(f >> 3) * 1024 + (f & 7) * 16;
            float (*part)[32] = reinterpret_cast<float (*)[32]>(slots);
            const int groups = 2 * a.blocks;
            float sum = 0.0f;
            for (int r = 0; r < groups; r += kBiasRound) {
                const int m = groups - r < kBiasRound ? groups - r : kBiasRound;
                for (int g = warp; g < m; g += kWeightThreads / 32) {
                    const uint8_t *p = src + (size_t)((r + g) >> 1) * (kHid * kChunkB * 2) + ((r + g) & 1) * 512;
                    float d[32];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(p + j * 128);
                        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            d[8 * j + 2 * e] = __uint_as_float(u[e] << 16);
                            d[8 * j + 2 * e + 1] = __uint_as_float(u[e] & 0xffff0000u);
                        }
                    }
#pragma unroll
                    for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
                        for (int e = 0; e < o; ++e) d[e] += d[e + o];
                    part[g][lane] = d[0];
                }
                __syncthreads();
                if (warp == 0)
                    for (int g = 0; g < m; ++g) sum += part[g][lane];
                __syncthreads();
            }
            if (warp == 0) update_param(a, (l == 0 ? ob1 : l == 1 ? ob2 : ob3) + f, sum);
        } else if (warp == 0) {
            float sum = 0.0f, loss = 0.0f;
            for (int b = lane; b < a.blocks * kChunkB; b += 32) {
                float s = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
                    a.b.dz4 + (size_t)(b / kChunkB) * 1024 + ((b % kChunkB) >> 3) * 128 + (b & 7) * 2));
                float l = a.b.sq[b];
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) {
                    s += __shfl_xor_sync(0xffffffffu, s, o);
                    l += __shfl_xor_sync(0xffffffffu, l, o);
                }
                sum += s;
                loss += l;
            }
            if (lane == 0) {
                update_param(a, ob4, sum);
                *a.loss += loss;
            }
        }
        return;
    }
    // a tile of dW = dZ^T H: rows mt * 128 .., columns nt * 16 ..; layer 0 .. 3
    const int layer = job < kJobW3 ? 1 : (job < kJobW1 ? 2 : (job < kJobW4 ? 0 : 3));
    const int mt = layer == 0 ? job - kJobW1 : (layer == 3 ? 0 : (job / kColTiles) & 1);
    const int nt = layer == 0 ? 0 : (layer == 3 ? job - kJobW4 : job % kColTiles);
    static_assert(kWTileN == kInPad, "every tile has the input layer's padded width");
    constexpr int kBlockBytes = kHid * kChunkB * 2, kBytesA = kTileM * kChunkB * 2;
    const uint8_t *A = layer == 3 ? a.b.dz4 : a.b.dZ[layer] + (size_t)mt * kBytesA;
    const uint8_t *B = layer == 0 ? a.b.X0 : a.b.H[layer - 1] + (size_t)nt * (kWTileN * kChunkB * 2);
    const size_t strideA = layer == 3 ? 1024 : kBlockBytes, strideB = layer == 0 ? kInPad * kChunkB * 2 : kBlockBytes;
    const uint32_t bytesA = layer == 3 ? 1024 : kBytesA, bytesB = kWTileN * kChunkB * 2;
    if (layer == 3) {
        // rows 8 .. 127 of the A operand are zero in every slot
        for (int i = tid; i < kWSlots * (kBytesA / 16); i += kWeightThreads)
            *reinterpret_cast<uint4 *>(slots + (i / (kBytesA / 16)) * kWSlotBytes + (i % (kBytesA / 16)) * 16) =
                make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                     "r"(32u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < kWSlots; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&empty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&accum)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&drain)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *s_abort = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    if (warp == 4) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (lane == 0) {
            asm volatile("fence.proxy.async;" ::: "memory");  // the operands were written by ordinary stores
            auto load = [&](int c) {
                const int s = c % kWSlots;
                mbar_expect(&full[s], bytesA + bytesB);
                bulk_load(slots + s * kWSlotBytes, A + (size_t)c * strideA, bytesA, &full[s]);
                bulk_load(slots + s * kWSlotBytes + kBytesA, B + (size_t)c * strideB, bytesB, &full[s]);
            };
            const uint32_t idesc = mma_idesc(kTileM, kWTileN);
            int issued = 0;
            for (; issued < kWSlots && issued < a.blocks; ++issued) load(issued);
            bool ok = true;
            for (int c = 0; c < a.blocks; ++c) {
                const int s = c % kWSlots;
                if (!(ok = mbar_wait_or_abort(&full[s], (uint32_t)((c / kWSlots) & 1), s_abort))) break;
                const uint32_t base = smem_addr(slots + s * kWSlotBytes);
                for (int k = 0; k < kChunkB / 16; ++k)
                    mma_bf16(tmem, smem_desc(base + k * 256, 128, 1024), smem_desc(base + kBytesA + k * 256, 128, 1024),
                             idesc, c > 0 || k > 0);
                mma_commit(&empty[s]);
                // refill the slot of the previous block once its products are done
                if (c >= 1 && issued < a.blocks) {
                    const int r = c - 1;
                    if (!(ok = mbar_wait_or_abort(&empty[r % kWSlots], (uint32_t)((r / kWSlots) & 1), s_abort))) break;
                    load(issued++);
                }
            }
            if (ok) {
                mma_commit(&accum);
            } else {
                if (!*s_abort) {
                    *s_abort = 1;
                    raise(a.err);
                }
                for (int c = issued > kWSlots ? issued - kWSlots : 0; c < issued; ++c)
                    mbar_wait(&full[c % kWSlots], (uint32_t)((c / kWSlots) & 1));
            }
            mma_commit(&drain);
            mbar_wait(&drain, 0);
        }
        __syncwarp();
    } else {
        // parameters of this thread's row of the tile; the previous step wrote
        // them before train_tiles of this step passed its wait, after which
        // this kernel may start, so they are read before this kernel's wait
        const int row = mt * kTileM + warp * 32 + lane;
        const int p0 = layer == 0 ? oW1 + row * kIn : (layer == 1 ? oW2 : oW3) + row * kHid + nt * kWTileN;
        const int nv = layer == 0 ? 1 : (layer == 3 ? 0 : kWTileN / 4);  // float4 of real columns
        float4 w[kWTileN / 4], m1[kWTileN / 4], m2[kWTileN / 4];
        if (!a.g) {
#pragma unroll
            for (int j = 0; j < kWTileN / 4; ++j)
                if (j < nv) {
                    w[j] = *reinterpret_cast<const float4 *>(a.w + p0 + 4 * j);
                    m1[j] = *reinterpret_cast<const float4 *>(a.m1 + p0 + 4 * j);
                    m2[j] = *reinterpret_cast<const float4 *>(a.m2 + p0 + 4 * j);
                }
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const bool ok = mbar_wait_or_abort(&accum, 0, s_abort);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
            const uint32_t trow = tmem + ((uint32_t)(32 * warp) << 16);
            float v[kWTileN];
            tmem_ld16(trow, v);
            if (layer == 3 && warp == 0) {
                // row 0 holds the gradient of W4: one column per lane
                __shared__ float s_row[kWTileN];
                if (lane == 0)
#pragma unroll
                    for (int e = 0; e < kWTileN; ++e) s_row[e] = v[e];
                __syncwarp();
                const int f = nt * kWTileN + lane;
                if (lane < kWTileN) {
                    const float w4 = update_param(a, oW4 + f, s_row[lane]);
                    if (!a.g)
                        *reinterpret_cast<__nv_bfloat16 *>(a.b.W4p + (f >> 3) * 128 + (f & 7) * 2) =
                            __float2bfloat16_rn(w4);
                }
            }
            uint32_t pk[kWTileN / 2];
#pragma unroll
            for (int j = 0; j < kWTileN / 4; ++j) {
                if (j >= nv) break;
                if (a.g) {
                    *reinterpret_cast<float4 *>(a.g + p0 + 4 * j) =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    continue;
                }
                w[j].x = adam_step(a, w[j].x, v[4 * j], m1[j].x, m2[j].x);
                w[j].y = adam_step(a, w[j].y, v[4 * j + 1], m1[j].y, m2[j].y);
                w[j].z = adam_step(a, w[j].z, v[4 * j + 2], m1[j].z, m2[j].z);
                w[j].w = adam_step(a, w[j].w, v[4 * j + 3], m1[j].w, m2[j].w);
                *reinterpret_cast<float4 *>(a.w + p0 + 4 * j) = w[j];
                *reinterpret_cast<float4 *>(a.m1 + p0 + 4 * j) = m1[j];
                *reinterpret_cast<float4 *>(a.m2 + p0 + 4 * j) = m2[j];
                const __nv_bfloat162 lo = __floats2bfloat162_rn(w[j].x, w[j].y);
                const __nv_bfloat162 hi = __floats2bfloat162_rn(w[j].z, w[j].w);
                pk[2 * j] = *reinterpret_cast<const uint32_t *>(&lo);
                pk[2 * j + 1] = *reinterpret_cast<const uint32_t *>(&hi);
            }
            if (!a.g && layer != 3) {
                if (layer == 0) {
                    *reinterpret_cast<uint2 *>(a.b.W1p + (row >> 3) * 256 + (row & 7) * 16) = make_uint2(pk[0], pk[1]);
                } else {
                    uint8_t *dst = (layer == 1 ? a.b.W2p : a.b.W3p) + (size_t)(row >> 3) * 4096 +
                                   nt * (kWTileN / 8) * 128 + (row & 7) * 16;
#pragma unroll
                    for (int g = 0; g < kWTileN / 8; ++g)
                        *reinterpret_cast<uint4 *>(dst + g * 128) =
                            make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
                }
            }
        } else if (!*s_abort) {
            *s_abort = 1;
            raise(a.err);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 4) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(32u));
    }
}

// The packed BF16 weights from the FP32 masters (padding zero).
__global__ void pack_train(const float *__restrict__ w, TrainBuffers b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;  // over 256 x 256
    if (i >= kHid * kHid) return;
    const int o = i / kHid, k = i % kHid;
    const int at = (o >> 3) * 4096 + (k >> 3) * 128 + (o & 7) * 16 + (k & 7) * 2;
    *reinterpret_cast<__nv_bfloat16 *>(b.W2p + at) = __float2bfloat16_rn(w[oW2 + i]);
    *reinterpret_cast<__nv_bfloat16 *>(b.W3p + at) = __float2bfloat16_rn(w[oW3 + i]);
    if (k < kInPad)
        *reinterpret_cast<__nv_bfloat16 *>(b.W1p + (o >> 3) * 256 + (k >> 3) * 128 + (o & 7) * 16 + (k & 7) * 2) =
            __float2bfloat16_rn(k < kIn ? w[oW1 + o * kIn + k] : 0.0f);
    if (o < kOutPad) *reinterpret_cast<__nv_bfloat16 *>(b.W4p + at) = __float2bfloat16_rn(o == 0 ? w[oW4 + k] : 0.0f);
}
