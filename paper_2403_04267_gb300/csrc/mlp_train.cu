// mlp_train.cu -- the surrogate MLP's training step (and inference on few samples) as three
// kernels: the forward and the backward pass of 32-sample tiles with the activations kept
// on chip (k_mlp_pass), every layer's weight gradient (k_mlp_dw), and the sum of their
// split-K partials with the Adam update (k_mlp_update).
//
// A step used to be 21 launches, a GEMM each for every layer's forward, activation-gradient
// and weight-gradient product with reductions between them: 319 us at 3675 samples, each
// kernel 15-30 us of its own latency (ncu: 5-10 % of the issue slots, the tensor pipe 1 %
// busy).  The arithmetic per element is that of those GEMMs: the same operands rounded to
// BF16, FP32 accumulation over K in the same order, the same K splits of the weight
// gradients, added in the same order.
#include "mlp_device.cuh"

namespace salec {
namespace mlp {

// ---------------------------------------------------------------------------------------
// The pass kernel: all five layers, and in training the backward pass, of a tile of 32
// samples, one CTA a tile (115 CTAs at 3675 samples).
//
// The products are formed transposed, Z^T = W H^T: the weights are the M side of the MMA (two
// blocks of 128 features, streamed by TMA as 128 x 64 K slices, 128-byte swizzled, into a
// ring of nine 16 KB stages), the samples its N side, so that a narrow tile of samples still
// fills the 128 lanes of tensor memory and no CTA needs another's columns.  (A tile of 128
// samples with its columns shared by a cluster of four CTAs needs an exchange of 48 KB per
// CTA and layer: shared-to-shared copies moved it at 16 bytes a clock, 3000 of the 7200
// cycles of a layer.)  The activations live in shared memory as the N-side operand (two
// buffers of 32 x 256 BF16: four 128-byte swizzled K slices).
//
// The pre-activations of the four hidden layers stay where the tensor cores left them, in
// tensor memory (4 layers x 2 blocks x 32 columns), so the backward pass reads gelu'(Z) from
// there: nothing but the transposed activations and gradients that the weight gradients
// contract over (HT, GT: a thread holds one feature of eight samples, 16 bytes) and Y - T for
// the loss goes to global memory.
//
// Products g with operand buffer g & 1 and accumulator columns (a block each 32):
//   0      W_1 X^T           64 g       K = 16
//   1..3   W_{g+1} H_g^T     64 g
//   4      W_5 H_4^T         256        66 features: one block
//   5      W_5^T G_5^T       320 + 64   K = 80 (66 padded)
//   6..8   W^T G^T           320 + 64 (g & 1)
// The two halves of an operand (K slices 0, 1 from feature block 0; 2, 3 from block 1) are
// signalled apart: a product starts on the first half of both its blocks while the epilogue
// of the second block of the product before still runs.  K runs in order in each block.
//
// An epilogue writes operand buffer (g + 1) & 1 once block 0 of product g is complete, which
// follows every MMA of product g - 1, the buffer's last readers.  The backward accumulators
// alternate, since block 1 of a product may start before the epilogue of block 1 of the one
// before has read its columns.  Every wait is bounded; one that runs out raises the abort
// flag and every role leaves its loop.  However its loop ends, the TMA thread waits for its
// copies and the MMA thread, on a barrier of its own behind every MMA it issued, for its MMAs.
//
// Warps: 0 TMA, 1 MMA, 2-17 epilogue (lane quarter q = warp & 3: features; samples 8 cq .. of
// cq = (warp - 2) >> 2), 18 the training state of the step.
// ---------------------------------------------------------------------------------------
constexpr int kPassThreads = 19 * 32;
constexpr int kNS = 32;                                    // samples of a tile
constexpr int kHidden = 256;
constexpr int kPassStages = 9;
constexpr uint32_t kOpSlice = kNS * 128;                   // operand K slice: 4 KB
constexpr uint32_t kOpBytes = 4 * kOpSlice;
constexpr uint32_t kW1Smem = kHidden * 16 * 2;             // layer 1, core matrices without swizzle
constexpr uint32_t kPassSmem = kPassStages * kSliceBytes + 2 * kOpBytes + kW1Smem + 1024;
constexpr int kAccOut = 256, kAccBwd = 320;                // accumulator columns

template <int NMEM>
struct PassArgs {
    NetMaps maps[NMEM];
    NetPtrs net[NMEM];
    const float* x;          // inference: FP32 inputs, rows of 5
    const float* t;          // training: targets
    float* y;                // inference: outputs
    const float* lr;         // training by a table: learning rates, or null
    float beta1, beta2, grad_scale;
    int B;
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v)
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

template <int NMEM, bool TRAIN>
__global__ void __launch_bounds__(kPassThreads, 1) k_mlp_pass(const __grid_constant__ PassArgs<NMEM> a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* ring = smem;
    unsigned char* op = smem + kPassStages * kSliceBytes;      // two operand buffers
    unsigned char* w1s = op + 2 * kOpBytes;
    __shared__ uint64_t wfull[kPassStages], wempty[kPassStages], hfull[2][2], accfull[2], drained;
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const NetMaps& maps = a.maps[NMEM == 1 ? 0 : blockIdx.y];
    const NetPtrs& n = a.net[NMEM == 1 ? 0 : blockIdx.y];
    const int m0 = (int)blockIdx.x * kNS;
    constexpr int kProducts = TRAIN ? 9 : 5;
    // feature blocks, K slices of a product
    auto blocks = [](int g) { return g == 4 ? 1 : 2; };

    if (tid == 0) {
        for (int k = 0; k < kPassStages; ++k) { mbar_init(&wfull[k], 1); mbar_init(&wempty[k], 1); }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&hfull[k][0], 16);
            mbar_init(&hfull[k][1], 16);
            mbar_init(&accfull[k], 1);
        }
        mbar_init(&drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // (inference is launched to overlap the kernel before it, whose weights or inputs it reads)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int c = tid; c < kHidden; c += kPassThreads) {
        *reinterpret_cast<uint4*>(w1s + cm_off(c, 0, kHidden)) = *reinterpret_cast<const uint4*>(n.W1 + (long)c * 8);
        *reinterpret_cast<uint4*>(w1s + cm_off(c, 1, kHidden)) = make_uint4(0u, 0u, 0u, 0u);
    }
    // the tile's inputs: 8 BF16 a sample, K padded to 16, in the first K slice of buffer 0
    if (warp == 18) {
        const int m = m0 + lane;
        uint4 xv = make_uint4(0u, 0u, 0u, 0u);
        if (m < a.B) {
            if (TRAIN) {
                xv = *reinterpret_cast<const uint4*>(n.X + (long)m * 8);
            } else {
                const float* x = a.x + (long)m * 5;
                const __nv_bfloat162 p0 = __floats2bfloat162_rn(x[0], x[1]), p1 = __floats2bfloat162_rn(x[2], x[3]);
                const __nv_bfloat162 p2 = __floats2bfloat162_rn(x[4], 0.0f);
                xv.x = *reinterpret_cast<const uint32_t*>(&p0);
                xv.y = *reinterpret_cast<const uint32_t*>(&p1);
                xv.z = *reinterpret_cast<const uint32_t*>(&p2);
            }
        }
        *reinterpret_cast<uint4*>(op + sw128_off(lane, 0)) = xv;
        *reinterpret_cast<uint4*>(op + sw128_off(lane, 1)) = make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;

    if (warp == 0) {
        // ---- weight slices, in the order the MMAs take them ----
        if (elect_one()) {
            int k = 0;
            auto slice = [&](const CUtensorMap* map, int kt, int blk) {
                const int st = k % kPassStages, use = k / kPassStages;
                if (use > 0 && !mbar_wait_idle(&wempty[st], (uint32_t)(use - 1) & 1u)) {
                    abort_flag = 1;
                    return;
                }
                mbar_expect_tx(&wfull[st], kSliceBytes);
                tma_load_2d(smem_u32(ring + st * kSliceBytes), map, kt * kBK, blk * kBM, &wfull[st]);
                ++k;
            };
            for (int g = 1; g < kProducts && !abort_flag; ++g) {
                const CUtensorMap* map = g < 5 ? &maps.w[g - 1] : &maps.wt[g - 5];
                for (int half = 0; half < (g == 5 ? 1 : 2); ++half)
                    for (int blk = 0; blk < blocks(g); ++blk)
                        for (int kt = 2 * half; kt < 2 * half + 2 && !abort_flag && !stalled(k); ++kt) slice(map, kt, blk);
            }
            // the last copy of each stage lands before the CTA's memory can go away
            for (int st = 0; st < kPassStages; ++st) {
                const int uses = k > st ? (k - 1 - st) / kPassStages + 1 : 0;
                if (uses > 0) mbar_drain(&wfull[st], (uint32_t)(uses - 1) & 1u);
            }
        }
    } else if (warp == 1) {
        // ---- MMAs ----
        if (elect_one()) {
            // descriptors by addition: a 16-wide K step is 32 bytes of a swizzled row of either
            // operand (formed anew at every step they took about 280 cycles of this one thread)
            const uint32_t idesc = idesc_bf16(kBM, kNS);
            const uint64_t ring_desc = sdesc_sw128(smem_u32(ring));
            int st = 0;
            uint32_t par = 0, hphase[2][2] = {{0u, 0u}, {0u, 0u}};
            bool good = true;
            for (int g = 0; g < kProducts && good; ++g) {
                const uint64_t h_desc = sdesc_sw128(smem_u32(op + (g & 1) * kOpBytes));
                const uint32_t acc = tmem + (uint32_t)(g < 4 ? 64 * g : g == 4 ? kAccOut : kAccBwd + 64 * (g & 1));
                if (g == 0) {
                    // (the inputs were there before the roles split)
                    for (int blk = 0; blk < 2; ++blk) {
                        mma_bf16(acc + blk * kNS, sdesc(smem_u32(w1s) + blk * (kBM * 16), kHidden * 16, 128), h_desc, idesc, 0u);
                        mma_commit(&accfull[blk]);
                    }
                    continue;
                }
                const int halves = g == 5 ? 1 : 2;
                for (int half = 0; half < halves && good; ++half) {
                    if (!mbar_wait_short(&hfull[g & 1][half], hphase[g & 1][half])) { good = false; break; }
                    hphase[g & 1][half] ^= 1u;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int blk = 0; blk < blocks(g) && good; ++blk) {
                        for (int kt = 2 * half; kt < 2 * half + 2; ++kt) {
                            if (!mbar_wait_short(&wfull[st], par)) { good = false; break; }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint64_t wd = ring_desc + (uint64_t)(st * (kSliceBytes >> 4));
                            const uint64_t hd = h_desc + (uint64_t)(kt * (kOpSlice >> 4));
                            mma_bf16(acc + blk * kNS, wd, hd, idesc, kt > 0 ? 1u : 0u);
                            if (g != 5 || kt == 0) {          // G_5 ends after five K steps
#pragma unroll
                                for (int kk = 1; kk < 4; ++kk) mma_bf16(acc + blk * kNS, wd + kk * 2, hd + kk * 2, idesc, 1u);
                            }
                            mma_commit(&wempty[st]);
                            if (++st == kPassStages) {
                                st = 0;
                                par ^= 1u;
                            }
                        }
                        if (good && half == halves - 1) mma_commit(&accfull[blk]);
                    }
                }
            }
            if (!good) abort_flag = 1;
            // every MMA issued finishes before the tensor memory is freed (an epilogue warp may
            // have given up on the last of them)
            mma_commit(&drained);
            mbar_drain(&drained, 0u);
        }
    } else if (warp < 18) {
        // ---- epilogues ----
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const int ms = m0 + cq * 8;                            // the thread's first sample
        const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cq * 8);
        // the operand half of buffer b is written: this warp's part reported
        auto publish = [&](int b, int half) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&hfull[b][half]);
        };
        // feature f of the thread's eight samples into operand buffer b
        auto store = [&](int b, int f, const uint32_t* w) {
            unsigned char* H = op + b * kOpBytes + (f >> 6) * kOpSlice + (f & 7) * 2;
            const int c = (f & 63) >> 3;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                *reinterpret_cast<unsigned short*>(H + sw128_off(cq * 8 + j, c)) = (unsigned short)(w[j >> 1] >> (16 * (j & 1)));
        };
        // row f of a transposed activation or gradient: eight samples, 16 bytes
        auto store_t = [&](__nv_bfloat16* P, int f, const uint32_t* w) {
            __nv_bfloat16* d = P + (long)f * n.ldT + ms;
            if (ms + 8 <= a.B) {
                *reinterpret_cast<uint4*>(d) = make_uint4(w[0], w[1], w[2], w[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (ms + j < a.B) reinterpret_cast<unsigned short*>(d)[j] = (unsigned short)(w[j >> 1] >> (16 * (j & 1)));
            }
        };
        // biases of the thread's features, and the targets of its outputs
        float bias[4][2];
        const int fo = q * 32 + lane;
        const bool out = fo < SALEC_MLP_OUT_N;
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            bias[l][0] = n.bias[l][fo];
            bias[l][1] = n.bias[l][kBM + fo];
        }
        const float bias_o = out ? n.bias[4][fo] : 0.0f;
        float tv[TRAIN ? 8 : 1];
        if (TRAIN) {
#pragma unroll
            for (int j = 0; j < 8; ++j) tv[j] = out && ms + j < a.B ? a.t[(long)(ms + j) * SALEC_MLP_OUT_N + fo] : 0.0f;
        }
        bool stop = false;
        auto wait_acc = [&](int blk, int use) {
            if (!__all_sync(0xffffffffu, mbar_wait_short(&accfull[blk], (uint32_t)use & 1u))) {
                abort_flag = 1;
                return false;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            return true;
        };
#pragma unroll
        for (int g = 0; g < kProducts; ++g) {
            if (stop) break;
            const int nb = (g + 1) & 1;
            if (g == 4) {
                // outputs; in training dL/dY = 2 (Y - T) / (B 66), zero beyond the 66 features and
                // the batch, and Y - T for the loss
                if (!wait_acc(0, 4)) break;
                float v[8];
                tmem_ld8(trow + kAccOut, v);
                if (TRAIN) {
                    float d[8], h[8];
                    uint32_t w[4];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const bool here = out && ms + j < a.B;
                        d[j] = (v[j] + bias_o) - tv[TRAIN ? j : 0];
                        h[j] = here ? d[j] * a.grad_scale : 0.0f;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const __nv_bfloat162 p = __floats2bfloat162_rn(h[2 * k], h[2 * k + 1]);
                        w[k] = *reinterpret_cast<const uint32_t*>(&p);
                    }
                    store(nb, fo, w);
                    publish(nb, 0);
                    if (out) {
                        store_t(n.GT[4], fo, w);
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (ms + j < a.B) n.D[(long)fo * n.ldT + ms + j] = d[j];
                    }
                } else if (out) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (ms + j < a.B) a.y[(long)(ms + j) * SALEC_MLP_OUT_N + fo] = v[j] + bias_o;
                }
            } else {
#pragma unroll
                for (int blk = 0; blk < 2; ++blk) {
                    // block 1 has one product fewer before the backward pass
                    if (!wait_acc(blk, g < 4 || blk == 0 ? g : g - 1)) {
                        stop = true;
                        break;
                    }
                    const int f = blk * kBM + fo;
                    uint32_t w[4];
                    if (g < 4) {
                        float v[8];
                        tmem_ld8(trow + (uint32_t)(64 * g + blk * kNS), v);
                        const f32x2 b = f2(bias[g < 4 ? g : 0][blk], bias[g < 4 ? g : 0][blk]);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const f32x2 h = gelu_pair(f2add(f2(v[2 * k], v[2 * k + 1]), b));
                            const __nv_bfloat162 p = __floats2bfloat162_rn(f2lo(h), f2hi(h));
                            w[k] = *reinterpret_cast<const uint32_t*>(&p);
                        }
                        store(nb, f, w);
                        publish(nb, blk);
                        if (TRAIN) store_t(n.HT[g < 4 ? g : 0], f, w);
                    } else {
                        // dL/dZ = (W^T G) gelu'(Z) of hidden layer l
                        const int l = g > 4 ? 8 - g : 0;
                        float v[8], z[8];
                        tmem_ld8(trow + (uint32_t)(kAccBwd + 64 * (g & 1) + blk * kNS), v);
                        tmem_ld8(trow + (uint32_t)(64 * l + blk * kNS), z);
                        const f32x2 b = f2(bias[l][blk], bias[l][blk]);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const f32x2 h = f2mul(f2(v[2 * k], v[2 * k + 1]), gelu_grad_pair(f2add(f2(z[2 * k], z[2 * k + 1]), b)));
                            const __nv_bfloat162 p = __floats2bfloat162_rn(f2lo(h), f2hi(h));
                            w[k] = *reinterpret_cast<const uint32_t*>(&p);
                        }
                        if (g + 1 < kProducts) {
                            store(nb, f, w);
                            publish(nb, blk);
                        }
                        store_t(n.GT[l], f, w);
                    }
                }
            }
            stop = stop || __any_sync(0xffffffffu, abort_flag != 0);
        }
    } else if (TRAIN && blockIdx.x == 0 && lane == 0) {
        // ---- the step's learning rate and Adam bias corrections (the double-precision
        // formula the single-step call evaluates on the host), and the loss sum cleared
        *n.loss = 0.0;
        if (a.lr) {
            TrainState* ts = n.ts;
            const int k = ts->k + 1;
            const double t = (double)(ts->t0 + k);
            ts->k = k;
            ts->lr = a.lr[k - 1];
            ts->c1 = (float)(1.0 / (1.0 - pow((double)a.beta1, t)));
            ts->c2 = (float)(1.0 / (1.0 - pow((double)a.beta2, t)));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_flag && tid == 0 && n.err) atomicOr(n.err, 8);
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// Weight gradients [dW_l | db_l] = G_l^T [H_{l-1} | 1] of every layer in one launch: a CTA
// per (layer, 128 x NT tile, K split), both operands K-major along the batch (GT, HT: the
// pass kernel left them transposed), 64-wide K slices by TMA (128-byte swizzled) into a
// ring of three stages.  Each split stores its partial transposed (ldp outputs a row, one row
// an input column), so that a warp's 32 accumulator lanes are 128 contiguous bytes;
// k_mlp_update adds them in split order.  The last CTAs of a member, one an output, sum the
// squared errors (the Y - T that the pass kernel left) in FP64.
// ---------------------------------------------------------------------------------------
constexpr int kDwThreads = 256;
constexpr int kDwStages = 3;
constexpr int kDwLossCtas = SALEC_MLP_OUT_N;

template <int NMEM>
struct DwArgs {
    NetMaps maps[NMEM];
    NetPtrs net[NMEM];
    DwPlan plan;
    int B;
};

template <int NMEM>
__global__ void __launch_bounds__(kDwThreads) k_mlp_dw(const __grid_constant__ DwArgs<NMEM> a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[kDwStages], empty[kDwStages];
    __shared__ uint32_t tmem_holder;
    __shared__ int ok_flag;
    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int member = NMEM == 1 ? 0 : blockIdx.y;
    const NetPtrs& n = a.net[member];
    if ((int)blockIdx.x >= a.plan.ctas) {
        __shared__ double part[kDwThreads / 32];
        const float* D = n.D + (long)((int)blockIdx.x - a.plan.ctas) * n.ldT;
        double s = 0.0;
        for (int m = tid; m < a.B; m += kDwThreads) s += (double)D[m] * (double)D[m];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) part[warp] = s;
        __syncthreads();
        if (tid == 0) {
            for (int k = 1; k < kDwThreads / 32; ++k) s += part[k];
            atomicAdd(n.loss, s);
        }
        return;
    }
    int l = 4;
    while (l > 0 && (int)blockIdx.x < a.plan.layer[l].first) --l;
    const DwLayer& L = a.plan.layer[l];
    const CUtensorMap* mapA = &a.maps[member].gt[l];
    const CUtensorMap* mapB = &a.maps[member].ht[l];
    const int idx = (int)blockIdx.x - L.first, tiles = L.mt * L.ntn;
    const int split = idx / tiles, tile = idx - split * tiles;
    const int tm0 = (tile % L.mt) * kBM, n0 = (tile / L.mt) * L.nt, NT = L.nt;
    const int kb = split * L.kchunk, ke = min(a.B, kb + L.kchunk), nk = (ke - kb + kBK - 1) / kBK;
    const uint32_t a_bytes = kBM * kBK * 2, b_bytes = (uint32_t)NT * kBK * 2;
    const uint32_t stage_bytes = a_bytes + (b_bytes + 1023u) / 1024u * 1024u;
    const uint32_t cols = NT <= 32 ? 32u : NT <= 64 ? 64u : NT <= 128 ? 128u : 256u;

    if (tid == 0) {
        for (int k = 0; k < kDwStages; ++k) { mbar_init(&full[k], 1); mbar_init(&empty[k], 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        ok_flag = 1;
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                     "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;

    if (warp == 0 && elect_one()) {
        const uint32_t idesc = idesc_bf16(kBM, NT);
        const uint32_t base = smem_u32(smem);
        const uint64_t a_desc = sdesc_sw128(base), b_desc = sdesc_sw128(base + a_bytes);
        auto load = [&](int kt) {
            const int st = kt % kDwStages;
            mbar_expect_tx(&full[st], a_bytes + b_bytes);
            tma_load_2d(base + st * stage_bytes, mapA, kb + kt * kBK, tm0, &full[st]);
            tma_load_2d(base + st * stage_bytes + a_bytes, mapB, kb + kt * kBK, n0, &full[st]);
        };
        bool good = true;
        int loaded = 0, committed = 0;
        for (; loaded < nk && loaded < kDwStages && !stalled(loaded); ++loaded) load(loaded);
        for (int kt = 0; kt < nk; ++kt) {
            const int st = kt % kDwStages;
            const uint32_t par = (uint32_t)(kt / kDwStages) & 1u;
            if (!mbar_wait_short(&full[st], par)) { good = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t off = (uint64_t)st * (stage_bytes >> 4);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
                mma_bf16(tmem, a_desc + off + kk * 2, b_desc + off + kk * 2, idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            mma_commit(&empty[st]);
            ++committed;
            if (loaded < nk && !stalled(loaded)) {
                if (!mbar_wait(&empty[st], par)) { good = false; break; }
                load(loaded++);
            }
        }
        if (good) good = mbar_wait(&empty[(nk - 1) % kDwStages], (uint32_t)((nk - 1) / kDwStages) & 1u);
        if (!good) {
            if (n.err) atomicOr(n.err, 16);
            // copies and MMAs still in flight finish first
            for (int k = committed; k < loaded; ++k) mbar_drain(&full[k % kDwStages], (uint32_t)(k / kDwStages) & 1u);
            if (committed > 0) mbar_drain(&empty[(committed - 1) % kDwStages], (uint32_t)((committed - 1) / kDwStages) & 1u);
            ok_flag = 0;
        }
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok_flag) {
        const int q = warp & 3, m = tm0 + q * 32 + lane;
        float* part = n.part[l] + (long)split * L.pstep + (long)n0 * L.ldp + m;
        for (int c0 = (warp >> 2) * 16; c0 < NT; c0 += 16 * (kDwThreads / 128)) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (n0 + c0 + j < L.N) part[(long)(c0 + j) * L.ldp] = v[j];
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// Split-K partials added in split order; the sum is the gradient (ADAM false: stored), or
// goes straight into Adam on the FP32 master parameters and the two BF16 copies of the
// weights.  A block takes 32 outputs x 32 input columns of a layer: the partials and the
// transposed weights run along the outputs, the parameters along the inputs, and the sums
// (then the new weights) change over in shared memory, so that every access is coalesced.
// ---------------------------------------------------------------------------------------
constexpr int kUpThreads = 256;

template <int NMEM>
struct UpdateArgs {
    NetPtrs net[NMEM];
    DwPlan plan;
    float* grad;             // ADAM false: destination
    AdamArgs adam;
};

template <int NMEM, bool ADAM>
__global__ void __launch_bounds__(kUpThreads) k_mlp_update(const __grid_constant__ UpdateArgs<NMEM> a)
{
    __shared__ float tile[32][33];
    const NetPtrs& n = a.net[NMEM == 1 ? 0 : blockIdx.y];
    int l = 4;
    while (l > 0 && (int)blockIdx.x < a.plan.layer[l].ufirst) --l;
    const DwLayer& L = a.plan.layer[l];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ni = L.N - 1;
    const int no32 = (L.M + 31) / 32, idx = (int)blockIdx.x - L.ufirst;
    const int o0 = (idx % no32) * 32, c0 = (idx / no32) * 32;
    constexpr int R = 32 / (kUpThreads / 32);         // rows of the tile a warp takes
    // lane = output
    float g[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int c = c0 + w * R + r;
        const float* part = n.part[l] + (long)c * L.ldp + o0 + lane;
        float p[kMaxSplit];
#pragma unroll
        for (int s = 0; s < kMaxSplit; ++s) p[s] = s < L.S && c < L.N ? part[s * L.pstep] : 0.0f;
        g[r] = 0.0f;
#pragma unroll
        for (int s = 0; s < kMaxSplit; ++s)
            if (s < L.S) g[r] += p[s];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) tile[w * R + r][lane] = g[r];
    __syncthreads();
    // lane = input column
    const int c = c0 + lane;
    float lr = a.adam.lr, c1 = a.adam.c1, c2 = a.adam.c2;
    if (ADAM && a.adam.table) {
        lr = n.ts->lr;
        c1 = n.ts->c1;
        c2 = n.ts->c2;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int o = o0 + w * R + r;
        if (o >= L.M || c >= L.N) continue;
        const long i = c < ni ? L.woff + (long)o * ni + c : L.boff + o;
        const float gr = tile[lane][w * R + r];
        if (!ADAM) {
            a.grad[i] = gr;
            continue;
        }
        // multiply-adds written out, so that every instantiation rounds alike
        const float mi = __fmaf_rn(1.0f - a.adam.beta1, gr, __fmul_rn(a.adam.beta1, n.m1[i]));
        const float vi = __fmaf_rn(__fmul_rn(1.0f - a.adam.beta2, gr), gr, __fmul_rn(a.adam.beta2, n.m2[i]));
        n.m1[i] = mi;
        n.m2[i] = vi;
        const float th = n.theta[i] - __fmul_rn(lr, __fmul_rn(mi, c1)) / (sqrtf(__fmul_rn(vi, c2)) + a.adam.eps);
        n.theta[i] = th;
        tile[lane][w * R + r] = th;
        if (c < ni) n.wbf[L.wbf_off + (long)o * L.w_ld + c] = __float2bfloat16_rn(th);
    }
    if (!ADAM || l == 0) return;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int cr = c0 + w * R + r, o = o0 + lane;
        if (o < L.M && cr < ni) n.wbfT[L.wbfT_off + (long)cr * L.wt_ld + o] = __float2bfloat16_rn(tile[w * R + r][lane]);
    }
}

// ---------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------
namespace {

// the device's SM count, with the kernels' shared-memory attributes set on first use
cudaError_t device_setup(int* sms)
{
    static int count[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!count[dev]) {
        auto set = [&](auto* k, size_t bytes) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        };
        set(k_mlp_pass<1, false>, kPassSmem);
        set(k_mlp_pass<1, true>, kPassSmem);
        set(k_mlp_pass<kMaxGroup, true>, kPassSmem);
        set(k_mlp_dw<1>, dw_smem_bytes(256));
        set(k_mlp_dw<kMaxGroup>, dw_smem_bytes(256));
        int c = 0;
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        count[dev] = c;
    }
    *sms = count[dev];
    return cudaSuccess;
}

template <int NMEM>
cudaError_t launch_pass(const TrainNet* const* nets, int count, const DwPlan& plan, const TrainLaunch& t, cudaStream_t s)
{
    PassArgs<NMEM> ca;
    DwArgs<NMEM> da;
    for (int k = 0; k < count; ++k) {
        ca.maps[k] = da.maps[k] = nets[k]->maps;
        ca.net[k] = da.net[k] = nets[k]->p;
    }
    ca.x = nullptr;
    ca.y = nullptr;
    ca.t = t.t;
    ca.lr = t.lr;
    ca.beta1 = t.adam.beta1;
    ca.beta2 = t.adam.beta2;
    ca.grad_scale = 2.0f / ((float)t.B * (float)SALEC_MLP_OUT_N);
    ca.B = da.B = t.B;
    da.plan = plan;
    const unsigned tiles = (unsigned)((t.B + kNS - 1) / kNS);
    k_mlp_pass<NMEM, true><<<dim3(tiles, (unsigned)count), kPassThreads, kPassSmem, s>>>(ca);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_mlp_dw<NMEM><<<dim3((unsigned)(plan.ctas + kDwLossCtas), (unsigned)count), kDwThreads, dw_smem_bytes(plan.max_nt), s>>>(da);
    return cudaGetLastError();
}

template <int NMEM, bool ADAM>
cudaError_t launch_update(const TrainNet* const* nets, int count, const DwPlan& plan, float* grad, const AdamArgs& adam,
                          cudaStream_t s)
{
    UpdateArgs<NMEM> u;
    for (int k = 0; k < count; ++k) u.net[k] = nets[k]->p;
    u.plan = plan;
    u.grad = grad;
    u.adam = adam;
    k_mlp_update<NMEM, ADAM><<<dim3((unsigned)plan.ublocks, (unsigned)count), kUpThreads, 0, s>>>(u);
    return cudaGetLastError();
}

}  // namespace

size_t dw_smem_bytes(int nt) { return (size_t)kDwStages * (kBM * kBK * 2 + ((size_t)nt * kBK * 2 + 1023) / 1024 * 1024) + 1024; }

// The plan of a batch's weight gradients: per layer 128-row by NT-column tiles (two column
// tiles of 144 for 257 columns) and K split over up to kMaxSplit CTAs a tile in whole
// 64-wide slices, at least two each: the few tiles of a layer (1 to 4) would leave most SMs
// idle otherwise.
DwPlan plan_dw(int B, int sms)
{
    DwPlan p = {};
    long woff = 0, wbf = 0, wbfT = 0;
    const int dims[6] = {5, kHidden, kHidden, kHidden, kHidden, SALEC_MLP_OUT_N};
    for (int l = 0; l < 5; ++l) {
        DwLayer& L = p.layer[l];
        const int ni = dims[l], no = dims[l + 1];
        L.M = no;
        L.N = ni + 1;
        L.mt = (no + kBM - 1) / kBM;
        L.ntn = (L.N + 255) / 256;
        L.nt = ((L.N + L.ntn - 1) / L.ntn + 15) / 16 * 16;
        L.ntn = (L.N + L.nt - 1) / L.nt;
        L.ldp = L.mt * kBM;
        L.pstep = (long)L.N * L.ldp;
        const int slices = (B + kBK - 1) / kBK;
        int S = 1;
        if (B >= 4 * kBK && L.mt * L.ntn < sms / 2) {
            S = (sms + L.mt * L.ntn - 1) / (L.mt * L.ntn);
            S = S < kMaxSplit ? S : kMaxSplit;
            S = S < (slices + 1) / 2 ? S : (slices + 1) / 2;
        }
        L.kchunk = (slices + S - 1) / S * kBK;
        L.S = (B + L.kchunk - 1) / L.kchunk;
        L.first = p.ctas;
        p.ctas += L.mt * L.ntn * L.S;
        L.ufirst = p.ublocks;
        p.ublocks += ((L.M + 31) / 32) * ((L.N + 31) / 32);
        if (L.nt > p.max_nt) p.max_nt = L.nt;
        L.woff = woff;
        L.boff = woff + (long)no * ni;
        woff = L.boff + no;
        L.w_ld = l == 0 ? 8 : ni;
        L.wbf_off = wbf;
        wbf += (long)no * L.w_ld;
        L.wt_ld = (no + 7) / 8 * 8;
        L.wbfT_off = l > 0 ? wbfT : 0;
        if (l > 0) wbfT += (long)ni * L.wt_ld;
    }
    return p;
}

// floats of layer l's partials at the largest split
size_t dw_part_floats(int l)
{
    const DwPlan p = plan_dw(1 << 20, 1 << 20);
    return (size_t)kMaxSplit * p.layer[l].pstep;
}

cudaError_t make_weight_maps(TrainNet* n)
{
    const NetPtrs& p = n->p;
    const DwPlan q = plan_dw(kBK, 1);
    bool ok = true;
    for (int l = 1; l < 5; ++l) {
        const DwLayer& L = q.layer[l];
        ok = ok && make_map_sw128(&n->maps.w[l - 1], p.wbf + L.wbf_off, L.M, L.N - 1, L.w_ld, kBM);
        ok = ok && make_map_sw128(&n->maps.wt[4 - l], p.wbfT + L.wbfT_off, L.N - 1, L.M, L.wt_ld, kBM);
    }
    n->maps_B = 0;
    return ok ? cudaSuccess : cudaErrorNotSupported;
}

cudaError_t make_batch_maps(TrainNet* n, int B)
{
    if (n->maps_B == B) return cudaSuccess;
    const NetPtrs& p = n->p;
    const DwPlan q = plan_dw(B, 1);
    bool ok = true;
    for (int l = 0; l < 5; ++l) {
        const DwLayer& L = q.layer[l];
        ok = ok && make_map_sw128(&n->maps.gt[l], p.GT[l], L.M, B, p.ldT, kBM);
        ok = ok && make_map_sw128(&n->maps.ht[l], l > 0 ? p.HT[l - 1] : p.XT, L.N, B, p.ldT, L.nt);
    }
    n->maps_B = ok ? B : 0;
    return ok ? cudaSuccess : cudaErrorNotSupported;
}

cudaError_t launch_train_pass(TrainNet* const* nets, int count, const TrainLaunch& t, float* grad, cudaStream_t s)
{
    if (count < 1 || count > kMaxGroup) return cudaErrorInvalidValue;
    int sms = 0;
    cudaError_t e = device_setup(&sms);
    for (int k = 0; k < count && e == cudaSuccess; ++k) e = make_batch_maps(nets[k], t.B);
    if (e != cudaSuccess) return e;
    const DwPlan plan = plan_dw(t.B, sms);
    e = count == 1 ? launch_pass<1>(nets, count, plan, t, s) : launch_pass<kMaxGroup>(nets, count, plan, t, s);
    if (e != cudaSuccess) return e;
    if (grad) return launch_update<1, false>(nets, 1, plan, grad, t.adam, s);
    return count == 1 ? launch_update<1, true>(nets, count, plan, nullptr, t.adam, s)
                      : launch_update<kMaxGroup, true>(nets, count, plan, nullptr, t.adam, s);
}

cudaError_t launch_infer_small(const TrainNet& n, const float* x, int B, float* y, cudaStream_t s, bool* done)
{
    int sms = 0;
    const cudaError_t e = device_setup(&sms);
    *done = false;
    if (e != cudaSuccess) return e;
    // Up to four tiles of 32 samples an SM: 128 samples 13.9 us (the persistent kernel's one CTA
    // for up to 256 samples: 36), 4864 samples 14.5 us (53), 14592 37 us (53), 19456 48.7 us
    // (53.6); 29184 samples would take 71 us (55).
    if ((B + kNS - 1) / kNS > 4 * sms) return cudaSuccess;
    *done = true;
    PassArgs<1> ca;
    ca.maps[0] = n.maps;
    ca.net[0] = n.p;
    ca.x = x;
    ca.y = y;
    ca.t = ca.lr = nullptr;
    ca.beta1 = ca.beta2 = ca.grad_scale = 0.0f;
    ca.B = B;
    // placed while the kernel before it in the stream ends (the kernel waits for that one
    // before it reads anything): a series of forward passes of 255 samples takes 10.6 us each
    // instead of 14.3
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)((B + kNS - 1) / kNS));
    c.blockDim = dim3(kPassThreads);
    c.dynamicSmemBytes = kPassSmem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k_mlp_pass<1, false>, ca);
}

}  // namespace mlp
}  // namespace salec
