// mlp_kernels.cu -- BF16 tensor-core kernels of the crater-surrogate MLP (5 -> 4 x 256 GELU
// -> 66): the bare GEMM, the inference pass over many samples, and the conversions of inputs
// and weights.  The training step and inference over few samples are in mlp_train.cu.
//
// The GEMM:
//     C[m][n] = sum_k A(m, k) B(n, k),   A(m, k) = A[m a_sm + k a_sk],  B(n, k) = B[n b_sn + k b_sk]
// with BF16 operands and an FP32 accumulator.  A CTA owns a 128 x NT tile of C (NT <= 128, a
// multiple of 16).  Its 128 threads gather 128 x 64 and NT x 64 operand tiles from global
// memory (any strides, zero outside the matrix) into shared memory in the tensor cores'
// canonical K-major layout without swizzle: 8-row x 16-byte core matrices, 128 bytes each,
// adjacent along M/N (stride 128 B) and then along K (stride rows x 16 B).  One elected
// thread issues tcgen05.mma (kind::f16, BF16 x BF16 -> FP32, M = 128, N = NT, K = 16) four
// times per 64-wide K slice, accumulating in tensor memory; tcgen05.commit arrives on the
// stage's mbarrier when those MMAs have read their operands, which frees the stage for the
// next gather (two stages).  The epilogue reads the accumulator back with tcgen05.ld (warp w
// owns TMEM lanes 32w..32w+31, i.e. rows 32w..32w+31 of the tile).
//
// Operands that are K-major rows of 16-byte multiples take a second kernel, k_gemm_bf16_tma,
// fed by TMA (below).
//
// Every wait on an mbarrier is bounded; on expiry the kernel records an error code, waits
// (bounded again) for its own MMAs, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mlp_device.cuh"

namespace salec {
namespace mlp {

// Gather 8 consecutive-in-k elements of row r into one 16-byte core-matrix row.
__device__ __forceinline__ uint4 gather8(const __nv_bfloat16* __restrict__ P, long s_r, long s_k, int r, int R, int k0,
                                         int K)
{
    union { uint4 u; __nv_bfloat16 h[8]; } w;
    if (r < R && s_k == 1 && k0 + 8 <= K && ((reinterpret_cast<uintptr_t>(P + r * s_r + k0) & 15) == 0)) {
        w.u = *reinterpret_cast<const uint4*>(P + r * s_r + k0);
        return w.u;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int k = k0 + e;
        w.h[e] = (r < R && k < K) ? P[r * s_r + (long)k * s_k] : __float2bfloat16_rn(0.0f);
    }
    return w.u;
}

// Epilogue: warp w reads TMEM lanes 32w..32w+31 (rows m0 + 32w + lane of the tile), 16
// columns at a time.  A row's 16 columns go out as 16-byte stores when they lie inside N and
// the rows are 16-byte aligned (each thread writes its own row: whole sectors, merged in
// L2); otherwise element by element.
__device__ __forceinline__ void epilogue(const GemmArgs& g, uint32_t tmem, int m0, int n0, int NT, bool any_k)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m = m0 + warp * 32 + lane;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    const bool vec = ((g.ldc * 4) & 15) == 0 && ((reinterpret_cast<uintptr_t>(g.C) & 15) == 0);
    for (int c0 = 0; c0 < NT; c0 += 16) {
        float v[16];
        tmem_ld16(trow + (uint32_t)c0, v);
        if (m >= g.M) continue;
        const int nb = n0 + c0;
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = any_k ? v[j] : 0.0f;    // K = 0: empty sum
        if (nb + 16 <= g.N && vec) {
            float4* dst = reinterpret_cast<float4*>(g.C + (long)m * g.ldc + nb);
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (nb + j < g.N) g.C[(long)m * g.ldc + nb + j] = v[j];
        }
    }
}

__global__ void __launch_bounds__(kGemmThreads) k_gemm_bf16(GemmArgs g)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // stage s: A tile at s * stage_bytes, B tile right after it
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t bars[2];
    __shared__ uint32_t tmem_holder;

    const int tid = threadIdx.x, warp = tid >> 5;
    const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * g.nt;
    const int NT = g.nt;
    const uint32_t a_bytes = kBM * kBK * 2, b_bytes = (uint32_t)NT * kBK * 2;
    const uint32_t stage_bytes = a_bytes + b_bytes;
    const uint32_t tmem_cols = g.tmem_cols;

    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;
    const uint32_t idesc = idesc_bf16(kBM, NT);

    const int nk = (g.K + kBK - 1) / kBK;
    bool ok = true;
    int issued = 0;                       // K slices whose MMAs were committed
    for (int kt = 0; kt < nk; ++kt) {
        const int s = kt & 1;
        // uniform decision: a barrier whose result every thread sees
        if (kt >= 2 && !__syncthreads_and(mbar_wait(&bars[s], ((kt - 2) >> 1) & 1))) { ok = false; break; }
        unsigned char* sa = smem + s * stage_bytes;
        unsigned char* sb = sa + a_bytes;
        const int k0 = kt * kBK;
        // A: thread tid gathers row tid; core matrix (row group rg, k group kg) at kg*2048 + rg*128
#pragma unroll
        for (int kg = 0; kg < 8; ++kg) {
            const uint4 w = gather8(g.A, g.a_sm, g.a_sk, m0 + tid, g.M, k0 + 8 * kg, g.K);
            *reinterpret_cast<uint4*>(sa + kg * (kBM * 16) + (tid >> 3) * 128 + (tid & 7) * 16) = w;
        }
        for (int r = tid; r < NT; r += kGemmThreads) {
#pragma unroll
            for (int kg = 0; kg < 8; ++kg) {
                const uint4 w = gather8(g.B, g.b_sn, g.b_sk, n0 + r, g.N, k0 + 8 * kg, g.K);
                *reinterpret_cast<uint4*>(sb + kg * (NT * 16) + (r >> 3) * 128 + (r & 7) * 16) = w;
            }
        }
        // generic-proxy writes -> visible to the tensor cores' (async proxy) reads
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(sa), b0 = smem_u32(sb);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk) {
                // K = 16 spans two core matrices along K
                const uint64_t ad = sdesc(a0 + kk * 2 * (kBM * 16), kBM * 16, 128);
                const uint64_t bd = sdesc(b0 + kk * 2 * (NT * 16), NT * 16, 128);
                mma_bf16(tmem, ad, bd, idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            }
            mma_commit(&bars[s]);
        }
        issued = kt + 1;
    }
    // all MMAs done: wait for the last commit of each stage (the later one covers every
    // earlier MMA; waiting for both leaves no arrive pending when the CTA exits)
    if (ok && issued >= 2) ok = __syncthreads_and(mbar_wait(&bars[(issued - 2) & 1], ((issued - 2) >> 1) & 1));
    if (ok && issued >= 1) ok = __syncthreads_and(mbar_wait(&bars[(issued - 1) & 1], ((issued - 1) >> 1) & 1));
    if (!ok) {
        if (g.err && tid == 0) atomicOr(g.err, 1);
        // MMAs still in flight finish before their memory goes away
        if (issued >= 1) mbar_drain(&bars[(issued - 1) & 1], ((issued - 1) >> 1) & 1);
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    if (ok) epilogue(g, tmem, m0, n0, NT, nk > 0);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// The same contraction when both operands are K-major rows (A[m][k], B[n][k], rows of
// 16-byte multiples).  One thread streams K slices into a ring of
// kStages shared-memory stages with TMA (cp.async.bulk.tensor, 2-D maps, boxes of 8
// elements x rows: one box is one column of core matrices, 16 bytes x rows, exactly the
// canonical no-swizzle K-major layout), each stage's mbarrier completing on the bytes
// delivered; the same thread issues the MMAs of a slice as soon as it lands and refills
// the stage once tcgen05.commit reports those MMAs done.  The tile is 128 x NT with NT up
// to 256 (a whole hidden layer, so the activations are read once).
// ---------------------------------------------------------------------------------------
constexpr int kStages = 4;
constexpr int kMaxNT_TMA = 256;

__global__ void __launch_bounds__(kGemmThreads) k_gemm_bf16_tma(const __grid_constant__ CUtensorMap mapA,
                                                                const __grid_constant__ CUtensorMap mapB, GemmArgs g)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[kStages], empty[kStages];
    __shared__ uint32_t tmem_holder;
    __shared__ int ok_flag;

    const int tid = threadIdx.x, warp = tid >> 5;
    const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * g.nt;
    const int NT = g.nt;
    const uint32_t a_bytes = kBM * kBK * 2, b_bytes = (uint32_t)NT * kBK * 2;
    const uint32_t stage_bytes = a_bytes + b_bytes;
    const uint32_t tmem_cols = g.tmem_cols;
    const int nk = (g.K + kBK - 1) / kBK;
    const int ns = g.stages;              // ring stages in use (1..kStages), set by the launcher

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapB)) : "memory");
        ok_flag = 1;
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;

    if (tid == 0) {
        const uint32_t idesc = idesc_bf16(kBM, NT);
        const uint32_t base = smem_u32(smem);
        auto load_slice = [&](int kt) {
            const int st = kt % ns;
            const uint32_t sa = base + st * stage_bytes, sb = sa + a_bytes;
            mbar_expect_tx(&full[st], stage_bytes);
            const int k0 = kt * kBK;
#pragma unroll
            for (int kg = 0; kg < kBK / 8; ++kg) {
                tma_load_2d(sa + kg * (kBM * 16), &mapA, k0 + 8 * kg, m0, &full[st]);
                tma_load_2d(sb + kg * (NT * 16), &mapB, k0 + 8 * kg, n0, &full[st]);
            }
        };
        bool good = true;
        int loaded = 0, committed = 0;  // slices whose copies were issued, whose MMAs were committed
        for (; loaded < nk && loaded < ns && !stalled(loaded); ++loaded) load_slice(loaded);
        for (int kt = 0; kt < nk && good; ++kt) {
            const int st = kt % ns;
            const uint32_t par = (uint32_t)(kt / ns) & 1u;
            if (!mbar_wait(&full[st], par)) { good = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = base + st * stage_bytes, b0 = a0 + a_bytes;
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk) {
                const uint64_t ad = sdesc(a0 + kk * 2 * (kBM * 16), kBM * 16, 128);
                const uint64_t bd = sdesc(b0 + kk * 2 * (NT * 16), NT * 16, 128);
                mma_bf16(tmem, ad, bd, idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            }
            mma_commit(&empty[st]);
            committed = kt + 1;
            if (loaded < nk && !stalled(loaded)) {
                // the stage is refilled once its MMAs have read it
                if (!mbar_wait(&empty[st], par)) { good = false; break; }
                load_slice(loaded++);
            }
        }
        // the last commit covers every MMA; wait for it (bounded)
        if (good && committed > 0)
            good = mbar_wait(&empty[(committed - 1) % ns], (uint32_t)((committed - 1) / ns) & 1u);
        if (!good) {
            if (g.err) atomicOr(g.err, 2);
            // copies and MMAs still in flight finish first
            for (int k = committed; k < loaded; ++k) mbar_drain(&full[k % ns], (uint32_t)(k / ns) & 1u);
            if (committed > 0) mbar_drain(&empty[(committed - 1) % ns], (uint32_t)((committed - 1) / ns) & 1u);
            ok_flag = 0;
        }
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok_flag) epilogue(g, tmem, m0, n0, NT, nk > 0);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// Shapes of the whole-network inference kernel below: hidden width 256, outputs padded to
// 80, an activation tile of 128 x 256 BF16, a weight slice of 256 rows x 64 K.
// ---------------------------------------------------------------------------------------
constexpr int kFusedHid = 256;
constexpr int kFusedOutPad = 80;      // 66 outputs padded to a multiple of 16
constexpr uint32_t kHBytes = kBM * kFusedHid * 2;          // 65536
constexpr uint32_t kWStageBytes = kFusedHid * kBK * 2;     // 32768

// ---------------------------------------------------------------------------------------
// The inference pass, persistent and warp-specialised: one CTA per SM takes 128-sample
// tiles two at a time and alternates them, so that the tensor cores work on one tile while
// the epilogue warps work on the other.  Per tile x (0, 1): an activation buffer H_x (BF16,
// canonical K-major, 64 KB) and a 256-column accumulator in tensor memory (both tiles: all
// 512 columns).  Warp 0 streams the weight slices (64-wide K slices, 256 rows x 128 bytes)
// with TMA into a 2-stage ring, 128-byte swizzled; warp 1 issues the MMAs of job (x, layer)
// once H_x holds that layer's input and frees each ring stage by tcgen05.commit; warps
// 2-17 run the epilogue of job (x, layer) when its accumulator is complete: gelu(Z + b) as
// BF16 back into H_x (the next layer's input), or Y for the output layer followed by the
// inputs of the tile's successor.  Jobs run in the order (pair, layer, tile) in every role.
// mbarriers: ring stage full / empty, accumulator x complete, H_x ready (16 epilogue warps).
// Every wait is bounded; a wait that runs out raises a shared abort flag that ends every
// role's loop.  However its loop ends, warp 0 waits for its copies and warp 1, on a barrier of
// its own behind every MMA it issued, for its MMAs; then the tensor memory is freed.
// ---------------------------------------------------------------------------------------
constexpr int kPPThreads = 18 * 32;
constexpr uint32_t kW1Bytes = kFusedHid * 16 * 2;          // layer-1 weights, K padded to 16
constexpr int kPPStages = 2;

size_t pp_smem_bytes() { return 2 * (size_t)kHBytes + kPPStages * (size_t)kWStageBytes + kW1Bytes + 1024; }

struct PPArgs {
    int B, ntiles, npairs;
    const __nv_bfloat16* X;
    int ld_x;
    const __nv_bfloat16* W1;
    const float* bias[5];
    float* Y;
    int* err;
};

__global__ void __launch_bounds__(kPPThreads, 1) k_mlp_forward_pp(const __grid_constant__ CUtensorMap mW2,
                                                                 const __grid_constant__ CUtensorMap mW3,
                                                                 const __grid_constant__ CUtensorMap mW4,
                                                                 const __grid_constant__ CUtensorMap mW5,
                                                                 PPArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* Hbuf = smem;                                   // H_0, H_1
    unsigned char* Wring = smem + 2 * kHBytes;                    // 2 stages, 1024-aligned
    unsigned char* W1s = Wring + kPPStages * kWStageBytes;        // layer-1 weights
    __shared__ __align__(16) float sbias[4 * kFusedHid + kFusedOutPad];
    __shared__ uint64_t wfull[kPPStages], wempty[kPPStages], accfull[2], hready[2], drained;
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x;
    if (tid == 0) {
        for (int k = 0; k < kPPStages; ++k) { mbar_init(&wfull[k], 1); mbar_init(&wempty[k], 1); }
        for (int x = 0; x < 2; ++x) { mbar_init(&accfull[x], 1); mbar_init(&hready[x], 16); }
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
    for (int k = tid; k < 4 * kFusedHid + kFusedOutPad; k += kPPThreads) {
        const int l = k / kFusedHid, n = k - l * kFusedHid;
        sbias[k] = l < 4 ? a.bias[l][n] : (n < SALEC_MLP_OUT_N ? a.bias[4][n] : 0.0f);
    }
    for (int n = tid; n < kFusedHid; n += kPPThreads) {
        *reinterpret_cast<uint4*>(W1s + cm_off(n, 0, kFusedHid)) = *reinterpret_cast<const uint4*>(a.W1 + (long)n * a.ld_x);
        *reinterpret_cast<uint4*>(W1s + cm_off(n, 1, kFusedHid)) = make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;
    // tile of slot x of the k-th pair of this CTA (-1: none)
    auto tile_of = [&](int k, int x) {
        const int t = 2 * (blockIdx.x + k * G) + x;
        return (blockIdx.x + k * G < a.npairs && t < a.ntiles) ? t : -1;
    };
    const int npairs_mine = a.npairs > (int)blockIdx.x ? (a.npairs - 1 - (int)blockIdx.x) / G + 1 : 0;

    if (warp == 0) {
        // ---- weight producer ----
        if (lane == 0) {
            int fills[kPPStages] = {0, 0};
            int stage = 0;
            for (int k = 0; k < npairs_mine && !abort_flag; ++k)
                for (int l = 1; l < 5 && !abort_flag; ++l)
                    for (int x = 0; x < 2 && !abort_flag; ++x) {
                        if (tile_of(k, x) < 0) continue;
                        const int N = l == 4 ? kFusedOutPad : kFusedHid;
                        const CUtensorMap* map = l == 1 ? &mW2 : l == 2 ? &mW3 : l == 3 ? &mW4 : &mW5;
                        for (int kt = 0; kt < kFusedHid / kBK && !stalled(fills[0] + fills[1]); ++kt) {
                            if (fills[stage] > 0 && !mbar_wait_idle(&wempty[stage], (uint32_t)(fills[stage] - 1) & 1u)) {
                                abort_flag = 1;
                                break;
                            }
                            mbar_expect_tx(&wfull[stage], (uint32_t)N * 128u);
                            tma_load_2d(smem_u32(Wring + stage * kWStageBytes), map, kt * kBK, 0, &wfull[stage]);
                            ++fills[stage];
                            stage ^= 1;
                        }
                    }
            // the last copies of each stage land before the CTA's memory can go away
            for (int st = 0; st < kPPStages; ++st)
                if (fills[st] > 0) mbar_drain(&wfull[st], (uint32_t)(fills[st] - 1) & 1u);
        }
    } else if (warp == 1) {
        // ---- MMA issuer ----
        if (lane == 0) {
            int used[kPPStages] = {0, 0}, hwait[2] = {0, 0};
            int stage = 0;
            const uint32_t w1 = smem_u32(W1s);
            for (int k = 0; k < npairs_mine && !abort_flag; ++k)
                for (int l = 0; l < 5 && !abort_flag; ++l)
                    for (int x = 0; x < 2 && !abort_flag; ++x) {
                        if (tile_of(k, x) < 0) continue;
                        if (!mbar_wait_idle(&hready[x], (uint32_t)(hwait[x]++) & 1u)) { abort_flag = 1; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const int N = l == 4 ? kFusedOutPad : kFusedHid;
                        const uint32_t idesc = idesc_bf16(kBM, N);
                        const uint32_t acc = tmem + (uint32_t)(x * kFusedHid);
                        const uint32_t hb = smem_u32(Hbuf + x * kHBytes);
                        if (l == 0) {
                            mma_bf16(acc, sdesc(hb, kBM * 16, 128), sdesc(w1, kFusedHid * 16, 128), idesc, 0u);
                        } else {
                            for (int kt = 0; kt < kFusedHid / kBK; ++kt) {
                                if (!mbar_wait(&wfull[stage], (uint32_t)(used[stage]++) & 1u)) { abort_flag = 1; break; }
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                                const uint32_t wb = smem_u32(Wring + stage * kWStageBytes);
#pragma unroll
                                for (int kk = 0; kk < kBK / 16; ++kk) {
                                    const uint64_t ad = sdesc(hb + (kt * (kBK / 8) + 2 * kk) * (kBM * 16), kBM * 16, 128);
                                    mma_bf16(acc, ad, sdesc_sw128(wb + kk * 32), idesc, (kt > 0 || kk > 0) ? 1u : 0u);
                                }
                                mma_commit(&wempty[stage]);
                                stage ^= 1;
                            }
                            if (abort_flag) break;
                        }
                        mma_commit(&accfull[x]);
                    }
            // every MMA issued finishes before the tensor memory is freed
            mma_commit(&drained);
            mbar_drain(&drained, 0u);
        }
    } else {
        // ---- epilogue: warps 2-17; lane quarter q (TMEM lanes 32q..), column quarter cq ----
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const int r = q * 32 + lane;                         // row of the tile
        const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
        int accw[2] = {0, 0};
        // the warp decides together: an abort seen by any lane ends the warp's loop
        auto aborted = [&]() { return __any_sync(0xffffffffu, abort_flag != 0); };
        // inputs of tile t into H_x: X rows (8 BF16 = one core-matrix row), K padded to 16
        auto stage_inputs = [&](int x, int t) {
            if (cq == 0) {
                const int m = t * kBM + r;
                uint4 xv = make_uint4(0u, 0u, 0u, 0u);
                if (m < a.B) xv = *reinterpret_cast<const uint4*>(a.X + (long)m * a.ld_x);
                unsigned char* H = Hbuf + x * kHBytes;
                *reinterpret_cast<uint4*>(H + cm_off(r, 0, kBM)) = xv;
                *reinterpret_cast<uint4*>(H + cm_off(r, 1, kBM)) = make_uint4(0u, 0u, 0u, 0u);
            }
        };
        auto release = [&](int x) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&hready[x]);
        };
        for (int x = 0; x < 2; ++x) {
            const int t = tile_of(0, x);
            if (t < 0) continue;
            stage_inputs(x, t);
            release(x);
        }
        bool stop = aborted();
        for (int k = 0; k < npairs_mine && !stop; ++k)
            for (int l = 0; l < 5 && !stop; ++l)
                for (int x = 0; x < 2 && !(stop = aborted()); ++x) {
                    const int t = tile_of(k, x);
                    if (t < 0) continue;
                    const bool ok = __all_sync(0xffffffffu, mbar_wait(&accfull[x], (uint32_t)(accw[x]++) & 1u));
                    if (!ok) {
                        abort_flag = 1;
                        stop = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t tacc = trow + (uint32_t)(x * kFusedHid);
                    const int m = t * kBM + r;
                    const bool live = m < a.B;
                    const float* bias = sbias + l * kFusedHid;
                    if (l < 4) {
                        unsigned char* H = Hbuf + x * kHBytes;
#pragma unroll 1
                        for (int c0 = cq * 64; c0 < cq * 64 + 64; c0 += 16) {
                            float v[16];
                            tmem_ld16(tacc + (uint32_t)c0, v);
                            uint32_t w[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
                            if (live) {
                                const float4* b4 = reinterpret_cast<const float4*>(bias + c0);
#pragma unroll
                                for (int qq = 0; qq < 4; ++qq) {
                                    const float4 b = b4[qq];
                                    const f32x2 glo = gelu_pair(f2add(f2(v[4 * qq], v[4 * qq + 1]), f2(b.x, b.y)));
                                    const f32x2 ghi = gelu_pair(f2add(f2(v[4 * qq + 2], v[4 * qq + 3]), f2(b.z, b.w)));
                                    const __nv_bfloat162 lo = __floats2bfloat162_rn(f2lo(glo), f2hi(glo));
                                    const __nv_bfloat162 hi = __floats2bfloat162_rn(f2lo(ghi), f2hi(ghi));
                                    w[2 * qq] = *reinterpret_cast<const uint32_t*>(&lo);
                                    w[2 * qq + 1] = *reinterpret_cast<const uint32_t*>(&hi);
                                }
                            }
                            *reinterpret_cast<uint4*>(H + cm_off(r, (c0 >> 3), kBM)) = make_uint4(w[0], w[1], w[2], w[3]);
                            *reinterpret_cast<uint4*>(H + cm_off(r, (c0 >> 3) + 1, kBM)) = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                        release(x);
                    } else {
                        for (int c0 = cq * 16; c0 < kFusedOutPad; c0 += 64) {
                            float v[16];
                            tmem_ld16(tacc + (uint32_t)c0, v);
                            if (live) {
                                float* y = a.Y + (long)m * SALEC_MLP_OUT_N + c0;
#pragma unroll
                                for (int j = 0; j < 16; ++j)
                                    if (c0 + j < SALEC_MLP_OUT_N) y[j] = v[j] + bias[c0 + j];
                            }
                        }
                        // the accumulator is read and H_x is free: the successor's inputs
                        const int tn = tile_of(k + 1, x);
                        if (tn >= 0) {
                            stage_inputs(x, tn);
                            release(x);
                        }
                    }
                }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_flag && tid == 0 && a.err) atomicOr(a.err, 4);
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// FP32 -> BF16 inputs of the first layer: rows of `cols` values into rows of `ld`, the
// padding zero.
__global__ void k_inputs_bf16(const float* __restrict__ x, int rows, int cols, int ld, __nv_bfloat16* __restrict__ y,
                              __nv_bfloat16* __restrict__ yT, long ldT)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long)rows * ld) return;
    const long r = i / ld;
    const int c = (int)(i - r * ld);
    const __nv_bfloat16 v = __float2bfloat16_rn(c < cols ? x[r * cols + c] : 0.0f);
    y[i] = v;
    if (yT && c < cols) yT[(long)c * ldT + r] = v;
}

__global__ void k_train_reset(TrainState* ts, int t0)
{
    ts->k = 0;
    ts->t0 = t0;
}

// BF16 copy of the weights from the FP32 parameters.
__global__ void k_refresh_bf16(const float* __restrict__ theta, long n, const int* __restrict__ wmap,
                               __nv_bfloat16* __restrict__ wbf, const int* __restrict__ wmapT,
                               __nv_bfloat16* __restrict__ wbfT)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int w = wmap[i];
    if (w >= 0) wbf[w] = __float2bfloat16_rn(theta[i]);
    if (wmapT) {
        const int wt = wmapT[i];
        if (wt >= 0) wbfT[wt] = __float2bfloat16_rn(theta[i]);
    }
}

size_t gemm_smem_bytes(int nt) { return 2 * (size_t)(kBM * kBK * 2 + nt * kBK * 2) + 1024; }

namespace {

size_t tma_smem_bytes(int nt, int stages = kStages) { return (size_t)stages * (kBM * kBK * 2 + nt * kBK * 2) + 1024; }

}  // namespace

// SM count and the TMA kernels' shared-memory attribute, per device (set once)
cudaError_t tma_device_setup(int dev, int* sms)
{
    static int sm_count[64] = {};
    static bool attr_tma[64] = {};
    cudaError_t e = cudaSuccess;
    if (!sm_count[dev]) {
        e = cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
    }
    if (!attr_tma[dev]) {
        e = cudaFuncSetAttribute(k_gemm_bf16_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tma_smem_bytes(kMaxNT_TMA));
        if (e != cudaSuccess) return e;
        attr_tma[dev] = true;
    }
    *sms = sm_count[dev];
    return cudaSuccess;
}

// The TMA-fed kernel's plan for one product: tile width, ring stages and tensor-memory
// columns (into g), and the grid (mt row tiles, ntl column tiles).
void plan_tma(GemmArgs& g, int sms, int* mt_out, int* ntl_out)
{
    const int mt = (g.M + kBM - 1) / kBM;
    auto round16 = [](int x) { return (x + 15) / 16 * 16; };
    auto tiles_n = [&](int w) { return (g.N + w - 1) / w; };
    int ntn = tiles_n(kMaxNT_TMA);
    int nt = round16((g.N + ntn - 1) / ntn);
    // narrower tiles (down to 32 columns) until the tiles fill the SMs: the epilogue of a
    // tile is the longest part of a CTA, and it shrinks with it
    while (mt * tiles_n(nt) < sms && nt > 32) {
        ntn *= 2;
        const int w = round16((g.N + ntn - 1) / ntn);
        nt = w > 32 ? w : 32;
    }
    g.nt = nt;
    int cols = 32;
    while (cols < nt) cols <<= 1;
    g.tmem_cols = cols;
    // narrow tiles keep two stages in flight: 41 KB of shared memory, five CTAs per SM, so
    // that concurrent GEMMs overlap
    g.stages = nt <= 64 ? 2 : kStages;
    *mt_out = mt;
    *ntl_out = tiles_n(nt);
}

cudaError_t launch_gemm(const GemmArgs& g0, cudaStream_t s)
{
    GemmArgs g = g0;
    if (g.M <= 0 || g.N <= 0) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    // both operands K-major with 16-byte rows: the TMA-fed kernel
    if (g.K > 0 && g.a_sk == 1 && g.b_sk == 1) {
        int sms = 0, mt = 0, ntl = 0;
        e = tma_device_setup(dev, &sms);
        if (e != cudaSuccess) return e;
        plan_tma(g, sms, &mt, &ntl);
        CUtensorMap ma, mb;
        if (make_map(&ma, g.A, g.M, g.K, g.a_sm, kBM) && make_map(&mb, g.B, g.N, g.K, g.b_sn, g.nt)) {
            k_gemm_bf16_tma<<<dim3((unsigned)mt, (unsigned)ntl), kGemmThreads, tma_smem_bytes(g.nt, g.stages), s>>>(ma, mb, g);
            return cudaGetLastError();
        }
    }
    const int nt = ((g.N < kMaxNT ? g.N : kMaxNT) + 15) / 16 * 16;
    g.nt = nt;
    int cols = 32;
    while (cols < nt) cols <<= 1;
    g.tmem_cols = cols;
    const size_t smem = gemm_smem_bytes(nt);
    // the attribute is per device
    static bool attr_set[64] = {};
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(k_gemm_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem_bytes(kMaxNT));
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    dim3 grid((unsigned)((g.M + kBM - 1) / kBM), (unsigned)((g.N + nt - 1) / nt));
    k_gemm_bf16<<<grid, kGemmThreads, smem, s>>>(g);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward_fused(const FusedLaunch& f, cudaStream_t s)
{
    if (f.B <= 0) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        // persistent ping-pong kernel: one CTA per SM, pairs of 128-sample tiles
        CUtensorMap m2, m3, m4, m5;
        if (!make_map_sw128(&m2, f.W[1], kFusedHid, kFusedHid, kFusedHid, kFusedHid) ||
            !make_map_sw128(&m3, f.W[2], kFusedHid, kFusedHid, kFusedHid, kFusedHid) ||
            !make_map_sw128(&m4, f.W[3], kFusedHid, kFusedHid, kFusedHid, kFusedHid) ||
            !make_map_sw128(&m5, f.W[4], SALEC_MLP_OUT_N, kFusedHid, kFusedHid, kFusedOutPad))
            return cudaErrorNotSupported;
        static bool attr_pp[64] = {};
        static int nsm[64] = {};
        if (!attr_pp[dev]) {
            e = cudaFuncSetAttribute(k_mlp_forward_pp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pp_smem_bytes());
            if (e != cudaSuccess) return e;
            e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            attr_pp[dev] = true;
        }
        PPArgs a;
        a.B = f.B;
        a.ntiles = (f.B + kBM - 1) / kBM;
        a.npairs = (a.ntiles + 1) / 2;
        a.X = f.X; a.ld_x = f.ld_x; a.W1 = f.W[0];
        for (int l = 0; l < 5; ++l) a.bias[l] = f.bias[l];
        a.Y = f.Y; a.err = f.err;
        const int grid = a.npairs < nsm[dev] ? a.npairs : nsm[dev];
        k_mlp_forward_pp<<<(unsigned)grid, kPPThreads, pp_smem_bytes(), s>>>(m2, m3, m4, m5, a);
        return cudaGetLastError();
    }
}

cudaError_t launch_inputs_bf16(const float* x, int rows, int cols, int ld, __nv_bfloat16* y, cudaStream_t s,
                               __nv_bfloat16* yT, long ldT)
{
    const long n = (long)rows * ld;
    if (n <= 0) return cudaSuccess;
    k_inputs_bf16<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, rows, cols, ld, y, yT, ldT);
    return cudaGetLastError();
}

cudaError_t launch_train_reset(TrainState* ts, int t0, cudaStream_t s)
{
    k_train_reset<<<1, 1, 0, s>>>(ts, t0);
    return cudaGetLastError();
}

cudaError_t launch_refresh_bf16(const float* theta, long n, const int* wmap, __nv_bfloat16* wbf, cudaStream_t s,
                                const int* wmapT, __nv_bfloat16* wbfT)
{
    k_refresh_bf16<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(theta, n, wmap, wbf, wmapT, wbfT);
    return cudaGetLastError();
}

}  // namespace mlp
}  // namespace salec
