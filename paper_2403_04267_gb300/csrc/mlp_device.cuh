// mlp_device.cuh -- tensor-core, TMA and mbarrier helpers of the surrogate-MLP kernels, the
// GELU, and the tensor maps of their operands (mlp_kernels.cu, mlp_train.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mlp_internal.cuh"
#include "salec_tma.cuh"

namespace salec {
namespace mlp {

constexpr int kBM = 128;          // rows of a C tile = TMEM lanes
constexpr int kBK = 64;           // K slice per stage
constexpr int kGemmThreads = 128;
constexpr int kMaxNT = 128;       // widest C tile (columns = TMEM columns)
// A wait on an mbarrier fails after 2 s.  Then the kernel still waits for its own copies and
// MMAs in flight, with a limit that is as long again: the shared memory they write or read and
// the tensor memory must not be given back under them.
// Failure detection is tested on a build of its own (SALEC_MLP_TEST_STALL = n): the thread that
// issues the operand copies of a tile stops after n of them, as if the others never landed, and
// the waits are short.
constexpr unsigned long long kDrainNs = 2000000000ull;
#ifdef SALEC_MLP_TEST_STALL
constexpr unsigned long long kWaitNs = 20000000ull;
__device__ __forceinline__ bool stalled(int copies) { return copies >= SALEC_MLP_TEST_STALL; }
#else
constexpr unsigned long long kWaitNs = 2000000000ull;
__device__ __forceinline__ bool stalled(int) { return false; }
#endif

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor of tcgen05: start address, leading-dimension byte offset
// (between core matrices adjacent along K), stride-dimension byte offset (between core
// matrices adjacent along M/N), the fixed field 0b001 at bits 46-48, no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator (bits 4-5 = 1), A and
// B BF16 (bits 7-9 = 1, bits 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits
// 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// bounded wait; false when the time limit ran out
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity)
{
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > kWaitNs) return false;
    return true;
}

// the wait for copies and MMAs in flight before their memory is given back
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity)
{
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > kDrainNs) return;
}

// mbar_wait for short waits on a critical path: the clock is only read once the first polls
// have failed (where other warps of the SM compute meanwhile, reading it between polls is the
// better use of the issue slots: the persistent forward kernel keeps mbar_wait)
__device__ __forceinline__ bool mbar_wait_short(uint64_t* bar, uint32_t parity)
{
    for (int k = 0; k < 64; ++k)
        if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait(bar, parity);
}

// True in one thread of the (converged) warp.  The tensor-core and bulk-copy instructions
// take their operands from uniform registers: in a branch on elect.sync the compiler knows
// that a single thread runs and moves them there once, in a branch on the lane number it has
// to serialise over the lanes that might be active, which cost about 130 cycles at every MMA.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// the warp's number as a value the compiler knows to be the same in all its lanes
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0); }

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// Packed FP32 pairs: every multiply, add and multiply-add of two values issues as one
// instruction, each lane rounded as the scalar instruction would.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 f2(float a, float b) { return (f32x2)__float_as_uint(a) | ((f32x2)__float_as_uint(b) << 32); }
__device__ __forceinline__ float f2lo(f32x2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f2hi(f32x2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f32x2 f2mul(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 f2fma(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 f2add(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// The normal CDF Phi(z) = (1 + erf(z / sqrt 2)) / 2 of two values, with the complementary
// error function of Abramowitz & Stegun, Handbook of Mathematical Functions, formula 7.1.26:
// for x >= 0, erfc(x) = t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) exp(-x^2) + e(x),
// t = 1 / (1 + p x), |e(x)| <= 1.5e-7.  Phi(z) is 1 - erfc(x) / 2 for z >= 0 and erfc(x) / 2
// for z < 0 (x = |z| / sqrt 2), so the left tail is formed without cancellation.  Also returns
// exp(-z^2 / 2) (the same exponential), which the GELU derivative needs.  The error is far
// below the BF16 rounding (2^-9 relative) that every activation goes through.
__device__ __forceinline__ f32x2 normal_cdf_pair(f32x2 z, f32x2* gauss)
{
    const float z0 = f2lo(z), z1 = f2hi(z);
    const f32x2 x = f2mul(f2(fabsf(z0), fabsf(z1)), f2(0.70710678118654752f, 0.70710678118654752f));
    const f32x2 d = f2fma(f2(0.3275911f, 0.3275911f), x, f2(1.0f, 1.0f));
    const f32x2 t = f2(__fdividef(1.0f, f2lo(d)), __fdividef(1.0f, f2hi(d)));
    f32x2 pol = f2fma(t, f2(1.061405429f, 1.061405429f), f2(-1.453152027f, -1.453152027f));
    pol = f2fma(t, pol, f2(1.421413741f, 1.421413741f));
    pol = f2fma(t, pol, f2(-0.284496736f, -0.284496736f));
    pol = f2fma(t, pol, f2(0.254829592f, 0.254829592f));
    const f32x2 nx2 = f2mul(f2(-f2lo(x), -f2hi(x)), x);
    const f32x2 e = f2(__expf(f2lo(nx2)), __expf(f2hi(nx2)));
    *gauss = e;
    const f32x2 h = f2mul(f2mul(f2(0.5f, 0.5f), f2mul(pol, t)), e);
    return f2(z0 >= 0.0f ? 1.0f - f2lo(h) : f2lo(h), z1 >= 0.0f ? 1.0f - f2hi(h) : f2hi(h));
}

// GELU in its erf form, z Phi(z), and its derivative Phi(z) + z phi(z)
__device__ __forceinline__ f32x2 gelu_pair(f32x2 z)
{
    f32x2 e;
    return f2mul(z, normal_cdf_pair(z, &e));
}
__device__ __forceinline__ f32x2 gelu_grad_pair(f32x2 z)
{
    f32x2 e;
    const f32x2 P = normal_cdf_pair(z, &e);
    return f2fma(f2mul(z, f2(0.39894228040143268f, 0.39894228040143268f)), e, P);
}


__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// core-matrix offset of (row r, 8-column group kg) in a K-major tile of `rows` rows
__device__ __forceinline__ uint32_t cm_off(int r, int kg, int rows) { return kg * (rows * 16) + (r >> 3) * 128 + (r & 7) * 16; }

// byte offset of 16-byte chunk c (8 columns) of row r in a 128-byte swizzled K slice: rows of
// 128 bytes, the chunks of a row permuted by its number modulo 8.  Warps writing one chunk of
// 32 consecutive rows meet no bank conflict, and the tensor cores read an A operand in it
// faster than in core matrices without swizzle (a 128 x 64 x 16 MMA every 100 cycles instead of
// every 165).
__device__ __forceinline__ uint32_t sw128_off(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }
constexpr uint32_t kSliceBytes = kBM * kBK * 2;      // a K slice of a 128-row tile: 16 KB

// descriptor of a K-major operand in the 128-byte swizzled layout: rows of 128 bytes, 8-row
// groups 1024 bytes apart (stride-dimension offset), swizzle mode 2 at bits 61-63; the
// leading-dimension offset is unused for K extents within one 128-byte row
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// bounded wait of a thread that has nothing else to do: it backs off between polls so
// that the warps doing arithmetic on its SM sub-partition keep the issue slots
__device__ __forceinline__ bool mbar_wait_idle(uint64_t* bar, uint32_t parity)
{
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (global_ns() - t0 > kWaitNs) return false;
        __nanosleep(64);
    }
    return true;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// cuTensorMapEncodeTiled from the driver (looked up once, shared with the solver's copy kernel)
inline TmaEncodeTiledFn encode_tiled() { return tma_encode_tiled(); }

// 2-D map of a row-major BF16 matrix [rows][K] with row stride ld elements; boxes of 8
// elements (16 bytes) x box_rows rows.  False when TMA cannot address it (alignment).
inline bool make_map(CUtensorMap* map, const void* base, long rows, long K, long ld, int box_rows)
{
    const TmaEncodeTiledFn fn = encode_tiled();
    if (!fn || rows < 1 || K < 1 || (reinterpret_cast<uintptr_t>(base) & 15) || ((ld * 2) & 15)) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    const cuuint32_t box[2] = {8u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same matrix as 64-element (128-byte) x box_rows boxes in the 128-byte swizzled
// layout (one box is one K slice of box_rows rows).
inline bool make_map_sw128(CUtensorMap* map, const void* base, long rows, long K, long ld, int box_rows)
{
    const TmaEncodeTiledFn fn = encode_tiled();
    if (!fn || rows < 1 || K < 1 || (reinterpret_cast<uintptr_t>(base) & 15) || ((ld * 2) & 15)) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace mlp
}  // namespace salec
