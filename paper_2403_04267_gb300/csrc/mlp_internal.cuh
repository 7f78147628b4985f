// mlp_internal.cuh -- argument blocks and launchers of the surrogate-MLP kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>

namespace salec {
namespace mlp {

// The bare GEMM: C = A B^T, BF16 operands with any element strides, FP32 result.
struct GemmArgs {
    int M, N, K;
    const __nv_bfloat16* A;
    long a_sm, a_sk;
    const __nv_bfloat16* B;
    long b_sn, b_sk;
    float* C;                 // FP32 output, row stride ldc
    long ldc;
    int* err;                 // error flag, or null
    int nt, tmem_cols;        // set by the launcher
    int stages;               // set by the launcher: shared-memory stages of the TMA-fed kernel
};

constexpr int kMaxSplit = 16;
constexpr int kMaxGroup = 8;      // ensemble members one group launch takes

constexpr int SALEC_MLP_OUT_N = 66;

// the fused inference pass over many samples: inputs, weights (BF16, W_1 rows padded like X),
// biases, outputs
struct FusedLaunch {
    int B;
    const __nv_bfloat16* X;
    int ld_x;
    const __nv_bfloat16* W[5];
    const float* bias[5];
    float* Y;
    int* err;
};

// Device state of a multi-step training call: k = steps of the call begun so far, t0 = Adam
// steps before the call; the step's learning rate and bias corrections, formed once per step.
struct TrainState {
    int k, t0;
    float lr, c1, c2;
};

struct AdamArgs {
    float lr, beta1, beta2, eps, c1, c2;   // c1 = 1 / (1 - beta1^t), c2 = 1 / (1 - beta2^t)
    bool table;                            // lr, c1, c2 from the net's TrainState instead
};

// A network's device arrays as the training kernels use them.
struct NetPtrs {
    const __nv_bfloat16* X;           // BF16 inputs, rows of 8
    const __nv_bfloat16* W1;          // layer-1 weights, rows of 8
    const float* bias[5];
    __nv_bfloat16* XT;                // inputs transposed, a row of ones under them
    __nv_bfloat16* HT[4];             // hidden activations transposed, a row of ones under them
    __nv_bfloat16* GT[5];             // dL/dZ_l transposed
    long ldT;                         // row stride of the transposed arrays
    float* D;                         // Y - T transposed (66 rows)
    float* part[5];                   // split-K partials of each layer's weight gradient
    float *theta, *m1, *m2;
    __nv_bfloat16 *wbf, *wbfT;        // BF16 weights and their transposes
    TrainState* ts;
    double* loss;                     // sum of squared errors
    int* err;
};

// TMA maps of a network: 128-row boxes of the weights and their transposes
// (wt[0] = W_5^T .. wt[3] = W_2^T), and for one batch size the transposed gradients and
// activations.
struct NetMaps {
    CUtensorMap w[4], wt[4], gt[5], ht[5];
};

struct TrainNet {
    NetPtrs p;
    NetMaps maps;
    int maps_B;                       // batch size that gt and ht were made for (0: none)
};

// One layer's part of the weight-gradient and update launches: an M x N product (N counts the
// bias column) in mt x ntn tiles of 128 x nt, K in S splits of kchunk, a split's partial N rows
// of ldp floats (pstep in all); its first CTA and first update block; its places in the parameter vector and in
// the BF16 weight blocks.
struct DwLayer {
    int M, N, mt, ntn, nt, S, kchunk, ldp, first, ufirst, w_ld, wt_ld;
    long woff, boff, wbf_off, wbfT_off, pstep;
};
struct DwPlan {
    DwLayer layer[5];
    int ctas, ublocks, max_nt;
};

struct TrainLaunch {
    int B;
    const float* t;                   // targets
    const float* lr;                  // learning-rate table, or null
    AdamArgs adam;
};

cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t s);
cudaError_t launch_mlp_forward_fused(const FusedLaunch& f, cudaStream_t s);
cudaError_t launch_inputs_bf16(const float* x, int rows, int cols, int ld, __nv_bfloat16* y, cudaStream_t s,
                               __nv_bfloat16* yT = nullptr, long ldT = 0);
// one thread: ts->k = 0, ts->t0 = t0
cudaError_t launch_train_reset(TrainState* ts, int t0, cudaStream_t s);
// BF16 copies of every weight from the FP32 parameters: at wmap[i], and transposed at wmapT[i]
cudaError_t launch_refresh_bf16(const float* theta, long n, const int* wmap, __nv_bfloat16* wbf, cudaStream_t s,
                                const int* wmapT, __nv_bfloat16* wbfT);

// mlp_train.cu.  A training pass of `count` networks (kMaxGroup at most, each with the plan it
// has alone): forward, backward, weight gradients, then the gradient of the one network into
// grad, or with grad null the Adam update of every network.
cudaError_t launch_train_pass(TrainNet* const* nets, int count, const TrainLaunch& t, float* grad, cudaStream_t s);
// inference of few samples by the training pass's tiles; *done = false, and nothing launched,
// for batches that fill the chip with the persistent kernel's larger tiles
cudaError_t launch_infer_small(const TrainNet& n, const float* x, int B, float* y, cudaStream_t s, bool* done);
cudaError_t make_weight_maps(TrainNet* n);
DwPlan plan_dw(int B, int sms);
size_t dw_part_floats(int layer);
size_t dw_smem_bytes(int nt);

}  // namespace mlp
}  // namespace salec
