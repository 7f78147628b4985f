// mlp_api.cu -- C ABI of the crater-surrogate MLP: parameters, forward pass, gradient and
// Adam training step on one caller-owned device buffer, plus the bare BF16 GEMM.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <new>
#include <string>
#include <vector>

#include "../../include/salec_mlp.h"
#include "mlp_internal.cuh"
#include "salec_trace.h"

using namespace salec::mlp;

namespace {

constexpr int kLayers = 5;
constexpr int kDims[kLayers + 1] = {SALEC_MLP_IN, 256, 256, 256, 256, SALEC_MLP_OUT};
constexpr int kHid = 256;
// BF16 row stride of the inputs and of W_1: 5 columns padded to 8 (16-byte rows, which the
// TMA-fed GEMM needs); the padding stays zero
constexpr int kInLd = 8;

// BF16 row stride of W_l
int w_ld(int l) { return l == 0 ? kInLd : kDims[l]; }
// BF16 row stride of W_l^T (n_in rows of n_out values, padded to 16-byte rows); layer 0
// needs none (no activation gradient below the first layer)
int wt_ld(int l) { return (kDims[l + 1] + 7) / 8 * 8; }
// rows of the transposed activation buffers: the layer's units, one row of ones (the bias
// gradients are the weight gradients of that row), padded
constexpr int kHidT = kHid + 16;
constexpr int kInT = 16;
long ld_t(int bmax) { return ((long)bmax + 7) / 8 * 8; }

size_t align_up(size_t x) { return (x + 255) & ~size_t(255); }

long n_params()
{
    long n = 0;
    for (int l = 0; l < kLayers; ++l) n += (long)kDims[l + 1] * kDims[l] + kDims[l + 1];
    return n;
}

long n_weights_bf16()
{
    long n = 0;
    for (int l = 0; l < kLayers; ++l) n += (long)kDims[l + 1] * w_ld(l);
    return n;
}

long n_weights_bf16_t()
{
    long n = 0;
    for (int l = 1; l < kLayers; ++l) n += (long)kDims[l] * wt_ld(l);
    return n;
}

// The weight gradients contract over the batch: the training kernel leaves the activations
// and the gradients of the pre-activations transposed (HT, XT, GT), and the BF16 weights are
// kept transposed as well (wbfT) for the activation gradients.
struct Layout {
    size_t theta, m1, m2, grad, wmap, wbf, wmapT, wbfT, X, XT, HT[4], D, GT[kLayers], part[kLayers], loss, err, ts,
        total;
    Layout(int bmax)
    {
        const long P = n_params(), W = n_weights_bf16(), WT = n_weights_bf16_t(), ldT = ld_t(bmax);
        size_t o = 0;
        auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes); return r; };
        theta = take(P * 4); m1 = take(P * 4); m2 = take(P * 4); grad = take(P * 4);
        wmap = take(P * 4);
        wbf = take(W * 2);
        wmapT = take(P * 4);
        wbfT = take(WT * 2);
        X = take((size_t)bmax * kInLd * 2);
        XT = take((size_t)kInT * ldT * 2);
        for (int l = 0; l < 4; ++l) HT[l] = take((size_t)kHidT * ldT * 2);
        D = take((size_t)SALEC_MLP_OUT * ldT * 4);
        for (int l = 0; l < kLayers; ++l) GT[l] = take((size_t)kDims[l + 1] * ldT * 2);
        for (int l = 0; l < kLayers; ++l) part[l] = take(dw_part_floats(l) * 4);   // split-K partials
        loss = take(16);          // the sum of squared errors, then the error flag
        err = loss + 8;
        ts = take(sizeof(TrainState));
        total = o;
    }
};

}  // namespace

struct salec_mlp {
    int bmax = 0;
    cudaStream_t stream = nullptr;
    std::string err;
    float *theta = nullptr, *m1 = nullptr, *m2 = nullptr, *grad = nullptr;
    int* wmap = nullptr;
    __nv_bfloat16* wbf = nullptr;
    int* wmapT = nullptr;
    __nv_bfloat16* wbfT = nullptr;
    __nv_bfloat16* X = nullptr;
    double* loss = nullptr;
    int* errflag = nullptr;
    TrainState* ts = nullptr;
    TrainNet net = {};                    // the arrays and TMA maps of the training kernels
    long steps = 0;                       // Adam steps taken
    // salec_mlp_train: a CUDA graph of kTrainChunk steps, for the arguments it was captured with
    cudaGraphExec_t tgraph = nullptr;
    const float* tg_t = nullptr;
    const float* tg_lr = nullptr;
    int tg_batch = 0;
    float tg_beta1 = 0.0f, tg_beta2 = 0.0f, tg_eps = 0.0f;
    bool tg_ok = true;                    // false after a capture failed: plain launches
    ~salec_mlp()
    {
        if (tgraph) cudaGraphExecDestroy(tgraph);
    }
    long woff[kLayers], boff[kLayers];    // offsets of W_l and b_l in theta
    long wbf_off[kLayers];                // offset of W_l in the BF16 weight block
    long wbfT_off[kLayers];               // offset of W_l^T in the transposed block (l >= 1)
};

namespace {

salec_status fail(salec_mlp* n, salec_status st, const std::string& msg)
{
    if (n) n->err = msg;
    return st;
}

salec_status cuda_fail(salec_mlp* n, cudaError_t e, const char* where)
{
    return fail(n, SALEC_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define MLP_CUDA(n, call, where)                                   \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return cuda_fail((n), e_, (where)); \
    } while (0)

salec_status check_batch(salec_mlp* n, int B)
{
    if (!n) return SALEC_EINVAL;
    if (B < 1 || B > n->bmax) return fail(n, SALEC_EINVAL, "batch outside 1..batch_max");
    return SALEC_OK;
}

constexpr int kTrainChunk = 25;

// the inputs as BF16 rows of 8 and transposed, for a training pass
cudaError_t inputs(salec_mlp* n, const float* x_dev, int B, cudaStream_t s)
{
    return launch_inputs_bf16(x_dev, B, SALEC_MLP_IN, kInLd, n->X, s, n->net.p.XT, n->net.p.ldT);
}

TrainLaunch train_launch(int B, const float* t_dev, const float* lr_dev, float beta1, float beta2, float eps)
{
    TrainLaunch t = {};
    t.B = B;
    t.t = t_dev;
    t.lr = lr_dev;
    t.adam.beta1 = beta1; t.adam.beta2 = beta2; t.adam.eps = eps;
    t.adam.table = lr_dev != nullptr;
    return t;
}

// One step of a multi-step call: its learning rate and bias corrections from the device
// state, then the gradient and the Adam update (the inputs are already in X).
salec_status train_one(salec_mlp* n, int B, const float* t_dev, const float* lr_dev, float beta1, float beta2,
                       float eps)
{
    TrainNet* net = &n->net;
    MLP_CUDA(n, launch_train_pass(&net, 1, train_launch(B, t_dev, lr_dev, beta1, beta2, eps), nullptr, n->stream),
             "mlp train step");
    return SALEC_OK;
}

// Capture kTrainChunk steps on a private stream (the graph can then be launched into any
// stream); false, with no error left pending, when capture is not possible.
bool capture_train(salec_mlp* n, int B, const float* t_dev, const float* lr_dev, float beta1, float beta2, float eps)
{
    if (n->tgraph) {
        cudaGraphExecDestroy(n->tgraph);
        n->tgraph = nullptr;
    }
    cudaStream_t cs;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    cudaStream_t keep = n->stream;
    n->stream = cs;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    salec_status st = SALEC_OK;
    for (int k = 0; k < kTrainChunk && e == cudaSuccess && st == SALEC_OK; ++k)
        st = train_one(n, B, t_dev, lr_dev, beta1, beta2, eps);
    const cudaError_t e2 = cudaStreamEndCapture(cs, &g);
    n->stream = keep;
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess && st == SALEC_OK) e = cudaGraphInstantiate(&n->tgraph, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess || st != SALEC_OK) {
        (void)cudaGetLastError();
        n->tgraph = nullptr;
        return false;
    }
    n->tg_t = t_dev; n->tg_lr = lr_dev; n->tg_batch = B;
    n->tg_beta1 = beta1; n->tg_beta2 = beta2; n->tg_eps = eps;
    return true;
}

}  // namespace

// Ensemble members trained together (salec_mlp_train_group): the member contexts and the
// CUDA graph of kTrainChunk steps captured for the arguments of the last call.
struct salec_mlp_group {
    std::vector<salec_mlp*> nets;
    cudaStream_t stream = nullptr;
    std::string err;
    cudaGraphExec_t tgraph = nullptr;
    const float* tg_t = nullptr;
    const float* tg_lr = nullptr;
    int tg_batch = 0;
    float tg_beta1 = 0.0f, tg_beta2 = 0.0f, tg_eps = 0.0f;
    bool tg_ok = true;
    ~salec_mlp_group()
    {
        if (tgraph) cudaGraphExecDestroy(tgraph);
    }
};

namespace {

salec_status gfail(salec_mlp_group* g, salec_status st, const std::string& msg)
{
    if (g) g->err = msg;
    return st;
}

#define GROUP_CUDA(g, call, where)                                                                                \
    do {                                                                                                          \
        cudaError_t e_ = (call);                                                                                  \
        if (e_ != cudaSuccess) return gfail((g), SALEC_ECUDA, std::string(where) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// One training step of every member, each kernel one launch for all members (the inputs are
// already in each X, X^T).
salec_status group_train_one(salec_mlp_group* G, cudaStream_t s, int B, const float* t_dev, const float* lr_dev,
                             float beta1, float beta2, float eps)
{
    TrainNet* nets[kMaxGroup];
    const int n = (int)G->nets.size();
    for (int k = 0; k < n; ++k) nets[k] = &G->nets[k]->net;
    GROUP_CUDA(G, launch_train_pass(nets, n, train_launch(B, t_dev, lr_dev, beta1, beta2, eps), nullptr, s), "group train step");
    return SALEC_OK;
}

// Capture kTrainChunk group steps on a private stream; false, with no error left pending,
// when capture is not possible.
bool capture_group(salec_mlp_group* G, int B, const float* t_dev, const float* lr_dev, float beta1, float beta2, float eps)
{
    if (G->tgraph) {
        cudaGraphExecDestroy(G->tgraph);
        G->tgraph = nullptr;
    }
    cudaStream_t cs;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    cudaGraph_t gr = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    salec_status st = SALEC_OK;
    for (int k = 0; k < kTrainChunk && e == cudaSuccess && st == SALEC_OK; ++k)
        st = group_train_one(G, cs, B, t_dev, lr_dev, beta1, beta2, eps);
    const cudaError_t e2 = cudaStreamEndCapture(cs, &gr);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess && st == SALEC_OK) e = cudaGraphInstantiate(&G->tgraph, gr, 0);
    if (gr) cudaGraphDestroy(gr);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess || st != SALEC_OK) {
        (void)cudaGetLastError();
        G->tgraph = nullptr;
        return false;
    }
    G->tg_t = t_dev; G->tg_lr = lr_dev; G->tg_batch = B;
    G->tg_beta1 = beta1; G->tg_beta2 = beta2; G->tg_eps = eps;
    return true;
}

}  // namespace

extern "C" {

int salec_mlp_n_params(void) { return (int)n_params(); }

salec_status salec_mlp_bytes(int batch_max, size_t* bytes)
{
    if (!bytes || batch_max < 1) return SALEC_EINVAL;
    *bytes = Layout(batch_max).total;
    return SALEC_OK;
}

salec_status salec_mlp_create(int batch_max, void* dev_buf, size_t bytes, void* stream, salec_mlp** out)
{
    if (!out || !dev_buf || batch_max < 1) return SALEC_EINVAL;
    *out = nullptr;
    Layout L(batch_max);
    if (bytes < L.total) return SALEC_ENOMEM;
    if (reinterpret_cast<uintptr_t>(dev_buf) & 255) return SALEC_EINVAL;
    salec_mlp* n = new (std::nothrow) salec_mlp();
    if (!n) return SALEC_ENOMEM;
    unsigned char* b = static_cast<unsigned char*>(dev_buf);
    n->bmax = batch_max;
    n->stream = static_cast<cudaStream_t>(stream);
    n->theta = reinterpret_cast<float*>(b + L.theta);
    n->m1 = reinterpret_cast<float*>(b + L.m1);
    n->m2 = reinterpret_cast<float*>(b + L.m2);
    n->grad = reinterpret_cast<float*>(b + L.grad);
    n->wmap = reinterpret_cast<int*>(b + L.wmap);
    n->wbf = reinterpret_cast<__nv_bfloat16*>(b + L.wbf);
    n->wmapT = reinterpret_cast<int*>(b + L.wmapT);
    n->wbfT = reinterpret_cast<__nv_bfloat16*>(b + L.wbfT);
    n->X = reinterpret_cast<__nv_bfloat16*>(b + L.X);
    n->loss = reinterpret_cast<double*>(b + L.loss);
    n->errflag = reinterpret_cast<int*>(b + L.err);
    n->ts = reinterpret_cast<TrainState*>(b + L.ts);
    // parameter offsets and the weight -> BF16 block map
    const long P = n_params();
    std::vector<int> wmap(P, -1), wmapT(P, -1);
    long o = 0, w = 0, wt = 0;
    for (int l = 0; l < kLayers; ++l) {
        const int ni = kDims[l], no = kDims[l + 1], ld = w_ld(l);
        n->woff[l] = o;
        n->wbf_off[l] = w;
        n->wbfT_off[l] = l > 0 ? wt : -1;
        for (int r = 0; r < no; ++r)
            for (int c = 0; c < ni; ++c) {
                wmap[o + (long)r * ni + c] = (int)(w + (long)r * ld + c);
                if (l > 0) wmapT[o + (long)r * ni + c] = (int)(wt + (long)c * wt_ld(l) + r);
            }
        o += (long)no * ni;
        w += (long)no * ld;
        if (l > 0) wt += (long)ni * wt_ld(l);
        n->boff[l] = o;
        o += no;
    }
    NetPtrs& p = n->net.p;
    p.X = n->X;
    p.W1 = n->wbf;
    for (int l = 0; l < kLayers; ++l) {
        p.bias[l] = n->theta + n->boff[l];
        p.GT[l] = reinterpret_cast<__nv_bfloat16*>(b + L.GT[l]);
        p.part[l] = reinterpret_cast<float*>(b + L.part[l]);
    }
    p.XT = reinterpret_cast<__nv_bfloat16*>(b + L.XT);
    for (int l = 0; l < 4; ++l) p.HT[l] = reinterpret_cast<__nv_bfloat16*>(b + L.HT[l]);
    p.ldT = ld_t(batch_max);
    p.D = reinterpret_cast<float*>(b + L.D);
    p.theta = n->theta; p.m1 = n->m1; p.m2 = n->m2;
    p.wbf = n->wbf; p.wbfT = n->wbfT;
    p.ts = n->ts; p.loss = n->loss; p.err = n->errflag;
    // the rows of ones under the transposed activations (BF16 1.0 = 0x3f80): columns past
    // the batch lie outside the tensor map and read as zero
    std::vector<uint16_t> ones((size_t)p.ldT, 0x3f80u);
    cudaError_t e = cudaMemsetAsync(dev_buf, 0, L.total, n->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(n->wmap, wmap.data(), P * sizeof(int), cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(n->wmapT, wmapT.data(), P * sizeof(int), cudaMemcpyHostToDevice, n->stream);
    for (int l = 0; l < 4 && e == cudaSuccess; ++l)
        e = cudaMemcpyAsync(p.HT[l] + (long)kHid * p.ldT, ones.data(), ones.size() * 2, cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p.XT + (long)SALEC_MLP_IN * p.ldT, ones.data(), ones.size() * 2, cudaMemcpyHostToDevice,
                            n->stream);
    if (e == cudaSuccess) e = make_weight_maps(&n->net);
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
    if (e != cudaSuccess) {
        delete n;
        return SALEC_ECUDA;
    }
    *out = n;
    return SALEC_OK;
}

salec_status salec_mlp_set_params(salec_mlp* n, const float* theta_host)
{
    if (!n || !theta_host) return SALEC_EINVAL;
    const long P = n_params();
    MLP_CUDA(n, cudaMemcpyAsync(n->theta, theta_host, P * 4, cudaMemcpyHostToDevice, n->stream), "set_params copy");
    MLP_CUDA(n, cudaMemsetAsync(n->m1, 0, P * 4, n->stream), "set_params reset");
    MLP_CUDA(n, cudaMemsetAsync(n->m2, 0, P * 4, n->stream), "set_params reset");
    MLP_CUDA(n, launch_refresh_bf16(n->theta, P, n->wmap, n->wbf, n->stream, n->wmapT, n->wbfT), "set_params bf16 copy");
    MLP_CUDA(n, cudaStreamSynchronize(n->stream), "set_params sync");
    n->steps = 0;
    return SALEC_OK;
}

salec_status salec_mlp_get_params(salec_mlp* n, float* theta_host)
{
    if (!n || !theta_host) return SALEC_EINVAL;
    MLP_CUDA(n, cudaMemcpyAsync(theta_host, n->theta, n_params() * 4, cudaMemcpyDeviceToHost, n->stream), "get_params");
    MLP_CUDA(n, cudaStreamSynchronize(n->stream), "get_params sync");
    return salec_mlp_check(n);
}

salec_status salec_mlp_forward(salec_mlp* n, const float* x_dev, int batch, float* y_dev)
{
    salec::HostRange range("salec_mlp_forward");
    salec_status st = check_batch(n, batch);
    if (st != SALEC_OK) return st;
    if (!x_dev || !y_dev) return fail(n, SALEC_EINVAL, "null pointer");
    bool done = false;
    MLP_CUDA(n, launch_infer_small(n->net, x_dev, batch, y_dev, n->stream, &done), "mlp forward");
    if (done) return SALEC_OK;
    MLP_CUDA(n, launch_inputs_bf16(x_dev, batch, SALEC_MLP_IN, kInLd, n->X, n->stream), "mlp input");
    FusedLaunch f;
    f.B = batch; f.X = n->X; f.ld_x = kInLd; f.Y = y_dev; f.err = n->errflag;
    for (int l = 0; l < kLayers; ++l) { f.W[l] = n->wbf + n->wbf_off[l]; f.bias[l] = n->theta + n->boff[l]; }
    MLP_CUDA(n, launch_mlp_forward_fused(f, n->stream), "mlp forward");
    return SALEC_OK;
}

salec_status salec_mlp_gradient(salec_mlp* n, const float* x_dev, const float* t_dev, int batch, float* grad_dev,
                                double* loss_host)
{
    salec::HostRange range("salec_mlp_gradient");
    salec_status st = check_batch(n, batch);
    if (st != SALEC_OK) return st;
    if (!x_dev || !t_dev) return fail(n, SALEC_EINVAL, "null pointer");
    float* grad = grad_dev ? grad_dev : n->grad;
    MLP_CUDA(n, inputs(n, x_dev, batch, n->stream), "mlp input");
    TrainNet* net = &n->net;
    MLP_CUDA(n, launch_train_pass(&net, 1, train_launch(batch, t_dev, nullptr, 0.0f, 0.0f, 0.0f), grad, n->stream),
             "mlp gradient");
    if (loss_host) {
        struct { double sse; int err, pad; } r;
        MLP_CUDA(n, cudaMemcpyAsync(&r, n->loss, sizeof(r), cudaMemcpyDeviceToHost, n->stream), "mlp loss read");
        MLP_CUDA(n, cudaStreamSynchronize(n->stream), "mlp loss sync");
        *loss_host = r.sse / ((double)batch * SALEC_MLP_OUT);
        if (r.err) return fail(n, SALEC_ECUDA, "a tensor-core wait ran out of time");
    }
    return SALEC_OK;
}

salec_status salec_mlp_train_step(salec_mlp* n, const float* x_dev, const float* t_dev, int batch, float lr,
                                  float beta1, float beta2, float eps, double* sse_dev)
{
    salec::HostRange range("salec_mlp_train_step");
    salec_status st = check_batch(n, batch);
    if (st != SALEC_OK) return st;
    if (!x_dev || !t_dev) return fail(n, SALEC_EINVAL, "null pointer");
    if (!(lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return fail(n, SALEC_EINVAL, "bad Adam hyper-parameters");
    MLP_CUDA(n, inputs(n, x_dev, batch, n->stream), "mlp input");
    n->steps += 1;
    TrainLaunch t = train_launch(batch, t_dev, nullptr, beta1, beta2, eps);
    t.adam.lr = lr;
    t.adam.c1 = (float)(1.0 / (1.0 - std::pow((double)beta1, (double)n->steps)));
    t.adam.c2 = (float)(1.0 / (1.0 - std::pow((double)beta2, (double)n->steps)));
    TrainNet* net = &n->net;
    MLP_CUDA(n, launch_train_pass(&net, 1, t, nullptr, n->stream), "mlp train step");
    if (sse_dev) MLP_CUDA(n, cudaMemcpyAsync(sse_dev, n->loss, 8, cudaMemcpyDeviceToDevice, n->stream), "mlp loss copy");
    return SALEC_OK;
}

salec_status salec_mlp_train(salec_mlp* n, const float* x_dev, const float* t_dev, int batch, int steps,
                             const float* lr_dev, float beta1, float beta2, float eps, double* sse_dev)
{
    salec::HostRange range("salec_mlp_train");
    salec_status st = check_batch(n, batch);
    if (st != SALEC_OK) return st;
    if (steps < 0) return fail(n, SALEC_EINVAL, "negative step count");
    if (steps == 0) return SALEC_OK;
    if (!x_dev || !t_dev || !lr_dev) return fail(n, SALEC_EINVAL, "null pointer");
    if (!(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return fail(n, SALEC_EINVAL, "bad Adam hyper-parameters");
    if (n->steps + (long)steps > 0x7fffffffL) return fail(n, SALEC_EINVAL, "step count overflow");
    MLP_CUDA(n, inputs(n, x_dev, batch, n->stream), "mlp input");
    MLP_CUDA(n, launch_train_reset(n->ts, (int)n->steps, n->stream), "mlp train reset");
    // the first step with plain launches (it also sets the kernels' attributes), then whole
    // chunks as graph replays, then the rest
    st = train_one(n, batch, t_dev, lr_dev, beta1, beta2, eps);
    if (st != SALEC_OK) return st;
    int done = 1;
    const int chunks = (steps - 1) / kTrainChunk;
    if (chunks > 0 && n->tg_ok) {
        const bool same = n->tgraph && n->tg_t == t_dev && n->tg_lr == lr_dev && n->tg_batch == batch &&
                          n->tg_beta1 == beta1 && n->tg_beta2 == beta2 && n->tg_eps == eps;
        if (!same && !capture_train(n, batch, t_dev, lr_dev, beta1, beta2, eps)) n->tg_ok = false;
        if (n->tgraph && n->tg_ok) {
            for (int c = 0; c < chunks; ++c) MLP_CUDA(n, cudaGraphLaunch(n->tgraph, n->stream), "mlp train graph");
            done += chunks * kTrainChunk;
        }
    }
    for (; done < steps; ++done) {
        st = train_one(n, batch, t_dev, lr_dev, beta1, beta2, eps);
        if (st != SALEC_OK) return st;
    }
    n->steps += steps;
    if (sse_dev) MLP_CUDA(n, cudaMemcpyAsync(sse_dev, n->loss, 8, cudaMemcpyDeviceToDevice, n->stream), "mlp loss copy");
    return SALEC_OK;
}

salec_status salec_mlp_check(salec_mlp* n)
{
    if (!n) return SALEC_EINVAL;
    int f = 0;
    MLP_CUDA(n, cudaMemcpyAsync(&f, n->errflag, 4, cudaMemcpyDeviceToHost, n->stream), "mlp flag read");
    MLP_CUDA(n, cudaStreamSynchronize(n->stream), "mlp flag sync");
    if (f) return fail(n, SALEC_ECUDA, "a tensor-core wait ran out of time");
    return SALEC_OK;
}

salec_status salec_gemm_bf16(int M, int N, int K, const void* A, long a_sm, long a_sk, const void* B, long b_sn,
                             long b_sk, float* C, long ldc, void* stream)
{
    if (M < 0 || N < 0 || K < 0) return SALEC_EINVAL;
    if (M > 0 && N > 0 && (!C || (K > 0 && (!A || !B)))) return SALEC_EINVAL;   // K = 0: C = 0, A and B unused
    GemmArgs g = {};
    g.M = M; g.N = N; g.K = K;
    g.A = static_cast<const __nv_bfloat16*>(A); g.a_sm = a_sm; g.a_sk = a_sk;
    g.B = static_cast<const __nv_bfloat16*>(B); g.b_sn = b_sn; g.b_sk = b_sk;
    g.C = C; g.ldc = ldc;
    if (launch_gemm(g, static_cast<cudaStream_t>(stream)) != cudaSuccess) return SALEC_ECUDA;
    return SALEC_OK;
}

salec_status salec_mlp_group_create(salec_mlp* const* nets, int n, void* stream, salec_mlp_group** out)
{
    if (!out || !nets || n < 1 || n > kMaxGroup) return SALEC_EINVAL;
    *out = nullptr;
    for (int k = 0; k < n; ++k) {
        if (!nets[k]) return SALEC_EINVAL;
        for (int j = 0; j < k; ++j)
            if (nets[j] == nets[k]) return SALEC_EINVAL;
    }
    salec_mlp_group* g = new (std::nothrow) salec_mlp_group();
    if (!g) return SALEC_ENOMEM;
    g->nets.assign(nets, nets + n);
    g->stream = static_cast<cudaStream_t>(stream);
    *out = g;
    return SALEC_OK;
}

salec_status salec_mlp_train_group(salec_mlp_group* G, const float* x_dev, const float* t_dev, int batch, int steps,
                                   const float* lr_dev, float beta1, float beta2, float eps)
{
    salec::HostRange range("salec_mlp_train_group");
    if (!G) return SALEC_EINVAL;
    if (steps < 0) return gfail(G, SALEC_EINVAL, "negative step count");
    if (steps == 0) return SALEC_OK;
    if (!x_dev || !t_dev || !lr_dev) return gfail(G, SALEC_EINVAL, "null pointer");
    if (!(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return gfail(G, SALEC_EINVAL, "bad Adam hyper-parameters");
    for (salec_mlp* m : G->nets) {
        if (batch < 1 || batch > m->bmax) return gfail(G, SALEC_EINVAL, "batch outside 1..batch_max of a member");
        if (m->steps + (long)steps > 0x7fffffffL) return gfail(G, SALEC_EINVAL, "step count overflow");
    }
    cudaStream_t s = G->stream;
    for (salec_mlp* m : G->nets) {
        GROUP_CUDA(G, inputs(m, x_dev, batch, s), "group input");
        GROUP_CUDA(G, launch_train_reset(m->ts, (int)m->steps, s), "group train reset");
    }
    // the first step with plain launches (it also sets the kernels' attributes), then whole
    // chunks as graph replays, then the rest
    salec_status st = group_train_one(G, s, batch, t_dev, lr_dev, beta1, beta2, eps);
    if (st != SALEC_OK) return st;
    int done = 1;
    const int chunks = (steps - 1) / kTrainChunk;
    if (chunks > 0 && G->tg_ok) {
        const bool same = G->tgraph && G->tg_t == t_dev && G->tg_lr == lr_dev && G->tg_batch == batch &&
                          G->tg_beta1 == beta1 && G->tg_beta2 == beta2 && G->tg_eps == eps;
        if (!same && !capture_group(G, batch, t_dev, lr_dev, beta1, beta2, eps)) G->tg_ok = false;
        if (G->tgraph && G->tg_ok) {
            for (int c = 0; c < chunks; ++c) GROUP_CUDA(G, cudaGraphLaunch(G->tgraph, s), "group train graph");
            done += chunks * kTrainChunk;
        }
    }
    for (; done < steps; ++done) {
        st = group_train_one(G, s, batch, t_dev, lr_dev, beta1, beta2, eps);
        if (st != SALEC_OK) return st;
    }
    for (salec_mlp* m : G->nets) m->steps += steps;
    return SALEC_OK;
}

const char* salec_mlp_group_last_error(const salec_mlp_group* g) { return g ? g->err.c_str() : "null group"; }

void salec_mlp_group_destroy(salec_mlp_group* g) { delete g; }

const char* salec_mlp_last_error(const salec_mlp* n) { return n ? n->err.c_str() : ""; }

void salec_mlp_destroy(salec_mlp* n) { delete n; }

}  // extern "C"
