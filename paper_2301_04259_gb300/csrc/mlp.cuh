// mlp.cuh -- the surrogate network (8 -> 4 x 256 GELU -> 129) on the tensor cores, whole chains
// of layers per kernel (mlp.cu).
#pragma once

#include "tc_gemm.cuh"

namespace soap {
namespace mlp {

constexpr int kIn = 8, kHidden = 256, kCoef = 128, kOut = kCoef + 1, kOutPad = 136;
constexpr int kFwd = 5;                      // forward products
constexpr int kBwd = 4;                      // products of the backward chain (dz)

// BF16 weights of one network as TMA maps (boxes of 64 K columns x 128 rows, 128-byte swizzle):
// W_l [out][in] for the forward products, W_l^T [in][out_pad] of layers 4 .. 1 for the backward.
struct Weights {
    CUtensorMap fwd[kFwd];
    CUtensorMap bwd[kBwd];
    const float* bias[kFwd];
};

// One training step's buffers.  TMA maps with boxes of 64 columns x 64 rows over the row-major
// BF16 activations and gradients: a_0 = scaled inputs [B][8], a_l [B][256], g_4 = dL/dy [B][136],
// g_l = dL/dz_l [B][256].  grad: GELU'(z_l) of every hidden layer in FP32, in the order of the
// threads that write and read it back (no other kernel reads it).
struct Step {
    CUtensorMap a[kFwd];
    CUtensorMap g[kFwd];
    const __nv_bfloat16* gp[kFwd];
    __nv_bfloat16* x0;
    float* grad[kFwd - 1];
};

struct TrainArgs {
    Weights w;
    Step s;
    const float* x;             // data set [n][8]
    const float* t;             // targets [n][129]
    const int* perm;            // shuffled row order, or NULL: rows in order
    const int* d_step;          // [0] step of the epoch
    const float* lohi;          // [2][8] input ranges
    const float* w_out;         // [129] loss weights
    double* loss;
    int B;
};

struct QueryArgs {
    Weights w[2];               // the network; the one that predicts the RV error (blockIdx.y = 1)
    int nets;                   // 1: the network predicts its own error
    const float* x;             // [n][8]
    int64_t n;
    const float* lohi;
    const float* mean;          // [128] coefficient scaling
    const float* sd;
    float thr_cms;
    uint8_t* accept;            // outputs, each may be NULL
    float* pred_err;
    float* coef;
    __nv_bfloat16* split;       // [n][3 x 128] rows [c_hi c_hi c_lo]
};

struct DwArgs {
    Step s;
    float* G;
    int64_t offW[kFwd], offb[kFwd];
    int* d_step;
    int B, steps, advance;
};

soap_status weight_maps(Weights& w, const __nv_bfloat16* const* W, const __nv_bfloat16* const* WT,
                        const float* const* bias);
// act: x0, a_1 .. a_4; grad: g_0 .. g_4
soap_status step_maps(Step& s, __nv_bfloat16* const* act, __nv_bfloat16* const* grad, int B);
// forward, loss and backward chain of one batch: activations, output and hidden gradients
soap_status train_step(const TrainArgs& a, cudaStream_t st, unsigned int* flags);
// weight and bias gradients of the batch; with `advance` the step counters move on
soap_status weight_grads(const DwArgs& a, cudaStream_t st, unsigned int* flags);
soap_status query(const QueryArgs& a, cudaStream_t st, unsigned int* flags);

}  // namespace mlp
}  // namespace soap
