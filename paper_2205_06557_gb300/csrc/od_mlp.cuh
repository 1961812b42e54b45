// The warm-start network as two kernels on the tensor cores (od_mlp.cu): a fused pass over
// 128-row tiles (forward, or forward, loss and backward data products) and the weight
// gradients.
#pragma once

#include "od_tc.cuh"

namespace od {
namespace mlp {

constexpr int IN = 7, K0 = 16, H = 256, OUTR = 4, OUTP = 16, G = 8;  // as in od_sur.cu
constexpr int TILE = 128;                     // rows (16 samples of 8 grains) per tile
constexpr int QUADS = 4;                      // 32-row quarters of a tile
constexpr int BIAS_LD = 4 * H + OUTP;         // bias-gradient partial row: b1, b2, b3, b4, b5
// output and input widths of a layer, and the offset of its W (then b) in the flat parameter
// vector (od_sur_get_params)
__host__ __device__ constexpr int out_of(int l) { return l == 4 ? OUTP : H; }
__host__ __device__ constexpr int in_of(int l) { return l == 0 ? K0 : l == 2 ? 2 * H : H; }
__host__ __device__ constexpr int w_off(int l) { return l == 0 ? 0 : w_off(l - 1) + out_of(l - 1) * (in_of(l - 1) + 1); }
constexpr int N_PARAMS = w_off(5);

// BF16 activations and backpropagated errors the weight gradients read, rows padded to tiles
struct Acts {
    __nv_bfloat16 *x0, *h1, *x3, *h3, *h4;       // [rows][16], [256], [512] (h2 | pooled mean), [256], [256]
    __nv_bfloat16 *dy, *dz4, *dz3, *dz2, *dz1;   // [rows][16], [256] ...
};

struct FusedMaps {
    CUtensorMap w[9];    // W1..W5, then W5^T, W4^T, W3^T, W2^T
    CUtensorMap act[8];  // h1, x3, h3, h4, dz4, dz3, dz2, dz1 (stores of 128 x 64 boxes)
};

struct GradMaps {
    CUtensorMap dz[5];  // of layer 1..5: dz1, dz2, dz3, dz4, dy (64 x 64 boxes)
    CUtensorMap x[5];   // x0, h1, x3, h3, h4
};

struct FusedArgs {
    const float* x;      // [rows][7]
    const float* mask;   // [rows]
    const float* tgt;    // [rows][4]
    const float* bias[5];
    float* y;            // [rows][4]
    float* row_loss;     // [tiles * 128]
    float* dbias;        // [CTAs * 4][BIAS_LD] column sums of the errors
    __nv_bfloat16 *x0, *dy;
    int rows, tiles;
    float inv_count;     // 1 / (present grains * 4)
    int* err;
};

bool encode_maps(const __nv_bfloat16* const wb[5], const __nv_bfloat16* const wt[5], const Acts& A, int rows_pad,
                 FusedMaps& F, GradMaps& D);
int launch_forward(const FusedMaps& M, const FusedArgs& A, int sms, cudaStream_t s);
// forward, row losses, errors of every layer (Acts) and the bias-gradient partials; *ctas:
// rows / 4 of the partials
int launch_forward_backward(const FusedMaps& M, const FusedArgs& A, int sms, int* ctas, cudaStream_t s);
// weight gradients over rows (split over CTAs into partial vectors part[splits][N_PARAMS]),
// then the whole gradient vector from the partials
int grad_splits(int rows, int sms);
int max_grad_splits(int max_rows, int sms);  // at least grad_splits of any rows up to max_rows
int launch_weight_grads(const GradMaps& M, float* part, int rows, int splits, int* err, cudaStream_t s);
int launch_grad_reduce(const float* part, int splits, const float* dbias, int bias_rows, float* grad, cudaStream_t s);

}  // namespace mlp
}  // namespace od
