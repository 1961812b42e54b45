// Learned warm start for the self-consistent grain charge: a small set-pooled MLP,
// trained on the GPU by the library's own forward, backward and Adam kernels.
//
// Network (per grain k of a sample, grains masked, at most 8 per sample):
//   x_k  = [global features (3), grain features (4)], padded to 16
//   h1_k = relu(W1 x_k + b1)            256
//   h2_k = relu(W2 h1_k + b2)           256
//   c    = mean over present grains of h2_k (set pooling)
//   h3_k = relu(W3 [h2_k, c] + b3)      256
//   h4_k = relu(W4 h3_k + b4)           256
//   y_k  = W5 h4_k + b5                 4 outputs (padded to 16)
// Weights are kept in FP32 (master copy for Adam) and used as BF16 in every matrix
// product (BF16 inputs, FP32 accumulation); activations are rounded to BF16 where they enter
// a product.  The loss is the mean squared error over present grains and the four outputs.
// By default the network runs as the fused kernels of od_mlp.cu on the fifth-generation tensor
// cores.  OD_GEMM_MMA_SYNC runs it layer by layer with warp-level mma.sync products
// (k_gemm_nt and the kernels below) as an independent cross-check.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "od_mlp.cuh"

namespace od {
namespace sur {

constexpr int IN = 7, K0 = 16, H = 256, OUTR = 4, OUTP = 16, G = 8;

// ------------------------------------------------------------------ GEMM
// C[M][N] = A[M][K] * B[N][K]^T (+ bias[N]) (relu) in FP32, optional BF16 copy.
// A, B BF16 row-major; M, N, K multiples of 16.  One warp per 16x16 output tile,
// two m16n8k16 products per k-step of 16.
__device__ __forceinline__ unsigned ld2(const __nv_bfloat16* p) { return *reinterpret_cast<const unsigned*>(p); }

__global__ void k_gemm_nt(const __nv_bfloat16* __restrict__ A, const __nv_bfloat16* __restrict__ B,
                          const float* __restrict__ bias, float* __restrict__ C, __nv_bfloat16* __restrict__ Cb,
                          int M, int N, int K, int relu)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int tiles_n = N / 16;
    if (warp >= (M / 16) * tiles_n) return;
    const int m0 = (warp / tiles_n) * 16, n0 = (warp % tiles_n) * 16;
    const int g = lane >> 2, t = lane & 3;
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    for (int k0 = 0; k0 < K; k0 += 16) {
        const __nv_bfloat16* a_lo = A + (long long)(m0 + g) * K + k0 + 2 * t;
        const __nv_bfloat16* a_hi = A + (long long)(m0 + g + 8) * K + k0 + 2 * t;
        const unsigned a0 = ld2(a_lo), a1 = ld2(a_hi), a2 = ld2(a_lo + 8), a3 = ld2(a_hi + 8);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const __nv_bfloat16* bp = B + (long long)(n0 + 8 * s + g) * K + k0 + 2 * t;
            const unsigned b0 = ld2(bp), b1 = ld2(bp + 8);
            asm volatile(
                "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                "{%0,%1,%2,%3};"
                : "+f"(acc[s][0]), "+f"(acc[s][1]), "+f"(acc[s][2]), "+f"(acc[s][3])
                : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = m0 + g + 8 * h;
            const int col = n0 + 8 * s + 2 * t;
            float v0 = acc[s][2 * h], v1 = acc[s][2 * h + 1];
            if (bias) {
                v0 += bias[col];
                v1 += bias[col + 1];
            }
            if (relu) {
                v0 = fmaxf(v0, 0.f);
                v1 = fmaxf(v1, 0.f);
            }
            C[(long long)row * N + col] = v0;
            C[(long long)row * N + col + 1] = v1;
            if (Cb) {
                Cb[(long long)row * N + col] = __float2bfloat16_rn(v0);
                Cb[(long long)row * N + col + 1] = __float2bfloat16_rn(v1);
            }
        }
}

// ---------------------------------------------------------------- helpers
__global__ void k_to_bf16(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = __float2bfloat16_rn(x[i]);
}

// out[c][r] = in[r][c] (BF16), in is R x C
__global__ void k_transpose(const __nv_bfloat16* __restrict__ in, __nv_bfloat16* __restrict__ out, int R, int C)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)R * C) return;
    const int r = (int)(i / C), c = (int)(i % C);
    out[(long long)c * R + r] = in[i];
}

// masked mean over the G grains of each sample: c[b][j] = sum_k m_bk h[bG+k][j] / n_b
__global__ void k_pool(const float* __restrict__ h, const float* __restrict__ mask, float* __restrict__ c, int Bn)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Bn * H) return;
    const int b = i / H, j = i % H;
    float s = 0.f, n = 0.f;
    for (int k = 0; k < G; ++k) {
        const float m = mask[b * G + k];
        s += m * h[(long long)(b * G + k) * H + j];
        n += m;
    }
    c[i] = n > 0.f ? s / n : 0.f;
}

// X3[row] = [h2[row], c[sample]] as BF16
__global__ void k_concat(const __nv_bfloat16* __restrict__ h2b, const float* __restrict__ c,
                         __nv_bfloat16* __restrict__ x3, int M)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)M * 2 * H) return;
    const int row = (int)(i / (2 * H)), j = (int)(i % (2 * H));
    x3[i] = j < H ? h2b[(long long)row * H + j] : __float2bfloat16_rn(c[(row / G) * H + (j - H)]);
}

// dY = 2 (y - t) / count on present grains and real outputs; loss partial sums per row
__global__ void k_loss(const float* __restrict__ y, const float* __restrict__ tgt, const float* __restrict__ mask,
                       float* __restrict__ dy, float* __restrict__ row_loss, int M, float inv_count)
{
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= M) return;
    const float m = mask[row];
    float l = 0.f;
    for (int o = 0; o < OUTP; ++o) {
        float d = 0.f;
        if (o < OUTR && m > 0.f) {
            const float e = y[row * OUTP + o] - tgt[row * OUTR + o];
            l += e * e;
            d = 2.f * e * inv_count;
        }
        dy[row * OUTP + o] = d;
    }
    row_loss[row] = l * inv_count;
}

// dZ = dA * (Z > 0) in place on dA (Z holds post-relu values: > 0 iff pre-activation > 0)
__global__ void k_relu_back(float* __restrict__ da, const float* __restrict__ a, __nv_bfloat16* __restrict__ dzb,
                            long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float v = a[i] > 0.f ? da[i] : 0.f;
    da[i] = v;
    dzb[i] = __float2bfloat16_rn(v);
}

// column sums of dZ [M][N] -> db[N] (fixed order per column)
__global__ void k_colsum(const float* __restrict__ dz, float* __restrict__ db, int M, int N)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    float s = 0.f;
    for (int r = 0; r < M; ++r) s += dz[(long long)r * N + j];
    db[j] = s;
}

// split dX3 [M][2H]: dA2 = first half + pooled share of the second half
__global__ void k_unpool(const float* __restrict__ dx3, const float* __restrict__ mask, float* __restrict__ da2, int M)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)M * H) return;
    const int row = (int)(i / H), j = (int)(i % H);
    const int b = row / G;
    float n = 0.f, dc = 0.f;
    for (int k = 0; k < G; ++k) {
        const float m = mask[b * G + k];
        n += m;
        dc += m * dx3[(long long)(b * G + k) * 2 * H + H + j];
    }
    const float share = n > 0.f ? mask[row] * dc / n : 0.f;
    da2[i] = dx3[(long long)row * 2 * H + j] + share;
}

// where parameter i of the flat vector lives in the BF16 copies: the element of wb (out x in per
// layer, one after another) and of wt (its transpose); false for a bias
__device__ __forceinline__ bool weight_place(int i, int& wb, int& wt)
{
    int base = 0;  // weights of the layers before
#pragma unroll
    for (int l = 0; l < 5; ++l) {
        const int rows = mlp::out_of(l), cols = mlp::in_of(l), k = i - mlp::w_off(l);
        if (k < rows * (cols + 1)) {
            wb = base + k;
            wt = base + (k % cols) * rows + k / cols;
            return k < rows * cols;
        }
        base += rows * cols;
    }
    return false;
}

// the BF16 copies of the weights and their transposes from the FP32 masters
__global__ void k_refresh(const float* __restrict__ p, __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int a, b;
    if (i >= mlp::N_PARAMS || !weight_place(i, a, b)) return;
    wb[a] = wt[b] = __float2bfloat16_rn(p[i]);
}

// Adam on the FP32 master parameters, then the BF16 copies of the weights: one launch over the
// whole vector
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt, float lr, float b1, float b2,
                       float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= mlp::N_PARAMS) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    int a, b;
    if (weight_place(i, a, b)) wb[a] = wt[b] = __float2bfloat16_rn(pi);
}

// the loss: row losses added in FP64 in a fixed order (one CTA)
__global__ void __launch_bounds__(256) k_loss_sum(const float* __restrict__ row_loss, int rows, double* __restrict__ loss)
{
    __shared__ double s[256];
    double a = 0.0;
    for (int r = threadIdx.x; r < rows; r += 256) a += (double)row_loss[r];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = s[0];
}

// inputs padded to K0 columns for the layer-by-layer products
__global__ void k_pad_inputs(const float* __restrict__ x, __nv_bfloat16* __restrict__ x0, int M)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * K0) return;
    const int r = i / K0, c = i % K0;
    x0[i] = __float2bfloat16_rn(c < IN ? x[r * IN + c] : 0.f);
}

// the four real outputs of the padded output layer
__global__ void k_take_outputs(const float* __restrict__ y, float* __restrict__ out, int M)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M * OUTR) out[i] = y[(i / OUTR) * OUTP + i % OUTR];
}

}  // namespace sur
}  // namespace od

using namespace od;
using namespace od::sur;

// ------------------------------------------------------------------- host
namespace {

struct Layer {
    int out, in;
    float *w = nullptr, *b = nullptr;            // FP32 master, in the flat parameter vector
    float *gw = nullptr, *gb = nullptr;          // gradients, likewise
    __nv_bfloat16 *wb = nullptr, *wt = nullptr;  // BF16 copy [out][in] and transpose [in][out]
};

}  // namespace

// results the host reads after a pass
struct SurOut {
    double loss;
    int err;  // tensor-core wait timeouts (bit 1)
    int pad;
};

struct od_sur {
    int maxB = 0, sms = 0;
    int splits_cap = 0;  // partial gradients (ranges of rows) `part` holds
    Layer L[5];
    float *p = nullptr, *g = nullptr, *am = nullptr, *av = nullptr;  // parameters, gradients, Adam moments
    __nv_bfloat16 *wb = nullptr, *wt = nullptr;
    // inputs, outputs and the fused pass's activations, rows padded to whole tiles
    float *x = nullptr, *mask = nullptr, *tgt = nullptr, *y = nullptr, *rowl = nullptr, *dbias = nullptr, *part = nullptr;
    mlp::Acts acts{};
    mlp::FusedMaps fmaps;
    mlp::GradMaps gmaps;
    SurOut* d_out = nullptr;
    SurOut* h_out = nullptr;  // page-locked
    // layer-by-layer engine, allocated when it is first selected (M = maxB * G rows)
    bool layers = false;
    __nv_bfloat16 *x0b = nullptr, *h1b = nullptr, *h2b = nullptr, *x3b = nullptr, *h3b = nullptr, *h4b = nullptr,
                  *dyb = nullptr, *dzb = nullptr, *tA = nullptr, *tB = nullptr;
    float *h1 = nullptr, *h2 = nullptr, *c = nullptr, *h3 = nullptr, *h4 = nullptr, *yp = nullptr, *dy = nullptr,
          *dx3 = nullptr, *da = nullptr;
    cudaStream_t stream = nullptr;
    cudaEvent_t ev_in = nullptr;  // after the copies of a batch's host arrays, in a call that reads no result
    long long adam_t = 0;
    int engine = OD_GEMM_TCGEN05;
    std::string err;
};

namespace {

thread_local std::string g_sur_error;

int sfail(od_sur* s, int code, const std::string& msg)
{
    if (s) s->err = msg;
    else g_sur_error = msg;
    return code;
}

#define SCK(s, call)                                                                                  \
    do {                                                                                              \
        cudaError_t e_ = (call);                                                                      \
        if (e_ != cudaSuccess) return sfail(s, OD_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

inline int blocks(long long n, int bt = 256) { return (int)((n + bt - 1) / bt); }

}  // namespace

namespace od {
int launch_gemm_tc(const __nv_bfloat16* A, const __nv_bfloat16* B, const float* bias, float* C, __nv_bfloat16* Cb,
                   int M, int N, int K, int relu, int* err, cudaStream_t s);

int gemm_bf16(const __nv_bfloat16* A, const __nv_bfloat16* B, const float* bias, float* C, __nv_bfloat16* Cb, int M,
              int N, int K, int relu, int engine, int* err, cudaStream_t stream)
{
    if (engine == OD_GEMM_TCGEN05) return launch_gemm_tc(A, B, bias, C, Cb, M, N, K, relu, err, stream);
    const long long warps = (long long)(M / 16) * (N / 16);
    k_gemm_nt<<<blocks(warps * 32, 128), 128, 0, stream>>>(A, B, bias, C, Cb, M, N, K, relu);
    return (int)cudaGetLastError();
}
}  // namespace od

namespace {

// a product of the layer-by-layer engine
int gemm(od_sur* s, const __nv_bfloat16* A, const __nv_bfloat16* B, const float* bias, float* C, __nv_bfloat16* Cb, int M,
         int N, int K, int relu)
{
    const int e = gemm_bf16(A, B, bias, C, Cb, M, N, K, relu, OD_GEMM_MMA_SYNC, &s->d_out->err, s->stream);
    return e == 0 ? OD_OK : sfail(s, OD_ECUDA, std::string("gemm launch failed: ") + cudaGetErrorString((cudaError_t)e));
}

// the pass's loss and error word, after everything queued on the stream
int read_out(od_sur* s)
{
    SCK(s, cudaMemcpyAsync(s->h_out, s->d_out, sizeof(SurOut), cudaMemcpyDeviceToHost, s->stream));
    SCK(s, cudaStreamSynchronize(s->stream));
    if (s->h_out->err) {
        SCK(s, cudaMemsetAsync(s->d_out, 0, sizeof(SurOut), s->stream));
        return sfail(s, OD_ETIMEOUT, "a tensor-core product's wait gave up");
    }
    return OD_OK;
}

void free_sur(od_sur* s)
{
    void* bufs[] = {s->p, s->g, s->am, s->av, s->wb, s->wt, s->x, s->mask, s->tgt, s->y, s->rowl, s->dbias, s->part,
                    s->acts.x0, s->acts.h1, s->acts.x3, s->acts.h3, s->acts.h4, s->acts.dy, s->acts.dz4, s->acts.dz3,
                    s->acts.dz2, s->acts.dz1, s->d_out, s->x0b, s->h1b, s->h2b, s->x3b, s->h3b, s->h4b, s->dyb, s->dzb,
                    s->tA, s->tB, s->h1, s->h2, s->c, s->h3, s->h4, s->yp, s->dy, s->dx3, s->da};
    for (void* p : bufs) cudaFree(p);
    cudaFreeHost(s->h_out);
    if (s->ev_in) cudaEventDestroy(s->ev_in);
}

// buffers of the layer-by-layer engine
int ensure_layers(od_sur* s)
{
    if (s->layers) return OD_OK;
    const long long M = (long long)s->maxB * G;
    struct {
        void** p;
        long long bytes;
    } want[] = {{(void**)&s->x0b, 2 * M * K0}, {(void**)&s->h1b, 2 * M * H}, {(void**)&s->h2b, 2 * M * H},
                {(void**)&s->x3b, 4 * M * H},  {(void**)&s->h3b, 2 * M * H}, {(void**)&s->h4b, 2 * M * H},
                {(void**)&s->dyb, 2 * M * OUTP}, {(void**)&s->dzb, 2 * M * H}, {(void**)&s->tA, 4 * M * H},
                {(void**)&s->tB, 4 * M * H},   {(void**)&s->h1, 4 * M * H},  {(void**)&s->h2, 4 * M * H},
                {(void**)&s->c, 4 * s->maxB * (long long)H}, {(void**)&s->h3, 4 * M * H}, {(void**)&s->h4, 4 * M * H},
                {(void**)&s->yp, 4 * M * OUTP}, {(void**)&s->dy, 4 * M * OUTP}, {(void**)&s->dx3, 8 * M * H},
                {(void**)&s->da, 8 * M * H}};
    for (auto& w : want)
        if (!*w.p && cudaMalloc(w.p, w.bytes) != cudaSuccess) {
            cudaGetLastError();
            return sfail(s, OD_ENOMEM, "surrogate: no memory for the layer-by-layer engine");
        }
    s->layers = true;
    return OD_OK;
}

// refresh the BF16 copies of every layer from the FP32 masters
int refresh_bf16(od_sur* s)
{
    k_refresh<<<blocks(mlp::N_PARAMS), 256, 0, s->stream>>>(s->p, s->wb, s->wt);
    return cudaGetLastError() == cudaSuccess ? OD_OK : sfail(s, OD_ECUDA, "weight refresh failed");
}

// forward pass layer by layer (rows a multiple of 16)
int forward_layers(od_sur* s, int Bn)
{
    const int M = Bn * G;
    int rc;
    k_pad_inputs<<<blocks((long long)M * K0), 256, 0, s->stream>>>(s->x, s->x0b, M);
    if ((rc = gemm(s, s->x0b, s->L[0].wb, s->L[0].b, s->h1, s->h1b, M, H, K0, 1))) return rc;
    if ((rc = gemm(s, s->h1b, s->L[1].wb, s->L[1].b, s->h2, s->h2b, M, H, H, 1))) return rc;
    k_pool<<<blocks((long long)Bn * H), 256, 0, s->stream>>>(s->h2, s->mask, s->c, Bn);
    k_concat<<<blocks((long long)M * 2 * H), 256, 0, s->stream>>>(s->h2b, s->c, s->x3b, M);
    if ((rc = gemm(s, s->x3b, s->L[2].wb, s->L[2].b, s->h3, s->h3b, M, H, 2 * H, 1))) return rc;
    if ((rc = gemm(s, s->h3b, s->L[3].wb, s->L[3].b, s->h4, s->h4b, M, H, H, 1))) return rc;
    if ((rc = gemm(s, s->h4b, s->L[4].wb, s->L[4].b, s->yp, nullptr, M, OUTP, H, 0))) return rc;
    return OD_OK;
}

// dW = dZ^T X over the M rows (NT product of the transposes), db = column sums
int weight_grad(od_sur* s, Layer& l, const float* dz, const __nv_bfloat16* dzb, const __nv_bfloat16* xb, int M)
{
    k_transpose<<<blocks((long long)M * l.out), 256, 0, s->stream>>>(dzb, s->tA, M, l.out);
    k_transpose<<<blocks((long long)M * l.in), 256, 0, s->stream>>>(xb, s->tB, M, l.in);
    int rc = gemm(s, s->tA, s->tB, nullptr, l.gw, nullptr, l.out, l.in, M, 0);
    if (rc) return rc;
    k_colsum<<<blocks(l.out), 256, 0, s->stream>>>(dz, l.gb, M, l.out);
    return OD_OK;
}

int backward_layers(od_sur* s, int Bn, float inv_count)
{
    const int M = Bn * G;
    int rc;
    k_loss<<<blocks(M), 256, 0, s->stream>>>(s->yp, s->tgt, s->mask, s->dy, s->rowl, M, inv_count);
    // output layer: dy (FP32) -> BF16
    k_to_bf16<<<blocks((long long)M * OUTP), 256, 0, s->stream>>>(s->dy, s->dyb, (long long)M * OUTP);
    if ((rc = weight_grad(s, s->L[4], s->dy, s->dyb, s->h4b, M))) return rc;
    // dh4 = dy W5  (B = W5^T [H][OUTP])
    if ((rc = gemm(s, s->dyb, s->L[4].wt, nullptr, s->da, nullptr, M, H, OUTP, 0))) return rc;
    k_relu_back<<<blocks((long long)M * H), 256, 0, s->stream>>>(s->da, s->h4, s->dzb, (long long)M * H);
    if ((rc = weight_grad(s, s->L[3], s->da, s->dzb, s->h3b, M))) return rc;
    if ((rc = gemm(s, s->dzb, s->L[3].wt, nullptr, s->da, nullptr, M, H, H, 0))) return rc;
    k_relu_back<<<blocks((long long)M * H), 256, 0, s->stream>>>(s->da, s->h3, s->dzb, (long long)M * H);
    if ((rc = weight_grad(s, s->L[2], s->da, s->dzb, s->x3b, M))) return rc;
    if ((rc = gemm(s, s->dzb, s->L[2].wt, nullptr, s->dx3, nullptr, M, 2 * H, H, 0))) return rc;
    k_unpool<<<blocks((long long)M * H), 256, 0, s->stream>>>(s->dx3, s->mask, s->da, M);
    k_relu_back<<<blocks((long long)M * H), 256, 0, s->stream>>>(s->da, s->h2, s->dzb, (long long)M * H);
    if ((rc = weight_grad(s, s->L[1], s->da, s->dzb, s->h1b, M))) return rc;
    if ((rc = gemm(s, s->dzb, s->L[1].wt, nullptr, s->da, nullptr, M, H, H, 0))) return rc;
    k_relu_back<<<blocks((long long)M * H), 256, 0, s->stream>>>(s->da, s->h1, s->dzb, (long long)M * H);
    if ((rc = weight_grad(s, s->L[0], s->da, s->dzb, s->x0b, M))) return rc;
    return cudaGetLastError() == cudaSuccess ? OD_OK : sfail(s, OD_ECUDA, "backward launch failed");
}

// The batch's arrays as they come; the layer-by-layer engine takes an even number of samples,
// the last of an odd batch absent and zero.  Copies of page-locked arrays are still under way on
// return: a call ends with read_out, or waits for them itself.
int upload_batch(od_sur* s, const float* x, const float* mask, const float* tgt, int Bn)
{
    const size_t M = (size_t)Bn * G;
    SCK(s, cudaMemcpyAsync(s->x, x, sizeof(float) * M * IN, cudaMemcpyHostToDevice, s->stream));
    SCK(s, cudaMemcpyAsync(s->mask, mask, sizeof(float) * M, cudaMemcpyHostToDevice, s->stream));
    if (tgt) SCK(s, cudaMemcpyAsync(s->tgt, tgt, sizeof(float) * M * OUTR, cudaMemcpyHostToDevice, s->stream));
    if (s->engine == OD_GEMM_MMA_SYNC && Bn % 2) {
        SCK(s, cudaMemsetAsync(s->x + M * IN, 0, sizeof(float) * G * IN, s->stream));
        SCK(s, cudaMemsetAsync(s->mask + M, 0, sizeof(float) * G, s->stream));
        SCK(s, cudaMemsetAsync(s->tgt + M * OUTR, 0, sizeof(float) * G * OUTR, s->stream));
    }
    return OD_OK;
}

// the end of a call that failed: the host arrays are the caller's again
int give_back(od_sur* s, int rc)
{
    cudaStreamSynchronize(s->stream);
    return rc;
}

mlp::FusedArgs fused_args(od_sur* s, int Bn)
{
    mlp::FusedArgs A{};
    A.x = s->x;
    A.mask = s->mask;
    A.tgt = s->tgt;
    for (int l = 0; l < 5; ++l) A.bias[l] = s->L[l].b;
    A.y = s->y;
    A.row_loss = s->rowl;
    A.dbias = s->dbias;
    A.x0 = s->acts.x0;
    A.dy = s->acts.dy;
    A.rows = Bn * G;
    A.tiles = (A.rows + mlp::TILE - 1) / mlp::TILE;
    A.err = &s->d_out->err;
    return A;
}

// outputs of the uploaded batch into s->y [rows][4]
int run_forward(od_sur* s, int Bn)
{
    if (s->engine == OD_GEMM_MMA_SYNC) {
        const int Bp = (Bn + 1) / 2 * 2;
        const int rc = forward_layers(s, Bp);
        if (rc) return rc;
        k_take_outputs<<<blocks((long long)Bp * G * OUTR), 256, 0, s->stream>>>(s->yp, s->y, Bp * G);
        return cudaGetLastError() == cudaSuccess ? OD_OK : sfail(s, OD_ECUDA, "forward launch failed");
    }
    const int e = mlp::launch_forward(s->fmaps, fused_args(s, Bn), s->sms, s->stream);
    return e == 0 ? OD_OK : sfail(s, OD_ECUDA, std::string("forward launch failed: ") + cudaGetErrorString((cudaError_t)e));
}

// loss and gradients of the uploaded batch into d_out and the gradient vector
int run_gradients(od_sur* s, int Bn, const float* mask_host)
{
    long long cnt = 0;
    for (int r = 0; r < Bn * G; ++r) cnt += mask_host[r] > 0.f;
    const float inv = cnt > 0 ? (float)(1.0 / ((double)cnt * OUTR)) : 0.f;
    int rows = Bn * G, rc, e;
    if (s->engine == OD_GEMM_MMA_SYNC) {
        const int Bp = (Bn + 1) / 2 * 2;
        rows = Bp * G;
        if ((rc = forward_layers(s, Bp)) || (rc = backward_layers(s, Bp, inv))) return rc;
    } else {
        mlp::FusedArgs A = fused_args(s, Bn);
        A.y = nullptr;
        A.inv_count = inv;
        const int splits = std::min(mlp::grad_splits(rows, s->sms), s->splits_cap);
        int ctas = 0;
        if ((e = mlp::launch_forward_backward(s->fmaps, A, s->sms, &ctas, s->stream)) ||
            (e = mlp::launch_weight_grads(s->gmaps, s->part, rows, splits, &s->d_out->err, s->stream)) ||
            (e = mlp::launch_grad_reduce(s->part, splits, s->dbias, ctas * mlp::QUADS, s->g, s->stream)))
            return sfail(s, OD_ECUDA, std::string("gradient launch failed: ") + cudaGetErrorString((cudaError_t)e));
    }
    k_loss_sum<<<1, 256, 0, s->stream>>>(s->rowl, rows, &s->d_out->loss);
    return cudaGetLastError() == cudaSuccess ? OD_OK : sfail(s, OD_ECUDA, "loss launch failed");
}

}  // namespace

extern "C" {

int od_sur_create(int max_batch, uint64_t seed, void* stream, od_sur** out)
{
    if (!out || max_batch < 1 || max_batch > (1 << 16)) return sfail(nullptr, OD_EINVAL, "bad surrogate arguments");
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return sfail(nullptr, OD_ENODEV, "no CUDA device");
    od_sur* s = new od_sur();
    s->maxB = (max_batch + 1) / 2 * 2;  // the layer-by-layer engine takes whole pairs of samples
    s->stream = (cudaStream_t)stream;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev);
    // He-uniform initial weights from a seeded host generator (splitmix64), zero biases
    unsigned long long st = seed * 0x9E3779B97F4A7C15ull + 12345ull;
    auto next = [&st]() {
        unsigned long long z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    bool ok = true;
    auto mb = [&](void** p, size_t bytes) { ok = ok && cudaMalloc(p, bytes) == cudaSuccess; };
    mb((void**)&s->p, sizeof(float) * mlp::N_PARAMS);
    mb((void**)&s->g, sizeof(float) * mlp::N_PARAMS);
    mb((void**)&s->am, sizeof(float) * mlp::N_PARAMS);
    mb((void**)&s->av, sizeof(float) * mlp::N_PARAMS);
    mb((void**)&s->wb, sizeof(__nv_bfloat16) * mlp::N_PARAMS);
    mb((void**)&s->wt, sizeof(__nv_bfloat16) * mlp::N_PARAMS);
    const long long M = ((long long)s->maxB * G + mlp::TILE - 1) / mlp::TILE * mlp::TILE;  // rows in whole tiles
    mb((void**)&s->x, 4 * M * IN);
    mb((void**)&s->mask, 4 * M);
    mb((void**)&s->tgt, 4 * M * OUTR);
    mb((void**)&s->y, 4 * M * OUTR);
    mb((void**)&s->rowl, 4 * M);
    mb((void**)&s->dbias, sizeof(float) * mlp::QUADS * mlp::BIAS_LD * (size_t)s->sms);
    s->splits_cap = mlp::max_grad_splits((int)M, s->sms);
    mb((void**)&s->part, sizeof(float) * mlp::N_PARAMS * (size_t)s->splits_cap);
    mb((void**)&s->acts.x0, 2 * M * K0);
    mb((void**)&s->acts.h1, 2 * M * H);
    mb((void**)&s->acts.x3, 4 * M * H);
    mb((void**)&s->acts.h3, 2 * M * H);
    mb((void**)&s->acts.h4, 2 * M * H);
    mb((void**)&s->acts.dy, 2 * M * OUTP);
    mb((void**)&s->acts.dz4, 2 * M * H);
    mb((void**)&s->acts.dz3, 2 * M * H);
    mb((void**)&s->acts.dz2, 2 * M * H);
    mb((void**)&s->acts.dz1, 2 * M * H);
    mb((void**)&s->d_out, sizeof(SurOut));
    ok = ok && cudaMallocHost((void**)&s->h_out, sizeof(SurOut)) == cudaSuccess &&
         cudaEventCreateWithFlags(&s->ev_in, cudaEventDisableTiming) == cudaSuccess;
    if (ok) {
        std::vector<float> p(mlp::N_PARAMS, 0.f);
        long long wo = 0;
        for (int li = 0; li < 5; ++li) {
            Layer& l = s->L[li];
            l.out = mlp::out_of(li);
            l.in = mlp::in_of(li);
            const int off = mlp::w_off(li), nw = l.out * l.in;
            l.w = s->p + off;
            l.b = l.w + nw;
            l.gw = s->g + off;
            l.gb = l.gw + nw;
            l.wb = s->wb + wo;
            l.wt = s->wt + wo;
            wo += nw;
            const int fan_in = li == 0 ? IN : l.in;
            const double bound = std::sqrt(6.0 / fan_in) * (li == 4 ? 0.1 : 1.0);
            for (int o = 0; o < l.out; ++o)
                for (int i = 0; i < l.in; ++i) {
                    const bool live = (li != 0 || i < IN) && (li != 4 || o < OUTR);
                    const double u = (double)(next() >> 11) * (1.0 / 9007199254740992.0);
                    p[(size_t)off + o * l.in + i] = live ? (float)((2.0 * u - 1.0) * bound) : 0.f;
                }
        }
        cudaMemcpyAsync(s->p, p.data(), sizeof(float) * p.size(), cudaMemcpyHostToDevice, s->stream);
        cudaMemsetAsync(s->g, 0, sizeof(float) * p.size(), s->stream);
        cudaMemsetAsync(s->am, 0, sizeof(float) * p.size(), s->stream);
        cudaMemsetAsync(s->av, 0, sizeof(float) * p.size(), s->stream);
        ok = cudaMemsetAsync(s->d_out, 0, sizeof(SurOut), s->stream) == cudaSuccess &&
             refresh_bf16(s) == OD_OK && cudaStreamSynchronize(s->stream) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        g_sur_error = "surrogate allocation failed";
        free_sur(s);
        delete s;
        return OD_ENOMEM;
    }
    const __nv_bfloat16 *wb[5], *wt[5];
    for (int l = 0; l < 5; ++l) wb[l] = s->L[l].wb, wt[l] = s->L[l].wt;
    if (!mlp::encode_maps(wb, wt, s->acts, (int)M, s->fmaps, s->gmaps)) {
        g_sur_error = "surrogate: tensor map encoding failed";
        free_sur(s);
        delete s;
        return OD_ECUDA;
    }
    *out = s;
    return OD_OK;
}

void od_sur_destroy(od_sur* s)
{
    if (!s) return;
    if (s->stream) cudaStreamSynchronize(s->stream);
    else cudaDeviceSynchronize();
    free_sur(s);
    delete s;
}

int od_sur_num_params(const od_sur* s) { return s ? mlp::N_PARAMS : 0; }

// FP32 master parameters, layer by layer: W (out x in, row-major) then b (out)
int od_sur_get_params(od_sur* s, float* host)
{
    if (!s || !host) return sfail(s, OD_EINVAL, "bad argument");
    SCK(s, cudaMemcpyAsync(host, s->p, sizeof(float) * mlp::N_PARAMS, cudaMemcpyDeviceToHost, s->stream));
    SCK(s, cudaStreamSynchronize(s->stream));
    return OD_OK;
}

int od_sur_set_params(od_sur* s, const float* host)
{
    if (!s || !host) return sfail(s, OD_EINVAL, "bad argument");
    SCK(s, cudaMemcpyAsync(s->p, host, sizeof(float) * mlp::N_PARAMS, cudaMemcpyHostToDevice, s->stream));
    int rc = refresh_bf16(s);
    if (rc) return rc;
    SCK(s, cudaStreamSynchronize(s->stream));
    return OD_OK;
}

// y[B][G][4] for inputs x[B][G][7] (host) and mask[B][G] (host)
int od_sur_forward(od_sur* s, const float* x, const float* mask, int Bn, float* y)
{
    if (!s || !x || !mask || !y || Bn < 1 || Bn > s->maxB) return sfail(s, OD_EINVAL, "bad forward arguments");
    int rc = upload_batch(s, x, mask, nullptr, Bn);
    if (rc || (rc = run_forward(s, Bn))) return give_back(s, rc);
    SCK(s, cudaMemcpyAsync(y, s->y, sizeof(float) * Bn * G * OUTR, cudaMemcpyDeviceToHost, s->stream));
    return read_out(s);
}

// loss and parameter gradients (layout of od_sur_get_params) without an update
int od_sur_gradients(od_sur* s, const float* x, const float* mask, const float* tgt, int Bn, double* loss, float* grads)
{
    if (!s || !x || !mask || !tgt || Bn < 1 || Bn > s->maxB) return sfail(s, OD_EINVAL, "bad gradient arguments");
    int rc = upload_batch(s, x, mask, tgt, Bn);
    const bool reads = grads || loss;  // else the call waits for the copies only, not for the kernels
    if (!rc && !reads) SCK(s, cudaEventRecord(s->ev_in, s->stream));
    if (rc || (rc = run_gradients(s, Bn, mask))) return give_back(s, rc);
    if (grads)
        SCK(s, cudaMemcpyAsync(grads, s->g, sizeof(float) * mlp::N_PARAMS, cudaMemcpyDeviceToHost, s->stream));
    if (!reads) {
        SCK(s, cudaEventSynchronize(s->ev_in));
        return OD_OK;
    }
    if ((rc = read_out(s))) return rc;
    if (loss) *loss = s->h_out->loss;
    return OD_OK;
}

// one Adam step on a minibatch; returns the minibatch loss
int od_sur_train_step(od_sur* s, const float* x, const float* mask, const float* tgt, int Bn, float lr, double* loss)
{
    int rc = od_sur_gradients(s, x, mask, tgt, Bn, loss, nullptr);
    if (rc) return rc;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    s->adam_t += 1;
    const float c1 = 1.f - std::pow(b1, (float)s->adam_t), c2 = 1.f - std::pow(b2, (float)s->adam_t);
    k_adam<<<blocks(mlp::N_PARAMS), 256, 0, s->stream>>>(s->p, s->g, s->am, s->av, s->wb, s->wt, lr, b1, b2, eps, c1, c2);
    if (cudaGetLastError() != cudaSuccess) return sfail(s, OD_ECUDA, "adam launch failed");
    return OD_OK;
}

const char* od_sur_last_error(const od_sur* s) { return s ? s->err.c_str() : g_sur_error.c_str(); }

int od_sur_set_gemm(od_sur* s, int engine)
{
    if (!s || (engine != OD_GEMM_TCGEN05 && engine != OD_GEMM_MMA_SYNC)) return sfail(s, OD_EINVAL, "bad engine");
    if (engine == OD_GEMM_MMA_SYNC) {
        const int rc = ensure_layers(s);
        if (rc) return rc;
    }
    s->engine = engine;
    return OD_OK;
}

int od_gemm_bf16(const uint16_t* A, const uint16_t* B, const float* bias, float* C, uint16_t* Cb, int M, int N, int K,
                 int relu, int engine, int* err, void* stream)
{
    if (!A || !B || !C || !err || M < 1 || N < 16 || K < 16 || N % 16 || K % 16) return OD_EINVAL;
    if (engine != OD_GEMM_TCGEN05 && (engine != OD_GEMM_MMA_SYNC || M % 16)) return OD_EINVAL;
    const int e = gemm_bf16((const __nv_bfloat16*)A, (const __nv_bfloat16*)B, bias, C, (__nv_bfloat16*)Cb, M, N, K,
                            relu, engine, err, (cudaStream_t)stream);
    return e == 0 ? OD_OK : OD_ECUDA;
}

}  // extern "C"
