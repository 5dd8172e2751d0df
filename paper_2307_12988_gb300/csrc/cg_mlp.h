// cg_mlp.h -- the training object of the learned initial guess, shared by
// cg_mlp.cu (entry points, any batch) and cg_train.cu (the training step on
// prepared operand images).
#pragma once
#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

namespace cg {
struct TrainImages;
}

struct cg_mlp_s {
    int device = 0;
    int n_in = 0, H = 0, n_out = 0, max_batch = 0;
    int64_t np = 0;
    int64_t step = 0;                 // Adam steps taken
    float* theta = nullptr;           // [np] parameters
    float* grad = nullptr;            // [np]
    float* m = nullptr;               // [np] Adam first moment
    float* v = nullptr;               // [np] Adam second moment
    // activations and gradients of one batch
    float *xb = nullptr, *tb = nullptr;          // gathered batch [max_batch][n_in / n_out]
    float *z1 = nullptr, *a1 = nullptr, *z2 = nullptr, *a2 = nullptr, *out = nullptr;
    float *g_out = nullptr, *g_z2 = nullptr, *g_z1 = nullptr;
    float* part = nullptr;            // [kLossBlocks] loss partial sums
    float* loss = nullptr;            // [1]
    float* ws = nullptr;              // K-split partial sums of the weight gradients
    int* err = nullptr;               // [1] set by a matrix-product block whose bounded wait ran out
    cg::TrainImages* img = nullptr;   // operand images of the training step (cg_train.cu)
    std::vector<float> in_mean, in_scale, out_mean, out_scale;
};

namespace cg {

constexpr int kLossBlocks = 256;
constexpr float kGeluK = 0.7978845608028654f;   // sqrt(2 / pi)
constexpr float kGeluC = 0.044715f;
constexpr int kGMaxSplit = 8;       // K ranges of one output tile at most
constexpr int kGK = 32;             // K elements per block (one 128-byte swizzle row of FP32)
constexpr int kGM = 128;            // rows per tile (MMA M)
constexpr int kTrainRows = 16384;   // batches up to this many rows take the training step on images

__device__ __forceinline__ float gelu_f(float z)
{
    const float t = tanhf(kGeluK * fmaf(kGeluC * z * z, z, z));
    return 0.5f * z * (1.0f + t);
}
__device__ __forceinline__ float gelu_grad_f(float z)
{
    const float t = tanhf(kGeluK * fmaf(kGeluC * z * z, z, z));
    return 0.5f * (1.0f + t) + 0.5f * z * (1.0f - t * t) * kGeluK * fmaf(3.0f * kGeluC, z * z, 1.0f);
}
// FP32 -> TF32, round to nearest (ties away), as a 32-bit pattern with the
// low 13 mantissa bits zero
__device__ __forceinline__ float tf32_rn(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

struct Offsets {
    int64_t W1, b1, W2, b2, W3, b3;
};
inline Offsets offsets(const cg_mlp_s* m)
{
    Offsets o;
    o.W1 = 0;
    o.b1 = o.W1 + static_cast<int64_t>(m->H) * m->n_in;
    o.W2 = o.b1 + m->H;
    o.b2 = o.W2 + static_cast<int64_t>(m->H) * m->H;
    o.W3 = o.b2 + m->H;
    o.b3 = o.W3 + static_cast<int64_t>(m->n_out) * m->H;
    return o;
}

// Tile width and K ranges of the generic product (cg_mlp.cu); the training
// step splits K the same way, so both give the same sums.
struct SplitRule {
    int bn, kb_per, splits;
};
SplitRule split_rule(int M, int N, int K, bool can_split);

// the training step on operand images (cg_train.cu); create: the weights' images
cudaError_t train_create(cg_mlp_s* m);
// *ready: batches of `rows` take the step on images (the first such call on a
// stream that is not capturing allocates the batch images)
cudaError_t train_ready(cg_mlp_s* m, int rows, cudaStream_t s, bool* ready);
void train_destroy(cg_mlp_s* m);
// weight images from the parameters (after the parameters were set)
cudaError_t train_refresh(cg_mlp_s* m, cudaStream_t s);
struct TrainBatch {
    const float *x, *t;        // [n_src][n_in], [n_src][n_out]
    int64_t n_src;
    const int32_t* perm;       // row i of the batch is row perm[i], or null (row i)
    int rows;
};
struct AdamStep {
    float lr, b1, b2, eps, bc1, bc2;
};
// an Adam step on m->grad
cudaError_t train_adam(cg_mlp_s* m, const AdamStep& a, cudaStream_t s);
// x of a batch into its images
cudaError_t train_prepare(cg_mlp_s* m, const TrainBatch& b, cudaStream_t s);
// forward and backward of the prepared batch; then the gradient (into
// m->grad), the loss and, where given, an Adam step and the next batch's images
cudaError_t train_step(cg_mlp_s* m, const TrainBatch& b, float* loss_copy, const AdamStep* adam,
                       const TrainBatch* next, cudaStream_t s);

}  // namespace cg
