// Kernels of the learned surrogate: a 4-level U-Net-like BF16 convolutional network on a
// coarse grid (16-32 channels), trained and run by the kernels in k_nn.cu.
//
// Tensors are channels-last [B][D][D][D][C] (x fastest, then y, z, batch), BF16 stored
// as uint16_t, D a power of two (D = 1 << lg).  A 3x3x3 convolution with zero padding is
// an implicit GEMM
//     out[m][n] = sum_k A[m][k] W[n][k],   k = tap * C + c,
//     A[m][tap*C + c] = x[m + offset(tap)][c]   (0 outside the grid),
//     tap = 9 (dz+1) + 3 (dy+1) + (dx+1),
// run on the tensor cores (tcgen05, BF16 in, FP32 accumulate in TMEM).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace sph {
namespace nn {

constexpr int NTAPS = 27;
// Weight image of a convolution, the B operand of k_conv_tc in its shared-memory layout: rows
// (2 - dz) N + n, columns k = (3 dy + dx) C + c, as chunks of 64 columns [3 N][64], each K-major
// with the 128-byte swizzle.  Elements (BF16):
__host__ __device__ constexpr int conv_image(int C, int N) { return (9 * C + 63) / 64 * 3 * N * 64; }

// Epilogues of a convolution beside the plain one (bias, ReLU, residual, mask), each in place of
// a pass over memory; all use the convolution's result as rounded to BF16.
enum {
    CONV_PLAIN = 0,
    CONV_POOL,     // out2[parent] = scale * (sum of the 8 children), 0 where mask2 <= 0 (mask2 given); out optional
    CONV_PAIR,     // out2 = out + add2 (add2 given), or out where mask2 > 0 and 0 elsewhere; out optional
    CONV_HEAD      // y = head weights . out + head bias (FP32); out optional
};

struct ConvArgs {
    const uint16_t *x;       // [nvox][C]
    const uint16_t *w;       // weight image, conv_image(C, N) elements
    const float *bias;       // [N] or nullptr
    const uint16_t *add;     // [nvox][N] or nullptr: added after the ReLU
    const uint16_t *mask;    // [nvox][N] or nullptr: zero where mask <= 0 (applied last)
    uint16_t *out;           // [nvox][N]
    int relu;
    int nvox, lg;
    int *err;                // bit 0: a bounded wait expired
    int up = 0;              // 1: x holds the grid of half the edge, read at each voxel's parent
    int epi = CONV_PLAIN;
    const uint16_t *add2 = nullptr, *mask2 = nullptr;
    uint16_t *out2 = nullptr;
    float scale = 1.f;
    const float *hw = nullptr;   // [34] head weights and bias
    float *y = nullptr;      // [nvox][2]
};

struct WgradArgs {
    const uint16_t *x;       // [nvox][C] layer input
    const uint16_t *dz;      // [nvox][N] gradient w.r.t. the layer's pre-activation
    float *part;             // [wgrad_splits][27 C + 1][N]: each CTA's sums, row 27 C the bias gradient's
    int nvox, lg;
    int *err;
    int up = 0;              // 1: x holds the grid of half the edge, read at each voxel's parent
};
// slices that one weight gradient writes (its CTAs)
int wgrad_splits(int C, int N, int lg, int nvox);

// Sums over the slices of several layers, each written as w [N][27][C] then b [N]; a layer with
// C = 0 is the head (N = 34 elements as they are, and the loss).
struct WgradSum {
    const float *part;
    float *grad;
    int C, N, splits, block0;
    __host__ __device__ int elems() const { return (NTAPS * C + 1) * N; }
};
struct WgradSums {
    WgradSum l[13];
    int layers = 0;
    const double *loss_part = nullptr;
    double *loss = nullptr;
};
void wgrad_sums(WgradSums &t, cudaStream_t st);
constexpr int HEAD_BLOCKS = 608;       // blocks of the head's loss / gradient kernel at most

// set the shared-memory limits of every instantiation (call once, outside graph capture)
void init_attributes();
// C, N in {16, 32}; returns 0, or -1 for an unsupported shape
int conv(const ConvArgs &a, int C, int N, cudaStream_t st);
int wgrad(const WgradArgs &a, int C, int N, cudaStream_t st);
// out [nvox][C] on the grid of edge 2^lg: coarse (half the edge) up-sampled + fine, or with a mask
// mask > 0 ? fine + coarse / 8 : 0
void expand(const uint16_t *coarse, const uint16_t *fine, const uint16_t *mask, uint16_t *out, int nvox, int lg, int C,
            cudaStream_t st);

// loss of the residual r = y0 against t and of the error head e = y1 against log(|r - t| + eps)
// (y[m][j] = sum_c hw[j][c] f[m][c] + hb[j]); writes the masked gradient of f (BF16) and each
// block's part of the head's gradient (part [blocks][34]) and of the loss (loss_part [blocks]);
// returns the number of blocks
int head_loss_backward(const uint16_t *f, const float *hw, const float *t, uint16_t *g_f, float *part, double *loss_part,
                       int nvox, float lambda, float eps, cudaStream_t st);

// parameters: per layer w [N][27][C] then b [N] (FP32 master copy)
void adam(float *p, const float *g, float *m, float *v, size_t n, float lr, float b1, float b2, float eps,
          float bc1, float bc2, cudaStream_t st);
void make_images(const float *w, int C, int N, uint16_t *img_fwd, uint16_t *img_dgrad, cudaStream_t st);
void f32_to_bf16(const float *in, uint16_t *out, size_t n, cudaStream_t st);

// coarse inputs of the network from pooled fields
// mean and largest value over f^3 blocks of an n_fine^3 field (avg or mx may be null)
void pool_f32(const float *fine, int n_fine, int f, float *avg, float *mx, cudaStream_t st);
void max4(const float *a, const float *b, const float *c, const float *d, size_t n, unsigned *maxbits,
          cudaStream_t st);
void make_inputs(const float *I, const float *E, const float *S, const float *Imax, const unsigned *maxbits,
                 uint16_t *x, size_t n, cudaStream_t st);
void make_target(const float *S_true, const float *S_base, float *t, size_t n, cudaStream_t st);

}  // namespace nn
}  // namespace sph

namespace sph {
namespace nn {
// ---- judge and fallback of the surrogate (single sample, coarse grid D = 1 << lgD, blocks of
// 8^3 coarse voxels, fine grid n = factor * D)
constexpr int JUDGE_BLOCK = 8;
// S_pred = S_coarse * exp(r) (use_net) or S_coarse
void apply_residual(const float *Sc, const float *y, int use_net, float *Sp, size_t n, cudaStream_t st);
// per block: max over its voxels of exp(e) (the error head's estimate of |ln S_pred - ln S|)
void block_pred_err(const float *y, int lgD, float *pe, cudaStream_t st);
// mark `samples` seeded coarse voxels per block: their factor^3 fine cells in mask (cleared here)
void judge_mask(int lgD, int factor, uint64_t seed, int samples, uint8_t *mask, int *sample_vox, cudaStream_t st);
// per block: max relative error of S_pred against the pooled fine S at the sampled voxels
void judge_err(const float *Sf, const float *Sp, const int *sample_vox, int lgD, int factor, int samples, float *err,
               cudaStream_t st);
// flags[b] = err > tol || (use_pred && pe > tol); counts: fallback, judged fail, predicted fail, max err bits
void fallback_flags(const float *err, const float *pe, int use_pred, float tol, int nblocks, int *flags,
                    unsigned *counts, cudaStream_t st);
void fallback_mask(const int *flags, int lgD, int factor, uint8_t *mask, cudaStream_t st);
void combine(const float *Sp, const float *Sf, const int *flags, int lgD, int factor, float *out, cudaStream_t st);
}  // namespace nn
}  // namespace sph
