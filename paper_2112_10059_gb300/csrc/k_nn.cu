// Kernels of the learned surrogate beside its convolutions (k_conv.cu): head and loss, Adam and
// weight images, input preparation, judge and fallback (see nn_kernels.cuh for layouts).
#include <math.h>

#include <algorithm>

#include "nn_kernels.cuh"
#include "nn_pack.cuh"
#include "sph_common.cuh"
#include "tc_sm103.cuh"

namespace sph {
namespace nn {

using namespace tc;

static unsigned blocks_for(size_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------- head and loss (FP32)
// Bound by memory: 68 B read and 32 B written per voxel.  Each thread keeps its 34 sums over the
// voxels of its stride, so that the warp reductions (5 shuffles a sum) are paid once per thread
// and not once per voxel, and the blocks' partials are few: at 64^3 x 4 the kernel and the sum of
// its partials take the place of 71 + 136 us (4096 blocks, summed by one after another).
__global__ void __launch_bounds__(256) k_head_loss_backward(const uint16_t *__restrict__ f, const float *__restrict__ hw,
                                                            const float *__restrict__ t, uint16_t *__restrict__ g_f,
                                                            float *__restrict__ part, double *__restrict__ loss_part,
                                                            int nvox, float lambda, float eps) {
    pdl_enter();
    __shared__ float wsum[8][34];
    __shared__ double lsum[8];
    float h[34], acc[34];
#pragma unroll
    for (int k = 0; k < 34; ++k) {
        h[k] = hw[k];
        acc[k] = 0.f;
    }
    double ld = 0.0;
    const float inv = 1.0f / (float)nvox;
    for (int m = blockIdx.x * 256 + threadIdx.x; m < nvox; m += gridDim.x * 256) {
        float a[16];
        unpack8(__ldg(reinterpret_cast<const uint4 *>(f + (size_t)m * 16)), a);
        unpack8(__ldg(reinterpret_cast<const uint4 *>(f + (size_t)m * 16 + 8)), a + 8);
        float r = h[32], e = h[33];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            r = fmaf(h[c], a[c], r);
            e = fmaf(h[16 + c], a[c], e);
        }
        const float d = r - t[m];
        const float le = logf(fabsf(d) + eps);
        ld += (double)(d * d + lambda * (e - le) * (e - le));
        const float gr = 2.f * d * inv, ge = 2.f * lambda * (e - le) * inv;
        float g[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            g[c] = a[c] > 0.f ? fmaf(h[c], gr, h[16 + c] * ge) : 0.f;
            acc[c] = fmaf(gr, a[c], acc[c]);
            acc[16 + c] = fmaf(ge, a[c], acc[16 + c]);
        }
        acc[32] += gr;
        acc[33] += ge;
        *reinterpret_cast<uint4 *>(g_f + (size_t)m * 16) = pack8(g);
        *reinterpret_cast<uint4 *>(g_f + (size_t)m * 16 + 8) = pack8(g + 8);
    }
    // head gradient: [j * 16 + c] = sum g_j f_c, [32 + j] = sum g_j
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 34; ++k) {
        float x = acc[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) wsum[warp][k] = x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ld += __shfl_down_sync(0xffffffffu, ld, o);
    if (lane == 0) lsum[warp] = ld;
    __syncthreads();
    if (threadIdx.x < 34) {
        float b = 0.f;
        for (int w = 0; w < 8; ++w) b += wsum[w][threadIdx.x];
        part[(size_t)blockIdx.x * 34 + threadIdx.x] = b;
    } else if (threadIdx.x == 64) {
        double b = 0.0;
        for (int w = 0; w < 8; ++w) b += lsum[w];
        loss_part[blockIdx.x] = b;
    }
}

int head_loss_backward(const uint16_t *f, const float *hw, const float *t, uint16_t *g_f, float *part, double *loss_part,
                       int nvox, float lambda, float eps, cudaStream_t st) {
    const int nb = std::min((int)blocks_for(nvox), HEAD_BLOCKS);
    launch_pdl(k_head_loss_backward, nb, 256, 0, st, f, hw, t, g_f, part, loss_part, nvox, lambda, eps);
    return nb;
}

// ---------------------------------------------------------------- parameters
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, size_t n, float lr, float b1, float b2, float eps, float bc1, float bc2) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
}

// element i of the image of a convolution with ci input and co output channels: its row and
// column, and whether a tap stands there (the last chunk may be padding)
__device__ __forceinline__ bool image_at(int i, int ci, int co, int &tap, int &c, int &n, size_t &at) {
    const int kc = i / (3 * co * 64), within = i % (3 * co * 64), row = within / 64, kk = within % 64, k = kc * 64 + kk;
    tap = 9 * (2 - row / co) + k / ci;
    c = k % ci;
    n = row % co;
    at = (size_t)kc * 3 * co * 64 + row * 64 + (((kk >> 3) ^ (row & 7)) << 3) + (kk & 7);
    return k < 9 * ci;
}

__global__ void k_images(const float *__restrict__ w, int C, int N, uint16_t *__restrict__ img_f,
                         uint16_t *__restrict__ img_d, int nf, int nd) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int tap, c, n;
    size_t at;
    if (i < nf) {
        const bool in = image_at(i, C, N, tap, c, n, at);
        img_f[at] = in ? f2bf(w[(size_t)(n * NTAPS + tap) * C + c]) : 0;
    } else if (i < nf + nd) {
        const bool in = image_at(i - nf, N, C, tap, c, n, at);   // the data gradient: flipped taps, channels exchanged
        img_d[at] = in ? f2bf(w[(size_t)(c * NTAPS + (NTAPS - 1 - tap)) * C + n]) : 0;
    }
}

__global__ void k_f32_to_bf16(const float *__restrict__ in, uint16_t *__restrict__ out, size_t n) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = f2bf(in[i]);
}

void adam(float *p, const float *g, float *m, float *v, size_t n, float lr, float b1, float b2, float eps, float bc1,
          float bc2, cudaStream_t st) {
    if (n) k_adam<<<blocks_for(n), 256, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, bc1, bc2);
}
void make_images(const float *w, int C, int N, uint16_t *img_fwd, uint16_t *img_dgrad, cudaStream_t st) {
    const int nf = conv_image(C, N);
    const int nd = img_dgrad ? conv_image(N, C) : 0;
    k_images<<<blocks_for((size_t)nf + nd), 256, 0, st>>>(w, C, N, img_fwd, img_dgrad, nf, nd);
}
void f32_to_bf16(const float *in, uint16_t *out, size_t n, cudaStream_t st) {
    if (n) k_f32_to_bf16<<<blocks_for(n), 256, 0, st>>>(in, out, n);
}

// ---------------------------------------------------------------- coarse inputs
// Mean and largest value over f^3 blocks (either output may be null), one thread per block, its
// cells in the order x, y, z.  Bound by memory: rows in 16-byte loads where the block edge and the
// pitch allow it (256^3 by 4: 16 us a field and output before, 17 for both outputs).
template <bool VEC>
__global__ void __launch_bounds__(256) k_pool(const float *__restrict__ fine, int nf, int f, float *__restrict__ avg,
                                              float *__restrict__ mx) {
    const int nc = nf / f, x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y, z = blockIdx.z;
    if (x >= nc || y >= nc) return;
    float s = 0.f, m = 0.f;
    for (int k = 0; k < f; ++k) {
        const float *row = fine + ((size_t)(z * f + k) * nf + (size_t)y * f) * nf + (size_t)x * f;
#pragma unroll 4
        for (int j = 0; j < f; ++j, row += nf) {
            if (VEC) {
                for (int i = 0; i < f; i += 4) {
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(row + i));
                    s += v.x; s += v.y; s += v.z; s += v.w;
                    m = fmaxf(fmaxf(m, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
                }
            } else {
                for (int i = 0; i < f; ++i) {
                    s += row[i];
                    m = fmaxf(m, row[i]);
                }
            }
        }
    }
    const size_t p = ((size_t)z * nc + y) * nc + x;
    if (avg) avg[p] = s / (float)(f * f * f);
    if (mx) mx[p] = m;
}

// maxima of up to four non-negative fields (b, d may be null) as float bits
__global__ void k_max4(const float *__restrict__ a, const float *__restrict__ b, const float *__restrict__ c,
                       const float *__restrict__ d, size_t n, unsigned *maxbits) {
    float m[4] = {0.f, 0.f, 0.f, 0.f};
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        m[0] = fmaxf(m[0], a[i]);
        if (b) m[1] = fmaxf(m[1], b[i]);
        m[2] = fmaxf(m[2], c[i]);
        if (d) m[3] = fmaxf(m[3], d[i]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[k] = fmaxf(m[k], __shfl_down_sync(0xffffffffu, m[k], o));
    }
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < 4; ++k) atomicMax(maxbits + k, __float_as_uint(m[k]));
}

// channel 0: log10(I / max I + 1e-8) / 8 + 1 (I averaged over the coarse cell); channel 1:
// |E| / max |E|; channel 2: ln(S / max S + 1e-12) / ln(1e12) + 1 (coarse FMM estimate);
// channel 3: as channel 0 for the largest fine-cell I in the coarse cell (sub-cell peak);
// channels 4..15 zero
__global__ void k_make_inputs(const float *__restrict__ I, const float *__restrict__ E, const float *__restrict__ S,
                              const float *__restrict__ Imax, const unsigned *__restrict__ maxbits,
                              uint16_t *__restrict__ x, size_t n) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float mi = __uint_as_float(maxbits[0]), me = __uint_as_float(maxbits[1]), ms = __uint_as_float(maxbits[2]);
    const float mx = __uint_as_float(maxbits[3]);
    float f[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) f[c] = 0.f;
    f[0] = mi > 0.f ? fmaxf(0.f, log10f(I[i] / mi + 1e-8f) * 0.125f + 1.f) : 0.f;
    f[1] = (E && me > 0.f) ? E[i] / me : 0.f;
    f[2] = ms > 0.f ? fmaxf(0.f, logf(S[i] / ms + 1e-12f) / 27.631021f + 1.f) : 0.f;
    f[3] = (Imax && mx > 0.f) ? fmaxf(0.f, log10f(Imax[i] / mx + 1e-8f) * 0.125f + 1.f) : 0.f;
    *reinterpret_cast<uint4 *>(x + i * 16) = pack8(f);
    *reinterpret_cast<uint4 *>(x + i * 16 + 8) = pack8(f + 8);
}

__global__ void k_make_target(const float *__restrict__ St, const float *__restrict__ Sb, float *__restrict__ t,
                              size_t n) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float a = St[i], b = Sb[i];
    t[i] = (a > 0.f && b > 0.f) ? logf(a / b) : 0.f;
}

void pool_f32(const float *fine, int n_fine, int f, float *avg, float *mx, cudaStream_t st) {
    const int nc = n_fine / f;
    if (nc == 0) return;
    const dim3 grid((nc + 31) / 32, (nc + 7) / 8, nc), block(32, 8);
    if (f % 4 == 0 && (reinterpret_cast<uintptr_t>(fine) & 15) == 0) k_pool<true><<<grid, block, 0, st>>>(fine, n_fine, f, avg, mx);
    else k_pool<false><<<grid, block, 0, st>>>(fine, n_fine, f, avg, mx);
}
void max4(const float *a, const float *b, const float *c, const float *d, size_t n, unsigned *maxbits,
          cudaStream_t st) {
    cudaMemsetAsync(maxbits, 0, 4 * sizeof(unsigned), st);
    if (n) k_max4<<<304, 256, 0, st>>>(a, b, c, d, n, maxbits);
}
void make_inputs(const float *I, const float *E, const float *S, const float *Imax, const unsigned *maxbits,
                 uint16_t *x, size_t n, cudaStream_t st) {
    if (n) k_make_inputs<<<blocks_for(n), 256, 0, st>>>(I, E, S, Imax, maxbits, x, n);
}
void make_target(const float *S_true, const float *S_base, float *t, size_t n, cudaStream_t st) {
    if (n) k_make_target<<<blocks_for(n), 256, 0, st>>>(S_true, S_base, t, n);
}


// ---------------------------------------------------------------- judge and fallback
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ int block_of(int v, int lgD) {
    const int D = 1 << lgD, dm = D - 1, nb = D / JUDGE_BLOCK;
    const int x = v & dm, y = (v >> lgD) & dm, z = v >> (2 * lgD);
    return ((z / JUDGE_BLOCK) * nb + y / JUDGE_BLOCK) * nb + x / JUDGE_BLOCK;
}

// coarse voxel j (0..511) of block b
__device__ __forceinline__ int voxel_in_block(int b, int j, int lgD) {
    const int D = 1 << lgD, nb = D / JUDGE_BLOCK;
    const int bx = b % nb, by = (b / nb) % nb, bz = b / (nb * nb);
    const int x = bx * JUDGE_BLOCK + (j & 7), y = by * JUDGE_BLOCK + ((j >> 3) & 7), z = bz * JUDGE_BLOCK + (j >> 6);
    return (z * D + y) * D + x;
}

__device__ __forceinline__ size_t fine_cell(int v, int lgD, int f, int a) {
    const int D = 1 << lgD, dm = D - 1, n = D * f;
    const int x = v & dm, y = (v >> lgD) & dm, z = v >> (2 * lgD);
    const int ax = a % f, ay = (a / f) % f, az = a / (f * f);
    return ((size_t)(z * f + az) * n + (y * f + ay)) * n + (x * f + ax);
}

__global__ void k_apply_residual(const float *__restrict__ Sc, const float *__restrict__ y, int use_net,
                                 float *__restrict__ Sp, size_t n) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < n) Sp[i] = use_net ? Sc[i] * expf(y[2 * i]) : Sc[i];
}

__global__ void __launch_bounds__(128) k_block_pred_err(const float *__restrict__ y, int lgD, float *__restrict__ pe) {
    const int b = blockIdx.x;                  // one CTA per block, four voxels a thread
    float m = 0.f;
#pragma unroll
    for (int j = threadIdx.x; j < JUDGE_BLOCK * JUDGE_BLOCK * JUDGE_BLOCK; j += 128)
        m = fmaxf(m, expf(y[2 * (size_t)voxel_in_block(b, j, lgD) + 1]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ float w[4];
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) pe[b] = fmaxf(fmaxf(w[0], w[1]), fmaxf(w[2], w[3]));
}

__global__ void k_judge_pick(int lgD, int f, uint64_t seed, int samples, uint8_t *__restrict__ mask,
                             int *__restrict__ sample_vox, int nblocks) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;   // a row of f fine cells of a sample
    const int e = i / (f * f), row = i % (f * f);
    if (e >= nblocks * samples) return;
    const int j = (int)(mix64(seed ^ ((uint64_t)e * 0xD1B54A32D192ED03ull)) & 511u);
    const int v = voxel_in_block(e / samples, j, lgD);
    if (row == 0) sample_vox[e] = v;
    const size_t c = fine_cell(v, lgD, f, row * f);
    for (int a = 0; a < f; ++a) mask[c + a] = 1;
}

// One warp per block, a lane per sample (its cells added in the order x, y, z).
__global__ void __launch_bounds__(128) k_judge_err(const float *__restrict__ Sf, const float *__restrict__ Sp,
                                                   const int *__restrict__ sample_vox, int lgD, int f, int samples,
                                                   float *__restrict__ err, int nblocks) {
    const int b = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= nblocks) return;
    float m = 0.f;
    for (int s = lane; s < samples; s += 32) {
        const int v = sample_vox[b * samples + s];
        float acc = 0.f;
#pragma unroll 4
        for (int r = 0; r < f * f; ++r) {
            const float *row = Sf + fine_cell(v, lgD, f, r * f);
            for (int a = 0; a < f; ++a) acc += row[a];
        }
        acc /= (float)(f * f * f);
        const float rel = acc > 0.f ? fabsf(Sp[v] - acc) / acc : (Sp[v] != 0.f ? INFINITY : 0.f);
        m = fmaxf(m, rel);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) err[b] = m;
}

__global__ void k_fallback_flags(const float *__restrict__ err, const float *__restrict__ pe, int use_pred,
                                 float tol, int nblocks, int *__restrict__ flags, unsigned *counts) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nblocks) return;
    const bool jf = !(err[b] <= tol);
    const bool pf = use_pred && !(pe[b] <= tol);
    flags[b] = (jf || pf) ? 1 : 0;
    if (jf || pf) atomicAdd(counts, 1u);
    if (jf) atomicAdd(counts + 1, 1u);
    if (pf) atomicAdd(counts + 2, 1u);
    atomicMax(counts + 3, __float_as_uint(fminf(err[b], 3.0e38f)));
}

// 16 fine cells of a row per thread (the edge f D is a multiple of 8): one store where they are whole
__global__ void __launch_bounds__(256) k_fallback_mask(const int *__restrict__ flags, int lgD, int f, uint8_t *__restrict__ mask) {
    const int D = 1 << lgD, n = D * f, nb = D / JUDGE_BLOCK, edge = f * JUDGE_BLOCK;
    const int per_row = (n + 15) / 16, i = blockIdx.x * 256 + threadIdx.x;
    if (i >= per_row * n) return;
    const int y = i / per_row, x0 = (i % per_row) * 16, z = blockIdx.y;
    const int *fl = flags + ((z / edge) * nb + y / edge) * nb;
    uint8_t *o = mask + ((size_t)z * n + y) * n + x0;
    uint32_t w[4] = {0, 0, 0, 0};
    int bx = x0 / edge, left = (bx + 1) * edge - x0;      // cells left in the block
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        if (x0 + a < n) w[a / 4] |= (uint32_t)(fl[bx] != 0) << (8 * (a % 4));
        if (--left == 0) {
            bx = min(bx + 1, nb - 1);
            left = edge;
        }
    }
    if ((n & 15) == 0 && (reinterpret_cast<uintptr_t>(mask) & 15) == 0) *reinterpret_cast<uint4 *>(o) = make_uint4(w[0], w[1], w[2], w[3]);
    else
        for (int a = 0; a < 16 && x0 + a < n; ++a) o[a] = (uint8_t)(w[a / 4] >> (8 * (a % 4)));
}

// Sp in passing blocks, the mean of the fine cells (in the order x, y, z) in failing ones
template <bool VEC>
__global__ void __launch_bounds__(256) k_combine(const float *__restrict__ Sp, const float *__restrict__ Sf,
                                                 const int *__restrict__ flags, int lgD, int f, float *__restrict__ out) {
    const int D = 1 << lgD, n = D * f;
    const int v = blockIdx.x * 256 + threadIdx.x;
    if (v >= D * D * D) return;
    if (!flags[block_of(v, lgD)]) {
        out[v] = Sp[v];
        return;
    }
    float acc = 0.f;
    const float *plane = Sf + fine_cell(v, lgD, f, 0);
    for (int k = 0; k < f; ++k, plane += (size_t)n * n) {
        const float *row = plane;
#pragma unroll 4
        for (int j = 0; j < f; ++j, row += n) {
            if (VEC) {
                for (int i = 0; i < f; i += 4) {
                    const float4 q = __ldg(reinterpret_cast<const float4 *>(row + i));
                    acc += q.x; acc += q.y; acc += q.z; acc += q.w;
                }
            } else {
                for (int i = 0; i < f; ++i) acc += row[i];
            }
        }
    }
    out[v] = acc / (float)(f * f * f);
}

static int nblocks_of(int lgD) {
    const int nb = (1 << lgD) / JUDGE_BLOCK;
    return nb * nb * nb;
}

void apply_residual(const float *Sc, const float *y, int use_net, float *Sp, size_t n, cudaStream_t st) {
    if (n) k_apply_residual<<<blocks_for(n), 256, 0, st>>>(Sc, y, use_net, Sp, n);
}
void block_pred_err(const float *y, int lgD, float *pe, cudaStream_t st) {
    k_block_pred_err<<<nblocks_of(lgD), 128, 0, st>>>(y, lgD, pe);
}
void judge_mask(int lgD, int factor, uint64_t seed, int samples, uint8_t *mask, int *sample_vox, cudaStream_t st) {
    const size_t n = (size_t)(factor << lgD);
    cudaMemsetAsync(mask, 0, n * n * n, st);
    const int nb = nblocks_of(lgD);
    k_judge_pick<<<blocks_for((size_t)nb * samples * factor * factor, 128), 128, 0, st>>>(lgD, factor, seed, samples, mask,
                                                                                        sample_vox, nb);
}
void judge_err(const float *Sf, const float *Sp, const int *sample_vox, int lgD, int factor, int samples, float *err,
               cudaStream_t st) {
    const int nb = nblocks_of(lgD);
    k_judge_err<<<blocks_for(nb, 4), 128, 0, st>>>(Sf, Sp, sample_vox, lgD, factor, samples, err, nb);
}
void fallback_flags(const float *err, const float *pe, int use_pred, float tol, int nblocks, int *flags,
                    unsigned *counts, cudaStream_t st) {
    cudaMemsetAsync(counts, 0, 4 * sizeof(unsigned), st);
    k_fallback_flags<<<blocks_for(nblocks, 128), 128, 0, st>>>(err, pe, use_pred, tol, nblocks, flags, counts);
}
void fallback_mask(const int *flags, int lgD, int factor, uint8_t *mask, cudaStream_t st) {
    const int n = factor << lgD;
    k_fallback_mask<<<dim3(blocks_for((size_t)((n + 15) / 16) * n), n), 256, 0, st>>>(flags, lgD, factor, mask);
}
void combine(const float *Sp, const float *Sf, const int *flags, int lgD, int factor, float *out, cudaStream_t st) {
    const size_t n = (size_t)1 << (3 * lgD);
    if (factor % 4 == 0 && (reinterpret_cast<uintptr_t>(Sf) & 15) == 0)
        k_combine<true><<<blocks_for(n), 256, 0, st>>>(Sp, Sf, flags, lgD, factor, out);
    else
        k_combine<false><<<blocks_for(n), 256, 0, st>>>(Sp, Sf, flags, lgD, factor, out);
}

}  // namespace nn
}  // namespace sph
