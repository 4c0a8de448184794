// 3x3x3 convolutions of the learned surrogate on tcgen05 (see nn_kernels.cuh for the tensors).
//
// k_conv_tc<C, N>: forward, or data gradient with a flipped, transposed weight image.  The
// implicit GEMM's A operand is never formed: a CTA keeps whole z-planes of its column's input
// (8 x 16 output voxels plus the halo, 10 x 18) in shared memory, one 16-byte unit of 8
// channels per voxel and channel group, x fastest.  Eight x-neighbours are then one
// unswizzled K-major core matrix (8 rows x 16 bytes), the 16 rows of the tile are its M
// repeats (stride one halo row), the channel groups its K repeats -- and the operand of any
// (dy, dx) tap is the same plane read from a start address moved by whole units.  A voxel's
// input is copied 1.4 times (halo) instead of 27 times.
// What bounds it is the tensor core's read of A, 4 KB per MMA: measured 39 clocks per M = 128,
// K = 16 MMA at N = 16, 40 at 32, 44 at 48, 56 at 96 (whatever the core matrices' alignment).
// So N is widened with the plane's other uses: plane z is the dz = 2, 1, 0 tap of the outputs
// z - 1, z, z + 1, whose accumulators lie side by side in TMEM (a ring of eight), and one MMA
// of N = 3 x out channels takes the place of three; an output still sums its taps in the order
// dz, dy, dx.  CTAs march in z through equal shares of the tiles, planes loaded three ahead, one
// warp issuing MMAs under the four others' copies and epilogues.
// 16 -> 16 channels at 64^3 x 4: 199 us gathering 27 taps, 38 with N = 16, 29 with N = 48;
// 32 -> 16: 391, 68, 53 (32 -> 32 at 32^3 x 4: 83, 21, 15).
//
// Every mbarrier wait is bounded; on expiry the kernel sets its error flag and carries
// on (the result is then invalid and the host reports it).
#include "nn_kernels.cuh"
#include "nn_pack.cuh"
#include "sph_common.cuh"
#include "tc_sm103.cuh"

namespace sph {
namespace nn {

using namespace tc;

constexpr uint32_t NN_WAIT = 1u << 22;

// ---------------------------------------------------------------- convolution (forward / data gradient)
constexpr int CX = 8, CY = 16;                  // output voxels of a tile: 8 (x) x 16 (y)
constexpr int PX = CX + 2, PY = CY + 2;         // its input plane with the halo
constexpr int AHEAD = 3;                        // planes loaded ahead of the one in use (forward: 223 us with 2, 206 with 3, 213 with 4)
constexpr int RING = AHEAD + 2;                 // planes in shared memory
constexpr int ACCS = 8;                         // accumulators in TMEM (at least 4)
// bytes between the channel groups of a plane: such that the 8 units a quarter-warp copies
// (2 groups x 4 voxels, or 4 groups x 2) fall into different banks
__host__ __device__ constexpr uint32_t group_bytes(int C) { return PX * PY * 16 + (C == 16 ? 0 : 32); }
__host__ __device__ constexpr uint32_t plane_bytes(int C) { return (uint32_t)(C / 8) * group_bytes(C); }
__host__ __device__ constexpr uint32_t weight_bytes(int C, int N) { return (uint32_t)conv_image(C, N) * 2; }
__host__ __device__ constexpr uint32_t conv_smem(int C, int N) {
    return 1024 + weight_bytes(C, N) + RING * plane_bytes(C) + 64;
}

__device__ __forceinline__ uint8_t *align1024(uint8_t *p) {
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

// until at most `pending` of this thread's copy groups are in flight
__device__ __forceinline__ void cp_async_wait_upto(int pending) {
    if (pending <= 0) cp_async_wait<0>();
    else if (pending == 1) cp_async_wait<1>();
    else if (pending == 2) cp_async_wait<2>();
    else cp_async_wait<3>();
}

// The planes a CTA passes through: for each column's run of output tiles zs .. ze - 1 the planes
// zs - 1 .. ze, in order.  An output is complete once the plane above it has been used.
struct PlaneCursor {
    int next, t1, lg;                         // the next run's first tile, the CTA's end
    int col = 0, z = 0, zs = 0, ze = -1;
    __device__ PlaneCursor(int t0, int t1_, int lg_) : next(t0), t1(t1_), lg(lg_) {}
    __device__ bool step() {                  // to the next plane; true where a run begins
        if (z < ze) {
            ++z;
            return false;
        }
        const int D = 1 << lg;
        col = next >> lg;
        zs = next & (D - 1);
        ze = min(D, zs + t1 - next);
        next += ze - zs;
        z = zs - 1;
        return true;
    }
};

template <int C, int N, int EPI>
__global__ void __launch_bounds__(160) k_conv_tc(ConvArgs a) {
    pdl_enter();
    constexpr int CG = C / 8;
    constexpr uint32_t GB = group_bytes(C), PB = plane_bytes(C), WB = weight_bytes(C, N);
    constexpr int NU = (PX * PY * CG + 127) / 128;   // units copied per thread and plane
    extern __shared__ uint8_t raw[];
    uint8_t *base = align1024(raw);
    // [0], [1]: a plane's MMAs are done; [2], [3]: it is in shared memory; [4]: weights
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + WB + RING * PB);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 5);
    int *eflag = reinterpret_cast<int *>(tslot + 1);
    __shared__ float sbias[N];
    __shared__ float shead[EPI == CONV_HEAD ? 34 : 1];

    const int r = threadIdx.x, warp = r >> 5;
    const int lg = a.lg, D = 1 << lg;
    const int ltx = lg > 3 ? lg - 3 : 0, lty = lg > 4 ? lg - 4 : 0;   // tiles per row and plane (log2)
    const int ntiles = (a.nvox >> (2 * lg)) << (ltx + lty);           // (batch x D) planes of tiles
    // equal shares of consecutive tiles (z fastest); whole z-pairs where the epilogue pools
    const int g2 = EPI == CONV_POOL ? 1 : 0;
    const int t0 = (int)((long long)(ntiles >> g2) * blockIdx.x / gridDim.x) << g2;
    const int t1 = (int)((long long)(ntiles >> g2) * (blockIdx.x + 1) / gridDim.x) << g2;
    if (t0 >= t1) return;                     // uniform over the CTA, before any allocation

    if (warp == 4) {
        tmem_alloc(smem_u32(tslot), ACCS * N);
        tmem_relinquish();
    }
    if (r < N) sbias[r] = a.bias ? a.bias[r] : 0.f;
    if constexpr (EPI == CONV_HEAD) {
        if (r < 34) shead[r] = a.hw[r];
    }
    if (r == 0) {
        mbar_init(smem_u32(&bar[0]), 1);
        mbar_init(smem_u32(&bar[1]), 1);
        mbar_init(smem_u32(&bar[2]), 128);
        mbar_init(smem_u32(&bar[3]), 128);
        mbar_init(smem_u32(&bar[4]), 1);
        *eflag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tslot;
    const uint32_t wbase = smem_u32(base), ring = wbase + WB;
    const int planes = t1 - t0 + 2 * (((t1 - 1) >> lg) - (t0 >> lg) + 1);

    if (warp == 4) {                          // ---- one thread issues every MMA
        if (elect_one()) {
            const uint64_t ad0 = sdesc_none(0, GB, PX * 16), bd0 = sdesc_sw128(0);
            mbar_expect_tx(smem_u32(&bar[4]), WB);
            bulk_g2s(wbase, a.w, WB, smem_u32(&bar[4]));
            if (!mbar_wait_bounded(smem_u32(&bar[4]), 0, NN_WAIT)) *eflag = 1;
            PlaneCursor p(t0, t1, lg);
            int q = 0;                        // outputs of the runs before this one
            for (int i = 0; i < planes; ++i) {
                const int len = p.ze - p.zs;
                if (p.step() && i > 0) q += len;
                if (!mbar_wait_bounded(smem_u32(&bar[2 + (i & 1)]), (i >> 1) & 1, NN_WAIT)) *eflag = 1;
                fence_after_sync();
                // the outputs lo .. hi use this plane: rows (lo - z + 1) N .. of the weight image
                const int lo = max(p.z - 1, p.zs), hi = min(p.z + 1, p.ze - 1), cnt = hi - lo + 1;
                const int blk = (q + lo - p.zs) % ACCS, c1 = min(cnt, ACCS - blk);   // c1 before the ring's end
                const uint64_t ad = ad0 + ((ring + (uint32_t)(i % RING) * PB) >> 4);
                const uint64_t bd = bd0 + ((wbase + (uint32_t)(lo - p.z + 1) * N * 128) >> 4);
                auto slice = [&](int k, int from, int to, uint32_t accumulate) {   // K = 16 slice k, outputs from .. to - 1
                    const int tap = k / (C / 16), h = k % (C / 16);
                    mma_bf16(tmem + (uint32_t)((blk + from) % ACCS * N),
                             ad + (((uint32_t)((tap / 3) * PX + tap % 3) * 16 + 2 * h * GB) >> 4),
                             bd + ((uint32_t)(k / 4) * 3 * N * 128 + (uint32_t)(k % 4) * 32 + (uint32_t)from * N * 128 >> 4),
                             idesc_bf16_f32(128, (to - from) * N), accumulate);
                };
                // the output that begins here takes its first slice without its accumulator
                const int old = hi == p.z + 1 ? cnt - 1 : cnt;
                if (old > 0) slice(0, 0, min(old, c1), 1u);
                if (old > c1) slice(0, c1, old, 1u);
                if (old < cnt) slice(0, old, cnt, 0u);
                if (c1 == cnt) {
#pragma unroll
                    for (int k = 1; k < 9 * C / 16; ++k) slice(k, 0, cnt, 1u);
                } else {
#pragma unroll
                    for (int k = 1; k < 9 * C / 16; ++k) {
                        slice(k, 0, c1, 1u);
                        slice(k, c1, cnt, 1u);
                    }
                }
                mma_commit(smem_u32(&bar[i & 1]));
            }
        }
    } else {                                  // ---- four warps copy planes and write results
        const int up = a.up, lgi = lg - up;   // input grid (half the edge when up-sampled on load)
        int off[NU], loaded = 0, slot = 0;    // off: a unit's place in its plane, and whether it is in the grid
        uint32_t in = 0, dst[NU];
        const uint16_t *xcol = a.x;
        PlaneCursor lp(t0, t1, lg);
#pragma unroll
        for (int j = 0; j < NU; ++j) {
            const int u = r + 128 * j;
            dst[j] = ring + (uint32_t)(u % CG) * GB + (uint32_t)(u / CG) * 16;
        }
        auto load_next = [&]() {              // the next plane, one copy group
            if (lp.step()) {                  // another column
                const int x0 = (lp.col & ((1 << ltx) - 1)) * CX - 1, y0 = ((lp.col >> ltx) & ((1 << lty) - 1)) * CY - 1;
                xcol = a.x + ((size_t)(lp.col >> (ltx + lty)) << (3 * lgi)) * C;
                in = 0;
#pragma unroll
                for (int j = 0; j < NU; ++j) {
                    const int u = r + 128 * j, v = u / CG, cg = u % CG;
                    const int x = x0 + v % PX, y = y0 + v / PX;
                    const bool ok = (unsigned)x < (unsigned)D && (unsigned)y < (unsigned)D;
                    off[j] = ok ? (((y >> up) << lgi) + (x >> up)) * C + cg * 8 : 0;
                    in |= (ok ? 16u : 0u) << j;
                }
            }
            const bool zin = (unsigned)lp.z < (unsigned)D;
            const uint32_t zmask = zin ? in : 0u;
            const uint16_t *xp = xcol + ((size_t)((zin ? lp.z : 0) >> up) << (2 * lgi)) * C;
#pragma unroll
            for (int j = 0; j < NU; ++j)
                if (r + 128 * j < PX * PY * CG) cp_async16(dst[j] + (uint32_t)slot * PB, xp + off[j], zmask >> j & 16u);
            slot = slot == RING - 1 ? 0 : slot + 1;
            cp_async_commit();
            ++loaded;
        };

        float pool[EPI == CONV_POOL ? N : 1];
        bool valid = false;                   // this thread's voxel of the run's tiles
        size_t at = 0, atp = 0;               // its place at z = 0, and its parent's
        auto place = [&](int col) {
            const int x = (col & ((1 << ltx) - 1)) * CX + (r & 7), y = ((col >> ltx) & ((1 << lty) - 1)) * CY + (r >> 3);
            const size_t b = (size_t)(col >> (ltx + lty));
            valid = x < D && y < D;
            at = (b << (3 * lg)) + ((size_t)y << lg) + x;
            if (EPI == CONV_POOL) atp = (b << (3 * lg - 3)) + ((size_t)(y >> 1) << (lg - 1)) + (x >> 1);
        };
        auto epilogue = [&](int z, int nth) { // output nth of the CTA's, at plane z of its run
            float v[N];
            const uint32_t acc = tmem + (uint32_t)(nth % ACCS * N) + ((uint32_t)(warp * 32) << 16);
            tmem_ld16(acc, v);
            if constexpr (N == 32) tmem_ld16(acc + 16, v + 16);
            fence_before_sync();              // read before this thread's next arrival frees the accumulator
            const size_t o = (at + ((size_t)z << (2 * lg))) * N;
            uint4 q[N / 8];
#pragma unroll
            for (int g = 0; g < N / 8; ++g) {
                float f[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float s = v[8 * g + j];
                    if (a.bias) s += sbias[8 * g + j];
                    if (a.relu) s = fmaxf(s, 0.f);
                    f[j] = s;
                }
                if constexpr (EPI == CONV_PLAIN) {
                    if (a.add && valid) {
                        float ad[8];
                        unpack8(*reinterpret_cast<const uint4 *>(a.add + o + 8 * g), ad);
#pragma unroll
                        for (int j = 0; j < 8; ++j) f[j] += ad[j];
                    }
                    if (a.mask && valid) {
                        float mk[8];
                        unpack8(*reinterpret_cast<const uint4 *>(a.mask + o + 8 * g), mk);
#pragma unroll
                        for (int j = 0; j < 8; ++j) f[j] = mk[j] > 0.f ? f[j] : 0.f;
                    }
                }
                q[g] = pack8(f);
                if (valid && (EPI == CONV_PLAIN || a.out)) *reinterpret_cast<uint4 *>(a.out + o + 8 * g) = q[g];
            }
            if constexpr (EPI == CONV_PAIR) {
                if (valid) {
#pragma unroll
                    for (int g = 0; g < N / 8; ++g) {
                        float f[8], s[8];
                        unpack8(q[g], f);
                        unpack8(__ldg(reinterpret_cast<const uint4 *>((a.add2 ? a.add2 : a.mask2) + o + 8 * g)), s);
#pragma unroll
                        for (int j = 0; j < 8; ++j) f[j] = a.add2 ? f[j] + s[j] : (s[j] > 0.f ? f[j] : 0.f);
                        *reinterpret_cast<uint4 *>(a.out2 + o + 8 * g) = pack8(f);
                    }
                }
            }
            if constexpr (EPI == CONV_POOL) {
                // children in the order x, y, z: this lane, its x, y and diagonal neighbour (lanes
                // r + 1, r + 8, r + 9 of the same warp), then the next plane's four
#pragma unroll
                for (int g = 0; g < N / 8; ++g) {
                    float s[8], f[8];
                    unpack8(q[g], s);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int src = (c & 1) + 8 * (c >> 1);
                        if (c > 0) {
                            uint4 n;
                            n.x = __shfl_down_sync(0xffffffffu, q[g].x, src);
                            n.y = __shfl_down_sync(0xffffffffu, q[g].y, src);
                            n.z = __shfl_down_sync(0xffffffffu, q[g].z, src);
                            n.w = __shfl_down_sync(0xffffffffu, q[g].w, src);
                            unpack8(n, f);
                        } else {
                            unpack8(q[g], f);
                        }
#pragma unroll
                        for (int j = 0; j < 8; ++j) pool[8 * g + j] = c == 0 && !(z & 1) ? 0.f + s[j] : pool[8 * g + j] + f[j];
                    }
                }
                if ((z & 1) && valid && !(r & 1) && !(r & 8)) {
                    const size_t op = (atp + ((size_t)(z >> 1) << (2 * lg - 2))) * N;
#pragma unroll
                    for (int g = 0; g < N / 8; ++g) {
                        float f[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) f[j] = a.scale * pool[8 * g + j];
                        if (a.mask2) {
                            float mk[8];
                            unpack8(__ldg(reinterpret_cast<const uint4 *>(a.mask2 + op + 8 * g)), mk);
#pragma unroll
                            for (int j = 0; j < 8; ++j) f[j] = mk[j] > 0.f ? f[j] : 0.f;
                        }
                        *reinterpret_cast<uint4 *>(a.out2 + op + 8 * g) = pack8(f);
                    }
                }
            }
            if constexpr (EPI == CONV_HEAD) {
                float f[16], r0 = shead[32], e0 = shead[33];
                unpack8(q[0], f);
                unpack8(q[1], f + 8);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    r0 = fmaf(shead[c], f[c], r0);
                    e0 = fmaf(shead[16 + c], f[c], e0);
                }
                if (valid) {                  // y is the caller's: its two floats need not be 8-byte aligned
                    float *y = a.y + o / N * 2;
                    if ((reinterpret_cast<uintptr_t>(a.y) & 7) == 0) {
                        *reinterpret_cast<float2 *>(y) = make_float2(r0, e0);
                    } else {
                        y[0] = r0;
                        y[1] = e0;
                    }
                }
            }
        };

        PlaneCursor p(t0, t1, lg);            // the plane whose MMAs are waited for
        int q = 0;
        for (int i = 0; i <= planes; ++i) {
            if (i < planes) {
                // plane i + AHEAD takes the slot of plane i - 2, whose MMAs are done (waited for below)
                while (loaded < planes && loaded <= i + AHEAD) load_next();
                cp_async_wait_upto(loaded - 1 - i);
                fence_proxy_async_smem();
                mbar_arrive(smem_u32(&bar[2 + (i & 1)]));
            }
            if (i > 0) {
                if (p.step()) place(p.col);
                if (!mbar_wait_bounded(smem_u32(&bar[(i - 1) & 1]), ((i - 1) >> 1) & 1, NN_WAIT)) *eflag = 1;
                if (p.z > p.zs) {
                    fence_after_sync();
                    epilogue(p.z - 1, q++);
                }
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    if (r == 0 && *eflag) atomicOr(a.err, 1);
    if (warp == 4) tmem_dealloc(tmem, ACCS * N);
}

// ---------------------------------------------------------------- weight gradient
// dW[n][tap][c] = sum over voxels m of dz[m][n] x[m + off(tap)][c]: M = (tap, c), N = out
// channels, K = voxels.  Both operands are K x M (N) with the channels contiguous, i.e. MN-major
// as the tensors lie: a core matrix is 8 x-neighbours of one 8-channel group, the same 16-byte
// units as above, so nothing is transposed or repeated.  Shared memory holds, per y row, the
// units of [z - 1, z, z + 1][channel group][x] at one stride; the core matrices of three
// neighbouring rows then follow each other at that stride in the order (dy, dz, group), which
// makes M tiles of 128 rows that cover the nine (dy, dz) taps (a tenth of the rows is padding).
// The three dx are dz at three x shifts, side by side as N = 3 x out channels: an MMA is bound by
// reading its 4 KB of x, whatever its N (16 -> 16 at 64^3 x 4: 289 us with both operands
// transposed in registers, 78 with the dx as three MMAs on shifted x, 40 so; 32 -> 16: 606,
// 187, 66).  A constant plane of ones behind the three z gives the bias gradient as one more
// row.  CTAs march in y through equal shares of the (sample, z, x segment) columns, 64 voxels an
// iteration, rows in a ring whose first slots are mirrored behind its last so that three rows
// always follow each other.  Each CTA's sums go to its own slice of `part`; k_wgrad_sum adds
// the slices in order (training is reproducible bit for bit).
__host__ __device__ constexpr int wg_block(int C) { return 3 * (C / 8) + 1; }               // core-matrix columns per row
__host__ __device__ constexpr int wg_tiles(int C) { return (3 * wg_block(C) + 15) / 16; }   // M tiles per dx
__host__ __device__ constexpr int wg_cols(int C, int N) {                                   // TMEM columns (power of 2)
    return 3 * wg_tiles(C) * N <= 128 ? 128 : 3 * wg_tiles(C) * N <= 256 ? 256 : 512;
}
// 64 voxels of one channel group of dz, padded as the x stride below; a slot holds three shifts
__host__ __device__ constexpr uint32_t wg_dz_group(int N) { return 1024 + (N == 16 ? 64 : 32); }
__host__ __device__ constexpr uint32_t wg_dz_slot(int N) { return 3 * (uint32_t)(N / 8) * wg_dz_group(N); }

struct WgradShape {      // how a layer's voxels are cut, from its edge alone
    int lgx;             // x segment of a row: 2^lgx voxels, 8 .. 64
    int rpi, lipc;       // rows per iteration, iterations per column (log2)
    int ring, mirror;    // rows in the ring, slots repeated behind it
    uint32_t stride;     // bytes between core-matrix columns
    int cols;            // core-matrix columns in shared memory
    int iters;           // iterations in all
};
static WgradShape wgrad_shape(int C, int lg, int nvox) {
    WgradShape s;
    const int lge = lg < 3 ? 3 : lg;
    s.lgx = lge > 6 ? 6 : lge;
    s.rpi = 64 >> s.lgx;
    s.lipc = lge - (6 - s.lgx);
    s.ring = 2 * (s.rpi + 2) + 1;
    s.mirror = s.lgx == 3 ? 3 : 2;
    // the 8 units a quarter-warp copies (2 groups x 4 voxels, or 4 x 2) in different banks
    s.stride = (16u << s.lgx) + (C == 16 ? 64 : 32);
    const int cb = wg_block(C);
    const int read = (s.ring - 1) * cb + 16 * wg_tiles(C) + (s.lgx == 3 ? cb : 0);   // the padding rows' reads end here
    s.cols = (s.ring + s.mirror) * cb > read ? (s.ring + s.mirror) * cb : read;
    s.iters = (nvox >> (2 * lg)) << (lge - s.lgx + s.lipc);
    return s;
}
static uint32_t wgrad_smem(int C, int N, const WgradShape &s) { return 128 + (uint32_t)s.cols * s.stride + 4 * wg_dz_slot(N) + 64; }

int wgrad_splits(int C, int N, int lg, int nvox) {
    const WgradShape s = wgrad_shape(C, lg, nvox);
    const int fit = 227 * 1024 / (int)(wgrad_smem(C, N, s) + 1024), tm = 512 / wg_cols(C, N);
    const int most = 152 * (fit < tm ? (fit < 2 ? fit : 2) : (tm < 2 ? tm : 2));
    const int n = (s.iters + 3) / 4;          // at least four iterations a CTA: each writes a slice of its own
    return n < 1 ? 1 : n < most ? n : most;
}

constexpr int WGT = 160;     // four warps copy, one issues the MMAs (eight copying: 29 us more per backward pass)

template <int C, int N>
__global__ void __launch_bounds__(WGT) k_wgrad_tc(WgradArgs a, WgradShape s) {
    pdl_enter();
    constexpr int CG = C / 8, CB = wg_block(C), NM = wg_tiles(C), TC = wg_cols(C, N);
    constexpr int LT = WGT - 32;              // copying threads
    constexpr int NU = (3 * CG * 64 + LT - 1) / LT, NZ = (3 * 64 * (N / 8) + LT - 1) / LT;
    constexpr uint32_t ZS = wg_dz_slot(N), ZG = wg_dz_group(N);
    extern __shared__ uint8_t raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 127) & ~(uintptr_t)127);
    const uint32_t xbytes = (uint32_t)s.cols * s.stride, blk = (uint32_t)CB * s.stride;
    // [0], [1]: an iteration's MMAs are done; [2], [3]: its rows are in shared memory
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + xbytes + 4 * ZS);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 4);
    int *eflag = reinterpret_cast<int *>(tslot + 1);
    const int r = threadIdx.x, warp = r >> 5;
    const int i0 = (int)((long long)s.iters * blockIdx.x / gridDim.x);
    const int n = (int)((long long)s.iters * (blockIdx.x + 1) / gridDim.x) - i0;   // >= 1: the grid is no larger than iters
    const int ipm = (1 << s.lipc) - 1;

    if (warp == LT / 32) {
        tmem_alloc(smem_u32(tslot), TC);
        tmem_relinquish();
    }
    if (r == 0) {
        mbar_init(smem_u32(&bar[0]), 1);
        mbar_init(smem_u32(&bar[1]), 1);
        mbar_init(smem_u32(&bar[2]), LT);
        mbar_init(smem_u32(&bar[3]), LT);
        *eflag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int e = r; e < (s.ring + s.mirror) << s.lgx; e += WGT) {   // the ones: channel 0 of each unit
        const int b = e >> s.lgx, x = e & ((1 << s.lgx) - 1);
        uint8_t *p = base + (size_t)(b * CB + CB - 1) * s.stride + (size_t)x * 16;
        *reinterpret_cast<uint4 *>(p) = make_uint4(0x3F80u, 0, 0, 0);
    }
    fence_proxy_async_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tslot;
    const uint32_t xb = smem_u32(base), zb = xb + xbytes;

    if (warp == LT / 32) {                          // ---- one thread issues every MMA
        if (elect_one()) {
            const uint32_t idesc = idesc_bf16_f32(128, 3 * N) | (3u << 15);  // both operands MN-major
            // MN-major without a swizzle: first stride along K (8 voxels), second along M or N
            const uint64_t ad0 = sdesc_none(0, s.lgx == 3 ? blk : 128, s.stride), bd0 = sdesc_none(0, 128, ZG);
            int f = 0;                        // sequence number of the iteration's first row
            for (int it = 0; it < n; ++it) {
                if (it > 0) f += s.rpi + (((i0 + it) & ipm) ? 0 : 2);
                if (!mbar_wait_bounded(smem_u32(&bar[2 + (it & 1)]), (it >> 1) & 1, NN_WAIT)) *eflag = 1;
                fence_after_sync();
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const int row = (16 * ks) >> s.lgx, x = (16 * ks) & ((1 << s.lgx) - 1);
                    const uint32_t sx = xb + (uint32_t)((f + row) % s.ring) * blk + (uint32_t)x * 16;
                    const uint64_t bd = bd0 + ((zb + (uint32_t)(it & 3) * ZS + (uint32_t)ks * 256) >> 4);
#pragma unroll
                    for (int j = 0; j < NM; ++j)
                        mma_bf16(tmem + (uint32_t)(j * 3 * N), ad0 + ((sx + (uint32_t)j * 16 * s.stride) >> 4), bd, idesc,
                                 (it > 0 || ks > 0) ? 1u : 0u);
                }
                mma_commit(smem_u32(&bar[it & 1]));
            }
        }
    } else {                                  // ---- the other warps copy
        const int lg = a.lg, D = 1 << lg, up = a.up, lgi = lg - up;
        const int lnx = lg > 6 ? lg - 6 : 0;  // x segments per row (log2)
        const int TX = 1 << s.lgx, nub = 3 * CG * TX;
        int off[NU], zoff[NZ];                // places in a row, and whether they are in the grid
        uint32_t in = 0, zin = 0, dst[NU], zdst[NZ];
        int slot = 0;
        const uint16_t *xcol = a.x, *zcol = a.dz;
        int x0 = 0, rows = -1;                // rows: sequence number of the last row copied
#pragma unroll
        for (int j = 0; j < NU; ++j) {
            const int u = r + LT * j, cg = u % CG, v = u / CG;
            dst[j] = xb + (uint32_t)((v >> s.lgx) * CG + cg) * s.stride + (uint32_t)(v & (TX - 1)) * 16;
        }
#pragma unroll
        for (int j = 0; j < NZ; ++j) {        // 3 shifts x 64 voxels x N / 8 units
            const int u = r + LT * j, ng = u % (N / 8), v = u / (N / 8) % 64, dx = u / (N / 8) / 64;
            zdst[j] = zb + (uint32_t)(dx * (N / 8) + ng) * ZG + (uint32_t)v * 16;
        }
        auto load_iter = [&](int k) {         // one copy group: the rows and gradients that iteration k adds
            const int i = i0 + k, y0 = (i & ipm) * s.rpi;
            const bool first = k == 0 || (i & ipm) == 0;
            if (first) {
                const int col = i >> s.lipc, z = (col >> lnx) & (D - 1), b = col >> (lnx + lg);
                x0 = (col & ((1 << lnx) - 1)) << 6;
                xcol = a.x + ((size_t)b << (3 * lgi)) * C;
                in = zin = 0;
                zcol = a.dz + (((size_t)b << (3 * lg)) + ((size_t)z << (2 * lg))) * N;
#pragma unroll
                for (int j = 0; j < NU; ++j) {
                    const int u = r + LT * j, cg = u % CG, v = u / CG;
                    const int x = x0 + (v & (TX - 1)), zz = z + (v >> s.lgx) - 1;
                    const bool ok = u < nub && (unsigned)x < (unsigned)D && (unsigned)zz < (unsigned)D;
                    off[j] = ok ? (((zz >> up) << (2 * lgi)) + (x >> up)) * C + cg * 8 : 0;
                    in |= (ok ? 16u : 0u) << j;
                }
#pragma unroll
                for (int j = 0; j < NZ; ++j) {
                    const int u = r + LT * j, ng = u % (N / 8), v = u / (N / 8) % 64, dx = u / (N / 8) / 64;
                    const int y = v >> s.lgx, x = x0 + (v & (TX - 1)) - (dx - 1);   // y: below the iteration's first
                    const bool ok = y < D && (unsigned)x < (unsigned)D;
                    zoff[j] = ok ? ((y << lg) + x) * N + ng * 8 : 0;
                    zin |= (ok ? 16u : 0u) << j;
                }
            }
            for (int y = first ? y0 - 1 : y0 + 1; y <= y0 + s.rpi; ++y) {
                ++rows;
                const bool yin = (unsigned)y < (unsigned)D;
                const uint32_t ymask = yin ? in : 0u, at = (uint32_t)slot * blk;
                const uint16_t *xr = xcol + ((size_t)((yin ? y : 0) >> up) << lgi) * C;
#pragma unroll
                for (int j = 0; j < NU; ++j)
                    if (r + LT * j < nub) cp_async16(dst[j] + at, xr + off[j], ymask >> j & 16u);
                if (slot < s.mirror) {
#pragma unroll
                    for (int j = 0; j < NU; ++j)
                        if (r + LT * j < nub) cp_async16(dst[j] + at + (uint32_t)s.ring * blk, xr + off[j], ymask >> j & 16u);
                }
                slot = slot == s.ring - 1 ? 0 : slot + 1;
            }
            const uint16_t *zr = zcol + ((size_t)y0 << lg) * N;
#pragma unroll
            for (int j = 0; j < NZ; ++j)
                if (r + LT * j < 3 * 64 * (N / 8)) cp_async16(zdst[j] + (uint32_t)(k & 3) * ZS, zr + zoff[j], zin >> j & 16u);
            cp_async_commit();
        };
        int f = 0, fprev = 0, k = 0;          // k: iterations copied
        for (int it = 0; it < n; ++it) {
            if (it > 0) {
                fprev = f;
                f += s.rpi + (((i0 + it) & ipm) ? 0 : 2);
            }
            // the MMAs of iteration it - 2 are done: rows before fprev and its gradients are free
            if (it >= 2 && !mbar_wait_bounded(smem_u32(&bar[it & 1]), ((it - 2) >> 1) & 1, NN_WAIT)) *eflag = 1;
            while (k < n && k <= it + 2 &&
                   rows + s.rpi + ((k == 0 || ((i0 + k) & ipm) == 0) ? 2 : 0) <= fprev + s.ring - 1)
                load_iter(k++);
            cp_async_wait_upto(k - 1 - it);
            fence_proxy_async_smem();
            mbar_arrive(smem_u32(&bar[2 + (it & 1)]));
        }
        // commits complete in order: the last iteration's covers every MMA
        if (!mbar_wait_bounded(smem_u32(&bar[(n - 1) & 1]), ((n - 1) >> 1) & 1, NN_WAIT)) *eflag = 1;
        fence_after_sync();
        float *part = a.part + (size_t)blockIdx.x * ((NTAPS * C + 1) * N);
        if (warp < 4) for (int q = 0; q < 3 * NM; ++q) {
            const int j = q / 3, dx = q % 3;
            float v[N];
            const uint32_t acc = tmem + (uint32_t)(q * N) + ((uint32_t)(warp * 32) << 16);
            tmem_ld16(acc, v);
            if constexpr (N == 32) tmem_ld16(acc + 16, v + 16);
            const int cm = 16 * j + (r >> 3), dy = cm / CB, rem = cm % CB;
            const int row = dy > 2 ? -1
                            : rem < CB - 1 ? (9 * (rem / CG) + 3 * dy + dx) * C + 8 * (rem % CG) + (r & 7)
                            : (dy == 0 && dx == 1 && (r & 7) == 0) ? NTAPS * C : -1;
            if (row >= 0) {
                float4 *o = reinterpret_cast<float4 *>(part + (size_t)row * N);
#pragma unroll
                for (int e = 0; e < N / 4; ++e) o[e] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    if (r == 0 && *eflag) atomicOr(a.err, 1);
    if (warp == LT / 32) tmem_dealloc(tmem, TC);
}

// Nearest up-sampling of `coarse` and the finer grid's own term: out = coarse + fine, or (mask)
// mask > 0 ? fine + coarse / 8 : 0, the gradient through a pooling.  One thread per 16-byte unit:
// as an epilogue of the coarse convolution the same passes had 128 threads per 1024 fine voxels
// and took 9 (8^3), 17 (16^3) and 40 us (32^3) more than the convolution alone, here 4, 6 and 16.
__global__ void __launch_bounds__(256) k_expand(const uint16_t *__restrict__ coarse, const uint16_t *__restrict__ fine,
                                                const uint16_t *__restrict__ mask, uint16_t *__restrict__ out,
                                                unsigned units, int lg, int lgG) {
    pdl_enter();
    const unsigned e = blockIdx.x * 256 + threadIdx.x;
    if (e >= units) return;
    const unsigned m = e >> lgG, g = e & ((1u << lgG) - 1), D = 1u << lg;
    const unsigned x = m & (D - 1), y = (m >> lg) & (D - 1), bz = m >> (2 * lg);
    const unsigned mc = ((((bz >> 1) << (lg - 1)) + (y >> 1)) << (lg - 1)) + (x >> 1);
    float f[8], s[8];
    const uint4 qf = __ldg(reinterpret_cast<const uint4 *>(coarse) + (((size_t)mc << lgG) + g));
    const uint4 qs = __ldg(reinterpret_cast<const uint4 *>(fine) + e);
    unpack8(qf, f);
    unpack8(qs, s);
    if (mask) {
        float k[8];
        unpack8(__ldg(reinterpret_cast<const uint4 *>(mask) + e), k);
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = k[j] > 0.f ? s[j] + 0.125f * f[j] : 0.f;
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] += s[j];
    }
    reinterpret_cast<uint4 *>(out)[e] = pack8(f);
}

void expand(const uint16_t *coarse, const uint16_t *fine, const uint16_t *mask, uint16_t *out, int nvox, int lg, int C,
            cudaStream_t st) {
    const unsigned units = (unsigned)nvox * (C / 8);
    launch_pdl(k_expand, (units + 255) / 256, 256, 0, st, coarse, fine, mask, out, units, lg, C == 32 ? 2 : 1);
}

// gradients of every layer of the table from the CTAs' slices: [27 C + 1][N] summed over the
// splits, written as w [N][27][C] then b [N].  32 elements x 8 groups of splits per block, the
// groups added in order.
__global__ void __launch_bounds__(256) k_wgrad_sum(WgradSums t) {
    pdl_enter();
    __shared__ float sm[8][32];
    int l = 0;
    while (l + 1 < t.layers && (int)blockIdx.x >= t.l[l + 1].block0) ++l;
    const WgradSum &w = t.l[l];
    const int elems = w.elems(), e = ((int)blockIdx.x - w.block0) * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5;
    float acc = 0.f;
    if (e < elems)
        for (int y = g; y < w.splits; y += 8) acc += w.part[(size_t)y * elems + e];
    sm[g][threadIdx.x & 31] = acc;
    __syncthreads();
    if (g == 0 && e < elems) {
#pragma unroll
        for (int k = 1; k < 8; ++k) acc += sm[k][threadIdx.x];
        const int k = e / w.N, nn = e % w.N;
        if (w.C == 0) w.grad[e] = acc;
        else w.grad[k < NTAPS * w.C ? nn * NTAPS * w.C + k : NTAPS * w.C * w.N + nn] = acc;
    }
    if (w.C == 0 && g == 1 && (int)blockIdx.x == w.block0) {   // the loss, its partials in a fixed order too
        double d = 0.0;
        for (int y = threadIdx.x & 31; y < w.splits; y += 32) d += t.loss_part[y];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if ((threadIdx.x & 31) == 0) *t.loss = d;
    }
}

template <int C, int N, int EPI>
static void set_conv() {
    cudaFuncSetAttribute(k_conv_tc<C, N, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, conv_smem(C, N));
}

void init_attributes() {
    static bool done = false;
    if (done) return;
    set_conv<16, 16, CONV_PLAIN>();
    set_conv<16, 32, CONV_PLAIN>();
    set_conv<32, 16, CONV_PLAIN>();
    set_conv<32, 32, CONV_PLAIN>();
    set_conv<16, 16, CONV_POOL>();
    set_conv<16, 32, CONV_POOL>();
    set_conv<32, 32, CONV_POOL>();
    set_conv<16, 16, CONV_PAIR>();
    set_conv<32, 16, CONV_PAIR>();
    set_conv<16, 16, CONV_HEAD>();
    cudaFuncSetAttribute(k_wgrad_tc<16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaFuncSetAttribute(k_wgrad_tc<16, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaFuncSetAttribute(k_wgrad_tc<32, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaFuncSetAttribute(k_wgrad_tc<32, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    done = true;
}

template <int C, int N, int EPI>
static int launch_conv(const ConvArgs &a, cudaStream_t st) {
    // as many CTAs as fit beside each other on an SM (227 KB shared memory, 512 columns of TMEM)
    constexpr int fit = 227 * 1024 / (int)(conv_smem(C, N) + 1024);
    constexpr int tm = 512 / (ACCS * N);
    constexpr int per_sm = fit < tm ? fit : tm;
    const int ltx = a.lg > 3 ? a.lg - 3 : 0, lty = a.lg > 4 ? a.lg - 4 : 0;
    const int tiles = (a.nvox >> (2 * a.lg)) << (ltx + lty);
    if (tiles > 0)
        launch_pdl(k_conv_tc<C, N, EPI>, tiles < 152 * per_sm ? tiles : 152 * per_sm, 160, conv_smem(C, N), st, a);
    return 0;
}

int conv(const ConvArgs &a, int C, int N, cudaStream_t st) {
    const int cn = C * 100 + N;
    switch (a.epi) {
        case CONV_HEAD: return cn == 1616 ? launch_conv<16, 16, CONV_HEAD>(a, st) : -1;
        case CONV_POOL:
            return cn == 1616   ? launch_conv<16, 16, CONV_POOL>(a, st)
                   : cn == 1632 ? launch_conv<16, 32, CONV_POOL>(a, st)
                   : cn == 3232 ? launch_conv<32, 32, CONV_POOL>(a, st)
                                : -1;
        case CONV_PAIR:
            return cn == 1616 ? launch_conv<16, 16, CONV_PAIR>(a, st) : cn == 3216 ? launch_conv<32, 16, CONV_PAIR>(a, st) : -1;
        default:
            return cn == 1616   ? launch_conv<16, 16, CONV_PLAIN>(a, st)
                   : cn == 1632 ? launch_conv<16, 32, CONV_PLAIN>(a, st)
                   : cn == 3216 ? launch_conv<32, 16, CONV_PLAIN>(a, st)
                   : cn == 3232 ? launch_conv<32, 32, CONV_PLAIN>(a, st)
                                : -1;
    }
}

template <int C, int N>
static int launch_wgrad(const WgradArgs &a, cudaStream_t st) {
    const WgradShape s = wgrad_shape(C, a.lg, a.nvox);
    if (s.iters > 0)
        launch_pdl(k_wgrad_tc<C, N>, wgrad_splits(C, N, a.lg, a.nvox), WGT, wgrad_smem(C, N, s), st, a, s);
    return 0;
}

int wgrad(const WgradArgs &a, int C, int N, cudaStream_t st) {
    if (C == 16 && N == 16) return launch_wgrad<16, 16>(a, st);
    if (C == 16 && N == 32) return launch_wgrad<16, 32>(a, st);
    if (C == 32 && N == 16) return launch_wgrad<32, 16>(a, st);
    if (C == 32 && N == 32) return launch_wgrad<32, 32>(a, st);
    return -1;
}

void wgrad_sums(WgradSums &t, cudaStream_t st) {
    int blocks = 0;
    for (int l = 0; l < t.layers; ++l) {
        t.l[l].block0 = blocks;
        blocks += (t.l[l].elems() + 31) / 32;
    }
    launch_pdl(k_wgrad_sum, blocks, 256, 0, st, t);
}

}  // namespace nn
}  // namespace sph
