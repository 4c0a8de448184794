// 3x3x3 convolutions of the learned surrogate on tcgen05 (see nn_kernels.cuh for the tensors).
//
// k_conv_tc<C, N>: forward, or data gradient with a flipped, transposed weight image.  The
// implicit GEMM's A operand is never formed: a CTA keeps whole z-planes of its column's input
// (8 x 16 output voxels plus the halo, 10 x 18) in shared memory, one 16-byte unit of 8
// channels per voxel and channel group, x fastest.  Eight x-neighbours are then one
// unswizzled K-major core matrix (8 rows x 16 bytes), the 16 rows of the tile are its M
// repeats (stride one halo row), the channel groups its K repeats -- and the operand of any
// of the 27 taps is the same plane read from a start address moved by whole units.
// A voxel's input is copied 1.4 times (halo) instead of 27 times; the copies per 128-voxel
// tile fall from 3584 (C = 16) to 360.
// CTAs march in z through equal shares of the tiles, planes in a ring of six loaded two
// ahead, the tile's MMAs (27 C / 16 of M = 128, N, K = 16, accumulated in tap order) running
// into one of two TMEM accumulators under the previous tile's epilogue.
// What bounds it: the tensor core reads 4 KB of A per MMA (about 32 clocks at 128 B/clock) for
// an N of only 16 or 32.
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
constexpr int RING = 6;                         // planes in shared memory
constexpr int AHEAD = 2;                        // planes loaded ahead of the tile's own three
// bytes between the channel groups of a plane: such that the 8 units a quarter-warp copies
// (2 groups x 4 voxels, or 4 groups x 2) fall into different banks
__host__ __device__ constexpr uint32_t group_bytes(int C) { return PX * PY * 16 + (C == 16 ? 0 : 32); }
__host__ __device__ constexpr uint32_t plane_bytes(int C) { return (uint32_t)(C / 8) * group_bytes(C); }
__host__ __device__ constexpr uint32_t weight_bytes(int C, int N) { return (uint32_t)conv_chunks(C) * N * 128; }
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
    else cp_async_wait<2>();
}

template <int C, int N>
__global__ void __launch_bounds__(128) k_conv_tc(ConvArgs a) {
    pdl_enter();
    constexpr int CG = C / 8;
    constexpr uint32_t GB = group_bytes(C), PB = plane_bytes(C), WB = weight_bytes(C, N);
    constexpr int NU = (PX * PY * CG + 127) / 128;   // units copied per thread and plane
    extern __shared__ uint8_t raw[];
    uint8_t *base = align1024(raw);
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + WB + RING * PB);   // [0], [1]: accumulators; [2]: weights
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 3);
    int *eflag = reinterpret_cast<int *>(tslot + 1);
    __shared__ float sbias[N];

    const int r = threadIdx.x;
    const int lg = a.lg, D = 1 << lg, dm = D - 1;
    const int ltx = lg > 3 ? lg - 3 : 0, lty = lg > 4 ? lg - 4 : 0;   // tiles per row and plane (log2)
    const int ntiles = (a.nvox >> (2 * lg)) << (ltx + lty);           // (batch x D) planes of tiles
    const int t0 = (int)((long long)ntiles * blockIdx.x / gridDim.x);
    const int t1 = (int)((long long)ntiles * (blockIdx.x + 1) / gridDim.x);
    if (t0 >= t1) return;                     // uniform over the CTA, before any allocation

    if (r < N) sbias[r] = a.bias ? a.bias[r] : 0.f;
    if (r < 32) {
        tmem_alloc(smem_u32(tslot), 2 * N);
        tmem_relinquish();
    }
    if (r == 0) {
        for (int s = 0; s < 3; ++s) mbar_init(smem_u32(&bar[s]), 1);
        *eflag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tslot;
    const uint32_t wbase = smem_u32(base), ring = wbase + WB;
    const uint32_t idesc = idesc_bf16_f32(128, N);
    if (r == 0) {
        mbar_expect_tx(smem_u32(&bar[2]), WB);
        bulk_g2s(wbase, a.w, WB, smem_u32(&bar[2]));
    }

    // ---- load cursor: the planes zs - 1 .. zs + len of each column's run of tiles, in order
    const int up = a.up, lgi = lg - up, Di = 1 << lgi;   // input grid (half the edge when up-sampled on load)
    int off[NU];
    const uint16_t *xcol = a.x;
    int ltile = t0, lz = 0, lze = -2, loaded = -1;
    auto load_next = [&]() {                  // the next plane, one copy group; false when none is left
        if (lz > lze) {                       // next column
            if (ltile >= t1) return false;
            const int col = ltile >> lg, zs = ltile & dm, len = min(D - zs, t1 - ltile);
            const int x0 = (col & ((1 << ltx) - 1)) * CX - 1, y0 = ((col >> ltx) & ((1 << lty) - 1)) * CY - 1;
            xcol = a.x + ((size_t)(col >> (ltx + lty)) << (3 * lgi)) * C;
#pragma unroll
            for (int j = 0; j < NU; ++j) {
                const int u = r + 128 * j, v = u / CG, cg = u % CG;
                const int x = x0 + v % PX, y = y0 + v / PX;
                off[j] = ((unsigned)x < (unsigned)D && (unsigned)y < (unsigned)D)
                             ? (((y >> up) << lgi) + (x >> up)) * C + cg * 8
                             : -1;
            }
            lz = zs - 1;
            lze = zs + len;
            ltile += len;
        }
        ++loaded;
        const uint32_t dst = ring + (uint32_t)(loaded % RING) * PB;
        const bool zin = (unsigned)lz < (unsigned)D;
        const uint16_t *xp = xcol + ((size_t)((zin ? lz : 0) >> up) << (2 * lgi)) * C;
#pragma unroll
        for (int j = 0; j < NU; ++j) {
            const int u = r + 128 * j;
            if (u < PX * PY * CG) {
                const bool in = zin && off[j] >= 0;
                cp_async16(dst + (uint32_t)(u % CG) * GB + (uint32_t)(u / CG) * 16, in ? xp + off[j] : a.x, in ? 16 : 0);
            }
        }
        cp_async_commit();
        ++lz;
        return lz <= lze || ltile < t1;
    };

    const int warp = r >> 5;
    auto epilogue = [&](int t, int it) {
        const int col = t >> lg, z = t & dm;
        const int x = (col & ((1 << ltx) - 1)) * CX + (r & 7), y = ((col >> ltx) & ((1 << lty) - 1)) * CY + (r >> 3);
        const size_t m = ((((size_t)(col >> (ltx + lty)) << lg) + z) << (2 * lg)) + ((size_t)y << lg) + x;
        if (!mbar_wait_bounded(smem_u32(&bar[it & 1]), (it >> 1) & 1, NN_WAIT)) *eflag = 1;
        fence_after_sync();
        float v[N];
        const uint32_t acc = tmem + (uint32_t)((it & 1) * N) + ((uint32_t)(warp * 32) << 16);
        tmem_ld16(acc, v);
        if constexpr (N == 32) tmem_ld16(acc + 16, v + 16);
        fence_before_sync();                  // ordered before the MMAs that overwrite it by the next barrier
        if (x < D && y < D) {
            const size_t o = m * N;
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
                if (a.add) {
                    float ad[8];
                    unpack8(*reinterpret_cast<const uint4 *>(a.add + o + 8 * g), ad);
#pragma unroll
                    for (int j = 0; j < 8; ++j) f[j] += ad[j];
                }
                if (a.mask) {
                    float mk[8];
                    unpack8(*reinterpret_cast<const uint4 *>(a.mask + o + 8 * g), mk);
#pragma unroll
                    for (int j = 0; j < 8; ++j) f[j] = mk[j] > 0.f ? f[j] : 0.f;
                }
                const uint4 q = pack8(f);
                *reinterpret_cast<uint4 *>(a.out + o + 8 * g) = q;
            }
        }
    };

    int f = 0, fprev = 0;                     // sequence number of the tile's first plane
    bool more = true;
    for (int it = 0; it < t1 - t0; ++it) {
        const int t = t0 + it;
        if (it > 0) {
            fprev = f;
            f += (t & dm) ? 1 : 3;
        }
        // a slot is free once the last tile that read it is done: the previous tile, whose MMAs
        // may still run, reads the planes from fprev on
        const int lim = min(f + 2 + AHEAD, fprev + RING - 1);
        while (more && loaded < lim) more = load_next();
        cp_async_wait_upto(loaded - (f + 2));
        fence_proxy_async_smem();
        __syncthreads();
        if (r == 0) {
            if (it == 0 && !mbar_wait_bounded(smem_u32(&bar[2]), 0, NN_WAIT)) *eflag = 1;
            fence_after_sync();
            const uint64_t ad0 = sdesc_none(0, GB, PX * 16), bd0 = sdesc_sw128(0);
            const uint32_t acc = tmem + (uint32_t)((it & 1) * N);
#pragma unroll
            for (int dz = 0; dz < 3; ++dz) {
                const uint32_t sp = ring + (uint32_t)((f + dz) % RING) * PB;
#pragma unroll
                for (int tap = 9 * dz; tap < 9 * dz + 9; ++tap) {
                    const uint32_t sv = sp + (uint32_t)((tap / 3 % 3) * PX + tap % 3) * 16;
#pragma unroll
                    for (int h = 0; h < C / 16; ++h) {
                        const int k = tap * (C / 16) + h;   // K = 16 slice of the weight image
                        mma_bf16(acc, ad0 + ((sv + 2 * h * GB) >> 4),
                                 bd0 + ((wbase + (uint32_t)(k / 4) * N * 128 + (uint32_t)(k % 4) * 32) >> 4), idesc,
                                 k > 0 ? 1u : 0u);
                    }
                }
            }
            mma_commit(smem_u32(&bar[it & 1]));
        }
        if (it > 0) epilogue(t - 1, it - 1);
    }
    epilogue(t1 - 1, t1 - 1 - t0);
    fence_before_sync();
    __syncthreads();
    if (r == 0 && *eflag) atomicOr(a.err, 1);
    if (r < 32) tmem_dealloc(tmem, 2 * N);
}

template <int C, int N>
static void set_conv() {
    cudaFuncSetAttribute(k_conv_tc<C, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, conv_smem(C, N));
}

void init_conv() {
    set_conv<16, 16>();
    set_conv<16, 32>();
    set_conv<32, 16>();
    set_conv<32, 32>();
}

template <int C, int N>
static void launch_conv(const ConvArgs &a, cudaStream_t st) {
    // as many CTAs as fit beside each other on an SM (227 KB shared memory, 4 of 128 threads at most)
    constexpr int per_sm = 227 * 1024 / (int)(conv_smem(C, N) + 1024) < 4 ? 227 * 1024 / (int)(conv_smem(C, N) + 1024) : 4;
    const int ltx = a.lg > 3 ? a.lg - 3 : 0, lty = a.lg > 4 ? a.lg - 4 : 0;
    const int tiles = (a.nvox >> (2 * a.lg)) << (ltx + lty);
    if (tiles > 0) launch_pdl(k_conv_tc<C, N>, tiles < 152 * per_sm ? tiles : 152 * per_sm, 128, conv_smem(C, N), st, a);
}

int conv(const ConvArgs &a, int C, int N, cudaStream_t st) {
    if (C == 16 && N == 16) launch_conv<16, 16>(a, st);
    else if (C == 16 && N == 32) launch_conv<16, 32>(a, st);
    else if (C == 32 && N == 16) launch_conv<32, 16>(a, st);
    else if (C == 32 && N == 32) launch_conv<32, 32>(a, st);
    else return -1;
    return 0;
}

}  // namespace nn
}  // namespace sph
