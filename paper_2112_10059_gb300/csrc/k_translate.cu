// Far-field translations as batched, gathered GEMMs (FP32 SIMT, register tiled).
//
// M2L (paper Section 2.4, far interactions through the hierarchy): for a tile of 64 V pairs (target
// box B, source box A) of one level and offset o,
//     d_B += M2L_o u_A,
// so that an operator is read once per tile instead of once per box pair.
//
// L2L: for a tile of 64 parent boxes P of level l-1 and one child slot c,
//     d_{child c of P} += L2L_c d_P.
//
// Tiling: CTA = 256 threads computes 128 operator rows x 64 boxes; thread
// (ty, tx) holds 8 rows x 4 boxes of FP32 accumulators; the K dimension (the
// operator columns) streams through shared memory 16 at a time.  Operators
// are stored transposed ([k][i], row stride npad), so an operator K-slab is a
// contiguous, coalesced read.
#include "sph_kernels.cuh"
#include "tc_sm103.cuh"

namespace sph {

constexpr int TM = 128, TN = 64, TK = 16;

// thread (ty, tx) owns operator rows ty*8 .. ty*8+7 and tile columns tx*4 .. tx*4+3
__device__ __forceinline__ void mma_tile(const float (*As)[TM], const float (*Bs)[TN], int ty, int tx,
                                         float acc[8][4]) {
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4 *>(&As[kk][ty * 8]);
        const float4 a1 = *reinterpret_cast<const float4 *>(&As[kk][ty * 8 + 4]);
        const float4 bv = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float b[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) acc[r][cc] = fmaf(a[r], b[cc], acc[r][cc]);
    }
}

// shared memory of a tile: two K slabs of each operand, then the staged results
constexpr int TS = TM + 4;                                  // row stride of a staged column
constexpr int TILE_FLOATS = TN * TS > 2 * TK * (TM + TN) ? TN * TS : 2 * TK * (TM + TN);

// acc += Op[i0.., :] * X[:, cols]: Op transposed [k][i] with row stride ldA and M valid rows (VEC:
// multiples of 4, 16-byte aligned), K = np; X columns = state rows src[col] (row stride np).  The
// next slab is loaded into registers under this slab's FMAs and stored into the other buffer:
// these launches have few CTAs, so a slab whose loads were waited for took three times its FMAs
// (L2L of the four levels of a 90 x 61 x 117 grid 125 us with the loads waited for and 32 scalar
// reductions a thread, 71 us so; M2L of its 32,013 pairs 116, 89).
template <bool VEC>
__device__ __forceinline__ void gemm_slab_g(const float *__restrict__ opT, int ldA, int M, int np, int i0,
                                            const float *__restrict__ state, const int *src, float *smem, float acc[8][4]) {
    float (*As)[TK][TM] = reinterpret_cast<float (*)[TK][TM]>(smem);
    float (*Bs)[TK][TN] = reinterpret_cast<float (*)[TK][TN]>(smem + 2 * TK * TM);
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int bc = tid % TN, bq = tid / TN, s = src[bc];    // this thread's column and quarter of a slab
    float a[8];
    float4 b;
    auto load = [&](int k0) {
        if (VEC) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int e = tid + 256 * j, i = i0 + e % 32 * 4;
                const float4 v = i < M ? __ldg(reinterpret_cast<const float4 *>(opT + (size_t)(k0 + e / 32) * ldA + i))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                a[4 * j] = v.x; a[4 * j + 1] = v.y; a[4 * j + 2] = v.z; a[4 * j + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int e = tid + 256 * j, i = i0 + e % TM;
                a[j] = i < M ? __ldg(opT + (size_t)(k0 + e / TM) * ldA + i) : 0.f;
            }
        }
        b = s >= 0 ? *reinterpret_cast<const float4 *>(state + (size_t)s * np + k0 + 4 * bq) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto store = [&](int buf) {
        if (VEC) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int e = tid + 256 * j;
                *reinterpret_cast<float4 *>(&As[buf][e / 32][e % 32 * 4]) = make_float4(a[4 * j], a[4 * j + 1], a[4 * j + 2], a[4 * j + 3]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) As[buf][(tid + 256 * j) / TM][(tid + 256 * j) % TM] = a[j];
        }
        Bs[buf][4 * bq][bc] = b.x;
        Bs[buf][4 * bq + 1][bc] = b.y;
        Bs[buf][4 * bq + 2][bc] = b.z;
        Bs[buf][4 * bq + 3][bc] = b.w;
    };
    load(0);
    store(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < np; k0 += TK, buf ^= 1) {
        if (k0 + TK < np) load(k0 + TK);
        mma_tile(As[buf], Bs[buf], ty, tx, acc);
        if (k0 + TK < np) store(buf ^ 1);
        __syncthreads();
    }
}

__device__ __forceinline__ void gemm_slab(const float *__restrict__ opT, int np, int i0,
                                          const float *__restrict__ state, const int *src, float *smem, float acc[8][4]) {
    gemm_slab_g<true>(opT, np, np, np, i0, state, src, smem, acc);
}

// out[dst[c]][i0 ..] += the tile's column c, a row of up to 128 values each by one bulk reduction
// (32 scalar reductions a thread, each warp's to 32 different rows, took as long as the FMAs).
// Ends with the staged columns read.
__device__ __forceinline__ void scatter_add(float *__restrict__ out, int np, int n, int i0, const int *dst,
                                            float *smem, const float acc[8][4]) {
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
#pragma unroll
    for (int cc = 0; cc < 4; ++cc)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = i0 + ty * 8 + 4 * h + r < n ? acc[4 * h + r][cc] : 0.f;
            *reinterpret_cast<float4 *>(smem + (tx * 4 + cc) * TS + ty * 8 + 4 * h) = make_float4(v[0], v[1], v[2], v[3]);
        }
    tc::fence_proxy_async_smem();
    __syncthreads();
    if (tid < TN && dst[tid] >= 0) {
        tc::bulk_reduce_add_f32(out + (size_t)dst[tid] * np + i0, tc::smem_u32(smem + tid * TS), (uint32_t)min(TM, np - i0) * 4u);
        tc::bulk_commit();
        tc::bulk_wait_read_all();
    }
    __syncthreads();
}

// ---------------------------------------------------------------- L2L
__global__ void __launch_bounds__(256) k_l2l_gemm(FmmDev F, int level, int parent_begin, int parent_count) {
    pdl_enter();
    __shared__ __align__(16) float tile_s[TILE_FLOATS];
    __shared__ int par[TN], dst[TN];
    const int tid = threadIdx.x;
    const int np = F.O.npad, n = F.O.n;
    const int t0 = blockIdx.x * TN;
    const int i0 = blockIdx.y * TM;
    const int c = blockIdx.z;
    const TreeDev &T = F.T;
    int any = 0;
    if (tid < TN) {
        int p = parent_begin + t0 + tid;
        int P = -1, C = -1;
        if (t0 + tid < parent_count && !T.b_leaf[p] && T.b_te[p] > T.b_tb[p]) {
            int ch = T.box_at[dense_off(level) + ((T.b_key[p] << 3) | (uint32_t)c)];
            if (ch >= 0 && T.b_te[ch] > T.b_tb[ch]) { P = p; C = ch; }
        }
        par[tid] = P;
        dst[tid] = C;
        any = C >= 0;
    }
    if (!__syncthreads_or(any)) return;
    float acc[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) acc[r][cc] = 0.f;
    gemm_slab(F.O.l2l_t + ((size_t)level * 8 + c) * np * np, np, i0, F.dchk, par, tile_s, acc);
    scatter_add(F.dchk, np, n, i0, dst, tile_s, acc);
}

// ---------------------------------------------------------------- V pairs grouped by offset
// key = level * 316 + slot.  The list kernels count the pairs per key, k_lists_layout (k_tree.cu)
// scans the counts and cuts every key's range into tiles of VPAIR_TILE pairs, and the list fill
// places every pair in its key's range (any order within a key) and writes the key of every tile.


// One CTA per tile of up to 64 V pairs sharing (level, offset): d_B += M2L_{l,o} u_A, scatter-added.
__global__ void __launch_bounds__(256) k_m2l_pairs(FmmDev F, PairsDev Pd) {
    pdl_enter();
    __shared__ __align__(16) float tile_s[TILE_FLOATS];
    __shared__ int trg[TN], src[TN];
    __shared__ int s_key;
    const int tid = threadIdx.x;
    const int np = F.O.npad, n = F.O.n;
    const int tile = blockIdx.x;
    if (tile >= Pd.tile_off[Pd.nkeys]) return;
    if (tid == 0) s_key = Pd.tile_key[tile];
    __syncthreads();
    const int key = s_key;
    const int level = key / NSLOT, slot = key % NSLOT;
    const int p0 = Pd.off[key] + (tile - Pd.tile_off[key]) * TN;
    const int p1 = min(p0 + TN, Pd.off[key + 1]);
    if (tid < TN) {
        int q = p0 + tid;
        const int2 pr = q < p1 ? Pd.pair[q] : make_int2(-1, -1);
        trg[tid] = pr.x;
        src[tid] = pr.y;
    }
    __syncthreads();
    const float *M = F.O.m2l_t + ((size_t)level * NSLOT + slot) * np * np;
    for (int i0 = 0; i0 < np; i0 += TM) {
        float acc[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) acc[r][cc] = 0.f;
        gemm_slab(M, np, i0, F.ueq, src, tile_s, acc);
        scatter_add(F.dchk, np, n, i0, trg, tile_s, acc);
    }
}

void fmm_m2l_pairs(const FmmDev &F, const PairsDev &Pd, int nV, int m2l_prec, cudaStream_t st) {
    (void)m2l_prec;
    if (nV <= 0) return;
    // upper bound on the tile count: every key adds at most one partial tile
    int grid = (nV + TN - 1) / TN + Pd.nkeys;
    launch_pdl(k_m2l_pairs, grid, 256, 0, st, F, Pd);
}

// ---------------------------------------------------------------- L2P for whole leaf boxes
// Chebyshev far field: S(cell m of leaf B) = sum_k E_l[m][k] d_B[k], E_l the interpolation
// table of the box's e^3 cells (rows in local Morton order, stored transposed [k][m]).
// A CTA handles 64 leaves of one level; its 128 x 64 result tile goes through shared
// memory to the leaves' targets, whose local Morton index is the low 3 log2(e) bits of
// their key.  Writes (=) every target of every leaf of this level.
__global__ void __launch_bounds__(256) k_l2p_gemm(FmmDev F, int level, int box_begin, int box_count,
                                                  float *__restrict__ out) {
    pdl_enter();
    __shared__ __align__(16) float tile[TM * (TN + 1)];     // the operands' slabs, then the results
    float (*Cs)[TN + 1] = reinterpret_cast<float (*)[TN + 1]>(tile);
    static_assert(TM * (TN + 1) >= 2 * TK * (TM + TN), "tile");
    __shared__ int col[TN];
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int np = F.O.npad;
    const TreeDev &T = F.T;
    const int t0 = blockIdx.x * TN;
    const int i0 = blockIdx.y * TM;
    const int e = 1 << (F.D - level);
    const int rows = e * e * e;
    int any = 0;
    if (tid < TN) {
        int b = box_begin + t0 + tid;
        int ok = t0 + tid < box_count && T.b_leaf[b] && T.b_te[b] > T.b_tb[b];
        col[tid] = ok ? b : -1;
        any = ok;
    }
    if (!__syncthreads_or(any)) return;
    float acc[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) acc[r][cc] = 0.f;
    gemm_slab_g<false>(F.O.e_tab + F.O.e_off[level], rows, rows, np, i0, F.dchk, col, tile, acc);
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) Cs[ty * 8 + r][tx * 4 + cc] = acc[r][cc];
    __syncthreads();
    const uint32_t lmask = (uint32_t)rows - 1u;
    // warp w handles columns w, w + 8, ...; lanes stride over the column's targets
    const int warp = tid >> 5, lane = tid & 31;
    for (int c = warp; c < TN; c += 8) {
        int b = col[c];
        if (b < 0) continue;
        for (int t = T.b_tb[b] + lane; t < T.b_te[b]; t += 32) {
            int m = (int)(F.trg_key[t] & lmask) - i0;
            if (m < 0 || m >= TM) continue;
            uint32_t pc = key_pc(F.trg_key[t]);
            out[(int64_t)pc_i(pc) + (int64_t)F.nx * ((int64_t)pc_j(pc) + (int64_t)F.ny * pc_k(pc))] = Cs[m][c];
        }
    }
}

void fmm_l2p_gemm_level(const FmmDev &F, int level, int box_begin, int box_count, float *out, cudaStream_t st) {
    if (box_count <= 0 || level < 2 || F.O.e_off[level] < 0) return;
    int e = 1 << (F.D - level);
    dim3 grid((box_count + TN - 1) / TN, (e * e * e + TM - 1) / TM);
    launch_pdl(k_l2p_gemm, grid, 256, 0, st, F, level, box_begin, box_count, out);
}

void fmm_l2l_gemm_level(const FmmDev &F, int level, int parent_begin, int parent_count, cudaStream_t st) {
    if (parent_count <= 0 || level < 3) return;
    dim3 grid((parent_count + TN - 1) / TN, (F.O.npad + TM - 1) / TM, 8);
    launch_pdl(k_l2l_gemm, grid, 256, 0, st, F, level, parent_begin, parent_count);
}

}  // namespace sph
