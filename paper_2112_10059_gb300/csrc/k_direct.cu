// Direct quadrature of Eq. summation over the selected sets (paper Section 2.4,
// Section 4 "Classical Int"): every (target, source) pair through the same
// kernel G.  The FP32 variant is the plain direct sum the FMM is compared with;
// the FP64 variant serves the small all-pairs case.
//
// Layout: sources and targets in Morton order as packed (i,j,k) + weights.  Distances come from
// integer cell offsets, R = h sqrt(d2), d2 = di^2 + dj^2 + dk^2 exact (below 2^24 in FP32).
#include <algorithm>

#include "sph_kernels.cuh"

namespace sph {

// ---------------------------------------------------------------- FP32
// Each thread sums two targets, each over every source in order, in packed FP32 pairs (one
// instruction for both targets, so the FMA work of a pair is half an issue slot an operation).
// Bound by the special-function unit: 3 results a pair (rsqrt at 16 per SM and clock, two ex2 at
// 32).  The sources of a tile come in chunks of 32 Morton neighbours with their bounding box; the
// distance between that box and the warp's 64 targets chooses, for the whole chunk, between
//   - far: e^{-(beta - alpha) R} < 2^-25, so that 1 - it is 1 in FP32 and its ex2 is left out;
//   - near: both exponentials;
//   - general: the boxes meet (a source may be the target's own cell) or R is small enough for
//     the series form of 1 - e^{-x} (general_term, pair by pair).
// A chunk is summed by itself before it joins a target's sum: in one chain the error grows with the
// sources (1,309 of them: 5e-6 of S, 2e-7 so).
// 160^3 cells, 7,072 sources (2.9e10 pairs): 28.2 ms pair by pair with integer offsets (their
// conversion is a fourth result of the same unit), 10.5 ms so.
constexpr int DS = 256;    // sources per shared-memory tile
constexpr int DC = 32;     // sources per chunk

struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 f2_get(F2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// FP32 constants in units of cells
struct DirectK {
    float a2, b2;       // alpha h log2(e), (beta - alpha) h log2(e)
    float wscale;       // source_scale C (the 1 / h^3 of G and the cell volume cancel)
    float self;         // ball integral / C, or 0
    float far2, near2;  // squared distances (cells) from which a chunk is far / near
    float bma_h;        // (beta - alpha) h
};

// A term w G h^3 / C of squared distance d2 (cells; 0: the self term) as the product of a and b, for any
// R: both forms of 1 - e^{-x} and selections, so that the pairs of a chunk overlap (one_minus_exp_neg
// branches).  Here and in the loops below the weight multiplies the exponential first:
// e^{-alpha R} / R^3 by itself has lost bits to FP32's smallest exponents at alpha R = 66 and a thousand
// cells, where w G has not.
__device__ __forceinline__ void general_term(float d2, float w, const DirectK &k, float &a, float &b) {
    const float ir = rsqrt_approx(fmaxf(d2, 1.f)), R = fmaxf(d2, 1.f) * ir, x = k.bma_h * R;
    const float em = x < 0.5f ? one_minus_exp_series(x) : 1.f - ex2_approx(-k.b2 * R);
    a = d2 > 0.f ? ex2_approx(-k.a2 * R) * w * em : k.self;
    b = d2 > 0.f ? ir * ir * ir : w;
}

constexpr int WARPS = 4;

__global__ void __launch_bounds__(32 * WARPS) k_direct_f32(const uint32_t *__restrict__ src_pc,
                                                    const float *__restrict__ src_q, int ns,
                                                    const uint32_t *__restrict__ trg_key, int nt, DirectK k, int nx,
                                                    int ny, float *__restrict__ out_dense) {
    __shared__ float4 sxy[DS], szs[DS];   // {x, x, y, y}, {z, z, x^2 + y^2 + z^2 twice}
    __shared__ float2 sw[DS];
    __shared__ int box[DS / DC][6];
    constexpr int Q = DS / DC / WARPS;     // chunks a warp stages
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t0 = (blockIdx.x * WARPS + warp) * 64 + lane;
    // targets past the end repeat the last one (their sums are not written)
    const uint32_t pa = key_pc(trg_key[min(t0, nt - 1)]), pb = key_pc(trg_key[min(t0 + 32, nt - 1)]);
    const int ax = pc_i(pa), ay = pc_j(pa), az = pc_k(pa), bx = pc_i(pb), by = pc_j(pb), bz = pc_k(pb);
    const int lx = __reduce_min_sync(~0u, min(ax, bx)), hx = __reduce_max_sync(~0u, max(ax, bx));
    const int ly = __reduce_min_sync(~0u, min(ay, by)), hy = __reduce_max_sync(~0u, max(ay, by));
    const int lz = __reduce_min_sync(~0u, min(az, bz)), hz = __reduce_max_sync(~0u, max(az, bz));
    const F2 tx = f2(-2.f * ax, -2.f * bx), ty = f2(-2.f * ay, -2.f * by), tz = f2(-2.f * az, -2.f * bz);
    const F2 tt = f2((float)(ax * ax + ay * ay + az * az), (float)(bx * bx + by * by + bz * bz));
    const F2 a2 = f2(-k.a2, -k.a2), b2 = f2(-k.b2, -k.b2);
    F2 acc = f2(0.f, 0.f);
    uint32_t np[Q];                        // the next tile's sources, loaded under this one's pairs
    float nq[Q];
    auto fetch = [&](int s0) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int s = min(s0 + (warp + i * WARPS) * DC + lane, ns - 1);
            np[i] = src_pc[s];
            nq[i] = src_q[s];
        }
    };
    if (ns > 0) fetch(0);
    for (int s0 = 0; s0 < ns; s0 += DS) {
        const int m = min(DS, ns - s0);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < Q; ++i) {          // a warp stages a chunk and its box (past the end: the last source)
            const int u = (warp + i * WARPS) * DC + lane;
            const int x = pc_i(np[i]), y = pc_j(np[i]), z = pc_k(np[i]);
            const float fx = (float)x, fy = (float)y, fz = (float)z, ss = (float)(x * x + y * y + z * z);
            const float w = nq[i] * k.wscale;
            sxy[u] = make_float4(fx, fx, fy, fy);
            szs[u] = make_float4(fz, fz, ss, ss);
            sw[u] = make_float2(w, w);
            const int b0 = __reduce_min_sync(~0u, x), b1 = __reduce_max_sync(~0u, x), b2_ = __reduce_min_sync(~0u, y);
            const int b3 = __reduce_max_sync(~0u, y), b4 = __reduce_min_sync(~0u, z), b5 = __reduce_max_sync(~0u, z);
            if (lane < 6) box[u / DC][lane] = lane == 0 ? b0 : lane == 1 ? b1 : lane == 2 ? b2_ : lane == 3 ? b3 : lane == 4 ? b4 : b5;
        }
        if (s0 + DS < ns) fetch(s0 + DS);
        __syncthreads();
        for (int c = 0; c < m; c += DC) {
            const int *b = box[c / DC];
            const int gx = max(max(b[0] - hx, lx - b[1]), 0), gy = max(max(b[2] - hy, ly - b[3]), 0),
                      gz = max(max(b[4] - hz, lz - b[5]), 0);
            const float g2 = (float)(gx * gx + gy * gy + gz * gz);
            const int end = min(c + DC, m);
            auto dist2 = [&](int u) {
                const float4 xy = sxy[u], zs = szs[u];
                F2 d = f2_add(tt, f2(zs.z, zs.w));
                d = f2_fma(tx, f2(xy.x, xy.y), d);
                d = f2_fma(ty, f2(xy.z, xy.w), d);
                return f2_fma(tz, f2(zs.x, zs.y), d);
            };
            F2 part = f2(0.f, 0.f);            // a chunk by itself, then into the sum
            if (g2 >= k.far2) {                // uniform over the warp, as every choice here
#pragma unroll 4
                for (int u = c; u < end; ++u) {
                    const F2 d = dist2(u);
                    const float2 dd = f2_get(d);
                    const F2 ir = f2(rsqrt_approx(dd.x), rsqrt_approx(dd.y));
                    const float2 e = f2_get(f2_mul(a2, f2_mul(d, ir)));
                    const F2 ew = f2_mul(f2(ex2_approx(e.x), ex2_approx(e.y)), f2(sw[u].x, sw[u].y));
                    part = f2_fma(ew, f2_mul(f2_mul(ir, ir), ir), part);
                }
            } else if (g2 >= k.near2) {
#pragma unroll 4
                for (int u = c; u < end; ++u) {
                    const F2 d = dist2(u);
                    const float2 dd = f2_get(d);
                    const F2 ir = f2(rsqrt_approx(dd.x), rsqrt_approx(dd.y));
                    const F2 R = f2_mul(d, ir);
                    const float2 e = f2_get(f2_mul(a2, R)), q = f2_get(f2_mul(b2, R));
                    const F2 m1 = f2(1.f - ex2_approx(q.x), 1.f - ex2_approx(q.y));
                    const F2 ew = f2_mul(f2(ex2_approx(e.x), ex2_approx(e.y)), f2(sw[u].x, sw[u].y));
                    part = f2_fma(f2_mul(ew, m1), f2_mul(f2_mul(ir, ir), ir), part);
                }
            } else {
#pragma unroll 4
                for (int u = c; u < end; ++u) {
                    const float2 dd = f2_get(dist2(u));
                    float a0, a1, b0, b1;
                    general_term(dd.x, sw[u].x, k, a0, b0);
                    general_term(dd.y, sw[u].y, k, a1, b1);
                    part = f2_fma(f2(a0, a1), f2(b0, b1), part);
                }
            }
            acc = f2_add(acc, part);
        }
    }
    const float2 r = f2_get(acc);
    if (t0 < nt) out_dense[(int64_t)ax + (int64_t)nx * ((int64_t)ay + (int64_t)ny * az)] = r.x;
    if (t0 + 32 < nt) out_dense[(int64_t)bx + (int64_t)nx * ((int64_t)by + (int64_t)ny * bz)] = r.y;
}

// The same sums with one target a thread and the general form throughout: where the targets are
// too few to fill the chip the longest warp counts, and a warp of 64 targets is long where its
// chunks are not far (37,692 targets x 218 sources: 62 us a call against 74 in pairs).
__global__ void __launch_bounds__(128) k_direct_f32_few(const uint32_t *__restrict__ src_pc,
                                                        const float *__restrict__ src_q, int ns,
                                                        const uint32_t *__restrict__ trg_key, int nt, DirectK k, int nx,
                                                        int ny, float *__restrict__ out_dense) {
    __shared__ float4 sp[512];
    const int t = blockIdx.x * 128 + threadIdx.x;
    const uint32_t tp = key_pc(trg_key[min(t, nt - 1)]);
    const float tx = (float)pc_i(tp), ty = (float)pc_j(tp), tz = (float)pc_k(tp);
    float acc = 0.f;
    for (int s0 = 0; s0 < ns; s0 += 512) {
        const int m = min(512, ns - s0);
        __syncthreads();
        for (int u = threadIdx.x; u < m; u += 128) {
            const uint32_t p = src_pc[s0 + u];
            sp[u] = make_float4((float)pc_i(p), (float)pc_j(p), (float)pc_k(p), src_q[s0 + u] * k.wscale);
        }
        __syncthreads();
        for (int c = 0; c < m; c += DC) {
            const int end = min(c + DC, m);
            float part = 0.f;
#pragma unroll 4
            for (int u = c; u < end; ++u) {
                const float4 p = sp[u];
                const float dx = tx - p.x, dy = ty - p.y, dz = tz - p.z, d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                float a, b;
                general_term(d2, p.w, k, a, b);
                part = fmaf(a, b, part);
            }
            acc += part;
        }
    }
    if (t < nt) out_dense[(int64_t)pc_i(tp) + (int64_t)nx * ((int64_t)pc_j(tp) + (int64_t)ny * pc_k(tp))] = acc;
}

// ---------------------------------------------------------------- FP64
// G h^3 times the source scale at squared cell offset d2, FP64 (d2 = 0: the self term)
__device__ __forceinline__ double pair_weight(int d2, const KParams64 &kp, int self_mode) {
    double v;
    if (d2) {
        const double R = kp.h * sqrt((double)d2);
        v = kp.C * exp(-kp.alpha * R) * (-expm1(-kp.bma * R)) / (R * R * R) * kp.vol;
    } else {
        v = self_mode ? kp.self_int : 0.0;
    }
    return v * kp.scale;
}

// Kahan-Babuska (Neumaier) compensated accumulation
__device__ __forceinline__ void neumaier(double &acc, double &comp, double term) {
    const double s = acc + term;
    comp += fabs(acc) >= fabs(term) ? (acc - s) + term : (term - s) + acc;
    acc = s;
}

// acc + comp += w q for w >= 0, the product unrounded.  eq: the biased exponent of q, less 1020.  Where |w q|
// is at most half of |acc| by the exponents, acc and the fused sum are so close that their difference
// is exact and one more FMA forms what the sum lost; the first terms, and one much larger than all
// before it, go by Neumaier's rule with the product's own rounding error.
__device__ __forceinline__ void add_product(double &acc, double &comp, double w, double q, int eq) {
    if ((__double2hiint(w) >> 20) + eq <= (__double2hiint(acc) >> 20 & 0x7ff)) {
        const double s = fma(w, q, acc);
        comp += fma(w, q, acc - s);
        acc = s;
    } else {
        const double t = w * q;
        comp += fma(w, q, -t);
        neumaier(acc, comp, t);
    }
}

__global__ void k_pair_table(KParams64 kp, int self_mode, int entries, double *__restrict__ table) {
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < entries; d += gridDim.x * blockDim.x)
        table[d] = pair_weight(d, kp, self_mode);
}

// On the grid a pair's weight depends on the integer d2 alone, so it is read from a table built
// for the call (the same arithmetic) instead of two exponentials, a root and a division in FP64
// per pair, about 250 instructions at 2 per SM and clock.  What is left is bound by the FP64 unit
// too: two FMAs and two additions a pair, each product compensated (this is the library's own
// reference: with one compensated addition per 16 products, 1.4 operations a pair, the rms error of
// a sum of weights of both signs was 4.0e-15, of positive ones over twelve decades 6.0e-17; each for
// itself, as pair by pair, 2.2e-15 and 5.1e-17, and with the products unrounded a tenth less).  32 targets per CTA; its eight warps take an
// eighth of each source tile and their sums are added in order.
// 24^3 cells, all pairs (1.9e8): 68.6 ms with G per pair, 0.64 with groups of 16, 1.5 ms so.
constexpr int DW = 8;            // warps per CTA
constexpr int DT64 = 512;        // sources per tile
constexpr int TABLE_SMEM = 12288;   // entries of a table kept in shared memory (96 KB)

template <bool SMEM>
__global__ void __launch_bounds__(32 * DW) k_direct_f64_table(const uint32_t *__restrict__ src_pc,
                                                              const float *__restrict__ src_q, int ns,
                                                              const uint32_t *__restrict__ trg_key, int nt,
                                                              const double *__restrict__ table, int entries, int nx,
                                                              int ny, double *__restrict__ out_dense) {
    __shared__ int4 sp[DT64];
    __shared__ double sq[DT64];
    __shared__ double part[DW][32][2];
    extern __shared__ double stab[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (SMEM)
        for (int e = threadIdx.x; e < entries; e += 32 * DW) stab[e] = table[e];
    const double *tab = SMEM ? stab : table;
    const int t = blockIdx.x * 32 + lane;
    const uint32_t tp = key_pc(trg_key[min(t, nt - 1)]);
    const int ti = pc_i(tp), tj = pc_j(tp), tk = pc_k(tp);
    double acc = 0.0, comp = 0.0;
    for (int s0 = 0; s0 < ns; s0 += DT64) {
        const int m = min(DT64, ns - s0);
        __syncthreads();
        for (int u = threadIdx.x; u < m; u += 32 * DW) {
            const uint32_t p = src_pc[s0 + u];
            const double q = (double)src_q[s0 + u];
            sp[u] = make_int4(pc_i(p), pc_j(p), pc_k(p), (__double2hiint(q) >> 20 & 0x7ff) - 1020);
            sq[u] = q;
        }
        __syncthreads();
        const int u1 = min(m, (warp + 1) * (DT64 / DW));
#pragma unroll 4
        for (int u = warp * (DT64 / DW); u < u1; ++u) {
            const int4 p = sp[u];
            const int di = ti - p.x, dj = tj - p.y, dk = tk - p.z;
            add_product(acc, comp, tab[di * di + dj * dj + dk * dk], sq[u], p.w);
        }
    }
    part[warp][lane][0] = acc;
    part[warp][lane][1] = comp;
    __syncthreads();
    if (warp == 0 && t < nt) {
        for (int w = 1; w < DW; ++w) {
            neumaier(acc, comp, part[w][lane][0]);
            comp += part[w][lane][1];
        }
        out_dense[(int64_t)ti + (int64_t)nx * ((int64_t)tj + (int64_t)ny * tk)] = acc + comp;
    }
}

// G per pair: for sets so small that the table would cost more than the pairs
__global__ void __launch_bounds__(256) k_direct_f64(const uint32_t *__restrict__ src_pc,
                                                    const float *__restrict__ src_q, int ns,
                                                    const uint32_t *__restrict__ trg_key, int nt,
                                                    KParams64 kp, int self_mode, int nx, int ny,
                                                    double *__restrict__ out_dense) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= nt) return;
    const uint32_t tp = key_pc(trg_key[t]);
    const int ti = pc_i(tp), tj = pc_j(tp), tk = pc_k(tp);
    double acc = 0.0, comp = 0.0;
    for (int s = 0; s < ns; ++s) {
        const uint32_t p = src_pc[s];
        const int di = ti - pc_i(p), dj = tj - pc_j(p), dk = tk - pc_k(p);
        neumaier(acc, comp, pair_weight(di * di + dj * dj + dk * dk, kp, self_mode) * (double)src_q[s]);
    }
    out_dense[(int64_t)ti + (int64_t)nx * ((int64_t)tj + (int64_t)ny * tk)] = acc + comp;
}

// A table entry costs as much as a pair without it: the table is built from two pairs an entry on.
int64_t direct_table_entries(int64_t ns, int64_t nt, int nx, int ny, int nz) {
    const int64_t n = (int64_t)(nx - 1) * (nx - 1) + (int64_t)(ny - 1) * (ny - 1) + (int64_t)(nz - 1) * (nz - 1) + 1;
    return ns * nt >= 2 * n ? n : 0;
}

int direct_launch(const DirectArgs &A, cudaStream_t st) {
    if (A.nt == 0) return 0;
    if (A.fp64 && A.table) {
        const int n = (int)A.table_entries;
        k_pair_table<<<std::min((n + 63) / 64, 152 * 16), 64, 0, st>>>(A.kp64, A.self_mode, n, A.table);
        const int grid = (A.nt + 31) / 32;
        if (n <= TABLE_SMEM) {
            cudaFuncSetAttribute(k_direct_f64_table<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TABLE_SMEM * 8);
            k_direct_f64_table<true><<<grid, 32 * DW, n * sizeof(double), st>>>(A.src_pc, A.src_q, A.ns, A.trg_key, A.nt, A.table,
                                                                                n, A.nx, A.ny, (double *)A.out);
        } else {
            k_direct_f64_table<false><<<grid, 32 * DW, 0, st>>>(A.src_pc, A.src_q, A.ns, A.trg_key, A.nt, A.table, n, A.nx, A.ny,
                                                                (double *)A.out);
        }
    } else if (A.fp64) {
        k_direct_f64<<<(A.nt + 255) / 256, 256, 0, st>>>(A.src_pc, A.src_q, A.ns, A.trg_key, A.nt, A.kp64, A.self_mode,
                                                         A.nx, A.ny, (double *)A.out);
    } else {
        const KParams64 &d = A.kp64;
        DirectK k;
        const double log2e = 1.4426950408889634;
        k.a2 = (float)(d.alpha * d.h * log2e);
        k.b2 = (float)(d.bma * d.h * log2e);
        k.wscale = (float)(d.scale * d.C);
        k.self = A.self_mode ? (float)(d.self_int / d.C) : 0.f;
        k.bma_h = (float)(d.bma * d.h);
        const double far = 25.5 / (d.bma * d.h * log2e), near = std::max(1.0, 0.5 / (d.bma * d.h));
        k.far2 = (float)std::max(far * far, near * near);
        k.near2 = (float)(near * near);
        // 64 targets a warp: four warps a CTA share the staged tile where that still fills the chip
        // pairs of targets from three CTAs of 256 targets an SM on
        if (A.nt >= 256 * 152 * 3)
            k_direct_f32<<<(A.nt + 255) / 256, 32 * WARPS, 0, st>>>(A.src_pc, A.src_q, A.ns, A.trg_key, A.nt, k, A.nx, A.ny,
                                                                    (float *)A.out);
        else
            k_direct_f32_few<<<(A.nt + 127) / 128, 128, 0, st>>>(A.src_pc, A.src_q, A.ns, A.trg_key, A.nt, k, A.nx, A.ny,
                                                                 (float *)A.out);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace sph
