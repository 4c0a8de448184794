"""The direct sums where their forms change: FP64 with the pair weights in shared memory, in global
memory or formed pair by pair; FP32 with chunks of sources that are far, near or meet the targets,
with and without the series form, one and four warps a CTA, and counts that fill no tile."""
import numpy as np
import pytest

import oracle
import sph_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sph():
    import __graft_entry__ as g
    g.build()
    import paper_2112_10059_gb300 as m
    return m


# nx, ny, nz, h (cm), pressure (Torr), share of the cells that are sources, targets (share of a random mask)
CASES = [(24, 24, 24, 0.2 / 24, 760.0, 1.0, 1.0),        # all pairs, weights in shared memory
         (40, 24, 33, 1e-3, 76.0, 0.02, 0.3),            # R small enough for the series form
         (40, 24, 33, 1e-2, 760.0, 0.02, 0.3),
         (200, 9, 7, 5e-3, 760.0, 0.03, 0.5),            # 39,702 weights: global memory
         (64, 50, 41, 1.0 / 64, 760.0, 3.5 / 131200, 3.5 / 131200),   # a few pairs: no table
         (96, 96, 96, 1.0 / 96, 380.0, 3e-4, 1.0),       # four warps a CTA, mostly far chunks
         (1, 1, 1, 0.01, 760.0, 1.0, 1.0)]


@pytest.mark.parametrize("case", CASES)
def test_direct_forms(sph, case):
    import torch
    nx, ny, nz, h, p, fs, ft = case
    n = nx * ny * nz
    u = si.uniform01(77, n)
    q = np.where(u <= fs, 0.5 + 0.5 * si.uniform01(78, n), 0.0).astype(np.float32)
    q[np.argmin(u)] = 1.0
    mask = (si.uniform01(79, n) <= ft).astype(np.uint8)
    mask[n // 2] = 1
    ctx = sph.Context(0)
    pO2 = si.pO2_of(p)
    sph.set_grid(ctx, nx, ny, nz, h, pO2)
    qd, md = torch.from_numpy(q).cuda(), torch.from_numpy(mask).cuda()
    sph.set_sources(ctx, qd, 0.01)
    sph.set_targets(ctx, mask=md)
    sph.set_criteria(ctx, 0.25)
    J = np.nonzero(q >= 0.25)[0].astype(np.int32)
    T = np.nonzero(mask)[0].astype(np.int32)
    if T.size * J.size > 2e8:                # a sample of the targets is checked
        S = T[:: max(1, int(T.size * J.size / 2e8) + 1)]
    else:
        S = T
    alpha, beta = oracle.alpha_beta(pO2, 0.035, 2.0)
    ref = oracle.sph(nx, ny, nz, h, alpha, beta, q, 0.01, J, S)
    d64 = sph.eval_direct(ctx, fp64=True).cpu().numpy()
    assert np.max(np.abs(d64[S] / ref - 1)) < 1e-13
    off = np.ones(n, bool)
    off[T] = False
    assert np.all(d64[off] == 0)
    d32 = sph.eval_direct(ctx, fp64=False).cpu().numpy().astype(np.float64)
    # positive terms added one after another in FP32, each within a few ulp of the approximate
    # exponentials and root (arguments up to 40 in log2 units: 2^-24 of them)
    tol = J.size * 2.0 ** -24 + 8e-6
    assert np.max(np.abs(d32[S] / ref - 1)) < tol
    assert np.all(d32[off] == 0)


@pytest.mark.parametrize("shape", [(16, 16, 16), (200, 9, 9)])     # weights in shared and in global memory
def test_fp64_sums_keep_what_large_terms_of_both_signs_cancel(sph, shape):
    """Weights +Q and -Q in cells opposite each other across the target cancel exactly, as their terms
    are the same product: what is left is the sum of the others, 1e-12 of the size.  A sum that adds
    several products before it compensates rounds them at the size of the largest, 1e-16 Q: 1e-5 of
    the result.  Compensated one by one the bound is that of the other sums here."""
    import torch
    nx, ny, nz = shape
    cx, cy, cz = nx // 2, ny // 2, nz // 2
    small = si.uniform01(91, nx * ny * nz).astype(np.float32).reshape(nz, ny, nx) + np.float32(0.5)
    small[cz, cy, cx] = 0.0
    q = small.copy()
    for k, (dx, dy, dz) in enumerate([(1, 0, 0), (2, 0, 0), (0, 1, 0), (0, 2, 1), (3, 1, 0)]):
        for s in (1, -1):
            small[cz + s * dz, cy + s * dy, cx + s * dx] = 0.0
            q[cz + s * dz, cy + s * dy, cx + s * dx] = s * 1e12 / (k + 1)
    mask = np.zeros((nz, ny, nx), np.uint8)
    mask[cz, cy, cx] = 1
    t = np.nonzero(mask.reshape(-1))[0].astype(np.int32)
    h, pO2 = 0.01, si.pO2_of(760.0)
    ctx = sph.Context(0)
    sph.set_grid(ctx, nx, ny, nz, h, pO2)
    qd, md = torch.from_numpy(q.reshape(-1)).cuda(), torch.from_numpy(mask.reshape(-1)).cuda()
    sph.set_sources(ctx, qd, 1.0)
    sph.set_targets(ctx, mask=md)
    sph.set_criteria(ctx, 0.0)
    d64 = sph.eval_direct(ctx, fp64=True).cpu().numpy()[t]
    ctx.close()
    alpha, beta = oracle.alpha_beta(pO2, 0.035, 2.0)
    ref = oracle.sph(nx, ny, nz, h, alpha, beta, small.reshape(-1), 1.0, np.nonzero(small.reshape(-1))[0].astype(np.int32), t)
    assert np.abs(d64 / ref - 1) < 1e-13


@pytest.mark.parametrize("ny,nz", [(3, 3), (12, 12)])     # one target a thread; pairs of targets
def test_fp32_terms_of_strongly_absorbed_sources(sph, ny, nz):
    """Sources at one end of 1024 cells of 0.0135 cm at atmospheric pressure: at the other end alpha R
    is 72 and e^{-alpha R} / d^3 in cells 5e-41, below FP32's normal range, while S = w G stays far above
    it.  The bound is that of the exponential's argument (105 in log2 units, 2^-24 of it, and the
    constants' rounding) and of 20 FP32 additions."""
    import torch
    nx, h, pO2 = 1024, 0.0135, 150.0
    q = np.zeros((nz, ny, nx), np.float32)
    q[:, :, 0] = 1.0 + np.arange(ny * nz, dtype=np.float32).reshape(nz, ny) / (ny * nz)
    ctx = sph.Context(0)
    sph.set_grid(ctx, nx, ny, nz, h, pO2)
    qd = torch.from_numpy(q.reshape(-1)).cuda()
    sph.set_sources(ctx, qd, 1e20)
    sph.set_targets(ctx)
    sph.set_criteria(ctx, 0.5)
    d32 = sph.eval_direct(ctx, fp64=False).cpu().numpy().astype(np.float64)
    ctx.close()
    alpha, beta = oracle.alpha_beta(pO2, 0.035, 2.0)
    T = np.arange(1000, 1024, dtype=np.int32)
    ref = oracle.sph(nx, ny, nz, h, alpha, beta, q.reshape(-1), 1e20, np.nonzero(q.reshape(-1))[0].astype(np.int32), T)
    assert np.all(ref > 1e-25)
    assert np.max(np.abs(d32[T] / ref - 1)) < 2 * 105 * 2.0 ** -24 + q[:, :, 0].size * 2.0 ** -24 + 2e-6


@pytest.mark.parametrize("ft", [0.01, 1.0])     # one target a thread; pairs of targets
def test_fp32_sums_of_many_small_terms_behind_a_large_one(sph, ft):
    """A source of weight 1, the first in Morton order, and 16,383 of 3e-8: at targets as far from all of
    them each small term is below half a unit in the last place of the sum, and one chain loses them all,
    up to 5e-4 of it.  32 terms are summed at a time, and the sums of the chunks: 32 + 16384 / 32
    roundings of 2^-24 one after another, whose errors add as squares, and 1e-6 at most for the
    approximate root and exponentials of a term (2^-22.9, cubed, and 2^-22.5)."""
    import torch
    nx, ny, nz, h, pO2 = 64, 64, 32, 1e-3, 150.0
    n = nx * ny * nz
    q = np.zeros((nz, ny, nx), np.float32)
    q[:16, :32, :32] = 3e-8 * (0.75 + 0.25 * si.uniform01(93, 16384).reshape(16, 32, 32))
    q[0, 0, 0] = 1.0
    mask = (si.uniform01(94, n) <= ft).astype(np.uint8)
    ctx = sph.Context(0)
    sph.set_grid(ctx, nx, ny, nz, h, pO2)
    qd, md = torch.from_numpy(q.reshape(-1)).cuda(), torch.from_numpy(mask).cuda()
    sph.set_sources(ctx, qd, 1.0)
    sph.set_targets(ctx, mask=md)
    sph.set_criteria(ctx, 1e-9)
    d32 = sph.eval_direct(ctx, fp64=False).cpu().numpy().astype(np.float64)
    ctx.close()
    T = np.nonzero(mask)[0].astype(np.int32)
    T = T[(T % nx >= 40) & (T // nx % ny >= 40)]
    T = T[:: max(1, T.size // 500)]
    J = np.nonzero(q.reshape(-1))[0].astype(np.int32)
    alpha, beta = oracle.alpha_beta(pO2, 0.035, 2.0)
    ref = oracle.sph(nx, ny, nz, h, alpha, beta, q.reshape(-1), 1.0, J, T)
    assert np.sqrt(np.mean((d32[T] / ref - 1) ** 2)) < 2.0 ** -24 * np.sqrt(32 + J.size / 32) + 1e-6
