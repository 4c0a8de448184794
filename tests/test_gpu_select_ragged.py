"""Selection on grids whose enclosing power-of-two cube is mostly empty: bricks of the cube that lie
outside the grid (known to select nothing, in every form of the selection), bricks that reach past
it, and statistics of fields and masks with and without 16-byte rows, against the oracle's rules."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [(130, 3, 1), (1, 200, 17), (40, 40, 1), (18, 33, 50), (64, 5, 37)]


@pytest.fixture(scope="module")
def sph():
    import __graft_entry__ as g
    g.build()
    import paper_2112_10059_gb300 as m
    return m


@pytest.mark.parametrize("form", ["default", "SPH_SELECT_LOOKBACK", "SPH_SELECT_TWO_PASS"])
@pytest.mark.parametrize("i_frac", [0.0, 0.4])
@pytest.mark.parametrize("targets", ["all", "emag", "mask", "block_mask"])
@pytest.mark.parametrize("shape", SHAPES)
def test_selection_of_ragged_grids(sph, monkeypatch, shape, targets, i_frac, form):
    import torch
    if form != "default":
        monkeypatch.setenv(form, "1")
    nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(n)
    q = rng.random(n).astype(np.float32)
    q[q < 0.2] = 0.0
    emag = mask = None
    if targets == "emag":
        emag = (rng.random(n) ** 3).astype(np.float32)
        emag[: n // 3] = 1.0               # whole bricks above the threshold
    elif targets == "mask":
        mask = (rng.random(n) < 0.3).astype(np.uint8)
    elif targets == "block_mask":
        mask = np.zeros(shape[::-1], np.uint8)
        mask[: (nz + 1) // 2, : (ny + 1) // 2, 16:] = 1
        mask[0, 0, 0] = 1
        mask = mask.reshape(-1).copy()
    c = sph.Context(0)
    sph.set_grid(c, nx, ny, nz, 1e-3, 150.0)
    sph.set_sources(c, torch.from_numpy(q).cuda(), 1.0)
    sph.set_targets(c, emag=None if emag is None else torch.from_numpy(emag).cuda(),
                    mask=None if mask is None else torch.from_numpy(mask).cuda())
    sph.set_criteria(c, i_frac, 0.5, 0.0)
    S = sph.eval_sph(c)[0].cpu().numpy()
    J, T = sph.get_selection(c)
    c.close()
    Jo, To = oracle.select(q, emag, mask, i_frac, 0.5, 0.0)
    assert np.array_equal(J, Jo) and np.array_equal(T, To)
    off = np.ones(n, bool)
    off[T] = False
    assert np.all(S[off] == 0) and np.all(S[T] > 0)
