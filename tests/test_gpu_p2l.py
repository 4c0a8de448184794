"""P2L (X lists) at the far end of a long grid: the same field, moved by a multiple of the largest
box, has the same tree and the same offsets, so S may differ by the rounding of sums alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sph():
    import __graft_entry__ as g
    g.build()
    import paper_2112_10059_gb300 as m
    return m


@pytest.mark.parametrize("far", ["chebyshev", "surface"])
def test_p2l_does_not_depend_on_the_place(sph, far):
    """Targets in a dense corner of 16^3 cells, sources beyond it in one leaf of edge 16: every other
    contribution is a U entry.  Positions of nodes and sources relative to the box are exact or rounded
    at the box's size, 2^-24 of at most 32 cells, so a term changes by nothing; order 8 (surface: 6)
    sums of 512 nodes and 24 sources in one fixed order."""
    import torch
    nx, n, edge = 1024, 64, 16
    rng = np.random.default_rng(8)
    src = np.unique(rng.integers(0, edge, (24, 3)), axis=0) + np.array([edge, 0, 0])
    w = (0.5 + rng.random(len(src))).astype(np.float32)
    S = []
    for x0 in (0, nx - n):
        q = np.zeros((n, n, nx), np.float32)
        q[src[:, 2], src[:, 1], x0 + src[:, 0]] = w
        m = np.zeros((n, n, nx), np.uint8)
        m[:edge, :edge, x0:x0 + edge] = 1
        c = sph.Context(0)
        sph.set_grid(c, nx, n, n, 1.0 / 1024, 150.0)
        sph.set_sources(c, torch.from_numpy(q.reshape(-1)).cuda(), 1.0)
        sph.set_targets(c, mask=torch.from_numpy(m.reshape(-1)).cuda())
        sph.set_criteria(c, 0.1, leaf_size=64, m2l_precision=sph.M2L_F32)
        sph.set_far_field(c, sph.FAR_CHEBYSHEV if far == "chebyshev" else sph.FAR_SURFACE, 8 if far == "chebyshev" else 6)
        out, st = sph.eval_sph(c, stats=True)
        S.append(out.cpu().numpy().astype(np.float64).reshape(n, n, nx)[:edge, :edge, x0:x0 + edge])
        assert st.n_x > 0 and st.n_w == 0 and st.n_v == 0
        c.close()
    assert np.all(S[0] > 0)
    assert np.max(np.abs(S[1] / S[0] - 1)) < 1e-6
