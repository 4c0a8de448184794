"""The near-field forms alone, against the FP64 oracle.

Every cell of a 16^3 grid is a source (i_frac 0), the weights are zero outside the first 12^3 cells
and the targets are the leaf of cells 4 .. 7 of each axis: all weights lie in the leaf and in its
neighbours, every source box beyond them sums to exactly zero, and S is the near field and nothing
else.  Its sums are taken in a fixed order, so a form's result is the same bits at every call.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N, LO, HI = 16, 4, 8
PAIRS, TABLE, MATRIX = {"SPH_NEAR_OVERLAP": "0"}, {"SPH_NEAR_MMA": "0"}, {"SPH_NEAR_MMA": "1"}


@pytest.fixture(scope="module")
def sph():
    import __graft_entry__ as g
    g.build()
    import paper_2112_10059_gb300 as m
    return m


def _targets():
    m = np.zeros((N, N, N), np.uint8)
    m[LO:HI, LO:HI, LO:HI] = 1
    return m.reshape(-1)


def _weights(kind, seed):
    u = np.random.default_rng(seed).random((N, N, N))
    q = {"uniform": 0.5 + 0.5 * u, "const": np.ones_like(u), "noise": u, "wide": 10.0 ** (-6.0 * u)}[kind]
    q[12:] = q[:, 12:] = q[:, :, 12:] = 0.0
    return q.astype(np.float32).reshape(-1)


def _near(sph, monkeypatch, form, q, h, pO2, scale=1.0):
    import torch
    for k in ("SPH_NEAR_OVERLAP", "SPH_NEAR_MMA"):
        monkeypatch.delenv(k, raising=False)
    for k, v in form.items():
        monkeypatch.setenv(k, v)
    c = sph.Context(0)
    sph.set_grid(c, N, N, N, h, pO2)
    sph.set_sources(c, torch.from_numpy(q).cuda(), scale)
    sph.set_targets(c, mask=torch.from_numpy(_targets()).cuda())
    sph.set_criteria(c, 0.0, leaf_size=64)
    out, _ = sph.eval_sph(c)
    S = out.cpu().numpy()[_targets() != 0]
    c.close()
    return S


def _exact(q, h, pO2, scale=1.0):
    a, b = oracle.alpha_beta(pO2, 0.035, 2.0)
    return oracle.sph(N, N, N, h, a, b, q, scale, np.nonzero(q)[0].astype(np.int32),
                      np.nonzero(_targets())[0].astype(np.int32))


# cell edge (cm) and pO2 (Torr): both sides of the series form, and a coarse grid
GRIDS = [(1.0 / 128, 150.0), (1e-3, 15.0), (1.0 / 24, 150.0)]


@pytest.mark.parametrize("kind", ["uniform", "const", "noise", "wide"])
@pytest.mark.parametrize("h,pO2", GRIDS)
def test_table_form_no_further_off_than_pair_by_pair(sph, monkeypatch, h, pO2, kind):
    """The offset table holds the values that the kernel of each pair has, so its sums must be no
    further from FP64 than those taken pair by pair (rms over eight fields)."""
    err = {"pairs": [], "table": []}
    for seed in range(8):
        q = _weights(kind, seed)
        ref = _exact(q, h, pO2)
        err["pairs"].append(_near(sph, monkeypatch, PAIRS, q, h, pO2) / ref - 1)
        err["table"].append(_near(sph, monkeypatch, TABLE, q, h, pO2) / ref - 1)
    rms = {k: np.sqrt(np.mean(np.square(v))) for k, v in err.items()}
    assert rms["table"] <= rms["pairs"], rms


@pytest.mark.parametrize("kind", ["uniform", "const", "noise", "wide"])
@pytest.mark.parametrize("h,pO2", GRIDS)
def test_matrix_form_no_further_off_than_pair_by_pair(sph, monkeypatch, h, pO2, kind):
    """The products of the three BF16 parts, summed by the tensor core, take the place of FP32 sums
    pair by pair and must be no further from FP64 (rms over eight fields).  The form did run: the
    table's sums of the same leaf differ from it in their last places."""
    err = {"pairs": [], "matrix": []}
    for seed in range(8):
        q = _weights(kind, seed)
        ref = _exact(q, h, pO2)
        S = _near(sph, monkeypatch, MATRIX, q, h, pO2)
        assert not np.array_equal(S, _near(sph, monkeypatch, TABLE, q, h, pO2))
        err["pairs"].append(_near(sph, monkeypatch, PAIRS, q, h, pO2) / ref - 1)
        err["matrix"].append(S / ref - 1)
    rms = {k: np.sqrt(np.mean(np.square(v))) for k, v in err.items()}
    assert rms["matrix"] <= rms["pairs"], rms


def test_matrix_form_sums_every_part(sph, monkeypatch):
    """Weights whose third BF16 part is nearly as large as it gets, and of one sign: 1 + 3 * 2^-10 +
    2^-17 - 2^-21 is 1 (hi) + 3 * 2^-10 (mid) + 2^-17 - 2^-21 (lo), so that a sum without lo hi would be
    7.1e-6 too small, one without lo hi and hi mid or mid hi far more.  What remains is at most a unit of
    2^-23 for the four accumulators an offset, 27 FP32 additions of 2^-24 each and 2^-22 of the kernel
    values' rounding and mean correction: 2e-6 in all."""
    h, pO2 = 1.0 / 128, 150.0
    # the near field multiplies the weights by C = 1 / (4 pi ln(chi ratio)): a scale that undoes it
    q = _weights("const", 0) * np.float32(1 + 3 * 2.0 ** -10 + 2.0 ** -17 - 2.0 ** -21)
    scale = 4 * np.pi * np.log(2.0 / 0.035)
    S = _near(sph, monkeypatch, MATRIX, q, h, pO2, scale)
    assert np.max(np.abs(S / _exact(q, h, pO2, scale) - 1)) < 2e-6


@pytest.mark.parametrize("value", [np.nan, np.inf, 2.0 ** 126, "small"])
def test_weights_that_the_matrix_form_leaves_to_the_table(sph, monkeypatch, value):
    """NaN, infinity, and weights whose BF16 parts would overflow or underflow: the table takes every
    leaf, with the same bits as where the matrix form is off."""
    q = _weights("uniform", 1)
    if value == "small":
        q = (q * np.float32(2.0 ** -90)).astype(np.float32)
    else:
        q = q.reshape(N, N, N)
        q[1, 2, 3] = value
        q = q.reshape(-1)
    h, pO2 = 1.0 / 128, 150.0
    a, b = _near(sph, monkeypatch, MATRIX, q, h, pO2), _near(sph, monkeypatch, TABLE, q, h, pO2)
    assert np.array_equal(a, b, equal_nan=True)
    if value == "small":
        assert np.all(a > 0)
    elif not np.isfinite(value):
        assert not np.any(np.isfinite(a))


@pytest.mark.parametrize("nx,ny,nz,leaf", [(16, 16, 16, 512), (16, 15, 13, 4096), (16, 16, 1, 64)])
def test_coarse_leaves_go_pair_by_pair(sph, monkeypatch, nx, ny, nz, leaf):
    """Leaves of edge 8 and 16, for which the offset table is not made: the near field beside the far
    field sums them as the kernel after it does (SPH_NEAR_OVERLAP=0), to the same bits.  All boxes are
    adjacent, so there is no far field."""
    import torch
    q = torch.from_numpy(np.random.default_rng(4).random(nx * ny * nz).astype(np.float32)).cuda()
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("SPH_NEAR_OVERLAP", flag)
        c = sph.Context(0)
        sph.set_grid(c, nx, ny, nz, 1.0 / 128, 150.0)
        sph.set_sources(c, q, 1.0)
        sph.set_targets(c)
        sph.set_criteria(c, 0.0, leaf_size=leaf)
        out.append(sph.eval_sph(c)[0].cpu().numpy())
        assert sph.get_tree(c)["V"].size == 0
        c.close()
    assert np.array_equal(out[0], out[1]) and np.all(out[0] > 0)
