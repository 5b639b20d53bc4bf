"""The Gram-matrix base case: panels at its size limits and block edges, and
ill-conditioned panels, which it must hand to the TSQR untouched, against the
oracle."""

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


# widths around the 32-wide blocks, from the smallest to the largest, at the
# least height (4 w) and odd taller ones
@pytest.mark.parametrize("w", [16, 17, 31, 32, 33, 64, 65, 96, 127, 128])
@pytest.mark.parametrize("tall", [0, 1])
def test_panel_matches_oracle(gb, ctx, orc, w, tall):
    m = 4 * w if not tall else 9 * w + 1001
    a = workloads.graded(m, w, 70 + w, 4.0 if tall else 0.0)
    VR, T, nb = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL, lda_pad=3 * tall)
    _gpu.compare_factor(a, VR, T, gb.GBQR_T_FULL, nb, orc, f"{m}x{w}")
    # the same panel by TSQR
    VR2, T2, _ = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL, gb.opts(cutoff_b=32))
    s = np.linalg.norm(a, axis=0)
    assert np.max(np.abs(np.tril(VR - VR2, -1))) <= 1e-12 and np.max(np.abs(T - T2)) <= 1e-12
    assert np.max(np.abs(np.triu(VR - VR2)) / s[None, :]) <= 1e-12


def _awkward(kind, m, w):
    a = workloads.gaussian(m, w, 90)
    if kind == "parallel":            # the last block's columns nearly the first one's
        a[:, w - 1] = a[:, 0] + 1e-9 * a[:, w - 1]
    elif kind == "correlated":        # every pivot small
        a = a + 30.0 * a[:, :1]
    elif kind == "triangular":        # R = -A, empty subcolumns
        a = workloads.upper_triangular(m, w, 91)
    return np.asfortranarray(a)


@pytest.mark.parametrize("kind", ["parallel", "correlated", "triangular"])
@pytest.mark.parametrize("w", [24, 100])
def test_awkward_panels(gb, ctx, orc, kind, w):
    """Same V, T, R as TSQR's, which the oracle pins elsewhere, up to the
    conditioning of the columns; a valid QR in any case."""
    a = _awkward(kind, 7 * w, w)
    VR, T, nb = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL)
    Q = _gpu.q_from_panels(VR, T, w)
    R = np.triu(VR[:w])
    scale = np.abs(a).max()
    assert np.linalg.norm(a / scale - Q @ (R / scale)) <= 1e-13 * np.linalg.norm(a / scale)
    assert np.linalg.norm(Q.T @ Q - np.eye(w)) <= 1e-13 * w
    if kind != "parallel":
        _gpu.compare_factor(a / scale, np.where(np.tri(*VR.shape, -1, dtype=bool), VR, VR / scale), T,
                            gb.GBQR_T_FULL, nb, orc, kind)


@pytest.mark.parametrize("scale", [1e-200, 1e200])
def test_gram_matrix_out_of_range(gb, ctx, scale):
    """Squares that underflow or overflow: the panel goes to the TSQR, whose
    result (which squares them as well) it is, bit for bit."""
    a = workloads.gaussian(168, 24, 94) * scale
    VR, T, _ = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL)
    VR2, T2, _ = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL, gb.opts(cutoff_b=24))
    assert np.array_equal(VR, VR2, equal_nan=True) and np.array_equal(T, T2, equal_nan=True)


def test_zero_and_nan_columns(gb, ctx):
    a = workloads.gaussian(600, 40, 92)
    a[:, 17] = 0.0
    VR, T, _ = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL)
    Q = _gpu.q_from_panels(VR, T, 40)
    assert np.linalg.norm(a - Q @ np.triu(VR[:40])) <= 1e-13 * np.linalg.norm(a)
    b = workloads.gaussian(600, 40, 93)
    b[599, 39] = np.nan
    VR, _, _ = _gpu.factor_gpu(ctx, b, gb.GBQR_T_FULL)
    st, info = ctx.sync()
    assert st == gb.GBQR_ENONFINITE and info.nonfinite
    assert not np.isfinite(VR[:, 39]).all()


@pytest.mark.parametrize("m,n", [(65537, 16), (70001, 130), (140000, 40)])
def test_panels_taller_than_the_usual_split(gb, ctx, m, n):
    """More rows than 128 splits of 512 hold: the Gram matrix's partials have
    their room (a valid QR, Q applied to the identity's columns by the panels)."""
    a = workloads.gaussian(m, n, 95)
    VR, T, nb = _gpu.factor_gpu(ctx, a, gb.GBQR_T_PANEL)
    Q = _gpu.q_from_panels(VR, T, nb)
    assert np.linalg.norm(a - Q @ np.triu(VR[:n])) <= 1e-13 * np.linalg.norm(a)
    assert np.linalg.norm(Q.T @ Q - np.eye(n)) <= 1e-13 * n
