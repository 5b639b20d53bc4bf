"""Panels whose columns share a direction: what the Gram-matrix base case
accepts keeps the orthogonality and the backward error of the TSQR."""

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu

U = np.finfo(float).eps / 2


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


def _columns(kind, m, w, seed):
    a = workloads.gaussian(m, w, seed)
    rng = np.random.default_rng(seed)
    if kind.startswith("mean"):             # a mean of so many standard deviations
        return a + float(kind[4:])
    if kind == "uniform":
        return rng.random((m, w))
    if kind == "intercept":                 # a column of ones beside columns with a mean
        a = a + 1.5
        a[:, 0] = 1.0
        return a
    if kind.startswith("factor"):           # a common column
        return a + float(kind[6:]) * rng.standard_normal((m, 1))
    if kind.startswith("chain"):            # each column correlated with the one before it
        r = float(kind[5:])
        for j in range(1, w):
            a[:, j] = r * a[:, j - 1] + np.sqrt(1 - r * r) * a[:, j]
        return a
    return a


KINDS = ["plain", "mean0.5", "mean0.7", "mean1", "mean2", "mean3", "uniform", "intercept", "factor1", "factor3", "chain0.5", "chain0.9"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("m,n", [(1024, 128), (512, 128), (8192, 128), (700, 64), (64, 16), (4096, 512)])
def test_no_less_accurate_than_the_tsqr(gb, ctx, kind, m, n):
    a = np.asfortranarray(_columns(kind, m, n, 600 + n))
    err = []
    for o in (None, gb.opts(cutoff_b=32)):
        VR, T, nb = _gpu.factor_gpu(ctx, a, gb.GBQR_T_PANEL, o)
        Q = _gpu.q_from_panels(VR, T, nb)
        err.append((np.linalg.norm(Q.T @ Q - np.eye(n), 2), np.linalg.norm(a - Q @ np.triu(VR[:n])) / np.linalg.norm(a)))
    # both are roundoff: half of the TSQR's more, and what the checker's own
    # products leave (a quarter of a unit per column summed)
    assert err[0][0] <= 1.5 * err[1][0] + n * U / 4, err
    assert err[0][1] <= 1.5 * err[1][1] + n * U / 4, err
