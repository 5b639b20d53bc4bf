"""Panels at scales whose products of squares leave the FP64 range, though the
squares do not: scaling by a power of two changes no digit of V and T."""

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


def _same(ref, got, s, a):
    (VR, T), (VR2, T2) = ref, got
    assert np.max(np.abs(np.tril(VR2 - VR, -1))) <= 1e-12 and np.max(np.abs(T2 - T)) <= 1e-12
    R, R2 = np.triu(VR[:VR.shape[1]]), np.triu(VR2[:VR.shape[1]]) / s
    assert np.max(np.abs(R2 - R) / np.linalg.norm(a, axis=0)) <= 1e-12


@pytest.mark.parametrize("e", [-460, -370, -300, -260, -245, -230, 230, 245, 260, 400])
@pytest.mark.parametrize("m,n", [(400, 40), (1024, 128)])
def test_scaled_panels(gb, ctx, m, n, e):
    a = workloads.gaussian(m, n, 800 + n)
    ref = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL)[:2]
    _same(ref, _gpu.factor_gpu(ctx, a * 2.0 ** e, gb.GBQR_T_FULL)[:2], 2.0 ** e, a)


@pytest.mark.parametrize("e", [-460, -300, -260, 260, 300])
def test_some_scaled_columns(gb, ctx, e):
    a = workloads.gaussian(600, 64, 810)
    s = np.ones(64)
    s[20:30] = 2.0 ** e
    s[60:] = 2.0 ** e
    ref = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL)[:2]
    _same(ref, _gpu.factor_gpu(ctx, a * s, gb.GBQR_T_FULL)[:2], s[None, :], a)


@pytest.mark.parametrize("e", [-100, 60, 100])
def test_fp32_scales(gb, ctx, e):
    """FP32 squares that leave FP32's range are FP64 numbers here."""
    import torch
    a = workloads.gaussian(700, 48, 820).astype(np.float32)
    out = []
    for s in (1.0, 2.0 ** e):
        A = torch.from_numpy(np.ascontiguousarray((a * np.float32(s)).T)).cuda().T
        T = torch.zeros((48, 48), dtype=torch.float32, device="cuda").T
        ctx.factor(A, T, gb.GBQR_T_FULL)
        assert ctx.sync()[0] == gb.GBQR_OK
        VR = A.cpu().numpy().astype(np.float64)
        out.append((np.tril(VR, -1), np.triu(VR[:48]) / s, T.cpu().numpy().astype(np.float64)))
    for p, q in zip(*out):
        assert np.max(np.abs(p - q)) <= 1e-4
