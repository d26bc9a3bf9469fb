"""The rounding of the implicit collision step. With dt = 2^-100 the streaming step leaves the
field as it is, and with kappa = x / dt, no emission and no scattering the collision step is
F / (1 + dt kappa): in double the quotient, in the mixed precision the float nearest to the
product with the reciprocal, subnormal floats among them."""
import numpy as np
import pytest
import torch

from gpu_common import T, cuda

pytestmark = pytest.mark.gpu

DT = 2.0 ** -100   # a power of two: dt kappa is exact


def _run(precision, F, kappa):
    ts = T()
    n = F.shape[1:]
    gg = ts.Grid(0.2, 1.0, *n, groups=F.shape[0], precision=precision,
                 scheme=ts.TS_RK4_SPLIT_IMPLICIT, bc=ts.TS_BC_NONE)
    gg.set_coeffs(kappa, 0 * kappa, 0 * kappa)
    X = cuda(F, torch.float64 if precision == ts.TS_FP64 else torch.float32)
    gg.step(X, DT, 1)
    ts.ts_sync_status(gg.handle)
    return X.cpu().numpy()


def _case(rng, dtype, scale):
    shape = (2, 5, 4, 6, 8, 12)
    F = (rng.standard_normal(shape) * scale).astype(dtype)
    kappa = np.exp(rng.uniform(-8, 8, size=shape[:4])) / DT
    return F, kappa, (1.0 + DT * kappa)[..., None, None]


@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e30])
def test_double_takes_the_quotient(scale):
    F, kappa, den = _case(np.random.default_rng(1), np.float64, scale)
    assert np.array_equal(_run(T().TS_FP64, F, kappa), F / den)


@pytest.mark.parametrize("scale", [1.0, 1e-37, 1e-39, 1e-43, 1e33])
def test_float_is_rounded_to_nearest(scale):
    F, kappa, den = _case(np.random.default_rng(2), np.float32, scale)
    want = (F.astype(np.float64) * (1.0 / den)).astype(np.float32)
    assert np.array_equal(_run(T().TS_FP32_R64, F, kappa), want)


def test_ties_go_to_even():
    """kappa dt = 2^k - 1: the reciprocal is a power of two. Subnormal quotients then lie half
    way between two floats in every second case."""
    F, kappa, _ = _case(np.random.default_rng(3), np.float32, 2.0 ** -124)
    kappa = (2.0 ** np.random.default_rng(4).integers(1, 6, size=kappa.shape) - 1.0) / DT
    den = (1.0 + DT * kappa)[..., None, None]
    assert np.all(np.log2(den) % 1 == 0)
    want = (F.astype(np.float64) * (1.0 / den)).astype(np.float32)
    assert np.array_equal(_run(T().TS_FP32_R64, F, kappa), want)
