"""Double-precision tensor-core passes on axes of 33 to 64 nodes, where a plan exists: matrices
wider than 256 accumulator columns, several 128-row tiles of a contraction, four-wide tiles
with one and two copies of the digits, and Fourier axes of 36 to 64 nodes. Each pair as (theta,
phi) and, where its first is even, as (Theta, Phi); forward, conservative and adjoint.

Tolerance: as in test_gpu_emulated.py, 1e-12 relative L2 or twice the oracle's own rounding
floor."""
import numpy as np
import pytest
import torch

from gpu_common import T, absorber_workload, cuda, host, pair, rel_l2
from oracle.conservative5d import ConservativeProblem, jacobian
from oracle.transport import Grid as OGrid, Problem as OProblem

pytestmark = pytest.mark.gpu

PAIRS = [(24, 40), (40, 12), (48, 4), (9, 60), (41, 8), (8, 64), (3, 64), (12, 48), (64, 2),
         (33, 12), (52, 8), (10, 44), (2, 64), (20, 36), (16, 64), (36, 24)]


def _sizes(pair_, where):
    a, b = pair_
    if where == "plane":
        return (5, a, b, 4, 6)
    if a % 2:
        pytest.skip("Theta needs an even number of nodes")
    return (5, 3, 4, a, b)


def _kernel(gg, form):
    if form == "linear":
        gg.set_scattering_anisotropy(-0.3)
        return dict(scatter_b=-0.3)
    if form == "thomson":
        gg.set_scattering_quadrupole(0.75)
        return dict(scatter_c=0.75)
    return {}


def _forms(where, n):
    return ["iso"] if where == "plane" or min(n[3], n[4]) < 4 else ["iso", "linear", "thomson"]


@pytest.mark.parametrize("where", ["plane", "angular"])
@pytest.mark.parametrize("axes", PAIRS, ids=str)
def test_forward(axes, where):
    n = _sizes(axes, where)
    dims = (0.2, 1.0) + n
    for form in _forms(where, n):
        og, gg = pair(*dims, G=2)
        kap, eta, ks, F0, g1, g2 = absorber_workload(og)
        kw = _kernel(gg, form)
        gg.set_coeffs(kap, eta, ks, g1, g2)
        ref = OProblem(og, kap, eta, ks, g1, g2, **kw).rhs(F0)
        other = OProblem(OGrid(*dims, groups=2, summation="library"), kap, eta, ks, g1, g2, **kw)
        tol = max(1e-12, 2 * rel_l2(other.rhs(F0), ref))
        assert rel_l2(host(gg.rhs(cuda(F0))), ref) < tol
        T().ts_sync_status(gg.handle)


@pytest.mark.parametrize("axes", [p for p in PAIRS if p[0] % 2 == 0], ids=str)
def test_conservative_form(axes):
    dims = (0.2, 1.0) + _sizes(axes, "angular")
    og, _ = pair(*dims, G=2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    J, h = jacobian(og), og.NT // 2
    X0 = np.ascontiguousarray(J * F0)
    c1, c2 = g1 * J[:, 0, :, :, :h], g2 * J[:, -1, :, :, h:]
    gc = T().Grid(*dims, groups=2, form=T().TS_FORM_CONSERVATIVE)
    gc.set_coeffs(kap, eta, ks, c1, c2)
    op = ConservativeProblem(og, kap, eta, ks, c1, c2)
    assert rel_l2(host(gc.rhs(cuda(X0))), op.rhs(X0)) < 1e-12


@pytest.mark.parametrize("where", ["plane", "angular"])
@pytest.mark.parametrize("axes", PAIRS, ids=str)
def test_adjoint(axes, where):
    n = _sizes(axes, where)
    dims = (0.2, 1.0) + n
    dt = 0.05 / (n[0] ** 2 + 4 * n[1] * n[2] + n[3] * n[4] * n[1])
    for form in _forms(where, n):
        og, gg = pair(*dims, G=2)
        kap, eta, ks, F0, g1, g2 = absorber_workload(og)
        kw = _kernel(gg, form)
        gg.set_coeffs(kap, eta, ks, g1, g2)
        op = OProblem(og, kap, eta, ks, g1, g2, **kw)
        lam0 = np.random.default_rng(5).standard_normal(og.shape)
        lam = cuda(lam0)
        gk = torch.zeros(gg.coef_shape, dtype=torch.float64, device="cuda")
        ge = torch.zeros_like(gk)
        gg.adjoint_step(cuda(F0), lam, gk, ge, dt)
        T().ts_sync_status(gg.handle)
        for a, b in zip((lam, gk, ge), op.adjoint_step(F0, lam0, dt)):
            assert rel_l2(host(a), b) < 1e-12
