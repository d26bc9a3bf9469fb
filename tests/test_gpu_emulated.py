"""Double-precision passes on the tensor cores (fixed-point digits, exact integer
products): parity with the oracle at the edges of their tiles and shapes, scaling,
non-finite data, and the bounded waits.

Tolerance: 1e-12 relative L2 as for every double-precision pass, or twice the oracle's
own rounding floor (the difference of its two summation orders) where that is higher.
Scaling a field by a power of two scales every fixed-point value, sum and rounding
alike: exact equality."""
import os

import numpy as np
import pytest
import torch

from gpu_common import T, absorber_workload, cuda, host, pair, rel_l2, setup_both
from oracle.conservative5d import ConservativeProblem, jacobian
from oracle.transport import Grid as OGrid, Problem as OProblem

pytestmark = pytest.mark.gpu

# (Nr, Ntheta, Nphi, NTheta, NPhi): one to three K cores on each axis, odd theta, ragged
# eight-block and four-column tiles, partial 128-row tiles, radial lines of one and two
# output groups with and without the leftover node, and lengths with K padding
SHAPES = [(3, 2, 2, 2, 2), (5, 3, 2, 6, 4), (9, 5, 4, 8, 6), (16, 4, 6, 10, 8), (17, 8, 8, 8, 8),
          (18, 7, 10, 14, 12), (25, 9, 16, 16, 10), (33, 6, 4, 24, 16), (32, 17, 2, 4, 20),
          (10, 16, 16, 16, 16), (7, 24, 16, 2, 24), (6, 16, 24, 24, 4), (12, 2, 32, 12, 32)]
# four-wide tiles, with two digit copies and with one (ragged blocks and columns, odd
# lengths of the DFS axis, one and two DFS tiles); streamed radial matrices
SHAPES += [(3, 24, 24, 6, 10), (3, 31, 32, 4, 6), (3, 32, 32, 4, 8), (5, 3, 2, 32, 32),
           (5, 3, 2, 30, 32), (4, 3, 4, 24, 24), (3, 25, 28, 26, 24), (65, 3, 4, 6, 10),
           (81, 2, 4, 12, 16), (72, 3, 2, 8, 12)]


def _rhs(gg, F):
    K = torch.full_like(F, float("nan"))
    T().ts_rhs(gg.handle, F, K)
    T().ts_sync_status(gg.handle)
    return K


@pytest.mark.parametrize("form", ["iso", "linear", "thomson"])
@pytest.mark.parametrize("n", SHAPES, ids=str)
def test_rhs_and_step_match_the_oracle(n, form):
    if form != "iso" and min(n[3], n[4]) < 4:
        pytest.skip("the anisotropic kernels need more directions")
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims, G=3)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    kw = {}
    if form == "linear":
        gg.set_scattering_anisotropy(-0.3)
        kw = dict(scatter_b=-0.3)
    elif form == "thomson":
        gg.set_scattering_quadrupole(0.75)
        kw = dict(scatter_c=0.75)
    gg.set_coeffs(kap, eta, ks, g1, g2)
    op = OProblem(og, kap, eta, ks, g1, g2, **kw)
    ref = op.rhs(F0)
    other = OProblem(OGrid(*dims, groups=3, summation="library"), kap, eta, ks, g1, g2, **kw)
    tol = max(1e-12, 2 * rel_l2(other.rhs(F0), ref))
    assert rel_l2(host(_rhs(gg, cuda(F0))), ref) < tol
    dt = 0.05 / (n[0] ** 2 + 4 * n[1] * n[2] + n[3] * n[4] * n[1])
    F = cuda(F0)
    gg.step(F, dt, 2)
    T().ts_sync_status(gg.handle)
    assert rel_l2(host(F), op.run(F0, dt, 2)) < 1e-12


@pytest.mark.parametrize("n", [SHAPES[3], SHAPES[5], SHAPES[9]], ids=str)
def test_conservative_rhs_matches_the_oracle(n):
    dims = (0.2, 1.0) + n
    og, _ = pair(*dims, G=2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    J, h = jacobian(og), og.NT // 2
    X0 = np.ascontiguousarray(J * F0)
    c1, c2 = g1 * J[:, 0, :, :, :h], g2 * J[:, -1, :, :, h:]
    gc = T().Grid(*dims, groups=2, form=T().TS_FORM_CONSERVATIVE)
    gc.set_coeffs(kap, eta, ks, c1, c2)
    gc.set_scattering_quadrupole(0.75)
    op = ConservativeProblem(og, kap, eta, ks, c1, c2, scatter_c=0.75)
    assert rel_l2(host(_rhs(gc, cuda(X0))), op.rhs(X0)) < 1e-12


@pytest.mark.parametrize("power", [-400, 300])
def test_powers_of_two_scale_exactly(power):
    dims = (0.2, 1.0, 17, 6, 8, 16, 16)
    og, gg = pair(*dims, G=1)
    kap, _, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, None, ks)
    F = cuda(F0)
    assert torch.equal(_rhs(gg, F) * 2.0 ** power, _rhs(gg, F * 2.0 ** power))


def test_zero_and_tiny_fields():
    dims = (0.2, 1.0, 17, 6, 8, 16, 16)
    og, gg = pair(*dims, G=1)
    kap, _, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, None, ks)
    for z in (0.0, -0.0):
        assert torch.all(_rhs(gg, torch.full(gg.shape, z, dtype=torch.float64, device="cuda")) == 0)
    K = _rhs(gg, cuda(F0) * 2.0 ** -1040)          # subnormal: lost at most, never garbage
    assert torch.all(torch.isfinite(K)) and float(K.abs().max()) < 1e-290


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_a_non_finite_point_spoils_its_lines_and_not_other_groups(bad):
    dims = (0.2, 1.0, 17, 6, 8, 16, 16)
    og, gg = pair(*dims, G=2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    gg.set_coeffs(kap, eta, ks, g1, g2)
    F = cuda(F0)
    good = _rhs(gg, F)
    F[1, 5, 2, 3, 4, 6] = bad
    K = _rhs(gg, F)
    assert torch.equal(K[0], good[0])
    assert not torch.any(torch.isfinite(K[1, 5, 2, 3]))              # its angular block
    assert not torch.any(torch.isfinite(K[1, :, 2, 3, 4, 6]))        # its radial line
    assert not torch.any(torch.isfinite(K[1, 5, :, 3, 4, 6]))        # and its theta line


def test_wide_range_between_blocks_keeps_each_blocks_precision():
    """Blocks 2^-40 below their neighbours: fixed point is relative to each block, so
    the angular terms keep full precision there (no radial or plane coupling: F depends
    on the direction alone within a block and the streaming of the others is compared
    on the large blocks only)."""
    dims = (0.2, 1.0, 9, 4, 8, 16, 16)
    og, gg = pair(*dims, G=1)
    kap, _, ks, F0, _, _ = absorber_workload(og)
    scale = 2.0 ** (-40 * (np.arange(og.Np) % 2))[None, None, None, :, None, None]
    F0 = F0 * scale
    gg.set_coeffs(kap, None, ks)
    os.environ["TS_GENERIC_PASSES"] = "1"
    try:
        plain = T().Grid(*dims, groups=1)
    finally:
        del os.environ["TS_GENERIC_PASSES"]
    plain.set_coeffs(kap, None, ks)
    F = cuda(F0)
    assert rel_l2(host(_rhs(gg, F)), host(_rhs(plain, F))) < 1e-13


def test_a_wait_that_runs_out_is_reported_and_the_grid_recovers():
    ts = T()
    dims = (0.2, 1.0, 17, 8, 8, 16, 16)
    og, gg = pair(*dims, G=2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    op = setup_both(og, gg, kap, eta, ks, g1, g2)
    ts.ts_set_wait_limit(gg.handle, -1)
    gg.step(cuda(F0), 1e-4, 1)
    with pytest.raises(ts.TSError) as e:
        ts.ts_sync_status(gg.handle)
    assert e.value.status == ts.TS_ERR_TIMEOUT
    ts.ts_sync_status(gg.handle)
    ts.ts_set_wait_limit(gg.handle, 0)
    assert rel_l2(host(_rhs(gg, cuda(F0))), op.rhs(F0)) < 1e-12


@pytest.mark.parametrize("form", ["iso", "linear", "thomson"])
@pytest.mark.parametrize("n", SHAPES[2:], ids=str)
def test_adjoint_step_matches_the_oracle(n, form):
    if form != "iso" and min(n[3], n[4]) < 4:
        pytest.skip("the anisotropic kernels need more directions")
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims, G=2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    kw = {}
    if form == "linear":
        gg.set_scattering_anisotropy(-0.3)
        kw = dict(scatter_b=-0.3)
    elif form == "thomson":
        gg.set_scattering_quadrupole(0.75)
        kw = dict(scatter_c=0.75)
    gg.set_coeffs(kap, eta, ks, g1, g2)
    op = OProblem(og, kap, eta, ks, g1, g2, **kw)
    dt = 0.05 / (n[0] ** 2 + 4 * n[1] * n[2] + n[3] * n[4] * n[1])
    lam0 = np.random.default_rng(5).standard_normal(og.shape)
    lam = cuda(lam0)
    gk = torch.zeros(gg.coef_shape, dtype=torch.float64, device="cuda")
    ge = torch.zeros_like(gk)
    gg.adjoint_step(cuda(F0), lam, gk, ge, dt)
    T().ts_sync_status(gg.handle)
    lo, gko, geo = op.adjoint_step(F0, lam0, dt)
    for a, b in ((lam, lo), (gk, gko), (ge, geo)):
        assert rel_l2(host(a), b) < 1e-12


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_captured_step_equals_the_plain_one(precision):
    """Passes start early outside a capture and are serialised within one."""
    og, gg, dtype = None, None, torch.float64
    if precision == "f64":
        og, gg = pair(0.2, 1.0, 17, 8, 8, 8, 8, G=2)
    else:
        dtype = torch.float32
        og = OGrid(0.2, 1.0, 17, 8, 8, 8, 8, groups=2)
        gg = T().Grid(0.2, 1.0, 17, 8, 8, 8, 8, groups=2, precision=T().TS_FP32)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    gg.set_coeffs(kap, eta, ks, g1, g2)
    plain, captured = cuda(F0).to(dtype), cuda(F0).to(dtype)
    gg.step(plain, 1e-4, 3)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gg.step(captured, 1e-4, 3)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(plain, captured)
