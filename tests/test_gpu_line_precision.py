"""Double precision on faint lines beside bright ones: every point of a right-hand side is as
exact as its own lines allow, whatever else its tile, block or field holds.

The measure: the error against extended precision in units of 2^-53 N, N the bound of the
point's terms from its own lines (extended.py). A contraction is off by at most 2 K 2^-57 of
row sum x largest value (digit products of order 8 and above, K <= 66 elements; the cut of the
data is 2^-61), 8 units for the largest K here; its coefficients and the sum of the three
passes take about a dozen roundings, which the terms share. Bar: 16 units. Lines cut relative
to a brighter neighbour's scale are off by 1e2 to 1e17 units."""
import numpy as np
import pytest
import torch

from extended import Extended, W
from gpu_common import T, absorber_workload, cuda, pair

pytestmark = pytest.mark.gpu

BAR = 16.0
SHAPES = [(17, 6, 8, 16, 16), (33, 4, 4, 12, 10), (65, 2, 4, 6, 8), (18, 3, 4, 8, 10)]


def field(kind, og, F0, rng):
    if kind == "beam":              # forward-peaked: directions fall off to e^-80
        mu = np.cos(og.Theta)[None, None, None, None, :, None]
        return F0 * np.exp(-40 * (1 - mu))
    if kind == "attenuated":        # 1e-10 across the shell
        return F0 * np.exp(-30 * (og.r - og.r[0]))[None, :, None, None, None, None]
    if kind == "pencil":            # one direction alone: the moments are far below its value
        F = np.zeros_like(F0)
        F[..., 3, 5] = F0[..., 3, 5]
        return F
    if kind.startswith("points"):   # a few bright points in a field 2^-p below them
        F = F0 * 2.0 ** -int(kind[6:])
        for _ in range(6):
            at = (0,) + tuple(rng.integers(0, n) for n in F0.shape[1:])
            F[at] = F0[at]
        return F
    if kind == "directions":        # every direction of its own magnitude, 2^-60 to 1
        return F0 * 2.0 ** -rng.integers(0, 60, size=(1, 1, 1, 1) + F0.shape[4:])
    if kind == "positions":         # every position
        return F0 * 2.0 ** -rng.integers(0, 60, size=F0.shape[:4] + (1, 1))
    if kind == "one side":          # e^-40 across the sphere
        return F0 * np.exp(-20 * (1 - np.cos(og.theta)))[None, None, :, None, None, None]
    raise ValueError(kind)


def units(got, want, bound):
    assert np.all(np.isfinite(got))
    some = bound > 0
    assert np.all(got[~some] == 0)
    return float((np.abs(got - want)[some] / (bound[some] * W(2) ** -53)).max())


def both(gg, op, F, coeffs, **kernel):
    L, N = op.streaming(F)
    K, M = op.rate(F, *coeffs, **kernel)
    x = cuda(F)
    return (units(gg.liouville(x).cpu().numpy(), L, N), units(gg.rhs(x).cpu().numpy(), K, M))


@pytest.mark.parametrize("kind", ["beam", "attenuated"])
@pytest.mark.parametrize("n", SHAPES, ids=str)
def test_radial_lines(n, kind):
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims)
    kap, eta, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, eta, ks)
    F = field(kind, og, F0, np.random.default_rng(11))
    assert max(both(gg, Extended(*dims), F, (kap, eta, ks))) < BAR


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_non_finite_point_reaches_no_other_radial_line(bad):
    """Of its radial neighbours in a tile, as in the passes on the FP64 units: no plane or
    angular line joins (theta, phi, Theta, Phi) below with the point's."""
    dims = (0.2, 1.0, 33, 5, 6, 16, 16)
    og, gg = pair(*dims)
    _, _, _, F0, _, _ = absorber_workload(og)
    gg.set_coeffs()
    F = cuda(F0)
    good = gg.liouville(F)
    F[0, 7, 1, 2, 3, 5] = bad
    K = gg.liouville(F)
    far = torch.ones(33, dtype=torch.bool)
    far[7] = False
    assert not torch.any(torch.isfinite(K[0, :, 1, 2, 3, 5]))
    same = K[0, far, 1, 2] == good[0, far, 1, 2]          # other nodes of the same (theta, phi)
    same[:, 3, 5] = True
    assert torch.all(same)


@pytest.mark.parametrize("kernel", [{}, {"b": -0.3}, {"c": 0.75}], ids=["iso", "linear", "thomson"])
@pytest.mark.parametrize("n", SHAPES + [(5, 3, 4, 32, 32), (6, 4, 2, 24, 16)], ids=str)
def test_moments_of_a_single_direction(n, kernel):
    """Directions off the bright one's lines hold exact zeros: their rate is the moments."""
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims)
    kap, eta, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, 0 * eta, 8 * ks)
    if "b" in kernel:
        gg.set_scattering_anisotropy(kernel["b"])
    if "c" in kernel:
        gg.set_scattering_quadrupole(kernel["c"])
    F = field("pencil", og, F0, None)
    assert max(both(gg, Extended(*dims), F, (kap, 0 * eta, 8 * ks), **kernel)) < BAR


LINES = ["points4", "points8", "points20", "points40", "points60", "directions", "positions",
         "one side"]
# eight- and four-wide tiles, two copies of the digits and one, odd theta, ragged columns
WIDE = [(17, 6, 8, 16, 16), (9, 16, 16, 8, 8), (33, 4, 4, 12, 10), (5, 7, 10, 14, 12),
        (4, 4, 4, 32, 32), (3, 32, 32, 4, 8), (3, 25, 28, 6, 10), (4, 3, 4, 24, 24)]


@pytest.mark.parametrize("kind", LINES)
@pytest.mark.parametrize("n", WIDE, ids=str)
def test_lines_of_all_axes(n, kind):
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims)
    kap, eta, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, eta, ks)
    F = field(kind, og, F0, np.random.default_rng(11))
    assert max(both(gg, Extended(*dims), F, (kap, eta, ks))) < BAR


@pytest.mark.parametrize("kind", ["points8", "points40", "directions"])
@pytest.mark.parametrize("n", [WIDE[0], WIDE[2], WIDE[4]], ids=str)
def test_lines_of_the_conservative_form(n, kind):
    ts = T()
    dims = (0.2, 1.0) + n
    og, _ = pair(*dims)
    F0 = absorber_workload(og)[3]
    gg = ts.Grid(*dims, form=ts.TS_FORM_CONSERVATIVE)
    gg.set_coeffs()
    F = field(kind, og, F0, np.random.default_rng(11))
    L, N = Extended(*dims, form="cons").streaming(F)
    assert units(gg.liouville(cuda(F)).cpu().numpy(), L, N) < BAR


@pytest.mark.parametrize("kind", LINES)
@pytest.mark.parametrize("n", [WIDE[0], WIDE[1], WIDE[2], WIDE[4], WIDE[5]], ids=str)
def test_lines_of_the_adjoint(n, kind):
    """One AB2 starting step backwards with dt = 2^200: the field itself is below the last
    place, what is left is -L^T times dt."""
    ts = T()
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims, scheme=ts.TS_AB2, bc=ts.TS_BC_NONE)
    F0 = absorber_workload(og)[3]
    gg.set_coeffs()
    F = field(kind, og, F0, np.random.default_rng(11))
    lam, prev = cuda(F), torch.zeros(gg.shape, dtype=torch.float64, device="cuda")
    gk = torch.zeros(gg.coef_shape, dtype=torch.float64, device="cuda")
    ts.ts_adjoint_step_ab2(gg.handle, cuda(F0), lam, prev, gk, torch.zeros_like(gk), 2.0 ** 200, True)
    ts.ts_sync_status(gg.handle)
    L, N = Extended(*dims).streaming_adjoint(F)
    assert units(lam.cpu().numpy() * 2.0 ** -200, -L, N) < BAR


@pytest.mark.parametrize("power", [-700, 600])
def test_far_powers_of_two_scale_exactly(power):
    dims = (0.2, 1.0, 17, 6, 8, 16, 16)
    og, gg = pair(*dims)
    kap, _, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, None, ks)
    F = field("points8", og, F0, np.random.default_rng(3))
    assert torch.equal(gg.rhs(cuda(F)) * 2.0 ** power, gg.rhs(cuda(F * 2.0 ** power)))


@pytest.mark.parametrize("n", [(17, 6, 8, 16, 16), (33, 4, 4, 12, 10), (4, 4, 4, 32, 32)], ids=str)
def test_tiny_blocks_and_lines_keep_their_digits(n):
    """Values near 2^-990 and, on most lines, 2^-8 below (2^-1022 is the smallest normal one).
    Results there are rounded by another rule at ties, so the bar is that of all lines."""
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims)
    kap, _, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, None, ks)
    F = field("points8", og, F0, np.random.default_rng(3)) * 2.0 ** -990
    assert max(both(gg, Extended(*dims), F, (kap, 0 * kap, ks))) < BAR


@pytest.mark.parametrize("bad", [float("nan"), -float("inf")])
@pytest.mark.parametrize("n", [(9, 6, 8, 16, 16), (4, 4, 4, 32, 32), (3, 32, 32, 4, 8)], ids=str)
def test_a_non_finite_point_reaches_its_own_lines(n, bad):
    """As in the passes on the FP64 units: its radial line, its circles over theta and Theta
    (the partner half turned by pi) and its lines over phi and Phi."""
    dims = (0.2, 1.0) + n
    og, gg = pair(*dims)
    F0 = absorber_workload(og)[3]
    gg.set_coeffs()
    _, Nt, Np, NT, NP = n
    i, j, l, k, m = 1, 2, 3, 1, 3
    F = F0.copy()
    F[0, i, j, l, k, m] = bad
    hit = np.zeros(F0.shape[1:], dtype=bool)
    l2, m2 = (l + Np // 2) % Np, (m + NP // 2) % NP
    hit[:, j, l, k, m] = True
    hit[i, :, l, k, m] = hit[i, :, l2, k, m2] = True
    hit[i, j, :, k, m] = True
    hit[i, j, l, :, m] = hit[i, j, l, :, m2] = True
    hit[i, j, l, k, :] = True
    K = gg.liouville(cuda(F)).cpu().numpy()[0]
    assert not np.any(np.isfinite(K[hit]))
    L, N = Extended(*dims).streaming(F0)
    off = np.abs(K - L[0])[~hit] / (N[0][~hit] * W(2) ** -53)
    assert np.all(np.isfinite(K[~hit])) and float(off.max()) < BAR


def test_what_a_block_gives_does_not_depend_on_the_other_groups():
    """Tiles of the angular pass run across groups (21 blocks a group): bit for bit."""
    dims = (0.2, 1.0, 7, 3, 2, 16, 16)
    og, gg = pair(*dims, G=3)
    kap, eta, ks, F0, _, _ = absorber_workload(og)
    gg.set_coeffs(kap, eta, ks)
    rng = np.random.default_rng(11)
    F = cuda(F0)
    good = gg.rhs(F)
    F[1] = cuda(field("points40", og, F0[1:2], rng)[0])
    K = gg.rhs(F)
    assert torch.equal(K[0], good[0]) and torch.equal(K[2], good[2])
