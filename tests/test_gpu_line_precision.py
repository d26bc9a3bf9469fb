"""Double precision on faint lines beside bright ones: every point of a right-hand side is as
exact as its own lines allow, whatever else its tile, block or field holds.

The measure: the error against extended precision in units of 2^-53 N, N the bound of the
point's terms from its own lines (extended.py). A contraction is off by at most 2 K 2^-57 of
row sum x largest value (digit products of order 8 and above, K <= 66 elements; the cut of the
data is 2^-61), 8 units for the largest K here; its coefficients and the sum of the three
passes take about a dozen roundings, which the terms share. Bar: 16 units. Lines cut relative
to a brighter neighbour's scale are off by 1e2 to 1e17 units."""
import os

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
