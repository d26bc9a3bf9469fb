"""ts_rhs writes the finished rate over the array that holds the angular and plane terms.
Every thread of a radial line needs the inflow node's entry of that array (the Tau rows),
so it has to be read before any thread of the line stores that node.

The derivative that an AB2 start step forms from the same input does not write over what
it reads. With dt = 2^200 (float: 2^60) the step's field is that derivative times dt, bit
for bit, wherever it is not zero: the field itself is below half a unit of the last place.

Double precision is also compared with the oracle: 1e-12 relative L2, or twice the oracle's
own rounding floor (the difference of its two summation orders; 4.5e-12 at 65 nodes, 1.7e-11
at 81). test_gpu_tensorcore.py compares the split products with it.
"""
import pytest
import torch

from gpu_common import T, absorber_workload, cuda, host, pair, rel_l2
from oracle.transport import Grid as OGrid, Problem as OProblem

pytestmark = pytest.mark.gpu


def _equal_to_the_start_step(precision, power, n, calls):
    ts = T()
    dims = (0.2, 1.0) + n
    dtype = torch.float64 if precision == ts.TS_FP64 else torch.float32
    og, rhs = pair(*dims, G=2, precision=precision)
    ab2 = ts.Grid(*dims, groups=2, precision=precision, scheme=ts.TS_AB2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    for g in (rhs, ab2):
        g.set_coeffs(kap, eta, ks, g1, g2)
    F = cuda(F0).to(dtype)
    step = F.clone()
    ab2.step(step, 2.0 ** power, 1)
    K = torch.empty_like(F)
    for _ in range(calls):
        K.fill_(float("nan"))
        ts.ts_rhs(rhs.handle, F, K)
        ts.ts_sync_status(rhs.handle)
        some = K != 0
        assert float(some.double().mean()) > 0.9
        assert torch.equal(K[some] * 2.0 ** power, step[some])
    ref = OProblem(og, kap, eta, ks, g1, g2).rhs(F0)
    other = OProblem(OGrid(*dims, groups=2, summation="library"), kap, eta, ks, g1, g2).rhs(F0)
    return rel_l2(host(K), ref), 2 * rel_l2(other, ref)


# two and four threads a line, one to three output groups, streamed matrices, partial tiles
@pytest.mark.parametrize("n", [(17, 4, 6, 8, 12), (33, 3, 4, 16, 16), (65, 2, 4, 10, 12),
                               (81, 2, 2, 8, 16)], ids=str)
def test_double_precision(n):
    off, floor = _equal_to_the_start_step(T().TS_FP64, 200, n, 20)
    assert off < max(1e-12, floor)


# split TF32 and split bf16: two threads a line
@pytest.mark.parametrize("n", [(17, 4, 6, 8, 16), (33, 3, 4, 16, 16), (41, 2, 4, 8, 24)], ids=str)
@pytest.mark.parametrize("precision", ["TS_TF32X3", "TS_BF16X3"])
def test_split_products(precision, n):
    _equal_to_the_start_step(getattr(T(), precision), 60, n, 20)
