"""The split-product radial passes at every number of K steps (8 nodes a step in split TF32,
16 in split bf16, up to 81 nodes), whole steps and padded ones. Bar and field as in
test_gpu_tensorcore.py: 1e-5 relative L2 of a right-hand side with 10 % noise."""
import numpy as np
import pytest
import torch

from gpu_common import T, absorber_workload, cuda, host, pair, rel_l2, setup_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [3, 4])   # TS_TF32X3, TS_BF16X3
@pytest.mark.parametrize("Nr", [3, 8, 16, 24, 25, 40, 41, 48, 56, 64, 72, 73, 80, 81])
def test_rhs_at_every_number_of_steps(Nr, prec):
    dims = (0.2, 1.0, Nr, 3, 4, 8, 12)
    og, gg = pair(*dims, G=2, precision=prec)
    kap, eta, ks, F0, gR1, gR2 = absorber_workload(og)
    op = setup_both(og, gg, kap, eta, ks, gR1, gR2)
    F = F0 + 0.1 * np.random.default_rng(3).standard_normal(og.shape)
    K = host(gg.rhs(cuda(F, torch.float32)))
    T().ts_sync_status(gg.handle)
    assert rel_l2(K, op.rhs(F)) < 1e-5
