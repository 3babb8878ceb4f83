"""The loss kernel at the edges of its blocks of 4096 values, for arrays that do
and do not start on 16 bytes, and for values whose squares leave the FP32 range.

Squares are FP32, sums FP64; 16 squares are added as an FP32 sum and its error,
which is off by at most 16 * 16 * 2^-48 of them."""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def shifted(a, k):
    t = torch.empty(a.size + k, device="cuda")[k:]
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("n", [1, 255, 4095, 4096, 4097, 512 * 4096 + 4095, 513 * 4096])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("grad", [True, False])
def test_loss_and_gradient(dn, n, shift, grad):
    rng = np.random.default_rng(n)
    D, Y = (rng.standard_normal(n).astype(np.float32) * 10.0 ** rng.uniform(-3, 3, n).astype(np.float32) for _ in range(2))
    P = 3
    g = shifted(np.full(n, np.nan, np.float32), shift) if grad else None
    L = dn.dnnmg_l2_loss(shifted(D, shift), shifted(Y, shift), P, g)
    e = D - Y
    assert L.item() == pytest.approx(math.fsum((e * e).astype(np.float64)) / P, rel=TOL)
    if grad:
        assert np.array_equal(g.cpu().numpy(), e * np.float32(2.0 / P))


@pytest.mark.parametrize("shift", [0, 1])
def test_sums_beyond_fp32_and_non_finite(dn, shift):
    D, Y = np.full(8192, 1.5e19, np.float32), np.zeros(8192, np.float32)
    L = dn.dnnmg_l2_loss(shifted(D, shift), shifted(Y, shift), 1)
    assert L.item() == pytest.approx(8192 * float(np.float32(1.5e19) * np.float32(1.5e19)), rel=TOL)
    for v in (np.inf, 1e30, np.nan):
        D[5000] = v
        L = dn.dnnmg_l2_loss(shifted(D, shift), shifted(Y, shift), 1).item()
        assert math.isnan(L) if v != v else L == math.inf
