"""The loss of one thread's 16 values (four float4, 1024 values apart) is the sum
of their FP32 squares to FP64 rounding: three FP64 additions."""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(40))
def test_loss_keeps_fp64_digits(seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    r = np.random.default_rng(seed)
    t = int(r.integers(256))
    D = np.zeros(4096, np.float32)
    D[(4 * (t + 256 * np.arange(4))[:, None] + np.arange(4)).ravel()] = r.standard_normal(16) * 10.0 ** r.uniform(-2, 2, 16)
    L = dnnmg.dnnmg_l2_loss(torch.from_numpy(D).cuda(), torch.zeros(4096, device="cuda"), 1).item()
    assert L == pytest.approx(math.fsum((D * D).astype(np.float64)), rel=4 * 2.0 ** -53)
