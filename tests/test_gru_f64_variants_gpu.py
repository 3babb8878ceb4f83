"""The FP64 network keeps its weights in shared memory while every CTA has one
tile of two patches, and reads them from L2 beyond that: the same bits row by
row on both sides of the border (1 to 6 CTAs an SM, by the layer)."""

import pytest
import torch

from paper_2008_11520_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,H,n_out", [(51, 16, 18), (51, 32, 18), (282, 16, 162), (51, 64, 18)])
def test_rows_do_not_depend_on_the_variant(n_in, H, n_out):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    net = dnnmg.Net(*synth.net_weights(n_in, H, n_out, 3), precision="f64")
    g = torch.Generator(device="cuda").manual_seed(H)
    most, ldx = 2 * 8 * sms, (n_in + 15) // 16 * 16
    X = torch.randn(most, ldx, device="cuda", generator=g, dtype=torch.float64)
    h0 = torch.rand(most, H, device="cuda", generator=g, dtype=torch.float64) - 0.5

    def run(P):
        h, d = h0[:P].clone(), torch.empty(P, n_out, device="cuda", dtype=torch.float64)
        dnnmg.dnnmg_gru_step(net, X[:P].contiguous(), h, d, P)
        return h, d

    h, d = run(most)
    for per in (1, 2, 3, 6):
        for P in (2 * per * sms - 1, 2 * per * sms, 2 * per * sms + 1):
            hp, dp = run(P)
            assert torch.equal(hp, h[:P]) and torch.equal(dp, d[:P])
