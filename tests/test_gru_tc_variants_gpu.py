"""The tensor-core network runs one or two CTAs an SM, by the number of 128-row
tiles and by what a layer takes of an SM; a row's results have the same bits
either way."""

import pytest
import torch

from paper_2008_11520_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [32, 64])
@pytest.mark.parametrize("n_in,n_out", [(51, 18), (99, 50), (267, 162)])
@pytest.mark.parametrize("off", [-1, 0, 1, 129])
def test_rows_do_not_depend_on_the_variant(H, n_in, n_out, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    P, few = 128 * sms + off, 300
    net = dnnmg.Net(*synth.net_weights(n_in, H, n_out, 3), precision="bf16")
    g = torch.Generator(device="cuda").manual_seed(H + n_in)
    X = torch.randn(P, (n_in + 15) // 16 * 16, device="cuda", generator=g).to(torch.bfloat16)
    h0 = torch.randn(P, H, device="cuda", generator=g).clamp(-0.5, 0.5)
    h, d = h0.clone(), torch.empty(P, n_out, device="cuda")
    dnnmg.dnnmg_gru_step(net, X, h, d, P)
    for rows in (slice(0, few), slice(P - few, P)):
        hs, ds = h0[rows].clone(), torch.empty(few, n_out, device="cuda")
        dnnmg.dnnmg_gru_step(net, X[rows].clone(), hs, ds, few)
        assert torch.equal(hs, h[rows]) and torch.equal(ds, d[rows])
    assert dnnmg.dnnmg_net_status(net) == 0
