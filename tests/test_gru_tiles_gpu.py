"""The FP32 / FP64 network's register-tiled kernel at the edges of its tiles
and variants: patch counts around a tile and around the count where the
weights move out of shared memory, states and outputs that are not multiples
of a tile, and shapes left to the one-column kernel."""

import numpy as np
import pytest
import torch

from helpers import TOL, rel_l2
from oracle import gru as ogru

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def step(dn, W, prec, X, h0):
    net = dn.Net(*W, precision=prec)
    P, n_out = X.shape[0], W[2].shape[0]
    h = torch.as_tensor(h0).to(net.real).cuda()
    d = torch.full((P, n_out), float("nan"), dtype=net.real, device="cuda")
    Xg = torch.zeros(P, (X.shape[1] + 15) // 16 * 16, dtype=net.real, device="cuda")
    Xg[:, :X.shape[1]] = torch.as_tensor(X).to(net.real)
    dn.dnnmg_gru_step(net, Xg, h, d, P)
    return h, d


# the last two: H not a multiple of 4, and more inputs than the tiled kernel stages
@pytest.mark.parametrize("n_in,H,n_out", [(99, 64, 50), (51, 32, 18), (1, 4, 1), (27, 20, 7), (30, 6, 5), (300, 64, 18)])
@pytest.mark.parametrize("P", [1, 31, 33, 64])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_matches_oracle(dn, n_in, H, n_out, P, prec):
    rng = np.random.default_rng(P + H)
    W = [rng.normal(0, 0.2, s) for s in ((3 * H, n_in), (3 * H, H), (n_out, H))]
    X, h0 = rng.normal(0, 1, (P, n_in)), rng.uniform(-0.5, 0.5, (P, H))
    if prec == "f32":
        W = [w.astype(np.float32).astype(np.float64) for w in W]
        X, h0 = (a.astype(np.float32).astype(np.float64) for a in (X, h0))
    h, d = step(dn, W, prec, X, h0)
    ho, do = ogru.gru_step(X, h0, *W)
    assert rel_l2(h.double().cpu().numpy(), ho) <= TOL[prec]
    assert rel_l2(d.double().cpu().numpy(), do) <= TOL[prec]


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_rows_do_not_depend_on_the_variant(dn, prec):
    # one tile an SM at most, and more: the same bits row by row
    rng = np.random.default_rng(3)
    n_in, H, n_out = 99, 64, 50
    W = [rng.normal(0, 0.2, s) for s in ((3 * H, n_in), (3 * H, H), (n_out, H))]
    X, h0 = rng.normal(0, 1, (5200, n_in)), rng.uniform(-0.5, 0.5, (5200, H))
    h, d = step(dn, W, prec, X, h0)
    for P in (70, 4830, 4870):
        hp, dp = step(dn, W, prec, X[:P], h0[:P])
        assert torch.equal(hp, h[:P]) and torch.equal(dp, d[:P])
