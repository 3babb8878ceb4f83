"""The fused training window at the edges of its range: rows
that end inside, at and past a 128-row tile, more tiles than CTAs, the
smallest and largest layers it takes, feature rows and arrays that do not
start on 16 bytes, no initial state, infinite features, and a precision
changed between a window's forward and backward."""

import numpy as np
import pytest
import torch

from helpers import rel_l2
from oracle import train as otrain
from test_train_gpu import cu, problem

pytestmark = pytest.mark.gpu

TOL = {"bf16": 2e-2, "f32": 1e-5}   # BF16 operands, FP32 products against FP64


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def off_by_one(a):
    """The same values in an array that starts 4 bytes past a 16-byte boundary."""
    t = torch.empty(a.numel() + 1, dtype=a.dtype, device=a.device)
    t[1:] = a.reshape(-1)
    return t[1:].view(a.shape)


@pytest.mark.parametrize("T,P,n_in,ldx,H,n_out,shift", [
    (1, 1, 1, 1, 32, 1, False), (2, 127, 33, 33, 64, 17, False), (2, 128, 64, 80, 32, 64, False),
    (3, 129, 64, 64, 64, 64, True), (2, 257, 51, 51, 64, 18, False), (1, 39000, 51, 64, 64, 18, False),
    (5, 700, 50, 52, 32, 18, True)])
@pytest.mark.parametrize("state", [True, False])
@pytest.mark.parametrize("prec", ["bf16", "f32"])
def test_window_matches_oracle(dn, T, P, n_in, ldx, H, n_out, shift, state, prec):
    (X, h0, Y), W = problem(T, P, n_in, ldx, H, n_out, seed=T + P)
    h0 = h0 if state else np.zeros_like(h0)
    tol = TOL[prec]
    wrap = off_by_one if shift else (lambda a: a)
    Xg, Wg = wrap(cu(X)), [wrap(cu(w)) for w in W]
    tr = dn.Trainer(n_in, ldx, H, n_out, T, P, precision=prec)
    D = wrap(torch.zeros(T, P, n_out, device="cuda"))
    tr.forward(Xg, wrap(cu(h0)) if state else None, *Wg, D)
    Do, cache = otrain.seq_forward(X[:, :, :n_in], h0, *W)
    dD = otrain.loss_grad_D(Do, Y)
    g = [torch.full_like(w, float("nan")) for w in Wg]
    dh0 = wrap(torch.zeros(P, H, device="cuda"))
    tr.backward(wrap(cu(dD)), Xg, Wg[1], Wg[2], *g, dh0=dh0)
    go = otrain.seq_backward(dD, cache, *W)
    torch.cuda.synchronize()
    assert tr.status() == 0
    assert rel_l2(D.cpu().numpy(), Do) <= tol
    assert rel_l2(tr.state().cpu().numpy(), cache["hs"][-1]) <= tol
    for a, b, name in zip(g + [dh0], go, ("Wx", "Uh", "Wfc", "h0")):
        assert rel_l2(a.cpu().numpy(), b) <= tol, name


@pytest.mark.parametrize("first,then", [("bf16", "f32"), ("f32", "bf16")])
def test_precision_changed_between_forward_and_backward(dn, first, then):
    # the backward reads what the other precision's forward saved
    T, P, n_in, ldx, H, n_out = 3, 150, 51, 64, 32, 18
    tol = TOL["bf16"]
    (X, h0, Y), W = problem(T, P, n_in, ldx, H, n_out, seed=2)
    Xg, Wg = cu(X), [cu(w) for w in W]
    tr = dn.Trainer(n_in, ldx, H, n_out, T, P)
    mode = lambda p: dn._check(dn.lib().dnnmg_trainer_set_precision(tr.handle, dn.PRECISIONS[p]))   # noqa: E731
    D = torch.empty(T, P, n_out, device="cuda")
    mode(first)
    tr.forward(Xg, cu(h0), *Wg, D)
    mode(then)
    Do, cache = otrain.seq_forward(X[:, :, :n_in], h0, *W)
    dD = otrain.loss_grad_D(Do, Y)
    g = [torch.empty_like(w) for w in Wg]
    tr.backward(cu(dD), Xg, Wg[1], Wg[2], *g)
    go = otrain.seq_backward(dD, cache, *W)
    torch.cuda.synchronize()
    for a, b, name in zip(g, go, ("Wx", "Uh", "Wfc")):
        assert rel_l2(a.cpu().numpy(), b) <= tol, name


def test_infinite_feature_saturates_the_gates(dn):
    # FP32 operands are clamped to the largest BF16 number before they are split
    T, P, n_in, ldx, H, n_out = 2, 5, 51, 64, 32, 18
    (X, h0, Y), W = problem(T, P, n_in, ldx, H, n_out, seed=4)
    X[0, 2, 7], X[1, 3, 9] = np.inf, -np.inf
    tr = dn.Trainer(n_in, ldx, H, n_out, T, P)
    D = torch.empty(T, P, n_out, device="cuda")
    tr.forward(cu(X), cu(h0), *[cu(w) for w in W], D)
    with np.errstate(over="ignore"):
        Do, _ = otrain.seq_forward(X[:, :, :n_in], h0, *W)
    assert np.isfinite(Do).all()
    assert rel_l2(D.cpu().numpy(), Do) <= TOL["f32"]
