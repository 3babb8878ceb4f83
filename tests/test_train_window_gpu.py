"""The fused training window (BF16 products) at the edges of its range: rows
that end inside, at and past a 128-row tile, more tiles than CTAs, the
smallest and largest layers it takes, feature rows and arrays that do not
start on 16 bytes, no initial state, and a precision changed between a
window's forward and backward."""

import numpy as np
import pytest
import torch

from helpers import rel_l2
from oracle import train as otrain
from test_train_gpu import cu, problem

pytestmark = pytest.mark.gpu

TOL = 2e-2   # BF16 operands against FP64


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
def test_window_matches_oracle(dn, T, P, n_in, ldx, H, n_out, shift, state):
    (X, h0, Y), W = problem(T, P, n_in, ldx, H, n_out, seed=T + P)
    h0 = h0 if state else np.zeros_like(h0)
    wrap = off_by_one if shift else (lambda a: a)
    Xg, Wg = wrap(cu(X)), [wrap(cu(w)) for w in W]
    tr = dn.Trainer(n_in, ldx, H, n_out, T, P, precision="bf16")
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
    assert rel_l2(D.cpu().numpy(), Do) <= TOL
    assert rel_l2(tr.state().cpu().numpy(), cache["hs"][-1]) <= TOL
    for a, b, name in zip(g + [dh0], go, ("Wx", "Uh", "Wfc", "h0")):
        assert rel_l2(a.cpu().numpy(), b) <= TOL, name


@pytest.mark.parametrize("first,then", [("bf16", "f32"), ("f32", "bf16")])
def test_precision_changed_between_forward_and_backward(dn, first, then):
    # the backward reads what the other precision's forward saved
    T, P, n_in, ldx, H, n_out = 3, 150, 51, 64, 32, 18
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
        assert rel_l2(a.cpu().numpy(), b) <= TOL, name
