"""Training windows with operands that are infinite, not numbers, or near the
ends of the FP32 range: outputs, state and gradients have the infinities, NaNs
and values that FP32 products give, and in BF16 those of rounded operands."""

import pytest
import torch

from test_train_gpu import problem

pytestmark = pytest.mark.gpu

TOL = {"bf16": 2e-2, "f32": 1e-5}   # as everywhere, on the finite values


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def reference(X, h0, Wx, Uh, Wfc, dD, bf16):
    """Outputs, states and gradients in FP32 on the CPU, one product at a time
    (operands rounded to BF16 if bf16)."""
    r = (lambda a: a.to(torch.bfloat16).float()) if bf16 else (lambda a: a)
    mm = lambda a, b: r(a) @ r(b)   # noqa: E731
    T, H = X.shape[0], Uh.shape[1]
    z, q, c, hs, D = [], [], [], [h0], []
    for s in range(T):
        g, u = mm(X[s], Wx.T), mm(hs[s], Uh[:2 * H].T)
        z.append(torch.sigmoid(g[:, :H] + u[:, :H]))
        q.append(torch.sigmoid(g[:, H:2 * H] + u[:, H:]))
        c.append(torch.tanh(g[:, 2 * H:] + mm(q[s] * hs[s], Uh[2 * H:].T)))
        hs.append(z[s] * hs[s] + (1 - z[s]) * c[s])
        D.append(mm(hs[s + 1], Wfc.T))
    gWx, gUh, gWfc, carry = 0.0, 0.0, 0.0, torch.zeros_like(h0)
    for s in reversed(range(T)):
        dh = mm(dD[s], Wfc) + carry
        dc, dz = dh * (1 - z[s]), dh * (hs[s] - c[s])
        az, ac = dz * z[s] * (1 - z[s]), dc * (1 - c[s] * c[s])
        drh = mm(ac, Uh[2 * H:])
        ar = drh * hs[s] * q[s] * (1 - q[s])
        carry = dh * z[s] + drh * q[s] + mm(torch.cat([az, ar], 1), Uh[:2 * H])
        gWx = gWx + mm(torch.cat([az, ar, ac], 1).T, X[s])
        gUh = gUh + torch.cat([mm(torch.cat([az, ar], 1).T, hs[s]), mm(ac.T, q[s] * hs[s])])
        gWfc = gWfc + mm(dD[s].T, hs[s + 1])
    return torch.stack(D), hs[-1], gWx, gUh, gWfc, carry


def run(dn, prec, X, h0, Wx, Uh, Wfc, dD):
    T, P, n_in = X.shape
    tr = dn.Trainer(n_in, n_in, Uh.shape[1], Wfc.shape[0], T, P, precision=prec)
    W = [w.cuda() for w in (Wx, Uh, Wfc)]
    D = torch.empty(dD.shape, device="cuda")
    g = [torch.empty_like(w) for w in W]
    dh0 = torch.empty(h0.shape, device="cuda")
    tr.forward(X.cuda(), h0.cuda(), *W, D)
    tr.backward(dD.cuda(), X.cuda(), W[1], W[2], *g, dh0=dh0)
    hT = tr.state().clone()
    assert tr.status() == 0
    return [a.cpu() for a in (D, hT, *g, dh0)]


def agree(got, want, tol):
    for name, a, b in zip(("D", "hT", "gWx", "gUh", "gWfc", "dh0"), got, want):
        assert torch.equal(torch.isnan(a), torch.isnan(b)), name
        for inf in (float("inf"), -float("inf")):
            assert torch.equal(a == inf, b == inf), name
        f = torch.isfinite(b)
        x, y = a[f].double(), b[f].double()
        assert float((x - y).norm()) <= tol * float(y.norm()), name


INF, NAN, BIG = float("inf"), float("nan"), 3.4e38   # (BIG is beyond the BF16 range)
SIZES = [(3, 150, 51, 64, 18), (2, 300, 99, 64, 50), (1, 40, 33, 32, 17)]
CASES = [("X", INF), ("X", -INF), ("X", NAN), ("X", BIG), ("X", 1e25), ("h0", INF), ("h0", NAN), ("h0", 1e30),
         ("Wx", INF), ("Wx", NAN), ("Wx", BIG), ("Uh", -INF), ("Wfc", INF), ("Wfc", NAN), ("Wfc", 1e30),
         ("dD", INF), ("dD", -INF), ("dD", NAN), ("dD", 1e36)]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("where,value", CASES)
def test_f32_range(dn, where, value, size):
    check_range(dn, "f32", where, value, size)


def check_range(dn, prec, where, value, size):
    T, P, n_in, H, n_out = size
    (X, h0, Y), W = problem(T, P, n_in, n_in, H, n_out, seed=5)
    t = {k: torch.tensor(a, dtype=torch.float32) for k, a in zip(("X", "h0", "Wx", "Uh", "Wfc"), (X, h0, *W))}
    t["dD"] = torch.randn(T, P, n_out, generator=torch.Generator().manual_seed(1))
    a = t[where].reshape(-1, t[where].shape[-1])
    a[a.shape[0] - 2, 3] = value
    if value in (INF, -INF):
        a[a.shape[0] // 2, 1] = -value
    agree(run(dn, prec, **t), reference(**t, bf16=prec == "bf16"), TOL[prec])


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("where,value", CASES)
def test_bf16_range(dn, where, value, size):
    # (sizes whose last tile has rows past the last patch)
    check_range(dn, "bf16", where, value, size)


@pytest.mark.parametrize("scale", [1e-30, 1e-33])
@pytest.mark.parametrize("size", SIZES)
def test_small_gradients_keep_their_digits(dn, size, scale):
    """The gradients are linear in dD also where the parts of its values are tiny."""
    T, P, n_in, H, n_out = size
    (X, h0, Y), W = problem(T, P, n_in, n_in, H, n_out, seed=6)
    t = {k: torch.tensor(a, dtype=torch.float32) for k, a in zip(("X", "h0", "Wx", "Uh", "Wfc"), (X, h0, *W))}
    t["dD"] = torch.randn(T, P, n_out, generator=torch.Generator().manual_seed(2)) * scale
    agree(run(dn, "f32", **t), reference(**t, bf16=False), TOL["f32"])


def test_state_of_the_window_before_as_h0(dn):
    """h0 may be the trainer's own state, which the window overwrites."""
    T, P, n_in, H, n_out = 2, 140, 51, 64, 18
    (X, h0, Y), W = problem(T, P, n_in, n_in, H, n_out, seed=7)
    t = {k: torch.tensor(a, dtype=torch.float32) for k, a in zip(("X", "h0", "Wx", "Uh", "Wfc"), (X, h0, *W))}
    t["X"][0, 3, 5] = INF
    tr = dn.Trainer(n_in, n_in, H, n_out, T, P)
    Xg, Wg = t["X"].cuda(), [t[k].cuda() for k in ("Wx", "Uh", "Wfc")]
    D = torch.empty(T, P, n_out, device="cuda")
    tr.forward(torch.nan_to_num(Xg, posinf=1.0), t["h0"].cuda(), *Wg, D)
    h1 = tr.state().cpu()
    tr.forward(Xg, tr.state(), *Wg, D)
    dD = torch.zeros(T, P, n_out)
    want = reference(t["X"], h1, t["Wx"], t["Uh"], t["Wfc"], dD, False)
    agree([D.cpu(), tr.state().cpu()], want, TOL["f32"])
