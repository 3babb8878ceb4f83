"""FP32 products of the training window on the tensor cores keep FP32's digits:
sums of one representable product are exact, and sums over many terms are
within four accumulations of an ulp (a missing product of the operands' parts
is worth 6e-7 or more on random operands)."""

import pytest
import torch

from test_train_window_range_gpu import dn, reference, run   # noqa: F401

pytestmark = pytest.mark.gpu

LIMIT = 4 * 2.0 ** -23   # 64 terms: four accumulations at full magnitude, each drops less than an ulp


@pytest.mark.parametrize("n_in,H,n_out", [(51, 64, 18), (1, 32, 1), (99, 64, 50), (64, 32, 64)])
@pytest.mark.parametrize("P", [1, 70])
def test_one_product_is_exact(dn, n_in, H, n_out, P):   # noqa: F811
    """z = 1 leaves h = h0: a row of h0 and of dD with one 1 picks entries of W_fc and dD."""
    g = torch.Generator().manual_seed(n_in + P)
    r = lambda *s: torch.randn(*s, generator=g)   # noqa: E731
    X = torch.ones(1, P, n_in)
    Wx = torch.zeros(3 * H, n_in)
    Wx[:H, 0] = 200.0
    Uh, Wfc = 0.1 * r(3 * H, H), r(n_out, H)
    h0, dD = torch.zeros(P, H), torch.zeros(1, P, n_out)
    hcol, ocol = torch.arange(P) % H, torch.arange(P) % n_out
    h0[torch.arange(P), hcol] = 1.0
    dD[0, torch.arange(P), ocol] = 1.0
    D, hT, _, _, _, dh0 = run(dn, "f32", X, h0, Wx, Uh, Wfc, dD)
    assert torch.equal(hT, h0)
    assert torch.equal(D[0], Wfc[:, hcol].T)
    assert torch.equal(dh0, Wfc[ocol])
    # gradient of W_fc: dD's row at the one patch whose state is that column's
    if P <= H:
        dD = r(1, P, n_out)
        gWfc = run(dn, "f32", X, h0, Wx, Uh, Wfc, dD)[4]
        want = torch.zeros(n_out, H)
        want[:, hcol] = dD[0].T
        assert torch.equal(gWfc, want)


@pytest.mark.parametrize("T,P,n_in,H,n_out", [(3, 500, 51, 64, 18), (1, 1, 1, 32, 1), (2, 300, 99, 64, 50),
                                              (2, 200, 16, 32, 17), (1, 5000, 64, 64, 64)])
@pytest.mark.parametrize("positive", [False, True])
def test_error_against_64_bits(dn, T, P, n_in, H, n_out, positive):   # noqa: F811
    g = torch.Generator().manual_seed(T + P)
    sign = torch.abs if positive else (lambda a: a)
    r = lambda *s: sign(torch.randn(*s, generator=g))   # noqa: E731
    scale = 0.02 if positive else 0.1
    t = dict(X=r(T, P, n_in), h0=r(P, H).clamp(-0.5, 0.5), Wx=scale * r(3 * H, n_in), Uh=scale * r(3 * H, H),
             Wfc=scale * r(n_out, H), dD=r(T, P, n_out))
    got = run(dn, "f32", **t)
    want = reference(**{k: a.double() for k, a in t.items()}, bf16=False)
    for name, a, b in zip(("D", "hT", "gWx", "gUh", "gWfc", "dh0"), got, want):
        assert float((a.double() - b).norm()) <= LIMIT * float(b.norm()), name
