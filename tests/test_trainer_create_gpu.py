"""A trainer made in a precision is the trainer switched to it: the same bits and
memory, and the same refusals."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,H,n_out", [(51, 64, 18), (99, 32, 50), (40, 48, 18)])   # (the last: one kernel per product)
@pytest.mark.parametrize("precision", ["f32", "bf16"])
def test_created_as_switched(n_in, H, n_out, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    T, P = 2, 200
    g = torch.Generator(device="cuda").manual_seed(0)
    r = lambda *s: 0.1 * torch.randn(*s, device="cuda", generator=g)   # noqa: E731
    X, h0, W, dD = r(T, P, n_in), r(P, H), [r(3 * H, n_in), r(3 * H, H), r(n_out, H)], r(T, P, n_out)

    def grads(tr):
        D, gs = torch.empty(T, P, n_out, device="cuda"), [torch.empty_like(w) for w in W]
        tr.forward(X, h0, *W, D)
        tr.backward(dD, X, W[1], W[2], *gs)
        return [D, tr.state().clone(), *gs]

    switched = dnnmg.Trainer(n_in, n_in, H, n_out, T, P)
    dnnmg._check(dnnmg.lib().dnnmg_trainer_set_precision(switched.handle, dnnmg.PRECISIONS[precision]))
    for a, b in zip(grads(dnnmg.Trainer(n_in, n_in, H, n_out, T, P, precision=precision)), grads(switched)):
        assert torch.equal(a, b)


def test_other_precisions_are_refused():
    from paper_2008_11520_gb300 import dnnmg
    h = ctypes.c_void_p()
    assert dnnmg.lib().dnnmg_trainer_create_precision(8, 8, 32, 4, 1, 1, dnnmg.PRECISIONS["f64"], ctypes.byref(h)) != 0
    assert not h.value
