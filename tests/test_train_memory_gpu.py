"""Device memory a trainer of the fused window's shapes holds: four saved
activations (H values a row and step, whole 128-row tiles), in FP32 the three
gates' gradients, and little else."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,n_out", [(51, 18), (99, 50)])
@pytest.mark.parametrize("precision,arrays", [("f32", 7), ("bf16", 4)])
def test_trainer_memory(n_in, n_out, precision, arrays):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    T, P, H = 10, 65536, 64
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    tr = dnnmg.Trainer(n_in, 112, H, n_out, T, P, precision=precision)
    held = before - torch.cuda.mem_get_info()[0]
    tr.close()
    # and h_T, its copy of h_0, dh_0 (3 of T rows), partial gradients (0.04 GB), allocation granularity
    assert held <= (arrays + 0.3) * 4 * H * T * P + (64 << 20)


def test_precision_back_and_forth():
    """BF16 products need no gate gradients in memory; FP32 ones get them back."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    T, P, n_in, H, n_out = 2, 200, 99, 64, 50
    g = torch.Generator(device="cuda").manual_seed(0)
    r = lambda *s: 0.1 * torch.randn(*s, device="cuda", generator=g)   # noqa: E731
    X, h0, W, dD = r(T, P, n_in), r(P, H), [r(3 * H, n_in), r(3 * H, H), r(n_out, H)], r(T, P, n_out)

    def grads(tr):
        D, gs = torch.empty(T, P, n_out, device="cuda"), [torch.empty_like(w) for w in W]
        tr.forward(X, h0, *W, D)
        tr.backward(dD, X, W[1], W[2], *gs)
        return [D, tr.state().clone(), *gs]

    mode = lambda tr, p: dnnmg._check(dnnmg.lib().dnnmg_trainer_set_precision(tr.handle, dnnmg.PRECISIONS[p]))   # noqa: E731
    tr = dnnmg.Trainer(n_in, n_in, H, n_out, T, P)
    first = grads(tr)
    for p in ("bf16", "bf16", "f32", "f32"):
        mode(tr, p)
    for a, b in zip(grads(tr), first):
        assert torch.equal(a, b)
