"""An update whose window kernels gave up a wait must not pass for a good one."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "bf16"])
def test_update_reports_a_wait_that_ran_out(precision, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg, train
    T, P, n_in, ldx, H, n_out = 2, 40, 51, 64, 32, 18
    tn = train.PatchNetTrainer(n_in, ldx, H, n_out, T, P, precision=precision)
    X, Y = torch.randn(T, P, ldx, device="cuda"), torch.randn(T, P, n_out, device="cuda")
    loss, _ = tn.train_window(X, Y)
    assert loss > 0
    monkeypatch.setattr(tn.trainer, "status", lambda reset=False: 1)   # as if one had
    with pytest.raises(dnnmg.DnnmgError, match="update 2: .*status is 1"):
        tn.train_window(X, Y)
