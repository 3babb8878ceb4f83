"""The fused training window with two 64-column chunks of features, at the
edges of its range: one and 64 columns in the second chunk, ragged rows, more
tiles than CTAs, arrays that do not start on 16 bytes; and the first size past
it, which one kernel per product takes."""

import pytest

import test_train_window_gpu as window
from test_train_window_gpu import dn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,P,n_in,ldx,H,n_out,shift", [
    (2, 1, 65, 65, 32, 1, False), (3, 129, 99, 112, 64, 50, False), (2, 257, 128, 128, 64, 64, True),
    (4, 300, 99, 99, 32, 50, False), (1, 20000, 99, 112, 64, 50, False), (2, 40, 129, 130, 32, 18, False)])
@pytest.mark.parametrize("state", [True, False])
@pytest.mark.parametrize("prec", ["bf16", "f32"])
def test_two_chunks_match_oracle(dn, T, P, n_in, ldx, H, n_out, shift, state, prec):  # noqa: F811
    window.test_window_matches_oracle(dn, T, P, n_in, ldx, H, n_out, shift, state, prec)
