"""The FP32 right-hand side whose warps walk up the all-fluid tiles (from 304
tiles on 4 rows at a time, from 4096 on 16) against the tile kernel of smaller
meshes: channels with the same cells and of different lengths must give the
same bits wherever their inputs agree, beside walls and obstacles too."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

H, NYC, SAME = 2.0 ** -8, 32, 280   # coarse spacing, coarse rows, coarse columns compared


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def obstacles(kind, wide):
    solid = np.zeros((NYC, wide), dtype=bool)
    if kind == "few":
        solid[12:18, 20:26] = solid[13:15, 90] = solid[0:3, 60] = True
    elif kind == "many":
        solid[np.random.default_rng(3).random(solid.shape) < 0.002] = True
    return solid


@pytest.mark.parametrize("kind", ["none", "few", "many"])
@pytest.mark.parametrize("nxc", [304, 4090, 4096])
def test_same_bits_as_small_meshes(dn, kind, nxc):
    solid = obstacles(kind, 4096)
    v = np.random.default_rng(1).standard_normal((2, 4 * NYC + 1, 4 * 4096 + 1))
    got = []
    for n in (296, nxc):
        mesh = dn.Mesh(dn.make_desc(n, NYC, 2, 1, precision="f32", solid=solid[:, :n], lx=n * H, ly=NYC * H))
        I = mesh.info
        r = mesh.fine(2)
        r.fill_(float("nan"))
        dn.dnnmg_rhs(mesh, mesh.pack(np.ascontiguousarray(v[:, :, :I.nxf + 1]).reshape(2, -1)), r)
        got.append(r.view(2, I.nyf + 1, I.pitch)[:, :, :I.nxf + 1].clone())
        assert torch.isfinite(got[-1]).all()
    assert torch.equal(got[0][:, :, :4 * SAME], got[1][:, :, :4 * SAME])
