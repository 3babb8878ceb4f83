"""The FP64 stencil passes at the tile counts where they change between 8 x 8 and
32 x 16-cell tiles (on 152 SMs, large ones from 92 tiles on, small ones again
from 153, large ones from 183): channels with the same cells, one some columns
longer, must give the same bits wherever their inputs agree."""
import numpy as np
import pytest
import torch

from test_tile_sizes_gpu import HX, HY, dn  # noqa: F401

pytestmark = pytest.mark.gpu
NYC, K = 32, 2   # 8 rows of tiles; a tile is 8 coarse columns wide


@pytest.mark.parametrize("tiles", [(88, 96), (152, 160), (176, 184)])
def test_same_bits(dn, tiles):  # noqa: F811
    rng = np.random.default_rng(sum(tiles))
    wide, same = tiles[1], tiles[0] - 16
    solid = np.zeros((NYC, wide), dtype=bool)
    solid[12:18, 20:26] = solid[13:15, 30] = solid[0:3, 60] = True
    xf = rng.standard_normal((3, 4 * NYC + 1, 4 * wide + 1))
    bf = rng.standard_normal((2, 4 * NYC + 1, 4 * wide + 1))
    dp = rng.standard_normal((NYC, wide, 50))
    got = []
    for nxc in tiles:
        sol = solid[:, :nxc]
        mesh = dn.Mesh(dn.make_desc(nxc, NYC, K, 1, precision="f64", solid=sol, lx=nxc * HX, ly=NYC * HY))
        I = mesh.info
        assert (-(-I.nxf // 32)) * (-(-I.nyf // 16)) == nxc
        cut = lambda a: np.ascontiguousarray(a[:, :, :I.nxf + 1]).reshape(a.shape[0], -1)   # noqa: E731
        nodes = lambda t: t.view(-1, I.nyf + 1, I.pitch)[:, :, :4 * same].clone()           # noqa: E731
        x, b = mesh.pack(cut(xf)), mesh.pack(cut(bf))
        d = torch.as_tensor(dp[:, :nxc][~sol]).cuda().contiguous()
        keep = torch.as_tensor((np.broadcast_to(np.arange(nxc), sol.shape) < same)[~sol])
        rf, X, v, r = mesh.fine(3), mesh.features(), mesh.fine(2), mesh.fine(2)
        dn.dnnmg_patch_features(mesh, x, b, X, rf=rf)
        dn.dnnmg_scatter_avg(mesh, d, x, v)
        dn.dnnmg_rhs(mesh, x[:2].contiguous(), r)
        got.append([nodes(rf), X.cpu()[keep], nodes(v), nodes(r)])
    for a, c in zip(*got):
        assert a.shape == c.shape and torch.equal(a, c)
