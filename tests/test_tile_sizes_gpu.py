"""The stencil passes on both sides of the tile count where they change from
8 x 8 to 32 x 16-cell tiles: two channels with the same cells, one some columns
longer (296 and 304 tiles of 32 x 16 cells), must give the same bits wherever
their inputs agree."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

HX, HY, NYC, SAME = 2.0 ** -8, 2.0 ** -8, 32, 280   # coarse spacing, coarse rows, coarse columns compared


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_same_bits_in_both_tile_sizes(dn, prec):
    rng = np.random.default_rng(1)
    wide = 304
    solid = np.zeros((NYC, wide), dtype=bool)
    solid[12:18, 20:26] = solid[13:15, 30] = solid[0:3, 60] = True
    xf = rng.standard_normal((3, 4 * NYC + 1, 4 * wide + 1))
    bf = rng.standard_normal((2, 4 * NYC + 1, 4 * wide + 1))
    xc = rng.standard_normal((3, NYC + 1, wide + 1))
    dp = rng.standard_normal((NYC, wide, 50))
    got = []
    for nxc in (296, wide):
        sol = solid[:, :nxc]
        mesh = dn.Mesh(dn.make_desc(nxc, NYC, 2, 1, precision=prec, solid=sol, lx=nxc * HX, ly=NYC * HY))
        I = mesh.info
        assert (-(-I.nxf // 32)) * (-(-I.nyf // 16)) == (296 if nxc == 296 else 304)
        cut = lambda a: np.ascontiguousarray(a[:, :, :I.nxf + 1]).reshape(a.shape[0], -1)   # noqa: E731
        nodes = lambda t: t.view(-1, I.nyf + 1, I.pitch)[:, :, :4 * SAME].clone()           # noqa: E731
        x, b = mesh.pack(cut(xf)), mesh.pack(cut(bf))
        d = torch.as_tensor(dp[:, :nxc][~sol]).to(mesh.real).cuda().contiguous()
        keep = torch.as_tensor((np.broadcast_to(np.arange(nxc), sol.shape) < SAME)[~sol])
        xcd = torch.as_tensor(np.ascontiguousarray(xc[:, :, :nxc + 1])).cuda().reshape(-1)
        out = []
        for given in (dict(xf=x), dict(xf=None, xc=xcd)):
            rf, X, v = mesh.fine(3), mesh.features(), mesh.fine(2)
            dn.dnnmg_patch_features(mesh, given["xf"], b, X, rf=rf, xc=given.get("xc"))
            dn.dnnmg_scatter_avg(mesh, d, given["xf"], v, xc=given.get("xc"))
            out += [nodes(rf), X.cpu()[keep], nodes(v)]
        r = mesh.fine(2)
        dn.dnnmg_rhs(mesh, x[:2].contiguous(), r)
        got.append(out + [nodes(r)])
    for a, b in zip(*got):
        assert a.shape == b.shape and torch.equal(a, b)
