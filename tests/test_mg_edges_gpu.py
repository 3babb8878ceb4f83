"""The multigrid kernels at the edges of their tiles and of their variants:
levels whose nodes end inside, at and past a 32 x 4-node tile, the smallest
levels, and FP32 sweeps on both sides of the size where the smoother changes
its form."""

import numpy as np
import pytest
import torch

from helpers import rel_l2
from paper_2008_11520_gb300 import solver
from parity import check
from test_mg_gpu import dev, flow, host_level, vanka_reference

pytestmark = pytest.mark.gpu

ELL = (0.4, 0.2, 0.12, 0.07)


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def inputs(nx, ny, seed):
    solid = solver.refine_mask(solver.ellipse_mask(nx // 2, ny // 2, ELL), 1)
    lev = host_level(nx, ny, solid)
    rng = np.random.default_rng(seed)
    x = flow(lev) + 0.05 * rng.standard_normal((3, lev.N))
    return solid, lev, x, rng.standard_normal((3, lev.N)), 0.1 * rng.standard_normal((3, lev.N))


# nodes: 5 x 5, 31 x 7, 33 x 5, 63 x 13, 65 x 17
@pytest.mark.parametrize("nx,ny", [(4, 4), (30, 6), (32, 4), (62, 12), (64, 16)])
def test_operators_and_sweep_at_tile_edges(dn, nx, ny):
    solid, lev, x, r, d0 = inputs(nx, ny, 3)
    mg = dn.MG(nx, ny, 1, solid, "f64")
    y = mg.field(0)
    mg.jvp(0, dev(x), dev(d0), y)
    check("mg J dx", rel_l2(y.cpu().numpy(), (lev.jacobian(x) @ d0.ravel()).reshape(3, -1)), 1e-12, "f64")
    mg.defect(0, dev(x), dev(r), 0.2, y)
    check("mg defect", rel_l2(y.cpu().numpy(), lev.defect(x, r, 0.2)), 1e-12, "f64")
    mg.rhs(0, dev(x), y)
    check("mg rhs", rel_l2(y.cpu().numpy()[:2], lev.rhs(x[:2])), 1e-12, "f64")
    d = dev(d0)
    mg.vanka(0, dev(x), dev(r), d, 0.8)
    check("mg Vanka sweep", rel_l2(d.cpu().numpy(), vanka_reference(lev, x, r, d0, 0.8)), 1e-11, "f64")


# cells of a colour: 64 and 9900 (eliminated ahead of the pass before), 10400 and 16384.
# FP64 sweeps carry about 500 roundings (5e-14 against the reference above): 500 x 6e-8 in FP32
@pytest.mark.parametrize("nx,ny", [(64, 16), (792, 200), (832, 200), (1024, 256)])
def test_fp32_sweep_equals_fp64(dn, nx, ny):
    solid, lev, x, r, d0 = inputs(nx, ny, 4)
    r = r * lev.hx * lev.hy / lev.k
    got = {}
    for prec, real in (("f64", torch.float64), ("f32", torch.float32)):
        mg = dn.MG(nx, ny, 1, solid, prec)
        d = dev(d0, real)
        x32, r32 = (dev(a.astype(np.float32).astype(np.float64), real) for a in (x, r))
        mg.vanka(0, x32, r32, d, 1.0)
        got[prec] = d.double().cpu().numpy()
    check("mg Vanka sweep", rel_l2(got["f32"], got["f64"]), 3e-5, "f32")
