"""Batched steps take other kernels than the instances alone when their tiles
together pass a threshold, when there are more instances than one launch takes,
and when v_corr of all does not fit the scratch.  An instance has the same bits
alone and in every such batch, also when steps alternate between streams."""

import numpy as np
import pytest
import torch

from helpers import Params, coarse_input, weights

pytestmark = pytest.mark.gpu

K_STEP = Params().k


@pytest.fixture(scope="module")
def dn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11520_gb300 import dnnmg
    return dnnmg


def instance(dn, K, s, nxc, nyc, seed):
    case = dict(nxc=nxc, nyc=nyc, K=K, s=s, H=64, prec="bf16")
    ellipse = None if seed % 3 == 0 else (0.3 + 0.1 * (seed % 5), 0.2, 0.05, 0.04)
    m = dn.Mesh(dn.make_desc(nxc, nyc, K, s, ellipse, precision="bf16"))
    I = m.info
    g = torch.Generator(device="cuda").manual_seed(seed)
    v, b0 = m.fine(2), m.fine(2)
    v.view(2, I.nyf + 1, I.pitch)[:, :, :I.nxf + 1] = 0.3 * torch.randn(2, I.nyf + 1, I.nxf + 1, device="cuda", generator=g)
    dn.dnnmg_rhs_restrict(m, v, b0, m.coarse(3))
    xc = torch.as_tensor(coarse_input(case, seed=seed)).cuda().contiguous()
    return dict(m=m, xc=xc, b0=b0)


def net_for(dn, m, K, s):
    I = m.info
    return dn.Net(*weights(dict(K=K, s=s, H=64, prec="bf16"), I.n_in, I.n_out), precision="bf16")


def alone(dn, net, q, steps):
    m = q["m"]
    h, bf, bc, ws = torch.zeros(m.info.P, 64, device="cuda"), q["b0"].clone(), m.coarse(3), m.workspace()
    for n in range(steps):
        dn.dnnmg_step(m, net, q["xc"], h, bf, bc, ws, n * K_STEP)
    return h, bf, bc


def compare(dn, net, insts, steps, run):
    srv = dn.Server(net, sum(-(-q["m"].info.P // 128) * 128 for q in insts))
    slots = [srv.admit(q["m"]) for q in insts]
    bf, bc = [q["b0"].clone() for q in insts], [q["m"].coarse(3) for q in insts]
    torch.cuda.synchronize()
    for n in range(steps):
        run(srv, n, [(slots[i], q["xc"], bf[i], bc[i], n * K_STEP) for i, q in enumerate(insts)])
    torch.cuda.synchronize()
    for i, q in enumerate(insts):
        h, b, c = alone(dn, net, q, steps)
        assert torch.equal(srv.state(slots[i]), h), i
        assert torch.equal(bf[i], b), i
        assert torch.equal(bc[i], c), i
        assert bool(torch.isfinite(b).all()) and float(h.abs().max()) > 0
    srv.close()


SMALL = [(32, 8), (48, 10), (40, 10), (64, 16)]
# 32 x 16-cell tiles of all instances, and what they are there for
BATCHES = {
    "boundary_tiles_304": (1, 1, [(256, 64)] * 10),              # 1280 tiles, over 304 of them with a boundary
    "tiles_4096": (1, 1, [(512, 128)] * 8),                      # the tall walk; alone 512: the short one
    "two_launches": (1, 1, SMALL * 10),                          # 40 instances: 32 and 8
    "large_and_small": (1, 1, SMALL * 5 + [(384, 96)] + SMALL * 5),
    "k2": (2, 1, [(128, 32)] * 9 + SMALL),                       # nine large: v_corr of eight fits
    "k2_two_cells": (2, 2, [(64, 16)] * 6 + SMALL),
    "k3_few": (3, 1, [(12, 6), (16, 8), (20, 4)]),               # no closed form: lists of all tiles, small
    "k3_many": (3, 1, [(64, 16)] * 3 + [(12, 6), (16, 8)]),      # and large
}


@pytest.mark.parametrize("name", list(BATCHES))
def test_batch_equals_alone_bitwise(dn, name):
    K, s, sizes = BATCHES[name]
    insts = [instance(dn, K, s, nx, ny, seed=i + 1) for i, (nx, ny) in enumerate(sizes)]
    net = net_for(dn, insts[0]["m"], K, s)
    compare(dn, net, insts, 2, lambda srv, n, items: srv.step(items))


def test_steps_on_two_streams_in_turn(dn):
    """The server's buffers serve one step at a time: a step waits for the one
    before it on another stream."""
    sizes = [(256, 64)] * 4 + SMALL
    insts = [instance(dn, 1, 1, nx, ny, seed=i + 1) for i, (nx, ny) in enumerate(sizes)]
    net = net_for(dn, insts[0]["m"], 1, 1)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]

    def run(srv, n, items):
        # two batches a step, each with instances of its own, on alternating streams
        for part in (0, 1):
            with torch.cuda.stream(streams[(n + part) % 2]):
                srv.step(items[part::2])
    compare(dn, net, insts, 6, run)
