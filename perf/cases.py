"""What the framework is timed on: the work its users have it do, through its public entry points.

Kinds of cases (the "kind" of a case), each over the sizes of the workloads in synth.py, the tests and bench.py:

* ``step``     one correction step (dnnmg_step) of one flow instance: the call a time loop makes once per time
               step.  FP64 on the plain instance (latency), FP32 fields and net, or FP32 fields with the BF16 net.
* ``serve``    one batched step of several instances with meshes of different sizes (Server.step): what the
               request loop runs whenever the GPU is free.
* ``train``    loss and gradients of one training window (PatchNetTrainer.loss, backward): what every update
               of the patch network does, FP32 or BF16 products.
* ``gru``      the patch network alone (dnnmg_gru_step): the network evaluated on given feature rows, as the
               accuracy evaluation (e_rel) and the training data path do.
* ``windows``  one time step of training data (dnnmg_rhs, dnnmg_prolongate, dnnmg_patch_features,
               dnnmg_scatter_avg on given fields): the single-pass entry points on whole fields.
* ``mg``       the way down one level of the plain multigrid solve (two Vanka sweeps, Newton-matrix product,
               axpby, restriction): the comparison method's hot loop.

Inputs are made on the GPU from the seed: a Poiseuille profile with drifting vortices as coarse solution, a fine
velocity with mesh-scale noise behind the right-hand side, weights and states of the workloads' distributions.
"""

import math

import numpy as np
import torch

from paper_2008_11520_gb300 import dnnmg, train

LX, LY, NU, DT, ALPHA0, U_MAX = 2.2, 0.41, 1e-3, 0.01, 0.1, 1.5
F64 = torch.float64


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: a 32 x 8 channel in FP64, latency and launches
        dict(name="step_plain_f64", kind="step", nxc=32, nyc=8, K=1, s=1, H=32, prec="f64", ay=0.06, ax=0.04),
        # an ordinary instance, FP32 net (the parity workload, 1024 x 256 fine cells)
        dict(name="step_channel_f32", kind="step", nxc=256, nyc=64, K=2, s=1, H=64, prec="f32", ay=0.04, ax=0.05),
        # the flagship: 16.8 M fine nodes, 2 x 2-cell patches, BF16 net
        dict(name="step_large_bf16", kind="step", nxc=2048, nyc=512, K=2, s=2, H=128, prec="bf16", ay=0.03, ax=0.05),
        # a full batch of the serving workload's one-level instances, 64 x 16 .. 512 x 128 coarse cells
        dict(name="serve_batch", kind="serve", n=20, lo=64, hi=512, K=1, H=64),
        # a lone request of the serving workload (most batches at its mean load hold one instance)
        dict(name="serve_one", kind="serve", n=1, lo=256, hi=256, K=2, H=64),
        # one update's gradients at the training workload's batch, BF16 products
        dict(name="train_bf16", kind="train", P=65536, T=10, nxc=128, K=1, H=64, prec="bf16"),
        # the same in FP32, the default precision of the trainer
        dict(name="train_f32", kind="train", P=65536, T=10, nxc=128, K=1, H=64, prec="f32"),
        # the accuracy experiment's update: three 32 x 8 flows side by side, FP32
        dict(name="train_small_f32", kind="train", P=762, T=10, nxc=32, K=1, H=32, prec="f32"),
        # the FP32 network alone at the parity workload's patches
        dict(name="gru_f32", kind="gru", P=16336, nxc=256, K=2, s=1, H=64, prec="f32"),
        # one time step of training data on the training workload's mesh
        dict(name="windows_f32", kind="windows", nxc=128, nyc=32, K=1, s=1, prec="f32", ay=0.04, ax=0.05),
        # plain multigrid on the parity workload's fine level, FP32
        dict(name="mg_f32", kind="mg", nx=1024, ny=256, prec="f32", ay=0.04, ax=0.05),
        # plain multigrid on the training workload's fine level, FP64
        dict(name="mg_f64", kind="mg", nx=256, ny=64, prec="f64", ay=0.04, ax=0.05),
    ]


def draw(rng):
    def size(lo, hi, step=1):
        return step * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)

    kind = rng.choice(["step", "step", "serve", "train", "train", "gru", "windows", "mg"])
    ay = round(rng.uniform(0.025, 0.06), 4)
    if kind == "step":
        prec = rng.choice(["f64", "f32", "bf16", "bf16"])
        hi = {"f64": 96, "f32": 512, "bf16": 1024}[prec]
        nxc = size(24, hi, 2)
        H = {"f64": 32, "f32": rng.choice([32, 64]), "bf16": rng.choice([64, 128])}[prec]
        return dict(kind=kind, nxc=nxc, nyc=max(6, 2 * round(nxc / rng.uniform(7.0, 9.0))), K=rng.choice([1, 2]),
                    s=rng.choice([1, 2]), H=H, prec=prec, ay=ay, ax=0.05)
    if kind == "serve":
        return dict(kind=kind, n=size(1, 20), lo=64, hi=rng.choice([128, 256, 512]), K=rng.choice([1, 2]), H=64)
    if kind == "train":
        prec = rng.choice(["f32", "bf16"])
        return dict(kind=kind, P=size(250, 60000), T=rng.choice([5, 10]), nxc=rng.choice([32, 64, 128]),
                    K=rng.choice([1, 1, 2]), H=rng.choice([32, 64]), prec=prec)
    if kind == "gru":
        return dict(kind=kind, P=size(500, 60000), nxc=rng.choice([64, 128, 256]), K=rng.choice([1, 2]), s=1,
                    H=rng.choice([32, 64]), prec=rng.choice(["f32", "bf16"]))
    if kind == "windows":
        nxc = size(32, 256, 2)
        return dict(kind=kind, nxc=nxc, nyc=max(8, 2 * round(nxc / 8)), K=rng.choice([1, 2]), s=1, prec="f32",
                    ay=ay, ax=0.05)
    nx = size(64, 1024, 8)
    return dict(kind="mg", nx=nx, ny=max(16, 8 * round(nx / 32)), prec=rng.choice(["f32", "f64"]) if nx <= 384
                else "f32", ay=ay, ax=0.05)


# ---------------------------------------------------------------- inputs
def _rng(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _flow(nx, ny, seed, obst):
    """Nodal (u, v, p) [3][ny+1][nx+1] of a Poiseuille profile with eight vortices, zero inside the obstacle."""
    r = np.random.default_rng(seed + 77)
    y, x = torch.meshgrid(torch.arange(ny + 1, dtype=F64, device="cuda") * (LY / ny),
                          torch.arange(nx + 1, dtype=F64, device="cuda") * (LX / nx), indexing="ij")
    wall = 4.0 * y * (LY - y) / LY ** 2
    u, v = U_MAX * wall, torch.zeros_like(x)
    for _ in range(8):
        x0, y0, rc = r.uniform(0.3, LX - 0.2), r.uniform(0.08, LY - 0.08), r.uniform(0.02, 0.06)
        g = float(r.choice([-0.15, 0.15])) / rc * wall * torch.exp(-((x - x0) ** 2 + (y - y0) ** 2) / rc ** 2)
        u = u - g * (y - y0)
        v = v + g * (x - x0)
    ax, ay = obst
    s = (((((x - 0.2) / ax) ** 2 + ((y - 0.2) / ay) ** 2) - 1.0) / 0.5).clamp(0.0, 1.0)
    s = s * s * (3.0 - 2.0 * s)
    return torch.stack([u * s, v * s, 8.0 * U_MAX * NU / LY ** 2 * (LX - x)])


def _solid(nx, ny, obst):
    """Cells [ny][nx] whose centroid lies inside the obstacle."""
    x = (np.arange(nx) + 0.5) * (LX / nx)
    y = (np.arange(ny) + 0.5) * (LY / ny)
    return ((x[None, :] - 0.2) / obst[0]) ** 2 + ((y[:, None] - 0.2) / obst[1]) ** 2 < 1.0


def _weights(n_in, H, n_out, seed, std=0.1):
    r = np.random.default_rng(seed + 5)
    return r.normal(0.0, std, (3 * H, n_in)), r.normal(0.0, std, (3 * H, H)), r.normal(0.0, std, (n_out, H))


def _sizes(K, s):
    S = s << K
    nf, nc = (S + 1) ** 2, (s + 1) ** 2
    return nf, nc, 3 * nf + 3 * nc + 12, 2 * nf


def _geometry(nxc, nyc, s):
    """The 12 geometry values of an s x s-cell patch: edges, aspect ratios, angles."""
    w, h = s * LX / nxc, s * LY / nyc
    return [w, h, w, h, w / h, w / h, 1.0, 1.0] + [math.pi / 2] * 4


def _feature_rows(lead, P, nxc, K, s, seed):
    """Feature rows [lead * P][n_in] of the size patches have: residuals, coarse velocities, Peclet numbers, geometry."""
    nf, nc, n_in, _ = _sizes(K, s)
    g = _rng(seed, 3)
    n = lead * P
    res = 1e-4 * torch.randn(n, 3 * nf, device="cuda", generator=g)
    vel = torch.cat([1.5 * torch.rand(n, nc, device="cuda", generator=g),
                     0.3 * torch.randn(n, nc, device="cuda", generator=g)], dim=1)
    pe = s * LX / nxc / NU * torch.sqrt(vel[:, :nc] ** 2 + vel[:, nc:] ** 2) * (1.0 if nxc >= 64 else 0.5)
    geo = torch.tensor(_geometry(nxc, nxc // 4, s), device="cuda", dtype=torch.float32).expand(n, 12)
    return torch.cat([res, vel, pe, geo], dim=1)


def _padded(X):
    """Rows padded with zeros to a multiple of 16 columns, the layout of the feature matrix."""
    n, n_in = X.shape
    out = torch.zeros(n, (n_in + 15) // 16 * 16, dtype=X.dtype, device=X.device)
    out[:, :n_in] = X
    return out


def _pitched(mesh, f):
    """Node values [comp][ny+1][nx+1] -> the mesh's pitched field [comp][plane]."""
    I = mesh.info
    out = torch.zeros(f.shape[0], I.nyf + 1, I.pitch, dtype=mesh.real, device="cuda")
    out[:, :, :I.nxf + 1] = f
    return out.reshape(f.shape[0], I.plane)


def _nodes(mesh, t):
    """The nodes of a pitched field (the row padding left out), as a view."""
    I = mesh.info
    return t.view(-1, I.nyf + 1, I.pitch)[:, :, :I.nxf + 1]


def _instance(c, seed):
    """Inputs of one instance: grid, coarse solution x_c, right-hand side b_f and state h, rounded as the call takes them."""
    obst = (c["ax"], c["ay"])
    real = F64 if c["prec"] == "f64" else torch.float32
    G = Grid(c["nxc"], c["nyc"], c["K"], c["s"], _solid(c["nxc"], c["nyc"], obst))
    xc = _flow(c["nxc"], c["nyc"], seed, obst)
    v = _flow(G.nx, G.ny, seed + 1, obst)[:2]
    v = v + 0.05 * U_MAX * (2.0 * torch.rand(v.shape, dtype=F64, device="cuda", generator=_rng(seed, 1)) - 1.0)
    bf = G.rhs(v).to(real)
    h = (torch.rand(G.P, c["H"], dtype=F64, device="cuda", generator=_rng(seed, 2)) - 0.5).to(real)
    return G, xc, bf, h


def _mesh(c):
    return dnnmg.Mesh(dnnmg.make_desc(c["nxc"], c["nyc"], c["K"], c["s"], (0.2, 0.2, c["ax"], c["ay"]),
                                      precision=c["prec"]))


def _serve_instances(c):
    """Meshes of a batch: coarse grids of the serving workload's range, one after the other over its logarithm."""
    out = []
    for i in range(c["n"]):
        f = (i + 0.5) / c["n"]
        nxc = 16 * round(c["lo"] * (c["hi"] / c["lo"]) ** f / 16)
        out.append(dict(nxc=nxc, nyc=nxc // 4, K=c["K"], s=1, H=c["H"], prec="bf16", ax=0.05,
                        ay=0.025 + 0.025 * ((7 * i) % 11) / 11))
    return out


def _train_inputs(c, seed):
    nf, nc, n_in, n_out = _sizes(c["K"], 1)
    T, P = c["T"], c["P"]
    X = _padded(_feature_rows(T, P, c["nxc"], c["K"], 1, seed)).view(T, P, -1)
    Y = 0.1 * torch.randn(T, P, n_out, device="cuda", generator=_rng(seed, 4))
    h0 = torch.rand(P, c["H"], device="cuda", generator=_rng(seed, 5)) - 0.5
    return X, Y, h0, n_in, n_out


def _mg_inputs(c, seed):
    obst = (c["ax"], c["ay"])
    real = F64 if c["prec"] == "f64" else torch.float32
    solid = _solid(c["nx"] // 2, c["ny"] // 2, obst).repeat(2, axis=0).repeat(2, axis=1)
    L = Grid(c["nx"], c["ny"], 0, 1, solid)
    x = _flow(c["nx"], c["ny"], seed, obst)
    x[0], x[1] = torch.where(L.dirichlet, L.inflow, x[0]), torch.where(L.dirichlet, 0.0, x[1])
    x[2] = torch.where(L.p_active, x[2], 0.0)
    r = torch.randn(3, L.ny + 1, L.nx + 1, dtype=F64, device="cuda", generator=_rng(seed, 6)) * (L.hx * L.hy / DT)
    r[:2] = torch.where(L.dirichlet, 0.0, r[:2])
    r[2] = torch.where(L.p_active, r[2], 0.0)
    return L, solid, x.to(real), r.to(real)


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        G, xc, bf, h = _instance(c, seed)
        mesh = _mesh(c)
        assert mesh.info.P == G.P
        net = dnnmg.Net(*_weights(mesh.info.n_in, c["H"], mesh.info.n_out, seed), precision=c["prec"])
        return dict(kind=kind, mesh=mesh, net=net, xc=xc.reshape(3, -1).contiguous(), h=h, bf=_pitched(mesh, bf),
                    bc=mesh.coarse(3), ws=mesh.workspace())
    if kind == "serve":
        nf, nc, n_in, n_out = _sizes(c["K"], 1)
        net = dnnmg.Net(*_weights(n_in, c["H"], n_out, seed), precision="bf16")
        made = []
        for i, ci in enumerate(_serve_instances(c)):
            G, xc, bf, h = _instance(ci, seed + 31 * i)
            made.append((_mesh(ci), xc.reshape(-1).contiguous(), bf, h))
        server = dnnmg.Server(net, sum((m.info.P + 127) // 128 * 128 for m, _, _, _ in made))
        items, states, out = [], [], []
        for mesh, xc, bf, h in made:
            slot = server.admit(mesh)
            st = server.state(slot)
            st.owner = server   # a view of the server's memory: it lives as long as the view
            st.copy_(h)
            bfp, bc = _pitched(mesh, bf), mesh.coarse(3)
            items.append((slot, xc, bfp, bc, 0.0))
            out.append((st, _nodes(mesh, bfp), bc))
        return dict(kind=kind, server=server, items=items, out=out)
    if kind == "train":
        X, Y, h0, n_in, n_out = _train_inputs(c, seed)
        tn = train.PatchNetTrainer(n_in, X.shape[2], c["H"], n_out, c["T"], c["P"], seed=seed % 100003, std=0.02,
                                   out_std=0.05, precision=c["prec"])
        return dict(kind=kind, tn=tn, X=X, Y=Y, h0=h0)
    if kind == "gru":
        nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
        net = dnnmg.Net(*_weights(n_in, c["H"], n_out, seed), precision=c["prec"])
        X = _padded(_feature_rows(1, c["P"], c["nxc"], c["K"], c["s"], seed)).to(net.feat)
        h = torch.rand(c["P"], c["H"], device="cuda", generator=_rng(seed, 5)) - 0.5
        return dict(kind=kind, net=net, X=X, h=h, d=torch.empty(c["P"], n_out, device="cuda"), P=c["P"])
    if kind == "windows":
        G, xc, bf, h = _instance(dict(c, H=1), seed)
        mesh = _mesh(c)
        prev = _flow(G.nx, G.ny, seed + 1, (c["ax"], c["ay"]))[:2]
        d = 0.05 * torch.randn(G.P, mesh.info.n_out, device="cuda", generator=_rng(seed, 7))
        return dict(kind=kind, mesh=mesh, xc=xc.reshape(-1).contiguous(), prev=_pitched(mesh, prev), d=d,
                    xf=mesh.fine(3), bf=mesh.fine(2), vc=mesh.fine(2), X=mesh.features())
    L, solid, x, r = _mg_inputs(c, seed)
    mg = dnnmg.MG(c["nx"], c["ny"], 2, solid, c["prec"])
    f = mg.field
    return dict(kind=kind, mg=mg, x=x.reshape(3, -1).contiguous(), r=r.reshape(3, -1).contiguous(), d=f(0), t=f(0),
                rc=f(1))


def run(s):
    kind = s["kind"]
    if kind == "step":
        dnnmg.dnnmg_step(s["mesh"], s["net"], s["xc"], s["h"], s["bf"], s["bc"], s["ws"], 0.0)
        return dict(h=s["h"], bf=_nodes(s["mesh"], s["bf"]), bc=s["bc"])
    if kind == "serve":
        s["server"].step(s["items"])
        return s["out"]
    if kind == "train":
        tn = s["tn"]
        for p in tn.params:
            p.grad = None
        L, D = tn.loss(s["X"], s["Y"], s["h0"])
        L.backward()
        return dict(loss=L.detach(), D=D.detach(), hT=tn.trainer.state().clone(), grads=[p.grad for p in tn.params])
    if kind == "gru":
        dnnmg.dnnmg_gru_step(s["net"], s["X"], s["h"], s["d"], s["P"])
        return dict(h=s["h"], d=s["d"])
    if kind == "windows":
        m = s["mesh"]
        dnnmg.dnnmg_prolongate(m, s["xc"], s["xf"], 0.0)
        dnnmg.dnnmg_rhs(m, s["prev"], s["bf"])
        dnnmg.dnnmg_patch_features(m, s["xf"], s["bf"], s["X"])
        dnnmg.dnnmg_scatter_avg(m, s["d"], s["xf"], s["vc"])
        return dict(xf=_nodes(m, s["xf"]), bf=_nodes(m, s["bf"]), X=s["X"], vc=_nodes(m, s["vc"]))
    mg, d, t = s["mg"], s["d"], s["t"]
    d.zero_()
    mg.vanka(0, s["x"], s["r"], d, 1.0)
    mg.vanka(0, s["x"], s["r"], d, 1.0)
    mg.jvp(0, s["x"], d, t)
    mg.axpby(1.0, s["r"], -1.0, t)
    mg.restrict(0, t, s["rc"])
    return dict(d=d, t=t, rc=s["rc"])


# ---------------------------------------------------------------- work
def _net_flops(rows, n_in, H, n_out):
    return 2.0 * rows * (3 * H * (n_in + H) + H * n_out)


def _step_work(c):
    nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
    fb = 8 if c["prec"] == "f64" else 4
    P = c["nxc"] * c["nyc"] // c["s"] ** 2
    Nf = ((c["nxc"] << c["K"]) + 1) * ((c["nyc"] << c["K"]) + 1)
    Nc = (c["nxc"] + 1) * (c["nyc"] + 1)
    # x_c in, b_c out, b_f and h read and written, weights; about 300 operations per fine node around the net
    by = 2 * 3 * Nc * 8 + 2 * 2 * Nf * fb + 2 * P * c["H"] * fb + (3 * c["H"] * (n_in + c["H"]) + c["H"] * n_out) * fb
    return by, _net_flops(P, n_in, c["H"], n_out) + 300.0 * Nf


def work(case):
    c, kind = case, case["kind"]
    if kind == "step":
        by, fl = _step_work(c)
    elif kind == "serve":
        w = [_step_work(i) for i in _serve_instances(c)]
        by, fl = sum(a for a, _ in w), sum(b for _, b in w)
    elif kind == "train":
        nf, nc, n_in, n_out = _sizes(c["K"], 1)
        n = c["T"] * c["P"]
        # X, Y and h_0 in, D and h_T out; forward, state gradients and weight gradients
        by = 4.0 * (n * (n_in + 2 * n_out) + 2 * c["P"] * c["H"])
        fl = 3.0 * _net_flops(n, n_in, c["H"], n_out)
    elif kind == "gru":
        nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
        by = c["P"] * (n_in * (2 if c["prec"] == "bf16" else 4) + 4 * (2 * c["H"] + n_out))
        fl = _net_flops(c["P"], n_in, c["H"], n_out)
    elif kind == "windows":
        nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
        P, Nf = c["nxc"] * c["nyc"], ((c["nxc"] << c["K"]) + 1) * ((c["nyc"] << c["K"]) + 1)
        # x_c, previous velocity and d in; x~, b_f, X and v_corr out
        by = 3 * (c["nxc"] + 1) * (c["nyc"] + 1) * 8 + 4.0 * (9 * Nf + P * (n_in + n_out))
        fl = 300.0 * Nf
    else:
        N = (c["nx"] + 1) * (c["ny"] + 1)
        fb = 8 if c["prec"] == "f64" else 4
        # x and the right-hand side in, the correction and the residual out, the coarse residual out; per cell and
        # sweep the assembly (about 1500) and solution (about 1300) of a 12 x 12 block and its defect (about 1200)
        by = fb * 3 * N * 4.25
        fl = 2 * 4000.0 * c["nx"] * c["ny"] + 400.0 * N
    return {"bytes": float(by), "flops": float(fl)}


# ---------------------------------------------------------------- the same in 64 bits
class Grid:
    """A masked channel grid (coarse cells nxc x nyc, K refinements) and the method's operators on it, 64 bits."""

    def __init__(self, nxc, nyc, K, s, solid):
        self.nxc, self.nyc, self.K, self.s, self.r, self.S = nxc, nyc, K, s, 1 << K, s << K
        self.nx, self.ny = nxc << K, nyc << K
        self.hx, self.hy = LX / self.nx, LY / self.ny
        self.solid_c = torch.as_tensor(np.asarray(solid, dtype=bool)).cuda()
        sol = self.solid_c.repeat_interleave(self.r, 0).repeat_interleave(self.r, 1)
        self.fluid = (~sol).to(F64)
        self.dirichlet, self.zero_bc, self.p_active = self._classes(sol)
        self.dirichlet_c = self._classes(self.solid_c)[0]
        y = torch.arange(self.ny + 1, dtype=F64, device="cuda") * self.hy
        prof = (U_MAX * 4.0 * y * (LY - y) / LY ** 2)[:, None]
        first = (torch.arange(self.nx + 1, device="cuda") == 0)[None, :] & ~self.zero_bc
        self.inflow = torch.where(first, prof, 0.0)
        self.npx, self.npy = nxc // s, nyc // s
        self.patch = ~self.solid_c.view(self.npy, s, self.npx, s).all(3).all(1)
        self.P = int(self.patch.sum())

    @staticmethod
    def _classes(sol):
        ny, nx = sol.shape
        ts = torch.zeros(ny + 1, nx + 1, dtype=torch.bool, device="cuda")
        tf = torch.zeros_like(ts)
        for b in (0, 1):
            for a in (0, 1):
                ts[b:b + ny, a:a + nx] |= sol
                tf[b:b + ny, a:a + nx] |= ~sol
        zero = ts.clone()
        zero[0] = zero[-1] = True
        dirichlet = zero.clone()
        dirichlet[:, 0] = True
        return dirichlet, zero, tf

    def _gauss(self):
        """(weight, shape values, x- and y-derivatives) of the four corners at the 2 x 2 Gauss points of a cell."""
        g = 0.5 / math.sqrt(3.0)
        for eta in (0.5 - g, 0.5 + g):
            for xi in (0.5 - g, 0.5 + g):
                ph = [(1 - xi) * (1 - eta), xi * (1 - eta), (1 - xi) * eta, xi * eta]
                dx = [-(1 - eta) / self.hx, (1 - eta) / self.hx, -eta / self.hx, eta / self.hx]
                dy = [-(1 - xi) / self.hy, -xi / self.hy, (1 - xi) / self.hy, xi / self.hy]
                yield self.hx * self.hy / 4.0, ph, dx, dy

    def _corner(self, f, a):
        return f[a >> 1:(a >> 1) + self.ny, a & 1:(a & 1) + self.nx]

    def _at(self, f, w):
        return sum(w[a] * self._corner(f, a) for a in range(4))

    def _velocity(self, u, v, sign, p=None):
        """(1/k) mass + sign/2 convection + sign nu/2 diffusion (- pressure gradient); with p the divergence too."""
        out = [torch.zeros_like(u) for _ in range(3 if p is not None else 2)]
        for w, ph, dx, dy in self._gauss():
            w = w * self.fluid
            uq, vq = self._at(u, ph), self._at(v, ph)
            ux, uy, vx, vy = self._at(u, dx), self._at(u, dy), self._at(v, dx), self._at(v, dy)
            mu = uq / DT + 0.5 * sign * (uq * ux + vq * uy)
            mv = vq / DT + 0.5 * sign * (uq * vx + vq * vy)
            pq = self._at(p, ph) if p is not None else 0.0
            for a in range(4):
                self._corner(out[0], a).add_(w * (mu * ph[a] + 0.5 * sign * NU * (ux * dx[a] + uy * dy[a]) - pq * dx[a]))
                self._corner(out[1], a).add_(w * (mv * ph[a] + 0.5 * sign * NU * (vx * dx[a] + vy * dy[a]) - pq * dy[a]))
                if p is not None:
                    self._corner(out[2], a).add_(w * (ux + vy) * ph[a])
        return out

    def lps_matrices(self):
        """[4][9][9]: the projection term's integrals over each cell of a 2 x 2-cell patch, on the patch's nodes."""
        Q = torch.eye(9, dtype=F64)
        for b in range(3):
            for a in range(3):
                X, Y = a / 2.0, b / 2.0
                for j, wt in ((0, (1 - X) * (1 - Y)), (2, X * (1 - Y)), (6, (1 - X) * Y), (8, X * Y)):
                    Q[3 * b + a, j] -= wt
        E = torch.zeros(4, 4, dtype=F64)
        for w, _, dx, dy in self._gauss():
            dx, dy = torch.tensor(dx, dtype=F64), torch.tensor(dy, dtype=F64)
            E += w * (torch.outer(dx, dx) + torch.outer(dy, dy))
        out = torch.zeros(4, 9, 9, dtype=F64)
        for c in range(4):
            ca, cb = c & 1, c >> 1
            ids = torch.tensor([3 * cb + ca, 3 * cb + ca + 1, 3 * cb + ca + 3, 3 * cb + ca + 4])
            F = torch.zeros(9, 9, dtype=F64)
            F[ids[:, None], ids[None, :]] = E
            out[c] = ALPHA0 * (self.hx ** 2 + self.hy ** 2) / NU * Q.T @ F @ Q
        return out.cuda()

    def lps(self, p):
        npy, npx = self.ny // 2, self.nx // 2
        at = lambda f, i: f[i // 3:i // 3 + 2 * npy - 1:2, i % 3:i % 3 + 2 * npx - 1:2]   # noqa: E731
        p9 = torch.stack([at(p, i) for i in range(9)]).reshape(9, -1)
        acc = torch.zeros_like(p9)
        for c, M in enumerate(self.lps_matrices()):
            acc += self.fluid[c >> 1::2, c & 1::2].reshape(1, -1) * (M @ p9)
        out = torch.zeros_like(p)
        for i in range(9):
            at(out, i).add_(acc[i].view(npy, npx))
        return out

    def rhs(self, v):
        b = torch.stack(self._velocity(v[0], v[1], -1.0))
        return torch.where(self.dirichlet, 0.0, b)

    def residual(self, x, bf):
        Au, Av, Ap = self._velocity(x[0], x[1], 1.0, x[2])
        Ap = Ap + self.lps(x[2])
        r = torch.stack([bf[0] - Au, bf[1] - Av, -Ap])
        r[:2] = torch.where(self.dirichlet, 0.0, r[:2])
        r[2] = torch.where(self.p_active, r[2], 0.0)
        return r

    def prolongate(self, xc):
        r = self.r

        def along(f, n):   # the last dimension, n coarse cells
            i = torch.arange(n * r + 1, device="cuda")
            ci = (i // r).clamp(max=n - 1)
            w = (i - ci * r).to(F64) / r
            return f[..., ci] * (1.0 - w) + f[..., ci + 1] * w

        x = along(along(xc, self.nxc).transpose(1, 2), self.nyc).transpose(1, 2).contiguous()
        x[0] = torch.where(self.dirichlet, self.inflow, x[0])
        x[1] = torch.where(self.dirichlet, 0.0, x[1])
        return x

    def restrict(self, bf, mask=None):
        for _ in range(self.K):
            for _ in range(2):   # along the last dimension, then the other
                even, odd = bf[..., 0::2].clone(), 0.5 * bf[..., 1::2]
                even[..., :-1] += odd
                even[..., 1:] += odd
                bf = even.transpose(1, 2)
        bf = bf.contiguous()
        return torch.cat([torch.where(self.dirichlet_c, 0.0, bf), torch.zeros_like(bf[:1])])

    def features(self, x, r):
        S, s, R = self.S, self.s, self.r
        rows = [f.unfold(0, S + 1, S).unfold(1, S + 1, S)[self.patch].reshape(self.P, -1) for f in r]
        co = [f[::R, ::R].unfold(0, s + 1, s).unfold(1, s + 1, s)[self.patch].reshape(self.P, -1) for f in x[:2]]
        pe = s * max(LX / self.nxc, LY / self.nyc) / NU * torch.sqrt(co[0] ** 2 + co[1] ** 2)
        geo = torch.tensor(_geometry(self.nxc, self.nyc, s), dtype=F64, device="cuda").expand(self.P, 12)
        return torch.cat(rows + co + [pe, geo], dim=1)

    def average(self, d, x):
        S, nf = self.S, (self.S + 1) ** 2
        g = torch.zeros(self.npy, self.npx, 2 * nf, dtype=F64, device="cuda")
        g[self.patch] = d
        tot = torch.zeros(2, self.ny + 1, self.nx + 1, dtype=F64, device="cuda")
        cnt = torch.zeros(self.ny + 1, self.nx + 1, dtype=F64, device="cuda")
        for j in range(S + 1):
            for i in range(S + 1):
                at = (slice(j, j + S * self.npy - S + 1, S), slice(i, i + S * self.npx - S + 1, S))
                cnt[at] += self.patch
                for comp in range(2):
                    tot[comp][at] += g[:, :, comp * nf + j * (S + 1) + i]
        return torch.where(self.dirichlet, x[:2], x[:2] + tot / cnt.clamp(min=1.0))

    # the Newton matrix of the level's system and the block smoother
    def newton_product(self, x, d):
        u, v = x[0], x[1]
        du, dv, dp = d
        out = [torch.zeros_like(u) for _ in range(3)]
        for w, ph, dx, dy in self._gauss():
            w = w * self.fluid
            U, V, Ux, Uy, Vx, Vy = (self._at(f, q) for f, q in ((u, ph), (v, ph), (u, dx), (u, dy), (v, dx), (v, dy)))
            a, b, ax, ay, bx, by = (self._at(f, q) for f, q in ((du, ph), (dv, ph), (du, dx), (du, dy), (dv, dx), (dv, dy)))
            pq = self._at(dp, ph)
            cu = a / DT + 0.5 * (U * ax + V * ay + a * Ux + b * Uy)
            cv = b / DT + 0.5 * (U * bx + V * by + a * Vx + b * Vy)
            for k in range(4):
                self._corner(out[0], k).add_(w * (cu * ph[k] + 0.5 * NU * (ax * dx[k] + ay * dy[k]) - pq * dx[k]))
                self._corner(out[1], k).add_(w * (cv * ph[k] + 0.5 * NU * (bx * dx[k] + by * dy[k]) - pq * dy[k]))
                self._corner(out[2], k).add_(w * (ax + by) * ph[k])
        y = torch.stack(out)
        y[2] += self.lps(dp)
        y[:2] = torch.where(self.dirichlet, d[:2], y[:2])
        y[2] = torch.where(self.p_active, y[2], dp)
        return y

    def element_matrices(self, x):
        """{(a, b, i, j): [ny+2][nx+2]} of the linearised element operator (no projection term), a ring of zeros."""
        u, v = x[0], x[1]
        E = {}
        for w, ph, dx, dy in self._gauss():
            w = w * self.fluid
            U, V, Ux, Uy, Vx, Vy = (self._at(f, q) for f, q in ((u, ph), (v, ph), (u, dx), (u, dy), (v, dx), (v, dy)))
            for a in range(4):
                for b in range(4):
                    lin = ph[a] * ph[b] / DT + 0.5 * NU * (dx[a] * dx[b] + dy[a] * dy[b])
                    nl = 0.5 * ph[a] * (U * dx[b] + V * dy[b])
                    pp = 0.5 * ph[a] * ph[b]
                    for key, val in (((0, 0), lin + nl + pp * Ux), ((0, 1), pp * Uy), ((1, 0), pp * Vx),
                                     ((1, 1), lin + nl + pp * Vy), ((0, 2), -ph[b] * dx[a]), ((1, 2), -ph[b] * dy[a]),
                                     ((2, 0), ph[a] * dx[b]), ((2, 1), ph[a] * dy[b])):
                        k = (a, b) + key
                        if k not in E:
                            E[k] = torch.zeros(self.ny + 2, self.nx + 2, dtype=F64, device="cuda")
                        E[k][1:-1, 1:-1] += w * val
        return E

    def vanka(self, x, r, d):
        E = self.element_matrices(x)
        Mc = self.lps_matrices()
        npy, npx = self.ny // 2, self.nx // 2
        S9 = torch.zeros(npy + 2, npx + 2, 9, 9, dtype=F64, device="cuda")
        for c in range(4):
            S9[1:-1, 1:-1] += self.fluid[c >> 1::2, c & 1::2][:, :, None, None] * Mc[c]
        fixed = torch.stack([self.dirichlet, self.dirichlet, ~self.p_active])
        d = d.clone()
        for cy in range(4):
            for cx in range(4):
                J, I = torch.meshgrid(torch.arange(cy, self.ny, 4, device="cuda"),
                                      torch.arange(cx, self.nx, 4, device="cuda"), indexing="ij")
                keep = self.fluid[J, I] > 0
                J, I = J[keep], I[keep]
                A = torch.zeros(J.numel(), 12, 12, dtype=F64, device="cuda")
                for (a, b, i, j), e in E.items():
                    for dj in (-1, 0, 1):
                        for di in (-1, 0, 1):
                            ra, rb, ka, kb = di + (a & 1), dj + (a >> 1), di + (b & 1), dj + (b >> 1)
                            if min(ra, rb, ka, kb) >= 0 and max(ra, rb, ka, kb) <= 1:
                                A[:, 3 * (ra + 2 * rb) + i, 3 * (ka + 2 * kb) + j] += e[J + 1 + dj, I + 1 + di]
                for n in range((cy - 1) >> 1, ((cy + 1) >> 1) + 1):
                    for m in range((cx - 1) >> 1, ((cx + 1) >> 1) + 1):
                        ids = [(cy + (a >> 1) - 2 * n, cx + (a & 1) - 2 * m) for a in range(4)]
                        S = S9[(J - cy) // 2 + n + 1, (I - cx) // 2 + m + 1]
                        for a, (ja, ia) in enumerate(ids):
                            for b, (jb, ib) in enumerate(ids):
                                if min(ia, ja, ib, jb) >= 0 and max(ia, ja, ib, jb) <= 2:
                                    A[:, 3 * a + 2, 3 * b + 2] += S[:, 3 * ja + ia, 3 * jb + ib]
                defect = r - self.newton_product(x, d)
                z = torch.zeros(J.numel(), 12, dtype=F64, device="cuda")
                for a in range(4):
                    for i in range(3):
                        z[:, 3 * a + i] = defect[i, J + (a >> 1), I + (a & 1)]
                        fx = fixed[i, J + (a >> 1), I + (a & 1)]
                        row = torch.zeros(12, dtype=F64, device="cuda")
                        row[3 * a + i] = 1.0
                        A[:, 3 * a + i] = torch.where(fx[:, None], row, A[:, 3 * a + i])
                z = _eliminate(A, z)
                for a in range(4):
                    for i in range(3):
                        d[i, J + (a >> 1), I + (a & 1)] += z[:, 3 * a + i]
        return torch.where(fixed, r, d)


def _eliminate(A, z):
    """Solutions of the systems A[n] by Gaussian elimination with partial pivoting; a vanishing pivot gives 0 there."""
    n = A.shape[0]
    M = torch.cat([A, z[:, :, None]], dim=2)
    tiny = 1e-12 * A.abs().amax(dim=(1, 2))
    at = torch.arange(n, device="cuda")
    dead = torch.zeros(n, 12, dtype=torch.bool, device="cuda")
    for k in range(12):
        piv = k + M[:, k:, k].abs().argmax(dim=1)
        rows = M[at, piv].clone()
        M[at, piv] = M[:, k]
        M[:, k] = rows
        dead[:, k] = M[:, k, k].abs() <= tiny
        unit = torch.zeros(13, dtype=F64, device="cuda")
        unit[k] = 1.0
        M[:, k] = torch.where(dead[:, k, None], unit, M[:, k])
        f = torch.where(dead[:, k, None], 0.0, M[:, k + 1:, k] / M[:, k, k, None])
        M[:, k + 1:] -= f[:, :, None] * M[:, None, k]
    x = torch.zeros(n, 12, dtype=F64, device="cuda")
    for k in range(11, -1, -1):
        x[:, k] = (M[:, k, 12] - (M[:, k, k + 1:12] * x[:, k + 1:]).sum(1)) / M[:, k, k]
    return x


def _gru(X, h, W):
    """One GRU step and the output layer: (h', d)."""
    Wx, Uh, Wfc = W
    H = h.shape[1]
    a = X @ Wx.T
    z = torch.sigmoid(a[:, :H] + h @ Uh[:H].T)
    r = torch.sigmoid(a[:, H:2 * H] + h @ Uh[H:2 * H].T)
    hn = z * h + (1.0 - z) * torch.tanh(a[:, 2 * H:] + (r * h) @ Uh[2 * H:].T)
    return hn, hn @ Wfc.T


def _dev(W):
    return [torch.as_tensor(np.asarray(w, dtype=np.float64)).cuda() for w in W]


def _exact_step(c, seed, W):
    G, xc, bf, h = _instance(c, seed)
    x = G.prolongate(xc)
    h, d = _gru(G.features(x, G.residual(x, bf.to(F64))), h.to(F64), W)
    bf = G.rhs(G.average(d, x))
    return dict(h=h, bf=bf, bc=G.restrict(bf).reshape(3, -1))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
        return _exact_step(c, seed, _dev(_weights(n_in, c["H"], n_out, seed)))
    if kind == "serve":
        nf, nc, n_in, n_out = _sizes(c["K"], 1)
        W = _dev(_weights(n_in, c["H"], n_out, seed))
        out = [_exact_step(ci, seed + 31 * i, W) for i, ci in enumerate(_serve_instances(c))]
        return [(o["h"], o["bf"], o["bc"].reshape(3, -1)) for o in out]
    if kind == "train":
        X, Y, h0, n_in, n_out = _train_inputs(c, seed)
        # PatchNetTrainer's initial weights, in FP32: N(0, 0.02^2) in the order Wx, Uh, Wfc, the last scaled to 0.05
        r = np.random.default_rng(seed % 100003)
        H, T, P = c["H"], c["T"], c["P"]
        W = [r.normal(0.0, 0.02, s) for s in ((3 * H, n_in), (3 * H, H), (n_out, H))]
        W[2] = W[2] * (0.05 / 0.02)
        W = [w.astype(np.float32) for w in W]
        W = [w.requires_grad_(True) for w in _dev(W)]
        h, D = h0.to(F64), []
        for t in range(T):
            h, d = _gru(X[t, :, :n_in].to(F64), h, W)
            D.append(d)
        D = torch.stack(D)
        loss = ((D - Y.to(F64)) ** 2).sum() / P
        loss.backward()
        return dict(loss=loss.detach(), D=D.detach(), hT=h.detach(), grads=[w.grad for w in W])
    if kind == "gru":
        nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
        W = _dev(_weights(n_in, c["H"], n_out, seed))
        X = _feature_rows(1, c["P"], c["nxc"], c["K"], c["s"], seed)
        X = X.to(torch.bfloat16) if c["prec"] == "bf16" else X
        h = torch.rand(c["P"], c["H"], device="cuda", generator=_rng(seed, 5)) - 0.5
        h, d = _gru(X.to(F64), h.to(F64), W)
        return dict(h=h, d=d)
    if kind == "windows":
        G, xc, _, _ = _instance(dict(c, H=1), seed)
        prev = _flow(G.nx, G.ny, seed + 1, (c["ax"], c["ay"]))[:2].to(torch.float32).to(F64)
        nf, nc, n_in, n_out = _sizes(c["K"], c["s"])
        d = 0.05 * torch.randn(G.P, n_out, device="cuda", generator=_rng(seed, 7))
        x, bf = G.prolongate(xc), G.rhs(prev)
        return dict(xf=x, bf=bf, X=_padded(G.features(x, G.residual(x, bf))), vc=G.average(d.to(F64), x))
    if c["nx"] * c["ny"] > 1 << 19:
        return None
    L, solid, x, r = _mg_inputs(c, seed)
    x, r = x.to(F64), r.to(F64)
    d = torch.zeros_like(r)
    for _ in range(2):
        d = L.vanka(x, r, d)
    t = r - L.newton_product(x, d)
    # the coarser level: its patches are solid where all 16 cells under them are
    f = torch.as_tensor(solid)
    sc = f.view(c["ny"] // 4, 4, c["nx"] // 4, 4).all(3).all(1).repeat_interleave(2, 0).repeat_interleave(2, 1)
    C = Grid(c["nx"] // 2, c["ny"] // 2, 0, 1, sc.numpy())
    g = t
    for _ in range(2):
        even, odd = g[..., 0::2].clone(), 0.5 * g[..., 1::2]
        even[..., :-1] += odd
        even[..., 1:] += odd
        g = even.transpose(1, 2)
    fixed = torch.stack([C.dirichlet, C.dirichlet, ~C.p_active])
    rc = torch.where(fixed, 0.0, g.contiguous())
    return dict(d=d.reshape(3, -1), t=t.reshape(3, -1), rc=rc.reshape(3, -1))
