"""The workloads whose speed is measured: what an elastic full-waveform
inversion with uncertainty quantification has the framework do, from the
smallest mesh to the 340 x 70 element benchmark mesh, through the public
entry points.

`listed()` and `draw()` give cases (plain dicts), `prepare()` what a program
holds before the call, `run()` one pass, `work()` the bytes and operations
a pass cannot do without, `exact()` the same outputs from plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2009_12663_gb300 as gb
from paper_2009_12663_gb300 import learned

DEV = "cuda:0"
AMP = 1e12                     # source amplitude (N m)
DAMP, SIGMA = 1.0, 100.0       # damping and smoothing length (m) of B0


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def sem(kind, nex, nez, h, nt, shots, nrec, f0, top=1, spl=1, streams=1, graph=0, ckpt=0, **more):
    return dict(kind=kind, nex=nex, nez=nez, h=h, nt=nt, shots=shots, nrec=nrec, f0=f0, top=top, spl=spl,
                streams=streams, graph=graph, ckpt=ckpt, **more)


def listed():
    return [
        # the smallest inversion mesh (600 m x 300 m, 15 Hz) at the default schedule: one gradient
        # of a study that runs thousands of them
        dict(sem("gradient", 12, 6, 50.0, 1500, 3, 13, 15.0), name="gradient 12x6, 3 shots"),
        # observed data of the 1000 m x 500 m model: one whole forward simulation
        dict(sem("forward", 40, 20, 25.0, 1200, 1, 41, 15.0), name="forward 40x20, 1 shot"),
        # one trial point of the line search on the benchmark mesh at the default schedule
        dict(sem("misfit", 340, 70, 50.0, 300, 24, 341, 5.0), name="misfit 340x70, 24 shots"),
        # the benchmark's gradient (its first steps): four full-history lanes replayed as graphs
        dict(sem("gradient", 340, 70, 50.0, 500, 24, 341, 5.0, streams=4, graph=1), name="gradient 340x70, lanes"),
        # the same in bounded memory: all shots in one launch, checkpoints and recomputation
        dict(sem("gradient", 340, 70, 50.0, 300, 24, 341, 5.0, spl=24, graph=1, ckpt=100),
             name="gradient 340x70, checkpoints"),
        # P4 of the experiments' model size, odd in both directions, before an inversion starts
        dict(sem("precond", 81, 21, 50.0, 800, 5, 82, 8.0, streams=4, graph=1, map=4), name="precond P4 81x21, 5 shots"),
        # search direction of the full-history BFGS late in an inversion of the benchmark model
        dict(kind="direction", n=1147323, k=50, name="direction n=1147323, 50 pairs"),
        # L-BFGS(5) on vp and vs of the 40 x 20 mesh: the store of the last pairs and its direction
        dict(kind="lbfgs", n=26082, k=5, name="L-BFGS n=26082, 5 pairs"),
        # the benchmark's uncertainty step
        dict(kind="uq", n=1147323, k=50, p=60, rank=50, form="randomized", name="UQ n=1147323, 60 probes"),
        # the exact decomposition after a short inversion of the 40 x 20 mesh (rho, vp, vs)
        dict(kind="uq", n=39123, k=20, p=0, rank=24, form="exact", name="UQ exact n=39123, 20 pairs"),
        # B0 from the learned preconditioner: features, U-Net, resampling, smoothing and inversion
        dict(sem("learned", 340, 70, 50.0, 10, 24, 341, 5.0, levels=4, base=32, height=256, width=1024),
             name="learned B0 340x70, 256x1024"),
        # one Adam step of its training at the size of the tests' maps, batch 4
        dict(kind="train", levels=4, base=32, height=32, width=128, batch=4, name="train 32x128, batch 4"),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gradient", "gradient", "forward", "misfit", "precond", "direction", "lbfgs", "uq", "learned",
                       "train"])
    if kind == "direction":
        return dict(kind=kind, n=log_int(rng, 2000, 1147323), k=rng.randint(1, 50))
    if kind == "lbfgs":
        return dict(kind=kind, n=log_int(rng, 2000, 764882), k=rng.randint(1, 8))
    if kind == "uq":
        form = rng.choice(["randomized", "twopass", "exact"])
        k = rng.randint(8, 50)
        p = rng.randint(k, min(2 * k, 60))
        return dict(kind=kind, n=log_int(rng, 5000, 1147323), k=k, p=p, rank=rng.randint(4, p), form=form)
    if kind == "train":
        return dict(kind=kind, levels=rng.randint(2, 4), base=8 * rng.randint(1, 4), height=8 * rng.randint(1, 8),
                    width=64 * rng.randint(1, 4), batch=rng.randint(1, 4))
    nex, nez = log_int(rng, 5, 340), log_int(rng, 3, 70)
    shots = rng.randint(1, 24)
    nodes = (4 * nex + 1) * (4 * nez + 1)
    budget = dict(gradient=1.0e9, precond=0.7e9).get(kind, 2.0e9)
    most = min(budget / nodes, 8000) / shots           # time steps a pass can afford
    nt = max(40, min(1500, int(most * rng.uniform(0.4, 1.0))))
    h = rng.choice([25.0, 40.0, 50.0])
    case = sem(kind, nex, nez, h, nt, shots, rng.randint(2, nex + 1), rng.choice([250.0, 400.0]) / h,
               top=rng.randint(0, 1), spl=rng.choice([1, 1, 2, 5, 24]), streams=rng.choice([1, 2, 4]),
               graph=rng.randint(0, 1))
    if kind == "gradient":
        case["ckpt"] = rng.choice([0, 0, max(8, nt // 6)])
    if kind == "precond":
        case["map"] = rng.randint(1, 4)
    if kind == "learned":
        case.update(nt=10, levels=rng.randint(2, 4), base=8 * rng.randint(1, 4), height=8 * rng.randint(4, 32),
                    width=64 * rng.randint(2, 16))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

DT = 5e-4


def generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def acquisition(case):
    """Sources 20 m deep evenly along the model, receivers at the surface."""
    L, dep = case["nex"] * case["h"], min(20.0, 0.4 * case["h"])
    src = [dict(x=L * (i + 0.5) / case["shots"], z=dep, type=0, f0=case["f0"], t0=1.2 / case["f0"], amp=AMP)
           for i in range(case["shots"])]
    rec = np.stack([np.linspace(0.0, L, case["nrec"]), np.zeros(case["nrec"])], axis=1)
    return src, rec


def gll():
    """GLL points, weights and the derivative matrix D[i][k] = l_k'(x_i) for five points."""
    a = math.sqrt(3.0 / 7.0)
    x = np.array([-1.0, -a, 0.0, a, 1.0])
    w = np.array([0.1, 49 / 90, 32 / 45, 49 / 90, 0.1])
    D = np.zeros((5, 5))
    for k in range(5):
        c = np.poly(np.delete(x, k))
        D[:, k] = np.polyval(np.polyder(c), x) / np.polyval(c, x[k])
    return x, w, D


def axis(ne, h):
    x, _, _ = gll()
    c = (np.arange(ne)[:, None] + (1 + x[None, :4]) / 2).reshape(-1)
    return np.append(c, ne) * h


def earth_model(case, seed):
    """Layered model with a fold: vp 1500 to 4500 m/s rising with depth (slower where the elements are
    small), vs = vp / 1.73, Gardner density, [3][nz][nx] on the GLL nodes."""
    g = generator(seed)
    r = torch.rand(8, generator=g, device=DEV, dtype=torch.float64)
    x = torch.tensor(axis(case["nex"], case["h"]), device=DEV) / (case["nex"] * case["h"])
    z = torch.tensor(axis(case["nez"], case["h"]), device=DEV) / (case["nez"] * case["h"])
    d = z[:, None] + (0.03 + 0.05 * r[0]) * torch.sin(2 * math.pi * ((1 + 2 * r[1]) * x[None] + r[2]))
    step = sum(torch.tanh((d - b) * 40) * a for a, b in zip(0.3 + r[3:7], (0.2, 0.4, 0.6, 0.8)))
    vp = 1500.0 + 3000.0 * (0.5 * d.clamp(0, 1) + 0.25 * (1 + step / (0.3 + r[3:7]).sum()))
    if case["h"] < 50.0:
        vp = 1500.0 + (vp - 1500.0) * 0.5
    return torch.stack([310.0 * vp ** 0.25, vp, vp / 1.73]).float().contiguous()


def observed(case, seed):
    """Observed data [shots][nrec][2][nt]: Ricker arrivals along two hyperbolas of seeded speeds."""
    g = generator(seed + 1)
    src, rec = acquisition(case)
    xs = torch.tensor([s["x"] for s in src], device=DEV)[:, None, None]
    r = (torch.tensor(rec[:, 0], device=DEV)[None, :, None] - xs).abs() + case["h"]
    t = DT * torch.arange(1, case["nt"] + 1, device=DEV)[None, None] - 1.2 / case["f0"]
    c = 1600.0 + 600.0 * torch.rand(2, generator=g, device=DEV)
    out = torch.empty(case["shots"], case["nrec"], 2, case["nt"], device=DEV)
    for comp in range(2):
        q = (math.pi * case["f0"] * (t - r / c[comp])) ** 2
        out[:, :, comp] = (50.0 / torch.sqrt(r) * (1 - 2 * q) * torch.exp(-q)).float()
    return out


def history(case, seed):
    """B0 and the pairs of a quadratic model: s ~ 1e-2 N(0, 1), y = A s with noise, A diagonal in [1, 10]."""
    g = generator(seed)
    n = case["n"]
    A = 1.0 + 9.0 * torch.rand(n, generator=g, device=DEV)
    B0 = (0.5 + 1.5 * torch.rand(n, generator=g, device=DEV)) / A
    pairs = []
    for _ in range(case["k"]):
        s = 1e-2 * torch.randn(n, generator=g, device=DEV)
        pairs.append((s, A * s + 5e-5 * torch.randn(n, generator=g, device=DEV)))
    return B0, pairs, torch.randn(n, generator=g, device=DEV)


def images(case, seed):
    """Training images: smooth random channels and maps a function of them."""
    g = generator(seed)
    H, W, b = case["height"], case["width"], case["batch"]
    low = torch.randn(b, 5, max(2, H // 8), max(2, W // 8), generator=g, device=DEV)
    x = torch.nn.functional.interpolate(low, size=(H, W), mode="bilinear", align_corners=True)
    t = torch.stack([x[:, 0] + 0.5 * x[:, 1], x[:, 1] * x[:, 2], x[:, 3] - x[:, 4]], dim=1)
    return x.contiguous(), t.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind in ("direction", "lbfgs", "uq"):
        n = case["n"]
        B0, pairs, grad = history(case, seed)
        if kind == "lbfgs":
            st.update(B0=B0, pairs=pairs, grad=grad[None].contiguous(), Z=torch.zeros(1, n, device=DEV))
            return st
        b = gb.Bfgs(n, case["k"], B0)
        for s, y in pairs:
            b.update(s, y)
        st["b"] = b
        if kind == "direction":
            st.update(grad=grad[None].contiguous(), Z=torch.zeros(1, n, device=DEV))
        else:
            st.update(V=torch.zeros(case["rank"], n, device=DEV), std=torch.zeros(n, device=DEV),
                      lam=torch.zeros(case["rank"], dtype=torch.float64, device=DEV))
        return st
    if kind == "train":
        net = gb.Unet(levels=case["levels"], base=case["base"], cin=5, cout=3, height=case["height"],
                      width=case["width"])
        net.set_params(learned.he_init(net, seed))
        st["net"] = net
        st["x"], st["t"] = images(case, seed)
        st["params"] = torch.zeros(net.num_params, device=DEV)
        return st
    src, rec = acquisition(case)
    m = gb.Mesh(case["nex"], case["nez"], case["h"], DT, case["nt"], src, rec, free_surface_top=case["top"])
    m.set_schedule(shots_per_launch=case["spl"], tile=0, use_graph=case["graph"], ckpt_every=case["ckpt"],
                   streams=case["streams"])
    model = earth_model(case, seed)
    st.update(mesh=m, model=model, ids=list(range(case["shots"])))
    shape = (case["shots"], case["nrec"], 2, case["nt"])
    if kind == "forward":
        st["seis"] = torch.zeros(shape, device=DEV)
    if kind in ("gradient", "misfit"):
        st["obs"] = observed(case, seed)
        st["grad"] = torch.zeros_like(model)
    if kind in ("precond", "learned"):
        st["H"], st["B0"] = torch.zeros_like(model), torch.zeros_like(model)
    if kind == "learned":
        net = gb.Unet(levels=case["levels"], base=case["base"], cin=5, cout=3, height=case["height"],
                      width=case["width"])
        st["lp"] = learned.LearnedPreconditioner(net, seed=seed)
        st["lp"].offset = torch.tensor([20.0, 30.0, 31.0]).reshape(3, 1, 1)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "direction":
        return st["b"].apply(st["grad"], st["Z"], gamma=0.9)
    if kind == "lbfgs":
        b = gb.Bfgs(case["n"], case["k"], st["B0"])
        for s, y in st["pairs"]:
            b.update(s, y)
        return b.apply(st["grad"], st["Z"], gamma=0.9)
    if kind == "uq":
        out = dict(V=st["V"], lam=st["lam"], std=st["std"])
        if case["form"] == "exact":
            st["b"].lowrank_exact(case["rank"], eps_prior=1.0, **out)
        elif case["form"] == "twopass":
            st["b"].lowrank_twopass(case["p"], case["rank"], seed=st["seed"], eps_prior=1.0, **out)
        else:
            st["b"].lowrank_invhess(case["p"], case["rank"], seed=st["seed"], eps_prior=1.0, **out)
        return out
    if kind == "train":
        loss = st["net"].train_step(st["x"], st["t"], 1e-4)
        return dict(loss=loss, params=st["net"].get_params(st["params"]))
    m, model = st["mesh"], st["model"]
    if kind == "learned":
        net = st["lp"].net
        ly = st["lp"].predict_log(learned.features(m, model, net.height, net.width)).contiguous()
        H = gb.resample(ly, st["H"], op=2)
        return dict(log_map=ly, B0=m.precond_from_hessian(H, SIGMA, DAMP, st["B0"]))
    m.set_model(model[0], model[1], model[2])
    if kind == "forward":
        return m.forward(st["ids"], st["seis"])
    if kind == "misfit":
        return m.misfit(st["ids"], st["obs"])
    if kind == "precond":
        m.precond_diag(st["ids"], case["map"], SIGMA, DAMP, st["H"], st["B0"])
        return dict(H=st["H"], B0=st["B0"])
    f = m.adjoint_gradient(st["ids"], st["obs"], st["grad"])
    return dict(misfit=f, grad=st["grad"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

STEP = 2300                    # operations of an element's force: 4 x 25 x 5 derivative terms, stress, 4 x 25 x 5 back
PRODUCT = 1300                 # of the strain products with the forward field (its derivatives, the products)
NODE = 12                      # of a node's update


def conv_layers(case):
    """(cout, cin, k, pixels) of every convolution of the network."""
    ch = [case["base"] << i for i in range(case["levels"])]
    px = [case["height"] * case["width"] >> (2 * i) for i in range(case["levels"])]
    out = []
    for i, c in enumerate(ch):
        out += [(c, 5 if i == 0 else ch[i - 1], 3, px[i]), (c, c, 3, px[i])]
    for i in range(case["levels"] - 2, -1, -1):
        out += [(ch[i], ch[i + 1] + ch[i], 3, px[i]), (ch[i], ch[i], 3, px[i])]
    return out + [(3, ch[0], 1, px[0])]


def work(case):
    kind = case["kind"]
    if kind in ("direction", "lbfgs"):
        n, k = case["n"], case["k"]
        pairs = 2 * k                                    # S and B0 Y (L-BFGS: S and Y, given with the call)
        return dict(bytes=4.0 * n * (pairs + 3), flops=2.0 * n * (2 * pairs + 1))
    if kind == "uq":
        n, k, r = case["n"], case["k"], case["rank"]
        p = 0 if case["form"] == "exact" else case["p"]
        return dict(bytes=4.0 * n * (2 * k + r + 2), flops=2.0 * n * (2 * k * p + 2 * k * r + 2 * r))
    if kind == "train":
        conv = sum(2.0 * o * i * k * k * px for o, i, k, px in conv_layers(case))
        par = sum(o * i * k * k for o, i, k, _ in conv_layers(case))
        px = case["height"] * case["width"]
        return dict(bytes=4.0 * (8 * case["batch"] * px + 7 * par), flops=3.0 * case["batch"] * conv)
    el, nodes = case["nex"] * case["nez"], (4 * case["nex"] + 1) * (4 * case["nez"] + 1)
    if kind == "learned":
        conv = sum(2.0 * o * i * k * k * px for o, i, k, px in conv_layers(case))
        return dict(bytes=4.0 * (6 * nodes + 3 * case["height"] * case["width"]), flops=conv)
    steps = float(case["shots"] * case["nt"])
    fwd = steps * (STEP * el + NODE * nodes)
    data = 4.0 * steps * case["nrec"] * 2
    if kind in ("forward", "misfit"):
        return dict(bytes=data + 12.0 * nodes, flops=fwd)
    if kind == "precond" and case["map"] in (1, 3):
        return dict(bytes=36.0 * nodes, flops=fwd + steps * PRODUCT * el)
    both = 2 * fwd + steps * (PRODUCT * el + 6 * nodes)
    return dict(bytes=data + 24.0 * nodes, flops=both)


# ---------------------------------------------------------------------------
# the same in FP64
# ---------------------------------------------------------------------------

class Sem64:
    """The spectral-element scheme on whole fields [shot][2][nz][nx]: Newmark (beta 0, gamma 1/2) with
    implicit first-order Stacey edges, and its discrete adjoint."""

    def __init__(self, case, model):
        self.case = case
        nex, nez, h = case["nex"], case["nez"], case["h"]
        self.nx, self.nz = 4 * nex + 1, 4 * nez + 1
        self.xi, w, D = gll()
        t64 = lambda a: torch.tensor(np.asarray(a, np.float64), device=DEV)  # noqa: E731
        self.D, self.w2 = t64(D), t64(np.outer(w, w))
        wx, wz = np.zeros(self.nx), np.zeros(self.nz)
        for n, v in ((nex, wx), (nez, wz)):
            for e in range(n):
                v[4 * e:4 * e + 5] += w * h / 2
        self.wx, self.wz = t64(wx), t64(wz)
        rho, vp, vs = model.double()
        self.rho, self.vp, self.vs = rho, vp, vs
        mu = rho * vs * vs
        self.lam, self.mu = self.elements(rho * vp * vp - 2 * mu), self.elements(mu)
        W = self.wz[:, None] * self.wx[None]
        wn, wt = torch.zeros(2, self.nz, self.nx, device=DEV, dtype=torch.float64), None
        wt = torch.zeros_like(wn)
        for ix in (0, self.nx - 1):
            wn[0, :, ix] += self.wz
            wt[1, :, ix] += self.wz
        for iz in ((self.nz - 1,) if case["top"] else (0, self.nz - 1)):
            wn[1, iz] += self.wx
            wt[0, iz] += self.wx
        self.wn, self.wt, self.W = wn, wt, W
        self.C = rho * vp * wn + rho * vs * wt
        self.inv = 1.0 / (rho * W + 0.5 * DT * self.C)
        src, rec = acquisition(case)
        self.sources = src
        self.rx, self.rz = self.point(rec[:, 0], nex), self.point(rec[:, 1], nez)

    def point(self, x, ne):
        """First node and Lagrange weights (and derivatives) of points along one axis."""
        h = self.case["h"]
        e = np.clip(np.ceil(np.asarray(x) / h).astype(int) - 1, 0, ne - 1)
        s = 2 * (np.asarray(x) - e * h) / h - 1
        val, der = np.zeros((len(e), 5)), np.zeros((len(e), 5))
        for k in range(5):
            c = np.poly(np.delete(self.xi, k))
            c = c / np.polyval(c, self.xi[k])
            val[:, k], der[:, k] = np.polyval(c, s), np.polyval(np.polyder(c), s) * 2 / h
        return 4 * e, val, der

    def elements(self, f):
        """Node field [...][nz][nx] -> element view [...][nez][nex][5][5]."""
        f = f.contiguous()
        st = f.stride()
        return f.as_strided(f.shape[:-2] + (self.case["nez"], self.case["nex"], 5, 5),
                            st[:-2] + (4 * self.nx, 4, self.nx, 1))

    def assemble(self, e):
        lead, nez, nex = e.shape[:-4], e.shape[-4], e.shape[-3]
        rows = e.new_zeros(lead + (nez, 5, self.nx))
        rows[..., :-1].view(lead + (nez, 5, nex, 4))[:] = e[..., :4].transpose(-3, -2)
        rows[..., 4::4] += e[..., 4].transpose(-2, -1)
        out = e.new_zeros(lead + (self.nz, self.nx))
        out[..., :-1, :].view(lead + (nez, 4, self.nx))[:] = rows[..., :4, :]
        out[..., 4::4, :] += rows[..., 4, :]
        return out

    def strains(self, u):
        e = self.elements(u)
        dx, dz = e @ self.D.T, self.D @ e
        return dx[:, 0], dz[:, 1], dz[:, 0] + dx[:, 1]

    def stiffness(self, u):
        xx, zz, g = self.strains(u)
        txx = self.w2 * ((self.lam + 2 * self.mu) * xx + self.lam * zz)
        tzz = self.w2 * (self.lam * xx + (self.lam + 2 * self.mu) * zz)
        txz = self.w2 * self.mu * g
        return self.assemble(torch.stack([txx @ self.D + self.D.T @ txz, txz @ self.D + self.D.T @ tzz], dim=1))

    def source_field(self, shots):
        f = torch.zeros(len(shots), 2, self.nz, self.nx, device=DEV, dtype=torch.float64)
        stf = np.zeros((len(shots), self.case["nt"] + 1))
        for q, i in enumerate(shots):
            s = self.sources[i]
            ix, lx, dx = self.point([s["x"]], self.case["nex"])
            iz, lz, dz = self.point([s["z"]], self.case["nez"])
            sl = (slice(iz[0], iz[0] + 5), slice(ix[0], ix[0] + 5))
            f[q, 0][sl] = torch.tensor(np.outer(lz[0], dx[0]), device=DEV)
            f[q, 1][sl] = torch.tensor(np.outer(dz[0], lx[0]), device=DEV)
            a = (math.pi * s["f0"] * (DT * np.arange(self.case["nt"] + 1) - s["t0"])) ** 2
            stf[q] = s["amp"] * (1 - 2 * a) * np.exp(-a)
        return f, torch.tensor(stf, device=DEV)

    def receivers(self):
        ix, lx, _ = self.rx
        iz, lz, _ = self.rz
        nodes = (iz[:, None, None] + np.arange(5)[:, None]) * self.nx + ix[:, None, None] + np.arange(5)
        return (torch.tensor(nodes.reshape(len(ix), 25), device=DEV),
                torch.tensor((lz[:, :, None] * lx[:, None, :]).reshape(len(ix), 25), device=DEV))

    def step(self, u, v, F):
        a = (F - self.stiffness(u) - self.C * v) * self.inv
        vn = v + DT * a
        return a, vn, u + DT * vn

    def forward(self, shots, keep=None, each=None):
        """Seismograms [shot][nrec][2][nt]; keep: list that receives u_0, u_1, ..; each(n, u_n, u_{n+1}, a)."""
        nt = self.case["nt"]
        f, stf = self.source_field(shots)
        at, wr = self.receivers()
        u0, u, v = torch.zeros_like(f), torch.zeros_like(f), torch.zeros_like(f)
        out = torch.empty(len(shots), 2, self.case["nrec"], nt, device=DEV, dtype=torch.float64)
        if keep is not None:
            keep += [u0, u]
        for n in range(nt):
            out[..., n] = (u.flatten(2)[:, :, at] * wr).sum(-1)
            a, v, nxt = self.step(u, v, f * stf[:, n + 1, None, None, None])
            if each:
                each(u0, u, a)
            u0, u = u, nxt
            if keep is not None:
                keep.append(u)
        return out.transpose(1, 2)

    def adjoint(self, signal, each):
        """The recurrence driven by P^T signal reversed in time; each(k, w, w_next, a, v) with the level k
        of the forward field that it meets."""
        nt, (at, wr) = self.case["nt"], self.receivers()
        w0 = torch.zeros(signal.shape[0], 2, self.nz, self.nx, device=DEV, dtype=torch.float64)
        w, v = torch.zeros_like(w0), torch.zeros_like(w0)
        for j in range(nt):
            F = torch.zeros_like(w0)
            s = signal[..., nt - 1 - j].transpose(1, 2)[..., None] * wr / DT
            F.flatten(2).index_add_(2, at.reshape(-1), s.flatten(2))
            a, vn, nxt = self.step(w, v, F)
            each(nt - j, w0, w, a, 0.5 * (v + vn))
            w0, w, v = w, nxt, vn

    def groups(self, levels):
        per = max(1, int(30e9 / (levels * 16.0 * self.nx * self.nz)))
        ids = list(range(self.case["shots"]))
        return [ids[i:i + per] for i in range(0, len(ids), per)]

    def misfit_gradient(self, obs):
        tot = torch.zeros(5, self.nz, self.nx, device=DEV, dtype=torch.float64)
        f = 0.0
        for ids in self.groups(self.case["nt"] + 2):
            u = []
            r = self.forward(ids, keep=u) - obs[ids].double()
            f += 0.5 * DT * float((r * r).sum())

            def meet(k, w0, w, a, v):
                ax, az, ag = self.strains(u[k])
                bx, bz, bg = self.strains(w)
                tot[0] += self.assemble(self.w2 * (ax + az) * (bx + bz)).sum(0)
                tot[1] += self.assemble(self.w2 * (2 * ax * bx + 2 * az * bz + ag * bg)).sum(0)
                tot[2] += (u[k] * a).sum((0, 1))
                tot[3] += (self.wn * u[k] * v).sum((0, 1))
                tot[4] += (self.wt * u[k] * v).sum((0, 1))
            self.adjoint(r, meet)
        gl, gm, ga, gp, gs = tot
        r, p, s = self.rho, self.vp, self.vs
        grad = torch.stack([gl * (p * p - 2 * s * s) + gm * s * s + self.W * ga + gp * p + gs * s,
                            2 * gl * r * p + gp * r, -4 * gl * r * s + 2 * gm * r * s + gs * r])
        return f, -DT * DT * grad

    def precond(self, kind):
        S = torch.zeros(4, self.nz, self.nx, device=DEV, dtype=torch.float64)

        def add(first, A, B):
            ax, az, ag = self.strains(A)
            bx, bz, bg = (ax, az, ag) if B is A else self.strains(B)
            S[0] += first.sum((0, 1))
            for q, v in enumerate(((ax + az) * (bx + bz), ax * bx + az * bz, ag * bg)):
                S[q + 1] += self.assemble(self.w2 * v).sum(0) / DT
        receiver = kind in (2, 4)
        for ids in self.groups(self.case["nt"] + 2 if receiver else 4):
            if not receiver:
                def square(u0, u, a):
                    d = u - u0
                    add(a * a * DT, d, d)
                self.forward(ids, each=square)
            else:
                u = []
                syn = self.forward(ids, keep=u)
                self.adjoint(syn, lambda k, w0, w, a, v: add((u[k + 1] - 2 * u[k] + u[k - 1]) * a / DT,
                                                             u[k + 1] - u[k], w - w0))
        H = (self.W * S[0].abs()).repeat(3, 1, 1)
        if kind >= 3:
            r2, p2, s2 = self.rho ** 2, self.vp ** 2, self.vs ** 2
            H[1] = 8 * r2 * p2 * S[1].abs()
            H[2] = 16 * r2 * s2 * S[2].abs() + 4 * r2 * s2 * S[3].abs()
        return H

    def invert_map(self, H):
        def smooth(f, c, w):
            d = c[:, None] - c[None]
            G = torch.exp(-d * d / (2 * SIGMA ** 2)) * w[None] * (d.abs() <= 5 * SIGMA)
            return f @ (G / G.sum(1, keepdim=True)).T
        cx = torch.tensor(axis(self.case["nex"], self.case["h"]), device=DEV)
        cz = torch.tensor(axis(self.case["nez"], self.case["h"]), device=DEV)
        S = smooth(smooth(H, cx, self.wx).transpose(1, 2), cz, self.wz).transpose(1, 2)
        return 1 / (S + DAMP * S.flatten(1).median(1).values[:, None, None])


def two_loop(B0, pairs, g, gamma):
    q, al = g.double().clone(), []
    for s, y in reversed(pairs):
        s, y = s.double(), y.double()
        al.append((s @ q) / (y @ s))
        q -= al[-1] * y
    z = gamma * B0.double() * q
    for (s, y), a in zip(pairs, reversed(al)):
        s, y = s.double(), y.double()
        z += (a - (y @ z) / (y @ s)) * s
    return z


def philox_normals(total, seed):
    """Standard normals from Philox4x32-10 (counter: element / 4) by Box-Muller on 24-bit uniforms."""
    M32 = 0xFFFFFFFF

    def mul(a, b):
        return (a * (b >> 16) + ((a * (b & 0xFFFF)) >> 16)) >> 16, (a * b) & M32
    blk = torch.arange((total + 3) // 4, device=DEV)
    c = [blk & M32, blk >> 32, torch.zeros_like(blk), torch.zeros_like(blk)]
    k0, k1 = seed & M32, seed >> 32
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    out = []
    for a, b in ((c[0], c[1]), (c[2], c[3])):
        r = torch.sqrt(-2 * torch.log(((a >> 8) + 1).double() / 2 ** 24))
        t = 2 * math.pi * (b >> 8).double() / 2 ** 24
        out += [r * torch.cos(t), r * torch.sin(t)]
    return torch.stack(out, 1).reshape(-1)[:total]


def decomposition(case, seed):
    """Eigenvalues of the low-rank part and the posterior std; eigenvectors are free in sign: no value."""
    B0, pairs, _ = history(case, seed)
    k, n = case["k"], case["n"]
    S = torch.stack([s for s, _ in pairs]).double()
    Y = torch.stack([y for _, y in pairs]).double()
    B = B0.double()
    R = (S @ Y.T).triu()
    Ri = torch.linalg.inv(R)
    M = torch.zeros(2 * k, 2 * k, device=DEV, dtype=torch.float64)
    M[:k, :k] = Ri.T @ (torch.diag(R.diag()) + (Y * B) @ Y.T) @ Ri
    M[:k, k:], M[k:, :k] = -Ri.T, -Ri
    Wm = torch.cat([S, B * Y])
    del S, Y
    if case["form"] == "exact":
        L = torch.linalg.cholesky(Wm @ Wm.T)
        Q = torch.linalg.solve_triangular(L, Wm, upper=False)
        Om = L.T @ M @ L
    else:
        X = philox_normals(case["p"] * n, seed).reshape(case["p"], n)
        E = (M @ (Wm @ X.T)).T @ Wm
        L = torch.linalg.cholesky(E @ E.T)
        Q = torch.linalg.solve_triangular(L, E, upper=False)
        if case["form"] == "twopass":
            QW = Q @ Wm.T
            Om = QW @ M @ QW.T
        else:
            Om = torch.linalg.solve((Q @ X.T).T, (Q @ E.T).T).T
        del X, E
    lam, U = torch.linalg.eigh(0.5 * (Om + Om.T))
    at = lam.abs().argsort(descending=True)[:case["rank"]]
    lam, V = lam[at], U[:, at].T @ Q
    std = torch.sqrt(((lam[:, None] * V * V).sum(0) + B).clamp(min=0))
    full = torch.zeros(case["rank"], device=DEV, dtype=torch.float64)
    full[:len(lam)] = lam
    return dict(V=None, lam=full, std=std)


def net64(case, params, x):
    """The U-Net on x [b][5][H][W] with FP64 parameters [(W, b), ..]."""
    F = torch.nn.functional
    it = iter(params)

    def conv(h, relu=True):
        W, b = next(it)
        h = F.conv2d(h, W, b, padding=W.shape[-1] // 2)
        return h.relu() if relu else h
    skips, h = [], x
    for i in range(case["levels"]):
        h = conv(conv(F.avg_pool2d(h, 2) if i else h))
        skips.append(h)
    for i in range(case["levels"] - 2, -1, -1):
        h = conv(conv(torch.cat([F.interpolate(h, scale_factor=2, mode="nearest"), skips[i]], 1)))
    return conv(h, relu=False)


def net_params(case, seed):
    """He-normal weights of the seed (numpy's PCG64, layer by layer), zero biases."""
    rng = np.random.default_rng(seed)
    out = []
    for o, i, k, _ in conv_layers(case):
        w = (rng.standard_normal((o, i, k, k)) * np.sqrt(2.0 / (i * k * k))).astype(np.float32)
        out.append((torch.tensor(w, device=DEV).double(), torch.zeros(o, device=DEV, dtype=torch.float64)))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("direction", "lbfgs"):
        B0, pairs, g = history(case, seed)
        return two_loop(B0, pairs, g, 0.9)[None]
    if kind == "uq":
        return decomposition(case, seed)
    if kind == "train":
        par = [(w.requires_grad_(), b.requires_grad_()) for w, b in net_params(case, seed)]
        x, t = images(case, seed)
        loss = ((net64(case, par, x.double()) - t.double()) ** 2).mean()
        loss.backward()
        flat = []
        for w, b in par:                                 # the first Adam step moves by lr g / (|g| + eps)
            w, b = (v.detach() - 1e-4 * v.grad / (v.grad.abs() + 1e-8) for v in (w, b))
            kc = w[0].numel()
            flat.append(torch.nn.functional.pad(w.flatten(1), (0, -kc % 8, 0, -len(w) % 8)).reshape(-1))
            flat.append(torch.nn.functional.pad(b, (0, -len(b) % 8)))
        return dict(loss=float(loss), params=torch.cat(flat))
    model = earth_model(case, seed)
    s = Sem64(case, model)
    if kind == "learned":
        sx = torch.tensor([[q["x"], q["z"]] for q in s.sources], device=DEV, dtype=torch.float64)
        rx = torch.tensor(acquisition(case)[1], device=DEV)
        cx = torch.tensor(axis(case["nex"], case["h"]), device=DEV)
        cz = torch.tensor(axis(case["nez"], case["h"]), device=DEV)
        ch = [s.vp / 4700, s.vs / 2700, s.rho / 2500]
        for pts in (sx, rx):
            e = 2 * learned.MASK_SIGMA_M ** 2
            g = torch.exp(-(cz[:, None] - pts[:, 1]) ** 2 / e) @ torch.exp(-(cx[:, None] - pts[:, 0]) ** 2 / e).T
            ch.append(g / g.max())
        up = lambda f, size: torch.nn.functional.interpolate(  # noqa: E731
            f[None], size=size, mode="bilinear", align_corners=True)[0]
        x = up(torch.stack(ch), (case["height"], case["width"]))
        ly = net64(case, net_params(case, seed), x[None])[0]
        ly = ly + torch.tensor([20.0, 30.0, 31.0], device=DEV).double().reshape(3, 1, 1)
        return dict(log_map=ly, B0=s.invert_map(torch.exp(up(ly, (s.nz, s.nx)))))
    if kind == "forward":
        return s.forward(list(range(case["shots"])))
    if kind == "misfit":
        f = 0.0
        obs = observed(case, seed).double()
        for ids in s.groups(4):
            f += 0.5 * DT * float(((s.forward(ids) - obs[ids]) ** 2).sum())
        return f
    if kind == "precond":
        H = s.precond(case["map"])
        return dict(H=H, B0=s.invert_map(H))
    f, g = s.misfit_gradient(observed(case, seed))
    return dict(misfit=f, grad=g)
