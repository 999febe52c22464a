"""Performance cases of the upscaled lattice Boltzmann library.

Each case is one call, or the short sequence of calls, that a user's program makes through the
public entry points: fine-grid time stepping in two and three dimensions, the coarse run, the
batched local problems that give K*, and the surrogate's inference and training. ``exact`` states
the same results in 64-bit torch, written from the equations (Eqs. 2, 6, 13, 15, 16, 17, 18),
where that takes seconds; the runs to a tolerance take up to 200,000 steps and have none.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1312_0195_gb300 as lbm
import synth

STORAGE = {"f32": lbm.LBM_F32, "f16": lbm.LBM_F16, "f64": lbm.LBM_F64}
ELEM = {"f32": 4, "f16": 2, "f64": 8}
G0 = 1e-6                      # body force of every workload, lattice units

# Largest work of one pass by path, the listed cases' own: lattice updates (fine grids), field cells
# (local problems), leaves (inference), samples (training).
MAX_LUP2 = 4096 * 4096 * 256
MAX_LUP3 = 256 ** 3 * 64


def listed():
    return [
        # the channel of Section 4.1's kind with bounce-back walls: the smallest grid in the tests, stepped
        # to a check interval at a time; launches and latency count
        dict(name="channel_128x64_f32", path="fine", nx=128, ny=64, storage="f32", walls=True, tau=1.0, steps=1024,
             check=64, guo=False, force=False, ell=8.0, sigma=1.0),
        # a mid-size lattice with odd sides: no aligned rows
        dict(name="fine_517x389_f32", path="fine", nx=517, ny=389, storage="f32", walls=False, tau=0.8, steps=512,
             check=128, guo=False, force=False, ell=16.0, sigma=1.5),
        # the headline fine-grid run
        dict(name="fine_4096_f32", path="fine", nx=4096, ny=4096, storage="f32", walls=False, tau=0.6, steps=256,
             check=64, guo=False, force=False, ell=32.0, sigma=2.0),
        # the same lattice with FP16 scaled storage, the option for larger fields
        dict(name="fine_4096_f16", path="fine", nx=4096, ny=4096, storage="f16", walls=False, tau=0.6, steps=256,
             check=64, guo=False, force=False, ell=32.0, sigma=2.0),
        # FP64 runs: the paper's 1000 x 1000 lattice (Section 4.2), where FP32 conditioning is too poor
        dict(name="fine_1000_f64", path="fine", nx=1000, ny=1000, storage="f64", walls=False, tau=0.6, steps=128,
             check=64, guo=False, force=False, ell=16.0, sigma=1.0),
        # the coarse run of the upscaled method: a 4096^2 field in 16 x 16 blocks
        dict(name="coarse_256", path="coarse", nx=256, ny=256, block=16, steps=1250, force=False),
        # K* of a quadtree's leaves (8 to 64 cells) to the tolerance, the method's main cost
        dict(name="leaves_quadtree_1536", path="leaves", field=1536, tree=3, kind="lognormal", ell=32.0, sigma=2.0,
             storage="f32", tol=1e-8, max_steps=200000),
        # K* of every 16 x 16 block of a channelised field
        dict(name="blocks16_2048", path="blocks", nx=2048, ny=2048, block=16, margin=0, tol=1e-8, max_steps=200000),
        # surrogate inference on a quadtree's leaves: planes, the ensemble's forward pass, the Darcy base
        dict(name="predict_quadtree_1024", path="predict", field=1024, tree=3, ell=16.0, sigma=1.5, models=4),
        # one epoch of surrogate training with the mini-batch the benchmark uses
        dict(name="train_4096", path="train", samples=4096, batch=256, models=4),
        # the D3Q19 fine grid
        dict(name="fine3d_256_f32", path="fine3d", nx=256, ny=256, nz=256, storage="f32", steps=64, ell=8.0, sigma=1.0),
        # 3-D K* of 16^3 cubes to the tolerance
        dict(name="cubes16_128", path="cubes", field=128, size=16, margin=0, sigma=1.0, storage="f32", tol=1e-8,
             max_steps=200000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["fine", "fine", "fine", "coarse", "leaves", "blocks", "predict", "train", "fine3d", "cubes"])
    if path == "fine":
        storage = rng.choice(["f32", "f32", "f16", "f64"])
        nx, ny = _log(rng, 48, 4096), _log(rng, 48, 4096)
        if rng.random() < 0.5:                       # half of the lattices have aligned rows
            nx = max(8, nx // 8 * 8)
        cells = nx * ny * (8 if storage == "f64" else 1)
        steps = max(16, min(1024, MAX_LUP2 // 4 // cells))
        return dict(path="fine", nx=nx, ny=ny, storage=storage, walls=rng.random() < 0.3,
                    tau=rng.choice([0.6, 0.8, 1.0]), steps=steps + rng.randrange(16), check=rng.choice([0, 64, 100]),
                    guo=rng.random() < 0.15, force=rng.random() < 0.2, ell=rng.choice([4.0, 8.0, 16.0]),
                    sigma=rng.choice([0.5, 1.0, 2.0]))
    if path == "coarse":
        nx, ny = _log(rng, 16, 1024), _log(rng, 16, 1024)
        steps = max(64, min(2000, MAX_LUP2 // 16 // (nx * ny)))
        return dict(path="coarse", nx=nx, ny=ny, block=rng.choice([8, 16, 32]), steps=steps, force=rng.random() < 0.5)
    if path == "leaves":
        if rng.random() < 0.5:                       # a fixed number of steps, any leaf size
            return dict(path="leaves", field=rng.choice([256, 384, 512]), tree=rng.randrange(1000),
                        kind=rng.choice(["lognormal", "ragged"]), ell=rng.choice([4.0, 8.0, 16.0]),
                        sigma=rng.choice([0.5, 1.0, 2.0]), storage=rng.choice(["f32", "f32", "f64"]), tol=0.0, max_steps=_log(rng, 100, 2000))
        return dict(path="leaves", field=rng.choice([192, 256, 512, 768]), tree=rng.randrange(1000),
                    kind="lognormal", ell=rng.choice([8.0, 16.0, 32.0]), sigma=rng.choice([0.5, 1.0, 2.0]),
                    storage="f32", tol=1e-8, max_steps=200000)
    if path == "blocks":
        block = rng.choice([8, 12, 16, 24, 32])
        n = max(2, _log(rng, 128, 1024) // block) * block
        return dict(path="blocks", nx=n, ny=n, block=block, margin=rng.choice([0, 0, 2, 4]), tol=1e-8,
                    max_steps=20000)
    if path == "predict":
        return dict(path="predict", field=rng.choice([128, 256, 512, 768, 1024]), tree=rng.randrange(1000),
                    ell=rng.choice([4.0, 8.0, 16.0]), sigma=rng.choice([0.5, 1.0, 2.0]), models=rng.choice([1, 2, 4]))
    if path == "train":
        return dict(path="train", samples=_log(rng, 256, 3000), batch=rng.choice([64, 100, 256]),
                    models=rng.choice([1, 2]))
    if path == "fine3d":
        nx, ny, nz = (_log(rng, 16, 256) for _ in range(3))
        storage = rng.choice(["f32", "f32", "f16", "f64"])
        cells = nx * ny * nz * (8 if storage == "f64" else 1)
        return dict(path="fine3d", nx=nx, ny=ny, nz=nz, storage=storage,
                    steps=max(8, min(256, MAX_LUP3 // 4 // cells)), ell=4.0, sigma=rng.choice([0.5, 1.0]))
    size = rng.choice([8, 12, 16])
    return dict(path="cubes", field=size * rng.choice([2, 3, 4]), size=size, margin=rng.choice([0, 0, 2]),
                sigma=rng.choice([0.5, 1.0]), storage="f32", tol=1e-8, max_steps=20000)


# ------------------------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _lognormal(shape, ell, sigma, seed, k0=1e-2):
    """Periodic log-normal permeability k0 exp(sigma Z), Z with covariance exp(-r^2 / (2 ell^2)):
    float32 on the GPU."""
    z = torch.randn(shape, generator=_gen(seed), device="cuda", dtype=torch.float32)
    k2 = torch.zeros([1] * len(shape), device="cuda")
    for d, n in enumerate(shape):
        k = 2.0 * math.pi * (torch.fft.rfftfreq(n) if d == len(shape) - 1 else torch.fft.fftfreq(n)).cuda()
        k2 = k2 + (k * k).reshape([-1 if i == d else 1 for i in range(len(shape))])
    z = torch.fft.irfftn(torch.fft.rfftn(z) * torch.exp(-0.25 * ell * ell * k2), s=shape)
    z = (z - z.mean()) / z.std()
    return (k0 * torch.exp(sigma * z)).contiguous()


def _ragged_leaves(n, seed):
    """Leaves of every side from 1 to 40 cells at seeded places of an n x n field."""
    r = np.random.Generator(np.random.PCG64(int(seed)))
    size = np.arange(1, 41)
    return np.stack([r.integers(0, n - size + 1), r.integers(0, n - size + 1), size], axis=1).astype(np.int32)


def _force_field(nx, ny):
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny
    gx = torch.sin(math.pi * x).expand(ny, nx)
    gy = torch.sin(math.pi * y)[:, None].expand(ny, nx)
    return (G0 * torch.stack([gx, gy])).float().contiguous()


def _coarse_tensors(nx, ny, seed):
    """Symmetric positive definite K* per coarse cell, [ny, nx, 4] float64 (fine lattice units)."""
    kx = _lognormal((ny, nx), 2.0, 1.0, seed).double()
    ky = _lognormal((ny, nx), 2.0, 1.0, seed + 1).double()
    c = 0.3 * torch.rand((ny, nx), generator=_gen(seed + 2), device="cuda", dtype=torch.float64) * torch.sqrt(kx * ky)
    return torch.stack([kx, c, c, ky], dim=-1).contiguous()


def _leaf_field(case, seed):
    n = case["field"]
    kappa = _lognormal((n, n), case["ell"], case["sigma"], seed)
    tree = case["tree"]                                 # the mesh is the case's, the field the seed's
    leaves = _ragged_leaves(n, tree) if case.get("kind") == "ragged" else synth.quadtree_leaves(n, n, tree)
    return kappa, leaves


def _weights(models, seed):
    """Network parameters per model in the library's layout (six 3x3 convolutions, a linear head)."""
    g = torch.Generator().manual_seed(int(seed) * 31 + 5)
    out = []
    for _ in range(models):
        p, cin = [], lbm.SURROGATE_PLANES
        for cout in (32, 32, 64, 64, 64, 64):
            p.append(torch.randn(cout * cin * 9, generator=g) * math.sqrt(2.0 / (9 * cin)))
            p.append(torch.randn(cout, generator=g) * 0.05)
            cin = cout
        p += [torch.randn(128, generator=g) / 8.0, torch.randn(2, generator=g) * 0.05]
        out.append(torch.cat(p).numpy())
    return out


# a trained ensemble's normalisation: log-K shift and scale, target means and deviations, wide
# statistics bounds, the Darcy target base (mode 3)
_NORM = np.array([-4.6, 1.5, -0.01, 0.06, -0.01, 0.06, -1e30, 1e30, -1e30, 1e30, -1e30, 1e30, 3.0], dtype=np.float32)


def _params2(case):
    return lbm.Params(nx=case["nx"], ny=case["ny"], tau=case["tau"], gx=0.0 if case["force"] else G0,
                      gy=0.0 if case["force"] else 0.25 * G0,
                      bc=lbm.LBM_BC_WALLS_Y if case["walls"] else lbm.LBM_BC_PERIODIC,
                      storage=STORAGE[case["storage"]],
                      force_model=1 if case["guo"] else 0)


def prepare(case, seed):
    path = case["path"]
    s = dict(case=case)
    if path == "fine":
        kappa = _lognormal((case["ny"], case["nx"]), case["ell"], case["sigma"], seed)
        force = _force_field(case["nx"], case["ny"]) if case["force"] else None
        s["grid"] = lbm.Grid(_params2(case), kappa, force)
    elif path == "coarse":
        b = case["block"]
        s["params"] = lbm.Params(nx=case["nx"] * b, ny=case["ny"] * b, tau=1.0, gx=0.0 if case["force"] else G0)
        s["keff"] = _coarse_tensors(case["nx"], case["ny"], seed)
        s["force"] = _force_field(case["nx"], case["ny"]) if case["force"] else None
        s["out"] = [torch.empty((case["ny"], case["nx"]), device="cuda") for _ in range(3)]
    elif path == "leaves":
        s["kappa"], leaves = _leaf_field(case, seed)
        s["leaves"] = torch.from_numpy(leaves).cuda()
        s["params"] = lbm.Params(nx=case["field"], ny=case["field"], tau=1.0, storage=STORAGE[case["storage"]])
    elif path == "blocks":
        nx, ny, b = case["nx"], case["ny"], case["block"]
        s["kappa"] = torch.from_numpy(synth.channel_kappa(nx, ny, seed)).cuda()
        s["params"] = lbm.Params(nx=nx, ny=ny, tau=1.0, margin=case["margin"])
        s["keff"] = torch.empty((ny // b, nx // b, 4), dtype=torch.float64, device="cuda")
    elif path == "predict":
        s["kappa"], leaves = _leaf_field(case, seed)
        s["leaves"] = torch.from_numpy(leaves).cuda()
        s["net"] = lbm.Surrogate(case["models"], seed)
        for m, w in enumerate(_weights(case["models"], seed)):
            s["net"].set_params(m, w)
        s["net"].set_normalization(_NORM)
    elif path == "train":
        n = case["samples"]
        kappa = _lognormal((512, 512), 8.0, 1.0, seed)
        r = np.random.Generator(np.random.PCG64(int(seed)))
        size = r.choice([8, 16, 32, 64], n)
        at = [r.integers(0, 512 // size) * size for _ in range(2)]
        leaves = torch.from_numpy(np.stack([*at, size], axis=1).astype(np.int32)).cuda()
        s["x"], s["stats"] = lbm.lbm_patches(kappa, leaves)
        mean = s["x"][:, :4].mean(dim=(1, 2, 3))
        noise = 0.1 * torch.randn((n, 2), generator=_gen(seed), device="cuda")
        s["y"] = (mean[:, None] + noise).contiguous()
        s["net"] = lbm.Surrogate(case["models"], seed)
    elif path == "fine3d":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        kappa = _lognormal((nz, ny, nx), case["ell"], case["sigma"], seed)
        s["grid"] = lbm.Grid3D(lbm.Params3D(nx=nx, ny=ny, nz=nz, tau=0.8, gx=G0, storage=STORAGE[case["storage"]]), kappa)
    else:
        n, b = case["field"], case["size"]
        s["kappa"] = _lognormal((n, n, n), 8.0, case["sigma"], seed)
        k = torch.arange(0, n, b, dtype=torch.int32)
        z, y, x = torch.meshgrid(k, k, k, indexing="ij")
        corner = torch.stack([x.ravel(), y.ravel(), z.ravel()], dim=1)
        s["leaves"] = torch.nn.functional.pad(corner, (0, 1), value=b).contiguous().cuda()
        s["params"] = lbm.Params3D(nx=n, ny=n, nz=n, tau=1.0, storage=STORAGE[case["storage"]], margin=case["margin"])
    return s


# --------------------------------------------------------------------------------------- runs

def run(s):
    case = s["case"]
    path = case["path"]
    if path == "fine":
        steps, resid, _ = s["grid"].step(case["steps"], 0.0, case["check"])
        rho, u, v = s["grid"].fields()
        return dict(rho=rho, u=u, v=v, steps=steps, resid=resid)
    if path == "coarse":
        rho, u, v = s["out"]
        _, steps = lbm.lbm_coarse_run(s["params"], case["block"], s["keff"], s["force"], max_steps=case["steps"],
                                      tol_rel=0.0, check_every=64, rho=rho, u=u, v=v)
        return dict(rho=rho, u=u, v=v, steps=steps)
    if path == "leaves":
        keff, status, steps, _ = lbm.local_keff(s["params"], s["kappa"], s["leaves"], G0, case["tol"],
                                                case["max_steps"], 64)
        return dict(keff=keff, status=status, steps=steps)
    if path == "blocks":
        lbm.lbm_upscale(s["params"], s["kappa"], case["block"], s["keff"], G0, case["tol"], case["max_steps"])
        return dict(keff=s["keff"])
    if path == "predict":
        x, stats = lbm.lbm_patches(s["kappa"], s["leaves"])
        return dict(y=s["net"].predict(x), stats=stats)
    if path == "train":
        loss = s["net"].train(s["x"], s["y"], s["stats"], epochs=1, batch=case["batch"], lr=2e-3, seed=1)
        return dict(loss=loss, params=[s["net"].get_params(m) for m in range(case["models"])])
    if path == "fine3d":
        s["grid"].step(case["steps"])
        rho, u, v, w = s["grid"].fields()
        return dict(rho=rho, u=u, v=v, w=w)
    keff, status, steps, _ = lbm.local_keff3(s["params"], s["kappa"], s["leaves"], G0, case["tol"], case["max_steps"], 64)
    return dict(keff=keff, status=status, steps=steps)


# --------------------------------------------------------------------------------------- work

def work(case):
    """Bytes a pass cannot do without (state in and out once, coefficients, outputs) and the
    floating-point operations of the lattice updates (about 85 in D2Q9, 180 in D3Q19) or of the
    network. A run to a tolerance counts the steps its workload takes on average."""
    path = case["path"]
    if path == "fine":
        n, e = case["nx"] * case["ny"], ELEM[case["storage"]]
        c = 8 if case["storage"] == "f64" else 4
        return dict(bytes=n * (18 * e + c * (3 if case["force"] else 1) + 12), flops=85.0 * n * case["steps"])
    if path == "coarse":
        n = case["nx"] * case["ny"]
        return dict(bytes=n * (32 + 12 + (8 if case["force"] else 0)), flops=95.0 * n * case["steps"])
    if path == "leaves":
        n = case["field"] ** 2
        cells = int((np.arange(1, 41) ** 2).sum()) if case["kind"] == "ragged" else n
        steps = case["max_steps"] if case["tol"] == 0.0 else 40000
        return dict(bytes=cells * 4.0, flops=85.0 * 2 * cells * steps)
    if path == "blocks":
        n = case["nx"] * case["ny"]
        grown = (1.0 + 2.0 * case["margin"] / case["block"]) ** 2
        return dict(bytes=4.0 * n + 32.0 * n / case["block"] ** 2, flops=85.0 * 2 * n * grown * 1500)
    if path == "predict":
        leaves = case["field"] ** 2 / 4096 * 17.5
        return dict(bytes=4.0 * case["field"] ** 2 + leaves * 8 * case["models"], flops=283.7e6 * leaves * case["models"])
    if path == "train":
        return dict(bytes=case["samples"] * 9 * 4096.0, flops=3 * 283.7e6 * case["samples"] * case["models"])
    if path == "fine3d":
        n, e = case["nx"] * case["ny"] * case["nz"], ELEM[case["storage"]]
        return dict(bytes=n * (38 * e + (8 if case["storage"] == "f64" else 4) + 16), flops=180.0 * n * case["steps"])
    n = case["field"] ** 3
    grown = (1.0 + 2.0 * case["margin"] / case["size"]) ** 3
    return dict(bytes=4.0 * n, flops=180.0 * 3 * n * grown * 5000)


# -------------------------------------------------------------------------- results in 64 bits

_E9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_E19 = [(0, 0, 0)] + [tuple(s if i == d else 0 for i in range(3)) for d in range(3) for s in (1, -1)] + \
    [tuple(s if i == a else (t if i == b else 0) for i in range(3)) for a, b in ((0, 1), (0, 2), (1, 2))
     for s, t in ((1, 1), (-1, -1), (1, -1), (-1, 1))]
_W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


class _Exact:
    """The scheme on deviations g = f - w rho0 in 64 bits: fields [..., (nz,) ny, nx], periodic
    (or half-way bounce-back walls in y). `drag(rx, ry, ..)` returns rho u from r = j + eps rho G / 2."""

    def __init__(self, shape, E, W, tau, G, drag, walls=False):
        self.E, self.W, self.tau, self.G, self.drag, self.walls = E, W, tau, G, drag, walls
        self.nd = len(E[0])
        self.opp = [E.index(tuple(-c for c in e)) for e in E]
        self.f = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in E]      # post-collision

    def streamed(self):
        out = []
        for a, e in enumerate(self.E):
            h = self.f[a]
            sh = [(c, -1 - d) for d, c in enumerate(e) if c]
            if sh:
                h = torch.roll(h, [c for c, _ in sh], [d for _, d in sh])
            if self.walls and e[1]:
                row = 0 if e[1] == 1 else -1
                h[..., row, :] = self.f[self.opp[a]][..., row, :]
            out.append(h)
        return out

    def moments(self, g):
        rho = 1.0 + sum(g)
        j = [sum(g[a] * e[d] for a, e in enumerate(self.E) if e[d]) for d in range(self.nd)]
        ru = self.drag(*[j[d] + 0.5 * rho * self.G[d] for d in range(self.nd)])
        return rho, j, ru

    def step(self):
        g = self.streamed()
        rho, j, ru = self.moments(g)
        tau = self.tau
        ue = [2.0 * tau * ru[d] + (1.0 - 2.0 * tau) * j[d] for d in range(self.nd)]
        for a, e in enumerate(self.E):
            eq = (rho - 1.0) + 3.0 * sum(ue[d] * e[d] for d in range(self.nd) if e[d])
            self.f[a] = g[a] + (self.W[a] * eq - g[a]) / tau

    def velocity(self):
        rho, _, ru = self.moments(self.streamed())
        return rho, [c / rho for c in ru]


def _scalar_drag(kappa, nu):
    k = kappa.double()
    d = 2.0 * k / (2.0 * k + nu)
    return lambda *r: [d * c for c in r]


def _exact_fine(case, seed):
    shape = (case["ny"], case["nx"])
    kappa = _lognormal(shape, case["ell"], case["sigma"], seed)
    G = list(_force_field(case["nx"], case["ny"]).double()) if case["force"] else [G0, 0.25 * G0]
    x = _Exact(shape, _E9, _W9, case["tau"], G, _scalar_drag(kappa, (case["tau"] - 0.5) / 3.0), case["walls"])
    old = None
    check, resid = case["check"], -1.0
    for t in range(1, case["steps"] + 1):
        at = check > 0 and t % check == 0
        if at:
            _, old = x.velocity()
        x.step()
        if at:
            _, new = x.velocity()
            du = max((a - b).abs().max().item() for a, b in zip(new, old))
            resid = du / max(c.abs().max().item() for c in new)
    rho, (u, v) = x.velocity()
    # with 11-bit storage the change of one step is the storage's own rounding: no 64-bit counterpart
    resid = None if case["storage"] == "f16" else torch.tensor(resid, dtype=torch.float64)
    return dict(rho=rho, u=u, v=v, steps=None, resid=resid)


def _exact_coarse(case, seed):
    r = case["block"]
    shape = (case["ny"], case["nx"])
    K = _coarse_tensors(case["nx"], case["ny"], seed) / r ** 2
    tau, nu = 0.5 + 0.5 / r, 1.0 / 6.0 / r
    c = 0.5 * nu                                       # rho u = (K + c I)^-1 K r
    a, b, p, q = K[..., 0] + c, K[..., 1], K[..., 2], K[..., 3] + c
    det = a * q - b * p

    def drag(rx, ry):
        kx, ky = K[..., 0] * rx + K[..., 1] * ry, K[..., 2] * rx + K[..., 3] * ry
        return [(q * kx - b * ky) / det, (a * ky - p * kx) / det]

    G = list(_force_field(case["nx"], case["ny"]).double() * r) if case["force"] else [G0 * r, 0.0]
    x = _Exact(shape, _E9, _W9, tau, G, drag)
    for _ in range(case["steps"]):
        x.step()
    rho, (u, v) = x.velocity()
    return dict(rho=rho, u=u, v=v, steps=None)


def _exact_leaves(case, seed):
    """Fixed-step local problems: every leaf of one size and both drives stepped together."""
    if case["tol"] > 0.0:
        return None
    kappa, leaves = _leaf_field(case, seed)
    keff = torch.zeros((len(leaves), 4), dtype=torch.float64, device="cuda")
    nu = 0.5 / 3.0
    for size in sorted(set(leaves[:, 2].tolist())):
        which = np.flatnonzero(leaves[:, 2] == size)
        k = torch.stack([kappa[y:y + size, x:x + size] for x, y, _ in leaves[which].tolist()])
        n = len(which)
        gx = torch.zeros((2 * n, 1, 1), dtype=torch.float64, device="cuda")
        gx[:n] = G0
        x = _Exact((2 * n, size, size), _E9, _W9, 1.0, [gx, G0 - gx], _scalar_drag(torch.cat([k, k]), nu))
        for _ in range(case["max_steps"]):
            x.step()
        _, (u, v) = x.velocity()
        u, v = (c.mean(dim=(1, 2)) * nu / G0 for c in (u, v))
        keff[torch.from_numpy(which).cuda()] = torch.stack([u[:n], u[n:], v[:n], v[n:]], dim=1)
    return dict(keff=keff, status=None, steps=None)


def _exact_fine3d(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    kappa = _lognormal(shape, case["ell"], case["sigma"], seed)
    x = _Exact(shape, _E19, _W19, 0.8, [G0, 0.0, 0.0], _scalar_drag(kappa, 0.3 / 3.0))
    for _ in range(case["steps"]):
        x.step()
    rho, (u, v, w) = x.velocity()
    return dict(rho=rho, u=u, v=v, w=w)


def _darcy(logk):
    """Finite-volume Darcy K*_xx, K*_yy of periodic patches [n, s, s] (harmonic faces, unit drive), by
    conjugate gradients in 64 bits to a relative residual of 1e-11."""
    k = torch.exp(logk.double())
    out = []
    kx, ky = (2.0 * k * torch.roll(k, -1, d) / (k + torch.roll(k, -1, d)) for d in (-1, -2))
    lx, ly = torch.roll(kx, 1, -1), torch.roll(ky, 1, -2)
    diag = kx + lx + ky + ly

    def apply(p):
        return diag * p - kx * torch.roll(p, -1, -1) - lx * torch.roll(p, 1, -1) - ky * torch.roll(p, -1, -2) - \
            ly * torch.roll(p, 1, -2)

    def dot(a, b):
        return (a * b).sum(dim=(-1, -2), keepdim=True)

    for d in (-1, -2):
        b = lx - kx if d == -1 else ly - ky
        p, r = torch.zeros_like(b), b.clone()
        q = r / diag
        rz, rr0 = dot(r, q), dot(b, b)
        for it in range(4000):
            ad = apply(q)
            dad = dot(q, ad)
            al = torch.where(dad > 0, rz / dad, torch.zeros_like(rz))
            p, r = p + al * q, r - al * ad
            z = r / diag
            new = dot(r, z)
            q = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * q
            rz = new
            if it % 32 == 31 and bool((dot(r, r) <= 1e-22 * rr0).all()):
                break
        face = kx if d == -1 else ky
        out.append((face * (p - torch.roll(p, -1, d) + 1.0)).mean(dim=(-1, -2)))
    return torch.stack(out, dim=-1)


def _exact_predict(case, seed):
    kappa, leaves = _leaf_field(case, seed)
    lk = torch.log(kappa.double())
    n = len(leaves)
    planes = torch.zeros((n, 9, 32, 32), dtype=torch.float64, device="cuda")
    stats = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    base = torch.zeros((n, 2), dtype=torch.float64, device="cuda")
    for size in sorted(set(leaves[:, 2].tolist())):
        which = torch.from_numpy(np.flatnonzero(leaves[:, 2] == size)).cuda()
        patch = torch.stack([lk[y:y + size, x:x + size] for x, y, _ in leaves[which.cpu().numpy()].tolist()])
        base[which] = torch.log(_darcy(patch))
        full = patch.repeat_interleave(64 // size, 1).repeat_interleave(64 // size, 2)
        ph = torch.stack([full[:, a::2, b::2] for a in (0, 1) for b in (0, 1)], dim=1)
        m = ph.mean(dim=1)
        row_h, row_a = -torch.log(torch.exp(-m).mean(2)), torch.log(torch.exp(m).mean(2))
        col_h, col_a = -torch.log(torch.exp(-m).mean(1)), torch.log(torch.exp(m).mean(1))
        planes[which, :4] = ph
        planes[which, 4] = math.log2(size) / 6.0
        planes[which, 5] = row_h[:, :, None].expand(-1, 32, 32)
        planes[which, 6] = row_a[:, :, None].expand(-1, 32, 32)
        planes[which, 7] = col_h[:, None, :].expand(-1, 32, 32)
        planes[which, 8] = col_a[:, None, :].expand(-1, 32, 32)
        var = (m * m).mean((1, 2)) - m.mean((1, 2)) ** 2
        grad = (m.diff(dim=1) ** 2).sum((1, 2)) + (m.diff(dim=2) ** 2).sum((1, 2))
        stats[which] = torch.stack([m.mean((1, 2)), var.clamp_min(0).sqrt(), 0.5 * grad / (32 * 31)], dim=1)
    x = (planes - float(_NORM[0])) / float(_NORM[1])
    x[:, 4] = planes[:, 4]
    y = torch.zeros((case["models"], n, 2), dtype=torch.float64, device="cuda")
    for m, w in enumerate(_weights(case["models"], seed)):
        w = torch.from_numpy(w).double().cuda()
        for i in range(0, n, 512):
            h, at, cin = x[i:i + 512], 0, 9
            for cout in (32, 32, 64, 64, 64, 64):
                k = w[at:at + cout * cin * 9].reshape(cout, cin * 9)
                at += cout * cin * 9
                h = torch.matmul(k, torch.nn.functional.unfold(h, 3, padding=1)) + w[at:at + cout, None]
                h = h.clamp_min(0).reshape(-1, cout, 32, 32)
                at += cout
                cin = cout
            h = h.mean((2, 3)) @ w[at:at + 128].reshape(2, 64).T + w[at + 128:at + 130]
            mean = torch.tensor([float(_NORM[2]), float(_NORM[4])], device="cuda", dtype=torch.float64)
            dev = torch.tensor([float(_NORM[3]), float(_NORM[5])], device="cuda", dtype=torch.float64)
            y[m, i:i + 512] = base[i:i + 512] + h * dev + mean
    return dict(y=y, stats=stats)


def exact(case, seed):
    path = case["path"]
    if path == "fine":
        return _exact_fine(case, seed)
    if path == "coarse":
        return _exact_coarse(case, seed)
    if path == "leaves":
        return _exact_leaves(case, seed)
    if path == "predict":
        return _exact_predict(case, seed)
    if path == "fine3d":
        return _exact_fine3d(case, seed)
    return None       # tolerance runs of up to 200,000 steps, and 64-bit training of whole ensembles
