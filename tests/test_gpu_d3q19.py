"""D3Q19 grids (Section 2's scheme in three dimensions) on the GPU against the D3Q19 oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _lbm():
    import paper_1312_0195_gb300 as lbm
    return lbm


def _field(nz, ny, nx, seed):
    rng = np.random.default_rng(seed)
    z = np.stack([synth.gaussian_random_field(nx, ny, 3.0, seed=seed * 100 + k) for k in range(nz)])
    z = 0.6 * z + 0.4 * rng.standard_normal((nz, ny, nx))
    return (1e-2 * np.exp(1.5 * z)).astype(np.float32)


def gpu3(kap, tau, nu, eps, g, steps, storage=0):
    import torch
    lbm = _lbm()
    nz, ny, nx = kap.shape
    p = lbm.Params3D(nx=nx, ny=ny, nz=nz, tau=tau, nu=nu, eps=eps, gx=g[0], gy=g[1], gz=g[2], storage=storage)
    with lbm.Grid3D(p, torch.from_numpy(np.ascontiguousarray(kap)).cuda()) as G:
        G.step(steps)
        out = [t.cpu().numpy().astype(np.float64) for t in G.fields()]
        mean = np.array(G.mean_velocity())
    return out, mean


def ora3(kap, tau, nu, eps, g, steps):
    p = oracle.Problem3D(tau, nu, eps, kappa=kap.astype(np.float64), g=g)
    f = p.rest()
    p.run(f, steps)
    return list(p.fields(f)), p.mean_velocity(f)


@pytest.mark.parametrize("shape", [(10, 12, 20), (7, 5, 131)])
def test_d3q19_fp32_matches_oracle(shape):
    kap = _field(*shape, seed=61)
    kap[1, 2, 3] = 0.0
    kap[2, 3, 4] = np.inf
    args = (kap, 0.8, 0.1, 0.9, (2e-6, -1e-6, 1.5e-6), 200)
    (r, u, v, w), mean = gpu3(*args)
    (ro, uo, vo, wo), mo = ora3(*args)
    scale = max(np.abs(uo).max(), np.abs(vo).max(), np.abs(wo).max())
    for a, b in ((u, uo), (v, vo), (w, wo)):
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-5 * scale)
    np.testing.assert_allclose(r, ro, rtol=0, atol=2.4e-7)
    assert u[1, 2, 3] == 0.0 and v[1, 2, 3] == 0.0 and w[1, 2, 3] == 0.0
    np.testing.assert_allclose(mean, mo, rtol=2e-5, atol=1e-6 * scale)


def test_d3q19_fp64_matches_oracle_to_roundoff():
    kap = _field(6, 9, 11, seed=62)
    args = (kap, 0.7, 0.05, 0.8, (1e-6, 2e-6, -1e-6), 300)
    (r, u, v, w), mean = gpu3(*args, storage=2)
    (ro, uo, vo, wo), mo = ora3(*args)
    scale = max(np.abs(uo).max(), np.abs(vo).max(), np.abs(wo).max())
    for a, b in ((u, uo), (v, vo), (w, wo)):
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-7 * scale)       # fields come back as float32
    np.testing.assert_allclose(mean, mo, rtol=1e-9, atol=1e-9 * scale)     # FP64 mean


def test_d3q19_full_size_sampled_against_oracle_windows():
    """256^3 (the benchmarked lattice, 16.8 M cells): after n steps a cell depends only on the
    cells within n of it, so periodic oracle windows of side 2 n + 9 reproduce sampled cells."""
    import torch
    lbm = _lbm()
    n, N = 6, 256
    rng = np.random.default_rng(63)
    kap = (1e-2 * np.exp(1.5 * rng.standard_normal((N, N, N)))).astype(np.float32)
    tau, nu, eps, g = 0.6, 0.2 / 6, 1.0, (1e-6, 0.0, 0.0)
    p = lbm.Params3D(nx=N, ny=N, nz=N, tau=tau, nu=nu, eps=eps, gx=g[0], gy=g[1], gz=g[2])
    pts = [tuple(int(v) for v in rng.integers(0, N, 3)) for _ in range(6)] + [(0, 0, 0), (N - 1, N - 1, N - 1)]
    with lbm.Grid3D(p, torch.from_numpy(kap).cuda()) as G:
        G.step(n)
        rho, u, v, w = G.fields()
        vals = [(float(u[z, y, x]), float(v[z, y, x]), float(w[z, y, x]), float(rho[z, y, x])) for (x, y, z) in pts]
    W = 2 * n + 9
    h = W // 2
    for (x, y, z), (ug, vg, wg, rg) in zip(pts, vals):
        zi = (np.arange(z - h, z - h + W) % N)[:, None, None]
        yi = (np.arange(y - h, y - h + W) % N)[None, :, None]
        xi = (np.arange(x - h, x - h + W) % N)[None, None, :]
        (ro, uo, vo, wo), _ = ora3(kap[zi, yi, xi], tau, nu, eps, g, n)
        s = max(abs(uo[h, h, h]), abs(vo[h, h, h]), abs(wo[h, h, h]), 1e-30)
        assert abs(ug - uo[h, h, h]) <= 1e-5 * s + 1e-13
        assert abs(vg - vo[h, h, h]) <= 1e-5 * s + 1e-13
        assert abs(wg - wo[h, h, h]) <= 1e-5 * s + 1e-13
        assert abs(rg - ro[h, h, h]) <= 2.4e-7


def test_d3q19_rejects_bad_input():
    import torch
    lbm = _lbm()
    kap = torch.full((4, 4, 4), 0.01, device="cuda")
    kap[1, 1, 1] = float("nan")
    with pytest.raises(lbm.LbmError):
        lbm.Grid3D(lbm.Params3D(nx=4, ny=4, nz=4, tau=1.0), kap)
    with pytest.raises(lbm.LbmError):
        lbm.Grid3D(lbm.Params3D(nx=4, ny=4, nz=4, tau=0.4), torch.full((4, 4, 4), 0.01, device="cuda"))


# ------------------------------------------------- three-dimensional local problems

def gpu_keff3(kap, leaves, tau, nu, eps, g, tol, max_steps, storage=0, k=64):
    import torch
    lbm = _lbm()
    nz, ny, nx = kap.shape
    p = lbm.Params3D(nx=nx, ny=ny, nz=nz, tau=tau, nu=nu, eps=eps, storage=storage)
    ke, st, steps, worst = lbm.local_keff3(p, torch.from_numpy(np.ascontiguousarray(kap, dtype=np.float32)).cuda(),
                                           torch.from_numpy(np.asarray(leaves, dtype=np.int32)).cuda(), g, tol,
                                           max_steps, k)
    return ke.cpu().numpy(), st.cpu().numpy(), steps.cpu().numpy(), worst


@pytest.mark.parametrize("storage", [0, 2])
def test_local_keff3_matches_oracle(storage):
    """Mixed cube sizes at fixed step counts (every drive the same number of steps on both sides)."""
    kap = _field(12, 14, 16, seed=71)
    leaves = [(0, 0, 0, 4), (8, 6, 4, 8), (3, 2, 1, 5), (12, 10, 8, 4), (0, 0, 0, 12)]
    ke, st, steps, _ = gpu_keff3(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 0.0, 600, storage)
    assert (steps == 600).all() and (st == 0).all()
    for i, (x0, y0, z0, s) in enumerate(leaves):
        cube = kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64)
        ref = oracle.local_keff3(cube, 1.0, 1.0 / 6.0, 1.0, 1e-6, tol=0.0, max_steps=600)["keff"]
        scale = np.abs(np.diag(ref)).max()
        tol = 1e-9 if storage == 2 else 1e-5
        np.testing.assert_allclose(ke[i], ref, rtol=0, atol=tol * scale)


def test_local_keff3_tolerance_stop_and_uniform_cube():
    """The stop rule gives the oracle's step counts; a uniform cube gives kappa I (Eq. 19 in 3-D)."""
    kap = _field(8, 8, 8, seed=72)
    kap[:4, :4, :4] = 3e-3
    leaves = [(0, 0, 0, 4), (0, 0, 0, 8)]
    ke, st, steps, worst = gpu_keff3(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 1e-7, 100000, storage=2)
    # stopped at tol 1e-7 per 64 steps, the uniform cube is within 1e-6 of its steady kappa
    np.testing.assert_allclose(np.diag(ke[0]), float(np.float32(3e-3)), rtol=1e-6)
    for i, (x0, y0, z0, s) in enumerate(leaves):
        ref = oracle.local_keff3(kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64), 1.0, 1.0 / 6.0, 1.0,
                                 1e-6, tol=1e-7, max_steps=100000)
        assert list(steps[i]) == ref["steps"]
        np.testing.assert_allclose(ke[i], ref["keff"], rtol=0, atol=1e-9 * np.abs(ref["keff"]).max())
    assert worst == 0 and (st == 0).all()


def test_local_keff3_rejects_bad_leaves():
    import torch
    lbm = _lbm()
    kap = torch.full((8, 8, 8), 0.01, device="cuda")
    p = lbm.Params3D(nx=8, ny=8, nz=8, tau=1.0)
    for bad in ([[4, 0, 0, 5]], [[0, 0, 0, 0]], [[-1, 0, 0, 2]]):
        with pytest.raises(lbm.LbmError):
            lbm.local_keff3(p, kap, torch.tensor(bad, dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("storage", [0, 2])
def test_local_keff3_cluster_slabs_match_oracle(storage):
    """Cubes wider than one CTA's shared memory: 16 and 15 cells (two slabs in FP32, four in
    FP64; 15 leaves the last slab one layer short) and 32 cells (sixteen slabs in FP32)."""
    kap = _field(32, 32, 32, seed=73)
    kap[20, 5, 17] = 0.0
    leaves = [(0, 0, 0, 16), (16, 8, 3, 15), (0, 0, 0, 32)]
    ke, st, steps, _ = gpu_keff3(kap, leaves, 0.8, 0.1, 0.9, 2e-6, 0.0, 300, storage)
    assert (steps == 300).all() and (st == 0).all()
    for i, (x0, y0, z0, s) in enumerate(leaves):
        cube = kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64)
        ref = oracle.local_keff3(cube, 0.8, 0.1, 0.9, 2e-6, tol=0.0, max_steps=300)["keff"]
        scale = np.abs(np.diag(ref)).max()
        np.testing.assert_allclose(ke[i], ref, rtol=0, atol=(1e-9 if storage == 2 else 1e-5) * scale)


@pytest.mark.parametrize("storage", [0, 2])
def test_local_keff3_cluster_and_global_paths_agree(storage, monkeypatch):
    """The shared-memory (cluster) path and the HBM path take the same arithmetic per cell;
    only the order of the FP64 velocity sums differs."""
    kap = _field(16, 16, 16, seed=74)
    leaves = [(0, 0, 0, 16), (4, 4, 4, 8), (1, 2, 3, 11), (0, 0, 0, 3)]
    a = gpu_keff3(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 0.0, 257, storage, k=16)
    monkeypatch.setenv("LBM_LOCAL3_GLOBAL", "1")
    b = gpu_keff3(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 0.0, 257, storage, k=16)
    assert (a[2] == 257).all() and (b[2] == 257).all()
    scale = np.abs(np.diagonal(b[0], axis1=1, axis2=2)).max()
    np.testing.assert_allclose(a[0], b[0], rtol=0, atol=1e-12 * scale)


def test_local_keff3_time_limit_gives_etimeout():
    """The launch's wall-clock bound on the cluster path: with a tiny limit every cluster
    abandons its job at its next check and the host sees LBM_ETIMEOUT; the context stays usable."""
    lbm = _lbm()
    kap = _field(32, 32, 32, seed=75)
    leaves = [(x, y, z, 16) for z in (0, 16) for y in (0, 16) for x in (0, 16)]
    try:
        lbm.lbm_set_time_limit(2e-4)
        ke, st, steps, worst = gpu_keff3(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 1e-14, 10_000_000)
        assert worst == lbm.LBM_ETIMEOUT
        assert (st == lbm.LBM_ETIMEOUT).all()
    finally:
        lbm.lbm_set_time_limit(600.0)
    ke, st, steps, worst = gpu_keff3(kap, leaves[:2], 1.0, 1.0 / 6.0, 1.0, 1e-6, 0.0, 100)
    assert worst == 0 and np.isfinite(ke).all()


def test_local_keff3_degenerate_and_large_cubes():
    """Cubes of 1, 2 and 3 cells (every neighbour is the cell itself or a wrapped copy), a cube
    of 36 (above the cluster limit, so on the HBM path) and an empty leaf list."""
    kap = _field(36, 36, 40, seed=76)
    leaves = [(5, 6, 7, 1), (0, 1, 2, 2), (30, 31, 32, 3), (2, 0, 0, 36)]
    ke, st, steps, _ = gpu_keff3(kap, leaves, 0.9, 0.12, 0.8, 1e-6, 0.0, 200)
    assert (steps == 200).all() and (st == 0).all()
    for i, (x0, y0, z0, s) in enumerate(leaves):
        cube = kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64)
        ref = oracle.local_keff3(cube, 0.9, 0.12, 0.8, 1e-6, tol=0.0, max_steps=200)["keff"]
        scale = np.abs(np.diag(ref)).max()
        np.testing.assert_allclose(ke[i], ref, rtol=0, atol=1e-5 * scale)
    # a single cell is a uniform cube: kappa on the diagonal, nothing off it (Eq. 19 in 3-D)
    np.testing.assert_allclose(np.diag(ke[0]), kap[7, 6, 5], rtol=1e-3)
    ke, st, steps, worst = gpu_keff3(kap, np.zeros((0, 4), np.int32), 0.9, 0.12, 0.8, 1e-6, 0.0, 200)
    assert worst == 0 and ke.shape == (0, 3, 3)


def test_local_keff3_full_size_sampled():
    """The benchmarked launch: all 4096 cubes of 16^3 of the 256^3 log-normal field in one call
    (clusters of two CTAs), a fixed 300 steps; seeded sample cubes against the oracle."""
    import torch
    lbm = _lbm()
    n, b = 256, 16
    kap = synth.lognormal_kappa3d(n, n, n, 8.0, 2.0, seed=7)
    cubes = [(x, y, z, b) for z in range(0, n, b) for y in range(0, n, b) for x in range(0, n, b)]
    p = lbm.Params3D(nx=n, ny=n, nz=n, tau=1.0, eps=1.0)
    ke, st, steps, _ = lbm.local_keff3(p, torch.from_numpy(kap).cuda(),
                                       torch.tensor(cubes, dtype=torch.int32, device="cuda"), 1e-6, 0.0, 300, 64)
    ke, steps = ke.cpu().numpy(), steps.cpu().numpy()
    assert (steps == 300).all() and (st.cpu().numpy() == 0).all()
    rng = np.random.default_rng(77)
    for i in list(rng.choice(len(cubes), 5, replace=False)) + [0, len(cubes) - 1]:
        x0, y0, z0, s = cubes[i]
        ref = oracle.local_keff3(kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64), 1.0, 1.0 / 6.0, 1.0,
                                 1e-6, tol=0.0, max_steps=300)["keff"]
        np.testing.assert_allclose(ke[i], ref, rtol=0, atol=1e-5 * np.abs(np.diag(ref)).max())


@pytest.mark.parametrize("storage,force_global", [(0, False), (2, False), (0, True)])
def test_local_keff3_oversampled_matches_oracle(storage, force_global, monkeypatch):
    """Oversampling (margin m): leaves grown by m cells on every side, cut from the field with
    periodic wrap (leaves at the field's edges wrap), inner-window mean; the cluster path and,
    forced, the HBM path against the oracle's oversampled problem."""
    import torch
    lbm = _lbm()
    if force_global:
        monkeypatch.setenv("LBM_LOCAL3_GLOBAL", "1")
    kap = _field(20, 18, 22, seed=78)
    leaves = [(0, 0, 0, 8), (14, 10, 12, 8), (5, 6, 7, 4), (18, 14, 16, 4)]
    for m in (2, 3):
        nz, ny, nx = kap.shape
        p = lbm.Params3D(nx=nx, ny=ny, nz=nz, tau=1.0, nu=1.0 / 6.0, eps=1.0, storage=storage, margin=m)
        ke, st, steps, _ = lbm.local_keff3(p, torch.from_numpy(kap).cuda(),
                                           torch.tensor(leaves, dtype=torch.int32, device="cuda"), 1e-6, 0.0, 300, 64)
        ke = ke.cpu().numpy()
        assert (steps.cpu().numpy() == 300).all() and (st.cpu().numpy() == 0).all()
        for i, (x0, y0, z0, s) in enumerate(leaves):
            grown = oracle.grown_cube(kap.astype(np.float64), x0, y0, z0, s, m)
            ref = oracle.local_keff3(grown, 1.0, 1.0 / 6.0, 1.0, 1e-6, tol=0.0, max_steps=300, margin=m)["keff"]
            tol = 1e-9 if storage == 2 else 1e-5
            np.testing.assert_allclose(ke[i], ref, rtol=0, atol=tol * np.abs(np.diag(ref)).max())


def test_local_keff3_margin_limits_are_rejected():
    import torch
    lbm = _lbm()
    kap = torch.full((8, 8, 8), 0.01, device="cuda")
    lv = torch.tensor([[0, 0, 0, 4]], dtype=torch.int32, device="cuda")
    for m in (33, 9, -1):
        with pytest.raises(lbm.LbmError):
            lbm.local_keff3(lbm.Params3D(nx=8, ny=8, nz=8, tau=1.0, margin=m), kap, lv)


def test_d3q19_fp16_storage_error_is_bounded():
    """FP16 scaled storage on the D3Q19 grid keeps 11 bits per population; in this Darcy-like
    regime the density deviations dominate every population. On this 12 x 16 x 40 box the
    error is measured at 1.199e-3 relative L2 (GB300, bit-reproducible); the test holds it to
    10 % above that."""
    kap = _field(12, 16, 40, seed=64)
    args = (kap, 1.0, 1.0 / 6.0, 1.0, (1e-6, 0.0, 0.0), 1500)
    (r, u, v, w), mean = gpu3(*args, storage=1)
    (ro, uo, vo, wo), mo = ora3(*args)
    num = np.sqrt(((u - uo) ** 2 + (v - vo) ** 2 + (w - wo) ** 2).sum())
    err = num / np.sqrt((uo ** 2 + vo ** 2 + wo ** 2).sum())
    print(f"D3Q19 FP16 storage rel L2 error on u: {err:.3e}")
    print(f"D3Q19 FP16 storage rel error of the mean u_x: {abs(mean[0] - mo[0]) / abs(mo[0]):.3e}")
    assert err < 1.1 * 1.199e-3
    assert abs(mean[0] - mo[0]) <= 3e-3 * abs(mo[0])
    np.testing.assert_allclose(r, ro, rtol=0, atol=1e-3)


@pytest.mark.parametrize("storage", [0, 1, 2])
def test_d3q19_checkpoint_restart_is_bitwise(storage):
    """Save after 80 steps, run 40 more; a new grid on the same field loads the state and runs the
    same 40 steps: the fields agree bit for bit (every storage type)."""
    import torch
    lbm = _lbm()
    kap = torch.from_numpy(_field(6, 8, 12, seed=66)).cuda()
    p = lbm.Params3D(nx=12, ny=8, nz=6, tau=0.8, nu=0.1, eps=0.9, gx=1e-6, gy=-0.5e-6, storage=storage)
    with lbm.Grid3D(p, kap) as a:
        a.step(80)
        st = a.save_state()
        a.step(40)
        fa = [t.cpu().numpy() for t in a.fields()]
    with lbm.Grid3D(p, kap) as b:
        b.load_state(st)
        b.step(40)
        fb = [t.cpu().numpy() for t in b.fields()]
    for x, y in zip(fa, fb):
        np.testing.assert_array_equal(x, y)
    # another parameter set (or a buffer of the wrong size) is rejected, not misread
    p2 = lbm.Params3D(nx=12, ny=8, nz=6, tau=0.9, nu=0.1, eps=0.9, gx=1e-6, gy=-0.5e-6, storage=storage)
    with lbm.Grid3D(p2, kap) as c:
        with pytest.raises(lbm.LbmError) as ei:
            c.load_state(st)
        assert ei.value.status == lbm.LBM_EINVAL
        with pytest.raises(lbm.LbmError) as ei:
            c.load_state(st[:-16])
        assert ei.value.status == lbm.LBM_EINVAL


@pytest.mark.parametrize("sides,tau,steps,k", [(range(1, 10), 1.0, 130, 64), (range(10, 19), 0.8, 77, 10)])
def test_local_keff3_two_jobs_a_cluster_match_oracle(sides, tau, steps, k):
    """FP32 cubes of up to 18 cells run two jobs to a cluster of one to six CTAs; every side (odd ones leave
    the last slab short) and a batch whose jobs are refilled more than once. 1e-5 is the FP32 bound above."""
    kap = _field(40, 40, 40, seed=79)
    kap[5, 6, 7] = 0.0
    leaves = [((3 * s) % (41 - s), (5 * s) % (41 - s), (7 * s) % (41 - s), s) for s in sides]
    leaves += [(x, y, z, 4) for z in range(0, 40, 4) for y in range(0, 40, 4) for x in range(0, 40, 4)] if 4 in sides else []
    ke, st, n, _ = gpu_keff3(kap, leaves, tau, 0.1, 0.9, 1e-6, 0.0, steps, k=k)
    assert (n == steps).all() and (st == 0).all()
    for i in range(min(len(leaves), 40)):
        x0, y0, z0, s = leaves[i]
        cube = kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64)
        ref = oracle.local_keff3(cube, tau, 0.1, 0.9, 1e-6, tol=0.0, max_steps=steps, check_every=k)["keff"]
        np.testing.assert_allclose(ke[i], ref, rtol=0, atol=1e-5 * np.abs(np.diag(ref)).max())


def test_local_keff3_time_limit_reaches_jobs_still_in_the_queue():
    """Past the wall-clock limit no leaf is reported as solved: neither the jobs that run nor those that wait in
    either size's queue (512 cubes of 8 and 125 of 12 cells, several times what the chip holds at once)."""
    import torch
    lbm = _lbm()
    kap = _field(64, 64, 64, seed=80)
    leaves = [(x, y, z, s) for s in (8, 12) for z in range(0, 65 - s, s) for y in range(0, 65 - s, s)
              for x in range(0, 65 - s, s)]
    try:
        lbm.lbm_set_time_limit(2e-4)
        ke, st, steps, worst = gpu_keff3(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 1e-14, 10_000_000)
        assert worst == lbm.LBM_ETIMEOUT
        assert (st == lbm.LBM_ETIMEOUT).all()
        assert (np.isnan(ke).all(axis=1) == (steps == 0)).all()
        _, n_notconv, worst = lbm.lbm3d_upscale(lbm.Params3D(nx=64, ny=64, nz=64, tau=1.0), torch.from_numpy(kap).cuda(), 8,
                                                1e-6, 1e-14, 10_000_000)
        assert worst == lbm.LBM_ETIMEOUT and n_notconv == 512
    finally:
        lbm.lbm_set_time_limit(600.0)


@pytest.mark.parametrize("side,n", [(3, 450), (4, 450), (7, 300), (8, 300), (12, 130), (13, 84), (14, 84), (16, 134), (17, 50), (18, 50)])
def test_local_keff3_batches_that_go_two_jobs_a_cluster_match_oracle(side, n):
    """Small batches of most sides run one job to a cluster; these are large enough for two, with refills, and checked
    like the batches above on a sample of their cubes."""
    kap = _field(40, 40, 40, seed=81)
    r = np.random.default_rng(side)
    leaves = [(*r.integers(0, 41 - side, 3), side) for _ in range(n)]
    ke, st, steps, _ = gpu_keff3(kap, leaves, 0.8, 0.1, 0.9, 1e-6, 0.0, 77, k=64)
    assert (steps == 77).all() and (st == 0).all()
    for i in [0, 1, n // 3, n // 2, n - 2, n - 1]:
        x0, y0, z0, s = leaves[i]
        cube = kap[z0:z0 + s, y0:y0 + s, x0:x0 + s].astype(np.float64)
        ref = oracle.local_keff3(cube, 0.8, 0.1, 0.9, 1e-6, tol=0.0, max_steps=77, check_every=64)["keff"]
        np.testing.assert_allclose(ke[i], ref, rtol=0, atol=1e-5 * np.abs(np.diag(ref)).max())
