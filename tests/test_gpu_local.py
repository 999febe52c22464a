"""GPU parity of the batched local problems (Section 3, Eq. 17) against the oracle,
and the paper's own K* values reproduced by the GPU solver.

The GPU solver stores FP32 deviations and reduces the means in FP64; the bar is
1e-4 relative on K*, the FP32 accuracy bar of the path. Off-diagonal entries are compared
relative to sqrt(K*_xx K*_yy), the scale of the tensor.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _lbm():
    import paper_1312_0195_gb300 as lbm
    return lbm


def gpu_keff(kap, leaves, tau, nu, eps, g, tol, max_steps, k=64, persistent=True, warm=0, storage=0):
    import torch
    lbm = _lbm()
    ny, nx = kap.shape
    p = lbm.Params(nx=nx, ny=ny, tau=tau, nu=nu, eps=eps, warm_start=warm, storage=storage)
    kt = torch.from_numpy(np.ascontiguousarray(kap, dtype=np.float32)).cuda()
    lt = torch.from_numpy(np.ascontiguousarray(leaves, dtype=np.int32)).cuda()
    keff, status, steps, worst = lbm.local_keff(p, kt, lt, g, tol, max_steps, k, persistent)
    return keff.cpu().numpy(), status.cpu().numpy(), steps.cpu().numpy(), worst


def oracle_keff(kap, leaf, tau, nu, eps, g, tol, max_steps, k=64, warm=False):
    x0, y0, s = (int(v) for v in leaf)
    patch = np.asarray(kap, dtype=np.float32)[y0:y0 + s, x0:x0 + s].astype(np.float64)
    return oracle.local_keff(patch, tau, nu, eps, g, tol=tol, max_steps=max_steps, check_every=k, warm=warm)


def assert_keff_close(a, b, rtol):
    scale = np.sqrt(abs(b[0] * b[3]))
    assert abs(a[0] - b[0]) <= rtol * abs(b[0]), (a, b)
    assert abs(a[3] - b[3]) <= rtol * abs(b[3]), (a, b)
    assert abs(a[1] - b[1]) <= rtol * scale, (a, b)
    assert abs(a[2] - b[2]) <= rtol * scale, (a, b)


def test_mixed_sizes_fixed_steps_match_oracle_and_per_leaf_launches():
    kap = synth.lognormal_kappa(128, 128, 8.0, 2.0, seed=21)
    leaves = synth.quadtree_leaves(128, 128, seed=3)
    assert set(leaves[:, 2]) == {8, 16, 32, 64} or len(set(leaves[:, 2])) >= 3
    tau, nu, eps, g = 1.0, 1.0 / 6.0, 1.0, 1e-6
    ke, st, steps, worst = gpu_keff(kap, leaves, tau, nu, eps, g, 0.0, 1500)
    assert worst == 0 and (st == 0).all() and (steps == 1500).all()
    for i in range(len(leaves)):
        ref = oracle_keff(kap, leaves[i], tau, nu, eps, g, 0.0, 1500)
        assert_keff_close(ke[i], ref["keff"], 1e-4)
    ke1, st1, steps1, _ = gpu_keff(kap, leaves, tau, nu, eps, g, 0.0, 1500, persistent=False)
    np.testing.assert_array_equal(ke1, ke)      # same arithmetic, same fixed-order reductions


def test_tolerance_stop_matches_oracle():
    kap = synth.lognormal_kappa(64, 64, 6.0, 1.0, seed=22)
    leaves = synth.uniform_leaves(64, 64, 16)
    tau, nu, eps, g = 1.0, 1.0 / 6.0, 1.0, 1e-6
    ke, st, steps, worst = gpu_keff(kap, leaves, tau, nu, eps, g, 1e-8, 200000)
    assert worst == 0 and (st == 0).all()
    for i in range(len(leaves)):
        ref = oracle_keff(kap, leaves[i], tau, nu, eps, g, 1e-8, 200000)
        assert_keff_close(ke[i], ref["keff"], 1e-4)
        assert (steps[i] % 64 == 0).all()


def test_odd_sizes_and_tiny_leaves():
    kap = synth.lognormal_kappa(60, 40, 5.0, 1.0, seed=23)
    leaves = np.array([[0, 0, 10], [10, 0, 10], [3, 7, 5], [50, 30, 10], [0, 20, 20], [59, 39, 1], [40, 0, 2]],
                      dtype=np.int32)
    tau, nu, eps, g = 0.8, 0.05, 0.8, 1e-6
    ke, st, steps, worst = gpu_keff(kap, leaves, tau, nu, eps, g, 0.0, 700, k=50)
    assert worst == 0
    for i in range(len(leaves)):
        ref = oracle_keff(kap, leaves[i], tau, nu, eps, g, 0.0, 700, k=50)
        assert_keff_close(ke[i], ref["keff"], 1e-4)


def test_fp64_local_solver_matches_oracle_to_roundoff():
    """storage = LBM_F64 selects the FP64 local solver (2048 resident cells, leaves up to 45)."""
    import torch
    lbm = _lbm()
    ex = synth.paper_experiment("E6_local")
    kap = np.asarray(ex["kappa"], dtype=np.float32)
    p = lbm.Params(nx=10, ny=10, tau=ex["tau"], nu=ex["nu"], eps=ex["eps"], storage=lbm.LBM_F64)
    lt = torch.tensor([[0, 0, 10]], dtype=torch.int32, device="cuda")
    ke, st, steps, worst = lbm.local_keff(p, torch.from_numpy(kap).cuda(), lt, ex["g_const"], 0.0, 20000, 64)
    ref = oracle.local_keff(kap.astype(np.float64), ex["tau"], ex["nu"], ex["eps"], ex["g_const"], tol=0.0,
                            max_steps=20000, check_every=64)
    np.testing.assert_allclose(ke.cpu().numpy()[0, [0, 3]], ref["keff"][[0, 3]], rtol=1e-9)
    big = torch.tensor([[0, 0, 46]], dtype=torch.int32, device="cuda")
    with pytest.raises(lbm.LbmError):
        lbm.local_keff(p, torch.zeros((64, 64), device="cuda") + 0.1, big)


def test_uniform_leaf_gives_kappa_identity():
    kap = np.full((64, 64), 0.037)
    leaves = np.array([[0, 0, 64], [0, 0, 8], [8, 8, 32]], dtype=np.int32)
    ke, st, _, _ = gpu_keff(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 1e-8, 100000)
    k32 = float(np.float32(0.037))
    for i in range(3):
        np.testing.assert_allclose(ke[i, [0, 3]], k32, rtol=1e-5)
        assert abs(ke[i, 1]) < 1e-6 * k32 and abs(ke[i, 2]) < 1e-6 * k32


@pytest.mark.parametrize("ratio", [2.0, 100.0, 1e4])
def test_gpu_reproduces_table1_and_table3(ratio):
    """Series layers (Table 1: harmonic mean) and the checkerboard (Table 3, 100^2 LBM column)
    solved as 20x20 periodic leaves by the GPU solver."""
    rows = {float(r[0]): r for r in (l.split() for l in open(
        __file__.replace("test_gpu_local.py", "golden/table3_checkerboard.txt")) if l.strip() and l[0] != "#")}
    ex = synth.paper_experiment("E2", ratio=ratio, ny=20)
    kap = ex["kappa"][:20, :20]
    ke, st, _, _ = gpu_keff(kap, np.array([[0, 0, 20]]), ex["tau"], ex["nu"], ex["eps"], ex["g"][0], 1e-10,
                            2000000)
    kxx = ke[0, 0] * 1e-4 / 1e-12
    exact = 2.0 / (1.0 + 1.0 / ratio)
    assert abs(kxx - exact) <= 1e-4 * exact
    ex = synth.paper_experiment("E4", ratio=ratio, n=100)
    kap = ex["kappa"][:20, :20]
    ke, st, _, _ = gpu_keff(kap, np.array([[0, 0, 20]]), ex["tau"], ex["nu"], ex["eps"], ex["g"][0], 1e-10,
                            2000000)
    kxx = ke[0, 0] * 1e-4 / 1e-12
    printed = float(rows[ratio][2])
    assert abs(kxx - printed) <= 1e-4 * printed


def test_gpu_reproduces_fiveblock_8485():
    ex = synth.paper_experiment("E5_local")
    ke, st, _, _ = gpu_keff(ex["kappa"], np.array([[0, 0, 10]]), ex["tau"], ex["nu"], ex["eps"], ex["g_const"],
                            1e-10, 1000000)
    k = ke[0] / ex["k_const"]
    assert abs(0.5 * (k[0] + k[3]) - 8.485) <= 1e-3


def test_full_size_quadtree_sampled():
    """4096^2 field (sigma 2, ell 32, seed 2) cut by the seeded quadtree (~71.6k leaves) in one
    persistent launch; sampled leaves against the oracle at the same fixed step count."""
    N = 4096
    kap = synth.lognormal_kappa(N, N, 32.0, 2.0, seed=2).astype(np.float32)
    leaves = synth.quadtree_leaves(N, N, seed=3)
    assert 65000 < len(leaves) < 78000
    tau, nu, eps, g = 1.0, 1.0 / 6.0, 1.0, 1e-6
    ke, st, steps, worst = gpu_keff(kap, leaves, tau, nu, eps, g, 0.0, 256)
    assert worst == 0 and np.isfinite(ke).all() and (steps == 256).all()
    rng = np.random.default_rng(1)
    for i in rng.choice(len(leaves), 24, replace=False):
        ref = oracle_keff(kap, leaves[i], tau, nu, eps, g, 0.0, 256)
        assert_keff_close(ke[i], ref["keff"], 1e-4)


def test_time_limit_gives_etimeout():
    """The launch's wall-clock bound: with a tiny limit the kernel abandons its jobs and the
    host sees LBM_ETIMEOUT (no device fault, the context stays usable)."""
    lbm = _lbm()
    kap = synth.lognormal_kappa(512, 512, 8.0, 1.0, seed=24)
    leaves = synth.uniform_leaves(512, 512, 64)
    try:
        lbm.lbm_set_time_limit(2e-4)
        ke, st, steps, worst = gpu_keff(kap, leaves, 1.0, 1.0 / 6.0, 1.0, 1e-6, 1e-12, 10_000_000)
        assert worst == lbm.LBM_ETIMEOUT
        assert (st == lbm.LBM_ETIMEOUT).any()
    finally:
        lbm.lbm_set_time_limit(600.0)
    ke, st, steps, worst = gpu_keff(kap, leaves[:4], 1.0, 1.0 / 6.0, 1.0, 1e-6, 0.0, 100)
    assert worst == 0 and np.isfinite(ke).all()


def test_invalid_leaves_rejected():
    import torch
    lbm = _lbm()
    kap = torch.full((32, 32), 0.1, device="cuda")
    p = lbm.Params(nx=32, ny=32, tau=1.0)
    for bad in ([[0, 0, 65]], [[30, 0, 8]], [[-1, 0, 4]], [[0, 0, 0]]):
        lt = torch.tensor(bad, dtype=torch.int32, device="cuda")
        with pytest.raises(lbm.LbmError) as ei:
            lbm.local_keff(p, kap, lt)
        assert ei.value.status == lbm.LBM_EINVAL


# ------------------------------------------------- oversampled local problems (Conclusions)

@pytest.mark.parametrize("storage", [0, 2])
def test_oversampled_leaves_match_oracle(storage):
    """margin > 0: each leaf's problem is solved on the leaf grown by `margin` cells (periodic wrap
    at the field edge) and K* averages the inner leaf. Leaves at the field corners exercise the
    wrap; fixed step counts make the comparison step for step."""
    import torch
    lbm = _lbm()
    kap = synth.lognormal_kappa(48, 40, 4.0, 1.5, seed=41).astype(np.float32)
    leaves = np.array([[0, 0, 8], [40, 32, 8], [16, 8, 16], [4, 24, 12], [32, 0, 8]], dtype=np.int32)
    for margin in (3, 8):
        p = lbm.Params(nx=48, ny=40, tau=1.0, nu=1.0 / 6.0, eps=1.0, storage=storage, margin=margin)
        ke, st, steps, _ = lbm.local_keff(p, torch.from_numpy(kap).cuda(), torch.from_numpy(leaves).cuda(), 1e-6,
                                          0.0, 1500, 64)
        ke = ke.cpu().numpy()
        for i, (x0, y0, s) in enumerate(leaves):
            ext = synth.crop_periodic(kap, x0 - margin, y0 - margin, s + 2 * margin, s + 2 * margin)
            ref = oracle.local_keff(ext.astype(np.float64), 1.0, 1.0 / 6.0, 1.0, 1e-6, tol=0.0, max_steps=1500,
                                    margin=margin)["keff"]
            scale = max(abs(ref[0]), abs(ref[3]))
            tol = 1e-9 if storage == 2 else 2e-5
            np.testing.assert_allclose(ke[i], ref, rtol=0, atol=tol * scale)


def test_oversampling_inner_window_on_parallel_layers():
    """The GPU counterpart of the oracle pin: parallel layers at tau = 1/2 with margin columns of
    a third permeability; the oversampled K*_yy is the mean over the inner leaf's columns."""
    import torch
    lbm = _lbm()
    ex = synth.paper_experiment("E3", ratio=10.0, ny=1)
    k1, k2 = float(ex["kappa"][0, 0]), float(ex["kappa"][0, 10])
    cols = np.array([5.0 * k2] * 10 + [k1] * 10 + [k2] * 10 + [5.0 * k2] * 10, dtype=np.float32)
    kap = np.tile(cols, (40, 1))
    p = lbm.Params(nx=40, ny=40, tau=ex["tau"], nu=ex["nu"], eps=ex["eps"], storage=lbm.LBM_F64, margin=10)
    lt = torch.tensor([[10, 10, 20]], dtype=torch.int32, device="cuda")
    ke, st, _, _ = lbm.local_keff(p, torch.from_numpy(kap).cuda(), lt, 1e-6, 1e-11, 20000, 64)
    kyy = float(ke[0, 3])
    inner = 0.5 * (float(np.float32(k1)) + float(np.float32(k2)))
    assert abs(kyy - inner) <= 2e-6 * inner


def test_oversampling_limits_are_rejected():
    import torch
    lbm = _lbm()
    kap = torch.full((64, 64), 0.01, device="cuda")
    lt = torch.tensor([[0, 0, 64]], dtype=torch.int32, device="cuda")
    for margin in (-1, 33):
        with pytest.raises(lbm.LbmError):
            lbm.local_keff(lbm.Params(nx=64, ny=64, tau=1.0, margin=margin), kap, lt)
    with pytest.raises(lbm.LbmError):          # 64 + 2 x 1 cells do not fit the resident patch
        lbm.local_keff(lbm.Params(nx=64, ny=64, tau=1.0, margin=1), kap, lt)


# ------------------------------------------------------------------ the Darcy start (warm_start = 1)

def test_darcy_start_fixed_steps_match_oracle():
    """warm_start = 1: runs on patches of 16 cells or more start from the patch's finite-volume
    Darcy state, solved in shared memory by conjugate gradients to a relative residual of 1e-5 (the
    oracle solves it directly in FP64). After a fixed 256 steps K* matches the oracle's warm-started
    run to 1e-4, for leaves of 8 (which start from rest), 16, 32 and 64 cells, in FP32 and FP64."""
    kap = synth.lognormal_kappa(128, 128, 6.0, 2.0, seed=27)
    leaves = np.array([[0, 0, 64], [64, 0, 32], [96, 0, 32], [64, 32, 16], [80, 32, 16], [96, 32, 8],
                       [0, 64, 64], [64, 64, 16]], dtype=np.int32)
    tau, nu, eps, g = 1.0, 1.0 / 6.0, 0.9, 1e-6
    ke, st, steps, worst = gpu_keff(kap, leaves, tau, nu, eps, g, 0.0, 256, warm=1)
    assert worst == 0 and (steps == 256).all()
    for i in range(len(leaves)):
        ref = oracle_keff(kap, leaves[i], tau, nu, eps, g, 0.0, 256, warm=True)
        assert_keff_close(ke[i], ref["keff"], 1e-4)
    cold, _, _, _ = gpu_keff(kap, leaves, tau, nu, eps, g, 0.0, 256)
    small = leaves[:, 2] < 16
    np.testing.assert_allclose(ke[small], cold[small], rtol=1e-6, atol=0)   # 8-cell leaves start from rest
    assert not np.array_equal(ke[~small], cold[~small])
    # the FP64 solver (leaves up to 45 cells) with the same start
    ke64, st64, _, w64 = gpu_keff(kap, leaves[leaves[:, 2] <= 32], tau, nu, eps, g, 0.0, 256, warm=1, storage=2)
    assert w64 == 0
    for i, leaf in enumerate(leaves[leaves[:, 2] <= 32]):
        ref = oracle_keff(kap, leaf, tau, nu, eps, g, 0.0, 256, warm=True)
        assert_keff_close(ke64[i], ref["keff"], 1e-4)


def test_darcy_start_converges_to_the_rest_start_k_star_in_fewer_steps():
    """Quadtree leaves of a 256^2 log-normal field (sigma 2) at tol 1e-8: the warm-started runs stop
    with the K* of the runs from rest within the stop test's band (2e-3: a run stops once its mean
    velocity drifts by less than tol x check_every per check, and the remaining error of either
    start decays over up to ~1e5 steps) and take fewer steps in total. Both starts are compared
    on every entry of K* (off-diagonal ones relative to sqrt(K*_xx K*_yy)): a Darcy-started run
    stops on the whole mean velocity vector, so its transverse component has settled too."""
    kap = synth.lognormal_kappa(256, 256, 8.0, 2.0, seed=29)
    leaves = synth.quadtree_leaves(256, 256, seed=29)
    tau, nu, eps, g = 1.0, 1.0 / 6.0, 1.0, 1e-6
    cold, sc, nc, _ = gpu_keff(kap, leaves, tau, nu, eps, g, 1e-8, 200000)
    warm, sw, nw, _ = gpu_keff(kap, leaves, tau, nu, eps, g, 1e-8, 200000, warm=1)
    ok = (sc == 0) & (sw == 0)
    assert ok.mean() > 0.8
    big = leaves[:, 2] >= 16
    sel = ok & big
    scale = np.sqrt(np.abs(cold[:, 0] * cold[:, 3]))
    d_diag = np.maximum(np.abs(warm[:, 0] / cold[:, 0] - 1), np.abs(warm[:, 3] / cold[:, 3] - 1))[sel]
    d_off = np.maximum(np.abs(warm[:, 1] - cold[:, 1]), np.abs(warm[:, 2] - cold[:, 2]))[sel] / scale[sel]
    cost = leaves[:, 2].astype(np.float64) ** 2
    uc, uw = (cost * nc.sum(axis=1))[big].sum(), (cost * nw.sum(axis=1))[big].sum()
    print(f"\n{sel.sum()} leaves: diagonal max {d_diag.max():.2e} median {np.median(d_diag):.2e}; "
          f"off-diagonal max {d_off.max():.2e} median {np.median(d_off):.2e}; "
          f"lattice updates {uw / uc:.3f} of the rest start's")
    assert d_diag.max() <= 2e-3 and np.median(d_diag) <= 1e-4
    assert d_off.max() <= 2e-3 and np.median(d_off) <= 1e-4
    assert uw < 0.8 * uc


def test_darcy_start_tolerance_stop_matches_oracle():
    """Darcy-started runs on high-contrast 16 x 16 patches (sigma 3) stopped at tol 1e-8 on the
    whole mean velocity vector, against the oracle's warm-started runs. Where both stop at the
    same check, K* agrees to 2e-4 (FP32 states on a contrast of e^+-9). The FP32 rounding of the
    mean velocity is a sizeable part of the drift allowed per check (6.4e-7 relative), so a stop
    decision often moves by a check or more; both results then lie in the stop test's band and
    agree to 1e-3."""
    kap = synth.lognormal_kappa(64, 64, 4.0, 3.0, seed=102)
    leaves = synth.uniform_leaves(64, 64, 16)
    tau, nu, eps, g = 1.0, 1.0 / 6.0, 1.0, 1e-6
    ke, st, steps, worst = gpu_keff(kap, leaves, tau, nu, eps, g, 1e-8, 200000, warm=1)
    assert worst == 0
    for i in range(len(leaves)):
        ref = oracle_keff(kap, leaves[i], tau, nu, eps, g, 1e-8, 200000, warm=True)
        eq = list(steps[i]) == list(ref["steps"])
        assert_keff_close(ke[i], ref["keff"], 2e-4 if eq else 1e-3)


def test_darcy_start_of_a_uniform_field_is_already_steady():
    """A uniform field: the Darcy start is Eq. 19's steady state, so every run on a warm-started
    patch stops at the first possible test (128 steps) with K* = kappa."""
    kap = np.full((96, 96), 0.05, dtype=np.float32)
    leaves = np.array([[0, 0, 64], [64, 0, 32], [64, 32, 16]], dtype=np.int32)
    ke, st, steps, worst = gpu_keff(kap, leaves, 0.8, 0.05, 0.9, 1e-6, 1e-7, 20000, warm=1)
    assert worst == 0 and (steps == 128).all()
    np.testing.assert_allclose(ke[:, 0], 0.05, rtol=2e-5)
    np.testing.assert_allclose(ke[:, 3], 0.05, rtol=2e-5)


def test_warm_start_value_is_checked():
    import torch
    lbm = _lbm()
    kap = torch.full((16, 16), 0.05, device="cuda")
    lt = torch.tensor([[0, 0, 16]], dtype=torch.int32, device="cuda")
    with pytest.raises(lbm.LbmError) as ei:
        lbm.local_keff(lbm.Params(nx=16, ny=16, tau=1.0, warm_start=2), kap, lt, 1e-6, 0.0, 10)
    assert ei.value.status == lbm.LBM_EINVAL


@pytest.mark.parametrize("tau,steps,k", [(1.0, 300, 64), (0.8, 130, 7), (1.0, 1, 64)])
def test_every_side_of_the_register_solver_matches_oracle(tau, steps, k):
    """Sides that are multiples of 4 keep their distributions in registers; each packs its rows into
    lanes and warps in another way (a part of a warp, one, two, four or sixteen warps, with idle lanes or
    without). 1e-4 is the FP32 bar of this file. The sides in between take the other solver in the same
    call."""
    kap = synth.lognormal_kappa(96, 96, 6.0, 1.0, seed=77)
    kap[5:9, 5:9] = 0.0
    sides = list(range(4, 65, 4)) + [5, 18, 63]
    leaves = np.array([[(7 * s) % (97 - s), (5 * s) % (97 - s), s] for s in sides + [8, 8, 8, 12, 16, 16]], dtype=np.int32)
    ke, st, n, worst = gpu_keff(kap, leaves, tau, 0.1, 0.9, 1e-6, 0.0, steps, k=k)
    assert worst == 0 and (n == steps).all()
    for i in range(len(leaves)):
        ref = oracle_keff(kap, leaves[i], tau, 0.1, 0.9, 1e-6, 0.0, steps, k=k)
        assert_keff_close(ke[i], ref["keff"], 1e-4)


@pytest.mark.parametrize("storage,warm", [(0, 0), (2, 0), (0, 1)])
def test_time_limit_reaches_jobs_still_in_the_queue(storage, warm):
    """Past the wall-clock limit no leaf is reported as solved: neither the jobs that run nor those that wait in a
    size's queue. Sides of the register solver (32, 8) and of the shared-memory one (30, 7), from rest and from the
    Darcy state, several times what the chip holds at once."""
    import torch
    lbm = _lbm()
    kap = torch.from_numpy(synth.lognormal_kappa(512, 512, 8.0, 1.0, seed=24).astype(np.float32)).cuda()
    leaves = np.concatenate([synth.uniform_leaves(512 // s * s, 512 // s * s, s) for s in (32, 30, 8, 7)] * 4)
    p = lbm.Params(nx=512, ny=512, tau=1.0, storage=storage, warm_start=warm)
    try:
        lbm.lbm_set_time_limit(2e-4)
        ke, st, steps, worst = lbm.local_keff(p, kap, torch.from_numpy(leaves.astype(np.int32)).cuda(), 1e-6, 1e-14,
                                              10_000_000, 64)
        assert worst == lbm.LBM_ETIMEOUT
        assert (st == lbm.LBM_ETIMEOUT).all()
        assert torch.isnan(ke.reshape(-1, 2, 2)[:, 0, :][steps == 0]).all()
    finally:
        lbm.lbm_set_time_limit(600.0)


@pytest.mark.parametrize("sizes,steps,tol", [(range(1, 41), 300, 0.0), ([16] * 40 + [15] * 900, 200000, 1e-6),
                                             ([64] * 3 + [12] * 500 + [63, 2], 200000, 1e-6)])
def test_batches_of_both_solvers_equal_their_halves(sizes, steps, tol):
    """A batch whose sides go to both solvers runs them side by side; K*, status and steps of a leaf are those of a batch of
    its own kind bit for bit, and the outputs are complete when the call returns (read at once, ten times over)."""
    import torch
    lbm = _lbm()
    kap = torch.from_numpy(synth.lognormal_kappa(512, 512, 8.0, 1.0, seed=27).astype(np.float32)).cuda()
    r = np.random.default_rng(5)
    size = r.permutation(np.array(list(sizes)))
    leaves = np.stack([r.integers(0, 513 - size), r.integers(0, 513 - size), size], axis=1).astype(np.int32)
    p = lbm.Params(nx=512, ny=512, tau=1.0)

    def run(lv):
        return [t.cpu() for t in lbm.local_keff(p, kap, torch.from_numpy(lv).cuda(), 1e-6, tol, steps, 64)[:3]]

    reg = (size >= 4) & (size % 4 == 0)
    ref = [torch.empty((len(leaves), *t.shape[1:]), dtype=t.dtype) for t in run(leaves[:1])]
    for which in (reg, ~reg):
        for a, b in zip(ref, run(leaves[which])):
            a[torch.from_numpy(which)] = b
    for _ in range(10):
        for a, b in zip(run(leaves), ref):
            assert torch.equal(a, b)


def test_time_limit_covers_both_solvers_of_a_batch():
    """The limit counts from the batch's first launch. With a queue built on the device the register solver takes every
    SM, and the shared-memory solver its jobs after it: a limit that either would meet alone, but not both, runs out.
    Leaves of 16 and 1 cells with a margin of 2 are patches of 20 (register solver) and 5 (shared-memory solver)."""
    import time

    import torch
    lbm = _lbm()
    kap = torch.from_numpy(synth.lognormal_kappa(512, 512, 8.0, 1.0, seed=29).astype(np.float32)).cuda()
    r = np.random.default_rng(6)
    p = lbm.Params(nx=512, ny=512, tau=1.0, margin=2)

    def leaves(s, n):
        return np.stack([r.integers(0, 513 - s, n), r.integers(0, 513 - s, n), np.full(n, s)], axis=1).astype(np.int32)

    reg, other = leaves(16, 4000), leaves(1, 16000)
    with lbm.Surrogate(2, 0) as sur:
        def run(lv):
            lv = torch.from_numpy(lv).cuda()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            st, nfb, worst = sur.keff(p, kap, lv, 1e-30, 1e-6, 0.0, 60000)[2:]
            return time.perf_counter() - t0, nfb, worst, st.cpu().numpy()

        run(reg[:10])
        t = [run(reg), run(other)]
        limit = 1.3 * max(t[0][0], t[1][0])
        assert [x[1:3] for x in t] == [(len(reg), lbm.LBM_OK), (len(other), lbm.LBM_OK)]
        assert t[0][0] + t[1][0] > 1.2 * limit, t
        try:
            lbm.lbm_set_time_limit(limit)
            both = run(np.concatenate([reg, other]))
            assert both[2] == lbm.LBM_ETIMEOUT and (both[3][:len(reg)] == lbm.LBM_OK).all()
        finally:
            lbm.lbm_set_time_limit(600.0)
