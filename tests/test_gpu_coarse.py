"""Coarse (upscaled) run, upscaling and block averages on the GPU.

Parity of the coarse step with the tensor drag of Eq. 18 is checked against the
oracle element by element. The fine-vs-coarse comparisons of Section 4.3 have
no printed numbers (the paper shows them as figures only), so those tests check
the orderings and sizes the paper states in words: the coarse run with K*
follows the block-averaged fine run, and in the Brinkman case (Section 4.3.2)
K* computed with nu_eff does better than K*err computed with nu_eff = 0.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _lbm():
    import paper_1312_0195_gb300 as lbm
    return lbm


def _t(a, dtype=np.float32):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def test_block_average_matches_reshape_mean():
    lbm = _lbm()
    a = np.random.default_rng(0).standard_normal((60, 80)).astype(np.float32)
    out = lbm.lbm_block_average(_t(a), 20).cpu().numpy()
    ref = a.astype(np.float64).reshape(3, 20, 4, 20).mean(axis=(1, 3))
    np.testing.assert_allclose(out, ref, rtol=1e-6, atol=1e-7)


@pytest.mark.parametrize("with_field", [False, True])
def test_coarse_run_tensor_drag_matches_oracle(with_field):
    """Coarse step with a full K* tensor per cell (Eq. 18) against the oracle's 2x2 solve."""
    import torch
    lbm = _lbm()
    rng = np.random.default_rng(5)
    r = 4
    cx, cy = 40, 28
    a = 10 ** rng.uniform(-2, 0, size=(cy, cx))
    b = 10 ** rng.uniform(-2, 0, size=(cy, cx))
    off = 0.4 * np.sqrt(a * b) * rng.uniform(-1, 1, size=(cy, cx))
    kf = np.stack([a, off, off * 0.9, b], axis=-1)            # fine lattice units, not symmetric
    fine = lbm.Params(nx=cx * r, ny=cy * r, tau=0.8, nu=0.05, eps=0.9, gx=2e-6, gy=-1e-6)
    gco = None
    if with_field:
        gco = np.ascontiguousarray(synth.sinusoidal_g_field(cx, 1e-6)[:, :cy, :cx])
    steps = 400
    u = torch.empty((cy, cx), device="cuda")
    v = torch.empty_like(u)
    rho = torch.empty_like(u)
    st, n = lbm.lbm_coarse_run(fine, r, _t(kf, np.float64), None if gco is None else _t(gco), steps, 0.0, 0,
                               rho, u, v)
    assert st == 0 and n == steps
    c = lbm.lbm_coarse_params(fine, r)
    assert abs(c.tau - (0.5 + 0.3 / r)) < 1e-15 and abs(c.nu - 0.05 / r) < 1e-15
    prob = oracle.Problem(c.tau, c.nu, c.eps, ktensor=kf / r ** 2, g=(c.gx, c.gy),
                          gfield=None if gco is None else gco.astype(np.float32).astype(np.float64) * r)
    f = prob.rest()
    prob.run(f, steps)
    ro, uo, vo = prob.fields(f)
    scale = max(np.abs(uo).max(), np.abs(vo).max())
    assert np.abs(u.cpu().numpy() - uo).max() <= 1e-5 * scale
    assert np.abs(v.cpu().numpy() - vo).max() <= 1e-5 * scale
    assert np.abs(rho.cpu().numpy() - ro).max() <= 1e-6


def test_upscale_lbm_only_matches_oracle_blocks():
    import torch
    lbm = _lbm()
    kap = synth.lognormal_kappa(64, 48, 6.0, 1.5, seed=31).astype(np.float32)
    p = lbm.Params(nx=64, ny=48, tau=1.0, eps=1.0)
    keff = torch.empty((3, 4, 4), dtype=torch.float64, device="cuda")
    st, nfb = lbm.lbm_upscale(p, _t(kap), 16, keff, 1e-6, 0.0, 640)
    assert st == 0 and nfb == 12
    ke = keff.cpu().numpy()
    for J in range(3):
        for I in range(4):
            patch = kap[J * 16:(J + 1) * 16, I * 16:(I + 1) * 16].astype(np.float64)
            ref = oracle.local_keff(patch, 1.0, 1.0 / 6.0, 1.0, 1e-6, tol=0.0, max_steps=640, check_every=64)
            np.testing.assert_allclose(ke[J, I, [0, 3]], ref["keff"][[0, 3]], rtol=1e-4)


def _fine_fields(lbm, p, kap, gfield, steps):
    with lbm.Grid(p, _t(kap), _t(gfield)) as G:
        G.step(steps, 0.0, 0)
        rho, u, v = G.fields()
        return (lbm.lbm_block_average(rho, 10), lbm.lbm_block_average(u, 10), lbm.lbm_block_average(v, 10))


def _coarse(lbm, p, keff, gco, steps):
    import torch
    u = torch.empty((40, 40), device="cuda")
    v = torch.empty_like(u)
    rho = torch.empty_like(u)
    lbm.lbm_coarse_run(p, 10, keff, _t(gco), steps, 0.0, 0, rho, u, v)
    return rho, u, v


def _rel(a, b):
    a = a.double().cpu().numpy()
    b = b.double().cpu().numpy()
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _iso(kappa_blocks):
    """[40, 40] scalar block permeability as an isotropic K* tensor field."""
    import torch
    k = np.zeros((40, 40, 4))
    k[..., 0] = kappa_blocks
    k[..., 3] = kappa_blocks
    return torch.from_numpy(k).cuda()


def test_fiveblock_darcy_upscaled_run_follows_fine_run():
    """Section 4.3.1 (E5): 400^2 fine grid, Eq. 23, G = (sin pi x, sin pi y), tau = 0.5; K* of every
    10x10 block by local LBM; 40^2 coarse run; compared near steady state (3e6 fine steps = 6
    time constants of the slowest pressure mode, 3e5 coarse steps, the same physical time).
    The coarse run with K* must follow the block-averaged fine run, and do so better than a
    coarse run with the naive block-mean permeability."""
    import torch
    lbm = _lbm()
    ex = synth.paper_experiment("E5_fine")
    kap = ex["kappa"].astype(np.float32)
    p = lbm.Params(nx=400, ny=400, tau=ex["tau"], nu=ex["nu"], eps=ex["eps"])
    keff = torch.empty((40, 40, 4), dtype=torch.float64, device="cuda")
    st, _ = lbm.lbm_upscale(p, _t(kap), 10, keff, 5e-7, 1e-9, 400000)
    assert st == 0
    k = keff.cpu().numpy() / ex["k_const"]
    mask = synth.fiveblock_coarse_kappa_eq24(40, 1.0, 0.0) == 1.0           # the five K = K_const blocks
    np.testing.assert_allclose(k[mask][:, [0, 3]], 1.0, rtol=1e-4)
    sin_blocks = k[~mask]
    assert abs(np.mean(0.5 * (sin_blocks[:, 0] + sin_blocks[:, 3])) - 8.485) < 1e-3
    gfine = ex["gfield"].astype(np.float32)
    gco = synth.sinusoidal_g_field(40, synth.LatticeUnits(0.0025, 2.5e-5).force(1.0))   # fine lattice units
    fine_steps = 3000000
    rf, uf, vf = _fine_fields(lbm, p, kap, gfine, fine_steps)
    _, uc, vc = _coarse(lbm, p, keff, gco, fine_steps // 10)
    naive = ex["kappa"].reshape(40, 10, 40, 10).mean(axis=(1, 3))           # arithmetic block mean of kappa
    _, un, vn = _coarse(lbm, p, _iso(naive), gco, fine_steps // 10)
    eu, ev = _rel(uc, uf), _rel(vc, vf)
    en = _rel(un, uf)
    print(f"E5 coarse vs block-averaged fine: rel L2 u {eu:.3e}, v {ev:.3e}; naive block mean: u {en:.3e}")
    assert eu < 0.05 and ev < 0.05
    assert eu < en


def test_fiveblock_brinkman_kstar_beats_kstar_err():
    """Section 4.3.2 (E6): with nu_eff > 0 the local problems must use the same nu_eff; K*err computed
    with nu_eff = 0 (the paper's 8.485 against 7.367) makes the coarse run deviate visibly."""
    import torch
    lbm = _lbm()
    ex = synth.paper_experiment("E6_fine")
    kap = ex["kappa"].astype(np.float32)
    p = lbm.Params(nx=400, ny=400, tau=ex["tau"], nu=ex["nu"], eps=ex["eps"])
    p_err = lbm.Params(nx=400, ny=400, tau=0.5, nu=ex["nu"], eps=ex["eps"])
    keff = torch.empty((40, 40, 4), dtype=torch.float64, device="cuda")
    keff_err = torch.empty_like(keff)
    # weak drag at tau ~ 1/2: per-step momentum increments are ~1e-5 of the momentum, below what FP32
    # storage resolves over 10^6 steps, so these local problems run on the FP64 local solver
    p64 = lbm.Params(nx=400, ny=400, tau=ex["tau"], nu=ex["nu"], eps=ex["eps"], storage=lbm.LBM_F64)
    p64_err = lbm.Params(nx=400, ny=400, tau=0.5, nu=ex["nu"], eps=ex["eps"], storage=lbm.LBM_F64)
    lbm.lbm_upscale(p64, _t(kap), 10, keff, 5e-7, 1e-10, 2000000)
    lbm.lbm_upscale(p64_err, _t(kap), 10, keff_err, 5e-7, 1e-10, 2000000)
    k = keff.cpu().numpy() / ex["k_const"]
    ke = keff_err.cpu().numpy() / ex["k_const"]
    mask = synth.fiveblock_coarse_kappa_eq24(40, 1.0, 0.0) == 1.0
    s_k = np.mean(0.5 * (k[~mask][:, 0] + k[~mask][:, 3]))
    s_e = np.mean(0.5 * (ke[~mask][:, 0] + ke[~mask][:, 3]))
    print(f"E6 K*/K_const {s_k:.5f} (paper 7.367), K*err/K_const {s_e:.5f} (paper 8.485)")
    assert abs(s_k - 7.367) < 1e-3 and abs(s_e - 8.485) < 1e-3
    gfine = ex["gfield"].astype(np.float32)
    gco = synth.sinusoidal_g_field(40, synth.LatticeUnits(0.0025, 2.5e-5).force(1.0))   # fine lattice units
    fine_steps = 100000
    rf, uf, vf = _fine_fields(lbm, p, kap, gfine, fine_steps)
    _, uc, vc = _coarse(lbm, p, keff, gco, fine_steps // 10)
    _, ue, ve = _coarse(lbm, p, keff_err, gco, fine_steps // 10)
    e_good, e_bad = _rel(uc, uf), _rel(ue, uf)
    print(f"E6 coarse vs fine: rel L2 u with K* {e_good:.3e}, with K*err {e_bad:.3e}")
    assert e_good < e_bad


@pytest.mark.parametrize("nx,ny", [(56, 8), (65, 31), (20, 130)])
def test_coarse_run_fused_passes_equal_single_steps_bitwise(nx, ny, monkeypatch):
    """The coarse run's tensor drag in passes of several steps against the one-step kernel."""
    import torch
    import paper_1312_0195_gb300 as lbm
    g = torch.Generator().manual_seed(nx)
    K = 0.05 * torch.rand((ny, nx, 4), generator=g, dtype=torch.float64)
    K[..., 0] += 0.2
    K[..., 3] += 0.2
    field = torch.rand((2, ny, nx), generator=g).cuda() * 1e-6
    for bc in (lbm.LBM_BC_PERIODIC, lbm.LBM_BC_WALLS_Y):
        for force in (None, field):
            got = []
            for single in (False, True):
                if single:
                    monkeypatch.setenv("LBM_STEP_VEC", "1")
                else:
                    monkeypatch.delenv("LBM_STEP_VEC", raising=False)
                out = [torch.empty((ny, nx), device="cuda") for _ in range(3)]
                lbm.lbm_coarse_run(lbm.Params(nx=4 * nx, ny=4 * ny, tau=1.0, gx=1e-6, bc=bc), 4, K.cuda(), force, 777,
                                   0.0, 64, *out)
                got.append(out)
            for a, b in zip(*got):
                assert torch.equal(a, b)


@pytest.mark.parametrize("nx,ny", [(777, 401), (1024, 520), (35001, 9)])
def test_coarse_run_of_large_lattices_equals_single_steps_bitwise(nx, ny, monkeypatch):
    """Coarse lattices too large to stay in shared memory go through passes of up to four steps, the tensor drag with and
    without a force field, walls, odd columns and few rows; fixed steps, with checks inside and beside a pass, and a
    stop at the tolerance. Fields and the step count equal the one-step kernel's."""
    import torch
    import paper_1312_0195_gb300 as lbm
    g = torch.Generator().manual_seed(nx)
    K = 0.05 * torch.rand((ny, nx, 4), generator=g, dtype=torch.float64)
    K[..., 0] += 0.2
    K[..., 3] += 0.2
    K = K.cuda()
    field = torch.rand((2, ny, nx), generator=g).cuda() * 1e-6
    for bc in (lbm.LBM_BC_PERIODIC, lbm.LBM_BC_WALLS_Y):
        for force in (None, field):
            got = []
            for single in (False, True):
                if single:
                    monkeypatch.setenv("LBM_STEP_VEC", "1")
                else:
                    monkeypatch.delenv("LBM_STEP_VEC", raising=False)
                runs = []
                for steps, tol, check in ((77, 0.0, 0), (77, 0.0, 19), (130, 0.0, 64), (400, 0.03, 13)):
                    out = [torch.empty((ny, nx), device="cuda") for _ in range(3)]
                    _, n = lbm.lbm_coarse_run(lbm.Params(nx=4 * nx, ny=4 * ny, tau=1.0, gx=1e-6, bc=bc), 4, K, force, steps,
                                              tol, check, *out)
                    runs.append((n, out))
                got.append(runs)
            for (n, a), (m, b) in zip(*got):
                assert n == m
                for x, y in zip(a, b):
                    assert torch.equal(x, y)
