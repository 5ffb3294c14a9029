"""The FP64 solve on the tensor cores (csrc/kernels_solve64.cu, N <= 64) where its tiling can go wrong: N around
the 16-deep steps and its maximum, rows around the 8-row groups, the 32-row halves and the 64-row tile,
several tiles per CTA (grid_blocks caps the CTAs), rows and members of very different size, zero columns.
Against the oracle's CG after a fixed number of steps (bar 1e-11, that of the existing FP64 iterates) and
the exact analysis (1e-8 at tol 1e-10)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed):
    side = max(4, int(np.ceil(np.sqrt(2 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=np.float64)


def _run(lib, p, **cfg):
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp64", **cfg)
    Xa = an.analyze(torch.from_numpy(np.ascontiguousarray(p.Xf)).cuda(), torch.from_numpy(p.y).cuda(), seed=6, counter=2)
    return an, Xa.cpu().numpy(), an.stats()


@pytest.mark.parametrize("pc", [0, 1])
@pytest.mark.parametrize("N,m,G", [(2, 9, 1), (15, 40, 1), (16, 64, 1), (17, 65, 1), (33, 97, 2), (40, 129, 1), (63, 500, 3), (64, 1500, 4), (64, 9000, 0)])
def test_iterates_and_analyses(lib, N, m, G, pc):
    p = _problem(N, m, 31 * N + m)
    p.r[:] = 0.8   # without preconditioning this path takes such R; with it the oracle's iterates are the same
    k = min(4, N, m)
    an, Xa, st = _run(lib, p, fixed_iters=k, precondition=pc, grid_blocks=G)
    E = oracle.obs_perturbations(6, 2, p.r, p.N)
    ref, info = oracle.cgd_enkf(p.Xf, p.rowptr, p.col, p.w, p.r, p.y, E, fixed_iters=k)
    _, _, Z, W = (t.cpu().numpy() for t in an.intermediates())
    assert np.linalg.norm(Z - info["Z"]) <= 1e-11 * np.linalg.norm(info["Z"])
    assert oracle.rel_frobenius(Xa, ref) <= 1e-11
    _, Xa, st = _run(lib, p, tol=1e-10, precondition=pc, grid_blocks=G)
    exact = oracle.enkf_exact(p.Xf, p.rowptr, p.col, p.w, p.r, p.y, E)
    assert st["status"] == "ok" and st["true_relres_max"] <= 2e-10
    assert oracle.rel_frobenius(Xa, exact) <= 1e-8


def test_rows_and_members_of_different_size(lib):
    p = _problem(48, 700, 9)
    rng = np.random.default_rng(1)
    p.Xf *= 10.0 ** rng.uniform(-1, 1, p.N)[None, :]
    p.w = p.w * np.repeat(10.0 ** rng.uniform(-4, 4, p.m), np.diff(p.rowptr))
    p.r[:] = 1.0
    k = 4
    an, Xa, st = _run(lib, p, fixed_iters=k, grid_blocks=3)
    E = oracle.obs_perturbations(6, 2, p.r, p.N)
    ref, info = oracle.cgd_enkf(p.Xf, p.rowptr, p.col, p.w, p.r, p.y, E, fixed_iters=k)
    Z = an.intermediates()[2].cpu().numpy()
    assert np.linalg.norm(Z - info["Z"]) <= 1e-11 * np.linalg.norm(info["Z"])


def test_zero_columns_and_statuses(lib):
    p = _problem(20, 300, 5)
    p.r[:] = 1.0
    X, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp64", tol=1e-10, grid_blocks=2)
    # E = H x_j - y for member 3: D_3 = 0, a column of no steps
    Zo = oracle.ensemble_stats(p.Xf, p.rowptr, p.col, p.w)[2]
    E = np.random.default_rng(2).standard_normal((p.m, p.N))
    E[:, 3] = Zo[:, 3] - p.y
    Xa = an.analyze_with_E(X, y, torch.from_numpy(E).cuda()).cpu().numpy()
    assert an.stats()["status"] == "ok"
    assert oracle.rel_frobenius(Xa, oracle.enkf_exact(p.Xf, p.rowptr, p.col, p.w, p.r, p.y, E)) <= 1e-8
    _, Xa, st = _run(lib, p, tol=1e-12, max_iter=3, grid_blocks=2)
    assert st["status"] == "not_converged" and st["iters_max"] == 3 and np.all(np.isfinite(Xa))
    p.Xf[p.col[3], 4] = np.nan
    _, _, st = _run(lib, p, tol=1e-8, grid_blocks=2)
    assert st["status"] == "nonfinite"


def test_varying_r(lib):
    # preconditioned, a varying R: the preconditioned persistent solve's system in whitened rows
    p = _problem(50, 1200, 8)
    p.r[:] = 10.0 ** np.random.default_rng(3).uniform(-2, 2, p.m)
    _, Xa, st = _run(lib, p, tol=1e-12, precondition=1, grid_blocks=5)
    E = oracle.obs_perturbations(6, 2, p.r, p.N)
    exact = oracle.enkf_exact(p.Xf, p.rowptr, p.col, p.w, p.r, p.y, E)
    assert st["status"] == "ok"
    assert oracle.rel_frobenius(Xa, exact) <= 1e-8


@pytest.mark.parametrize("N,m,pc,varying", [(64, 1500, 1, True), (40, 900, 0, False), (24, 700, 0, True), (20, 90, 1, True)])
def test_the_allocation_free_entry_point_takes_the_same_route(lib, N, m, pc, varying):
    # the same analysis through a handle and on the fixed array; without preconditioning the latter does not
    # know whether R is constant and keeps the m-vector solve, whose result agrees to the tolerance
    p = _problem(N, m, 3 * N + m)
    if not varying:
        p.r[:] = 0.9
    _, Xa, st = _run(lib, p, tol=1e-11, precondition=pc)
    cfg = lib.default_config(p.n, p.m, p.N, precision="fp64", tol=1e-11, precondition=pc)
    dev = (torch.from_numpy(p.rowptr).cuda(), torch.from_numpy(p.col).cuda(), torch.from_numpy(p.w).cuda(), torch.from_numpy(p.r).cuda())
    X2, st2 = lib.analyze_noalloc(cfg, *dev, torch.from_numpy(np.ascontiguousarray(p.Xf)).cuda(), torch.from_numpy(p.y).cuda(), seed=6, counter=2)
    assert st["status"] == "ok" and st2["status"] == "ok"
    X2 = X2.cpu().numpy()
    if pc or varying:
        assert np.array_equal(Xa, X2)
    else:
        assert oracle.rel_frobenius(X2, Xa) <= 1e-9
