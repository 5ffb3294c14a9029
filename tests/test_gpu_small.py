"""The small-problem solve (csrc/kernels_small.cu: a thread-block cluster per column) for every
cluster size and around its tiles: FP64 iterates after a fixed number of steps and converged
FP32 analyses, against the oracle's CG and exact analysis and against the persistent solve of the
same problem (grid_blocks > 0 selects it). Bars: 1e-11 for FP64 iterates (as for the persistent
solve's), 1e-6 for FP32 analyses."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed, dtype):
    side = max(4, int(np.ceil(np.sqrt(2 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=dtype)


def _run(lib, p, prec, **cfg):
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision=prec, **cfg)
    dt = torch.float64 if prec == "fp64" else torch.float32
    Xa = an.analyze(torch.from_numpy(np.ascontiguousarray(p.Xf)).to("cuda", dt), torch.from_numpy(p.y).cuda(), seed=6, counter=2)
    return an, Xa.double().cpu().numpy(), an.stats()


def _small(st, N):
    # N clusters of one to eight CTAs (how many of a size are resident at once is the chip's)
    return st["grid_blocks"] % N == 0 and 1 <= st["grid_blocks"] // N <= 8


# one CTA per column and no row beyond it, odd sizes, up to eight CTAs with ragged blocks
FP64 = [(2, 1), (20, 20), (33, 31), (64, 150), (128, 90), (64, 301), (37, 530), (17, 1100)]


@pytest.mark.parametrize("pc", [0, 1])
@pytest.mark.parametrize("N,m", FP64)
def test_fp64_iterates_match_the_oracle(lib, N, m, pc):
    p = _problem(N, m, 31 * N + m, np.float64)
    p.r[:] = 0.8   # without preconditioning FP64 takes this path for such R; with it the oracle's iterates are the same
    k = min(4, N)
    an, Xa, st = _run(lib, p, "fp64", fixed_iters=k, precondition=pc)
    assert _small(st, N), st
    E = oracle.obs_perturbations(6, 2, p.r, p.N)
    ref, info = oracle.cgd_enkf(p.Xf, p.rowptr, p.col, p.w, p.r, p.y, E, fixed_iters=k)
    _, D, Z, W = (t.cpu().numpy() for t in an.intermediates())
    if m >= k:   # before the Krylov space is exhausted
        assert np.linalg.norm(Z - info["Z"]) <= 1e-11 * np.linalg.norm(info["Z"])
    assert oracle.rel_frobenius(Xa, ref) <= 1e-11
    an2, X2, st2 = _run(lib, p, "fp64", tol=1e-10, precondition=pc)
    an3, X3, st3 = _run(lib, p, "fp64", tol=1e-10, precondition=pc, grid_blocks=3)
    assert st2["status"] == "ok" and st3["status"] == "ok" and st2["true_relres_max"] <= 2e-10
    assert oracle.rel_frobenius(X2, X3) <= 1e-8


@pytest.mark.parametrize("N,m", [(2, 3), (20, 200), (31, 500), (128, 380), (64, 900), (37, 3001), (18, 5003)])
def test_fp32_plain_analyses_match_the_exact_and_the_persistent_solve(lib, N, m):
    p = _problem(N, m, 17 * N + m, np.float32)
    an, Xa, st = _run(lib, p, "fp32", tol=1e-8)
    assert _small(st, N) and st["status"] == "ok" and st["true_relres_max"] <= 1e-8, st
    E = oracle.obs_perturbations(6, 2, p.r, p.N)
    ref = oracle.enkf_exact(p.Xf.astype(np.float64), p.rowptr, p.col, p.w, p.r, p.y, E)
    assert oracle.rel_frobenius(Xa, ref) <= 1e-6
    _, X2, st2 = _run(lib, p, "fp32", tol=1e-8, grid_blocks=5)
    assert oracle.rel_frobenius(Xa, X2) <= 1e-6


def test_statuses(lib):
    p = _problem(20, 300, 5, np.float64)
    p.r[:] = 1.0
    _, Xa, st = _run(lib, p, "fp64", tol=1e-12, max_iter=3)
    assert st["status"] == "not_converged" and st["iters_max"] == 3 and np.all(np.isfinite(Xa))
    p.Xf[p.col[3], 4] = np.nan
    _, _, st = _run(lib, p, "fp64", tol=1e-8)
    assert st["status"] == "nonfinite"
