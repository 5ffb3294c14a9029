"""The preconditioned solve in Krylov coordinates (csrc/krylov.cuh) where its N x N recurrences are hard:
variances of R far below the ensemble's, a member far larger than the others, a step limit, and inputs
that are not numbers.

Bar of the analyses: Z, HA and the sums hold about 47 bits and the residual of a rounded Z is up to
lambda = the largest eigenvalue of HA^T R^-1 HA/(N-1) times its rounding, so the increment X_a - X_f is off by
at most 1e-6 (the FP32 path's bar) + 2^-46 lambda of its size, converged or not."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed):
    side = max(4, int(np.ceil(np.sqrt(2 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=np.float32)


def _run(lib, p, prec="fp32", **cfg):
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision=prec, precondition=1, tol=1e-8, **cfg)
    Xa = an.analyze(torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda(), seed=6, counter=2).double().cpu().numpy()
    st = an.stats()
    an.close()
    return Xa, st


def _check(lib, p, prec):
    X = p.Xf.astype(np.float64)
    HA = oracle.ensemble_stats(X, p.rowptr, p.col, p.w)[4]
    lam = np.linalg.eigvalsh(HA.T @ (HA / p.r[:, None]) / (p.N - 1)).max()
    ref = oracle.enkf_exact(X, p.rowptr, p.col, p.w, p.r, p.y, oracle.obs_perturbations(6, 2, p.r, p.N), m_dense=0)
    Xa, st = _run(lib, p, prec)
    assert st["status"] in ("ok", "not_converged"), st
    err = np.linalg.norm(Xa - ref) / np.linalg.norm(ref - X)
    assert err <= 1e-6 + 2.0 ** -46 * lam, (err, lam, st)


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("N,m", [(20, 4000), (64, 1024), (100, 2000)])
@pytest.mark.parametrize("decades", [4, 8])
def test_observations_far_more_accurate_than_the_ensemble(lib, N, m, decades, prec):
    p = _problem(N, m, 3)
    p.r = p.r * 10.0 ** -decades
    _check(lib, p, prec)


@pytest.mark.parametrize("factor", [1e2, 1e4])
def test_a_member_far_larger_than_the_others(lib, factor):
    p = _problem(64, 1024, 6)
    p.Xf[:, 5] *= np.float32(factor)
    _check(lib, p, "fp32")


@pytest.mark.parametrize("N,m", [(20, 300), (64, 2000), (100, 2000)])
@pytest.mark.parametrize("steps", [1, 3])
def test_a_step_limit_leaves_no_column_worse_than_no_analysis(lib, N, m, steps):
    # (r, R^-1 r) <= (d, R^-1 d) for every column, so ||r|| <= sqrt(max r / min r) ||d||
    p = _problem(N, m, 8)
    _, st = _run(lib, p, max_iter=steps)
    assert st["status"] == "not_converged" and st["iters_max"] <= steps
    assert 0 < st["true_relres_max"] <= np.sqrt(p.r.max() / p.r.min()) * (1 + 1e-6), st


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_an_observation_that_is_no_number_leaves_the_forecast(lib, prec, bad):
    p = _problem(64, 1024, 7)
    p.y[500] = bad
    Xa, st = _run(lib, p, prec)
    assert st["status"] == "nonfinite" and np.array_equal(Xa, p.Xf.astype(np.float64)), st
