"""The preconditioned solve in Krylov coordinates (csrc/krylov.cuh) where its N x N recurrences end early: a
step limit, and inputs that are not numbers."""
import numpy as np
import pytest

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
