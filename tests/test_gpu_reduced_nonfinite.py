"""Inputs that are not numbers in the Reduced form: its N x N CG (csrc/kernels_reduced.cu) ends at once on a
right-hand side with a NaN or an infinity, and the analysis has to say so instead of reporting a
converged one of zero steps."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed, dt):
    side = max(4, int(np.ceil(np.sqrt(1.5 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=dt)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["y", "X", "E"])
@pytest.mark.parametrize("N,fixed", [(20, 0), (64, 0), (100, 0), (64, 5)])
def test_status_and_residuals_say_nonfinite(lib, prec, bad, where, N, fixed):
    dt = np.float64 if prec == "fp64" else np.float32
    p = _problem(N, 300, 7, dt)
    E = np.random.default_rng(1).standard_normal((p.m, N))
    if where == "y":
        p.y[150] = bad
    elif where == "X":
        p.Xf[p.col[100], 3] = bad
    else:
        E[150, 3] = bad
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision=prec, variant="reduced", fixed_iters=fixed)
    X, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    an.analyze_with_E(X, y, torch.from_numpy(E).cuda())
    st = an.stats()
    assert st["status"] == "nonfinite", st
    it, rel, true = an.column_stats()
    hit = np.arange(N) == 3 if where == "E" else np.ones(N, bool)   # a column of M, or all of them
    assert np.all(it[hit] == 0) and np.all(np.isnan(rel[hit])) and np.all(np.isnan(true[hit]))
    assert np.all(np.isfinite(rel[~hit])) and st["columns_converged"] == (N if fixed else int(np.sum(~hit)))
    # the handle's next analysis starts afresh
    p = _problem(N, 300, 7, dt)
    an.analyze(torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda(), seed=1)
    assert an.stats()["status"] == "ok"
    an.close()
