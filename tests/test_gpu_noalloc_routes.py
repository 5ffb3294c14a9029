"""FP32 with CG preconditioned by R through a handle (Krylov coordinates) and through the allocation-free entry point
(recurrences on m-vectors, or a cluster per column): different solves of the same system, both certified by
their true residual. Bar: the FP32 path's 1e-6 against the exact analysis for each."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,m,grid", [(2, 40, 0), (20, 300, 0), (33, 1500, 0), (64, 1024, 0), (64, 1024, 7), (128, 700, 0)])
def test_preconditioned_fp32(lib, N, m, grid):
    side = max(4, int(np.ceil(np.sqrt(1.5 * m))))
    p = synth.grf_problem(side, max(1.0, side / 10), N, m, 0.25, 1.5, 7 * N + m, dtype=np.float32)
    X, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp32", precondition=1, grid_blocks=grid)
    Xa = an.analyze(X, y, seed=6, counter=2).double().cpu().numpy()
    st = an.stats()
    cfg = lib.default_config(p.n, p.m, p.N, precision="fp32", precondition=1, grid_blocks=grid)
    dev = [torch.from_numpy(a).cuda() for a in (p.rowptr, p.col, p.w, p.r)]
    X2, st2 = lib.analyze_noalloc(cfg, *dev, X, y, seed=6, counter=2)
    exact = oracle.enkf_exact(p.Xf.astype(np.float64), p.rowptr, p.col, p.w, p.r, p.y, oracle.obs_perturbations(6, 2, p.r, N))
    for s, x in ((st, Xa), (st2, X2.double().cpu().numpy())):
        assert s["status"] == "ok" and 0 <= s["true_relres_max"] <= 1e-8, s
        assert oracle.rel_frobenius(x, exact) <= 1e-6
    an.close()
