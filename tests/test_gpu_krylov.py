"""The preconditioned solve in Krylov coordinates (csrc/krylov.cuh) at the sizes where its tiling
can go wrong: N around the column tiles (32, 64, 128) and odd, m around the 64-row tile and
the row blocks of several grids, one CTA for two column groups, variances spread over four
decades, and members of very different spread. Against the exact FP64 analysis; the bar is the
FP32 path's (1e-6 relative Frobenius error: X_a is stored in FP32) and the certificate the true
residual within tol."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed, r_decades=0.0, outlier=1.0):
    rng = np.random.default_rng(seed)
    n = max(2 * m, 8)
    side = int(np.ceil(np.sqrt(n)))
    p = synth.grf_problem(side, max(1.0, side / 12), N, m, 0.5, 1.5, seed, dtype=np.float32)
    p.r = p.r * 10.0 ** rng.uniform(-r_decades / 2, r_decades / 2, m)
    p.Xf[:, 0] *= np.float32(outlier)
    return p


def _check(lib, p, prec="fp32", tol=1e-8, bar=1e-6, **cfg):
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision=prec, precondition=1, tol=tol, **cfg)
    Xa = an.analyze(torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda(), seed=4, counter=9)
    st = an.stats()
    E = oracle.obs_perturbations(4, 9, p.r, p.N)
    ref = oracle.enkf_exact(p.Xf.astype(np.float64), p.rowptr, p.col, p.w, p.r, p.y, E)
    err = oracle.rel_frobenius(Xa.double().cpu().numpy(), ref)
    assert st["status"] == "ok" and 0 <= st["true_relres_max"] <= tol, st
    assert bar is None or err <= bar, (err, st)
    an.close()


@pytest.mark.parametrize("N", [2, 3, 31, 32, 33, 63, 64, 65, 96, 127, 128])
@pytest.mark.parametrize("m,G", [(1, 0), (63, 0), (64, 1), (65, 2), (450, 3), (700, 5)])
def test_tile_edges(lib, N, m, G):
    _check(lib, _problem(N, m, 1000 * N + m), grid_blocks=G)


@pytest.mark.parametrize("N", [20, 64, 100])
def test_spread_variances_and_members(lib, N):
    _check(lib, _problem(N, 900, 7 + N, r_decades=4.0))
    # one member 300 times the others (condition about 1e7): the solve has to reach its certificate;
    # X_a itself is limited by the FP32 perturbations and update (1.0e-5 from the recurrences on
    # m-vectors as well)
    _check(lib, _problem(N, 900, 9 + N, outlier=300.0), bar=None)


def test_tight_tolerance_takes_another_cycle(lib):
    _check(lib, _problem(64, 4000, 3), tol=1e-12)


def test_fixed_step_counts_keep_the_recurrences_on_m_vectors(lib):
    # a step count fixed by the caller is about the m-vectors: more steps than N are taken
    p = _problem(32, 500, 21)
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp32", precondition=1, fixed_iters=70)
    Xa = an.analyze(torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda(), seed=4, counter=9)
    E = oracle.obs_perturbations(4, 9, p.r, p.N)
    ref = oracle.enkf_exact(p.Xf.astype(np.float64), p.rowptr, p.col, p.w, p.r, p.y, E)
    assert an.stats()["status"] == "ok"
    assert oracle.rel_frobenius(Xa.double().cpu().numpy(), ref) <= 1e-4
    it, _, _ = an.column_stats()
    assert np.all(it <= 70) and it.max() > 32
