"""The FP64 ensembles' Gram pass of the Reduced and sEnKF variants on the tensor cores
(csrc/kernels_reduced.cu, gram64_kernel) where its tiling can go wrong: N around its 64-column blocks,
m around the 16-row steps and the 80-row tile, and several tiles per CTA; members, rows and weights of very
different size. Bars: those of the existing FP64 tests of these variants (1e-12 for G, 1e-10 for X_a)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed):
    side = max(4, int(np.ceil(np.sqrt(1.5 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=np.float64)


def _check(lib, p, X, E, tol_g=1e-12, solve=True):
    Xf, y = torch.from_numpy(X).cuda(), torch.from_numpy(p.y).cuda()
    e = None if E is None else torch.from_numpy(E).cuda()
    _, _, _, _, HA = oracle.ensemble_stats(X, p.rowptr, p.col, p.w)
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp64", variant="reduced", tol=1e-12)
    Xa = an.analyze_with_E(Xf, y, e)
    _, G = an.intermediates_reduced()
    ref = np.eye(p.N) + HA.T @ (HA / p.r[:, None]) / (p.N - 1)
    assert np.linalg.norm(G.cpu().numpy() - ref) <= tol_g * np.linalg.norm(ref)
    if solve:
        exact = oracle.enkf_exact(X, p.rowptr, p.col, p.w, p.r, p.y, E)
        assert oracle.rel_frobenius(Xa.cpu().numpy(), exact) <= 1e-10
    an.close()
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp64", variant="senkf")
    Xa = an.analyze_with_E(Xf, y, e)
    ref = oracle.senkf_alg3(X, p.rowptr, p.col, p.w, p.r, p.y, E)
    assert oracle.rel_frobenius(Xa.cpu().numpy(), ref) <= 1e-10
    an.close()


@pytest.mark.parametrize("N", [2, 33, 63, 64, 65, 127, 128])
@pytest.mark.parametrize("m", [1, 17, 81, 700])
def test_reduced_and_senkf(lib, N, m):
    p = _problem(N, m, 100 * N + m)
    E = np.random.default_rng(N).standard_normal((m, N)) * np.sqrt(p.r)[:, None]
    for e in (E, None):
        _check(lib, p, p.Xf, e)


def test_several_tiles_per_cta(lib):
    p = _problem(70, 152 * 200 + 13, 3)   # 201 rows per CTA: three tiles
    _check(lib, p, p.Xf, None)


def test_members_rows_and_weights_of_different_size(lib):
    p = _problem(40, 500, 4)
    rng = np.random.default_rng(5)
    p.r[:] = 10.0 ** rng.uniform(-3, 3, p.m)
    X = p.Xf * 10.0 ** rng.uniform(-2, 2, p.N)[None, :]
    # (G's condition is 2.6e6: CG stopped at 1e-12, the oracle's too, leaves 5e-8 of X_a, so G and the sEnKF's X_a only)
    _check(lib, p, X, None, 1e-11, solve=False)


def test_infinities_reach_every_member(lib):
    p = _problem(20, 300, 5)
    X = p.Xf.copy()
    X[p.col[3], 4] = np.inf   # an observed value: the row's mean, then every entry of W
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp64", variant="senkf")
    Xa = an.analyze(torch.from_numpy(X).cuda(), torch.from_numpy(p.y).cuda(), seed=1, counter=0)
    assert torch.isnan(Xa).all()
