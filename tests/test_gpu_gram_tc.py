"""The FP32 ensembles' Gram pass of the Reduced and sEnKF variants on the tensor cores
(csrc/kernels_reduced.cu, gram_tc_kernel) where its tiling can go wrong: N around the column tiles,
m around the 64-row tile and past the 512-row chunk of a CTA, explicit perturbations and E = 0.
G, M's solution and W against the oracle on the FP32-rounded ensemble; the bars are those of the
existing tests of these variants (1e-11 for G, 1e-6 for X_a)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _problem(N, m, seed):
    side = max(4, int(np.ceil(np.sqrt(1.5 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=np.float32)


@pytest.mark.parametrize("N", [2, 31, 32, 33, 64, 65, 100, 128])
@pytest.mark.parametrize("m", [1, 63, 65, 640])
def test_reduced_and_senkf(lib, N, m):
    p = _problem(N, m, 100 * N + m)
    X = p.Xf.astype(np.float64)
    E = np.random.default_rng(N).standard_normal((m, N)) * np.sqrt(p.r)[:, None]
    Xf, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    _, _, _, _, HA = oracle.ensemble_stats(X, p.rowptr, p.col, p.w)
    for e in (E, None):
        an = lib.Analysis(p.n, m, N, p.rowptr, p.col, p.w, p.r, precision="fp32", variant="reduced", tol=1e-10)
        Xa = an.analyze_with_E(Xf, y, None if e is None else torch.from_numpy(e).cuda())
        assert an.stats()["status"] == "ok"
        _, G = an.intermediates_reduced()
        ref = np.eye(N) + HA.T @ (HA / p.r[:, None]) / (N - 1)
        assert np.linalg.norm(G.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
        exact = oracle.enkf_exact(X, p.rowptr, p.col, p.w, p.r, p.y, e)
        assert oracle.rel_frobenius(Xa.double().cpu().numpy(), exact) <= 1e-6
        an.close()
        an = lib.Analysis(p.n, m, N, p.rowptr, p.col, p.w, p.r, precision="fp32", variant="senkf")
        Xa = an.analyze_with_E(Xf, y, None if e is None else torch.from_numpy(e).cuda())
        ref = oracle.senkf_alg3(X, p.rowptr, p.col, p.w, p.r, p.y, e)
        assert oracle.rel_frobenius(Xa.double().cpu().numpy(), ref) <= 1e-6
        an.close()


def test_several_chunks_per_cta(lib):
    # 152 CTAs of more than 512 rows each: the products of a CTA's second chunk are added to the first's
    N, m = 24, 152 * 512 + 40000
    p = _problem(N, m, 3)
    Xf, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    an = lib.Analysis(p.n, m, N, p.rowptr, p.col, p.w, p.r, precision="fp32", variant="reduced", tol=1e-10)
    Xa = an.analyze(Xf, y, seed=2, counter=1)
    E = oracle.obs_perturbations(2, 1, p.r, N)
    exact = oracle.enkf_exact(p.Xf.astype(np.float64), p.rowptr, p.col, p.w, p.r, p.y, E)
    assert an.stats()["status"] == "ok"
    assert oracle.rel_frobenius(Xa.double().cpu().numpy(), exact) <= 1e-6
