"""The FP64 ensembles' update on the tensor cores (csrc/kernels_update64.cu) where its tiling can go wrong: N
around its 64-member blocks and 16-deep steps, n around the 80-row tile and several tiles per CTA, both
forms (X_f + A W, X_f V), rows of very different size. The analysis leaves W, so the update is
compared with the same W: a K-term FP64 dot product is off by at most about K 2^-53 of |a| |b|; bar 1e-14 of
|X_f| + |A| |W| per row."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("variant", ["cgd", "reduced"])
@pytest.mark.parametrize("N,n", [(2, 1), (16, 80), (17, 81), (63, 500), (64, 152 * 32 + 1), (65, 161), (100, 4000), (128, 152 * 33)])
def test_update(lib, N, n, variant):
    rng = np.random.default_rng(N + n)
    m = max(1, min(n, 50))
    X = rng.standard_normal((n, N)) * 10.0 ** rng.uniform(-6, 6, (n, 1)) + rng.standard_normal((n, 1))
    r = np.ones(m)
    col = np.sort(rng.choice(n, m, replace=False)).astype(np.int32)
    cfg = dict(precondition=1, tol=1e-10) if variant == "cgd" else dict(variant="reduced", tol=1e-10)
    an = lib.Analysis(n, m, N, np.arange(m + 1, dtype=np.int32), col, np.ones(m), r, precision="fp64", max_iter=50, **cfg)
    Xf, y = torch.from_numpy(X).cuda(), torch.from_numpy(rng.standard_normal(m)).cuda()
    Xa = an.analyze(Xf, y, seed=1, counter=2).cpu().numpy()
    W = (an.intermediates()[3] if variant == "cgd" else an.intermediates_reduced()[0]).cpu().numpy()
    A = X - X.mean(1, keepdims=True) if variant == "cgd" else X
    ref = A.astype(np.longdouble) @ W.astype(np.longdouble)
    if variant == "cgd":
        ref = X + ref
    scale = np.linalg.norm(X, axis=1) + np.linalg.norm(A, axis=1) * np.linalg.norm(W)
    assert np.max(np.linalg.norm((Xa - ref).astype(np.float64), axis=1) / scale) <= 1e-14
