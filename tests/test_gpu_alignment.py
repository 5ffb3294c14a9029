"""X_f and X_a at addresses that are aligned for their elements only (a view into a larger tensor): every route
gives what it gives at 16-byte boundaries, bit for bit (the same arithmetic behind narrower accesses)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROUTES = [("fp32", dict(precondition=1)), ("fp16", dict(precondition=1)), ("fp32", dict()), ("fp32", dict(grid_blocks=3)),
          ("fp16", dict(lowprec_terms=1)), ("fp32", dict(variant="reduced")), ("fp32", dict(variant="senkf")),
          ("fp64", dict()), ("fp64", dict(variant="reduced")), ("fp64", dict(precondition=1))]


def _problem(N, m, seed, dt):
    side = max(4, int(np.ceil(np.sqrt(1.5 * m))))
    return synth.grf_problem(side, max(1.0, side / 10), N, m, 0.5, 1.5, seed, dtype=dt)


def _at(x, off):
    """A copy of x that begins `off` elements behind a 256-byte boundary."""
    buf = torch.empty(x.numel() + off, dtype=x.dtype, device="cuda")
    v = buf[off:].view(x.shape)
    v.copy_(x)
    return v


@pytest.mark.parametrize("prec,cfg", ROUTES)
@pytest.mark.parametrize("N", [20, 64, 100, 33])
def test_single_analyses(lib, prec, cfg, N):
    p = _problem(N, 300, N, np.float64 if prec == "fp64" else np.float32)
    X, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision=prec, max_iter=60, **cfg)
    ref = an.analyze(X, y, seed=4).clone()
    for a, b in ((1, 0), (0, 1), (1, 3), (2, 2)):
        assert torch.equal(an.analyze(_at(X, a), y, seed=4, out=_at(X, b)), ref), (a, b)
    Xi = _at(X, 1)   # in place
    assert torch.equal(an.analyze(Xi, y, seed=4, out=Xi), ref)
    # page-locked host arrays: read by the innovations and written by the update themselves
    hX, hXa = (torch.empty(p.n * N + 1, dtype=X.dtype, pin_memory=True)[1:].view(p.n, N) for _ in range(2))
    hX.copy_(torch.from_numpy(p.Xf))
    assert torch.equal(an.analyze_host(hX, torch.from_numpy(p.y), seed=4, out=hXa).cuda(), ref)
    an.close()


def test_batches(lib):
    probs = [_problem(N, m, N, np.float32) for N, m in ((16, 500), (64, 900), (100, 300), (33, 200))]
    X, y = [torch.from_numpy(p.Xf).cuda() for p in probs], [torch.from_numpy(p.y).cuda() for p in probs]
    an = lib.BatchAnalysis([dict(n=p.n, m=p.m, N=p.N, rowptr=p.rowptr, col=p.col, w=p.w, r=p.r) for p in probs])
    ref = [o.clone() for o in an.analyze(X, y, [1, 2, 3, 4])]
    out = an.analyze([_at(x, 1) for x in X], y, [1, 2, 3, 4], out=[_at(x, 2) for x in X])
    assert all(torch.equal(a, b) for a, b in zip(out, ref))
    an.close()
