"""Handles bound to a stream that is not ordered with the legacy default stream: everything their creation
uploads is there when the handle's kernels read it. R of the preconditioned solves (and, in
double-float, 1/R and its root, formed at creation), of the batch and of the other forms, at sizes whose uploads
do not fit one staging buffer; results are bitwise those of a handle on the default stream."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FORMS = [("fp32", dict(precondition=1)), ("fp16", dict(precondition=1)), ("fp32", dict()), ("fp16", dict(lowprec_terms=1)),
         ("fp32", dict(variant="reduced")), ("fp64", dict(precondition=1)), ("fp64", dict(variant="senkf"))]


def _problem(side, N, seed, dt):
    return synth.grf_problem(side, side / 16, N, side * side // 2, 0.25, 2.0, seed, dtype=dt)


@pytest.mark.parametrize("prec,cfg", FORMS)
def test_single_handles(lib, prec, cfg):
    dt = np.float64 if prec == "fp64" else np.float32
    p = _problem(400, 8, 5, dt)
    X, y = torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda()
    torch.cuda.synchronize()
    out = []
    for stream in [torch.cuda.current_stream()] + [torch.cuda.Stream() for _ in range(3)]:
        an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, stream=stream, precision=prec, max_iter=50, **cfg)
        with torch.cuda.stream(stream):
            out.append(an.analyze(X, y, seed=2).clone())
        an.close()
        torch.cuda.synchronize()
    assert all(torch.equal(out[0], o) for o in out[1:])


def test_batches(lib):
    probs = [_problem(s, N, s, np.float32) for s, N in ((300, 8), (64, 40), (400, 16))]
    X, y = [torch.from_numpy(p.Xf).cuda() for p in probs], [torch.from_numpy(p.y).cuda() for p in probs]
    torch.cuda.synchronize()
    out = []
    for stream in [torch.cuda.current_stream()] + [torch.cuda.Stream() for _ in range(3)]:
        an = lib.BatchAnalysis([dict(n=p.n, m=p.m, N=p.N, rowptr=p.rowptr, col=p.col, w=p.w, r=p.r) for p in probs], stream=stream)
        with torch.cuda.stream(stream):
            out.append([o.clone() for o in an.analyze(X, y, [1, 2, 3])])
        an.close()
        torch.cuda.synchronize()
    for o in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], o))
