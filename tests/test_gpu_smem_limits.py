"""Limits on dynamic shared memory belong to a kernel, not to a handle: a handle created for fewer members
must not lower the limit that an older one's launches need."""
import numpy as np
import pytest

import oracle
import synth
from synth.mlp_init import init_params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _warm(lib, N, precondition):
    p = synth.grf_problem(40, 4.0, N, 400, 0.5, 1.5, 3, dtype=np.float32)
    K = 32
    shape = (K + N, 32, 1, N)
    params = torch.from_numpy(init_params(*shape, seed=1, out_scale=0.3)).cuda()
    an = lib.Analysis(p.n, p.m, p.N, p.rowptr, p.col, p.w, p.r, precision="fp32", precondition=precondition, warm_start=1)
    an.set_warm_model(shape, params)
    return p, an, params


@pytest.mark.parametrize("precondition", [0, 1])
def test_a_handle_of_fewer_members_leaves_an_older_one_working(lib, precondition):
    p, an, params = _warm(lib, 128, precondition)
    _, other, params2 = _warm(lib, 104, precondition)
    Xa = an.analyze(torch.from_numpy(p.Xf).cuda(), torch.from_numpy(p.y).cuda(), seed=5, counter=1)
    assert an.stats()["status"] == "ok"
    E = oracle.obs_perturbations(5, 1, p.r, p.N)
    ref = oracle.enkf_exact(p.Xf.astype(np.float64), p.rowptr, p.col, p.w, p.r, p.y, E)
    assert oracle.rel_frobenius(Xa.double().cpu().numpy(), ref) <= 1e-6
    other.close()
    an.close()
