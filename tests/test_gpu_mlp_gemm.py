"""The dense layers' matrix product (csrc/kernels_mlp.cu, mlp_gemm_kernel) where its tiling can go wrong: one
row, one input, sizes around the 64 x 64 tile and the 32-deep step, odd leading dimensions (no 16-byte
loads) and depths that split over 1 to 8 CTAs. Against a 64-bit evaluation; a K-term FP32 dot product of
unit-variance terms is off by at most about sqrt(K) 2^-24 of its norm, three layers deep: bar 1e-5."""
import numpy as np
import pytest

from oracle import warmstart as ows
from synth.mlp_init import init_params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# (in, hidden, layers, out, batch)
@pytest.mark.parametrize("dims", [(1, 1, 1, 1, 1), (3, 5, 2, 2, 7), (63, 64, 1, 65, 64), (64, 63, 2, 64, 65), (33, 31, 3, 129, 130),
                                  (1088, 512, 1, 64, 2), (1500, 20, 1, 3, 256), (130, 128, 2, 33, 1000)])
def test_forward_and_gradient(lib, dims):
    shape, B = dims[:4], dims[4]
    p = init_params(*shape, seed=7, out_scale=1.0)
    rng = np.random.default_rng(8)
    X = rng.standard_normal((B, shape[0])).astype(np.float32)
    T = rng.standard_normal((B, shape[3])).astype(np.float32)
    tp, tX = torch.from_numpy(p).cuda(), torch.from_numpy(X).cuda()
    Y = lib.mlp_forward(shape, tp, tX).cpu().numpy()
    ref = ows.forward(p.astype(np.float64), shape, X.astype(np.float64))
    assert np.linalg.norm(Y - ref) <= 1e-5 * np.linalg.norm(ref)
    loss, grad = lib.mlp_loss_grad(shape, tp, tX, torch.from_numpy(T).cuda())
    L, g = ows.loss_grad(p.astype(np.float64), shape, X.astype(np.float64), T.astype(np.float64))
    assert abs(loss.item() - L) <= 1e-5 * L
    a, off = grad.cpu().numpy()[:g.size], 0
    for fi, fo in ows.layer_dims(*shape):
        for cnt in (fi * fo, fo):
            assert np.linalg.norm(a[off:off + cnt] - g[off:off + cnt]) <= 1e-5 * np.linalg.norm(g[off:off + cnt]), (fi, fo, cnt)
            off += cnt
