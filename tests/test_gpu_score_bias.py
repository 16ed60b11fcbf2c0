"""Bias gradients of columns that hold infinities: what a sum in the order of
the rows gives, infinity of the term's sign, NaN where both signs meet, and the
other columns' bits as without them."""
import numpy as np
import pytest

from paper_2603_12550_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M", [128, 512, 8192])
def test_infinite_terms(M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    ctx = vds.Context(0)
    D = 9
    layers = inputs.mlp_init((D, 256, 256, 256, D), seed=3)
    x = torch.from_numpy(np.random.default_rng(M).standard_normal((M, D)).astype(np.float32)).cuda()
    t = torch.zeros((M, D), device="cuda")
    _, ref = vds.Score(ctx, D, layers).fit_step(x, t, 0.0, want_grads=True)
    t[M // 2, 2] = -float("inf")  # residual s - t
    t[M - 1, 4] = float("inf")
    t[0, 8], t[M - 1, 8] = float("inf"), -float("inf")
    _, got = vds.Score(ctx, D, layers).fit_step(x, t, 0.0, want_grads=True)
    b, r = got[-1][1], ref[-1][1]
    assert b[2] == np.inf and b[4] == -np.inf
    assert np.isnan(b[8])
    rest = [0, 1, 3, 5, 6, 7]
    assert np.isfinite(r).all() and (b[rest] == r[rest]).all()
    ctx.close()
