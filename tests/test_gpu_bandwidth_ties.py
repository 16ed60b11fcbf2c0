"""The median rule on clouds whose distances take few values, in compact clouds
where the screen still resolves the bracket: the sample has to say that the
bracket holds too many keys (a pass that collected 2 / 3 of all pairs one by one
took five times the histograms), and nothing changes in the value: 1e-6 of the
FP64 oracle, as in test_gpu_bandwidth.py."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TRIANGLE = np.array([[0.0, 0.0], [1.0, 0.0], [0.5, 0.75 ** 0.5]], dtype=np.float32)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    c = vds.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("N,sites", [(2897, 3), (4096, 3), (9000, 12), (9000, 40)])
def test_value(orc, ctx, N, sites):
    pts = TRIANGLE if sites == 3 else np.random.default_rng(2).standard_normal((sites, 2)).astype(np.float32)
    q = pts[np.arange(N) % sites]
    h = ctx.vds_bandwidth(torch.from_numpy(np.ascontiguousarray(q)).cuda(), 0)
    assert abs(h / orc.median_bandwidth(q.astype(np.float64)) - 1) <= 1e-6


def test_time(ctx):
    """Not slower than twice the cloud that takes the histograms for another reason (an outlier)."""
    N = 65536
    ties = torch.from_numpy(TRIANGLE[np.arange(N) % 3]).cuda()
    far = torch.randn((N, 2), device="cuda", generator=torch.Generator(device="cuda").manual_seed(0))
    far[0] = 1e4
    best = {}
    for name, q in (("ties", ties), ("far", far)) * 3:
        t0 = time.perf_counter()
        ctx.vds_bandwidth(q, 0)
        best[name] = min(best.get(name, 1e9), time.perf_counter() - t0)
    assert best["ties"] <= 2.0 * best["far"], best
