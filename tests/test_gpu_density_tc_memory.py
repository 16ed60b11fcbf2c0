"""The tensor-core density where device memory is short: the row sums of a whole
cloud (N^2 / 128 bytes) do not fit, and it goes in more launches of fewer column
tiles, with the pass's documented accuracy against the FP64 oracle (1e-4, 1e-5
for the median particle)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,nb,left_mb", [(262144, 3, 300), (131072, 2, 160)])
def test_short_memory(orc, N, nb, left_mb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    q = torch.randn((N, 3 * nb), device="cuda", generator=torch.Generator(device="cuda").manual_seed(N))
    p = vds.params(nb, 3, h=0.7)
    rho = torch.full((N,), float("nan"), device="cuda")
    ctx = vds.Context(0)
    ctx.vds_density_tc(q[:1000], p, rho)  # loads the kernels
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (left_mb << 20), dtype=torch.uint8, device="cuda")
    left = torch.cuda.mem_get_info()[0]
    try:
        ctx.vds_density_tc(q, p, rho)
        torch.cuda.synchronize()
    finally:
        del hog
        torch.cuda.empty_cache()
    ctx.close()
    assert left < (left_mb + 64) << 20
    rows = np.random.default_rng(4).choice(N, 96, replace=False)
    rows[:3] = [0, N - 1, N // 2]
    want = orc.density_rows(q.cpu().numpy().astype(np.float64), 0.7, rows)
    got = rho.cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    rel = np.abs(got[rows] - want) / want
    assert rel.max() <= 1e-4 and np.median(rel) <= 1e-5, (rel.max(), np.median(rel))
