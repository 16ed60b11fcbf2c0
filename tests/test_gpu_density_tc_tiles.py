"""The tensor-core density where its triangle of tiles can go wrong: one
particle either side of a row tile (128) and a column tile (256), clouds whose
tiles are fewer or just more than the SMs, and one large enough for several
launches (more than about 370000 particles), against the FP64 oracle: 1e-4
everywhere, 1e-5 for the median particle, the pass's documented accuracy."""
import numpy as np
import pytest

from paper_2603_12550_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def vds():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds as v
    return v


@pytest.fixture(scope="module")
def ctx(vds):
    c = vds.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("N,nb", [(2, 2), (127, 3), (128, 2), (256, 3), (385, 3), (511, 2), (513, 3), (2944, 3),
                                  (3073, 2), (4096, 3), (9999, 2)])
def test_tiles_match_oracle(orc, vds, ctx, N, nb):
    q = inputs.equilibrium_cloud(N, nb, 3, seed=N + nb)
    rho = torch.full((N,), float("nan"), device="cuda")
    qd = torch.from_numpy(q).cuda()
    ctx.vds_density_tc(qd, vds.params(nb, 3, h=0.8), rho)
    want = orc.density(q.astype(np.float64), 0.8)
    rel = np.abs(rho.cpu().numpy().astype(np.float64) - want) / want
    assert rel.max() <= 1e-4 and np.median(rel) <= 1e-5, (rel.max(), np.median(rel))
    again = torch.empty_like(rho)
    ctx.vds_density_tc(qd, vds.params(nb, 3, h=0.8), again)
    assert torch.equal(rho, again)


def test_several_launches(orc, vds, ctx):
    N = 400001
    q = inputs.equilibrium_cloud(N, 2, 3, seed=1)
    rho = torch.full((N,), float("nan"), device="cuda")
    ctx.vds_density_tc(torch.from_numpy(q).cuda(), vds.params(2, 3, h=0.7), rho)
    rows = np.random.default_rng(4).choice(N, 96, replace=False)
    rows[:4] = [0, N - 1, 262143, 375000]
    want = orc.density_rows(q.astype(np.float64), 0.7, rows)
    got = rho.cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    rel = np.abs(got[rows] - want) / want
    assert rel.max() <= 1e-4 and np.median(rel) <= 1e-5, (rel.max(), np.median(rel))
