"""The symmetric pair passes (one kernel value per unordered pair) against the
FP64 oracle at the sizes where their tiling can go wrong: the smallest cloud
that takes them, one particle either side of an i-tile (128 threads x 4, 6 or 8
particles), of a j-chunk (32 or 64 records) and of the record padding (256),
and the switch to the larger tiles, for every supported dimension.

Tolerance 1e-5 relative, the bar of the full-order path: FP32 sums of 256 or
fewer terms compensated beyond, and ex2.approx's 2^-22.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2603_12550_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def vds():
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds as v
    return v


@pytest.fixture(scope="module")
def ctx(vds):
    c = vds.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


CASES = [(1, 2, 2048), (1, 2, 3073), (1, 3, 2049), (1, 3, 33000), (2, 2, 2111), (2, 3, 2304), (2, 3, 4609),
         (3, 2, 2305), (4, 2, 2081), (3, 3, 2047), (3, 3, 2048), (3, 3, 2560), (3, 3, 2561), (3, 3, 4095),
         (3, 3, 32767), (3, 3, 32769), (5, 2, 2049), (6, 2, 2177), (4, 3, 2559), (7, 2, 2050), (5, 3, 2051),
         (8, 2, 3001)]


@pytest.mark.parametrize("nb,s,N", CASES)
def test_symmetric_passes_match_oracle(orc, vds, ctx, nb, s, N):
    h = 0.6 * np.sqrt(nb)
    q32 = inputs.equilibrium_cloud(N, nb, s, seed=N + nb)
    E_o, g_o, rho_o = orc.energy_grad(q32.astype(np.float64), orc.params(nb, s, h=h))
    q = torch.from_numpy(q32).cuda()
    g, rho = torch.full_like(q, float("nan")), torch.full((N,), float("nan"), device="cuda")
    E = ctx.vds_energy_grad(q, vds.params(nb, s, h=h), g=g, rho=rho)
    assert np.max(np.abs(rho.cpu().numpy() - rho_o) / rho_o) <= 1e-5
    assert abs(E - E_o) <= 1e-5 * (1 + abs(E_o))
    assert np.max(np.abs(g.cpu().numpy() - g_o)) <= 1e-5 * np.max(np.abs(g_o))
    # the schedule does not enter the sums
    g2 = torch.empty_like(q)
    ctx.vds_energy_grad(q, vds.params(nb, s, h=h), g=g2)
    assert torch.equal(g, g2)
