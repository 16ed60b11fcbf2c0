"""The pair passes of a cloud against itself -- small clouds in one launch with
the epilogue, larger ones over unordered pairs -- against the FP64 oracle at the
sizes where their tiling can go wrong: one particle, the switches between the
forms (1216, 2432, 4864 or 6144 particles) and between tile sizes (32768,
49152), one particle either side of an i-tile and of a j-chunk, for every
supported dimension.

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


CASES = [(1, 2, 1), (3, 3, 2), (3, 3, 7), (2, 3, 9), (4, 3, 33),
         (3, 3, 1216), (3, 3, 1217), (8, 2, 1216), (8, 2, 1217), (1, 3, 2432), (3, 3, 2433), (2, 3, 2433),
         (5, 2, 2433), (6, 2, 2177), (7, 2, 2050), (5, 3, 2051), (1, 2, 6144), (1, 2, 6145), (1, 3, 6145),
         (2, 2, 6147), (2, 3, 6144), (2, 3, 6145), (3, 2, 7169), (4, 2, 4865), (3, 3, 4864), (3, 3, 4865),
         (3, 3, 5376), (3, 3, 5377), (3, 3, 5381), (5, 2, 4865), (6, 2, 5121), (4, 3, 5120), (7, 2, 4866),
         (5, 3, 4867), (8, 2, 5000), (3, 3, 32767), (3, 3, 32769), (1, 3, 33000), (3, 3, 49153), (2, 2, 50001)]


@pytest.mark.parametrize("nb,s,N", CASES)
def test_passes_match_oracle(orc, vds, ctx, nb, s, N):
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


@pytest.mark.parametrize("N,nb,s,steps", [(700, 3, 3, 5), (700, 3, 3, 6), (1300, 2, 3, 8), (3000, 1, 2, 7)])
def test_steps_replayed_in_pairs_equal_single_steps(vds, ctx, N, nb, s, steps):
    # small clouds alternate between two record arrays, and replays advance two
    # steps at a time: any number of steps gives what single calls give
    q0 = torch.from_numpy(inputs.equilibrium_cloud(N, nb, s, seed=3)).cuda()
    p = vds.params(nb, s, h=0.7, dt=0.002, kappa=inputs.shear_kappa(s, 1.0))
    a, b = q0.clone(), q0.clone()
    ctx.vds_step(a, p, steps)
    for _ in range(steps):
        ctx.vds_step(b, p, 1)
    assert torch.equal(a, b)
