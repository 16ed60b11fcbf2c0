"""Batched ensembles over unordered pairs where their units can go wrong: one
particle either side of the size that takes them (2048), of an i-tile (640 to
1536 particles by dimension) and of a run of j-chunks (1024 particles), next to
small ensembles over ordered pairs: against the FP64 oracle (1e-5), the same
bits alone as in a batch and in every shape of the ordered items, explicit and
implicit steps."""
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


CASES = [(2, 3, [2047, 2048, 300, 2049, 3073, 1]), (3, 3, [2303, 2305, 40, 3100]), (1, 2, [2048, 3072, 3073, 9]),
         (1, 3, [2050, 4097]), (2, 2, [2100, 50]), (4, 2, [2304, 2049]), (4, 3, [2561, 77, 2048])]


def _setup(vds, ctx, nb, s, sizes, **kw):
    rng = np.random.default_rng(5)
    qs = [inputs.equilibrium_cloud(n, nb, s, seed=200 + e) for e, n in enumerate(sizes)]
    h = rng.uniform(0.5, 0.9, len(sizes)) * np.sqrt(nb)
    kap = np.stack([inputs.shear_kappa(s, r) for r in 10.0 ** rng.uniform(-1, 1, len(sizes))])
    return qs, h, kap, vds.Batch(ctx, sizes, nb * s, vds.params(nb, s, **kw), h, kap)


@pytest.mark.parametrize("nb,s,sizes", CASES)
def test_evaluation_matches_oracle(orc, vds, ctx, nb, s, sizes):
    qs, h, kap, b = _setup(vds, ctx, nb, s, sizes)
    q_all = torch.from_numpy(np.concatenate(qs)).cuda()
    g, rho = torch.full_like(q_all, float("nan")), torch.full((q_all.shape[0],), float("nan"), device="cuda")
    E = b.energy_grad(q_all, g=g, rho=rho)
    off = np.concatenate([[0], np.cumsum(sizes)])
    for e, q in enumerate(qs):
        sl = slice(off[e], off[e + 1])
        E_o, g_o, rho_o = orc.energy_grad(q.astype(np.float64), orc.params(nb, s, h=h[e]))
        assert np.max(np.abs(rho[sl].cpu().numpy() - rho_o) / rho_o) <= 1e-5
        assert abs(E[e] - E_o) <= 1e-5 * (1 + abs(E_o))
        assert np.max(np.abs(g[sl].cpu().numpy() - g_o)) <= 1e-5 * max(np.max(np.abs(g_o)), 1e-30)
        b1 = vds.Batch(ctx, [sizes[e]], nb * s, vds.params(nb, s), h[e:e + 1], kap[e:e + 1])
        g1 = torch.empty((sizes[e], nb * s), device="cuda")
        b1.energy_grad(q_all[sl].contiguous(), g=g1)
        assert torch.equal(g1, g[sl])
    for cfg in range(vds.BATCH_CONFIGS):
        b.set_config(cfg)
        g2 = torch.empty_like(g)
        b.energy_grad(q_all, g=g2)
        assert torch.equal(g2, g)


@pytest.mark.parametrize("scheme,dt", [(0, 0.005), (1, 0.01)])
def test_steps_match_oracle(orc, vds, ctx, scheme, dt):
    nb, s, sizes = 2, 3, [2049, 500, 3073]
    qs, h, kap, b = _setup(vds, ctx, nb, s, sizes, dt=dt, scheme=scheme, tol=1e-6, jfloor=1e-9)
    q_all = torch.from_numpy(np.concatenate(qs)).cuda()
    b.step(q_all, 2)
    got, off = q_all.cpu().numpy(), 0
    for e, q in enumerate(qs):
        po = orc.params(nb, s, h=h[e], dt=dt, kappa=kap[e], tol=1e-10)
        q64 = q.astype(np.float64)
        q_o = orc.explicit_steps(q64, po, 2) if scheme == 0 else orc.implicit_steps(q64, po, 2)[0]
        assert np.max(np.abs(got[off:off + len(q)] - q_o)) <= 1e-5 * np.max(np.abs(q_o))
        off += len(q)
