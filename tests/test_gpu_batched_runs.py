"""Batched ensembles either side of the sizes where the length of a unit changes
(8 chunks of 32 particles up to 4064 particles, a sixteenth of the ensemble from
there, 32 chunks from 16385): against the FP64 oracle (1e-5, as for the other
batched passes), and the same bits alone as next to others."""
import numpy as np
import pytest

from paper_2603_12550_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nb,s,sizes", [(1, 3, [4064, 4096, 4321]), (3, 3, [4095, 4097]), (2, 3, [8191, 2048]),
                                        (1, 2, [16384, 16417])])
def test_lengths_of_units(orc, nb, s, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    ctx = vds.Context(0)
    qs = [inputs.equilibrium_cloud(n, nb, s, seed=n) for n in sizes]
    h = np.linspace(0.5, 0.7, len(sizes)) * np.sqrt(nb)
    kap = np.zeros((len(sizes), s, s))
    q_all = torch.from_numpy(np.concatenate(qs)).cuda()
    g, rho = torch.full_like(q_all, float("nan")), torch.full((q_all.shape[0],), float("nan"), device="cuda")
    vds.Batch(ctx, sizes, nb * s, vds.params(nb, s), h, kap).energy_grad(q_all, g=g, rho=rho)
    off = np.concatenate([[0], np.cumsum(sizes)])
    for e, q in enumerate(qs):
        sl = slice(off[e], off[e + 1])
        _, g_o, rho_o = orc.energy_grad(q.astype(np.float64), orc.params(nb, s, h=h[e]))
        assert np.max(np.abs(rho[sl].cpu().numpy() - rho_o) / rho_o) <= 1e-5
        assert np.max(np.abs(g[sl].cpu().numpy() - g_o)) <= 1e-5 * np.max(np.abs(g_o))
        g1 = torch.empty((sizes[e], nb * s), device="cuda")
        vds.Batch(ctx, [sizes[e]], nb * s, vds.params(nb, s), h[e:e + 1], kap[e:e + 1]).energy_grad(
            q_all[sl].contiguous(), g=g1)
        assert torch.equal(g1, g[sl])
    ctx.close()
