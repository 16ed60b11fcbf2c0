"""Implicit steps with phase timing on: the gradient count is the number of
evaluations that the steps report, every gradient follows at least one density,
and the results are the bits of the untimed call."""
import pytest

from paper_2603_12550_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,nb,s,h,dt,steps", [(512, 1, 2, 0.3, 0.01, 5), (300, 1, 2, 0.4, 0.15, 3),
                                               (7000, 2, 3, 0.7, 0.02, 2), (256, 3, 3, 0.9, 0.01, 70)])
def test_counts_are_evaluations(N, nb, s, h, dt, steps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    ctx = vds.Context(0)
    p = vds.params(nb, s, h=h, dt=dt, kappa=inputs.shear_kappa(s, 1.0), scheme=1, tol=1e-6, jfloor=1e-9)
    a = torch.from_numpy(inputs.equilibrium_cloud(N, nb, s, seed=N)).cuda()
    b = a.clone()
    want = ctx.vds_step(a, p, steps, want_iters=True)
    ctx.vds_timing(True)
    its = ctx.vds_step(b, p, steps, want_iters=True)
    _, n, _ = ctx.vds_timing_read()
    ctx.vds_timing(False)
    assert its == want and torch.equal(a, b)
    assert n[1] == sum(its) and n[0] >= sum(its), (n, its)
    ctx.close()
