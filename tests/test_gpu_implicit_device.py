"""Implicit steps with the minimiser on the device, where its rounds can go
wrong: steps that need more gradients than are enqueued per step (a large time
step), more steps than the host runs ahead (64), steps split over calls, the
small-cloud and the symmetric passes, FENE bonds, and iteration limits, against
the FP64 oracle's minimiser (1e-5, as for the other implicit steps)."""
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


@pytest.mark.parametrize("N,nb,s,h,dt,spring,steps", [(300, 1, 2, 0.4, 0.15, 0, 3), (500, 3, 3, 0.9, 0.1, 0, 3),
                                                      (400, 2, 3, 0.8, 0.05, 1, 4), (5000, 3, 3, 0.8, 0.05, 0, 2),
                                                      (7000, 1, 3, 0.5, 0.08, 1, 2)])
def test_steps_of_many_gradients_match_oracle(orc, vds, ctx, N, nb, s, h, dt, spring, steps):
    b = 50.0
    kap = inputs.shear_kappa(s, 1.0)
    q32 = inputs.equilibrium_cloud(N, nb, s, seed=N, fene_b=b if spring else None)
    kw = dict(h=h, dt=dt, kappa=kap, spring=spring, b=b, tol=1e-6, jfloor=1e-9)
    q_o, _, _ = orc.implicit_steps(q32.astype(np.float64), orc.params(nb, s, **kw), steps)
    q = torch.from_numpy(q32).cuda()
    its = ctx.vds_step(q, vds.params(nb, s, scheme=1, **kw), steps, want_iters=True)
    assert len(its) == steps and all(k >= 3 for k in its), its
    assert np.max(np.abs(q.cpu().numpy() - q_o)) <= 1e-5 * np.max(np.abs(q_o))


def test_many_steps_and_steps_over_calls(vds, ctx):
    N, nb, s = 256, 1, 2
    kw = dict(h=0.35, dt=0.01, kappa=inputs.shear_kappa(s, 0.5), scheme=1, tol=1e-6, jfloor=1e-9)
    q0 = torch.from_numpy(inputs.equilibrium_cloud(N, nb, s, seed=4)).cuda()
    p = vds.params(nb, s, **kw)
    a, b = q0.clone(), q0.clone()
    its = ctx.vds_step(a, p, 150, want_iters=True)
    assert len(its) == 150 and all(1 <= k <= 50 for k in its)
    for _ in range(3):
        ctx.vds_step(b, p, 50)
    assert torch.isfinite(a).all()
    # a call's first step starts from q*, a later one from the last correction: same minimiser
    assert float((a - b).abs().max()) <= 1e-4 * float(a.abs().max())


def test_iteration_limit_updates_q_and_stops(vds, ctx):
    N, nb, s = 400, 3, 3
    q = torch.from_numpy(inputs.equilibrium_cloud(N, nb, s, seed=9)).cuda()
    q0 = q.clone()
    p = vds.params(nb, s, h=0.9, dt=0.1, scheme=1, tol=1e-12, max_iter=2, jfloor=1e-9)
    with pytest.raises(vds.VdsError) as e:
        ctx.vds_step(q, p, 5)
    assert e.value.code == vds.VDS_ENOCONV
    assert not torch.equal(q, q0) and torch.isfinite(q).all()
    ctx.vds_step(q, vds.params(nb, s, h=0.9, dt=0.01, scheme=1, tol=1e-6, jfloor=1e-9), 2)
