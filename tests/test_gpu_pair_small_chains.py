"""Accuracy of the small-cloud passes where a lane's records are cut in two
chains (3073 particles and more).  With a wide kernel every value is near one
and the rounding of the sums is all that is left of the density's error: it has
to be no larger than that of the ordered passes (vds_energy_grad_noalloc), whose
chains of 64 records are Kahan-summed, against the FP64 oracle.  (Chains of 48
and less leave about sqrt(48 / 64) of it; one chain of N / 64 = 58 to 96 records
left more than all of it.)"""
import numpy as np
import pytest

from paper_2603_12550_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nb,s,N", [(1, 3, 6000), (2, 2, 6143), (2, 3, 6144), (3, 3, 4863), (4, 3, 4864), (8, 2, 4801)])
def test_errors_of_two_chains(orc, nb, s, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    ctx = vds.Context(0)
    h = 4.0 * np.sqrt(nb * s)
    p = vds.params(nb, s, h=h)
    err = np.zeros(2)
    for seed in range(4):
        q32 = inputs.equilibrium_cloud(N, nb, s, seed=seed)
        rho_o = orc.density(q32.astype(np.float64), h)
        q = torch.from_numpy(q32).cuda()
        for k, call in enumerate((ctx.vds_energy_grad, vds.energy_grad_noalloc)):
            rho = torch.full((N,), float("nan"), device="cuda")
            call(q, p, rho=rho)
            err[k] += np.linalg.norm(rho.cpu().numpy() - rho_o) / np.linalg.norm(rho_o)
    assert err[0] <= err[1], err / 4
    ctx.close()
