"""The bracketed median selection at the sizes where it can go wrong: the last
cloud that writes all keys and the first that takes the bracket (2896 and 2897
particles), one particle either side of an i-tile (512 or 1024) and a j-chunk
(64), the smallest clouds, and clouds whose many equal distances overflow the
bracket (the histograms take over).  1e-6 relative, as in
test_gpu_bandwidth.py: an exact selection on FP32 squared distances."""
import numpy as np
import pytest

from paper_2603_12550_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


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


@pytest.mark.parametrize("N,nb,s", [(2, 3, 3), (5, 2, 2), (2896, 3, 3), (2897, 3, 3), (2897, 1, 2), (3072, 1, 3),
                                    (3073, 2, 3), (4095, 2, 2), (4097, 3, 3), (3585, 8, 2), (3000, 5, 2),
                                    (3001, 4, 3), (2999, 7, 2), (3137, 5, 3), (3136, 4, 2)])
def test_median_matches_oracle_at_the_edges(orc, ctx, N, nb, s):
    q32 = inputs.equilibrium_cloud(N, nb, s, seed=N + nb)
    q = torch.from_numpy(q32).cuda()
    h = ctx.vds_bandwidth(q, 0)
    h_o = orc.median_bandwidth(q32.astype(np.float64))
    assert abs(h / h_o - 1) <= 1e-6
    assert ctx.vds_bandwidth(q, 0) == h


@pytest.mark.parametrize("N,sites", [(3000, 3), (3000, 2), (6000, 40)])
def test_median_among_few_distinct_distances(orc, ctx, N, sites):
    # at two sites half the distances are zero and the median is the other one or zero
    q32 = inputs.equilibrium_cloud(sites, 3, 3, seed=7)[np.arange(N) % sites]
    if sites == 2:
        q32[:200] = q32[1]  # uneven, so that the median is the zero distance
        from paper_2603_12550_gb300 import vds
        with pytest.raises(vds.VdsError) as e:
            ctx.vds_bandwidth(torch.from_numpy(q32).cuda(), 0)
        assert e.value.code == vds.VDS_ENAN
        return
    h = ctx.vds_bandwidth(torch.from_numpy(q32).cuda(), 0)
    assert abs(h / orc.median_bandwidth(q32.astype(np.float64)) - 1) <= 1e-6
