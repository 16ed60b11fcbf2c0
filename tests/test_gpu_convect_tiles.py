"""The convection step in blocks of nodes (values per node a multiple of four,
aligned arrays) at the edges of blocks and value ranges, and arrays one float
off alignment, which take the other kernel: against the FP64 oracle's upwind
step, 1e-6 of the field's largest value as in test_gpu_convect.py, and the same
bits in both kernels."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("shape,M,bc", [((1, 1, 1), 4, 0), ((64, 1, 1), 128, 0), ((65, 1, 1), 4, 1), ((2, 1, 1), 260, 0),
                                        ((9, 5, 3), 132, 0), ((4, 4, 4), 124, 1), ((5, 8, 1), 1000, 0),
                                        ((1, 3, 17), 516, 1), ((8, 8, 8), 384, 0)])
def test_blocks_match_oracle(orc, vds, ctx, shape, M, bc):
    G = shape[0] * shape[1] * shape[2]
    rng = np.random.default_rng(M + G)
    Q = rng.standard_normal((G, M)).astype(np.float32)
    u = rng.uniform(-1.5, 1.5, (G, 3)).astype(np.float32)
    u[::3, 1] = 0.0
    dx, dt = (0.4, 0.3, 0.5), 0.06
    ud = torch.from_numpy(u).cuda()
    want = orc.convect_upwind(Q.astype(np.float64), u.astype(np.float64), shape, dx, dt, bc)
    outs = []
    for shift in (0, 1):  # floats off a 16-byte boundary
        q_in = torch.empty(G * M + 4, device="cuda")[shift:shift + G * M].view(G, M)
        q_in.copy_(torch.from_numpy(Q))
        q_out = torch.full((G * M + 4,), float("nan"), device="cuda")
        ctx.vds_convect(q_in, q_out[shift:shift + G * M], shape, ud, dx, dt, bc)
        assert torch.isnan(q_out[G * M + shift:]).all() and torch.isnan(q_out[:shift]).all()
        outs.append(q_out[shift:shift + G * M].view(G, M).clone())
        got = outs[-1].cpu().numpy().astype(np.float64)
        assert np.max(np.abs(got - want)) <= 1e-6 * np.max(np.abs(Q))
    assert torch.equal(outs[0], outs[1])
