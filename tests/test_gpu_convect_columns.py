"""The convection step where a CTA takes several groups of columns (few nodes,
many values per node) and where the blocks of an axis are not a power of two:
the same bits as the kernel for unaligned arrays, which takes a node per CTA,
and 1e-6 of the field's largest value against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,M,bc", [((1, 1, 1), 311300, 0), ((1, 1, 1), 1245188, 1), ((2, 1, 1), 622596, 0),
                                        ((3, 1, 1), 400004, 1), ((7, 1, 1), 200068, 0), ((12, 1, 1), 160004, 1),
                                        ((5, 5, 1), 100004, 0), ((9, 9, 1), 1540, 1), ((3, 3, 3), 40004, 0),
                                        ((11, 1, 9), 772, 0)])
def test_columns_and_blocks(orc, shape, M, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    ctx = vds.Context(0)
    G = shape[0] * shape[1] * shape[2]
    rng = np.random.default_rng(M)
    Q = rng.standard_normal((G, M)).astype(np.float32)
    u = rng.uniform(-1.5, 1.5, (G, 3)).astype(np.float32)
    dx, dt = (0.4, 0.3, 0.5), 0.06
    ud = torch.from_numpy(u).cuda()
    outs = []
    for shift in (0, 1):  # floats off a 16-byte boundary
        q_in = torch.empty(G * M + 4, device="cuda")[shift:shift + G * M].view(G, M)
        q_in.copy_(torch.from_numpy(Q))
        q_out = torch.full((G * M + 4,), float("nan"), device="cuda")
        ctx.vds_convect(q_in, q_out[shift:shift + G * M], shape, ud, dx, dt, bc)
        assert torch.isnan(q_out[G * M + shift:]).all() and torch.isnan(q_out[:shift]).all()
        outs.append(q_out[shift:shift + G * M].view(G, M).clone())
    assert torch.equal(outs[0], outs[1])
    want = orc.convect_upwind(Q.astype(np.float64), u.astype(np.float64), shape, dx, dt, bc)
    assert np.max(np.abs(outs[0].cpu().numpy() - want)) <= 1e-6 * np.max(np.abs(Q))
    ctx.close()
