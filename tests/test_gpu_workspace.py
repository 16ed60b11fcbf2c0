"""Large workspaces leave the memory to the program around the library: where
little is free, what a call takes beyond its small buffers stays within a quarter
of it, and its results are those with memory to spare (1e-5 for the passes, the
same bandwidth)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MB = 1 << 20


@pytest.fixture(scope="module")
def vds():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds as v
    return v


def _gradient(vds, ctx, q):
    g = torch.empty_like(q)
    ctx.vds_energy_grad(q, vds.params(3, 3, h=0.7), g=g, want_energy=False)
    return g


def _bandwidth(vds, ctx, q):
    return ctx.vds_bandwidth(q, 0)


def _batch(vds, ctx, q):
    n = [16384] * (q.shape[0] // 16384)
    b = vds.Batch(ctx, n, 9, vds.params(3, 3), np.full(len(n), 0.7), np.zeros((len(n), 3, 3)))
    g = torch.empty_like(q)
    b.energy_grad(q, g=g, want_energy=False)
    return g, b


# small: the call's buffers that grow with N alone
@pytest.mark.parametrize("call,small", [(_gradient, 72), (_bandwidth, 16), (_batch, 72)])
def test_a_quarter_of_what_is_free(vds, call, small):
    q = torch.randn((131072, 9), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    ctx = vds.Context(0)
    want = call(vds, ctx, q)
    ctx.close()
    torch.cuda.synchronize()
    want, got = want[0] if isinstance(want, tuple) else want, None
    ctx = vds.Context(0)
    call(vds, ctx, q[:16384])  # loads the kernels
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 320 * MB, dtype=torch.uint8, device="cuda")
    spare = torch.empty_like(q)  # what the call's result will take of the allocator
    del spare
    left = torch.cuda.mem_get_info()[0]
    try:
        got = call(vds, ctx, q)
        torch.cuda.synchronize()
        taken = left - torch.cuda.mem_get_info()[0]
    finally:
        del hog
        torch.cuda.empty_cache()
    assert left < 384 * MB
    assert taken <= left / 4 + small * MB, (taken, left)
    got = got[0] if isinstance(got, tuple) else got
    if isinstance(want, float):
        assert got == want
    else:
        assert float((got - want).abs().max()) <= 1e-5 * float(want.abs().max())
    ctx.close()
