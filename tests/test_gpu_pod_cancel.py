"""The basis products X V Lambda^-1/2 where they cancel: every snapshot holds the
first mode, and the last one kept is 1000 times smaller (lambda_r / lambda_1 =
1e-6), so the terms of its column are 1000 times the column.  Whatever the
eigenvectors, the basis lies in the column space of X; what lies outside, by an
FP64 projection, is rounding: of the columns as stored (2^-24 each, twice, with
the two steps of the orthonormalisation) 4e-7 at most, where FP32 products would
leave 1e-5 to 1e-4.  Snapshots scaled to the ends of what the Gram takes too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Ns,M,r,scale", [(6000, 12, 6, 1.0), (6000, 12, 12, 1.0), (30000, 64, 20, 1.0),
                                          (6000, 12, 6, 1e15), (6000, 12, 6, 1e-15)])
def test_basis_stays_in_the_column_space(Ns, M, r, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_12550_gb300 import build
    build.build()
    from paper_2603_12550_gb300 import vds
    rng = np.random.default_rng(3)
    U = np.linalg.qr(rng.standard_normal((Ns, M)))[0]
    V = np.linalg.qr(rng.standard_normal((M, M)))[0]
    sig = 1e-3 ** (np.arange(M) / (r - 1))
    sig[r:] = 1e-3 * 0.7 ** np.arange(1, M - r + 1)
    X = ((U * sig) @ V.T * 100.0 * scale).astype(np.float32)
    ctx = vds.Context(0)
    basis, got = ctx.pod_build(torch.from_numpy(np.ascontiguousarray(X.T)).cuda(), Ns, M, 3, r_fixed=r)
    assert got == r
    phi = basis.phi().cpu().numpy().astype(np.float64)
    Q = np.linalg.qr(X.astype(np.float64) / scale)[0]
    out = np.linalg.norm(phi - Q @ (Q.T @ phi), axis=0)
    assert out.max() <= 4e-7, out
    basis.free()
    ctx.close()
