"""gemv of matrices whose pitch is whole 16-byte granules and whose rows end
inside one: the default entry point on both sides of the rules for such rows,
against the FP64 oracle, with NaN between N and lda."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(3, 67), (3, 255), (40, 257), (4001, 511), (3999, 513), (4000, 513),
                                 (4000, 1023), (4000, 1025), (3999, 2047), (4001, 2047)])
@pytest.mark.parametrize("granule", [4, 8])
def test_gemv(M, N, granule):
    from paper_1502_02389_gb300 import build, lift as L
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    L.lift_init(0)
    rng = np.random.default_rng(M + N)
    A, x, y = (rng.uniform(-1, 1, s).astype(np.float32) for s in ((M, N), N, M))
    lda = (N + granule - 1) // granule * granule
    Ap = np.full((M, lda), np.nan, np.float32)
    Ap[:, :N] = A
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    Ad, xd, yd = dev(Ap), dev(x), dev(y)
    L.lift_gemv(M, N, 1.25, Ad, lda, xd, 0.5, yd)
    ref = blas.gemv(A.astype(np.float64), x.astype(np.float64), y.astype(np.float64), 1.25, 0.5)
    tol = blas.tolerance(N, 1.0) * blas.gemv_row_terms(A, x, y, 1.25, 0.5)
    assert np.all(np.abs(yd.cpu().numpy().astype(np.float64) - ref) <= tol)
    if N < 256 or (M >= 4000 and 512 <= N < 1024):       # rows folded in 4-byte vectors: variant 0's bits
        y0 = dev(y)
        L.lift_gemv_v(0, M, N, 1.25, Ad, lda, xd, 0.5, y0)
        assert torch.equal(yd, y0)
