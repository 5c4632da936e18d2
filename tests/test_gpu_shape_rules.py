"""The FIXED policy's choices by shape and alignment: the default entry points
on both sides of every threshold, with matrices whose rows, pointers and
vectors are and are not whole 16-byte granules, against the FP64 oracle
within the parity bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blas

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_02389_gb300 import build, lift
    build.build()
    torch.cuda.set_device(0)
    lift.lift_init(0)
    yield lift
    torch.cuda.synchronize()
    assert lift.lift_read_status() == 0


def at(a, off):
    """A device copy of the fp32 array a, `off` elements past a 256-byte
    boundary, NaN around it: (buffer, address)."""
    b = torch.full((a.size + 128,), float("nan"), device="cuda")
    b[64 + off:64 + off + a.size] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()
    return b, b.data_ptr() + 4 * (64 + off)


# (M, N) around the rules' thresholds, ragged and whole; (pad, offsets of A, x, y)
FORMS = [(0, 0, 0, 0), (0, 1, 2, 3), (1, 0, 0, 0), (4, 0, 0, 1), (8, 0, 0, 0)]
GEMV = [(1, 1), (3, 0), (7, 255), (7, 256), (40, 1023), (9, 1024), (5, 2047), (999, 2048),
        (1000, 2048), (2000, 2050), (499, 4096), (500, 4097), (3, 8192), (2000, 8192), (4000, 1025),
        (4001, 3001), (2, 65535), (3, 65536), (5, 70003)]


@pytest.mark.parametrize("M,N", GEMV)
def test_gemv(L, M, N):
    rng = np.random.default_rng(M * 131 + N)
    A = rng.uniform(-1, 1, (M, N)).astype(np.float32)
    x, y = rng.uniform(-1, 1, N).astype(np.float32), rng.uniform(-1, 1, M).astype(np.float32)
    for pad, oa, ox, oy in FORMS:
        Ap = np.full((M, N + pad), np.nan, np.float32)
        Ap[:, :N] = A
        bufs = [at(Ap, oa), at(x, ox)]
        for beta in (0.5, 0.0):
            out, py = at(y, oy)
            L.lift_gemv(M, N, 1.25, bufs[0][1], N + pad, bufs[1][1], beta, py)
            got = out[64 + oy:64 + oy + M].cpu().numpy().astype(np.float64)
            ref = blas.gemv(A.astype(np.float64), x.astype(np.float64), y.astype(np.float64), 1.25, beta)
            tol = blas.tolerance(max(N, 2), 1.0) * blas.gemv_row_terms(A, x, y, 1.25, beta)
            assert np.all(np.abs(got - ref) <= tol), (pad, oa, ox, oy, beta)
            assert torch.isnan(out[:64 + oy]).all() and torch.isnan(out[64 + oy + M:]).all()


GEMV_T = [(1, 1), (0, 5), (5, 3), (33, 256), (128, 300), (129, 512), (129, 513), (9999, 100),
          (10000, 256), (10001, 257), (130, 1040), (130, 1044), (2048, 16384), (2049, 16380), (3, 65536),
          (70, 40001), (300, 600)]


@pytest.mark.parametrize("M,N", GEMV_T)
def test_gemv_t(L, M, N):
    rng = np.random.default_rng(M * 137 + N)
    A = rng.uniform(-1, 1, (M, N)).astype(np.float32)
    x, y = rng.uniform(-1, 1, M).astype(np.float32), rng.uniform(-1, 1, N).astype(np.float32)
    A64, x64, y64 = (t.astype(np.float64) for t in (A, x, y))
    for pad, oa, ox, oy in FORMS:
        Ap = np.full((M, N + pad), np.nan, np.float32)
        Ap[:, :N] = A
        bufs = [at(Ap, oa), at(x, ox)]
        for beta in (0.5, 0.0):
            out, py = at(y, oy)
            L.lift_gemv_t(M, N, 1.25, bufs[0][1], N + pad, bufs[1][1], beta, py)
            got = out[64 + oy:64 + oy + N].cpu().numpy().astype(np.float64)
            ref = blas.gemv_t(A64, x64, y64, 1.25, beta)
            terms = 1.25 * (np.abs(A64).T @ np.abs(x64)) + np.abs(beta * y64)
            assert np.all(np.abs(got - ref) <= blas.tolerance(max(M, 2), 1.0) * terms), \
                (pad, oa, ox, oy, beta)
            assert torch.isnan(out[:64 + oy]).all() and torch.isnan(out[64 + oy + N:]).all()


# the default vector entry points on slices: every pair of offsets, sizes
# around the vectors and tiles (2048 elements for the maps, 4096 for the
# reductions), NaN on both sides of every array
@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 2045, 2048, 4093, 4096, 4099, 8195, 20001, 1300001])
def test_unaligned_vectors(L, n):
    rng = np.random.default_rng(n)
    x, y = rng.standard_normal(n).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    x64, y64 = x.astype(np.float64), y.astype(np.float64)
    scal = (x64 * 1.5).astype(np.float32)
    axpy = (np.float32(-0.75) * x + y).astype(np.float32)      # fl(fl(a x) + y): two roundings
    nrm = float(np.sqrt(np.sum(x64 * x64)))
    want = [(L.lift_asum, blas.asum(x64), blas.asum_terms(x)), (L.lift_asum_comp, blas.asum(x64), None),
            (L.lift_sum, float(np.sum(x64)), blas.asum_terms(x)), (L.lift_nrm2, nrm, nrm)]
    for ox in range(4):
        bx, px = at(x, ox)
        for f, ref, terms in want:
            r = torch.full((1,), -7.0, device="cuda")
            f(px, n, r)
            tol = blas.tolerance(max(2, n), terms) if terms is not None else 2.0 ** -22 * abs(ref)
            assert abs(float(r.item()) - ref) <= tol, (f.__name__, ox)
        for oy in range(4):
            by, py = at(y, oy)
            r = torch.full((2,), -7.0, device="cuda")
            L.lift_dot(px, py, n, r[0:1])
            L.lift_dot_comp(px, py, n, r[1:2])
            ref, terms = blas.dot(x64, y64), blas.dot_terms(x, y)
            got = r.cpu().numpy().astype(np.float64)
            assert np.all(np.abs(got - ref) <= blas.tolerance(max(2, n), terms)), (ox, oy)
            L.lift_axpy(n, -0.75, px, py)
            assert np.array_equal(by[64 + oy:64 + oy + n].cpu().numpy().view(np.uint32),
                                  axpy.view(np.uint32)), (ox, oy)
            L.lift_scal(n, 1.5, px, py)
            assert np.array_equal(by[64 + oy:64 + oy + n].cpu().numpy().view(np.uint32),
                                  scal.view(np.uint32)), (ox, oy)
            assert torch.isnan(by[:64 + oy]).all() and torch.isnan(by[64 + oy + n:]).all()
        L.lift_scal(n, 1.5, px, px)                            # in place
        assert np.array_equal(bx[64 + ox:64 + ox + n].cpu().numpy().view(np.uint32),
                              scal.view(np.uint32)), ox
        assert torch.isnan(bx[:64 + ox]).all() and torch.isnan(bx[64 + ox + n:]).all()
    v = torch.ones(n + 8, device="cuda")                       # Inf and NaN propagate
    v[1 + n // 2] = float("inf")
    r = torch.zeros(1, device="cuda")
    L.lift_asum(v.data_ptr() + 4, n, r)
    assert r.item() == float("inf")
    L.lift_asum(v.data_ptr() + 8, 0, r)                        # an empty slice
    assert r.item() == 0.0
