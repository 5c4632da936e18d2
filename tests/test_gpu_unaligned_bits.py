"""Default reductions of slices, bit for bit: the FP64 sum of the partials
against the form's low-level expression at every offset, from one tile to
several per CTA and on both sides of the second launch (16 MiB read), calls
repeated back to back; the compensated ones within their bound."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blas
from oracle import lowlevel as ll
from oracle.patterns import evaluate

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


def slice_of(a, off):
    b = torch.full((a.size + 16,), float("nan"), device="cuda")
    b[off:off + a.size] = torch.from_numpy(a).cuda()
    return b, b.data_ptr() + 4 * off


def expected(op, n, m, x, y, sms):
    """The FP64 sums that the expression gives, one for each number of CTAs
    per SM that the device may hold."""
    T = math.ceil((n + m) / ll.UNALIGNED_TILE)
    grids = {math.ceil(T / math.ceil(T / (sms * k))) for k in range(1, 9)}
    out = set()
    for g in grids:
        e, ln = ll.unaligned_reduce(op, n, m, g, cast32=False)
        pad = lambda v: np.concatenate([np.zeros(m, np.float32), v, np.zeros(ln - n - m, np.float32)])  # noqa: E731,B023
        v = evaluate(e, (pad(x), pad(y)) if op == "dot" else pad(x), mode="f32")[0]
        out.add(float(v))
    return out


# (n, offsets of x, offsets of y); one and two inputs change to two launches
# at 2^22 and 2^21 elements
SIZES = [(5, (1, 2, 3), (0, 3)), (4093, (1, 2, 3), (1, 2)), (20001, (1, 3), (0, 1, 2)),
         (600000, (2,), (1,)), ((1 << 21) - 1, (1,), (1, 3)), ((1 << 21) + 3, (3,), (0, 3)),
         ((1 << 22) - 1, (1,), (2,)), ((1 << 22) + 5, (2,), (2, 3)), ((1 << 23) + 43, (1,), (3,))]


@pytest.mark.parametrize("n,xs,ys", SIZES)
def test_reductions(L, n, xs, ys):
    rng = np.random.default_rng(n)
    x, y = (rng.standard_normal(n).astype(np.float32) for _ in range(2))
    sms = L.lift_sm_count()
    r, r64 = torch.zeros(64, device="cuda"), torch.zeros(64, device="cuda", dtype=torch.float64)
    for ox in xs:
        bx, px = slice_of(x, ox)
        for op, f in (("asum", L.lift_asum_v), ("sum", L.lift_sum_v), ("nrm2", L.lift_nrm2_v)):
            for k in range(8):                      # back to back
                f(-1, px, n, r[k:k + 1], r64[k:k + 1])
            got, got32 = r64[:8].cpu().numpy(), r[:8].cpu().numpy()
            assert np.all(got == got[0]) and np.all(got32 == np.float32(got[0])), op
            assert float(got[0]) in expected(op, n, ox, x, None, sms), op
        for oy in ys:
            by, py = slice_of(y, oy)
            for k in range(8):
                L.lift_dot_v(-1, px, py, n, r[k:k + 1], r64[k:k + 1])
            got, got32 = r64[:8].cpu().numpy(), r[:8].cpu().numpy()
            assert np.all(got == got[0]) and np.all(got32 == np.float32(got[0]))
            assert float(got[0]) in expected("dot", n, ox, x, y, sms), (ox, oy)


@pytest.mark.parametrize("n", [(1 << 21) - 1, (1 << 21) + 3, (1 << 22) - 1, (1 << 22) + 5, (1 << 24) + 43])
def test_compensated(L, n):
    rng = np.random.default_rng(n)
    x, y = (rng.standard_normal(n).astype(np.float32) for _ in range(2))
    # terms per pair: at most every vector lane of a thread, 4 per lane and tile
    m = 4 * 4 * math.ceil(math.ceil((n + 3) / ll.UNALIGNED_TILE) / L.lift_sm_count())
    r, r64 = torch.zeros(8, device="cuda"), torch.zeros(8, device="cuda", dtype=torch.float64)
    exact, terms = blas.asum_exact(x), blas.asum_terms(x)
    bx, px = slice_of(x, 1)
    for k in range(8):
        L.lift_asum_comp(px, n, r[k:k + 1], r64[k:k + 1])
    got = r.cpu().numpy().astype(np.float64)
    assert np.all(got == got[0]) and torch.all(r64 == r64[0])
    assert abs(got[0] - exact) <= blas.compensated_tolerance(exact, terms, m)
    exact, terms = blas.dot_exact(x, y), blas.dot_terms(x, y)
    for oy in (1, 3):
        by, py = slice_of(y, oy)
        for k in range(8):
            L.lift_dot_comp(px, py, n, r[k:k + 1], r64[k:k + 1])
        got = r.cpu().numpy().astype(np.float64)
        assert np.all(got == got[0]) and torch.all(r64 == r64[0])
        assert abs(got[0] - exact) <= blas.compensated_tolerance(exact, terms, m)
