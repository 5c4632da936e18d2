"""A batch run again and again: the queue and the per-op counters return to
their start by themselves, in both schedules and on any stream, for batches
smaller and larger than the grid, with gemv rows and columns around the
row groups and steps of each processing mode."""
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


def make(L, count, seed):
    rng = np.random.default_rng(seed)
    descs, checks, keep = [], [], []
    for i in range(count):
        if i % 2:
            M = int(rng.choice([1, 3, 15, 16, 17, 33, 200]))
            N = int(rng.choice([1, 31, 127, 128, 129, 255, 256, 257, 384, 1024, 1029, 4096]))
            off = int(rng.integers(0, 2))
            A = rng.uniform(-1, 1, (M, N)).astype(np.float32)
            x, y = rng.uniform(-1, 1, N).astype(np.float32), rng.uniform(-1, 1, M).astype(np.float32)
            buf = torch.zeros(M * N + 8, device="cuda")
            buf[off:off + M * N] = torch.from_numpy(A.reshape(-1)).cuda()
            xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
            beta = float(rng.choice([0.0, 0.5]))
            descs.append({"op": L.OP_GEMV, "variant": -1, "M": M, "N": N, "lda": N, "alpha": 1.25,
                          "beta": beta, "A": buf.data_ptr() + 4 * off, "x": xd, "out": yd})
            ref = blas.gemv(A.astype(np.float64), x.astype(np.float64), y.astype(np.float64), 1.25, beta)
            tol = blas.tolerance(max(2, N), 1.0) * blas.gemv_row_terms(A, x, y, 1.25, beta)
            keep += [buf, xd]
            checks.append((yd, torch.from_numpy(y).cuda(), ref, tol))
        else:
            n = int(rng.choice([0, 1, 300, 4095, 4097, 20000, 300001]))
            x = rng.uniform(-1, 1, n).astype(np.float32)
            xd, out = torch.from_numpy(x).cuda(), torch.zeros(1, device="cuda")
            scal = i % 4 == 0
            if scal:
                out = torch.zeros(n + 4, device="cuda")
            descs.append({"op": L.OP_SCAL if scal else L.OP_ASUM, "variant": -1, "n": n, "alpha": 1.5,
                          "x": xd, "out": out})
            ref = np.concatenate([x.astype(np.float64) * 1.5, np.zeros(4)]) if scal else \
                np.array([blas.asum(x.astype(np.float64)) if n else 0.0])
            tol = np.abs(ref) * 2.0 ** -24 if scal else blas.tolerance(max(2, n), blas.asum_terms(x))
            keep.append(xd)
            checks.append((out, torch.zeros_like(out), ref, tol))
    return descs, checks, keep


@pytest.mark.parametrize("count", [1, 7, 3000])
def test_reruns(L, count):
    descs, checks, keep = make(L, count, count)
    h = L.lift_batch_create(descs)
    streams = [torch.cuda.current_stream(), torch.cuda.Stream()]
    first = None
    try:
        for k in range(6):
            L.lift_batch_set_schedule(h, L.BATCH_PER_ITEM if k in (2, 3) else L.BATCH_QUEUE)
            for out, start, _, _ in checks:
                out.copy_(start)
            torch.cuda.synchronize()
            L.lift_batch_run(h, streams[k % 2])
            torch.cuda.synchronize()
            got = [c[0].cpu().numpy() for c in checks]
            for i, (g, (_, _, ref, tol)) in enumerate(zip(got, checks)):
                assert np.all(np.abs(g.astype(np.float64) - ref) <= tol), (k, i, descs[i])
            if first is None:
                first = got
            assert all(np.array_equal(a, b) for a, b in zip(first, got)), k
    finally:
        L.lift_batch_destroy(h)
