"""Host threads that share a stream: a call of two launches (partials, then
their combine) is submitted as one, so calls that several threads make on one
stream at the same time give the bits that each gives alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1502_02389_gb300 import synth

pytestmark = pytest.mark.gpu

THREADS, REPEATS = 4, 60


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


# a call's inputs are the thread's own; every call here takes two launches
def _calls(L, k):
    rng = np.random.default_rng(100 + k)
    n = 1 << 22
    vals = (rng.standard_normal(n + 8) * (k + 1)).astype(np.float32)
    x = torch.from_numpy(vals).cuda()
    y = torch.from_numpy(rng.standard_normal(n + 8).astype(np.float32)).cuda()
    xb = torch.cat([x, x, y]).bfloat16()
    q, s = synth.encode_fp8_blocks(np.tile(vals[:n].astype(np.float64), 4))
    q, s = torch.from_numpy(q).cuda(), torch.from_numpy(s).cuda()
    A = torch.from_numpy((rng.standard_normal((8, 131072)) * (k + 1)).astype(np.float32)).cuda()
    B = torch.from_numpy((rng.standard_normal((4097, 301)) * (k + 1)).astype(np.float32)).cuda()
    xu, yu = x.data_ptr() + 4, y.data_ptr() + 12
    return [
        (1, lambda st, r: L.lift_asum(x, n, r, st)),
        (1, lambda st, r: L.lift_dot(x, y, n, r, st)),
        (1, lambda st, r: L.lift_asum_comp(x, n, r, stream=st)),
        (1, lambda st, r: L.lift_dot_comp(x, y, n, r, stream=st)),
        (1, lambda st, r: L.lift_asum(xu, n, r, st)),
        (1, lambda st, r: L.lift_nrm2(xu, n, r, st)),
        (1, lambda st, r: L.lift_dot_comp(xu, yu, n, r, stream=st)),
        (1, lambda st, r: L.lift_asum_ex(L.BF16, xb, None, 3 * n, r, stream=st)),
        (1, lambda st, r: L.lift_asum_ex(L.FP8_E4M3, q, s, 4 * n, r, stream=st)),
        (8, lambda st, r: L.lift_gemv(8, 131072, 1.0, A, 131072, x, 0.0, r, st)),
        (8, lambda st, r: L.lift_gemv(8, 131071, 1.0, A, 131072, xu, 0.0, r, st)),
        (301, lambda st, r: L.lift_gemv_t(4097, 301, 1.0, B, 301, y, 0.0, r, st)),
        (131072, lambda st, r: L.lift_gemv_t(8, 131072, 1.0, A, 131072, y, 0.0, r, st)),
    ], (x, y, xb, q, s, A, B)


def test_threads_on_one_stream(L):
    st = torch.cuda.Stream()
    work = [_calls(L, k) for k in range(THREADS)]
    want = []
    for calls, _ in work:
        out = [torch.full((m,), -7.0, device="cuda") for m, _ in calls]
        torch.cuda.synchronize()
        for (_, f), r in zip(calls, out):
            f(st, r)
            st.synchronize()
        want.append(out)
    got = [[[torch.full((m,), -7.0, device="cuda") for _ in range(2)] for m, _ in calls]
           for calls, _ in work]
    bad = [torch.zeros(len(calls), dtype=torch.int64, device="cuda") for calls, _ in work]
    torch.cuda.synchronize()
    errors = []
    gate = threading.Barrier(THREADS)

    def run(k):
        try:
            calls = work[k][0]
            gate.wait(60)
            for rep in range(REPEATS):
                for j in range(len(calls)):
                    # another order in each thread, so that different calls meet
                    i = (j * (2 * k + 1) + rep) % len(calls)
                    calls[i][1](st, got[k][i][rep % 2])
                    with torch.cuda.stream(st):
                        bad[k][i] += (got[k][i][rep % 2] != want[k][i]).any()
        except Exception as e:               # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(THREADS)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for k in range(THREADS):
        assert bad[k].sum().item() == 0, (k, bad[k].tolist())
