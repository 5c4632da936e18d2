"""More streams than workspace slots: default gemv calls of few rows, and
fp32 reductions of one launch, keep their partials in scratch of the
stream's own, so calls on many streams at once give the bits of the same
calls one after another; streams beyond the last own scratch run forms that
keep none, and graphs captured on one stream may be replayed side by side.
In a process of its own: the streams stay assigned until the
library is finalised."""
import os
import subprocess
import sys
import textwrap

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_CHILD = textwrap.dedent(
    """
    import ctypes
    import numpy as np
    import torch
    from paper_1502_02389_gb300 import build, lift as L

    build.build()
    L.lift_init(0)
    STREAMS, CHECKED = 264, 24          # own scratch is for the first 256
    rt = torch.cuda.cudart()
    streams = []
    for _ in range(STREAMS):
        h = ctypes.c_ulonglong(0)
        assert rt.cudaStreamCreate(ctypes.addressof(h)) == 0
        streams.append(h.value)
    r = torch.zeros(STREAMS, device="cuda")
    one = torch.ones(64, device="cuda")
    torch.cuda.synchronize()
    for k, s in enumerate(streams):                       # every stream is known to the library
        L.lift_asum(one, 64, r[k:k + 1], s)
    torch.cuda.synchronize()
    assert torch.all(r == 64)

    def calls(k, s, out):
        A, x, z = data[k]
        L.lift_gemv(6, 120000, 1.0, A, 120000, x, 0.0, out[0:6], s)
        L.lift_gemv(6, 119999, 1.0, A, 119999, x.data_ptr() + 4, 0.0, out[6:12], s)
        L.lift_asum(z, 1 << 18, out[12:13], s)
        L.lift_dot(z, z, 3 << 18, out[13:14], s)
        L.lift_sum(z, 1 << 20, out[14:15], s)

    g = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda *n: torch.randn(*n, device="cuda", generator=g)
    data = [(rnd(6, 120000) * (k + 1), rnd(120001), rnd(1 << 21) * (k + 1)) for k in range(CHECKED)]
    for first in (8, STREAMS - CHECKED):   # with own scratch; the last eight without
        use = streams[first:first + CHECKED]
        want = torch.zeros(CHECKED, 16, device="cuda")
        got = torch.zeros(40, CHECKED, 16, device="cuda")
        torch.cuda.synchronize()
        for k, s in enumerate(use):
            calls(k, s, want[k])
            torch.cuda.synchronize()
        for rep in range(40):
            for k, s in enumerate(use):
                if k < CHECKED - 8 or first == 8:
                    calls(k, s, got[rep, k])
                else:                      # reductions on shared slots may race: gemv alone
                    A, x, z = data[k]
                    L.lift_gemv(6, 120000, 1.0, A, 120000, x, 0.0, got[rep, k][0:6], s)
                    L.lift_gemv(6, 119999, 1.0, A, 119999, x.data_ptr() + 4, 0.0, got[rep, k][6:12], s)
                    got[rep, k][12:15] = want[k][12:15]
        torch.cuda.synchronize()
        assert torch.equal(got, want[None].expand_as(got)), first
        ref = torch.stack([(A.double() @ x[:120000].double()) for A, x, _ in data])
        assert torch.all((want[:, :6] - ref).abs() <= 1e-5 * ref.abs().max())
    # graphs captured on one stream, replayed side by side on others
    cap, side = torch.cuda.Stream(), [torch.cuda.Stream() for _ in range(3)]
    out = torch.zeros(3, 40, 12, device="cuda")
    graphs = []
    for k in range(3):
        A, x, _ = data[k]
        gr = torch.cuda.CUDAGraph()
        with torch.cuda.graph(gr, stream=cap):
            for i in range(40):
                L.lift_gemv(6, 120000, 1.0, A, 120000, x, 0.0, out[k, i][0:6], cap)
                L.lift_gemv(6, 119999, 1.0, A, 119999, x.data_ptr() + 4, 0.0, out[k, i][6:12], cap)
        graphs.append(gr)
    for _ in range(20):
        for gr, s in zip(graphs, side):
            with torch.cuda.stream(s):
                gr.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want[:3, None, :12].expand_as(out))
    assert L.lift_read_status() == 0
    print("OK")
    """
)


def test_more_streams_than_slots():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = subprocess.run([sys.executable, "-c", _CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert p.returncode == 0 and "OK" in p.stdout, p.stdout[-2000:] + p.stderr[-4000:]
