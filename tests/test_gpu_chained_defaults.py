"""Default calls chained on one stream with no host synchronisation: slices,
the calls whose combine is a second kernel, gemv and gemv-T by shape, and the
cost model's training launches.  Each call reads what the call before it wrote
or overwrites what it read; the results must be the bits of the same chain
synchronised after every call, and so must a CUDA graph of it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1502_02389_gb300 import synth

pytestmark = pytest.mark.gpu

N = (1 << 22) + 41            # two passes from 16 MiB, slices
ROUNDS, RES = 6, 12


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


class Chain:
    def __init__(self, L):
        self.L = L
        rng = np.random.default_rng(3)
        f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()  # noqa: E731
        q, s = synth.encode_fp8_blocks(rng.standard_normal(1 << 24))
        self.start = {"x": f(N + 8), "y": f(N + 8), "g": f(70000), "h": f(4100),
                      "p": f(12 * 64 + 64 + 64 * 64 + 64 + 64 * 33 + 33) * 0.1,
                      "m": torch.zeros(12 * 64 + 64 + 64 * 64 + 64 + 64 * 33 + 33, device="cuda")}
        self.start["v"] = self.start["m"] + 1e-4
        self.const = {"A": f(33, 70001), "B": f(4097, 1001), "xb": f(1 << 23).bfloat16(),
                      "q": torch.from_numpy(q).cuda(), "s": torch.from_numpy(s).cuda(),
                      "X": f(500, 12), "T": f(500, 33), "M": (f(500, 33) > 0).float()}
        self.d = {k: v.clone() for k, v in self.start.items()}
        self.res = torch.zeros(ROUNDS * RES, device="cuda")
        self.work = torch.zeros(L.lift_mlp_work_count(500, 64, 64), device="cuda")
        self.P, self.dP = torch.zeros(500, 33, device="cuda"), torch.zeros(500, 33, device="cuda")
        self.grads = torch.zeros_like(self.d["p"])

    def reset(self):
        for k, v in self.start.items():
            self.d[k].copy_(v)
        for t in (self.res, self.work, self.P, self.dP, self.grads):
            t.zero_()
        torch.cuda.synchronize()

    def issue(self, s, sync):
        L, d, c = self.L, self.d, self.const
        x, y = d["x"].data_ptr() + 4, d["y"].data_ptr() + 12
        count = d["p"].numel()

        def step(f, *a, **k):
            f(*a, **k)
            if sync:
                s.synchronize()

        for r in range(ROUNDS):
            o = lambda k: self.res[r * RES + k:r * RES + k + 1]  # noqa: B023, E731
            step(L.lift_scal, N, 0.5, x, x, s)                   # slices, in place
            step(L.lift_dot_comp, x, y, N, o(0), stream=s)
            step(L.lift_axpy, N, 0.25, x, y, s)
            step(L.lift_nrm2, y, N, o(1), s)
            step(L.lift_asum_comp, y, N, o(2), stream=s)
            step(L.lift_sum, x, N, o(3), s)
            step(L.lift_dot, x, y, N, o(4), s)
            step(L.lift_asum_comp, d["x"], N, o(5), stream=s)    # aligned, two kernels
            step(L.lift_asum_ex, L.BF16, c["xb"], None, 1 << 23, o(6), stream=s)
            step(L.lift_asum_ex, L.FP8_E4M3, c["q"], c["s"], 1 << 24, o(7), stream=s)
            step(L.lift_asum, d["y"], 1 << 18, o(8), s)          # one launch
            step(L.lift_gemv, 33, 70001, 0.01, c["A"], 70001, y, 0.5, d["h"], s)
            step(L.lift_gemv_t, 33, 70000, 0.1, c["A"], 70001, d["h"], 0.5, d["g"], s)
            step(L.lift_gemv_t, 4097, 1001, 0.01, c["B"], 1001, d["h"], 0.5, d["g"], s)
            step(L.lift_gemv, 4097, 1001, 0.01, c["B"], 1001, d["g"], 0.5, d["h"], s)
            step(L.lift_mlp_forward, 12, 64, 64, 33, d["p"], c["X"], 500, self.work, self.P, s)
            step(L.lift_mlp_loss, self.P, c["T"], c["M"], 500 * 33, 1e-3, self.dP, o(9), s)
            step(L.lift_mlp_backward, 12, 64, 64, 33, d["p"], c["X"], 500, self.work, self.dP,
                 self.grads, s)
            step(L.lift_mlp_adam, d["p"], self.grads, d["m"], d["v"], count, r + 1, 1e-3, 0.9, 0.999,
                 1e-8, s)
            step(L.lift_asum, d["p"], count, o(10), s)

    def state(self):
        torch.cuda.synchronize()
        return {k: t.clone() for k, t in dict(self.d, res=self.res, P=self.P, grads=self.grads).items()}


def test_chain_of_defaults(L):
    ch = Chain(L)
    s = torch.cuda.Stream()
    ch.reset()
    ch.issue(s, sync=True)
    want = ch.state()
    assert all(torch.isfinite(t).all() for t in want.values())
    for _ in range(3):
        ch.reset()
        ch.issue(s, sync=False)
        got = ch.state()
        for k in want:
            assert torch.equal(got[k], want[k]), k
    ch.reset()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        ch.issue(s, sync=False)
    ch.reset()
    graph.replay()
    got = ch.state()
    for k in want:
        assert torch.equal(got[k], want[k]), k
