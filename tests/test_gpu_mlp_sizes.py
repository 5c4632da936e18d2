"""The cost model's kernels at the edges of their tiles: the fused network
(64 units in both hidden layers) with batches, inputs and outputs around the
row groups, column tiles and staged chunks, other sizes on the one-operation
kernels, and unaligned loss arrays, against the FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_02389_gb300 import build, lift
    build.build()
    torch.cuda.set_device(0)
    lift.lift_init(0)
    return lift


def rel(a, b):
    return float(np.max(np.abs(a - b)) / max(1e-30, np.max(np.abs(b))))


# (d_in, h1, h2, V, B)
SIZES = [(12, 64, 64, 1, 1), (1, 64, 64, 31, 15), (13, 64, 64, 33, 17), (64, 64, 64, 288, 16),
         (12, 64, 64, 289, 33), (7, 64, 64, 600, 100), (12, 64, 64, 265, 2308), (65, 64, 64, 20, 9),
         (12, 32, 64, 40, 50), (5, 64, 48, 265, 70)]


@pytest.mark.parametrize("d,h1,h2,V,B", SIZES)
@pytest.mark.parametrize("off", [0, 1])
def test_forward_loss_gradients(L, d, h1, h2, V, B, off):
    rng = np.random.default_rng(d + 3 * V + B)
    f32 = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    X, T = rng.random((B, d)).astype(np.float32), f32(B, V)
    M = (rng.random((B, V)) < 0.5).astype(np.float32)
    M[0, 0] = 1.0
    p = {"W1": f32(d, h1), "b1": f32(h1), "W2": f32(h1, h2) / 8, "b2": f32(h2), "W3": f32(h2, V) / 8,
         "b3": f32(V)}
    names = list(mlp.PARAM_NAMES)
    flat = np.concatenate([p[k].reshape(-1) for k in ("W1", "b1", "W2", "b2", "W3", "b3")])
    p64 = {k: v.astype(np.float64) for k, v in p.items()}
    inv = float(np.float32(1.0 / M.sum()))

    def dev(a):                      # off: 4 bytes past a 16-byte boundary
        b = torch.zeros(a.size + 8, device="cuda")
        b[off:off + a.size] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()
        return b, b.data_ptr() + 4 * off

    keep = {k: dev(v) for k, v in dict(X=X, T=T, M=M, p=flat, P=np.zeros((B, V), np.float32),
                                       dP=np.zeros((B, V), np.float32), g=np.zeros_like(flat)).items()}
    q = {k: v[1] for k, v in keep.items()}
    work = torch.zeros(L.lift_mlp_work_count(B, h1, h2), device="cuda")
    loss = torch.zeros(1, device="cuda")
    L.lift_mlp_forward(d, h1, h2, V, q["p"], q["X"], B, work, q["P"])
    L.lift_mlp_loss(q["P"], q["T"], q["M"], B * V, inv, q["dP"], loss)
    L.lift_mlp_backward(d, h1, h2, V, q["p"], q["X"], B, work, q["dP"], q["g"])
    torch.cuda.synchronize()
    out = lambda k, n: keep[k][0][off:off + n].cpu().numpy()  # noqa: E731
    Pref, cache = mlp.forward(p64, X.astype(np.float64))
    assert rel(out("P", B * V).reshape(B, V), Pref) <= 1e-5
    lref = mlp.masked_mse(Pref, T.astype(np.float64), M)
    assert abs(float(loss.item()) - lref) <= 1e-5 * lref
    gref = mlp.backward(p64, cache, Pref, T.astype(np.float64), M)
    g, o = out("g", flat.size), 0
    for k in ("W1", "b1", "W2", "b2", "W3", "b3"):
        n = p[k].size
        assert rel(g[o:o + n].reshape(p[k].shape), gref[k]) <= 1e-4, k
        o += n
    assert set(names) == set(p)
    # nothing before or after the arrays is written
    for k, n in (("P", B * V), ("dP", B * V), ("g", flat.size)):
        b = keep[k][0]
        assert torch.all(b[:off] == 0) and torch.all(b[off + n:] == 0), k
