"""The cost model's fused kernels where they stage their inputs in pieces:
output columns on both sides of what the forward (736) and the backward
launch (544) hold at once and several chunks beyond, and batches on both
sides of the rows that a CTA of the weight gradients holds (512 of an eighth
of the batch), against the FP64 oracle; repeated calls give the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp

pytestmark = pytest.mark.gpu

KEYS = ("W1", "b1", "W2", "b2", "W3", "b3")


def rel(a, b):
    return float(np.max(np.abs(a - b)) / max(1e-30, np.max(np.abs(b))))


# (d_in, V, B)
@pytest.mark.parametrize("d,V,B", [(12, 544, 20), (13, 545, 33), (12, 736, 17), (12, 737, 33), (13, 1300, 20),
                                   (7, 1700, 16), (13, 40, 2432), (12, 33, 2433), (12, 40, 4096),
                                   (13, 31, 4104), (64, 265, 5000), (5, 20, 9001)])
@pytest.mark.parametrize("off", [0, 1])
def test_pieces(d, V, B, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_02389_gb300 import build, lift as L
    build.build()
    L.lift_init(0)
    rng = np.random.default_rng(d + 3 * V + B)
    f32 = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    X, T = rng.random((B, d)).astype(np.float32), f32(B, V)
    M = (rng.random((B, V)) < 0.5).astype(np.float32)
    p = {"W1": f32(d, 64), "b1": f32(64), "W2": f32(64, 64) / 8, "b2": f32(64), "W3": f32(64, V) / 8,
         "b3": f32(V)}
    flat = np.concatenate([p[k].reshape(-1) for k in KEYS])
    p64 = {k: v.astype(np.float64) for k, v in p.items()}
    inv = float(np.float32(1.0 / M.sum()))

    def dev(a):                      # off: 4 bytes past a 16-byte boundary
        b = torch.zeros(a.size + 8, device="cuda")
        b[off:off + a.size] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()
        return b, b.data_ptr() + 4 * off

    z = np.zeros((B, V), np.float32)
    keep = {k: dev(v) for k, v in dict(X=X, T=T, M=M, p=flat, P=z, dP=z, g=np.zeros_like(flat)).items()}
    q = {k: v[1] for k, v in keep.items()}
    work = torch.zeros(L.lift_mlp_work_count(B, 64, 64) + 1, device="cuda")
    loss = torch.zeros(1, device="cuda")
    out = lambda k, n: keep[k][0][off:off + n].cpu().numpy().copy()  # noqa: E731
    runs = []
    for _ in range(3):
        L.lift_mlp_forward(d, 64, 64, V, q["p"], q["X"], B, work.data_ptr() + 4 * off, q["P"])
        L.lift_mlp_loss(q["P"], q["T"], q["M"], B * V, inv, q["dP"], loss)
        L.lift_mlp_backward(d, 64, 64, V, q["p"], q["X"], B, work.data_ptr() + 4 * off, q["dP"], q["g"])
        torch.cuda.synchronize()
        runs.append((out("P", B * V), out("g", flat.size), float(loss.item())))
    for r in runs[1:]:
        assert np.array_equal(r[0], runs[0][0]) and np.array_equal(r[1], runs[0][1]) and r[2] == runs[0][2]
    Pref, cache = mlp.forward(p64, X.astype(np.float64))
    assert rel(runs[0][0].reshape(B, V), Pref) <= 1e-5
    lref = mlp.masked_mse(Pref, T.astype(np.float64), M)
    assert abs(runs[0][2] - lref) <= 1e-5 * lref
    # a unit within rounding of 0 may be on in fp32 and off in 64 bits, and its
    # row then counts as a whole: the gates are the kernel's own (Z1 and Z2 of
    # the work buffer), which may differ from the reference's only there
    Xc, Z1, H1, Z2, H2 = cache
    zs = work[off:off + 4 * B * 64].cpu().numpy().reshape(4, B, 64)
    for Z, z in ((Z1, zs[0]), (Z2, zs[2])):
        flips = (z > 0) != (Z > 0)
        assert flips.sum() <= 8 and np.all(np.abs(Z[flips]) <= 1e-6)
    gref = mlp.backward(p64, (Xc, zs[0], H1, zs[2], H2), Pref, T.astype(np.float64), M)
    o = 0
    for k in KEYS:
        n = p[k].size
        assert rel(runs[0][1][o:o + n].reshape(p[k].shape), gref[k]) <= 1e-4, k
        o += n
    for k, n in (("P", B * V), ("dP", B * V), ("g", flat.size)):
        b = keep[k][0]
        assert torch.all(b[:off] == 0) and torch.all(b[off + n:] == 0), k
