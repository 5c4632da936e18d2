"""The combines of partial sums in the kernel expressions carry their rounding
errors: adding fp32 partials costs one rounding of the result, however many
partials there are and in whichever order a kernel adds them.

With one row per block (gemv-T) or one element per thread (split-row gemv)
and x = 1 the partials are the matrix's own entries, so the exact sum is
known.  A pair (sum, compensation) that goes through every add leaves the
final rounding, u |S|, and second-order terms: at most m adds, each of whose
errors is added to the compensation with one rounding, (m u)^2 sum|t|
doubled as for a compensated sum."""
import math

import numpy as np
import pytest

from oracle import blas
from oracle import lowlevel as ll
from oracle.patterns import TreeComp, evaluate

U = blas.U_FP32


def columns(m, n, seed):
    """m x n values of mixed sign and magnitude, exactly fp32."""
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((m, n)) * 2.0 ** rng.integers(-3, 4, (m, n))).astype(np.float32)


def sums(A, axis):
    return np.array([math.fsum(v) for v in np.moveaxis(A.astype(np.float64), axis, -1)])


@pytest.mark.parametrize("passes,cluster", [(1, 1), (2, 1)])
@pytest.mark.parametrize("RB", [2, 31, 32, 33, 94, 512])
def test_gemv_t_block_combine(RB, passes, cluster):
    A = columns(RB, 200, RB)
    z = evaluate(ll.gemv_t_z_variant(RB, 200, 1.0, 1, RB, passes, cluster), A, mode="f32",
                 env={"x": np.ones(RB, np.float32)})
    exact = sums(A, 0)
    tol = U * np.abs(exact) + 2 * (RB * U) ** 2 * np.abs(A.astype(np.float64)).sum(0)
    assert np.all(np.abs(z.astype(np.float64) - exact) <= tol)


@pytest.mark.parametrize("threads,S", [(128, 1), (256, 1), (128, 2), (256, 40), (128, 94)])
def test_gemv_split_row_combine(threads, S):
    N = threads * S
    A = columns(64, N, threads + S)
    z = evaluate(ll.gemv_split_z_variant(64, N, 1.0, 1, threads, threads, S), A, mode="f32",
                 env={"x": np.ones(N, np.float32)})
    exact = sums(A, 1)
    parts = np.abs(A.astype(np.float64).reshape(64, S, threads).sum(2)).sum(1) if S > 1 else 0.0
    tol = U * (np.abs(exact) + 1.01 * parts) + \
        2 * ((threads + S) * U) ** 2 * np.abs(A.astype(np.float64)).sum(1)
    assert np.all(np.abs(z.astype(np.float64) - exact) <= tol)


def test_tree_comp_values():
    # 1 and 63 terms of 2^-24, one per lane: a plain fp32 tree loses terms
    x = np.full((64, 1), 2.0 ** -24, np.float32)
    x[0] = 1.0
    assert evaluate(TreeComp(), x, mode="f32")[0] == np.float32(1 + 63 * 2.0 ** -24)
    i = np.arange(64 * 5).reshape(64, 5)
    assert evaluate(TreeComp(), i, mode="int")[0] == i.sum()
    for v in (np.inf, -np.inf, np.nan):              # non-finite sums stay what they are
        x[40] = v
        assert np.array_equal(evaluate(TreeComp(), x, mode="f32"), [v], equal_nan=True)
    x[41] = np.inf                                   # NaN + Inf
    assert np.isnan(evaluate(TreeComp(), x, mode="f32")[0])


# Row blocks (rows each, how many) of the one-pass form that 4-byte rows took
# and of the form that they take, on a device of 152 SMs
@pytest.mark.parametrize("M,old,new", [(40, 4, 8), (576, 4, 4), (689, 8, 12), (3147, 4, 8),
                                       (9534, 8, 20), (4097, 44, 48), (8191, 216, 252),
                                       (20000, 52, 60), (52140, 44, 104)])
def test_gemv_t_of_4_byte_rows_is_no_less_accurate(M, old, new):
    n = max(64, min(4096, (1 << 22) // M))
    rng = np.random.default_rng(M)
    A = rng.uniform(-1, 1, (M, n)).astype(np.float32)
    x = rng.uniform(-1, 1, M).astype(np.float32)
    exact = A.T.astype(np.float64) @ x.astype(np.float64)      # error far below fp32's
    err = []
    for B, passes in ((old, 1), (new, 4)):
        z = evaluate(ll.gemv_t_z_variant(M, n, 1.0, B, -(-M // B), passes), A, mode="f32", env={"x": x})
        err.append(np.linalg.norm(z.astype(np.float64) - exact))
    # 2 %: the roundings of the products are the same in both, those of the sums are not
    assert err[1] <= 1.02 * err[0]


@pytest.mark.parametrize("N", [256, 320, 512, 776, 1024, 1272])
def test_gemv_rows_of_8_float_vectors_are_no_less_accurate(N):
    # against the 4-float vectors that such rows were read in before; six
    # matrices, whose errors differ by 1 to 6 % and scatter by 1 % each
    M = (1 << 21) // N
    err = [0.0, 0.0]
    for seed in range(6):
        rng = np.random.default_rng(N + seed * 7919)
        A = rng.uniform(-1, 1, (M, N)).astype(np.float32)
        x = rng.uniform(-1, 1, N).astype(np.float32)
        exact = A.astype(np.float64) @ x.astype(np.float64)
        for i, vw in enumerate((4, 8)):
            z = evaluate(ll.gemv_z_variant(M, N, 1.0, vw), A, mode="f32", env={"x": x})
            err[i] += np.sum((z.astype(np.float64) - exact) ** 2)
    assert err[1] <= err[0]
