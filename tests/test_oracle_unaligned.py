"""The expression of a default reduction of a slice: on integer inputs every
order gives the exact sum, so a dropped element, vector, tile or warp would
show."""
import numpy as np
import pytest

from oracle import lowlevel as ll
from oracle.patterns import evaluate


@pytest.mark.parametrize("op", ["asum", "dot", "nrm2", "sum"])
@pytest.mark.parametrize("n,m,grid", [(1, 3, 1), (4095, 1, 1), (4094, 2, 1), (4093, 3, 1), (9000, 1, 2),
                                      (20001, 2, 2), (70000, 3, 5)])
def test_exact_on_integers(op, n, m, grid):
    rng = np.random.default_rng(n + m)
    x, y = (rng.integers(-9, 9, n).astype(float) for _ in range(2))
    e, L = ll.unaligned_reduce(op, n, m, grid, cast32=False)
    pad = lambda v: np.concatenate([np.zeros(m), v, np.zeros(L - n - m)])  # noqa: E731
    got = evaluate(e, (pad(x), pad(y)) if op == "dot" else pad(x))[0]
    want = {"asum": np.abs(x).sum(), "dot": x @ y, "sum": x.sum(), "nrm2": np.sqrt(x @ x)}[op]
    assert got == want
