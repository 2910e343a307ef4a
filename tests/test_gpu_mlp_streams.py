"""The network's forward kernel with several tiles in flight per CTA: a row's
outputs depend on that row alone, so every row of a large ragged batch must
equal, bit for bit, the same row evaluated in a batch of one tile."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TILE, SMS = 128, 152


# tiles per CTA around the number in flight (5): fewer, equal, one more, twice
# and a ragged last tile of one row
@pytest.mark.parametrize("n", [2 * TILE + 1, 4 * SMS * TILE + 1, 5 * SMS * TILE, 5 * SMS * TILE + 1,
                               10 * SMS * TILE + TILE - 1])
def test_rows_do_not_depend_on_the_batch(n):
    from paper_2501_06717_gb300 import bats as B
    rng = np.random.default_rng(n)
    P = (0.3 * rng.normal(size=B.BATS_MLP_NPARAM)).astype(np.float32)
    X = rng.normal(size=(n, 40)).astype(np.float32)
    m = B.Mlp(P)
    Y = m.forward(X)
    assert Y.shape == (n, 8) and np.isfinite(Y).all()
    starts = sorted({0, TILE, n - 1} | {int(i) for i in rng.integers(0, n - 1, 12)})
    for i in starts:
        Yi = m.forward(X[i:i + TILE])
        assert np.array_equal(Yi.view(np.uint32), Y[i:i + TILE].view(np.uint32)), i
    m.close()
