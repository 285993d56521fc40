"""The marking's sort in chunks and its 32-way search of the running sums, at the edges of a
chunk, of the chunk lengths and of the longest merged array: the marked set equals the
oracle's (whole numbers: no tolerance)."""
import numpy as np
import pytest

import oracle as O
from paper_1901_08393_gb300 import bem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = bem.Context()
    yield c
    c.close()


@pytest.mark.parametrize("N", [1023, 1024, 1025, 2047, 3073, 16384, 16385, 18433, 65537, 131072, 131073])
def test_marked_set_at_chunk_edges(ctx, N):
    rng = np.random.default_rng(N)
    cases = (rng.random(N) ** 6,
             rng.integers(0, 5, N) / 4.0,                        # ties across every chunk, zeros
             np.sort(rng.random(N))[::-1].copy(),                # sorted already
             np.where(np.arange(N) == N - 1, 1.0, 1e-12))        # one key before all others
    for eta2 in cases:
        for theta in (0.01, 0.5, 1.0):
            m, n = bem.dorfler(ctx, eta2, theta)
            ref = O.dorfler(eta2, theta)
            assert np.array_equal(m, ref) and n == int(ref.sum())
