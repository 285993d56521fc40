"""The room a batch sets aside for its far-field work lists holds the tiles it lists."""
import ctypes

import pytest

from paper_1901_08393_gb300 import bem

# rows x columns of the far-field variants (include/bem.h)
TILES = [(32, 256), (16, 256), (64, 256), (8, 128), (16, 128), (32, 128), (8, 128), (16, 128), (32, 128), (4, 128),
         (8, 64), (4, 64), (2, 64), (1, 64)]


def _bound(tile, N):
    from paper_1901_08393_gb300 import build

    build.build()
    f = getattr(ctypes.CDLL(bem.LIB_PATH), "_ZN3bem21far_batch_items_boundEil")  # bem::far_batch_items_bound(int, long)
    f.argtypes, f.restype = [ctypes.c_int, ctypes.c_long], ctypes.c_double
    return f(tile, N)


def _listed(R, C, N):
    """The tiles of R x C entries that reach the diagonal or above."""
    return sum(len(range(i0 // C * C, N, C)) for i0 in range(0, N, R))


@pytest.mark.parametrize("tile", range(len(TILES)), ids=lambda k: "x".join(map(str, TILES[k])))
def test_bound_holds_the_list(tile):
    assert len(TILES) == bem.FAR_TILE_VARIANTS
    R, C = TILES[tile]
    for N in sorted({4, 12, 63, 64, 65, 257} | {k * C + e for k in (1, 2, 3, 8, 9, 39, 94) for e in (-1, 0, 1, R)}):
        listed = _listed(R, C, N)
        assert _bound(tile + 1, N) == listed, N
        if N < 1024 or R * C >= 512:  # the variants that timing may choose for a batch
            assert _bound(0, N) >= listed, N
