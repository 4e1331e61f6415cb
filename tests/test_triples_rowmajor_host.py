"""CPU restatement of the tile across a corner in the row-major walking order
(corner_tile_rowmajor in csrc/sg_compact_stencil.cu), against the geometry."""
import pytest

import oracle


def _corner_tile_rowmajor(q, kind, rb):
    at = (1, 2, 0)[kind]
    width = 3 ** (rb // 2)
    w, v = divmod(q, width)                  # the word of the next digit, the other
    pw, pv, ones, d, j = width, 1, 0, at, 0
    while j < rb:
        n, d = divmod(w, 3)
        if d != at:
            break
        ones += pw
        w, v, pw, pv, j = v, n, pv, 3 * pw, j + 1
    above = d == 0
    if j == rb or (kind != 0 and d != 1):
        return None, above
    return q + (d - at) * ones + (at - d) * pw, above


@pytest.mark.parametrize("rb", range(9))
def test_corner_tiles_of_the_rowmajor_order(rb):
    bx, by = oracle.block_map(rb, oracle.ORDER_ROWMAJOR)
    index = {(int(x), int(y)): q for q, (x, y) in enumerate(zip(bx, by))}
    for (x, y), q in index.items():
        left, up = index.get((x - 1, y)), index.get((x, y - 1))
        got, above = _corner_tile_rowmajor(q, 0, rb)
        assert got == (left if up is None else up)
        assert got is None or above == (up is not None)
        assert _corner_tile_rowmajor(q, 1, rb)[0] == index.get((x + 1, y))
        assert _corner_tile_rowmajor(q, 2, rb)[0] == index.get((x, y + 1))
