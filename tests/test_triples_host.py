"""CPU restatement of how a compact tile finds the tile across each of its
corners from the digits of its launch index (corner_tile in
csrc/sg_compact_stencil.cu), against the geometry."""
import pytest

import oracle


def _corner_tile(q, kind, rb):
    at = (1, 2, 0)[kind]
    pw, rest, d, j = 1, q, at, 0
    while j < rb:
        rest, d = divmod(rest, 3)
        if d != at:
            break
        j, pw = j + 1, 3 * pw
    above = d == 0
    if j == rb or (kind != 0 and d != 1):
        return None, above
    ones = (pw - 1) // 2
    if kind == 0:
        return q - ones - d * pw + pw + (2 * ones if d == 2 else 0), above
    return q - at * ones - pw + at * pw + ones, above


@pytest.mark.parametrize("rb", range(8))
def test_corner_tiles_match_the_geometry(rb):
    bx, by = oracle.block_map(rb, oracle.ORDER_INTERLEAVED)
    index = {(int(x), int(y)): q for q, (x, y) in enumerate(zip(bx, by))}
    for (x, y), q in index.items():
        left, up = index.get((x - 1, y)), index.get((x, y - 1))
        assert left is None or up is None
        got, above = _corner_tile(q, 0, rb)
        assert got == (left if up is None else up)
        assert got is None or above == (up is not None)
        assert _corner_tile(q, 1, rb)[0] == index.get((x + 1, y))
        assert _corner_tile(q, 2, rb)[0] == index.get((x, y + 1))
