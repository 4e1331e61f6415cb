"""CPU restatement of the fused CA on words (csrc/sg_words.cuh): units of 64-tiles
with the three tiles at their corners, triples of cells, one neighbour at most
at each corner.  Compared with the oracle over partial tiles, grid edges, every
unit depth and the deepest light cone."""
import numpy as np
import pytest

import oracle
from paper_1706_04552_gb300 import inputs


def _digits(x, y, levels):
    return sum((((x >> j) & 1) + 2 * ((y >> j) & 1)) * 3 ** j for j in range(levels))


def _coords(p, levels):
    x = y = 0
    for j in range(levels):
        d = p // 3 ** j % 3
        x |= (d == 1) << j
        y |= (d == 2) << j
    return x, y


def _neighbour(x, y, n, corner):
    near = {"A": [(x - 1, y), (x, y - 1)], "B": [(x + 1, y), (x + 1, y - 1)],
            "C": [(x, y + 1), (x - 1, y + 1)]}[corner]
    live = [0 <= a < n and 0 <= b < n and (a & b) == 0 for a, b in near]
    assert sum(live) <= 1                       # at each corner at most one triangle
    for k in (0, 1):
        if live[k]:
            return (k + 1,) + near[k]
    return 0, x, y


def _maj(a, b, c):
    return (a & b) | (c & (a ^ b))


# 16-blocks of a corner tile that are read, by corner and kind of contact
_NEED = {("A", 1): 1 << 4, ("A", 2): 1 << 8, ("B", 1): 1 | 1 << 2, ("B", 2): 1 << 8,
         ("C", 1): 1 | 1 << 1, ("C", 2): 1 << 4}
_TRIPLES = [[_neighbour(*_coords(p, 5), 32, c) for c in "ABC"] for p in range(243)]


def _unit(g, r, ux, uy, depth, k):
    n, nb = g.shape[0], max(1, g.shape[0] >> 6)
    l = min(depth, max(0, r - 6))
    ox, oy, far = ux << l, uy << l, (1 << l) - 1
    tiles = [(ox + _coords(t, l)[0], oy + _coords(t, l)[1]) for t in range(3 ** l)]
    blocks = [0x1FF] * len(tiles)
    for c, (x, y) in zip("ABC", ((ox, oy), (ox + far, oy), (ox, oy + far))):
        kind, a, b = _neighbour(x, y, nb, c)
        tiles.append((a, b) if kind else None)
        blocks.append(_NEED[c, kind] if kind else 0)
    lanes = len(tiles)
    w = np.zeros((3, 243, lanes), np.uint8)
    for t in range(lanes):
        for p in range(243):
            if not (blocks[t] >> (p // 27)) & 1:
                continue
            x, y = _coords(p, 5)
            for c, (dx, dy) in enumerate(((0, 0), (1, 0), (0, 1))):
                xx, yy = tiles[t][0] * 64 + 2 * x + dx, tiles[t][1] * 64 + 2 * y + dy
                if xx < n and yy < n:
                    w[c, p, t] = g[yy, xx]
    at = {tile: t for t, tile in enumerate(tiles) if tile is not None}
    links = []
    for t in range(lanes):
        row = []
        for c in "ABC":
            kind, a, b = _neighbour(*tiles[t], nb, c) if tiles[t] else (0, 0, 0)
            row.append((kind, at[a, b]) if kind and (a, b) in at else (0, 0))
        links.append(row)
    zero = np.zeros(lanes, np.uint8)
    for _ in range(k):
        new = np.zeros_like(w)
        P, L, U, Q1, Q2, R1, R2 = (zero.copy() for _ in range(7))
        for t, ((ka, sa), (kb, sb), (kc, sc)) in enumerate(links):
            L[t], U[t] = ka == 1, ka == 2
            P[t] = w[1, 121, sa] if ka == 1 else w[2, 242, sa] if ka == 2 else 0
            Q1[t] = w[0, 0, sb] if kb == 1 else w[2, 242, sb] if kb == 2 else 0
            Q2[t] = w[2, 0, sb] if kb == 1 else 0
            R1[t] = w[0, 0, sc] if kc == 1 else w[1, 121, sc] if kc == 2 else 0
            R2[t] = w[1, 0, sc] if kc == 1 else 0
        for p in range(243):
            x, y = _coords(p, 5)
            if 2 * x >= n or 2 * y >= n:
                continue                        # outside a grid smaller than the tile
            (ka, ax, ay), (kb, bx, by), (kc, cx, cy) = _TRIPLES[p]
            ia, ib, ic = _digits(ax, ay, 5), _digits(bx, by, 5), _digits(cx, cy, 5)
            a, b, c = w[:, p]
            pp = w[1, ia] if ka == 1 else w[2, ia] if ka == 2 else zero
            pl, pu = (pp if ka == 1 else zero), (pp if ka == 2 else zero)
            q1 = w[0, ib] if kb == 1 else w[2, ib] if kb == 2 else zero
            q2 = w[2, ib] if kb == 1 else zero
            r1 = w[0, ic] if kc == 1 else w[1, ic] if kc == 2 else zero
            r2 = w[1, ic] if kc == 1 else zero
            if p == 0:
                pp, pl, pu = P, P & L, P & U
            if p == 121:
                q1, q2 = Q1, Q2
            if p == 242:
                r1, r2 = R1, R2
            new[0, p] = _maj(b, c, pp) & ((b ^ c ^ pp) | a)
            s = a ^ c ^ pu
            new[1, p] = ((s ^ q1 ^ q2) | b) & (_maj(a, c, pu) ^ _maj(s, q1, q2))
            s = a ^ b ^ pl
            new[2, p] = ((s ^ r1 ^ r2) | c) & (_maj(a, b, pl) ^ _maj(s, r1, r2))
        w = new
    return tiles[:3 ** l], w


@pytest.mark.parametrize("r,depth", [(4, 3), (5, 3), (6, 3), (8, 2), (9, 3), (10, 2), (10, 3)])
@pytest.mark.parametrize("k", [1, 16])
def test_words_match_the_oracle(r, depth, k):
    n = 1 << r
    g = inputs.ca_seed_grid(r, 0.45, 7 * r + k)
    want = oracle.ca_steps(r, g, k)
    side = max(1, n >> (6 + min(depth, max(0, r - 6))))
    for ux, uy in [(a, b) for a in range(side) for b in range(side) if (a & b) == 0][:5]:
        tiles, w = _unit(g, r, ux, uy, depth, k)
        for t, (bx, by) in enumerate(tiles):
            for p in range(243):
                x, y = _coords(p, 5)
                for c, (dx, dy) in enumerate(((0, 0), (1, 0), (0, 1))):
                    xx, yy = bx * 64 + 2 * x + dx, by * 64 + 2 * y + dy
                    inside = xx < n and yy < n
                    assert w[c, p, t] == (want[yy, xx] if inside else 0)


@pytest.mark.parametrize("off_in,off_out", [(0, 0), (1, 15), (7, 3), (8, 8), (15, 1)])
def test_compact_runs_shift_to_any_alignment(off_in, off_out):
    # a 729-byte run read in aligned 16-byte pieces: cells 96 W + 32 i .. + 31 of
    # warp W come from a funnel shift of its pieces' bits; the way out shifts
    # the same groups to the output's alignment
    cells = np.random.default_rng(off_in).integers(0, 2, 729)
    flat = np.concatenate([np.ones(off_in, int), cells, np.ones(64, int)])   # neighbours around
    groups = {}
    for warp in range(8):
        b = [0, 0, 0, 0]
        for i in range(7):
            start = 96 * warp + 16 * i
            if start < off_in + 729:
                v = sum(int(x) << j for j, x in enumerate(flat[start:start + 16]))
                b[i >> 1] |= v << (16 * (i & 1))
        for i in range(3):
            if 3 * warp + i <= 22:
                x = ((b[i] | b[i + 1] << 32) >> off_in) & 0xFFFFFFFF
                groups[3 * warp + i] = x
    for e in range(729):
        assert (groups[e >> 5] >> (e & 31)) & 1 == cells[e]
    valid = {g: v if g < 22 else v & ((1 << 25) - 1) for g, v in groups.items()}
    out = np.full(off_out + 729 + 64, -1)
    for warp in range(8):
        g = [valid.get(3 * warp - 1 + i, 0) for i in range(4)]
        for i in range(3):
            v = (((g[i + 1] << 32 | g[i]) << off_out) >> 32) & 0xFFFFFFFF
            for h in range(2):
                first = 96 * warp + 32 * i + 16 * h - off_out
                for j in range(16):
                    if 0 <= first + j < 729:
                        assert out[off_out + first + j] == -1          # stored once
                        out[off_out + first + j] = (v >> (16 * h + j)) & 1
    assert np.array_equal(out[off_out:off_out + 729], cells)
    assert (out[:off_out] == -1).all() and (out[off_out + 729:] == -1).all()


def _corner_tile_index(q, at, rbu, l):
    pw, rest, d, j = 1, q, at, 0
    while j < rbu:
        rest, d = divmod(rest, 3)
        if d != at:
            break
        j, pw = j + 1, 3 * pw
    if j == rbu:
        return None
    per = 3 ** l
    return (q + (at - d) * (pw - (pw - 1) // 2)) * per + d * ((per - 1) // 2)


@pytest.mark.parametrize("rb,l", [(0, 0), (1, 0), (2, 2), (3, 2), (4, 3), (5, 3), (5, 2), (6, 3)])
def test_corner_tiles_of_a_unit(rb, l):
    # the tile across each corner of a unit, and the tiles inside it, by the
    # digits of the interleaved order
    bx, by = oracle.block_map(rb, oracle.ORDER_INTERLEAVED)
    place = [(int(x), int(y)) for x, y in zip(bx, by)]
    index = {p: q for q, p in enumerate(place)}
    ux, uy = oracle.block_map(rb - l, oracle.ORDER_INTERLEAVED)
    far, nb = (1 << l) - 1, 1 << rb
    for q in range(3 ** (rb - l)):
        ox, oy = int(ux[q]) << l, int(uy[q]) << l
        for lane in range(3 ** l):
            x, y = _coords(lane, l)
            within = sum((lane // 3 ** j % 3 + 1) % 3 * 3 ** j for j in range(l))
            assert place[q * 3 ** l + within] == (ox + x, oy + y)
        for c, at, x, y in (("A", 1, ox, oy), ("B", 2, ox + far, oy), ("C", 0, ox, oy + far)):
            kind, a, b = _neighbour(x, y, nb, c)
            assert _corner_tile_index(q, at, rb - l, l) == (index[a, b] if kind else None)


@pytest.mark.parametrize("s", [4, 5, 6])
def test_cell_tables_of_smaller_tiles(s):
    # element e of a 64-tile's run of 729 -> its cell, for tile sides 16, 32, 64
    rho, cells = 1 << s, []
    for q in range(3 ** (6 - s)):
        x0 = y0 = 0
        for j in range(s, 6):
            d = q // 3 ** (j - s) % 3
            x0 |= (d == 2) << j
            y0 |= (d == 0) << j
        cells += [(x, y) for y in range(y0, y0 + rho) for x in range(x0, x0 + rho) if x & y == 0]
    xs, ys = oracle.compact_cells(6, s, oracle.ORDER_INTERLEAVED)
    assert cells == list(zip(xs.tolist(), ys.tolist()))
