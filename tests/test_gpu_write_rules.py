"""Write passes where their dispatch changes: the compact write four elements at a
time (every alignment, partial units, each value kind), and the sector stores
in row groups (small grids, edges of the rule).  Against the oracle, exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_1706_04552_gb300 as sg

pytestmark = pytest.mark.gpu

KINDS = {"const": oracle.VAL_CONST, "linear31": oracle.VAL_LINEAR31, "hash": oracle.VAL_HASH}


def _embedded(r, kind, seed, dtype):
    g = np.zeros((1 << r, 1 << r), dtype=dtype)
    oracle.map_write(r, g, KINDS[kind], seed)
    return g


@pytest.mark.parametrize("r,rho,dtype,kind,shift,order", [
    (4, 16, "u8", "hash", 0, "interleaved"), (5, 16, "u8", "hash", 3, "rowmajor"),
    (5, 32, "f32", "hash", 1, "interleaved"), (6, 64, "u8", "linear31", 1, "interleaved"),
    (6, 64, "f32", "hash", 2, "rowmajor"), (8, 16, "f32", "linear31", 3, "interleaved"),
    (9, 64, "u8", "hash", 2, "interleaved"), (9, 32, "u8", "const", 5, "rowmajor"),
    (10, 64, "u8", "hash", 7, "rowmajor"), (11, 16, "f32", "hash", 0, "interleaved"),
])
def test_compact_write_at_any_alignment(r, rho, dtype, kind, shift, order):
    dt, nd = (torch.uint8, np.uint8) if dtype == "u8" else (torch.float32, np.float32)
    seed = 5 if dtype == "u8" or kind != "const" else 0x3F800000
    c = 3 ** r
    buf = torch.full((c + 16,), 77, dtype=dt, device="cuda")
    sg.compact_map_write(buf[shift:shift + c], r, rho, kind, seed, order=order)
    oid = {"rowmajor": oracle.ORDER_ROWMAJOR, "interleaved": oracle.ORDER_INTERLEAVED}[order]
    want = oracle.compact_pack(r, rho.bit_length() - 1, _embedded(r, kind, seed, nd), oid)
    got = buf.cpu().numpy()
    assert np.array_equal(got[shift:shift + c], want)
    assert (got[:shift] == 77).all() and (got[shift + c:] == 77).all()


@pytest.mark.parametrize("r,rho,dtype,store,order", [
    (5, 32, "u8", "merge", "interleaved"), (6, 64, "u8", "sector", "rowmajor"),
    (7, 32, "u8", "masked", "rowmajor"), (10, 64, "u8", "merge", "rowmajor"),
    (3, 8, "f32", "merge", "interleaved"), (4, 16, "f32", "sector", "rowmajor"),
    (6, 64, "f32", "masked", "interleaved"), (9, 16, "f32", "merge", "rowmajor"),
    (11, 32, "f32", "merge", "interleaved"), (12, 64, "u8", "merge", "interleaved"),
])
def test_sector_stores_in_row_groups(r, rho, dtype, store, order):
    nd = np.uint8 if dtype == "u8" else np.float32
    n = 1 << r
    rng = np.random.default_rng(r)
    g0 = rng.integers(1, 200, (n, n)).astype(nd)
    if store == "sector":
        g0[:] = 0                                   # write-only: a zero grid
    want = g0.copy()
    oracle.map_write(r, want, oracle.VAL_HASH, 9)
    g = torch.from_numpy(g0.ravel()).cuda()
    sg.map_write(g, r, rho, "lambda", "hash", 9, store=store, order=order)
    assert np.array_equal(g.cpu().numpy().reshape(n, n), want)


def test_sector_stores_agree_on_both_sides_of_the_rule():
    # uint8: row groups up to level 15 (1845 groups of units), whole units at 16
    for r in (15, 16):
        g = torch.zeros(1 << (2 * r), dtype=torch.uint8, device="cuda")
        sg.map_write(g, r, 64, "lambda", "hash", 3, store="merge")
        h = torch.zeros_like(g)
        sg.map_write(h, r, 64, "lambda_unroll", "hash", 3, store="fill")
        assert torch.equal(g, h)
        del g, h
