"""The fused CA on words of 32 tiles (csrc/sg_words.cuh) at the sizes where its
dispatch and its packing change: around the levels where it takes over from the
rows of bits, at every unit depth, on buffers that are 16- but not 32-byte
aligned, and in batches whose small gaskets share a word.  Bit for bit against
the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

pytestmark = pytest.mark.gpu


def _state(r, seed, p=0.45):
    return inputs.ca_seed_grid(r, p, seed)


@pytest.mark.parametrize("r,rho,k,order,shift", [
    (11, 16, 8, "interleaved", 0),       # rows of bits
    (11, 16, 9, "interleaved", 0),       # words, units of 9 tiles
    (11, 64, 16, "rowmajor", 16),        # 16-byte stores
    (12, 32, 8, "rowmajor", 0),          # rows of bits on 32-tiles
    (12, 32, 15, "interleaved", 16),
    (13, 64, 2, "interleaved", 0),       # units of 27 tiles
    (13, 16, 15, "rowmajor", 0),
    (13, 32, 16, "interleaved", 16),
])
def test_ca_steps_around_the_dispatch(r, rho, k, order, shift):
    n = 1 << r
    s0 = _state(r, 10 * r + k)
    a = torch.zeros(n * n + 64, dtype=torch.uint8, device="cuda")[shift:shift + n * n]
    b = torch.zeros(n * n + 64, dtype=torch.uint8, device="cuda")[shift:shift + n * n]
    a.copy_(torch.from_numpy(s0.ravel()))
    sg.ca_steps(a, b, r, rho, k, order=order)
    assert np.array_equal(b.cpu().numpy().reshape(n, n), oracle.ca_steps(r, s0, k))
    assert np.array_equal(a.cpu().numpy().reshape(n, n), s0)


@pytest.mark.parametrize("rho,levels", [
    # levels 4 and 5 fill part of a tile; more than 32 gaskets in one window
    (16, [4] * 40 + [5, 12, 4, 6, 5, 7, 9, 8, 6, 10]),
    (32, [5] * 9 + [13, 6, 8, 7, 5, 9, 6, 11]),
    (64, [6] * 35 + [8, 9, 7, 6, 8, 10, 11, 6, 12]),
])
@pytest.mark.parametrize("k", [3, 16])
def test_batch_packs_small_gaskets(rho, levels, k):
    host = [_state(r, 100 + i) for i, r in enumerate(levels)]
    a = [torch.from_numpy(h.ravel()).cuda() for h in host]
    b = [torch.zeros_like(t) for t in a]
    batch = sg.CABatch(levels, a, b, rho=rho)
    batch.steps(k, 0)
    for i, r in enumerate(levels):
        n = 1 << r
        want = oracle.ca_steps(r, host[i], k)
        assert np.array_equal(b[i].cpu().numpy().reshape(n, n), want), (i, r)


@pytest.mark.parametrize("rho,levels,k", [
    (16, [12], 2), (16, [10] * 6, 4), (16, [9, 10, 10], 11), (16, [8] * 18, 11), (16, [8] * 19, 9),
    (32, [11] * 6, 4), (32, [8, 9, 10, 11] * 3, 8), (32, [8, 9, 10, 11] * 3 + [9], 8),
    (32, [9, 10, 10], 11), (32, [8] * 19, 9), (32, [9], 12),
])
def test_batch_around_the_dispatch(rho, levels, k):
    host = [_state(r, 700 + i) for i, r in enumerate(levels)]
    a = [torch.from_numpy(h.ravel()).cuda() for h in host]
    b = [torch.zeros_like(t) for t in a]
    sg.CABatch(levels, a, b, rho=rho).steps(k, 0)
    for i, r in enumerate(levels):
        n = 1 << r
        assert np.array_equal(b[i].cpu().numpy().reshape(n, n),
                              oracle.ca_steps(r, host[i], k)), (i, r)


def test_scheduler_mixes_step_counts_in_a_word():
    # gaskets that share a word, each with its own step count per iteration
    levels = [6, 7, 6, 8, 9, 6, 7, 10, 6, 8]
    host = [_state(r, 300 + i) for i, r in enumerate(levels)]
    bufs = [(torch.from_numpy(h.ravel()).cuda(), torch.zeros(h.size, dtype=torch.uint8, device="cuda"))
            for h in host]
    sched = sg.Sched(levels, 64, 16)
    for i, (x, y) in enumerate(bufs):
        sched.set_buffers(i, x.data_ptr(), y.data_ptr())
    steps = [9, 16, 1, 12, 10, 14, 11, 15, 23, 13]
    sched.submit(list(range(len(levels))), list(range(len(levels))), steps)
    stream = torch.cuda.current_stream()
    while sched.step(stream).iteration:
        pass
    torch.cuda.synchronize()
    for i, (x, y) in enumerate(bufs):
        n = 1 << levels[i]
        cur = x if sched.gasket(i).cur == x.data_ptr() else y
        assert np.array_equal(cur.cpu().numpy().reshape(n, n),
                              oracle.ca_steps(levels[i], host[i], steps[i])), i
    sched.close()


@pytest.mark.parametrize("r,k,order,shift_in,shift_out", [
    (6, 1, "interleaved", 0, 0), (6, 16, "interleaved", 5, 11), (7, 3, "rowmajor", 15, 0),
    (8, 16, "rowmajor", 0, 1), (9, 2, "interleaved", 1, 15), (10, 16, "interleaved", 3, 8),
    (12, 16, "rowmajor", 0, 0), (13, 7, "interleaved", 0, 4),
])
def test_compact_steps_at_any_alignment(r, k, order, shift_in, shift_out):
    n, c = 1 << r, 3 ** r
    oid = {"rowmajor": oracle.ORDER_ROWMAJOR, "interleaved": oracle.ORDER_INTERLEAVED}[order]
    s0 = _state(r, 50 + r)
    src = torch.full((c + 64,), 1, dtype=torch.uint8, device="cuda")
    dst = torch.full((c + 64,), 7, dtype=torch.uint8, device="cuda")
    a, b = src[shift_in:shift_in + c], dst[shift_out:shift_out + c]
    a.copy_(torch.from_numpy(oracle.compact_pack(r, 6, s0, oid)))
    sg.compact_ca_steps(a, b, r, 64, k, order=order)
    want = oracle.compact_pack(r, 6, oracle.ca_steps(r, s0, k), oid)
    got = dst.cpu().numpy()
    assert np.array_equal(got[shift_out:shift_out + c], want)
    assert (got[:shift_out] == 7).all() and (got[shift_out + c:] == 7).all()


def test_single_steps_on_words_match_the_general_path():
    # level 14 is the smallest a single step takes on words (embedded, compact
    # and batched); the bounding-box map runs the general tile kernel
    r = 14
    n = 1 << r
    idx, val = inputs.ca_seed_sparse(r, 0.4, 5)
    a = torch.zeros(n * n, dtype=torch.uint8, device="cuda")
    a[torch.from_numpy(idx).cuda()] = torch.from_numpy(val).cuda()
    want, got = torch.zeros_like(a), torch.zeros_like(a)
    sg.ca_step(a, want, r, 64, "bbox")
    for rho in (4, 64):
        got.zero_()
        sg.ca_step(a, got, r, rho)
        assert torch.equal(got, want)
    c, d, e = (torch.zeros(3 ** r, dtype=torch.uint8, device="cuda") for _ in range(3))
    sg.compact_pack(a, c, r, 64)
    sg.compact_ca_step(c, d, r, 64)
    sg.compact_pack(want, e, r, 64)
    assert torch.equal(d, e)
    small = torch.from_numpy(_state(7, 1).ravel()).cuda()
    sa, sb = [small, a], [torch.zeros_like(small), torch.zeros_like(a)]
    sg.CABatch([7, r], sa, sb, rho=32).step(0)
    assert torch.equal(sb[1], want)
    assert np.array_equal(sb[0].cpu().numpy().reshape(128, 128), oracle.ca_steps(7, _state(7, 1), 1))


@pytest.mark.parametrize("r", [6, 9, 10, 12, 13])
@pytest.mark.parametrize("rho", [1, 8, 16, 64])
def test_single_step_kernel_is_picked_by_level(r, rho):
    n = 1 << r
    a = torch.from_numpy(_state(r, r).ravel()).cuda()
    want, got = torch.zeros_like(a), torch.zeros_like(a)
    sg.ca_step(a, want, r, 16, "bbox")
    sg.ca_step(a, got, r, rho)
    assert torch.equal(got, want)


@pytest.mark.parametrize("r,rho,shift_in,shift_out", [
    (6, 16, 0, 3), (7, 32, 9, 0), (9, 16, 1, 15), (10, 32, 0, 0), (12, 16, 5, 2), (13, 32, 0, 8),
])
def test_compact_step_on_smaller_tiles(r, rho, shift_in, shift_out):
    c = 3 ** r
    s = rho.bit_length() - 1
    s0 = _state(r, 70 + r)
    src = torch.full((c + 64,), 1, dtype=torch.uint8, device="cuda")
    dst = torch.full((c + 64,), 7, dtype=torch.uint8, device="cuda")
    a, b = src[shift_in:shift_in + c], dst[shift_out:shift_out + c]
    a.copy_(torch.from_numpy(oracle.compact_pack(r, s, s0)))
    sg.compact_ca_step(a, b, r, rho)
    got = dst.cpu().numpy()
    assert np.array_equal(got[shift_out:shift_out + c],
                          oracle.compact_pack(r, s, oracle.ca_steps(r, s0, 1)))
    assert (got[:shift_out] == 7).all() and (got[shift_out + c:] == 7).all()
