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
