"""Both sides of the lines at which a step changes kernels, in both walking
orders and on buffers that are 16- but not 32-byte aligned: bit for bit the
general path (the bounding box, a batch's gaskets alone) or the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

pytestmark = pytest.mark.gpu


def _board(r, seed, shift=0):
    """A random state of level r, `shift` bytes past a 512-byte boundary."""
    n2 = 1 << (2 * r)
    a = torch.zeros(n2 + shift, dtype=torch.uint8, device="cuda")[shift:]
    idx, val = inputs.ca_seed_sparse(r, 0.4, seed)
    a[torch.from_numpy(idx).cuda()] = torch.from_numpy(val).cuda()
    return a


@pytest.mark.parametrize("r", [13, 14, 15])
def test_one_ca_step_by_level_and_order(r):
    for shift in (0, 16):
        a = _board(r, r, shift)
        want, got = torch.zeros_like(a), torch.zeros(a.numel() + shift, dtype=torch.uint8,
                                                     device="cuda")[shift:]
        sg.ca_step(a, want, r, 64, "bbox")
        for rho in (16, 64):
            for order in ("interleaved", "rowmajor"):
                got.zero_()
                sg.ca_step(a, got, r, rho, order=order)
                assert torch.equal(got, want), (shift, rho, order)


@pytest.mark.parametrize("levels", [
    # cells in units of 3^14: small gaskets, below and from 1.0 on; levels 9 and
    # 10 alone, 1.0; mixed with smaller ones, below and from 9.0 on
    [8] * 728, [8] * 729, [9, 10] * 62, [10, 8] * 100, [10, 8] * 657,
    # above level 10, below and from 3.0 on
    [13, 13, 12, 9, 7], [13] * 8 + [12, 6, 12, 12],
])
def test_one_step_of_a_batch_by_cells_and_levels(levels):
    boards = {r: [_board(r, 31 * r + i) for i in range(2)] for r in set(levels)}
    want = {}
    for r, some in boards.items():
        for i, a in enumerate(some):
            want[r, i] = torch.zeros_like(a)
            sg.ca_step(a, want[r, i], r, 16, "bbox")
    pick = [i % 2 for i in range(len(levels))]
    a = [boards[r][i].clone() for r, i in zip(levels, pick)]
    for order in ("interleaved", "rowmajor"):
        b = [torch.zeros_like(t) for t in a]
        sg.CABatch(levels, a, b, rho=64).step(0, order=order)
        for j, (r, i) in enumerate(zip(levels, pick)):
            assert torch.equal(b[j], want[r, i]), (j, r, order)


@pytest.mark.parametrize("r,rho", [(7, 8), (8, 8), (9, 8), (10, 8), (10, 16), (11, 16), (12, 16)])
def test_one_diffusion_step_by_level_and_tile_side(r, rho):
    # every kernel updates a cell with the same operations in the same order
    n2 = 1 << (2 * r)
    idx, val = inputs.uniform_sparse(r, 3 * r)
    for shift in (0, 4):                         # floats: 16 bytes
        a, want, got = (torch.zeros(n2 + shift, device="cuda")[shift:] for _ in range(3))
        a[torch.from_numpy(idx).cuda()] = torch.from_numpy(val).cuda()
        sg.diffuse_step(a, want, r, 64, 0.2, "bbox")
        for order in ("interleaved", "rowmajor"):
            got.zero_()
            sg.diffuse_step(a, got, r, rho, 0.2, order=order)
            assert torch.equal(got, want), (shift, order)


@pytest.mark.parametrize("r,rho,k,order,shift", [
    (10, 16, 16, "interleaved", 0),          # rows of bits on 16-tiles
    (10, 64, 16, "rowmajor", 16),
    (11, 32, 8, "interleaved", 16),          # the last of them
    (11, 32, 9, "rowmajor", 0),              # words
    (12, 16, 4, "interleaved", 0),           # rows of bits on 32-tiles
    (12, 64, 4, "rowmajor", 16),
    (12, 32, 3, "interleaved", 0),
    (12, 16, 5, "rowmajor", 0),              # words
    (12, 32, 5, "interleaved", 16),
])
def test_ca_steps_by_level_and_count(r, rho, k, order, shift):
    n = 1 << r
    s0 = inputs.ca_seed_grid(r, 0.45, 20 * r + k)
    a, b = (torch.zeros(n * n + shift, dtype=torch.uint8, device="cuda")[shift:] for _ in range(2))
    a.copy_(torch.from_numpy(s0.ravel()))
    sg.ca_steps(a, b, r, rho, k, order=order)
    assert np.array_equal(b.cpu().numpy().reshape(n, n), oracle.ca_steps(r, s0, k))


@pytest.mark.parametrize("rho", [16, 32, 64])
@pytest.mark.parametrize("levels", [
    [12, 12, 11, 9, 10, 12],                 # 3^13 cells and more, none below level 9
    [12, 11, 9, 10, 9],                      # fewer
    [12, 12, 12, 6, 8],                      # as many, with small ones
])
def test_batch_units_with_and_without_small_gaskets(levels, rho):
    host = [inputs.ca_seed_grid(r, 0.4, 900 + i) for i, r in enumerate(levels)]
    a = [torch.from_numpy(h.ravel()).cuda() for h in host]
    for k, order in ((13, "interleaved"), (16, "rowmajor")):
        b = [torch.zeros_like(t) for t in a]
        sg.CABatch(levels, a, b, rho=rho).steps(k, 0, order=order)
        for i, r in enumerate(levels):
            n = 1 << r
            assert np.array_equal(b[i].cpu().numpy().reshape(n, n),
                                  oracle.ca_steps(r, host[i], k)), (i, r, k)


@pytest.mark.parametrize("rho,levels,k", [
    # a CTA an SM is 1216 tiles on 152 SMs: the last batch on rows of bits at each
    # number of steps, and the first on words
    (16, [8] * 90, 2), (16, [8] * 91, 2), (16, [8] * 75, 4), (16, [8] * 76, 3),
    (16, [8] * 45, 8), (16, [9] * 15 + [6], 5), (16, [8] * 15, 9), (16, [8] * 16, 11),
    (16, [9] * 10, 10), (16, [9] * 10 + [7], 9), (16, [8] * 15, 16), (16, [8, 8, 9, 9, 9, 9, 4], 12),
    (32, [10] * 30, 2), (32, [10] * 31, 2), (32, [10] * 20, 4), (32, [10] * 20 + [5], 4),
    (32, [10] * 15, 6), (32, [10] * 15 + [6], 5), (32, [10] * 10, 8), (32, [10] * 10 + [7], 7),
    (32, [10] * 5, 9), (32, [10] * 5 + [5], 11), (32, [8] * 3, 10), (32, [9, 6], 12),
])
def test_batch_steps_by_tiles_and_count(rho, levels, k):
    boards = {r: [_board(r, 17 * r + i) for i in range(2)] for r in set(levels)}
    want = {}
    for r, some in boards.items():
        for i, a in enumerate(some):
            want[r, i] = torch.zeros_like(a)
            if r > 4:
                sg.ca_steps(a, want[r, i], r, 16, k, "bbox")
            else:
                s0 = a.cpu().numpy().reshape(1 << r, 1 << r)
                want[r, i].copy_(torch.from_numpy(oracle.ca_steps(r, s0, k).ravel()))
    pick = [i % 2 for i in range(len(levels))]
    a = [boards[r][i].clone() for r, i in zip(levels, pick)]
    for order in ("interleaved", "rowmajor"):
        b = [torch.zeros_like(t) for t in a]
        sg.CABatch(levels, a, b, rho=rho).steps(k, 0, order=order)
        for j, (r, i) in enumerate(zip(levels, pick)):
            assert torch.equal(b[j], want[r, i]), (j, r, order)


@pytest.mark.parametrize("dtype,r,rho", [
    (torch.uint8, 13, 64), (torch.uint8, 14, 32), (torch.float32, 10, 16), (torch.float32, 11, 64),
    (torch.float32, 12, 32), (torch.float32, 12, 16),
])
@pytest.mark.parametrize("store", ["merge", "masked", "sector"])
def test_grids_in_host_memory_by_size(dtype, r, rho, store):
    # row groups apart or whole units; the device grid takes the first at these sizes
    n2 = 1 << (2 * r)
    if store == "sector":
        start = torch.zeros(n2, dtype=dtype)
    elif dtype == torch.uint8:
        start = torch.arange(n2, dtype=torch.int32).remainder_(251).to(dtype)
    else:
        start = torch.arange(n2, dtype=torch.float32).remainder_(1009.0)
    host = start.clone().pin_memory()
    sg.map_write_mapped(host, r, rho, "lambda", "hash", 5, store=store)
    dev = start.cuda()
    sg.map_write(dev, r, rho, "lambda", "hash", 5, store="scatter")
    torch.cuda.synchronize()
    assert torch.equal(host, dev.cpu())
