"""Diffusion with a warp per 64-tile (csrc/sg_diffuse_tile.cu) against the general
tile kernels (the bounding-box map's) step by step, bit for bit: every step
count, both orders, tile sides on both sides of its dispatch, grids aligned to
16 bytes only, several tiles per warp, and non-finite values."""
import pytest
import torch

import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

pytestmark = pytest.mark.gpu


def _buffers(r, shift, field):
    n = 1 << (2 * r)
    bufs = [torch.zeros(n + 16, device="cuda")[shift:shift + n] for _ in range(4)]
    bufs[0].copy_(field)
    return bufs


def _check(r, rho, k, order, shift, field, ctas=None, alpha=0.2):
    a, b, x, y = _buffers(r, shift, field)
    sg.diffuse_steps(a, b, r, rho, k, alpha, order=order, ctas_per_sm=ctas)
    x.copy_(a)
    for _ in range(k):
        sg.diffuse_step(x, y, r, 32, alpha, "bbox")
        x, y = y, x
    assert torch.equal(b.view(torch.int32), x.view(torch.int32))
    assert torch.equal(a.view(torch.int32), field.view(torch.int32))


@pytest.mark.parametrize("r,rho,k,order,shift,ctas", [
    (6, 64, 1, "interleaved", 0, None), (6, 32, 8, "rowmajor", 4, None),
    (7, 64, 3, "rowmajor", 0, None), (8, 16, 4, "interleaved", 0, None),
    (8, 16, 5, "interleaved", 4, None), (9, 64, 8, "interleaved", 0, None),
    (10, 16, 1, "rowmajor", 0, None), (10, 4 * 8, 7, "interleaved", 4, None),
    (11, 16, 1, "interleaved", 0, None), (12, 32, 8, "rowmajor", 0, 1),
    (13, 64, 2, "interleaved", 4, 1),
])
def test_steps_match_the_general_path(r, rho, k, order, shift, ctas):
    field = torch.from_numpy(inputs.uniform_grid(r, 3 * r + k).ravel()).cuda()
    _check(r, rho, k, order, shift, field, ctas)


@pytest.mark.parametrize("rho", [1, 2, 4, 8])
def test_single_step_at_any_tile_side(rho):
    r = 8
    field = torch.from_numpy(inputs.uniform_grid(r, 2).ravel()).cuda()
    want, got = torch.zeros_like(field), torch.zeros_like(field)
    sg.diffuse_step(field, want, r, 32, 0.25, "bbox")
    sg.diffuse_step(field, got, r, rho, 0.25)
    assert torch.equal(want.view(torch.int32), got.view(torch.int32))


def test_signed_zeros_and_infinities():
    r = 8
    idx, val = inputs.uniform_sparse(r, 4)
    v = torch.from_numpy(val) - 0.5
    v[::7] = -0.0
    field = torch.zeros(1 << (2 * r))
    field[torch.from_numpy(idx)] = v
    _check(r, 64, 8, "interleaved", 0, field.cuda())
    v[5], v[3000] = float("inf"), float("-inf")
    field[torch.from_numpy(idx)] = v
    a, b, x, y = _buffers(r, 0, field.cuda())
    sg.diffuse_steps(a, b, r, 64, 6, 0.2)
    x.copy_(a)
    for _ in range(6):
        sg.diffuse_step(x, y, r, 32, 0.2, "bbox")
        x, y = y, x
    assert torch.equal(torch.nan_to_num(b, 7.0), torch.nan_to_num(x, 7.0))
