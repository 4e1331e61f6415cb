"""The compact diffusion step on triples (csrc/sg_compact_stencil.cu): partial
units, several units per CTA, both walking orders and arrays at any 4-byte
address, against the embedded step, bit for bit."""
import numpy as np
import pytest
import torch

import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,rho,order,shift,ctas", [
    (4, 16, "interleaved", 0, None), (5, 16, "rowmajor", 1, None), (5, 32, "interleaved", 3, None),
    (6, 64, "interleaved", 1, None), (7, 16, "rowmajor", 0, None), (8, 32, "rowmajor", 2, None),
    (9, 64, "rowmajor", 0, None), (12, 16, "interleaved", 1, 1), (12, 64, "rowmajor", 3, 1),
    (13, 32, "interleaved", 0, 2),
])
def test_triples_match_the_embedded_step(r, rho, order, shift, ctas):
    n, c = 1 << r, 3 ** r
    g = torch.from_numpy(inputs.uniform_grid(r, r).ravel()).cuda()
    want_grid = torch.zeros_like(g)
    sg.diffuse_step(g, want_grid, r, 4 if r > 4 else 2, 0.2)
    src = torch.full((c + 8,), 9.0, device="cuda")
    dst = torch.full((c + 8,), 9.0, device="cuda")
    a, b = src[shift:shift + c], dst[shift:shift + c]
    want = torch.empty(c, device="cuda")
    sg.compact_pack(g, a, r, rho, order=order)
    sg.compact_pack(want_grid, want, r, rho, order=order)
    sg.compact_diffuse_step(a, b, r, rho, 0.2, order=order, ctas_per_sm=ctas)
    assert torch.equal(b, want)
    assert bool((dst[:shift] == 9.0).all()) and bool((dst[shift + c:] == 9.0).all())
