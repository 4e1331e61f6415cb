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
