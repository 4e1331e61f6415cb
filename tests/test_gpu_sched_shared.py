"""Gaskets of a scheduler that share memory: their launches run one behind the
other, the shorter advances' class first (include/sg_sched.h)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho,r", [(64, 11), (32, 9), (16, 6)])
def test_a_gasket_steps_what_another_has_written(rho, r):
    n = 1 << r
    s0 = inputs.ca_seed_grid(r, 0.4, r)
    a = torch.from_numpy(s0.ravel()).cuda()
    b, c, d = (torch.zeros_like(a) for _ in range(3))
    sched = sg.Sched([r, r, r], rho, 16)
    sched.set_buffers(0, a.data_ptr(), b.data_ptr())
    sched.set_buffers(1, b.data_ptr(), c.data_ptr())      # reads what 0 writes
    sched.set_buffers(2, c.data_ptr(), d.data_ptr())      # reads what 1 writes
    sched.submit([0, 1, 2], [0, 1, 2], [1, 4, 16])
    res = sched.step(torch.cuda.current_stream())
    assert res.launches == 3
    for got, k in ((b, 1), (c, 5), (d, 21)):
        assert np.array_equal(got.cpu().numpy().reshape(n, n), oracle.ca_steps(r, s0, k)), k
    # buffers of their own again: stepped beside one another, each on its own
    own = [(a.clone(), torch.zeros_like(a)) for _ in range(3)]
    for i, (x, y) in enumerate(own):
        sched.set_buffers(i, x.data_ptr(), y.data_ptr())
    sched.submit([0, 1, 2], [3, 4, 5], [1, 4, 16])
    sched.step(torch.cuda.current_stream())
    for (_, y), k in zip(own, (1, 4, 16)):
        assert np.array_equal(y.cpu().numpy().reshape(n, n), oracle.ca_steps(r, s0, k)), k
    sched.close()
