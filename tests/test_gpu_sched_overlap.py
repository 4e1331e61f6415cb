"""The launches of one scheduler iteration may overlap on the device
(csrc/sg_sched.cu).  What follows the iteration on the stream, or on a stream
that waits for it, must follow all of them: a long launch in front of short
ones, every pair of kernels, read right after each call."""
import pytest
import torch

import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

pytestmark = pytest.mark.gpu


def _alone(a, r, steps):
    a, b = a.clone(), torch.zeros_like(a)
    for _ in range(steps):
        sg.ca_step(a, b, r, 16)
        a, b = b, a
    return a


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("rho,levels,steps", [
    # classes: single step, 2..4, 5..8, 9..16; the largest gasket in the first
    (64, [13, 6, 7, 6, 9, 8], [1, 3, 7, 16, 33, 20]),
    (64, [6, 13, 6, 7, 8, 6], [1, 4, 6, 12, 17, 18]),
    (32, [13, 12, 6, 6, 5, 7], [1, 2, 8, 16, 19, 35]),       # warps, words, rows of bits
    (16, [12, 12, 5, 4, 10, 6], [1, 4, 8, 9, 24, 3]),
])
def test_work_after_an_iteration_sees_all_its_launches(rho, levels, steps, own_stream):
    init = [torch.from_numpy(inputs.ca_seed_grid(r, 0.4, 50 + i).ravel()).cuda()
            for i, r in enumerate(levels)]
    bufs = [(a.clone(), torch.zeros_like(a)) for a in init]
    sched = sg.Sched(levels, rho, 16)
    for i, (a, b) in enumerate(bufs):
        sched.set_buffers(i, a.data_ptr(), b.data_ptr())
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    side = torch.cuda.Stream()
    ids = list(range(len(levels)))
    sched.submit(ids, ids, steps)
    snaps = []
    while sched.step(stream).iteration:
        now = [sched.gasket(i) for i in ids]
        cur = [a if now[i].cur == a.data_ptr() else b for i, (a, b) in enumerate(bufs)]
        with torch.cuda.stream(stream):
            here = [c.clone() for c in cur]
        side.wait_stream(stream)
        with torch.cuda.stream(side):
            there = [c.clone() for c in cur]
        stream.wait_stream(side)                 # the next iteration writes what was read
        snaps.append(([int(x.steps_done) for x in now], here, there))
    torch.cuda.synchronize()
    assert snaps[-1][0] == steps
    for done, here, there in snaps:
        for i in ids:
            want = _alone(init[i], levels[i], done[i])
            assert torch.equal(here[i], want) and torch.equal(there[i], want), (i, done[i])
    sched.close()
