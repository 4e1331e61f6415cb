"""Which buffers a scheduler holds share memory (csrc/sg_spans.h), against a
search over all pairs."""
import os
import random
import shutil
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(__file__), "host_src", "spans.cpp")


def test_spans_refuse_what_meets_a_held_range(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "spans"
    subprocess.run([gxx, "-std=c++17", "-O1", SRC, "-o", str(exe)], check=True)
    rng = random.Random(7)
    top = 2 ** 64 - 2 ** 33                      # ranges up to the end of the address space
    held, lines, want = {}, [], []
    for _ in range(4000):
        if held and rng.random() < 0.4:
            start = rng.choice(list(held))
            del held[start]
            lines.append(f"- {start}")
            continue
        start = 16 * rng.randrange(1, 400) + rng.choice((0, top))
        size = 1 << rng.randrange(4, 11) if rng.random() < 0.98 else 1 << 32
        meets = any(start < s + n and s < start + size for s, n in held.items())
        lines.append(f"+ {start} {size}")
        want.append(0 if meets else 1)
        if not meets:
            held[start] = size
    out = subprocess.run([str(exe)], input="\n".join(lines), capture_output=True, text=True,
                         check=True).stdout.split()
    assert [int(v) for v in out] == want
    assert 0 < sum(want) < len(want)
