"""The work a user of this package has it do, as cases that can be measured.

Every case goes through the package's tensor functions (``map_write``,
``ca_step`` / ``ca_steps``, ``diffuse_step`` / ``diffuse_steps``, the
``compact_*`` forms, ``CABatch`` and ``Sched``).  Levels, tile sides, values
and step counts are those of ``workloads`` and of ``serve.ServeConfig``; the
drawn cases spread over the levels between them.

Bytes counted in ``work``: on an embedded grid the 32-byte sectors that hold
gasket cells (the smallest piece of memory that can be read or written), on a
compact array its 3^r elements; each input once, each output once.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_1706_04552_gb300 as sg
from paper_1706_04552_gb300 import inputs

DEV = "cuda"


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The paper's experiment at its largest size, and the headline of the
        # benchmark: write v(x, y) into the gasket of a zero 65536 x 65536 matrix.
        dict(name="write_u8_r16_fill", op="write", r=16, dtype="u8", rho=64,
             map="lambda_unroll", store="fill"),
        # A small float grid that already holds other data off the gasket, with
        # the library's own choice of stores: a call that latency decides.
        dict(name="write_f32_r11", op="write", r=11, dtype="f32", rho=16, map="lambda",
             store="auto"),
        # The same write for a program that keeps only the gasket's cells.
        dict(name="compact_write_u8_r16", op="compact_write", r=16, dtype="u8", rho=64),
        # One generation of the automaton on a large board: an interactive
        # simulation that looks at each generation.
        dict(name="ca_step_r15", op="ca", r=15, rho=64, k=1),
        # The small end-to-end workload's board, 16 generations a call.
        dict(name="ca_steps_r10_k16", op="ca", r=10, rho=16, k=16),
        # A long run on a large board, 16 generations a call.
        dict(name="ca_steps_r15_k16", op="ca", r=15, rho=64, k=16),
        # One diffusion step of a medium field (a solver that couples every step).
        dict(name="diffuse_step_r14", op="diffuse", r=14, rho=32, k=1),
        # A long diffusion run on a large field, 8 steps a call.
        dict(name="diffuse_steps_r15_k8", op="diffuse", r=15, rho=32, k=8),
        # The long CA run of a program that keeps only the gasket's cells.
        dict(name="compact_ca_r15_k16", op="compact_ca", r=15, rho=64, k=16),
        # A diffusion step on a compact field.
        dict(name="compact_diffuse_r15", op="compact_diffuse", r=15, rho=64),
        # Many boards of uneven levels stepped together, 16 generations a launch.
        dict(name="batch_32_k16", op="batch", count=32, lo=8, hi=14, level_seed=2, rho=64, k=16),
        # The serving core: a burst of requests of 1..32 generations on small
        # resident boards, served until none is left.
        dict(name="serve_48", op="serve", count=48, lo=6, hi=11, level_seed=3, rho=64, fuse=16,
             requests=96),
    ]


def draw(rng):
    op = rng.choice(("write", "write", "compact_write", "ca", "ca", "diffuse", "diffuse",
                     "compact_ca", "compact_diffuse", "batch", "serve"))
    if op == "write":
        dtype = rng.choice(("u8", "f32"))
        rho = rng.choice((8, 16, 32, 64))
        stores = ["auto"]
        if rho * (1 if dtype == "u8" else 4) >= 16:
            stores.append("fill")
        return dict(op=op, r=rng.randint(8, 15 if dtype == "u8" else 14), dtype=dtype, rho=rho,
                    map=rng.choice(("lambda", "lambda_unroll", "lambda_lut")),
                    store=rng.choice(stores))
    if op == "compact_write":
        dtype = rng.choice(("u8", "f32"))
        return dict(op=op, r=rng.randint(8, 16 if dtype == "u8" else 15), dtype=dtype,
                    rho=rng.choice((16, 32, 64)))
    if op == "ca":
        return dict(op=op, r=rng.randint(6, 15), rho=rng.choice((16, 32, 64)),
                    k=rng.randint(1, 16))
    if op == "diffuse":
        return dict(op=op, r=rng.randint(6, 14), rho=rng.choice((16, 32, 64)), k=rng.randint(1, 8))
    if op == "compact_ca":
        k = rng.randint(1, 16)
        return dict(op=op, r=rng.randint(6, 15), rho=64 if k > 1 else rng.choice((16, 32, 64)), k=k)
    if op == "compact_diffuse":
        return dict(op=op, r=rng.randint(6, 14), rho=rng.choice((16, 32, 64)))
    if op == "batch":
        lo = rng.randint(6, 9)
        return dict(op=op, count=rng.randint(3, 32), lo=lo, hi=rng.randint(lo + 1, 13),
                    level_seed=rng.randint(0, 999), rho=rng.choice((16, 32, 64)),
                    k=rng.randint(1, 16))
    return dict(op="serve", count=rng.randint(5, 48), lo=6, hi=rng.randint(8, 11),
                level_seed=rng.randint(0, 999), rho=64, fuse=rng.choice((4, 8, 16)),
                requests=rng.randint(16, 96))


# ------------------------------------------------------------------- inputs

def _cells(r):
    """Flat row-major indices of the 3^r gasket cells, on the GPU."""
    x = torch.zeros(1, dtype=torch.int64, device=DEV)
    y = torch.zeros(1, dtype=torch.int64, device=DEV)
    for j in range(r):
        h = 1 << j
        x, y = torch.cat([x, x + h, x]), torch.cat([y, y, y + h])
    return (y << r) | x


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _ca_values(n, g, p=0.3):
    return (torch.rand(n, generator=g, device=DEV) < p).to(torch.uint8)


def _ca_state(r, g):
    s = torch.zeros(1 << (2 * r), dtype=torch.uint8, device=DEV)
    s[_cells(r)] = _ca_values(3 ** r, g)
    return s


def _field(r, g):
    s = torch.zeros(1 << (2 * r), dtype=torch.float32, device=DEV)
    s[_cells(r)] = torch.rand(3 ** r, generator=g, device=DEV)
    return s


def _levels(case):
    return inputs.batch_levels(case["count"], case["lo"], case["hi"], case["level_seed"])


def _requests(case):
    """(gasket, steps) of each request: uniform gaskets, 1..32 steps."""
    rng = np.random.default_rng(case["level_seed"] + 1)
    n = case["requests"]
    return (rng.integers(0, case["count"], n).astype(np.int32),
            rng.integers(1, 33, n).astype(np.int32))


def prepare(case, seed):
    op, g = case["op"], _gen(seed)
    st = dict(case, seed=int(seed))
    if op == "write":
        n = 1 << (2 * case["r"])
        dt = torch.uint8 if case["dtype"] == "u8" else torch.float32
        if case["store"] == "fill":           # a zero matrix, as the paper writes into
            st["grid"] = torch.zeros(n, dtype=dt, device=DEV)
        elif case["dtype"] == "u8":
            st["grid"] = torch.randint(0, 256, (n,), dtype=dt, device=DEV, generator=g)
        else:
            st["grid"] = torch.rand(n, dtype=dt, device=DEV, generator=g)
    elif op == "compact_write":
        dt = torch.uint8 if case["dtype"] == "u8" else torch.float32
        st["out"] = torch.zeros(3 ** case["r"], dtype=dt, device=DEV)
    elif op == "ca":
        st["inp"] = _ca_state(case["r"], g)
        st["out"] = torch.zeros_like(st["inp"])
    elif op == "diffuse":
        st["inp"] = _field(case["r"], g)
        st["out"] = torch.zeros_like(st["inp"])
    elif op == "compact_ca":
        st["inp"] = _ca_values(3 ** case["r"], g)
        st["out"] = torch.zeros_like(st["inp"])
    elif op == "compact_diffuse":
        st["inp"] = torch.rand(3 ** case["r"], generator=g, device=DEV)
        st["out"] = torch.zeros_like(st["inp"])
    elif op == "batch":
        levels = _levels(case)
        st["a"] = [_ca_state(r, g) for r in levels]
        st["b"] = [torch.zeros_like(a) for a in st["a"]]
        st["batch"] = sg.CABatch(levels, st["a"], st["b"], rho=case["rho"])
    elif op == "serve":
        levels = _levels(case)
        st["bufs"] = [(_ca_state(r, g), torch.zeros(1 << (2 * r), dtype=torch.uint8, device=DEV))
                      for r in levels]
        st["sched"] = sg.Sched(levels, case["rho"], case["fuse"])
        for i, (a, b) in enumerate(st["bufs"]):
            st["sched"].set_buffers(i, a.data_ptr(), b.data_ptr())
        st["gaskets"], st["steps"] = _requests(case)
        st["ids"] = np.arange(case["requests"], dtype=np.int64)
    else:
        raise ValueError(op)
    return st


# ------------------------------------------------------------------ one pass

def run(st):
    op = st["op"]
    if op == "write":
        return sg.map_write(st["grid"], st["r"], st["rho"], st["map"], "hash", st["seed"],
                            store=None if st["store"] == "auto" else st["store"])
    if op == "compact_write":
        return sg.compact_map_write(st["out"], st["r"], st["rho"], "hash", st["seed"])
    if op == "ca":
        if st["k"] == 1:
            return sg.ca_step(st["inp"], st["out"], st["r"], st["rho"])
        return sg.ca_steps(st["inp"], st["out"], st["r"], st["rho"], st["k"])
    if op == "diffuse":
        if st["k"] == 1:
            return sg.diffuse_step(st["inp"], st["out"], st["r"], st["rho"], 0.2)
        return sg.diffuse_steps(st["inp"], st["out"], st["r"], st["rho"], st["k"], 0.2)
    if op == "compact_ca":
        if st["k"] == 1:
            return sg.compact_ca_step(st["inp"], st["out"], st["r"], st["rho"])
        return sg.compact_ca_steps(st["inp"], st["out"], st["r"], st["rho"], st["k"])
    if op == "compact_diffuse":
        return sg.compact_diffuse_step(st["inp"], st["out"], st["r"], st["rho"], 0.2)
    if op == "batch":
        if st["k"] == 1:
            st["batch"].step(0)
        else:
            st["batch"].steps(st["k"], 0)
        return st["b"]
    sched, stream = st["sched"], torch.cuda.current_stream()
    sched.submit(st["gaskets"], st["ids"], st["steps"])
    while sched.step(stream).iteration:
        pass
    return [a if sched.gasket(i).cur == a.data_ptr() else b
            for i, (a, b) in enumerate(st["bufs"])]


# ---------------------------------------------------------- what it cannot avoid

def _sector_bytes(r, elem):
    """Bytes of the 32-byte sectors of a level-r grid that hold gasket cells: a
    sector of 2^g elements at column x on row y does iff (x >> g) & (y >> g) == 0."""
    if r == 0:
        return 32
    g = min(r, 5 if elem == 1 else 3)
    return (1 << g) * 3 ** (r - g) * (elem << g)


def work(case):
    op = case["op"]
    elem = 1 if case.get("dtype") == "u8" or op in ("ca", "compact_ca", "batch", "serve") else 4
    if op == "write":
        touched = _sector_bytes(case["r"], elem)
        return {"bytes": touched * (1 if case["store"] == "fill" else 2), "flops": 0}
    if op == "compact_write":
        return {"bytes": elem * 3 ** case["r"], "flops": 0}
    if op == "ca":
        return {"bytes": 2 * _sector_bytes(case["r"], 1), "flops": 0}
    if op == "diffuse":
        # about 4 additions, a multiplication and a fused multiply-add a cell and step
        return {"bytes": 2 * _sector_bytes(case["r"], 4), "flops": 7 * case["k"] * 3 ** case["r"]}
    if op == "compact_ca":
        return {"bytes": 2 * 3 ** case["r"], "flops": 0}
    if op == "compact_diffuse":
        return {"bytes": 8 * 3 ** case["r"], "flops": 7 * 3 ** case["r"]}
    levels = _levels(case)
    if op == "serve":
        levels = [levels[i] for i in sorted(set(_requests(case)[0].tolist()))]
    return {"bytes": sum(2 * _sector_bytes(r, 1) for r in levels), "flops": 0}


# ------------------------------------------------------------- in 64 bits

def _hash01(key, seed):
    """(h >> 40) * 2^-24 of the SplitMix64 output for (seed * gamma) ^ key, in
    64-bit integers (shifts of negative values masked to logical ones)."""
    def i64(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >> 63 else v

    def shr(z, n):
        return (z >> n) & ((1 << (64 - n)) - 1)

    z = (key ^ i64(seed * 0x9E3779B97F4A7C15)) + i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
    z = z ^ shr(z, 31)
    return shr(z, 40).double() * 2.0 ** -24


def _diffuse64(u, idx, r, k, alpha):
    """k steps on the embedded float64 grid u (0 off the gasket), in place."""
    n = 1 << r
    x, y = idx & (n - 1), idx >> r
    deg = torch.zeros(idx.numel(), dtype=torch.float64, device=DEV)
    near = []
    for dx, dy in ((-1, 0), (1, 0), (0, -1), (0, 1)):
        ok = ((x + dx >= 0) & (x + dx < n) & (y + dy >= 0) & (y + dy < n) &
              (((x + dx) & (y + dy)) == 0))
        deg += ok
        near.append(torch.where(ok, idx + dx + (dy << r if dy > 0 else -(1 << r) if dy else 0),
                                torch.full_like(idx, -1)))
    for _ in range(k):
        v = u[idx]
        s = -deg * v
        for j in near:
            s += torch.where(j >= 0, u[j.clamp(min=0)], torch.zeros_like(s))
        u[idx] = v + alpha * s
    return u


def _compact_index(r, rho):
    """Flat grid index of each element of a compact array (default walking
    order: the digits of the tile's launch index q are the levels' choices,
    finest first, mirrored vertically)."""
    s = rho.bit_length() - 1
    rb = r - s
    q = torch.arange(3 ** rb, dtype=torch.int64, device=DEV)
    bx = torch.zeros_like(q)
    ly = torch.zeros_like(q)
    for j in range(rb):
        d = q // 3 ** j % 3
        bx += (d >> 1) << j
        ly += (d - (d >> 1)) << j
    by = (1 << rb) - 1 - ly
    t = _cells(s).sort().values                       # the tile's cells, row by row
    tx, ty = t & (rho - 1), t >> s
    return ((((by[:, None] << s) + ty) << r) + (bx[:, None] << s) + tx).reshape(-1)


def exact(case, seed):
    op = case["op"]
    if op == "write" and case["dtype"] == "f32":
        st = prepare(case, seed)
        out, idx = st["grid"].double(), _cells(case["r"])
        out[idx] = _hash01(idx, int(seed))
        return out
    if op == "compact_write" and case["dtype"] == "f32":
        return _hash01(_compact_index(case["r"], case["rho"]), int(seed))
    if op == "diffuse":
        u = prepare(case, seed)["inp"].double()
        return _diffuse64(u, _cells(case["r"]), case["r"], case["k"], float(np.float32(0.2)))
    if op == "compact_diffuse":
        v = prepare(case, seed)["inp"].double()
        idx = _compact_index(case["r"], case["rho"])
        u = torch.zeros(1 << (2 * case["r"]), dtype=torch.float64, device=DEV)
        u[idx] = v
        return _diffuse64(u, idx, case["r"], 1, float(np.float32(0.2)))[idx]
    return None                     # bytes: equal or not
