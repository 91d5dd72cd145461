"""The work that the speed of this library is judged by.

A case is one call pattern of a user's program: a grid (or a batch of grids)
that lives on the GPU, advanced by a few steps through the public entry points.
Sizes, densities and rules are those of the workloads that the tests and the
benchmark use (16384^2 radius sweep, 32768^2 precision variants, the batch of
uneven grids, the multi-state rule R10 C16) or generic ones.  `run` steps the
grid on from where it is, as a simulation loop does, and returns the whole
state.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2406_17284_gb300 import cat, inputs

U8, BIT1, NIB4 = cat.STORE_U8, cat.STORE_BIT1, cat.STORE_NIB4


def listed() -> list[dict]:
    return [
        # the textbook run: 100 generations of Conway's rule on a small board,
        # every launch a latency (options left to the library)
        dict(name="conway_256", kind="single", H=256, W=256, r=1, C=2, M=0, rule="conway", p=0.5, storage=U8,
             boundary=0, kernel="auto", dtype="auto", steps=100),
        # the radius sweep as the benchmark and the Grid class's defaults run it
        # (FP8 operands): a small radius ...
        dict(name="sweep_r4_fp8", kind="single", H=16384, W=16384, r=4, C=2, M=1, rule="scaled", p=0.5, storage=U8,
             boundary=0, kernel="tcgen05", dtype="fp8", steps=1),
        # ... and a large one
        dict(name="sweep_r12_fp8", kind="single", H=16384, W=16384, r=12, C=2, M=1, rule="scaled", p=0.5, storage=U8,
             boundary=0, kernel="tcgen05", dtype="fp8", steps=1),
        # the same sweep in the paper's own precision
        dict(name="sweep_r10_fp16", kind="single", H=16384, W=16384, r=10, C=2, M=1, rule="scaled", p=0.5, storage=U8,
             boundary=0, kernel="tcgen05", dtype="fp16", steps=1),
        # an odd-sized simulation with every option left to the library
        dict(name="ragged_r9", kind="single", H=9001, W=12347, r=9, C=2, M=0, rule="scaled", p=0.5, storage=U8,
             boundary=0, kernel="auto", dtype="auto", steps=1),
        # large packed grids, one bit per cell: a small and the largest radius
        dict(name="bits_r2", kind="single", H=32768, W=32768, r=2, C=2, M=1, rule="scaled", p=0.35, storage=BIT1,
             boundary=0, kernel="auto", dtype="auto", steps=1),
        dict(name="bits_r16", kind="single", H=32768, W=32768, r=16, C=2, M=1, rule="scaled", p=0.35, storage=BIT1,
             boundary=0, kernel="auto", dtype="auto", steps=1),
        # multi-state rule (Generations reading), one byte and four bits per cell
        dict(name="c16_u8", kind="single", H=24576, W=24576, r=10, C=16, M=1, rule="multistate", p=0.65, storage=U8,
             boundary=0, kernel="auto", dtype="auto", steps=1),
        dict(name="c16_nib4", kind="single", H=24576, W=24576, r=10, C=16, M=1, rule="multistate", p=0.65,
             storage=NIB4, boundary=0, kernel="auto", dtype="auto", steps=1),
        # a parameter study: many uneven grids, each with its own radius and
        # rule, on buffers of the caller's allocator, in one call
        dict(name="batch_uneven", kind="batch", count=512, side_lo=64, side_hi=2048, kernel="auto", dtype="auto",
             draw_seed=2024, steps=4),
        # the paper's boundary: a torus
        dict(name="periodic_r6", kind="single", H=8192, W=8192, r=6, C=2, M=1, rule="scaled", p=0.5, storage=U8,
             boundary=1, kernel="auto", dtype="auto", steps=2),
        # a radius beyond the paper's 16
        dict(name="wide_r24", kind="single", H=8192, W=8192, r=24, C=2, M=1, rule="scaled", p=0.5, storage=U8,
             boundary=0, kernel="auto", dtype="auto", steps=2),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["u8", "u8", "fp8", "fp8", "fp16", "bits", "bits", "c16", "batch", "periodic", "wide"])
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 16, 512), side_lo=64, side_hi=rng.choice([512, 1024, 2048]),
                    kernel="auto", dtype="auto", draw_seed=rng.randrange(1 << 30), steps=2 * rng.randint(1, 2))
    # areas from a small board to the benchmark's, sides of every residue
    top = {"bits": 30, "c16": 28, "wide": 27, "periodic": 27}.get(kind, 28)
    area = 2.0 ** rng.uniform(16, top)
    H = max(64, int(round(math.sqrt(area) * 2.0 ** rng.uniform(-1, 1))))
    W = max(64, int(round(area / H)))
    if rng.random() < 0.3:   # sizes that people type
        H, W = max(64, H // 64 * 64), max(64, W // 64 * 64)
    steps = max(1, min(64, int(2.0 ** (top - 2) / (H * W))))
    if kind == "periodic":
        steps = max(2, steps)
    r = rng.randint(17, 32) if kind == "wide" else rng.randint(1, 16)
    # densities at which the scaled rule keeps boards of every radius alive
    c = dict(kind="single", H=H, W=W, r=r, C=2, M=rng.randint(0, 1), rule="scaled", p=round(rng.uniform(0.48, 0.56), 3),
             storage=U8, boundary=0, kernel="auto", dtype="auto", steps=steps)
    if kind in ("fp8", "fp16"):
        c.update(kernel="tcgen05", dtype=kind)
    elif kind == "bits":
        c.update(storage=BIT1)
    elif kind == "c16":
        c.update(C=rng.choice([3, 4, 8, 16]), storage=rng.choice([U8, NIB4]), p=round(rng.uniform(0.64, 0.72), 3))
    elif kind == "periodic":
        c.update(boundary=1)
    return c


def _rule(case: dict) -> dict:
    if case["rule"] == "conway":
        return dict(inputs.CONWAY)
    if case["rule"] == "multistate":
        return dict(inputs.MULTISTATE_R10_C16)
    return inputs.scaled_rule(case["r"], case["M"], case["C"])


def _gen(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _board(H: int, W: int, p: float, C: int, g: torch.Generator) -> torch.Tensor:
    """Cells alive with probability p; with C > 2 a quarter of the cells is in one of the decaying states."""
    x = torch.rand((H, W), generator=g, device="cuda", dtype=torch.float32)
    s = (x < p).to(torch.uint8)
    if C > 2:
        d = torch.randint(0, 4 * (C - 2), (H, W), generator=g, device="cuda", dtype=torch.uint8)
        s = torch.where(d < C - 2, d + 2, s)
    return s


def _specs(case: dict) -> list[dict]:
    return inputs.batch_instances(case["count"], case["draw_seed"], case["side_lo"], case["side_hi"])


def _pitch(W: int) -> int:
    return (W + 15) // 16 * 16


def _arena(case: dict, seed: int):
    """One buffer for all grids of a batch, each at a multiple of 256 bytes, and its grids' places."""
    specs, at, n = _specs(case), [], 0
    for d in specs:
        at.append(n)
        n += (d["H"] * _pitch(d["W"]) + 255) // 256 * 256
    a = torch.zeros(n, dtype=torch.uint8, device="cuda")
    g = _gen(seed)
    for d, o in zip(specs, at):
        P = _pitch(d["W"])
        a[o:o + d["H"] * P].view(d["H"], P)[:, :d["W"]] = _board(d["H"], d["W"], d["p"], 2, g)
    return specs, at, a


def prepare(case: dict, seed: int):
    if case["kind"] == "batch":
        specs, at, a = _arena(case, seed)
        b = torch.zeros_like(a)
        grids = []
        for d, o in zip(specs, at):
            g = cat.Grid(d["H"], d["W"], d["rule"], kernel=case["kernel"], dtype=case["dtype"])
            cat.cat_bind(g.handle, a.data_ptr() + o, b.data_ptr() + o, _pitch(d["W"]))
            grids.append(g)
        return dict(case=case, grids=grids, handles=[g.handle for g in grids], a=a, b=b)
    g = cat.Grid(case["H"], case["W"], _rule(case), kernel=case["kernel"], dtype=case["dtype"],
                 boundary=case["boundary"], storage=case["storage"])
    g.set_state(_board(case["H"], case["W"], case["p"], case["C"], _gen(seed)))
    return dict(case=case, grid=g)


class _Rows:
    """The rows of a grid's current device buffer; a tensor made from them keeps the grid (and its memory) alive."""

    def __init__(self, grid: cat.Grid):
        self.grid = grid
        ptr, pitch = cat.cat_state_ptr(grid.handle)
        cols = {BIT1: (grid.W + 7) // 8, NIB4: (grid.W + 1) // 2}.get(grid.storage, grid.W)
        self.__cuda_array_interface__ = {"shape": (grid.H, cols), "strides": (pitch, 1), "typestr": "|u1",
                                         "data": (ptr, False), "version": 3}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":   # an even number of steps: the states are back in the first buffer
        cat.cat_batch_step(state["handles"], case["steps"])
        return state["a"]
    state["grid"].step(case["steps"])
    return torch.as_tensor(_Rows(state["grid"]), device="cuda")


def _cells(case: dict) -> int:
    if case["kind"] == "batch":
        return sum(d["H"] * d["W"] for d in _specs(case))
    return case["H"] * case["W"]


def work(case: dict) -> dict:
    """The state read once and written once; per cell and step a running box sum (an addition and a subtraction in each
    direction) and the comparisons with the rule's bounds."""
    cells = _cells(case)
    per_cell = {U8: 1.0, BIT1: 0.125, NIB4: 0.5}[case.get("storage", U8)]
    return {"bytes": 2.0 * per_cell * cells, "flops": 8.0 * cells * case["steps"]}


def _window_sums(x: torch.Tensor, r: int, dim: int) -> torch.Tensor:
    """Sums over 2r + 1 consecutive entries along dim (the result is 2r shorter)."""
    c = torch.cumsum(x, dim, dtype=torch.int64)
    n = x.shape[dim]
    out = c.narrow(dim, 2 * r, n - 2 * r).clone()
    out.narrow(dim, 1, n - 2 * r - 1).sub_(c.narrow(dim, 0, n - 2 * r - 1))
    return out


def _step(s: torch.Tensor, rule: dict, periodic: bool) -> torch.Tensor:
    H, W = s.shape
    r, C = rule["r"], rule["C"]
    out = torch.empty_like(s)
    cols = torch.arange(-r, W + r, device=s.device) % W
    rows = max(1, min(H, (1 << 25) // W))
    for y in range(0, H, rows):
        n = min(rows, H - y)
        if periodic:
            a = (s[torch.arange(y - r, y + n + r, device=s.device) % H] == 1)[:, cols]
        else:
            a = torch.zeros((n + 2 * r, W + 2 * r), dtype=torch.bool, device=s.device)
            lo, hi = max(0, y - r), min(H, y + n + r)
            a[lo - y + r:hi - y + r, r:r + W] = s[lo:hi] == 1
        k = _window_sums(_window_sums(a, r, 0), r, 1)
        c = s[y:y + n]
        k = k - (c == 1).to(torch.int64) if rule["M"] == 0 else k
        born = ((k >= rule["b1"]) & (k <= rule["b2"])).to(torch.uint8)
        kept = (k >= rule["s1"]) & (k <= rule["s2"])
        lost = 2 if C > 2 else 0
        aged = torch.where(c + 1 == C, torch.zeros_like(c), c + 1)
        out[y:y + n] = torch.where(c == 0, born, torch.where(c == 1, torch.where(kept, 1, lost).to(torch.uint8), aged))
    return out


def _packed(s: torch.Tensor, storage: int) -> torch.Tensor:
    """The bytes that a packed grid holds: the lowest cell in the lowest bits."""
    per = {BIT1: 8, NIB4: 2}[storage]
    H, W = s.shape
    n = (W + per - 1) // per
    out = torch.zeros((H, n), dtype=torch.uint8, device=s.device)
    for i in range(per):
        v = s[:, i::per]
        out[:, :v.shape[1]] |= v << (i * 8 // per)
    return out


def exact(case: dict, seed: int):
    if case["kind"] == "batch":
        specs, at, a = _arena(case, seed)
        for d, o in zip(specs, at):
            P = _pitch(d["W"])
            v = a[o:o + d["H"] * P].view(d["H"], P)[:, :d["W"]]
            s = v.clone()
            for _ in range(case["steps"]):
                s = _step(s, d["rule"], False)
            v.copy_(s)
        return a
    s = _board(case["H"], case["W"], case["p"], case["C"], _gen(seed))
    for _ in range(case["steps"]):
        s = _step(s, _rule(case), case["boundary"] == 1)
    return s if case["storage"] == U8 else _packed(s, case["storage"])
