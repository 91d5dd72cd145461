"""The bit-plane box-sum kernel (options left to the library) vs the CPU
oracle: radii at the edges of its plane counts, widths around 32-cell words
and the words a warp writes, strips shorter and longer than the grid, every
storage, both boundaries, and buffers whose bytes past W belong to the caller.
All values are whole numbers, so every comparison is exact.
"""
import numpy as np
import pytest

from oracle import oracle
from paper_2406_17284_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (9, 16), (40, 33), (33, 961), (70, 1031), (700, 95)]


@pytest.fixture(scope="module")
def cat():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2406_17284_gb300 import build
    build.build()
    from paper_2406_17284_gb300 import cat as catmod
    catmod.load()
    return catmod


def board(H, W, C, seed):
    g = inputs.bernoulli(H, W, 0.5, seed)
    if C > 2:
        u = inputs.uniform_states(H, W, C, seed + 1)
        g = np.where((u >= 2) & (inputs.bernoulli(H, W, 0.3, seed + 2) == 1), u, g)
    return g.astype(np.uint8)


def check(cat, H, W, rule, storage, boundary=0, steps=3):
    grid = board(H, W, rule["C"], 7 * H + W + rule["r"])
    g = cat.Grid(H, W, rule, kernel="auto", dtype="auto", storage=storage, boundary=boundary)
    try:
        g.set_state(grid)
        g.step(steps)
        got = g.get_state()
        assert g.status() == cat.CAT_OK
    finally:
        g.close()
    want = oracle.step(grid, oracle.Rule(**rule), boundary=boundary, n_steps=steps)
    assert np.array_equal(got, want), (H, W, rule, storage, boundary, int((got != want).sum()))


def rules(r, C):
    s = inputs.scaled_rule(r, M=r & 1, C=C)
    top = (2 * r + 1) ** 2
    # empty survival range, birth of everything; survival of full boxes only
    return [s, dict(s, s1=3, s2=2, b1=0, b2=top), dict(s, M=1, s1=top, s2=1 << 30, b1=1, b2=top // 2)]


@pytest.mark.parametrize("storage,C,radii", [(0, 2, (1, 2, 3, 7, 8, 9)), (1, 2, (1, 2, 3, 5, 7, 8, 15, 16)),
                                             (2, 2, (1, 9)), (2, 16, (1, 10, 16)), (0, 3, (1, 15)), (0, 16, (2, 10))])
def test_planes_match_the_oracle(cat, storage, C, radii):
    for r in radii:
        for H, W in SHAPES:
            for rule in rules(r, C):
                check(cat, H, W, rule, storage)


@pytest.mark.parametrize("C", [2, 5])
def test_planes_on_a_torus(cat, C):
    for r in (1, 6, 9):
        for H, W in [(20, 17), (33, 64), (70, 1031)]:
            check(cat, H, W, inputs.scaled_rule(r, C=C), 0, boundary=1)


@pytest.mark.parametrize("r", [1, 4, 7])
def test_packed_steps_on_a_torus(cat, r):
    """Several steps in one call: the one-bit ghost frame at every word offset of W."""
    for H, W in [(5, 64), (20, 79), (33, 80), (40, 81), (64, 95), (70, 96), (33, 1031)]:
        for n in (2, 3, 6):
            check(cat, H, W, inputs.scaled_rule(r, M=1), 0, boundary=1, steps=n)


@pytest.mark.parametrize("r", [8, 16])
@pytest.mark.parametrize("H,W", [(5611, 5807), (33, 1048577)])
def test_packed_steps_on_a_large_torus(cat, r, H, W):
    """The larger radii take the bits from 30 * 2^20 cells on: against the
    tensor-core kernel's steps from the same state."""
    import torch
    rule, host = inputs.scaled_rule(r), board(H, W, 2, r)
    a = cat.Grid(H, W, rule, kernel="auto", dtype="auto", boundary=1)
    b = cat.Grid(H, W, rule, kernel="tcgen05", dtype="fp8", boundary=1)
    try:
        for g in (a, b):
            g.set_state(host)
            g.step(9)
        assert torch.equal(a.state_tensor(), b.state_tensor())
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("C", [2, 16])
def test_bytes_past_the_grid_are_not_read_or_written(cat, C):
    """Bound buffers with a pitch above W, the gap full of other data."""
    import torch
    for H, W, pitch in [(50, 37, 48), (50, 1000, 1024), (9, 97, 112)]:
        rule = inputs.scaled_rule(4, C=C)
        grid = board(H, W, C, W)
        a = torch.full((H, pitch), 255, dtype=torch.uint8, device="cuda")
        b = torch.full((H, pitch), 254, dtype=torch.uint8, device="cuda")
        a[:, :W] = torch.from_numpy(grid).cuda()
        g = cat.Grid(H, W, rule, kernel="auto", dtype="auto")
        try:
            cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), pitch)
            g.step(3)
            torch.cuda.synchronize()
        finally:
            g.close()
        assert np.array_equal(b[:, :W].cpu().numpy(), oracle.step(grid, oracle.Rule(**rule), n_steps=3))
        assert bool((a[:, W:] == 255).all()) and bool((b[:, W:] == 254).all())


@pytest.mark.parametrize("r", [1, 4, 16])
def test_packed_steps_between_uint8_states(cat, r):
    """Several steps in one call keep the states between packed, inside the
    grid's own rows: any number of steps, the state where the parity puts it,
    no byte past W touched."""
    import torch
    rule = inputs.scaled_rule(r, M=1)
    for H, W, pitch in [(40, 64, 64), (33, 97, 112), (130, 1031, 1056)]:
        grid = board(H, W, 2, W + r)
        for n in (2, 3, 4, 5, 9):
            a = torch.full((H, pitch), 255, dtype=torch.uint8, device="cuda")
            b = torch.full((H, pitch), 254, dtype=torch.uint8, device="cuda")
            a[:, :W] = torch.from_numpy(grid).cuda()
            g = cat.Grid(H, W, rule, kernel="auto", dtype="auto")
            try:
                cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), pitch)
                g.step(n)
                torch.cuda.synchronize()
                got = (b if n & 1 else a)[:, :W].cpu().numpy()
                assert cat.cat_state_ptr(g.handle)[0] == (b if n & 1 else a).data_ptr()
            finally:
                g.close()
            assert np.array_equal(got, oracle.step(grid, oracle.Rule(**rule), n_steps=n)), (H, W, r, n)
            assert bool((a[:, W:] == 255).all()) and bool((b[:, W:] == 254).all())


def test_packed_batch_of_uneven_grids(cat):
    """cat_batch_step with the options left to the library: every radius, grids
    narrower and wider than a warp's words, and one large enough for the batch
    to step on bit planes; calls of different lengths one after the other (also
    short and captured ones, which take the tiles)."""
    import torch
    specs = [dict(r=r, H=H, W=W, M=r & 1) for r, H, W in
             [(r, 20 + 7 * r, 64 + 61 * (r % 5)) for r in range(1, 17)] + [(3, 300, 1031), (16, 90, 961), (9, 1, 64)]]
    grids, hosts = [], []
    for i, d in enumerate(specs):
        rule = inputs.scaled_rule(d["r"], M=d["M"])
        host = board(d["H"], d["W"], 2, 50 + i)
        g = cat.Grid(d["H"], d["W"], rule, kernel="auto", dtype="auto")
        g.set_state(host)
        grids.append(g)
        hosts.append((host, oracle.Rule(**rule)))
    rule, large = inputs.scaled_rule(2), board(5801, 5803, 2, 9)
    big = cat.Grid(5801, 5803, rule, kernel="auto", dtype="auto")
    ref = cat.Grid(5801, 5803, rule, kernel="tcgen05", dtype="fp8")
    big.set_state(large)
    ref.set_state(large)
    handles = [g.handle for g in grids] + [big.handle]

    def compare(done):
        for g, (host, rule) in zip(grids, hosts):
            assert np.array_equal(g.get_state(), oracle.step(host, rule, n_steps=done)), (done, rule, host.shape)
        assert torch.equal(big.state_tensor(), ref.state_tensor()), done
    try:
        done = 0
        for n, captured in ((8, False), (4, True), (9, False), (1, False), (11, False), (4, False), (2, True)):
            if captured:   # (the first one comes before any call has taken the tiles)
                s = torch.cuda.Stream()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    cat.cat_batch_step(handles, n, s)
                graph.replay()
                torch.cuda.synchronize()
            else:
                cat.cat_batch_step(handles, n)
            ref.step(n)
            done += n
            compare(done)
        with pytest.raises(cat.CatError):
            cat.cat_batch_step(handles + handles[:1], 4)
    finally:
        for g in grids + [big, ref]:
            g.close()


@pytest.mark.parametrize("storage,H,W,r,n", [(1, 300, 700, 1, 2), (1, 300, 700, 1, 8), (1, 130, 2000, 1, 100),
                                             (1, 300, 700, 4, 4), (1, 300, 700, 10, 2), (1, 50, 90, 16, 4),
                                             (0, 300, 700, 1, 8), (0, 300, 700, 10, 6), (0, 130, 1031, 4, 2),
                                             (2, 200, 333, 3, 2)])
def test_captured_steps_with_the_options_left(cat, storage, H, W, r, n):
    """An even number of steps of a default grid, captured into a graph in one
    call and replayed three times, then a plain call of an odd number."""
    import torch
    rule = inputs.scaled_rule(r, M=1, C=5 if storage == 2 else 2)
    host = board(H, W, rule["C"], 3 * r + n)
    g = cat.Grid(H, W, rule, kernel="auto", dtype="auto", storage=storage)
    try:
        g.set_state(host)
        at = cat.cat_state_ptr(g.handle)[0]
        s = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            g.step(n, s)
        assert cat.cat_state_ptr(g.handle)[0] == at
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        want = oracle.step(host, oracle.Rule(**rule), n_steps=3 * n)
        assert np.array_equal(g.get_state(), want)
        g.step(3)
        assert cat.cat_state_ptr(g.handle)[0] != at
        assert np.array_equal(g.get_state(), oracle.step(want, oracle.Rule(**rule), n_steps=3))
    finally:
        g.close()


@pytest.mark.parametrize("H,W", [(450000, 33), (840000, 16), (450000, 64), (450000, 65), (300000, 90), (300000, 120)])
@pytest.mark.parametrize("r", [3, 13, 16])
def test_tall_grids(cat, H, W, r):
    """Narrow and tall: where the choice between bit planes and tensor cores
    depends on the words of a row, both give the same states."""
    import torch
    for C, boundary, n in ((16, 0, 2), (2, 0, 1), (2, 0, 8), (2, 1, 3)):
        rule = inputs.scaled_rule(r, M=1, C=C)
        host = board(H, W, C, W + r)
        a = cat.Grid(H, W, rule, kernel="auto", dtype="auto", boundary=boundary)
        b = cat.Grid(H, W, rule, kernel="tcgen05", dtype="fp8", boundary=boundary)
        try:
            for g in (a, b):
                g.set_state(host)
                g.step(n)
            assert torch.equal(a.state_tensor(), b.state_tensor()), (C, boundary, n)
        finally:
            a.close()
            b.close()


def test_foreign_kernels_between_default_steps(cat):
    """Kernels without the early-launch trigger on both sides of every call: they
    read the state just stepped and rewrite parts of it, in place, on one stream
    with grids of other storages, each stepped in turn."""
    import torch
    H, W, pitch = 600, 700, 720
    rule = inputs.scaled_rule(4)
    grid = board(H, W, 2, 31)
    a = torch.zeros((H, pitch), dtype=torch.uint8, device="cuda")
    b = torch.zeros((H, pitch), dtype=torch.uint8, device="cuda")
    a[:, :W] = torch.from_numpy(grid).cuda()
    bound = cat.Grid(H, W, rule, kernel="auto", dtype="auto")
    cat.cat_bind(bound.handle, a.data_ptr(), b.data_ptr(), pitch)
    others = []
    for r, C, storage, boundary in ((2, 2, 1, 0), (9, 2, 1, 0), (1, 2, 0, 0), (5, 5, 2, 0), (3, 16, 0, 0), (4, 2, 0, 1)):
        rr, host = inputs.scaled_rule(r, C=C), board(300 + 7 * r, 401, C, r)
        g = cat.Grid(*host.shape, rr, kernel="auto", dtype="auto", storage=storage, boundary=boundary)
        g.set_state(host)
        others.append([g, oracle.Rule(**rr), host, boundary])
    try:
        cur, other, want = a, b, grid
        for k, n in enumerate((1, 2, 5, 1, 4)):
            bound.step(n)
            if n & 1:
                cur, other = other, cur
            snap, want = cur[:, :W].clone(), oracle.step(want, oracle.Rule(**rule), n_steps=n)
            cur[50 + 40 * k:90 + 40 * k, :W] ^= 1
            cur[:, 9 * k:9 * k + 20] = 0
            for o in others:
                o[0].step(n)
                o[2] = oracle.step(o[2], o[1], boundary=o[3], n_steps=n)
                if o[0].storage == 0:    # the first row dies, by a torch kernel
                    o[0].state_tensor()[0] = 0
                    o[2] = o[2].copy()
                    o[2][0] = 0
            assert np.array_equal(snap.cpu().numpy(), want), k
            want = want.copy()
            want[50 + 40 * k:90 + 40 * k] ^= 1
            want[:, 9 * k:9 * k + 20] = 0
        for g, rr, host, boundary in others:
            assert np.array_equal(g.get_state(), host), (rr, boundary)
    finally:
        for g in [bound] + [o[0] for o in others]:
            g.close()


@pytest.mark.parametrize("r,n", [(10, 4), (10, 8), (3, 6), (2, 32), (1, 32)])
def test_tiles_of_as_many_steps_as_they_take(cat, r, n):
    """The most steps per launch: two at r = 10, after which 30 of the 32 cells of
    a neighbouring word are stale."""
    for H, W in [(40, 33), (200, 961), (90, 1031)]:
        check(cat, H, W, inputs.scaled_rule(r, M=1), 1, steps=n)
        if W >= 64:
            check(cat, H, W, inputs.scaled_rule(r, M=1), 0, steps=n + 1)
