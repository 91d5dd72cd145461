"""cat_bind: an instance stepping two caller-owned device buffers (torch tensors).

The state is read from the first buffer as it is, steps alternate between the
two (as cat_state_ptr reports), results match the CPU oracle, and the buffers
stay the caller's after cat_destroy.
"""
import numpy as np
import pytest

from oracle import oracle
from paper_2406_17284_gb300 import inputs

pytestmark = pytest.mark.gpu


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


def orule(d):
    return oracle.Rule(d["r"], d["C"], d["M"], d["s1"], d["s2"], d["b1"], d["b2"], d.get("nbhd", "M"))


@pytest.mark.parametrize("kernel,dtype,k", [("tcgen05", "fp8", 1), ("tcgen05", "fp8", 3), ("tcgen05", "fp16", 1),
                                            ("mma_sync", "fp16", 1), ("stencil", "auto", 1),
                                            ("runsum", "auto", 1)])
def test_steps_on_torch_buffers(cat, kernel, dtype, k):
    import torch
    H, W, pitch = 333, 517, 544            # pitch above the minimum, a multiple of 16
    rule = inputs.scaled_rule(7)
    grid = inputs.bernoulli(H, W, 0.5, 90)
    a = torch.zeros((H, pitch), dtype=torch.uint8, device="cuda")
    b = torch.full((H, pitch), 7, dtype=torch.uint8, device="cuda")   # garbage the step must overwrite
    a[:, :W] = torch.from_numpy(grid).cuda()
    g = cat.Grid(H, W, rule, kernel=kernel, dtype=dtype, steps_per_launch=k)
    try:
        cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), pitch)
        assert cat.cat_state_ptr(g.handle) == (a.data_ptr(), pitch)
        g.step(1)
        torch.cuda.synchronize()
        assert g.status() == cat.CAT_OK
        assert cat.cat_state_ptr(g.handle)[0] == b.data_ptr()
        assert np.array_equal(b[:, :W].cpu().numpy(), oracle.step(grid, orule(rule)))
        g.step(4)
        torch.cuda.synchronize()
        assert g.status() == cat.CAT_OK
        assert cat.cat_state_ptr(g.handle)[0] == b.data_ptr()
        want = oracle.step(grid, orule(rule), n_steps=5)
        assert np.array_equal(b[:, :W].cpu().numpy(), want)
        assert np.array_equal(g.get_state(), want)
    finally:
        g.close()
    a.fill_(3)                              # still the caller's memory
    torch.cuda.synchronize()
    assert int(a[0, 0]) == 3


def test_rejections(cat):
    import torch
    rule = inputs.scaled_rule(3)
    a = torch.zeros((64, 64), dtype=torch.uint8, device="cuda")
    b = torch.zeros((64, 64), dtype=torch.uint8, device="cuda")
    g = cat.Grid(64, 64, rule, boundary=cat.BOUNDARY_PERIODIC)
    try:
        with pytest.raises(cat.CatError) as e:
            cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), 64)
        assert e.value.code == cat.CAT_ERR_UNSUPPORTED
    finally:
        g.close()
    g = cat.Grid(64, 60, rule)
    try:
        for args in ((a.data_ptr(), b.data_ptr(), 40), (a.data_ptr(), a.data_ptr(), 64),
                     (a.data_ptr(), b.data_ptr(), 56)):
            with pytest.raises(cat.CatError) as e:
                cat.cat_bind(g.handle, *args)
            assert e.value.code == cat.CAT_ERR_INVALID_ARG, args
        host = np.zeros((64, 64), np.uint8)
        with pytest.raises(cat.CatError) as e:
            cat.cat_bind(g.handle, host.ctypes.data, b.data_ptr(), 64)
        assert e.value.code == cat.CAT_ERR_INVALID_ARG
        cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), 64)
        with pytest.raises(cat.CatError) as e:
            cat.cat_set_options(g.handle, cat.KERNEL_TCGEN05, cat.DTYPE_FP8_E4M3, cat.STORE_BIT1)
        assert e.value.code == cat.CAT_ERR_UNSUPPORTED
    finally:
        g.close()


@pytest.mark.parametrize("n", [1, 5])
def test_pitch_above_four_gib(cat, n):
    """Rows more than 2^32 bytes apart, with every option left to the library."""
    import torch
    H, W, pitch = 3, 200, (1 << 32) + 4096
    size = (H - 1) * pitch + 4096
    if torch.cuda.mem_get_info()[0] < 3 * size:
        pytest.skip("not enough device memory")
    rule = inputs.scaled_rule(4)
    grid = inputs.bernoulli(H, W, 0.5, 17)
    a = torch.zeros(size, dtype=torch.uint8, device="cuda")
    b = torch.zeros(size, dtype=torch.uint8, device="cuda")
    rows = [torch.as_strided(t, (H, W), (pitch, 1)) for t in (a, b)]
    rows[0].copy_(torch.from_numpy(grid))
    g = cat.Grid(H, W, rule, kernel="auto", dtype="auto")
    try:
        cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), pitch)
        g.step(n)
        torch.cuda.synchronize()
        assert g.status() == cat.CAT_OK
    finally:
        g.close()
    assert np.array_equal(rows[n & 1].cpu().numpy(), oracle.step(grid, orule(rule), n_steps=n))
    for t in (a, b):    # nothing between the rows
        assert not bool(t[4096:pitch].any()) and not bool(t[pitch + 4096:2 * pitch].any())


@pytest.mark.parametrize("H,W,pitch,r,n", [(130, 1024, 1024, 4, 2), (130, 1024, 1024, 4, 3), (70, 97, 112, 1, 9),
                                           (300, 517, 544, 12, 4), (2600, 2700, 2704, 2, 8)])
def test_the_other_buffer_holds_the_generation_before(cat, H, W, pitch, r, n):
    """A caller's two buffers after several steps in one call, every option left
    to the library: the state, and the generation before it (cat_step and
    cat_batch_step)."""
    import torch
    rule = inputs.scaled_rule(r)
    grid = inputs.bernoulli(H, W, 0.5, H + n)
    before = oracle.step(grid, orule(rule), n_steps=n - 1)
    after = oracle.step(before, orule(rule))
    for batch in (False, True):
        a = torch.zeros((H, pitch), dtype=torch.uint8, device="cuda")
        b = torch.zeros((H, pitch), dtype=torch.uint8, device="cuda")
        a[:, :W] = torch.from_numpy(grid).cuda()
        g = cat.Grid(H, W, rule, kernel="auto", dtype="auto")
        try:
            cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), pitch)
            if batch:
                cat.cat_batch_step([g.handle], n)
            else:
                g.step(n)
            torch.cuda.synchronize()
            state, other = (b, a) if n & 1 else (a, b)
            assert cat.cat_state_ptr(g.handle)[0] == state.data_ptr()
        finally:
            g.close()
        assert np.array_equal(state[:, :W].cpu().numpy(), after), batch
        assert np.array_equal(other[:, :W].cpu().numpy(), before), batch


@pytest.mark.parametrize("kernel,dtype,r,tile", [("tcgen05", "fp8", 4, 0), ("tcgen05", "fp8", 9, 0), ("tcgen05", "fp16", 9, 0),
                                                 ("tcgen05", "fp4", 9, 0), ("tcgen05", "fp8", 24, 0),
                                                 ("tcgen05", "fp8", 24, 96), ("mma_sync", "fp16", 4, 0),
                                                 ("stencil", "auto", 4, 0), ("runsum", "auto", 4, 0), ("auto", "auto", 4, 0),
                                                 ("auto", "auto", 9, 0)])
def test_no_byte_past_a_rows_last_unit_is_touched(cat, kernel, dtype, r, tile):
    """A pitch above W, births everywhere: the bytes from W to the next multiple
    of 16 are the library's, those beyond stay, by cat_step and cat_batch_step."""
    import torch
    H, W, pitch, unit = 150, 101, 144, 112
    rule = dict(inputs.scaled_rule(r), b1=0, b2=(2 * r + 1) ** 2)
    grid = inputs.bernoulli(H, W, 0.5, r)
    for batch in (False, True):
        a = torch.full((H, pitch), 255, dtype=torch.uint8, device="cuda")
        b = torch.full((H, pitch), 254, dtype=torch.uint8, device="cuda")
        a[:, :W] = torch.from_numpy(grid).cuda()
        g = cat.Grid(H, W, rule, kernel=kernel, dtype=dtype, tile=tile)
        try:
            cat.cat_bind(g.handle, a.data_ptr(), b.data_ptr(), pitch)
            for n in (1, 2):
                if batch:
                    cat.cat_batch_step([g.handle], n)
                else:
                    g.step(n)
            torch.cuda.synchronize()
            assert g.status() == cat.CAT_OK
        finally:
            g.close()
        assert np.array_equal(b[:, :W].cpu().numpy(), oracle.step(grid, orule(rule), n_steps=3)), batch
        assert bool((a[:, unit:] == 255).all()) and bool((b[:, unit:] == 254).all()), batch
