"""The ghost frame of a periodic uint8 grid vs the CPU oracle: every remainder
of W by 16, grids as small as the frame is wide and smaller, so that each frame
cell, the corners too, is read by the step after it.
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


@pytest.mark.parametrize("kernel,dtype,r", [("tcgen05", "fp8", 16), ("auto", "auto", 4)])
@pytest.mark.parametrize("H", [1, 15, 16, 40])
def test_frame_of_every_width(cat, kernel, dtype, r, H):
    rule = inputs.scaled_rule(r, M=1)
    for W in [15, *range(16, 33), 47, 1025]:
        grid = inputs.bernoulli(H, W, 0.5, H * W)
        g = cat.Grid(H, W, rule, kernel=kernel, dtype=dtype, boundary=1)
        try:
            g.set_state(grid)
            for _ in range(2):
                g.step(1)
            assert np.array_equal(g.get_state(), oracle.step(grid, oracle.Rule(**rule), boundary=1, n_steps=2)), W
        finally:
            g.close()


@pytest.mark.parametrize("kernel,dtype,r,n", [("tcgen05", "fp8", 16, 2), ("auto", "auto", 4, 1), ("auto", "auto", 4, 3)])
@pytest.mark.parametrize("H", [16383, 16384, 1 << 19])
def test_frame_of_tall_grids(cat, kernel, dtype, r, n, H):
    """Sides in chunks of 16 cells from 16384 rows on, where W is a multiple of 16,
    and by the looping kernel from 2^19."""
    rule = inputs.scaled_rule(r, M=1)
    for W in (16, 48, 64, 65):
        grid = inputs.bernoulli(H, W, 0.5, H + W)
        g = cat.Grid(H, W, rule, kernel=kernel, dtype=dtype, boundary=1)
        try:
            g.set_state(grid)
            g.step(n)
            assert np.array_equal(g.get_state(), oracle.step(grid, oracle.Rule(**rule), boundary=1, n_steps=n)), W
        finally:
            g.close()
