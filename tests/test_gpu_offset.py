"""The FP8 kernel with H - 16 as pass 2's operand (two states, uint8, r = 8 ..
15) vs the CPU oracle, with the radii on either side: tiles cut at every edge,
counts at both ends of their range, ranges that are empty or hold everything,
one step and several per launch.  All values are whole numbers, so every
comparison is exact.
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


@pytest.mark.parametrize("r", [7, 8, 11, 15, 16])
@pytest.mark.parametrize("shape", [(1, 1), (127, 129), (300, 273)])
def test_offset_pass2(cat, r, shape):
    top = (2 * r + 1) ** 2
    s = inputs.scaled_rule(r)
    boards = [inputs.bernoulli(*shape, 0.5, r), np.ones(shape, np.uint8), np.zeros(shape, np.uint8)]
    for rule in (s, dict(s, s1=3, s2=2, b1=0, b2=0), dict(s, M=1, s1=top, s2=1 << 30, b1=0, b2=top)):
        for grid in boards:
            for per_launch in (1, 3):
                g = cat.Grid(*shape, rule, kernel="tcgen05", dtype="fp8", steps_per_launch=per_launch)
                try:
                    g.set_state(grid)
                    assert np.array_equal(g.box_sums(), oracle.box_sums(grid, r))
                    g.step(3)
                    got = g.get_state()
                    assert g.status() == cat.CAT_OK
                finally:
                    g.close()
                assert np.array_equal(got, oracle.step(grid, oracle.Rule(**rule), n_steps=3)), (rule, per_launch)


@pytest.mark.parametrize("r", [16, 32])
def test_ranges_of_the_wide_tile(cat, r):
    """Its counts are compared as f32: the same edges of the rule's ranges."""
    top = (2 * r + 1) ** 2
    s = inputs.scaled_rule(r)
    grid = inputs.bernoulli(131, 200, 0.5, r)
    for g0 in (grid, np.ones_like(grid)):
        for rule in (s, dict(s, s1=3, s2=2, b1=0, b2=0), dict(s, M=1, s1=top, s2=1 << 30, b1=1, b2=top // 2)):
            g = cat.Grid(131, 200, rule, kernel="tcgen05", dtype="fp8", tile=96)
            try:
                g.set_state(g0)
                g.step(2)
                got = g.get_state()
            finally:
                g.close()
            assert np.array_equal(got, oracle.step(g0, oracle.Rule(**rule), n_steps=2)), rule
