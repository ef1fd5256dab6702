"""Two steps per launch of the 3D sets with diagonal velocities against single steps, at the edges of its tiles
(30 x 14 cells) and segments."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu

# Columns and rows of the plane: one tile, one cell less and more than whole tiles, several ragged tiles, odd widths.
# The planes fill the grid up to the size from which runs take two steps per launch.
PLANES = [(60, 14), (59, 13), (61, 28), (120, 15), (178, 41), (97, 55), (256, 72)]
SETS = [("D3Q9", 9, 3728271), ("D3Q13", 13, 1290556), ("D3Q19", 19, 883012)]


def _run(lee, monkeypatch, name, shape, n, g0, single=False):
    for k in ("LEE_TB_STEPS", "LEE_SINGLE_STEP", "LEE_T3_TMA"):
        monkeypatch.delenv(k, raising=False)
    if single:
        monkeypatch.setenv("LEE_SINGLE_STEP", "1")
    g = np.empty_like(g0)
    with lee.Solver(name, shape, 0.57, storage="f32") as sv:
        sv.set_populations(g0)
        for k in n:
            sv.step(k)
        sv.get_populations(g)
    return g


@pytest.mark.parametrize("plane", PLANES)
@pytest.mark.parametrize("name,q,cells", SETS)
def test_fp32_runs_equal_single_steps(gpu_lib, monkeypatch, name, q, cells, plane):
    """One launch, a launch and a single step, a replayed graph, and calls that start in either copy."""
    lee = gpu_lib
    shape = (*plane, cells // (plane[0] * plane[1]) + 8)
    g0 = inputs.random_populations(q, int(np.prod(shape)), seed=8)
    for n in ((2,), (3,), (21, 21, 2)):
        a = _run(lee, monkeypatch, name, shape, n, g0)
        b = _run(lee, monkeypatch, name, shape, n, g0, single=True)
        assert np.array_equal(a, b), n
