"""The 3D plane pipeline: four steps per launch against single steps, at the edges of its tiles and
segments."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu

# (grids of fewer cells take single steps) narrower than the halo, a row or a plane thin, long in each
# direction, ragged tiles, strips and segments of several sizes
SHAPES = [(4, 300, 700), (8, 1, 98400), (786436, 1, 1), (12, 65539, 1), (1600, 520, 1), (400, 3, 700), (132, 83, 75),
          (100, 97, 91), (256, 72, 48),
          # widths that are not multiples of 4
          (1, 1600, 1400), (3, 911, 815), (49, 230, 191), (2097155, 1, 1), (193, 107, 110)]


def _run(lee, monkeypatch, name, shape, storage, n, g0, single=False, **kw):
    for k in ("LEE_TB_STEPS", "LEE_SINGLE_STEP", "LEE_T3_TMA"):
        monkeypatch.delenv(k, raising=False)
    if single:
        monkeypatch.setenv("LEE_SINGLE_STEP", "1")
    g = np.empty_like(g0)
    with lee.Solver(name, shape, 0.57, storage=storage, **kw) as sv:
        sv.set_populations(g0)
        for k in n if isinstance(n, tuple) else (n,):
            sv.step(k)
        sv.get_populations(g)
    return g


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("name", ["D3Q7", "D3Q7_DI"])
def test_fp32_runs_equal_single_steps(gpu_lib, monkeypatch, name, shape):
    """One launch, a launch with every remainder, a replayed graph, and calls that start in either copy."""
    lee = gpu_lib
    g0 = inputs.random_populations(7, int(np.prod(shape)), seed=8)
    for n in (4, 5, 7, 43, (43, 43, 4)):
        a = _run(lee, monkeypatch, name, shape, "f32", n, g0)
        b = _run(lee, monkeypatch, name, shape, "f32", n, g0, single=True)
        assert np.array_equal(a, b), n
