"""Global sums of FP64 states: momentum adds up the differences of opposite populations, cell by cell, so it is as exact as
they are however large the populations themselves; and sums with cells at the edges of a thread's group."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SETS = ["D1Q3", "D2Q5", "D2Q5_DI", "D3Q7", "D3Q7_DI", "D3Q9", "D3Q13", "D3Q19"]
UNIT = 2.0 ** -53


def _shape(info, cells):
    return (cells, 1, 1) if info["D"] == 1 else (cells // 7, 7, 1) if info["D"] == 2 else (cells // 35, 7, 5)


@pytest.mark.parametrize("cells", [35, 1015, 116725, 116970, 467005])
@pytest.mark.parametrize("name", SETS)
def test_momentum_beside_large_populations(gpu_lib, name, cells):
    """Opposite populations that differ by 1e-9 of themselves.  A difference of two such values is exact; its sums round at
    most 64 times in the longest chain (a thread's groups, the warp, the block, the blocks)."""
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    D, q, c, f = info["D"], info["q"], np.array(info["c"]), np.array(info["f"])[:, None]
    rng = np.random.default_rng(cells)
    g = np.empty((q, cells))
    g[0] = rng.uniform(0.5, 1.0, cells)
    g[1::2] = rng.uniform(0.5, 1.0, (q // 2, cells))
    g[2::2] = g[1::2] * (1.0 + 1e-9 * rng.normal(size=(q // 2, cells)))
    red = np.empty(D + 4)
    with lee.Solver(name, _shape(info, cells), 0.6, storage="f64") as sv:
        sv.set_populations(g)
        sv.reduce(red)
    assert abs(red[0] - math.fsum(g.ravel())) <= 64 * UNIT * g.sum()
    for a in range(D):
        d = (c[1::2, a, None] * (g[1::2] - g[2::2])).ravel()
        assert abs(red[1 + a] - math.fsum(d)) <= 64 * UNIT * np.abs(d).sum()
    assert abs(red[D + 2] - math.fsum((g * g / f).ravel())) <= 64 * UNIT * (g * g / f).sum()
    assert red[D + 3] == 0


@pytest.mark.parametrize("name", SETS)
def test_values_that_are_not_finite(gpu_lib, name):
    """Each is counted and left out of the sums; the others of its cell and group stay."""
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    D, q, cells, c = info["D"], info["q"], 1015, np.array(info["c"])
    rng = np.random.default_rng(3)
    g = rng.uniform(0.5, 1.0, (q, cells))
    red = np.empty(D + 4)
    for i, x, v in [(0, 0, np.nan), (1, 0, np.inf), (q - 1, cells - 1, -np.inf), (2, 256, np.nan), (2, 512, np.nan)]:
        g[i, x] = v
    with lee.Solver(name, _shape(info, cells), 0.6, storage="f64") as sv:
        sv.set_populations(g)
        sv.reduce(red)
    fine = np.where(np.isfinite(g), g, 0.0)
    assert red[D + 3] == 5
    assert abs(red[0] - math.fsum(fine.ravel())) <= 64 * UNIT * fine.sum()
    for a in range(D):
        assert abs(red[1 + a] - math.fsum((c[:, a, None] * fine).ravel())) <= 64 * UNIT * fine.sum()
