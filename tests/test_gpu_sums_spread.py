"""Moments and global sums where populations of very different size meet in a cell or in neighbouring cells: each sum is
as near its own terms as FP64 sums of them are, whatever the other populations hold."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SETS = [("D1Q3", (1023, 1, 1)), ("D2Q5", (61, 37, 1)), ("D2Q5_DI", (64, 33, 1)), ("D3Q7", (13, 11, 29)),
        ("D3Q9", (16, 9, 17)), ("D3Q13", (16, 9, 11)), ("D3Q19", (13, 11, 9))]
UNIT = 2.0 ** -53


def _sizes(kind, c, shape, rng):
    """Size of each velocity's populations, per cell."""
    q, cells = len(c), int(np.prod(shape))
    s = np.ones((q, cells))
    if kind == "tiny moving":
        s[1:] = 1e-15
    elif kind == "denormal moving":
        s[1:] = 1e-39
    elif kind == "all tiny":  # normal numbers below the integer form's range, and denormals
        s *= 1e-30
        s[:, ::3] = 1e-40
    elif kind == "tiny rest":
        s[0] = 1e-14
    elif kind == "last axis tiny":  # velocities along the last axis alone; only they carry its momentum in the axis sets
        last = max(a for a in range(3) if any(v[a] for v in c))
        s[[i for i in range(q) if any(c[i]) and not any(c[i][:last])]] = 1e-13
    elif kind == "one cell in four":
        s[:, np.arange(cells) % 4 != 1] = 1e-16
    elif kind == "falling off":  # a tail: 2^-3 per cell and back
        x = np.arange(cells) % 40
        s *= 2.0 ** (-3.0 * np.minimum(x, 40 - x))
    elif kind == "edge of the integer form":  # 2^33 and 2^34 apart
        s[rng.integers(0, q, cells), np.arange(cells)] = 2.0 ** -rng.integers(31, 36, cells)
    return s


@pytest.mark.parametrize("kind", ["tiny moving", "denormal moving", "all tiny", "tiny rest", "last axis tiny", "one cell in four",
                                  "falling off", "edge of the integer form"])
@pytest.mark.parametrize("storage", ["f32", "bf16", "bfp16"])
@pytest.mark.parametrize("name,shape", SETS)
def test_each_sum_against_its_own_terms(gpu_lib, name, shape, storage, kind):
    """Bounds: 24 roundings of a cell's terms (at most 18 additions and the coefficients); 64 of all cells' terms for the
    global sums, and for the terms in one thread's group of cells and one block's."""
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    D, q, cells = info["D"], info["q"], int(np.prod(shape))
    rng = np.random.default_rng(11)
    c, f = np.array(info["c"]), np.array(info["f"])[:, None]
    g0 = rng.uniform(0.5, 1.0, (q, cells)) * _sizes(kind, info["c"], shape, rng) * rng.choice([-1.0, 1.0], (q, 1))
    rho, u, red, g = np.empty(cells), np.empty((D, cells)), np.empty(D + 4), np.empty((q, cells))
    with lee.Solver(name, shape, 0.6, storage=storage) as sv:
        sv.set_populations(np.ascontiguousarray(g0))
        sv.get_populations(g)
        sv.moments(rho, u)
        sv.reduce(red)
    for x in range(cells):
        assert abs(rho[x] - math.fsum(g[:, x])) <= 24 * UNIT * np.abs(g[:, x]).sum()
        for a in range(D):
            j = c[:, a] * g[:, x] / info["rho0"]
            assert abs(u[a, x] - math.fsum(j)) <= 24 * UNIT * np.abs(j).sum()
    w = 0.5 * ((c ** 2).sum(1) + np.array(info["beta"]))[:, None]
    for got, terms in [(red[0], g), (red[D + 1], w * g), (red[D + 2], g * g / f)] + [(red[1 + a], c[:, a, None] * g) for a in range(D)]:
        assert abs(got - math.fsum(terms.ravel())) <= 64 * UNIT * np.abs(terms).sum()
    assert red[D + 3] == 0
