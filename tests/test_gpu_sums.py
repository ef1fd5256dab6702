"""Moments and global sums of FP32 and 16-bit states, which the kernels add as integers, against exact sums:
magnitudes, spreads and special values at the edges of the integer form."""
import math

import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu


def _cases(rng, q, cells):
    """Populations by cells: all of one size; spread over 2^-40 of the largest; tiny next to normal; signed zeros and
    denormals; a cell of zeros; a cell of values below the integer form's range."""
    g = rng.normal(size=(q, cells)).astype(np.float32)
    k = cells // 6
    g[:, k:2 * k] *= (2.0 ** -rng.integers(0, 40, size=(q, k))).astype(np.float32)
    g[:, 2 * k:3 * k] *= np.float32(1e-30)
    g[0, 2 * k:3 * k] = 1.0
    g[1:, 3 * k:4 * k] = rng.choice(np.array([0.0, -0.0, 1e-42, -1e-42], np.float32), size=(q - 1, k))
    g[:, 4 * k:5 * k] = 0.0
    g[:, 5 * k:] *= np.float32(1e-25)
    return g


@pytest.mark.parametrize("name,shape", [("D1Q3", (1023, 1, 1)), ("D2Q5", (61, 37, 1)), ("D2Q5_DI", (64, 64, 1)),
                                        ("D3Q7", (13, 11, 29)), ("D3Q13", (16, 9, 11)), ("D3Q19", (13, 11, 9))])
def test_fp32_moments_and_sums_are_exact_sums_rounded_once(gpu_lib, name, shape):
    """Each FP64 result within 4 roundings of its exactly summed terms (and 2^-56 of the largest term, the
    integer form's unit)."""
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    D, q, cells = info["D"], info["q"], int(np.prod(shape))
    g = _cases(np.random.default_rng(3), q, cells).astype(np.float64)
    rho, u, red = np.empty(cells), np.empty((D, cells)), np.empty(D + 4)
    with lee.Solver(name, shape, 0.6, storage="f32") as sv:
        sv.set_populations(g)
        held = np.empty_like(g)
        sv.get_populations(held)
        assert np.array_equal(held, g)
        sv.moments(rho, u)
        sv.reduce(red)
    c = np.array(info["c"])
    unit = 2.0 ** -53
    for x in range(cells):
        most = np.abs(g[:, x]).max()
        want = math.fsum(g[:, x])
        assert abs(rho[x] - want) <= 4 * unit * abs(want) + 3 * 2.0 ** -56 * most
        for a in range(D):
            j = math.fsum(c[:, a] * g[:, x]) / info["rho0"]
            assert abs(u[a, x] - j) <= 4 * unit * abs(j) + 3 * 2.0 ** -56 * most
    # global sums: the integer units, and FP64 sums of one value per thread, group and velocity
    rows = 8 * math.sqrt(cells) * unit
    size = np.abs(g).sum()
    assert abs(red[0] - math.fsum(g.ravel())) <= rows * size
    for a in range(D):
        assert abs(red[1 + a] - math.fsum((c[:, a, None] * g).ravel())) <= rows * size
    f = np.array(info["f"])[:, None]
    want = math.fsum((g * g / f).ravel())
    assert abs(red[D + 2] - want) <= 8 * unit * math.sqrt(cells) * want
    assert red[D + 3] == 0


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("cells", [1, 255, 1025, 4099])
def test_non_finite_values_beside_finite_ones(gpu_lib, storage, cells):
    """Groups with infinities and NaN: counted, and every finite value of the same cells still summed."""
    lee = gpu_lib
    g = inputs.random_populations(3, cells, seed=2)
    kw = {"store_scale": 1024.0} if storage in ("f16", "bf16") else {}
    bad = [(0, 0, np.nan), (2, cells - 1, np.inf), (1, cells // 2, -np.inf)]
    for i, x, v in bad:
        g[i, x] = v
    red = np.empty(5)
    with lee.Solver("D1Q3", (cells, 1, 1), 0.6, storage=storage, **kw) as sv:
        sv.set_populations(g)
        held = np.empty_like(g)
        sv.get_populations(held)
        sv.reduce(red)
    fine = np.where(np.isfinite(held), held, 0.0)
    assert red[-1] == len(bad) == np.count_nonzero(~np.isfinite(held))
    np.testing.assert_allclose(red[0], math.fsum(fine.ravel()), rtol=0, atol=1e-14 * np.abs(fine).sum())
    np.testing.assert_allclose(red[1], math.fsum((fine[1] - fine[2])), rtol=0, atol=1e-14 * np.abs(fine).sum())
