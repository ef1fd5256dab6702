"""Moments and global sums of populations of one sign and size, whose integer sums are the longest: every mantissa
bit set, and fields at rest, which store one number for all velocities of a shell (and, in 16 bits, of the set)."""
import math

import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu

SETS = [("D1Q3", (1023, 1, 1)), ("D2Q5", (61, 37, 1)), ("D2Q5_DI", (64, 64, 1)), ("D3Q7", (13, 11, 29)),
        ("D3Q7_DI", (13, 11, 29)), ("D3Q9", (16, 9, 17)), ("D3Q13", (16, 9, 11)), ("D3Q19", (13, 11, 9))]
STORAGES = ["f32", "f16", "bf16", "bfp16"]
UNIT = 2.0 ** -53


def _check(lee, name, shape, storage, fill):
    """Sums of one sign lose nothing by cancellation: each result within 64 roundings of the exact sum of its terms,
    which covers a thread's and a block's additions at these sizes and the coefficients."""
    info = lee.lee_velset_info(name)
    D, q, cells = info["D"], info["q"], int(np.prod(shape))
    rho, red, g = np.empty(cells), np.empty(D + 4), np.empty((q, cells))
    with lee.Solver(name, shape, 0.6, storage=storage) as sv:
        fill(sv, info)
        sv.get_populations(g)
        sv.moments(rho)
        sv.reduce(red)
    c, f, beta = np.array(info["c"]), np.array(info["f"])[:, None], np.array(info["beta"])
    np.testing.assert_allclose(rho, [math.fsum(v) for v in g.T], rtol=64 * UNIT)
    size = math.fsum(np.abs(g).ravel())
    np.testing.assert_allclose(red[0], math.fsum(g.ravel()), rtol=0, atol=64 * UNIT * size)
    for a in range(D):
        np.testing.assert_allclose(red[1 + a], math.fsum((c[:, a, None] * g).ravel()), rtol=0, atol=64 * UNIT * size)
    w = 0.5 * ((c ** 2).sum(1) + beta)[:, None]
    np.testing.assert_allclose(red[D + 1], math.fsum((w * g).ravel()), rtol=0, atol=64 * UNIT * math.fsum((w * np.abs(g)).ravel()))
    np.testing.assert_allclose(red[D + 2], math.fsum((g * g / f).ravel()), rtol=64 * UNIT)
    assert red[D + 3] == 0


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("name,shape", SETS)
def test_all_mantissa_bits_set(gpu_lib, name, shape, sign, storage):
    """The stored values are all the same, with every mantissa bit of the storage set."""

    def fill(sv, info):
        bits = {"f32": 24, "f16": 11, "bf16": 8, "bfp16": 15}[storage]
        v = sign * (2.0 - 2.0 ** (1 - bits)) * 2.0 ** -7
        f = np.array(info["f"])[:, None] if storage in ("f16", "bf16") else 1.0
        sv.set_populations(np.full((info["q"], int(np.prod(shape))), v) * f)

    _check(gpu_lib, name, shape, storage, fill)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("isentropic", [True, False])
@pytest.mark.parametrize("name,shape", SETS)
def test_fields_at_rest(gpu_lib, name, shape, isentropic, storage):
    """A uniform density with its isentropic temperature and one without any; a pulse on top of it."""
    lee = gpu_lib
    cells = int(np.prod(shape))
    for rho in (np.full(cells, 1e-3), 1e-3 + inputs.gaussian_pulse(shape, 8e-4, 4.0, [n / 2 for n in shape])):

        def fill(sv, info):
            th = (info["gamma"] - 1.0) * info["theta0"] / info["rho0"] * rho if isentropic else np.zeros(cells)
            sv.init_fields(np.ascontiguousarray(rho), np.zeros((info["D"], cells)), np.ascontiguousarray(th))

        _check(lee, name, shape, storage, fill)
