"""The scale of 16-bit storage, which an FP32 estimate of the largest population decides where it can, against the
largest population of the FP64 equilibrium: at powers of two and next to them, and outside the estimate's range."""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SETS = [("D1Q3", (301, 1, 1)), ("D2Q5", (61, 37, 1)), ("D2Q5_DI", (64, 33, 1)), ("D3Q7", (13, 11, 29)), ("D3Q9", (13, 11, 9)),
        ("D3Q13", (16, 9, 11)), ("D3Q19", (13, 11, 9))]


def _largest(name, f, rho, u, theta):
    """max |g^eq / f*| as FP32, NaN left out."""
    g = np.abs(oracle.equilibrium(name, rho, u, theta) / np.asarray(f)[:, None])
    with np.errstate(over="ignore"):
        return float(np.float32(np.max(np.where(np.isnan(g), 0.0, g))))


def _scale(lee, name, shape, rho, u, theta, storage):
    with lee.Solver(name, shape, 0.6, storage=storage) as sv:
        sv.init_fields(rho, u, theta)
        return sv.store_scale


@pytest.mark.parametrize("name,shape", SETS)
def test_scale_at_powers_of_two(gpu_lib, name, shape):
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    cells, D = int(np.prod(shape)), info["D"]
    rng = np.random.default_rng(5)
    f0 = [rng.normal(size=cells), rng.normal(size=(D, cells)), rng.normal(size=cells)]
    m0 = np.max(np.abs(oracle.equilibrium(name, *f0) / np.asarray(info["f"])[:, None]))
    for k in (-20, -3, 0, 7):
        for d in (0.0, 2.0 ** -22, -2.0 ** -22, 2.0 ** -17, -2.0 ** -17, 0.3):
            f = [v * (2.0 ** k * (1 + d) / m0) for v in f0]
            m = _largest(name, info["f"], *f)
            want = 2.0 ** math.floor(math.log2(1024.0 / m))
            for storage in ("f16", "bf16"):
                assert _scale(lee, name, shape, *f, storage) == want, (k, d, storage)


@pytest.mark.parametrize("name,shape", SETS)
@pytest.mark.parametrize("what", ["zero", "tiny", "huge", "inf", "nan", "nan_u", "all_nan"])
def test_scale_of_special_fields(gpu_lib, name, shape, what):
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    cells, D = int(np.prod(shape)), info["D"]
    rng = np.random.default_rng(6)
    f = [rng.normal(size=cells), rng.normal(size=(D, cells)), rng.normal(size=cells)]
    if what == "zero":
        f = [0 * v for v in f]
    elif what == "tiny":
        f = [v * 1e-36 for v in f]
    elif what == "huge":
        f = [v * 1e33 for v in f]
    elif what == "inf":
        f[0][cells // 2] = np.inf
    elif what == "nan":
        f[0][cells // 2] = np.nan
    elif what == "nan_u":
        f[1][0, cells // 3] = np.nan
    else:
        f[0][:] = np.nan
    # (the oracle's order of operations turns an infinite field into NaN for some sets)
    m = np.inf if what == "inf" else _largest(name, info["f"], *f)
    want = 2.0 ** math.floor(math.log2(1024.0 / m)) if 0.0 < m < np.inf else 1.0
    assert _scale(lee, name, shape, *f, "f16") == want
