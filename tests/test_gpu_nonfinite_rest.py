"""A rest population that is not finite: it stays in its cell where a step leaves rest populations alone, is counted there, and
does not change any other population."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("bc", ["periodic", "open_zero", "open_sponge"])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("name,shape", [("D2Q5", (64, 33, 1)), ("D2Q5_DI", (37, 20, 1)), ("D3Q7", (12, 11, 9)),
                                        ("D3Q9", (12, 11, 9)), ("D3Q13", (12, 11, 9))])
def test_it_stays_in_its_cell(gpu_lib, name, shape, storage, bc, value):
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    D, q, cells = info["D"], info["q"], int(np.prod(shape))
    x = cells // 2 + shape[0] // 2
    g0 = inputs.random_populations(q, cells, seed=4)
    kw = {"store_scale": 1024.0} if storage == "f16" else {}
    if bc == "open_sponge":
        kw.update(sponge_width=2, sponge_strength=0.25)
    out = []
    for g in (g0, g0.copy()):
        if out:
            g[0, x] = value
        with lee.Solver(name, shape, 0.6, storage=storage, bc=bc, **kw) as sv:
            sv.set_populations(g)
            now, red, rho = np.empty_like(g), np.empty(D + 4), np.empty(cells)
            for n in (1, 2, 9):
                sv.step(n)
            sv.get_populations(now)
            sv.reduce(red)
            sv.moments(rho)
        out.append((now, red, rho))
    (a, ra, ma), (b, rb, mb) = out
    assert ra[D + 3] == 0 and rb[D + 3] == 1
    assert not np.isfinite(b[0, x]) and not np.isfinite(mb[x])
    a[0, x] = b[0, x] = 0.0
    assert np.array_equal(a, b)
    ma[x] = mb[x] = 0.0
    assert np.array_equal(ma, mb)
