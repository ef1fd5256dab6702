"""Runs of the 1D set without a frame: one move of the populations against single steps."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["periodic", "open_zero"])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("nx", [1, 2, 3, 255, 1000, 70001])
def test_runs_equal_single_steps(gpu_lib, monkeypatch, bc, storage, nx):
    """Moves by less than, as much as and more than the grid, and runs that start in either copy."""
    lee = gpu_lib
    kw = {"store_scale": 1024.0} if storage in ("f16", "bf16") else {}
    g0 = inputs.random_populations(3, nx, seed=1)
    for n in (2, 3, nx + 1, 2 * min(nx, 300) + 5):
        if nx > 1000 and n > 1000:
            continue
        outs = []
        for single in (False, True):
            monkeypatch.delenv("LEE_TB_STEPS", raising=False)
            monkeypatch.setenv("LEE_SINGLE_STEP", "1" if single else "0")
            with lee.Solver("D1Q3", (nx, 1, 1), 0.8, storage=storage, bc=bc, **kw) as sv:
                sv.set_populations(g0)
                if single:
                    for _ in range(2 * n + 1):
                        sv.step(1)
                else:
                    sv.step(n)
                    sv.step(1)
                    sv.step(n)
                assert sv.steps_done == 2 * n + 1
                g = np.empty((3, nx))
                sv.get_populations(g)
                outs.append(g)
        assert np.array_equal(outs[0], outs[1]), n


def test_long_runs(gpu_lib):
    lee = gpu_lib
    nx, n = 1000, 10 ** 12 + 7
    g0 = inputs.random_populations(3, nx, seed=1)
    with lee.Solver("D1Q3", (nx, 1, 1), 0.8, storage="f64") as sv:
        sv.set_populations(g0)
        sv.step(n)
        g = np.empty((3, nx))
        sv.get_populations(g)
    assert np.array_equal(g, np.stack([g0[0], np.roll(g0[1], n % nx), np.roll(g0[2], -(n % nx))]))
    with lee.Solver("D1Q3", (nx, 1, 1), 0.8, storage="f64", bc="open_zero") as sv:
        sv.set_populations(g0)
        sv.step(n)
        sv.get_populations(g)
    assert np.array_equal(g[0], g0[0]) and not g[1:].any()
