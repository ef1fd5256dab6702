"""The 2D row pipeline: eight steps per launch against single steps, at the edges of its strips and
segments."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu

# narrower than a strip's halo, one strip less one chunk, one strip, one more chunk, several strips; rows
# fewer than the levels, odd, and many segments
SHAPES = [(4, 3, 1), (12, 5, 1), (108, 7, 1), (112, 16, 1), (116, 9, 1), (240, 4, 1), (260, 41, 1), (456, 1003, 1),
          # widths that are not multiples of 4
          (1, 3, 1), (2, 5, 1), (3, 4, 1), (13, 9, 1), (113, 16, 1), (115, 7, 1), (222, 33, 1), (457, 1003, 1)]


def _state(lee, monkeypatch, shape, storage, n, g0, single, name="D2Q5", **kw):
    for k in ("LEE_TB_STEPS", "LEE_SINGLE_STEP"):
        monkeypatch.delenv(k, raising=False)
    if single:
        monkeypatch.setenv("LEE_SINGLE_STEP", "1")
    g = np.empty_like(g0)
    with lee.Solver(name, shape, 0.55, storage=storage, **kw) as sv:
        sv.set_populations(g0)
        for k in n if isinstance(n, tuple) else (n,):
            sv.step(k)
        sv.get_populations(g)
    return g


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("name", ["D2Q5", "D2Q5_DI"])
def test_fp32_runs_equal_single_steps(gpu_lib, monkeypatch, name, shape):
    """Runs of one launch of eight, of every remainder, of a replayed graph (77 steps: 9 launches of
    eight, one of four, one single step) and of calls that start in either copy."""
    lee = gpu_lib
    g0 = inputs.random_populations(5, int(np.prod(shape)), seed=5)
    for n in (8, 11, 14, 77, (77, 77, 8, 8)):
        a = _state(lee, monkeypatch, shape, "f32", n, g0, False, name)
        b = _state(lee, monkeypatch, shape, "f32", n, g0, True, name)
        assert np.array_equal(a, b), n


@pytest.mark.parametrize("shape", [(4, 3, 1), (12, 5, 1), (104, 7, 1), (112, 16, 1), (120, 9, 1), (264, 41, 1), (456, 203, 1)])
@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_16bit_launch_of_eight_is_two_of_four(gpu_lib, monkeypatch, storage, shape):
    """The state is rounded to the storage after every four steps, whether one launch takes four or eight, so
    runs give the same bits however the calls cut them at multiples of four."""
    lee = gpu_lib
    g0 = inputs.random_populations(5, int(np.prod(shape)), seed=6)
    kw = {"store_scale": 1024.0}
    a = _state(lee, monkeypatch, shape, storage, 24, g0, False, **kw)
    b = _state(lee, monkeypatch, shape, storage, (4, 16, 4), g0, False, **kw)
    held = _state(lee, monkeypatch, shape, storage, 0, g0, False, **kw)
    f = _state(lee, monkeypatch, shape, "f32", 4, held, True)
    for _ in range(5):  # D2Q5's weights and the scale are powers of two: the FP32 steps round alike
        f = _state(lee, monkeypatch, shape, "f32", 4, _state(lee, monkeypatch, shape, storage, 0, f, False, **kw), True)
    c = _state(lee, monkeypatch, shape, storage, 0, f, False, **kw)
    assert np.array_equal(a, b) and np.array_equal(a, c)
