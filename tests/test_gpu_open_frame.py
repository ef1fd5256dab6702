"""Rest populations at open edges, where a frame damps them and every other cell leaves them alone: each population of a
run against the same run of one-cell-per-thread kernels, and the rest ones against their own recursion, at the edges of vectors, blocks and
frames."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu

# widths of whole vectors and blocks, odd ones, grids that are frame but for one cell, and grids of one warp
SHAPES = [("D2Q5", (32, 9, 1), 4), ("D2Q5", (136, 37, 1), 7), ("D2Q5", (37, 5, 1), 2), ("D2Q5_DI", (8, 40, 1), 3),
          ("D2Q5_DI", (100, 64, 1), 31), ("D3Q7", (24, 10, 6), 2), ("D3Q7", (13, 9, 11), 4), ("D3Q9", (40, 7, 8), 3),
          ("D3Q13", (16, 9, 7), 3), ("D3Q19", (16, 9, 7), 3), ("D1Q3", (20000, 1, 1), 100)]


def _run(lee, name, shape, storage, g0, steps, **kw):
    out = []
    with lee.Solver(name, shape, 0.7, storage=storage, **({"store_scale": 1024.0} if storage in ("f16", "bf16") else {}), **kw) as sv:
        sv.set_populations(g0)
        for n in steps:
            sv.step(n)
            g = np.empty_like(g0)
            sv.get_populations(g)
            out.append(g)
    return out


def _damp(shape, D, w, smax, dtype):
    """The frame's factor of each cell, with the roundings of the storage's arithmetic."""
    d = np.zeros(shape[::-1], int)
    for a in range(D):
        x = np.arange(shape[a])
        e = np.maximum(np.maximum(w - x, x - (shape[a] - 1 - w)), 0)
        d = np.maximum(d, e.reshape([-1 if b == a else 1 for b in (2, 1, 0)]))
    r = dtype(d.ravel()) / dtype(w)
    # 1 - (smax r) r with one rounding: exact in long double for these short factors
    return dtype(np.longdouble(1) - np.longdouble(dtype(smax) * r) * np.longdouble(r))


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16", "bfp16"])
@pytest.mark.parametrize("bc", ["open_zero", "open_sponge"])
@pytest.mark.parametrize("name,shape,w", SHAPES)
def test_vectors_equal_single_cells(gpu_lib, monkeypatch, name, shape, w, bc, storage):
    lee = gpu_lib
    kw = dict(bc=bc, **(dict(sponge_width=w, sponge_strength=0.25) if bc == "open_sponge" else {}))
    info = lee.lee_velset_info(name)
    g0 = inputs.random_populations(info["q"], int(np.prod(shape)), seed=6)
    steps = (1, 1, 2, 9)
    a = _run(lee, name, shape, storage, g0, steps, **kw)
    monkeypatch.setenv("LEE_FORCE_SCALAR", "1")
    b = _run(lee, name, shape, storage, g0, steps, **kw)
    for n, (x, y) in enumerate(zip(a, b)):
        assert np.array_equal(x, y), n


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("name,shape,w", [s for s in SHAPES if s[0] != "D3Q19"])
def test_rest_populations_are_damped_in_the_frame_alone(gpu_lib, name, shape, w, storage):
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    dtype = np.float64 if storage == "f64" else np.float32
    g0 = inputs.random_populations(info["q"], int(np.prod(shape)), seed=6).astype(dtype).astype(np.float64)
    damp = _damp(shape, info["D"], w, 0.25, dtype)
    assert (damp == 1).any() and (damp != 1).any()
    want = g0[0].astype(dtype)
    for n, g in zip((1, 1, 2, 5), _run(lee, name, shape, storage, g0, (1, 1, 2, 5), bc="open_sponge", sponge_width=w, sponge_strength=0.25)):
        for _ in range(n):
            want = want * damp
        if storage == "f32":  # (FP64's factor may be rounded twice in long double: one unit per step)
            assert np.array_equal(g[0], want.astype(np.float64))
        else:
            np.testing.assert_allclose(g[0], want, rtol=1e-14)
