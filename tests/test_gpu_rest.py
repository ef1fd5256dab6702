"""Rest populations of the sets with one moving shell: the collision conserves them cell by cell, so a
step leaves them alone and both state copies hold them."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,shape", [("D1Q3", (1030, 1, 1)), ("D2Q5", (132, 9, 1)), ("D2Q5_DI", (37, 6, 1)),
                                        ("D3Q7", (36, 5, 4)), ("D3Q7_DI", (13, 6, 5)), ("D3Q9", (16, 5, 4)),
                                        ("D3Q13", (13, 6, 5))])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16", "bfp16"])
def test_rest_populations_keep_their_bits(gpu_lib, name, shape, storage):
    """After runs that end in either copy (1, 2 and 9 steps) the rest populations are those stored at
    the start."""
    lee = gpu_lib
    info = lee.lee_velset_info(name)
    cells = int(np.prod(shape))
    g = inputs.random_populations(info["q"], cells, seed=4)
    with lee.Solver(name, shape, 0.7, storage=storage, **({"store_scale": 1024.0} if storage in ("f16", "bf16") else {})) as sv:
        sv.set_populations(g)
        first, now = np.empty_like(g), np.empty_like(g)
        sv.get_populations(first)
        for n in (1, 2, 9):
            sv.step(n)
            sv.get_populations(now)
            assert np.array_equal(now[0], first[0]), n
        if info["D"] > 1:  # (the 1D set moves its populations without relaxing them)
            assert not np.array_equal(np.sort(now[1:].ravel()), np.sort(first[1:].ravel()))


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("before", [1, 2, 3])
def test_network_takes_over_from_a_sponge_fallback(gpu_lib, storage, before):
    """The fallback frame damps rest populations from copy to copy; a network installed after it goes on
    from the current ones, as a handle does that starts from that state."""
    lee = gpu_lib
    shape, cells = (40, 33, 1), 40 * 33
    params = np.load(lee.__path__[0] + "/data/boundary_d2q5_tau0.6.npy").astype(np.float32)
    rho, u, th = inputs.random_fields(shape, 2, 6)
    kw = dict(storage=storage, bc="open_learned", sponge_width=4, sponge_strength=0.5)
    with lee.Solver("D2Q5", shape, 0.6, **kw) as a, lee.Solver("D2Q5", shape, 0.6, **kw) as b:
        a.init_fields(rho, u, th)
        a.step(before)
        g = np.empty((5, cells))
        a.get_populations(g)
        a.set_boundary_mlp(params)
        b.set_boundary_mlp(params)
        b.set_populations(g)
        out = [np.empty_like(g), np.empty_like(g)]
        for n in (1, 2):
            for sv, o in zip((a, b), out):
                sv.step(n)
                sv.get_populations(o)
            assert np.array_equal(out[0], out[1])
