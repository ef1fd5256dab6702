"""Calls that the caller captures into a CUDA graph of its own: each replay advances the state, wherever the launches of a call
can leave it in the copy they found it in."""
import numpy as np
import pytest

from paper_1601_08103_gb300 import inputs

pytestmark = pytest.mark.gpu

EVERY = (2, 3, 4, 5, 6, 7, 8, 9, 10, 15, 16, 20, 24, 31, 72)
EVEN = (2, 4, 6, 8, 10, 16, 72)
CASES = [("D1Q3", (1000, 1, 1), "f64", "periodic", EVERY), ("D1Q3", (30000, 1, 1), "f32", "open_zero", EVERY),
         ("D1Q3", (1000, 1, 1), "f32", "open_sponge", EVERY), ("D2Q5", (64, 33, 1), "f32", "periodic", EVERY),
         ("D2Q5", (63, 33, 1), "f32", "periodic", EVERY), ("D2Q5", (64, 33, 1), "f64", "periodic", EVEN),
         ("D2Q5", (64, 33, 1), "f32", "open_zero", EVEN),
         # 16-bit states, rounded every four steps: an even number of fours and ones
         ("D2Q5", (64, 33, 1), "f16", "periodic", (2, 5, 7, 8, 10, 16, 24, 32, 72)),
         ("D2Q5", (64, 33, 1), "bfp16", "periodic", (2, 5, 7, 8, 10, 16, 24, 72)),
         ("D3Q7", (16, 9, 7), "f32", "periodic", EVEN), ("D3Q7", (132, 83, 75), "f32", "periodic", (3, 4, 7, 8, 12, 16, 20)),
         ("D3Q7", (193, 107, 110), "f32", "periodic", (2, 4, 6, 8, 12, 20)),
         ("D3Q19", (120, 84, 100), "f32", "periodic", EVEN)]


def _solver(lee, name, shape, storage, bc, stream, g0):
    kw = {"store_scale": 1024.0} if storage in ("f16", "bf16") else {}
    if bc == "open_sponge":
        kw.update(sponge_width=7, sponge_strength=0.25)
    sv = lee.Solver(name, shape, 0.57, storage=storage, bc=bc, stream=stream, **kw)
    sv.set_populations(g0)
    return sv


@pytest.mark.parametrize("name,shape,storage,bc,counts", CASES)
def test_each_replay_advances_the_state(gpu_lib, name, shape, storage, bc, counts):
    import torch

    lee = gpu_lib
    st = torch.cuda.Stream()
    q, cells = lee.lee_velset_info(name)["q"], int(np.prod(shape))
    g0 = inputs.random_populations(q, cells, seed=1)
    a, b = np.empty_like(g0), np.empty_like(g0)
    for n in counts:
        with _solver(lee, name, shape, storage, bc, st, g0) as sv:
            sv.sync()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                sv.step(n)
            with torch.cuda.stream(st):
                for _ in range(3):
                    graph.replay()
            st.synchronize()
            sv.get_populations(a)
        with _solver(lee, name, shape, storage, bc, st, g0) as sv:
            for _ in range(3):
                sv.step(n)
            sv.get_populations(b)
        assert np.array_equal(a, b), n


@pytest.mark.parametrize("mode", ["launch", "graph"])
@pytest.mark.parametrize("unit", [1, 2, 4])
def test_batch(gpu_lib, mode, unit):
    import torch

    lee = gpu_lib
    st = torch.cuda.Stream()
    domains = [(64, 32, 0.6), (132, 40, 0.8)]
    fields = [inputs.random_fields((nx, ny, 1), 2, 5) for nx, ny, _ in domains]

    def batch():
        b = lee.Batch("D2Q5", "f32", domains, stream=st)
        b.set_shape(256, 4, unit)
        for d, f in enumerate(fields):
            b.init_fields(d, *f)
        b.sync()
        return b

    def populations(b):
        out = [np.empty((5, nx * ny)) for nx, ny, _ in domains]
        for d, o in enumerate(out):
            b.get_populations(d, o)
        return out

    for n in (2 * unit, 8, 16, 24, 72):
        with batch() as b:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                b.step(n, mode)
            with torch.cuda.stream(st):
                for _ in range(3):
                    graph.replay()
            st.synchronize()
            got = populations(b)
        with batch() as b:
            for _ in range(3):
                b.step(n, mode)
            want = populations(b)
        for x, y in zip(got, want):
            assert np.array_equal(x, y), n
