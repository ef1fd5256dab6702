"""The number of launches of a call, as the library reports it, against the rules of its header."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,shape,storage,bc,want", [
    ("D2Q5", (64, 33, 1), "f32", "periodic", {0: 0, 1: 1, 2: 1, 8: 1, 9: 2, 15: 3, 1000: 125}),
    ("D2Q5", (63, 33, 1), "f32", "periodic", {1: 1, 3: 1, 8: 1, 15: 3}),
    ("D2Q5", (64, 33, 1), "f16", "periodic", {1: 1, 3: 3, 8: 1, 12: 2, 15: 5}),
    ("D2Q5", (64, 33, 1), "bfp16", "periodic", {3: 3, 8: 2, 9: 3}),
    ("D2Q5", (64, 33, 1), "f64", "periodic", {8: 8}),
    ("D2Q5", (64, 33, 1), "f32", "open_zero", {8: 8}),
    ("D1Q3", (1000, 1, 1), "f64", "periodic", {1: 1, 2000: 1}),
    ("D1Q3", (1000, 1, 1), "f64", "open_sponge", {1: 1, 2000: 1}),
    ("D3Q7", (16, 9, 7), "f32", "periodic", {2: 1, 5: 3, 7: 4, 8: 8}),
    ("D3Q7", (64, 64, 72), "f32", "periodic", {5: 5, 8: 8}),
    ("D3Q7", (15, 9, 7), "f32", "periodic", {5: 5}),
    ("D3Q7", (132, 83, 75), "f32", "periodic", {3: 2, 4: 1, 8: 2, 43: 12}),
    ("D3Q19", (120, 84, 100), "f32", "periodic", {2: 1, 5: 3}),
])
def test_counts(gpu_lib, name, shape, storage, bc, want):
    kw = {"sponge_width": 7, "sponge_strength": 0.25} if bc == "open_sponge" else {}
    with gpu_lib.Solver(name, shape, 0.6, storage=storage, bc=bc, **kw) as sv:
        assert {n: sv.run_launches(n) for n in want} == want


def test_batch(gpu_lib):
    with gpu_lib.Batch("D2Q5", "f32", [(64, 32, 0.6), (132, 40, 0.8)]) as b:
        with pytest.raises(gpu_lib.LeeError):
            b.run_launches(8)  # no launch shape yet
        for unit, want in ((1, 17), (2, 9), (3, 7), (4, 3)):
            b.set_shape(256, 4, unit)
            assert b.run_launches(17) == want
