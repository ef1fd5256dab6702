"""Global sums of populations that do not lie on whole vectors: the same bits from every start, pitch and width, since each
thread adds the same cells."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("name,cells", [("D1Q3", 1), ("D1Q3", 5), ("D2Q5", 1023), ("D2Q5", 4100), ("D3Q7", 1026), ("D3Q19", 2049)])
def test_starts_and_pitches(gpu_lib, name, cells, storage):
    import torch

    lee = gpu_lib
    info = lee.lee_velset_info(name)
    q, D = info["q"], info["D"]
    dtype = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage]
    values = torch.from_numpy(np.random.default_rng(cells).normal(size=(q, cells))).to("cuda", dtype)
    results = set()
    for start in (0, 1, 2, 4, 7):
        for pitch in (cells, cells + 1, (cells + 63) // 64 * 64):
            buf = torch.full((start + q * pitch + 8,), float("nan"), dtype=dtype, device="cuda")
            for i in range(q):
                buf[start + i * pitch:start + i * pitch + cells] = values[i]
            out = torch.empty(D + 4, dtype=torch.float64, device="cuda")
            lee.lee_reduce_noalloc(name, storage, buf[start:], cells, pitch, out)
            results.add(tuple(out.cpu().tolist()))
    assert len(results) == 1
    (got,) = results
    assert got[D + 3] == 0
