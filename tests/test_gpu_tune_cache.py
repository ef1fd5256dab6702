"""The autotuner's file: a shape measured on the kernels in use is taken from it, one of earlier kernels is measured anew."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TUNE = """
import paper_1601_08103_gb300 as lee
with lee.Batch("D2Q5", "f32", [(68, 36, 0.6), (140, 44, 0.7)]) as b:
    print(b.tune_shape()["us_per_step"])
"""


def _tuned(path):
    env = {k: v for k, v in os.environ.items() if k not in ("LEE_TB_STEPS", "LEE_SINGLE_STEP")}
    out = subprocess.run([sys.executable, "-c", TUNE], env=dict(env, LEE_AUTOTUNE_CACHE=str(path)), cwd=ROOT,
                         capture_output=True, text=True, check=True, timeout=120)
    return float(out.stdout)


def test_shapes_of_earlier_kernels_are_not_used(gpu_lib, tmp_path):
    path = tmp_path / "shapes"
    first = _tuned(path)
    key, *shape = path.read_text().split()
    assert float(shape[-1]) == pytest.approx(first, abs=1e-3)
    shape[-1] = "12345.0"
    path.write_text(" ".join([key, *shape]) + "\n")
    assert _tuned(path) == 12345.0
    path.write_text(" ".join(["batch2/" + key.split("/", 1)[1], *shape]) + "\n")
    assert _tuned(path) < 1000.0
    assert path.read_text().splitlines()[-1].split()[0] == key
