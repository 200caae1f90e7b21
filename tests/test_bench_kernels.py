"""The bench names the 2-D FP32 kernels by the launchers' rules (no GPU)."""
import importlib

import pytest


@pytest.mark.parametrize("shape,r,t,dims,tile,name", [
    ("box", 2, 1, (16384, 16384), [1, 32, 256], "cu2d_march"), ("box", 2, 2, (16384, 16384), [1, 64, 128], "cu2d_march"),
    ("star", 3, 2, (1000, 1000), [1, 64, 64], "cu2d_march"), ("box", 3, 2, (1000, 1000), [1, 64, 64], "cu2d_sweep"),
    ("box", 3, 1, (512, 512), [1, 16, 32], "cu2d_sweep"), ("box", 3, 1, (512, 500), [1, 16, 32], "cu2d_march"),
    ("box", 3, 1, (16384, 16384), [1, 64, 128], "cu2d_march"), ("box", 2, 3, (2000, 2000), [1, 64, 64], "cu2d_sweep"),
    ("star", 4, 1, (2000, 2000), [1, 64, 64], "cu2d_sweep")])
def test_fp32_kernel_names(shape, r, t, dims, tile, name):
    bench = importlib.import_module("bench")
    info = {"path": 1, "t": t, "precision_name": "native", "tile": tile}
    assert bench.kernel_name(info, 2, "f32", shape, r, dims) == name
    assert bench.kernel_name(info, 2, "f64", shape, r, dims) == "cu2d_sweep"
