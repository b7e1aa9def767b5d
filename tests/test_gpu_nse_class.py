"""GPU checks of the two-level streaming NSE kernels in class form (FP32 / FP64) against the
one-node-per-thread kernel: widths around the lane, strip and ghost widths, heights around the item
heights, 3D widths from the 65 columns they take.

Tolerance: both sum the same few dozen products per node in another order, two steps deep: 16 units in
the last place of each field's largest value (FP32 2e-6), FP64 1e-12."""

import numpy as np
import pytest

import gpu_cases as G
from test_gpu_lean import case, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


GRIDS2 = [(128, 1), (129, 2), (131, 7), (233, 16), (236, 33), (241, 9)]
GRIDS3 = [(65, 1, 1), (66, 5, 3), (95, 17, 2), (127, 4, 9), (128, 16, 4), (131, 9, 5)]


def compare(mm, lat, n, storage, steps, force=None):
    kw, prob = case(lat, "s", 2, list(n), storage)
    level = G.random_level(prob, np.random.default_rng(sum(n)))
    kern, _, _, a = run(mm, kw, level, steps=steps, force=force)
    direct, _, _, b = run(mm, kw, level, steps=steps, force="direct")
    assert "march" in kern and "direct" in direct
    tol = 1e-12 if storage == "fp64" else 2e-6
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= tol * np.abs(y).max(), (n, kern)


@pytest.mark.parametrize("storage", ["fp64", "fp32"])
@pytest.mark.parametrize("n", GRIDS2)
def test_2d(mm, n, storage):
    compare(mm, "D2Q9", n, storage, 2)


@pytest.mark.parametrize("force", [None, "lean3d_rows16"])
@pytest.mark.parametrize("n", GRIDS3)
def test_3d_fp32(mm, n, force):
    compare(mm, "D3Q19", n, "fp32", 2, force)


@pytest.mark.parametrize("n", GRIDS3)
def test_3d_fp64(mm, n):
    compare(mm, "D3Q19", n, "fp64", 2)
