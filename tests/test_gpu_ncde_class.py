"""GPU checks of the NCDE kernels in class form (equal spacings; FP32 / FP64) against the
one-node-per-thread kernel: one flux polynomial on every axis or one per axis, two and three levels,
widths around the lane, strip and ghost widths.

Tolerance: the same products in another order, two steps deep: 16 units in the last place of the largest
value (FP32 2e-6), FP64 1e-12."""

import numpy as np
import pytest

import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


def run(mm, kw, level, levels, force, monkeypatch):
    if force:
        monkeypatch.setenv("MMFD_FORCE_KERNEL", force)
    else:
        monkeypatch.delenv("MMFD_FORCE_KERNEL", raising=False)
    s = mm.Solver(mm.make_desc(**kw))
    try:
        s.set_fields(level)
        if levels == 3:
            s.set_fields([0.98 * x for x in level], 1)
        s.step(2)
        return s.fields(0)[0], s.get_info().kernel.decode()
    finally:
        s.close()


GRIDS = [("D2Q9", n) for n in [(128, 1), (129, 2), (131, 7), (236, 33), (241, 9)]]
GRIDS += [("D3Q19", n) for n in [(65, 1, 1), (66, 5, 3), (127, 4, 9), (128, 8, 4), (131, 9, 5)]]


@pytest.mark.parametrize("storage", ["fp64", "fp32"])
@pytest.mark.parametrize("shared", [True, False])
@pytest.mark.parametrize("levels", [2, 3])
@pytest.mark.parametrize("lat,n", GRIDS)
def test_ncde_class(mm, monkeypatch, lat, n, levels, shared, storage):
    kw, prob = G.case(lat, "NCDE", levels, n, storage)
    kw["dx"] = [1.0] * len(n)
    if shared:
        kw["flux"] = [kw["flux"][0]] * len(n)
    level = G.random_level(prob, np.random.default_rng(sum(n)))
    a, kern = run(mm, kw, level, levels, None, monkeypatch)
    b, direct = run(mm, kw, level, levels, "direct", monkeypatch)
    assert "march" in kern and "direct" in direct
    assert np.abs(a - b).max() <= (1e-12 if storage == "fp64" else 2e-6) * np.abs(b).max()
