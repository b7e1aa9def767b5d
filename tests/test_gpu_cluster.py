"""GPU checks of the cluster kernel (all steps of a small 2D solve in one launch): the same bits as one
launch per step, for every lattice, PDE, level count and storage, at row counts around the cluster's
sixteen CTAs and widths around the vector and ghost widths."""
import numpy as np
import pytest

import gpu_cases as G

pytestmark = pytest.mark.gpu

CASES = [(lat, pde, lev) for lat, pde, lev in G.SUPPORTED if lat.startswith("D2")]
GRIDS = [(8, 1), (9, 2), (13, 15), (16, 16), (31, 17), (47, 33), (64, 40), (33, 70)]


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


def run(mm, kw, fields, steps):
    s = mm.Solver(mm.make_desc(**kw))
    try:
        s.set_fields(fields)
        for n in steps:
            s.step(n)
        info = s.get_info()
        return [s.fields(l) for l in range(1 if kw["levels"] == 2 else 2)], info.steps_done
    finally:
        s.close()


@pytest.mark.parametrize("storage", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("lat,pde,levels", CASES)
def test_cluster_equals_single_steps(mm, lat, pde, levels, storage):
    for n in GRIDS:
        kw, prob = G.case(lat, pde, levels, list(n), storage)
        if storage == "bf16" and n[0] % 2:
            kw.update(flags=mm.MMFD_FLAG_STOCHASTIC_ROUND, seed=5)
        fields = G.random_level(prob, np.random.default_rng(n[0] + 100 * n[1]))
        a, da = run(mm, kw, fields, [5])                  # one launch
        b, db = run(mm, kw, fields, [1] * 5)              # one launch per step
        c, dc = run(mm, kw, fields, [2, 1, 2])
        assert da == db == dc == 5
        for x, y, z in zip(a, b, c):
            assert all(np.array_equal(p, q) and np.array_equal(p, r) for p, q, r in zip(x, y, z)), (n, storage)
