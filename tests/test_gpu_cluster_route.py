"""GPU checks that the cluster kernel is the one that runs (MMFD_FORCE_KERNEL=cluster fails where it does
not), against the direct kernel bit for bit, up to the widest grids and the last row count its rule
takes."""
import numpy as np
import pytest

import gpu_cases as G

pytestmark = pytest.mark.gpu

CASES = [(lat, pde, lev, st) for lat, pde, lev in G.SUPPORTED if lat.startswith("D2")
         for st in ("fp64", "fp32", "bf16") if st != "fp64" or pde == "LCDE"]


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


def run(mm, monkeypatch, force, kw, fields, steps):
    monkeypatch.setenv("MMFD_FORCE_KERNEL", force)
    s = mm.Solver(mm.make_desc(**kw))
    try:
        s.set_fields(fields)
        for n in steps:
            s.step(n)
        return [s.fields(l) for l in range(1 if kw["levels"] == 2 else 2)]
    finally:
        s.close()


@pytest.mark.parametrize("lat,pde,levels,storage", CASES)
def test_cluster_runs_and_equals_the_direct_kernel(mm, monkeypatch, lat, pde, levels, storage):
    cost = {"LCDE": 2, "NCDE": 3, "NSE": 5}[pde] * (levels - 1) * (5 if storage == "fp64" else 1)
    most = 65536 // cost
    for n in [(65, 17), (100, min(33, most // 100)), (127, most // 127), (13, 40)]:
        kw, prob = G.case(lat, pde, levels, list(n), storage)
        if storage == "bf16" and n[0] % 2:
            kw.update(flags=mm.MMFD_FLAG_STOCHASTIC_ROUND, seed=5)
        fields = G.random_level(prob, np.random.default_rng(n[0]))
        a = run(mm, monkeypatch, "cluster", kw, fields, [4, 3])
        b = run(mm, monkeypatch, "direct", kw, fields, [7])
        assert all(np.array_equal(p, q) for x, y in zip(a, b) for p, q in zip(x, y)), n


@pytest.mark.parametrize("lat,pde,levels,storage", [("D2Q9", "NSE", 2, "fp32"), ("D2Q9", "LCDE", 3, "fp64"),
                                                    ("D2Q9", "NCDE", 3, "bf16")])
def test_autotuning_a_cluster_solver_leaves_its_levels(mm, monkeypatch, tmp_path, lat, pde, levels, storage):
    monkeypatch.setenv("MMFD_FORCE_KERNEL", "cluster")
    kw, prob = G.case(lat, pde, levels, [90, 25], storage)
    fields = G.random_level(prob, np.random.default_rng(3))
    s, plain = mm.Solver(mm.make_desc(**kw)), mm.Solver(mm.make_desc(**kw))
    try:
        for x in (s, plain):
            x.set_fields(fields)
            x.step(3)
        info = s.autotune(str(tmp_path / "tune.txt"))
        assert info.candidates == 1 and info.ms_per_step > 0 and s.get_info().steps_done == 3
        for steps in (0, 4):
            s.step(steps)
            plain.step(steps)
            for l in range(levels - 1):
                assert all(np.array_equal(a, b) for a, b in zip(s.fields(l), plain.fields(l))), (steps, l)
    finally:
        s.close()
        plain.close()
