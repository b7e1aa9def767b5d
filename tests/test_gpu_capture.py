"""GPU check of mmfd_step under stream capture: the captured launches (plain dependencies instead of chained
ones; the cluster kernel's one launch), replayed once, give the bits of the same steps outside a capture,
for every kind of step kernel, on a solver that has and one that has not stepped before."""
import numpy as np
import pytest

import gpu_cases as G

pytestmark = pytest.mark.gpu

LBGK = dict(a=(1.0, 0.0, 0.0), abar=(1.0, 0.0, 0.0))
STEPS = [
    ("D2Q9", "LCDE", 2, [64, 48], "fp32", {}),                                             # cluster
    ("D2Q9", "NSE", 2, [40, 20], "bf16", {}),
    ("D2Q9", "NSE", 3, [50, 30], "fp64", {}),                                              # direct
    ("D3Q19", "LCDE", 2, [20, 9, 8], "fp32", {}),
    ("D2Q9", "NCDE", 3, [200, 33], "fp32", {}),                                            # marching kernels
    ("D2Q9", "LCDE", 2, [301, 40], "fp32", dict(temporal_depth=3)),
    ("D2Q9", "NSE", 2, [256, 40], "fp32", dict(dx=[1.0] * 2, temporal_depth=3, **LBGK)),
    ("D2Q9", "NSE", 2, [256, 40], "bf16", dict(dx=[1.0] * 2, temporal_depth=2, **LBGK)),
    ("D3Q19", "NSE", 2, [70, 12, 9], "fp32", dict(dx=[1.0] * 3, **LBGK)),
    ("D3Q7", "LCDE", 2, [130, 12, 9], "fp32", {}),
    ("D2Q9", "LCDE", 2, [200, 64], "fp32", dict(theta=0.5, temporal_depth=4, targets=[0, -1, -1, 0, 0.5])),
]


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


@pytest.mark.parametrize("lat,pde,levels,n,storage,more", STEPS)
def test_captured_steps_equal_the_same_steps(mm, lat, pde, levels, n, storage, more):
    import torch
    kw, prob = G.case(lat, pde, levels, n, storage)
    kw.update(flags=mm.MMFD_FLAG_ALLOW_UNSTABLE)
    if "targets" in more:
        del kw["a"], kw["ahat"]
    kw.update({k: v for k, v in more.items() if k != "theta"})
    make = dict(kw, **({"theta": more["theta"]} if "theta" in more else {}))
    fields = G.random_level(prob, np.random.default_rng(7))
    side = torch.cuda.Stream()
    plain = mm.Solver(mm.make_desc(**make))
    s = mm.Solver(mm.make_desc(**make), stream=side)
    try:
        assert plain.get_info().kernel == s.get_info().kernel
        for first in (True, False):
            if first:
                plain.set_fields(fields)
                s.set_fields(fields)
            else:
                plain.step(2)
                s.step(2)
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                s.step(7)
            with torch.cuda.stream(side):
                graph.replay()
            plain.step(7)
            torch.cuda.synchronize()
            assert s.get_info().steps_done == plain.get_info().steps_done
            for l in range(levels - 1):
                for a, b in zip(s.fields(l), plain.fields(l)):
                    assert np.isfinite(b).all() and np.array_equal(a, b), first
    finally:
        plain.close()
        s.close()
