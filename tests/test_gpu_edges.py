"""GPU checks of the marching kernels' edge stores: grid widths of every remainder modulo a lane's four
nodes, against the one-node-per-thread kernel.  Two steps, so that the second reads the first one's
ghost images (BF16: rounding may differ by a few units in the last place after two steps)."""

import numpy as np
import pytest

import gpu_cases as G

pytestmark = pytest.mark.gpu

GRIDS = [("D2Q9", "LCDE", (n, 5)) for n in (128, 129, 130, 131, 133)]
GRIDS += [("D2Q9", "NSE", (n, 3)) for n in (129, 134, 135, 252)]
GRIDS += [("D2Q9", "LCDE", (131, 1)), ("D2Q9", "NSE", (130, 1))]
GRIDS += [("D3Q7", "LCDE", (n, 5, 3)) for n in (128, 129, 130, 131)]
GRIDS += [("D3Q19", "NSE", (n, 4, 2)) for n in (129, 130, 135)] + [("D3Q19", "NSE", (131, 1, 3)), ("D3Q7", "LCDE", (133, 6, 1))]


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


@pytest.mark.parametrize("storage", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("lat,pde,n", GRIDS)
def test_edge_widths(mm, monkeypatch, lat, pde, n, storage):
    kw, prob = G.case(lat, pde, 2, list(n), storage)
    fields = G.random_level(prob, np.random.default_rng(n[0]))
    out = {}
    for force in ("", "direct"):
        if force:
            monkeypatch.setenv("MMFD_FORCE_KERNEL", force)
        else:
            monkeypatch.delenv("MMFD_FORCE_KERNEL", raising=False)
        s = mm.Solver(mm.make_desc(**kw))
        try:
            assert ("direct" in s.get_info().kernel.decode()) == (force == "direct")
            s.set_fields(fields)
            s.step(2)
            out[force] = s.fields(0)
        finally:
            s.close()
    refs = [1.0] + [0.0] * prob.dim if pde == "NSE" else [0.0]
    for f, (a, b) in enumerate(zip(out[""], out["direct"])):
        if storage == "bf16":
            assert np.all(np.abs(a - b) <= 4 * G.bf16_ulp(b - refs[f]) + 1e-5 * np.abs(b - refs[f]).max())
        else:
            assert np.abs(a - b).max() <= (1e-12 if storage == "fp64" else 2e-6) * max(np.abs(b).max(), 1e-30)
