"""GPU check that the class-form kernels cost no accuracy: their FP32 error (root mean square against the
FP64 levels of the same solve, which differ from the oracle by some 1e-15) is no larger than the
general pair form's, which takes every coefficient of the scheme rounded once.  Both errors are dominated
by what the coefficients' roundings do to the sum a uniform field gets in every step; the class forms keep
that sum, so theirs may only be smaller, up to the scatter of the single roundings (10 % allowed)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


def modes(rng, shape, amp):
    x = np.meshgrid(*[np.arange(s) / s for s in shape], indexing="ij")
    p = sum(rng.normal() * np.cos(2 * np.pi * sum(int(rng.integers(-4, 5)) * a for a in x) + rng.uniform(0, 6))
            for _ in range(8))
    return (amp * p / np.abs(p).max()).astype(np.float32).astype(np.float64)


def errors(mm, monkeypatch, kw, steps, level):
    """RMS error per field, class form and general form, over three initial levels."""
    out = {}
    for force in ("", "generic"):
        if force:
            monkeypatch.setenv("MMFD_FORCE_KERNEL", force)
        else:
            monkeypatch.delenv("MMFD_FORCE_KERNEL", raising=False)
        e2 = []
        for seed in range(3):
            fields = level(np.random.default_rng(seed), kw["n"][::-1])
            got = {}
            for storage in ("fp64", "fp32"):
                s = mm.Solver(mm.make_desc(**kw, storage=storage, temporal_depth=1, flags=mm.MMFD_FLAG_ALLOW_UNSTABLE))
                try:
                    s.set_fields(fields)
                    s.step(steps)
                    got[storage] = s.fields()
                finally:
                    s.close()
            e2.append([np.mean((a - b) ** 2) for a, b in zip(got["fp32"], got["fp64"])])
        out[force] = np.sqrt(np.mean(e2, axis=0))
    return out[""], out["generic"]


@pytest.mark.parametrize("a0", [0.0, 0.1, 0.25, 0.5])
@pytest.mark.parametrize("lat,n,d0,steps", [("D2Q9", [200, 160], None, 50), ("D2Q9", [200, 160], 0.3, 50),
                                            ("D3Q19", [66, 40, 36], None, 30), ("D3Q19", [129, 40, 36], None, 30)])
def test_nse(mm, monkeypatch, lat, n, d0, steps, a0):
    dim = len(n)
    # streaming momentum: (abar-, abar+) = (1 - a0) (a+, a-)
    kw = dict(pde="NSE", lattice=lat, levels=2, n=n, dt=1.0, dx=[1.0] * dim, ref=[1.0] + [0.0] * dim, a=(1.0, 0.0, 0.0),
              abar=(1.0 - a0, a0, 0.0))
    if d0:
        kw["d0"] = [d0] * dim
    cls, gen = errors(mm, monkeypatch, kw, steps,
                      lambda rng, sh: [1.0 + modes(rng, sh, 0.01)] + [modes(rng, sh, 0.05) for _ in range(dim)])
    assert np.all(cls <= 1.1 * gen), (cls, gen)


@pytest.mark.parametrize("a", [(0.95, 0.1, -0.05), (0.8, 0.4, -0.2), None])
@pytest.mark.parametrize("lat,n", [("D2Q9", [200, 160]), ("D3Q19", [130, 40, 36])])
@pytest.mark.parametrize("shared", [True, False])
def test_ncde(mm, monkeypatch, lat, n, a, shared):
    dim = len(n)
    kw = dict(pde="NCDE", lattice=lat, n=n, dt=0.8, dx=[1.0] * dim, diff=[0.15, 0, 0.05, 0],
              flux=([[0, 0.05, 0.1, 0]] * 3 if shared else [[0, 0.05, 0.1, 0], [0, -0.03, 0.1, 0], [0, 0, 0.06, 0.02]])[:dim])
    if a:
        kw.update(levels=2, a=a)
    else:
        kw.update(levels=3, a=(7 / 8, 0.0, 1 / 8), ahat=(1 / 8, 0.0, -1 / 8))
    cls, gen = errors(mm, monkeypatch, kw, 40, lambda rng, sh: [0.5 + modes(rng, sh, 0.2)])
    assert np.all(cls <= 1.1 * gen), (cls, gen)
