"""GPU check that fusing the Jacobi sweeps of a theta-scheme step costs no accuracy: the FP32 error against
the 64-bit oracle, fused and with one sweep per launch.  The last four sweeps of either round alike and
earlier ones' rounding has shrunk by rho^4 (rho, the sweep's contraction, at most 0.7 here) by the end, so
the two errors are equal to within a few percent; 5 % is allowed.  (With every sweep starting from the
rounded r / d the fused error was 1.16, 2.24 and 1.53 times the other in the first, second and
last of these cases.)"""
import numpy as np
import pytest

from oracle import oracle as orc
from oracle import params as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


@pytest.mark.parametrize("scale,dt,theta", [(1, 8, 0.5), (2, 4, 0.5), (1, 8, 0.9), (1, 2, 0.5), (5, 6, 0.3), (1, 8, 0.0)])
def test_fused_sweeps_are_as_accurate_as_single_ones(mm, scale, dt, theta):
    nx, ny, steps = 192, 160, 6
    K = [[0.02 * scale, 0.005 * scale], [0.005 * scale, 0.01 * scale]]
    u = [0.1 / scale ** 0.5, 0.05 / scale ** 0.5]
    a = P.two_level_from_a0(0.0)
    prob = P.problem_lcde("D2Q9", 2, [nx, ny], dt, [1.0, 1.0], K, u, a)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    err = {0: [], 1: []}
    for seed in range(3):
        rng = np.random.default_rng(seed)
        p = sum(rng.normal() * np.cos(2 * np.pi * (int(rng.integers(0, 9)) * x / nx + int(rng.integers(0, 9)) * y / ny) +
                                      rng.uniform(0, 6)) for _ in range(12))
        phi = 1.0 + (0.5 * p / np.abs(p).max()).astype(np.float32).astype(np.float64)
        ref = orc.theta_run(prob, [phi], steps, theta)[0]
        for depth in err:
            s = mm.Solver(mm.make_desc("LCDE", "D2Q9", 2, [nx, ny], dt, [1.0, 1.0], K=K, u=u, a=a, storage="fp32",
                                       ref=[1.0], theta=theta, temporal_depth=depth))
            try:
                s.set_fields([phi])
                s.step(steps)
                assert s.get_info().temporal_depth == (4 if depth == 0 else 1)
                err[depth].append(np.mean((s.fields()[0] - ref) ** 2))
            finally:
                s.close()
    fused, single = (np.sqrt(np.mean(err[d])) for d in (0, 1))
    assert fused <= 1.05 * single, (fused, single)
