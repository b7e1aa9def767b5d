"""What the library's launchers ask of the CUDA runtime, on a runtime without a GPU
(fake_cudart/fake_cudart.cpp, loaded in a child process before the library): errors of one call stay
with it, and what a launch needs is set on the device that it goes to."""
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, sys
fake = C.CDLL({fake!r}, mode=C.RTLD_GLOBAL)
fake.fake_launches.restype = C.c_char_p
sys.path[:0] = [{root!r}, {tests!r}]
import numpy as np
import gpu_cases as G
from paper_2505_17057_gb300 import mmfd as M

def put(name, value):
    fake.fake_set(name.encode(), value)

def launches():
    # (device, kernel, (gx, gy, gz), threads, chained, cluster) since the last call
    out = []
    for line in fake.fake_launches().decode().splitlines():
        w = line.split()
        out.append((int(w[0]), w[1], tuple(int(v) for v in w[2:5]), int(w[5]), w[7] == "1", int(w[8])))
    fake.fake_clear()
    return out

class Solver:
    def __init__(self, **kw):
        self.desc = M.make_desc(**kw)
        self.h = M.mmfd_create(self.desc)
        self.nf = M.mmfd_get_info(self.h).nf
        n = kw["n"]
        self.data = [np.ones(tuple(reversed(n))) for _ in range(self.nf)]
        self.set()
        launches()
    def set(self):
        M.mmfd_set_fields(self.h, 0, [d.ctypes.data for d in self.data], M.MMFD_DEVICE, M.MMFD_DT_F64)
    def step(self, n):
        M.mmfd_step(self.h, n)
        return launches()

def solver(lat, pde, levels, n, storage="fp32", **more):
    kw, _ = G.case(lat, pde, levels, n, storage)
    kw.update(more)
    return Solver(**kw)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    home = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    lib = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(home, "include"), "-o", lib,
                    os.path.join(HERE, "fake_cudart", "fake_cudart.cpp")], check=True)

    def run(script):
        env = {k: v for k, v in os.environ.items() if k != "MMFD_FORCE_KERNEL"}
        p = subprocess.run([sys.executable, "-c", PRELUDE.format(fake=lib, root=ROOT, tests=HERE) + script],
                           capture_output=True, text=True, timeout=300, env=env)
        assert p.returncode == 0, p.stdout + p.stderr
    return run


def test_a_failed_launch_leaves_no_error_behind(fake):
    fake("""
for lat, pde, n in [("D2Q9", "NSE", [256, 64]), ("D2Q9", "LCDE", [200, 40]), ("D3Q19", "NCDE", [128, 9, 8]), ("D2Q9", "NCDE", [20, 2000])]:
    s = solver(lat, pde, 2, n)
    put("fail_next", 701)                      # out of resources
    try:
        s.step(1)
        raise SystemExit("the failed launch went unnoticed")
    except M.MMFDError as e:
        assert e.code == M.MMFD_ERR_CUDA, e.code
    s.set()                                    # the next calls run as if nothing had happened
    launches()
    assert len(s.step(1)) == 1
""")


def test_cluster_launch_on_every_device_and_the_way_back(fake):
    fake("""
for dev in (0, 1, 0, 3):
    fake.fake_device(dev)
    for storage, pde in [("fp32", "LCDE"), ("bf16", "NSE"), ("fp64", "LCDE")]:
        s = solver("D2Q9", pde, 2, [64, 48], storage)
        for got in (s.step(5), s.step(2)):         # one launch for all steps of a call
            assert len(got) == 1 and "k_cluster" in got[0][1] and got[0][0] == dev and got[0][5] == 16, got
# a cluster that the device does not take after all: the steps run one by one, and go on doing so
s = solver("D2Q9", "LCDE", 2, [64, 48])
for code in (912, 701, 1):
    put("fail_next", code)
    got = s.step(5)
    assert len(got) == 5 and all("k_direct" in g[1] for g in got), (code, got)
    s = solver("D2Q9", "LCDE", 2, [64, 48])
""")


def test_device_without_such_clusters(fake):
    fake("""
put("clusters", 0)
s = solver("D2Q9", "LCDE", 2, [64, 48])
assert ["k_direct" in g[1] for g in s.step(3)] == [True] * 3
fake.fake_device(1)
put("clusters", 1)                                  # another device of the machine has room for them
s = solver("D2Q9", "LCDE", 2, [64, 48])
got = s.step(3)
assert len(got) == 1 and "k_cluster" in got[0][1], got
""")


@pytest.mark.parametrize("lat,pde,levels,n,more", [
    ("D3Q19", "NSE", 2, [96, 20, 18], dict(dx=[1.0] * 3, a=(1.0, 0.0, 0.0), abar=(1.0, 0.0, 0.0))),
    ("D3Q19", "NCDE", 3, [70, 20, 18], dict(dx=[1.0] * 3)),
    ("D3Q19", "NSE", 2, [128, 20, 18], {}),
    ("D3Q7", "LCDE", 2, [256, 64, 20], {}),
    ("D2Q9", "NSE", 2, [256, 64], dict(dx=[1.0] * 2, a=(1.0, 0.0, 0.0), abar=(1.0, 0.0, 0.0), temporal_depth=3)),
    ("D2Q9", "NCDE", 2, [256, 64], dict(temporal_depth=1)),
    ("D2Q9", "LCDE", 2, [256, 64], dict(storage="fp64", temporal_depth=2)),
])
def test_marching_kernels_on_every_device(fake, lat, pde, levels, n, more):
    fake(f"""
kw = dict(flags=M.MMFD_FLAG_ALLOW_UNSTABLE, **{more!r})
storage = kw.pop("storage", "fp32")
grids = set()
for dev in (0, 1, 2, 0):
    fake.fake_device(dev)
    got = solver({lat!r}, {pde!r}, {levels}, {n!r}, storage, **kw).step(3)
    assert got and all(g[0] == dev and "k_march" in g[1] for g in got), got
    grids.add(tuple(g[1:] for g in got))
assert len(grids) == 1, grids
# as does a device that the library keeps no answer for
fake.fake_device(100)
assert solver({lat!r}, {pde!r}, {levels}, {n!r}, storage, **kw).step(3)
""")


def test_cluster_on_request_only_where_the_rule_takes_it(fake):
    fake("""
import os
os.environ["MMFD_FORCE_KERNEL"] = "cluster"

def takes(lat, pde, levels, n, storage, **more):
    try:
        s = solver(lat, pde, levels, n, storage, **more)
    except M.MMFDError as e:
        assert e.code == M.MMFD_ERR_UNSUPPORTED, e
        return False
    assert "k_cluster" in s.step(2)[0][1]
    put("fail_next", 912)
    try:
        s.step(2)
    except M.MMFDError as e:
        assert e.code == M.MMFD_ERR_CUDA
        return True
    raise SystemExit("went back to one launch per step in silence")

for lat, pde, levels in [c for c in G.SUPPORTED if c[0].startswith("D2")]:
    cost = {"LCDE": 2, "NCDE": 3, "NSE": 5}[pde] * (levels - 1)
    for storage in ("fp64", "fp32", "bf16"):
        f64 = storage == "fp64"
        if f64 and pde != "LCDE":
            assert not takes(lat, pde, levels, [16, 16], storage)
            continue
        most = 65536 // (cost * (5 if f64 else 1))
        assert takes(lat, pde, levels, [100, 33] if most >= 3300 else [100, most // 100], storage), (lat, pde, levels, storage)
        assert takes(lat, pde, levels, [127, most // 127], storage), (lat, pde, levels, storage)
        assert not takes(lat, pde, levels, [127, most // 127 + 1], storage), (lat, pde, levels, storage)
assert not takes("D2Q9", "LCDE", 2, [128, 16], "fp32")          # the marching kernels' widths
assert not takes("D3Q7", "LCDE", 2, [16, 16, 4], "fp32")
assert not takes("D2Q9", "LCDE", 2, [32, 16], "fp32", boundary="dirichlet")
""")


def test_autotuner_times_the_launches_that_steps_make(fake):
    fake("""
for lat, pde, levels, n, kernel in [("D2Q9", "NCDE", 2, [200, 40], "k_march2d"), ("D3Q19", "NSE", 2, [40, 9, 8], "k_direct"),
                                    ("D2Q9", "LCDE", 2, [64, 48], "k_cluster"), ("D2Q5", "LCDE", 3, [64, 48], "k_cluster")]:
    s = solver(lat, pde, levels, n)
    for before in (0, 2):                          # tuned before the first step, and after one
        if before:
            assert all(kernel in g[1] for g in s.step(before))
        info = M.mmfd_autotune(s.h)
        got = launches()
        assert info.candidates >= 1 and got
        # trials are programmatic dependents, as steps are (the cluster's one launch depends on nothing)
        assert all(kernel in g[1] and g[4] == (kernel != "k_cluster") for g in got), got[:3]
        if kernel == "k_cluster":
            assert (info.temporal_depth, info.rows_per_item, info.candidates) == (1, 0, 1)
            assert abs(info.ms_per_step - 1.0 / 64) < 1e-9     # the fake events lie 1 ms apart
    assert all(kernel in g[1] for g in s.step(2))
""")


def test_ctas_per_sm_of_the_plain_linear_step(fake):
    # (4 SMs and 1 MB of L2, so that small grids fill the GPU)
    fake("""
put("sms", 4)
put("l2_kb", 1024)

def ctas(lat, levels, n, storage="fp32"):
    grid = solver(lat, "LCDE", levels, n, storage, temporal_depth=1).step(1)[0][2]
    assert grid[1] == grid[2] == 1
    return -(-grid[0] // 4)                            # (equal segments may leave part of the last round idle)

for lat in ("D2Q5", "D2Q9"):
    # at 7 CTAs per SM that fit: four while two levels stay below 1.5 times the L2, three beyond
    assert ctas(lat, 2, [200, 256]) == 4               # 0.4 MB
    assert ctas(lat, 2, [256, 700]) == 4               # 1.44 MB
    assert ctas(lat, 2, [256, 800]) == 3               # 1.64 MB
    assert ctas(lat, 2, [700, 800]) == 3
    for levels, storage in [(2, "fp64"), (2, "bf16"), (3, "fp32")]:
        assert ctas(lat, levels, [256, 700], storage) == 7
# below that also three where they queue no more stages than four.  152 SMs: 4 (3) CTAs are 2432 (1824) warps;
# 768^2, 6 strips: items of 2 (3) rows, 2 (3) stages; 800^2, 7 strips: 3 (4) rows, 3 stages; 1024^2, 8 strips:
# 4 (5) rows, 3 (4) stages; 1100^2, 9 strips: 5 (6) rows, 4 stages
put("sms", 152)
put("l2_kb", 129 << 10)
fake.fake_device(2)
for n, ctas_of in [(768, 6 * 384 / 4), (800, 7 * 200 / 4), (1024, 8 * 256 / 4), (1100, -(-9 * 184 // 4))]:
    grid = solver("D2Q9", "LCDE", 2, [n, n], temporal_depth=1).step(1)[0][2]
    assert grid == (ctas_of, 1, 1), (n, grid)
put("sms", 4)
put("l2_kb", 1024)
put("ctas_per_sm", 2)                                  # a device with room for fewer (another one: kept per device)
fake.fake_device(1)
assert ctas("D2Q9", 2, [256, 800]) == 2
""")
