"""The files that guard a committed traffic figure (no GPU): for every kernel name a solver reports, bench.py
hashes the sources that hold the kernels run under it, their launchers and all they include."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2505_17057_gb300", "csrc")


def text(name):
    with open(os.path.join(CSRC, name)) as fh:
        return fh.read()


# kernel name -> the global functions that run under it
RUNS = {
    "k_march2d": {"k_march2d", "k_march2d_nse", "k_march2d_ncde"},
    "k_march2d_tb": {"k_march2d_tb"},
    "k_march2d_nse_s": {"k_march2d", "k_march2d_nse"},
    "k_march2d_tb_nse": {"k_march2d_tb_nse", "k_march2d_nse"},
    "k_march2d_src": {"k_march2d"},
    "k_march2d_theta": {"k_theta", "k_march2d"},
    "k_march3d": {"k_march3d", "k_march3d_nse", "k_march3d_ncde"},
    "k_march3d_nse_s": {"k_march3d", "k_march3d_nse"},
    "k_direct": {"k_direct", "k_cluster"},
}


def globals_in(files):
    """Names of the __global__ functions defined in the files."""
    found = set()
    for f in files:
        found |= set(re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text(f)))
    return found


@pytest.mark.parametrize("name", sorted(RUNS))
def test_sources_hold_the_kernels(name):
    files = bench.kernel_sources(name)
    assert RUNS[name] <= globals_in(files), (RUNS[name] - globals_in(files), files)


@pytest.mark.parametrize("name", sorted(bench.KERNEL_SOURCES))
def test_sources_are_closed_under_includes(name):
    files = set(bench.kernel_sources(name))
    for f in files:
        for inc in re.findall(r'#include "([^"]+)"', text(f)):
            assert inc in files or not os.path.exists(os.path.join(CSRC, inc)), (f, inc)
    # the heights of the work items, which set the halo rows a launch reads
    if "march" in name:
        assert "launch.cuh" in files


def test_a_header_changes_the_hash(monkeypatch, tmp_path):
    import shutil
    base = tmp_path / "pkg"                       # the headers beside the package are included by relative path
    shutil.copytree(CSRC, base / "csrc")
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    before = {k: bench.kernel_source_sha(k) for k in RUNS}
    monkeypatch.setattr(bench, "CSRC", str(base / "csrc"))
    assert {k: bench.kernel_source_sha(k) for k in RUNS} == before
    with open(base / "csrc" / "nse_class.cuh", "a") as fh:
        fh.write("\n")
    after = {k: bench.kernel_source_sha(k) for k in RUNS}
    assert {k for k in RUNS if after[k] != before[k]} == {"k_march2d", "k_march2d_nse_s", "k_march2d_tb_nse", "k_march3d",
                                                          "k_march3d_nse_s"}
