"""The library's host code against a CUDA runtime made of host memory (tests/host_driver_check.cu, tests/fake_cudart.cc): what a handle holds
after an allocation failed, which buffers a replayed graph may use, what a handle remembers between budgets.  Nothing
runs on a GPU."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess

import pytest

from paper_2508_20403_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    nvcc = build._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc on this machine")
    build.build()
    out = str(tmp_path_factory.mktemp("host_driver") / "check")
    flags = [f for f in build.NVCC_FLAGS if f not in ("-O3", "-lineinfo")]
    objs = [o for o in sorted(glob.glob(os.path.join(build.BUILD, "*.o"))) if os.path.basename(o) != "pdg_api.o"]
    subprocess.run([nvcc, *flags, "-O1", "-Xcompiler", "-D_GLIBCXX_ASSERTIONS", "-cudart", "none",
                    os.path.join(HERE, "host_driver_check.cu"), os.path.join(HERE, "fake_cudart.cc"), *objs, "-o", out], check=True)
    return out


def _run(checker, name, **env):
    r = subprocess.run([checker, name], capture_output=True, text=True, timeout=300, env={**os.environ, **env})
    assert r.returncode == 0, (name, r.returncode, r.stderr[-2000:])
    return r


@pytest.mark.parametrize("name", ["oom_join", "oom_table", "oom_tiers", "oom_table_keeps_size"])
def test_calls_after_a_failed_allocation(checker, name):
    """Each allocation of a recovery fails once (candidate buffers, the join's table and its growth, the tiers'
    buffers); the call reports it, the next call has every buffer its kernels use, nothing is freed twice."""
    _run(checker, name)


def test_a_graph_ends_with_its_buffers(checker):
    """A budget, captured and replayed; a larger one that runs out of memory; the first again: the buffers are new ones
    of the old sizes, so the old graph must not run."""
    _run(checker, "graph_of_old_buffers")


def test_late_weights_need_no_more_memory(checker):
    """Host weights that follow on a second stream need the places of the mirror images; where memory is short of them
    but enough for the plain order, init still succeeds."""
    _run(checker, "late_weights_memory")


def test_report_of_a_failed_index_check(checker):
    _run(checker, "failed_index_check", PDG_DEBUG_BOUNDS="1")


def test_tiers_are_remembered_by_budget(checker):
    """A budget whose candidates fill the join's cells is decided by the tiers, and from the start the next time; smaller
    budgets of the same handle keep the join."""
    _run(checker, "tiers_by_budget")
