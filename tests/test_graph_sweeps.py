"""The op graph's executor built for the host: batches, shared and reused cotangent
arrays, sums in parts and the lean layout against a node-by-node sweep of the graph of
one node per primitive."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


@pytest.mark.parametrize("fwd,rev", [(24, 32), (4, 3)])
def test_batched_sweeps_equal_node_by_node(tmp_path, fwd, rev):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "graph_sweeps")
    src = os.path.join(HERE, "host_emulation", "graph_sweeps.cpp")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-DSTG_FWD_MAX=%d" % fwd,
                        "-DSTG_REV_MAX=%d" % rev, "-I", CUDA_INC, "-o", exe, src],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    assert "FAIL" not in r.stdout
    sums = [int(m) for m in re.findall(r"longest sum (\d+)", r.stdout)]
    assert (max(sums) > rev) == (rev == 3), r.stdout   # the small batches split sums
