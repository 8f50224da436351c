"""The order of the library's calls to the CUDA runtime, without a GPU: its
objects are linked with a runtime that executes nothing before it has to
(fake_cudart.h), and the scenarios of host_calls.cpp check what it saw."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="session")
def host_calls(libgsr_path, tmp_path_factory):
    from paper_2507_15683_gb300 import build as B
    exe = str(tmp_path_factory.mktemp("host_calls") / "host_calls")
    objs = [os.path.join(B.OBJ_DIR, os.path.basename(s) + ".o") for s in B._sources()]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    cmd = [B.NVCC, "-std=c++17", "-O1", "-cudart", "none", "-I", B.INCLUDE, "-I", HERE,
           os.path.join(HERE, "host_calls.cpp")] + objs + ["-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return exe


@pytest.mark.parametrize("scenario", ["batches_of_changing_size", "two_devices", "early_starts", "sizes_in_pairs", "other_scenes",
                                      "no_memory_for_graphs", "callers_capture"])
def test_host_calls(host_calls, scenario):
    r = subprocess.run([host_calls, scenario], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
