"""The library's host code on a stand-in for the CUDA runtime (CPU): the
order of work across streams and what a call leaves behind when it fails.
host_runtime.cpp says how the stand-in works and what each scenario does."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2401_11029_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    include = os.path.join(CUDA, "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    out = tmp_path_factory.mktemp("host_runtime")
    exe = str(out / "host_runtime")
    flags = ["-O1", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I",
             include, "-include", "cuda_runtime.h"]
    # (launches that no scenario reaches have no definition)
    subprocess.run([cxx, *flags, "-x", "c++", os.path.join(HERE, "host_runtime.cpp"),
                    os.path.join(CSRC, "runtime.cu"), os.path.join(CSRC, "grammar.cpp"),
                    "-o", exe, "-no-pie", "-Wl,--unresolved-symbols=ignore-all",
                    "-ldl", "-lpthread"], check=True)
    return exe


@pytest.mark.parametrize("scenario", ["batch_across_streams", "failed_readouts",
                                      "failed_products", "failed_buffers",
                                      "failed_batch_tables", "readout_without_map",
                                      "budget_after_failed_readouts", "failed_growths",
                                      "load_without_roomy_sets", "per_thread_stream"])
def test_scenario(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
