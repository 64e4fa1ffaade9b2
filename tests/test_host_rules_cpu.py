"""Rules that decide where a kernel may store and in which order, compiled for
the host from the kernels' own headers (host_rules.cu): faults in them would be
stores out of range, to memory of another GPU, or in an undefined order, so they
are tested without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _nvcc():
    for cand in (os.environ.get("CUDA_HOME"), "/usr/local/cuda"):
        if cand and os.path.exists(os.path.join(cand, "bin", "nvcc")):
            return os.path.join(cand, "bin", "nvcc")
    return shutil.which("nvcc")


@pytest.fixture(scope="module")
def host_rules(tmp_path_factory):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("host_rules") / "host_rules")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2209_08189_gb300", "csrc"),
           os.path.join(ROOT, "tests", "host_rules.cu"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stdout + res.stderr
    return exe


@pytest.mark.parametrize("group", ["result_arrays", "scatter_boxes", "conv_schedule"])
def test_host_rules(host_rules, group):
    run = subprocess.run([host_rules, group], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0 and run.stdout.strip() == "OK", run.stdout + run.stderr
