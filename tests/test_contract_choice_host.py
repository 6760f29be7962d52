"""The rule that chooses between the two tensor-core contraction kernels (tcs_wins of
csrc/contract_tcs.cu), on the host: random tile lists against the rule restated, in the
order in which plans build them and shuffled, and that a column window is scanned once
however many tiles share it.  tests/host_tcs_rule.cu is compiled with nvcc; it makes
no CUDA call."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_choice_of_the_contraction_kernel(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path / "host_tcs_rule"
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2",
                        "-I", os.path.join(ROOT, "paper_2506_10526_gb300", "csrc"),
                        "-I", os.path.join(ROOT, "include"), "-o", str(out),
                        os.path.join(HERE, "host_tcs_rule.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(out)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    lists, bad, wins, ratio, _ = r.stdout.split()
    assert int(bad) == 0
    assert 0.05 < int(wins) / int(lists) < 0.95
    # scanned tile by tile the two take the same time; 2560 tiles of 5 windows
    assert float(ratio) < 0.5
