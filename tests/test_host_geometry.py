"""The evaluation's CTA of 128 threads is part of the whole-cluster evaluation's
geometry (a row is two 64-particle columns) and of the piece groups' counters: a
build with another size must not compile (it compiled and summed half of the
particles or counted two groups together)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("threads,ok", [(128, True), (64, False), (256, False)])
def test_cta_size(tmp_path, threads, ok):
    nvcc = next((c for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc") if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    r = subprocess.run([nvcc, "-std=c++17", "-O0", "-gencode", "arch=compute_103a,code=sm_103a",
                        f"-DNB_EVAL_TPB={threads}", "-c", os.path.join(HERE, "host", "sym_check.cu"),
                        "-o", str(tmp_path / "x.o")], capture_output=True, text=True, timeout=600)
    assert (r.returncode == 0) == ok, r.stdout + r.stderr
    if not ok:
        assert "128 threads" in r.stdout + r.stderr
