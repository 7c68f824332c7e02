"""1/sqrt(r^2 + eps^2) as the potentials take it (`csrc/nb_fixed.cuh`), on the CPU over
all separations.  Compiles `tests/host/root_check.cpp`."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_root_over_all_separations(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "root_check")
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off",
                    os.path.join(HERE, "host", "root_check.cpp"), "-o", exe],
                   check=True, capture_output=True, timeout=600)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.splitlines()[-1].startswith("ok"), r.stdout
