"""The FP64 evaluation's pair vectors (`csrc/nb_fixed.cuh`, fx_vectors) component by
component on the CPU: in systems thin along an axis, chains, bulk motion and at the
ends of the range no component of jerk or snap may be less exact against its own
summands than in plain doubles.  Compiles `tests/host/components_check.cpp`."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_components_as_exact_as_doubles(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "components_check")
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off",
                    os.path.join(HERE, "host", "components_check.cpp"), "-o", exe],
                   check=True, capture_output=True, timeout=600)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.splitlines()[-1].startswith("ok"), r.stdout
