"""The block fixed-point pair terms of the FP64 evaluation (`csrc/nb_fixed.cuh`)
on the CPU: against long double and beside the same terms in plain doubles, over
separations, velocities, accelerations and softenings of any scale.  Compiles
`tests/host/fixed_check.cpp`; every class's rms error must not exceed the double
form's, and what vanishes, is excluded or is not finite must stay so."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_pair_terms(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "fixed_check")
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off",
                    os.path.join(HERE, "host", "fixed_check.cpp"), "-o", exe],
                   check=True, capture_output=True, timeout=600)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.splitlines()[-1].startswith("ok"), r.stdout
