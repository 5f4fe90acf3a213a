"""Every order of the warps of a CTA of the 2D FP64 sweep that its waits allow (f64_waits_model.cpp, with the wait
thresholds the kernel is compiled with): nothing is overwritten before its readers are done, every block's moments are
written once, no warp waits for ever.  (units of rows, velocity groups, rows a unit, columns, moment warps); blocks of
three columns, so that 7 columns are the fewest with three blocks."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1712_01132_gb300", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs g++")
    exe = str(tmp_path_factory.mktemp("waits") / "model")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "f64_waits_model.cpp"), "-o", exe], check=True)
    return lambda *a: subprocess.run([exe] + [str(v) for v in a], check=True, capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("units,groups,rows,n1,moment_warps", [
    (1, 2, 2, 6, 2), (1, 2, 2, 7, 2), (1, 2, 2, 8, 2), (1, 2, 2, 9, 1), (1, 2, 2, 10, 2), (1, 3, 2, 8, 2), (1, 3, 2, 7, 3),
    (1, 2, 1, 7, 2), (1, 2, 1, 10, 2), (2, 1, 2, 8, 2), (3, 1, 1, 8, 2), (2, 2, 2, 7, 2), (2, 2, 1, 7, 2)])
def test_every_order_is_sound(model, units, groups, rows, n1, moment_warps):
    assert model(units, groups, rows, n1, moment_warps, 1)[0] == "ok"


@pytest.mark.parametrize("units,groups,rows,n1", [(1, 2, 2, 7), (1, 3, 2, 8), (1, 2, 1, 10), (2, 2, 2, 7)])
def test_the_model_sees_a_missing_wait(model, units, groups, rows, n1):
    """Without the wait of the moment warps for the unit's other groups, sums of two blocks meet in one buffer."""
    assert model(units, groups, rows, n1, 2, 0) == ["violation", "group", "sum"]
