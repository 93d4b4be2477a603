"""The FP64 angle searches decided by the FP32 model, on the CPU, against the searches that evaluate every angle.

dp_search64.cuh is compiled for the host (tests/host) and run node by node on
random fields: the same code, the same bits of the value at it and the same
frozen foot are asked for.  Half of the coordinates put the foot of some table
angle within 2e-5 of a cell face, where a rounding decides which cell an angle
is in, with displacements from a fraction of a cell to the longest that a
dimension of 1,024 nodes allows (the FP32 displacement is off by 3e-5 of a cell
there), and the periodic angle and reduced node sets among them.

The bounds that the decisions rest on are measured against extended precision:
no error may be larger than its bound, whichever term dominates.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = os.path.join(ROOT, "tests", "host")
CSRC = os.path.join(ROOT, "paper_2407_14675_gb300", "csrc")


def compile_host(tmp, name):
    from paper_2407_14675_gb300 import build
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    exe = str(tmp / name)
    subprocess.run([shutil.which("g++") or "g++", "-std=gnu++17", "-O2", "-ffp-contract=off", "-I" + cuda, "-I" + HOST,
                    "-I" + CSRC, os.path.join(HOST, name + ".cpp"), "-o", exe], check=True)
    return exe


@pytest.fixture(scope="module")
def searches(tmp_path_factory):
    return compile_host(tmp_path_factory.mktemp("host"), "search64_host")


@pytest.mark.parametrize("kind", ["box", "polar", "band"])
@pytest.mark.parametrize("angles", [30, 64, 1024])
@pytest.mark.parametrize("cells,thrust", [(2, 3e-1), (30, 1e-2), (127, 1e-3), (450, 3e-4), (1022, 3e-4), (1022, 1e-3)])
def test_the_model_decides_as_fp64_does(searches, cells, thrust, angles, kind):
    count = 20000 if angles == 1024 else 100000
    out = subprocess.run([searches, "1", str(count), str(cells), str(thrust), str(angles), str(int(kind == "polar")),
                          str(int(kind == "band")), "2e-5"], check=True, capture_output=True, text=True).stdout
    n, model, wrong = map(int, out.split())
    assert n == count and wrong == 0
    assert model > 0.01 * count    # the model is what was tested


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    return compile_host(tmp_path_factory.mktemp("host"), "search64_bounds")


@pytest.mark.parametrize("polar", [0, 1])
@pytest.mark.parametrize("angles", [16, 30, 64, 1024])
def test_errors_stay_within_their_bounds(bounds, angles, polar):
    out = subprocess.run([bounds, "1", "400000", str(angles), str(polar)], check=True, capture_output=True, text=True).stdout
    slope, value, fraction, fp64, looked = map(float, out.split())
    assert looked > 300000
    assert max(slope, value, fraction, fp64) <= 1.0
