"""The spreading kernel lists, for a brick of grid points, the atoms of a range of cells: exactly in single precision,
that range holds every atom whose stencil reaches the brick (no GPU; the driver says how).  Without the margin that the
range carries for rounding, the same check finds violations, so it can see them."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_01377_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

pytestmark = pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA_INC),
                                reason="no compiler or CUDA headers")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("spread") / "spread_range")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CUDA_INC, "-I", CSRC,
                    os.path.join(ROOT, "tests", "host_sanitize", "spread_range_driver.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    return exe


def test_every_reaching_atom_is_in_the_range(driver):
    r = subprocess.run([driver], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
    assert "violations 0" in r.stdout


def test_the_check_sees_a_range_without_margin(driver):
    r = subprocess.run([driver, "0.0"], capture_output=True, text=True, timeout=600)
    assert r.returncode == 1 and "violations 0" not in r.stdout, r.stdout
