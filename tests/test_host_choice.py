"""riccati_choice (csrc/spock_internal.h) on the CPU: one meaning of
SPOCK_RICCATI_KERNELS, which single problems and batches share."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2212_01110_gb300", "csrc")
INC = os.path.join(HERE, "..", "include")

DRIVER = r"""
#include "spock_internal.h"
int main() { return (int)spock::riccati_choice(); }
"""
AUTO, DIRECT, STAGED = 0, 1, 2


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.isdir(cuda):
        pytest.skip("g++ or the CUDA headers are missing")
    tmp = tmp_path_factory.mktemp("choice")
    src, exe = tmp / "driver.cpp", tmp / "driver"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-I", INC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    return exe


@pytest.mark.parametrize("value,want", [(None, AUTO), ("", AUTO), ("auto", AUTO), ("direct", DIRECT), ("d", DIRECT),
                                        ("staged", STAGED), ("tma", STAGED), ("grp", STAGED), ("t", STAGED),
                                        ("autos", STAGED)])
def test_choice(driver, value, want):
    env = {k: v for k, v in os.environ.items() if k != "SPOCK_RICCATI_KERNELS"}
    if value is not None:
        env["SPOCK_RICCATI_KERNELS"] = value
    assert subprocess.run([str(driver)], env=env).returncode == want


def test_one_reader():
    """No kernel file and no part of the solver reads the variable by itself."""
    readers = [f for f in sorted(os.listdir(CSRC))
               if re.search(r'getenv\("SPOCK_RICCATI_KERNELS"\)', open(os.path.join(CSRC, f)).read())]
    assert readers == ["spock_internal.h"]
