"""backward_blocks (csrc/factor.cpp) on the CPU: [K | K + W^T | Rt^-1] of every
node becomes [E | K | Rt^-1] with E = Rt^-1 (K + W^T), in place, whatever the
number of host threads.  E is a sum of nu products; tolerance nu + 1 roundoffs of
the sum of their absolute values."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2212_01110_gb300", "csrc")
INC = os.path.join(HERE, "..", "include")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "spock_internal.h"
int main(int argc, char** argv) {
  const int nx = atoi(argv[3]), nu = atoi(argv[4]), threads = atoi(argv[5]);
  std::vector<double> v((size_t)atoll(argv[6]));
  FILE* f = fopen(argv[1], "rb");
  if (fread(v.data(), 8, v.size(), f) != v.size()) return 2;
  fclose(f);
  spock::backward_blocks(nx, nu, v, threads);
  f = fopen(argv[2], "wb");
  fwrite(v.data(), 8, v.size(), f);
  return fclose(f);
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.isdir(cuda):
        pytest.skip("g++ or the CUDA headers are missing")
    tmp = tmp_path_factory.mktemp("blocks")
    src, exe = tmp / "driver.cpp", tmp / "driver"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O2", "-g", "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
                    "-I", CSRC, "-I", INC, "-I", cuda, str(src), os.path.join(CSRC, "factor.cpp"), "-o", str(exe),
                    "-lpthread"], check=True)
    return tmp, exe


@pytest.mark.parametrize("nx,nu,nodes", [(1, 1, 1), (3, 2, 7), (2, 5, 130), (20, 7, 300)])
@pytest.mark.parametrize("threads", [1, 3])
def test_blocks(driver, nx, nu, nodes, threads):
    tmp, exe = driver
    rng = np.random.default_rng(nx + 10 * nu)
    kx, size = nu * nx, 2 * nu * nx + nu * nu
    nb = rng.standard_normal((nodes, size)) * 10.0 ** rng.uniform(-6, 6, (nodes, size))
    (tmp / "in").write_bytes(nb.tobytes())
    subprocess.run([str(exe), str(tmp / "in"), str(tmp / "out"), str(nx), str(nu), str(threads), str(nb.size)],
                   check=True)
    out = np.frombuffer((tmp / "out").read_bytes()).reshape(nodes, size)
    C, R = nb[:, kx:2 * kx].reshape(nodes, nu, nx), nb[:, 2 * kx:].reshape(nodes, nu, nu)
    bound = (nu + 1) * 2.0 ** -53 * (np.abs(R) @ np.abs(C)).reshape(nodes, kx)
    assert np.all(np.abs(out[:, :kx] - (R.astype(np.longdouble) @ C.astype(np.longdouble)).reshape(nodes, kx)) <= bound)
    assert np.array_equal(out[:, kx:2 * kx], nb[:, :kx])
    assert np.array_equal(out[:, 2 * kx:], nb[:, 2 * kx:])
