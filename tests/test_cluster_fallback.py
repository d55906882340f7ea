"""The choice of a smaller cluster where the device refuses a size (lb_cluster.h), on the host: a compiled
program in whose place of a launch stands a function that takes clusters up to a given size."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include <cstdio>
#include <cstdlib>
#include "lb_cluster.h"
int main(int, char** argv) {
  const int want = atoi(argv[1]), most = atoi(argv[2]);
  const cudaError_t refusal = (cudaError_t)atoi(argv[3]);
  int tries = 0, last = 0;
  const cudaError_t e = gblb::launch_in_clusters(want, [&](int size) {
    ++tries;
    last = size;
    return size <= most ? cudaSuccess : refusal;
  });
  printf("%d %d %d\\n", (int)e, last, tries);
}
"""
INVALID_CLUSTER_SIZE, OUT_OF_RESOURCES, ILLEGAL_ADDRESS = 912, 701, 700


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda = next((d for d in ("/usr/local/cuda/include", "/usr/include") if os.path.exists(os.path.join(d, "driver_types.h"))), None)
    if cxx is None or cuda is None:
        pytest.skip("no C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("cluster")
    (d / "p.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-I", cuda, "-I", os.path.join(ROOT, "paper_0903_5067_gb300", "csrc"), str(d / "p.cpp"), "-o",
                    str(d / "p")], check=True)
    return lambda *a: tuple(int(v) for v in subprocess.run([str(d / "p"), *map(str, a)], check=True, capture_output=True,
                                                           text=True).stdout.split())


@pytest.mark.parametrize("want,most,refusal,status,size,tries", [
    (16, 16, INVALID_CLUSTER_SIZE, 0, 16, 1),  # taken as asked
    (16, 8, INVALID_CLUSTER_SIZE, 0, 8, 2),
    (10, 9, OUT_OF_RESOURCES, 0, 8, 2),
    (9, 1, INVALID_CLUSTER_SIZE, 0, 1, 5),
    (6, 2, OUT_OF_RESOURCES, 0, 1, 3),  # 6, 3, 1
    (1, 0, OUT_OF_RESOURCES, OUT_OF_RESOURCES, 1, 1),  # nothing smaller
    (16, 8, ILLEGAL_ADDRESS, ILLEGAL_ADDRESS, 16, 1),  # not a matter of the size
])
def test_smaller_clusters(program, want, most, refusal, status, size, tries):
    assert program(want, most, refusal) == (status, size, tries)
