"""Which scenes the one-cluster binning takes, and with how many CTAs: up to 8192 Gaussians and 512 cells, a CTA for every 64
Gaussians up to 16, and none where the device (or the share of it that the process has) cannot hold a cluster of that size -
those scenes take the grid-wide kernels, as larger ones do.  The rule is host code: compiled and called here."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def ctas(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("route")
    (d / "route.cpp").write_text('#include <cstdio>\n#include "gs_device.cuh"\nint main() {\n  long long n; int cells, limit;\n'
                                 '  while (scanf("%lld %d %d", &n, &cells, &limit) == 3) printf("%d\\n", gs::cluster_ctas(n, cells, limit));\n}\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2609_05255_b200", "csrc"), str(d / "route.cpp"), "-o", str(d / "route")], check=True)

    def call(rows):
        text = "\n".join("%d %d %d" % r for r in rows)
        return [int(v) for v in subprocess.run([str(d / "route")], input=text, capture_output=True, text=True, check=True).stdout.split()]
    return call


def test_cluster_sizes(ctas):
    expect = {(1, 1): 1, (64, 1): 1, (65, 1): 2, (128, 1): 2, (129, 1): 4, (512, 1): 8, (513, 1): 16, (1000, 512): 16, (8192, 512): 16,
              (8193, 1): 0, (1000, 513): 0}
    assert ctas([(n, c, 16) for n, c in expect]) == list(expect.values())


@pytest.mark.parametrize("limit", [0, 1, 2, 4, 8, 16])
def test_a_cluster_that_does_not_fit_is_not_asked_for(ctas, limit):
    ns = [1, 64, 65, 100, 300, 600, 2000, 8192]
    full = ctas([(n, 12, 16) for n in ns])
    for n, want, got in zip(ns, full, ctas([(n, 12, limit) for n in ns])):
        assert got == (want if want <= limit else 0)
        assert got == 0 or n <= 1024 * got                       # the kernel gives a thread one Gaussian at most
