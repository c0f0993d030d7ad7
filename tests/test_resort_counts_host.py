"""CPU check of the number of movers that the near-sorted re-sort takes from its scan.

The scan runs over [all | stayers | movers] as one array of 32-bit words, so its last word is twice
the number of particles and wraps from 2^31 particles on, while the word before the movers may
not.  The difference has to be the number of movers all the same (a context takes up to 2^32 - 2
particles); widened before the subtraction it was negative and taken for no movers at all.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_13394_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "pm_internal.cuh"
int main(int argc, char** argv) {
  for (int i = 1; i + 1 < argc; i += 2)
    std::printf("%lld\n", (long long)pmnu::scan_difference((uint32_t)std::strtoull(argv[i], nullptr, 10),
                                                           (uint32_t)std::strtoull(argv[i + 1], nullptr, 10)));
  return 0;
}
"""


@pytest.fixture(scope="module")
def movers(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("movers")
    src, exe = d / "movers.cu", d / "movers"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True, capture_output=True)

    def run(pairs):
        args = [str(x) for p in pairs for x in p]
        out = subprocess.run([str(exe), *args], check=True, capture_output=True, text=True).stdout
        return [int(x) for x in out.split()]
    return run


def test_movers_of_any_capacity(movers):
    want, pairs = [], []
    for n in (1, 1000, 2 ** 31 - 1, 2 ** 31, 2 ** 31 + 7, 3 * 10 ** 9, 2 ** 32 - 2):
        for m in sorted({0, 1, n // 3, n - 1, n}):
            stay = n - m
            words = np.cumsum(np.array([n, stay, m], dtype=np.uint64)).astype(np.uint32)  # as the device holds them
            want.append(m)
            pairs.append((int(words[1]), int(words[2])))
    assert movers(pairs) == want


def test_the_kernels_use_it():
    text = open(os.path.join(CSRC, "k_sort.cu")).read()
    body = text[text.index("int64_t movers_of("):]
    body = body[:body.index("\n}")]
    assert "scan_difference(" in body and "(int64_t)bstart3" not in body
