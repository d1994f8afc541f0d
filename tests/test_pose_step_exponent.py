"""The bias correction of the pose step takes its exponent from the caller's device memory: whatever
that holds, its loop ends. The helper is compiled here as plain C++ (no GPU runs it)."""
import os
import re
import subprocess

import pytest

from paper_2601_00705_gb300 import build

MAIN = """
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#define __device__
#define __forceinline__ inline
%s
int main(int, char** argv) {
  std::printf("%%.17g\\n", power(std::strtod(argv[1], nullptr), std::strtoll(argv[2], nullptr, 10)));
  return 0;
}
"""


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    text = open(os.path.join(build.CSRC, "track.cu")).read()
    found = re.search(r"__device__ __forceinline__ double power\(.*?\n}\n", text, re.S)
    out = tmp_path_factory.mktemp("power")
    (out / "power.cpp").write_text(MAIN % found.group(0))
    subprocess.run(["g++", "-O1", "-std=c++17", str(out / "power.cpp"), "-o", str(out / "power")],
                   check=True)
    return str(out / "power")


# The exponent is the step count plus one: counts of -2 and below (memory that was never zeroed)
# and 2^31 - 1 included.
@pytest.mark.parametrize("step", [0, 1, 29, 1000, -1, -2, -7, 2 ** 31 - 1, -2 ** 31])
@pytest.mark.parametrize("base", [0.0, 0.5, 0.9, 0.999])
def test_power_ends_for_every_step_count(helper, base, step):
    r = subprocess.run([helper, repr(base), str(step + 1)], capture_output=True, text=True,
                       timeout=10, check=True)
    try:
        expect = base ** (step + 1)
    except (ZeroDivisionError, OverflowError):
        expect = float("inf")
    assert float(r.stdout) == pytest.approx(expect, rel=1e-12 * max(1, abs(step)) + 1e-15)
