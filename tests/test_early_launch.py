"""Which grids are launched early (pdl): at most half a CTA per SM or at least
eight per SM, on any number of SMs (host code of the launch header alone)."""
import shutil
import subprocess

import pytest

from paper_2206_06996_gb300 import build

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include "launch.cuh"
int main(int argc, char** argv) {
  for (int i = 2; i < argc; ++i) printf("%d", (int)scr::early_grid(atoll(argv[i]), atoi(argv[1])));
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or shutil.which("/usr/local/cuda/bin/nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("early")
    (d / "p.cu").write_text(PROGRAM)
    r = subprocess.run([nvcc] + build.FLAGS + ["-I", build.CSRC, str(d / "p.cu"), "-o", str(d / "p")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "p")


@pytest.mark.parametrize("sms", [152, 148, 132, 76, 7])
def test_early_launches_follow_the_number_of_sms(program, sms):
    grids = [1, sms // 2, sms // 2 + 1, sms, 8 * sms - 1, 8 * sms, 100 * sms]
    out = subprocess.run([program, str(sms)] + [str(g) for g in grids], capture_output=True, text=True).stdout
    assert out == "".join(str(int(2 * g <= sms or g >= 8 * sms)) for g in grids) == "1100011"
