"""What set-ups leave behind and share: lists of long rows for any number of
levels."""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2206_06996_gb300 as pkg  # noqa: E402
from paper_2206_06996_gb300 import build as cuda_build  # noqa: E402

pkg.load_library(build_if_missing=True)

HERE = os.path.dirname(os.path.abspath(__file__))


def test_long_row_lists_of_more_patterns_than_a_page(tmp_path):
    """130 patterns (a hierarchy queues two per level, without a bound on its
    levels): every one gets its list."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    lib = cuda_build.build()
    exe = str(tmp_path / "long_rows_client")
    cmd = [nvcc] + cuda_build.FLAGS + ["-I", cuda_build.CSRC, os.path.join(HERE, "long_rows_client.cu"), "-cudart",
                                       "shared", "-o", exe, lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
