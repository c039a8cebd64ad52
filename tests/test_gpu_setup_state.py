"""What set-ups leave behind and share: lists of long rows for any number of
levels, device memory over numeric re-set-ups."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

import fsi_inputs as F

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


def _pool_bytes(attr=7):
    """Bytes in use in the device's memory pool, which the library allocates
    from (attribute 7: current, 8: the highest since it was last reset)."""
    path = next(l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l)
    rt = C.CDLL(path)
    pool, v = C.c_void_p(), C.c_uint64()
    assert rt.cudaDeviceGetDefaultMemPool(C.byref(pool), torch.cuda.current_device()) == 0
    assert rt.cudaMemPoolGetAttribute(pool, attr, C.byref(v)) == 0
    return v.value


@pytest.mark.parametrize("precision", [pkg.SCR_FP64, pkg.SCR_MIXED])
@pytest.mark.parametrize("loops", [0, 2])
def test_numeric_resetups_keep_the_device_memory(precision, loops):
    """A Newton iteration's numeric re-set-up and solve hold the same device
    memory each time, with V-cycles replayed by the host's loops (whose
    vectors are the set-up's) and with device loops."""
    s = F.tube_system("tube_mini")
    used = []
    with pkg.BlockSolver(precision=precision, graph_krylov=loops) as sol:
        sol.setup(s.A, s.B, s.C, s.D)
        for _ in range(5):
            sol.update_values(s.A, s.B, s.C, s.D)
            sol.solve(s.b.copy())
            torch.cuda.synchronize()
            used.append(_pool_bytes())
    assert used[0] > 0 and used[1:] == used[:1] * 4
