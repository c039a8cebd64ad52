"""What set-ups leave behind and share: lists of long rows for any number of
levels, device memory over numeric re-set-ups, set-ups of several threads, set-ups with
other timed kernels, timed kernels of BF16 levels; and set-ups of operators far
from the usual scales."""
import ctypes as C
import os
import shutil
import subprocess
import threading

import numpy as np
import pytest

import fsi_inputs as F
from oracle import amg
from oracle.sparse import to_csr

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


def _pool_bytes(attr=7, reset=False):
    """Bytes in use in the device's memory pool, which the library allocates
    from (attribute 7: current, 8: the highest since it was last reset)."""
    path = next(l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l)
    rt = C.CDLL(path)
    pool, v = C.c_void_p(), C.c_uint64()
    assert rt.cudaDeviceGetDefaultMemPool(C.byref(pool), torch.cuda.current_device()) == 0
    if reset:
        assert rt.cudaMemPoolSetAttribute(pool, attr, C.byref(v)) == 0
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


def _dense(n, seed):
    """A full matrix of n rows with a dominant diagonal, as 1x1 blocks."""
    a = np.random.default_rng(seed).uniform(-1.0, 1.0, (n, n)) + 2.0 * n * np.eye(n)
    return a, F.BSR(1, 1, n, n, np.arange(n + 1, dtype=np.int32) * n, np.tile(np.arange(n, dtype=np.int32), n),
                    a.reshape(-1))


def test_inverses_of_two_sizes_in_several_threads():
    """Coarsest levels of 20 rows in six threads beside one of 560 rows,
    inverted at once: the launch limits of one do not reach into another's (an
    explicit inverse's residual is at most 8 n eps cond(A); cond < 4 here)."""
    errors, done = [], threading.Event()

    def work(n, times):
        try:
            a, L = _dense(n, n)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream), pkg.BlockSolver(amg_max_levels=1, autotune=0) as sol:
                b = torch.ones(3 * n, dtype=torch.float64, device="cuda")
                for k in range(times):
                    sol.mesh_setup(L)
                    if n < 100 and done.is_set():
                        break
                x = sol.amg_apply(pkg.SCR_HIER_MESH, b).cpu().numpy().reshape(n, 3)
            assert np.abs(a @ x - 1.0).max() <= 32 * n * np.finfo(float).eps * n
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(f"{n} rows: {e}")

    small = [threading.Thread(target=work, args=(20, 20000)) for _ in range(6)]
    large = threading.Thread(target=work, args=(560, 300))
    for t in small + [large]:
        t.start()
    large.join()
    done.set()
    for t in small:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("share", [1.0, 0.1])
def test_vcycle_with_a_diagonal_next_to_zero_matches_oracle(share):
    """Rows whose diagonal is 1e-36 of the others' entries give D^{-1} A an
    eigenvalue of 1e36: its power iteration, the Chebyshev guard and the V-cycle
    stay finite and equal the oracle's on the exported hierarchy (its V-cycle
    moves by 2e-16 when its matrices do, so FP64 sums in another order stay
    below 1e-10)."""
    L = F.tube_system("tube_small").L
    rows = np.repeat(np.arange(L.nb_rows), np.diff(L.row_ptr))
    small = np.random.default_rng(1).random(L.nb_rows) < share
    L.val[(L.col == rows) & small[rows]] *= 1e-36
    with pkg.BlockSolver() as sol:
        sol.mesh_setup(L)
        nl = sol.amg_levels(pkg.SCR_HIER_MESH)
        As = [to_csr(sol.export(pkg.SCR_HIER_MESH, l, pkg.SCR_EXPORT_OPERATOR)) for l in range(nl)]
        Ps = [to_csr(sol.export(pkg.SCR_HIER_MESH, l, pkg.SCR_EXPORT_PROLONGATOR)) for l in range(nl - 1)]
        b = np.random.default_rng(3).standard_normal(3 * L.nb_rows)
        x = sol.amg_apply(pkg.SCR_HIER_MESH, torch.as_tensor(b, device="cuda")).cpu().numpy().reshape(-1, 3)
    assert nl > 1
    ref = amg.vcycle(amg.hierarchy_from_matrices(As, Ps, 1, 1, 1, "cheb", 3), b.reshape(-1, 3))
    assert np.all(np.isfinite(x)) and np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)


def test_smoother_data_do_not_depend_on_the_timed_kernels(tmp_path):
    """Set-ups (and numeric re-set-ups) with two files of product kernels hold
    the same smoother data: V-cycles of all hierarchies, run with one forced
    kernel, are bit-identical."""
    s = F.tube_system("tube_small")
    with pkg.BlockSolver() as sol:  # every pattern is in the table
        sol.setup(s.A, s.B, s.C, s.D)
        sol.mesh_setup(s.L)
    pkg.tune_save(str(tmp_path / "timed.txt"))
    lines = (tmp_path / "timed.txt").read_text().splitlines()
    for name, codes in (("one", ("101", "101")), ("two", ("402", "104"))):
        rows = [l.split() for l in lines if not l.startswith("#")]
        text = "".join(" ".join(r[:7] + [codes[0] if r[3] == "3" else codes[1]]) + "\n" for r in rows)
        (tmp_path / name).write_text(text)
    rng = np.random.default_rng(2)
    b = {w: torch.as_tensor(rng.standard_normal(n), device="cuda")
         for w, n in ((pkg.SCR_HIER_A, 3 * s.n_v), (pkg.SCR_HIER_SHAT, s.n_p), (pkg.SCR_HIER_MESH, 3 * s.L.nb_rows))}
    sols = []
    try:
        for name in ("one", "two"):
            pkg.tune_load(str(tmp_path / name))
            sols.append(pkg.BlockSolver().setup(s.A, s.B, s.C, s.D))
            sols[-1].mesh_setup(s.L)
        assert [x.stats()["kernel_A"] for x in sols] == [101, 402]
        for again in range(2):
            if again:
                pkg.BlockSolver().close()  # no forced kernel
                for x in sols:
                    x.update_values(s.A, s.B, s.C, s.D)
            pkg.BlockSolver(spmv_group=102).close()  # forces every product's kernel from here
            for which, rhs in b.items():
                one, two = (x.amg_apply(which, rhs).cpu().numpy() for x in sols)
                np.testing.assert_array_equal(one, two)
    finally:
        pkg.tune_load(str(tmp_path / "timed.txt"))
        pkg.BlockSolver().close()
        for x in sols:
            x.close()


def test_levels_with_bf16_values_have_timed_kernels_of_their_own(tmp_path):
    """Coarse levels of the same sizes with BF16 and with FP32 values run
    different kernels: the table of timed choices holds an entry for each
    (value bytes 4, and 204 with BF16 values)."""
    s = F.tube_system("tube_small")
    for bf16 in (1, 0):
        with pkg.BlockSolver(precision=pkg.SCR_MIXED, amg_coarse_bf16=bf16) as sol:
            sol.setup(s.A, s.B, s.C, s.D)
            P1 = sol.export(pkg.SCR_HIER_A, 1, pkg.SCR_EXPORT_PROLONGATOR)
    pkg.tune_save(str(tmp_path / "t.txt"))
    rows = [l.split() for l in (tmp_path / "t.txt").read_text().splitlines() if not l.startswith("#")]
    key = [str(v) for v in (len(P1.col), P1.nb_rows, P1.nb_cols, 3, 3)]
    assert {r[5] for r in rows if r[:5] == key and r[6] == "1"} >= {"4", "204"}


def test_only_the_16_byte_kernels_build_a_padded_copy():
    """A product with a forced kernel builds what that kernel reads: triples of
    lanes (401) hold no more than the scalar-row kernel (101), the 16-byte
    kernels (304) their padded copy beside it."""
    A = pkg.DeviceBSR.from_host(F.tube_system("tube_small").A)
    x = torch.ones(3 * A.nb_cols, dtype=torch.float64, device="cuda")
    peak = {}
    for code in (101, 401, 304):
        with pkg.BlockSolver(spmv_group=code, autotune=0):
            low = _pool_bytes(8, reset=True)
            pkg.bsr_spmv(A, x)
            peak[code] = _pool_bytes(8) - low
    pkg.BlockSolver().close()  # no forced kernel from here
    values = 8 * 9 * A.nnzb
    assert values <= peak[101] < 1.5 * values and peak[401] == peak[101] and peak[304] > 2 * values
