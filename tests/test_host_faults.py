"""Host-side failures of matrix creation and multigrid set-up, without a GPU: the library's objects linked with a fake
CUDA runtime on host memory (fake_cudart.cpp) whose allocations, or whose operator new, fail on request."""

import glob
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SETUP = """
import ctypes, sys
sys.path.insert(0, sys.argv[2])
import gen
from paper_1711_10622_gb300 import _native as N
L, fake = N.lib(), ctypes.CDLL(sys.argv[1])
for f in ("fake_pending", "fake_live", "fake_bytes"):
    getattr(fake, f).restype = ctypes.c_long

def create(op):
    A = ctypes.c_void_p()
    st = L.ens_create_matrix(op.n, op.nnz, op.row_ptr.ctypes.data, op.col_idx.ctypes.data, op.val.ctypes.data, 0, None, ctypes.byref(A))
    assert (st == N.ENS_OK) == bool(A)
    return st, A

def destroy(A):
    assert L.ens_destroy_matrix(A) == N.ENS_OK
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1711_10622_gb300 import build

    build.build()
    lib = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-o", lib, os.path.join(ROOT, "tests", "fake_cudart.cpp"),
                    *sorted(glob.glob(os.path.join(build.OBJ_DIR, "*.o"))), "-lpthread"], check=True)
    return lib


def _run(fake, script):
    """In a process of its own: an exception that leaves the library ends the process."""
    r = subprocess.run([sys.executable, "-c", SETUP + script, fake, ROOT], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, ENSEMBLE_SOLVE_LIB=fake))
    assert r.returncode == 0, r.stderr[-2000:]


def test_create_matrix_without_host_memory(fake):
    """Each host allocation of the call fails in turn: the call returns a matrix or ENS_ERR_OOM and keeps nothing."""
    _run(fake, """
op = gen.dirichlet_box(41)  # large enough for row boxes
seen = set()
for k in range(1, 100000):
    fake.fake_fail_new(ctypes.c_long(k))
    st, A = create(op)
    reached = not fake.fake_pending()
    fake.fake_fail_new(ctypes.c_long(0))
    assert st in (N.ENS_OK, N.ENS_ERR_OOM), st
    seen.add(st)
    if A:
        destroy(A)
    assert fake.fake_live() == 0
    if not reached:
        break
assert N.ENS_OK in seen and k > 20
""")


def test_create_matrix_without_device_memory(fake):
    """Each device allocation fails in turn: without its boxes' memory the matrix works, without its own the call ends."""
    _run(fake, """
op = gen.dirichlet_box(41)
seen = []
for k in range(1, 1000):
    fake.fake_fail_alloc(ctypes.c_long(k))
    st, A = create(op)
    reached = not fake.fake_pending()
    fake.fake_fail_alloc(ctypes.c_long(0))
    seen.append(st)
    if A:
        destroy(A)
    assert fake.fake_live() == 0
    if not reached:
        break
assert set(seen) == {N.ENS_OK, N.ENS_ERR_OOM} and seen[0] == N.ENS_ERR_OOM and seen.count(N.ENS_OK) >= 2, seen
""")


def test_amg_setup_without_device_memory(fake):
    """The coarsest level's dense matrix (the last three allocations of the set-up) is left out where it does not fit;
    every other failed allocation ends the call with the matrix as it was."""
    _run(fake, """
op = gen.dirichlet_box(16)
seen = []
for k in range(1, 1000):
    st, A = create(op)
    held = fake.fake_live()
    fake.fake_fail_alloc(ctypes.c_long(k))
    st = L.ens_amg_setup(A, None, None)
    reached = not fake.fake_pending()
    fake.fake_fail_alloc(ctypes.c_long(0))
    assert st == N.ENS_OK or (st == N.ENS_ERR_OOM and fake.fake_live() == held), st
    destroy(A)
    assert fake.fake_live() == 0
    if not reached:
        break
    seen.append(st)
assert seen[-3:] == [N.ENS_OK] * 3 and seen.count(N.ENS_ERR_OOM) >= 10, seen
""")


def test_scaled_copy_uses_its_levels_boxes(fake):
    """The column-scaled copy of a multigrid level takes the row boxes of the level (the same rows and columns) and holds
    only values of its own."""
    _run(fake, """
import numpy as np
op = gen.dirichlet_box(41)
b0 = fake.fake_bytes()
st, A = create(op)
b1 = fake.fake_bytes()
o = N.AmgOpts()
L.ens_default_amg_opts(ctypes.byref(o))
o.max_levels = 2
assert L.ens_amg_setup(A, ctypes.byref(o), None) == N.ENS_OK
b2 = fake.fake_bytes()
rows, nnz = (ctypes.c_int64 * 16)(), (ctypes.c_int64 * 16)()
assert L.ens_amg_info(A, None, rows, nnz) == N.ENS_OK and rows[1] > 512
C = gen.Operator("level", (rows[1], 1, 1), ("x",) * 3, np.empty(rows[1] + 1, np.int32), np.empty(nnz[1], np.int32), np.empty(nnz[1]), False)
assert L.ens_amg_level(A, 1, C.row_ptr.ctypes.data, C.col_idx.ctypes.data, C.val.ctypes.data, None) == N.ENS_OK
b3 = fake.fake_bytes()
st, B = create(C)
maps = 4 * (op.n + op.n + rows[1] + 1)
copy = (b2 - b1) - maps - (fake.fake_bytes() - b3)
shape = op.n // 256 * (256 + 576) * 4  # at least this for rows and columns of the boxes
assert copy <= (b1 - b0) - shape, (copy, b1 - b0, shape)
destroy(B)
destroy(A)
assert fake.fake_live() == 0
""")
