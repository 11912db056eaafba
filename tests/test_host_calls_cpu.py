"""The library's host code on a CUDA runtime without a GPU (fake_cuda.cpp):
which device waits before memory is freed, what an error leaves behind, which
form a call takes.  Kernels do nothing here; their results are the GPU tests'."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1511_02494_gb300 import _abi, build as lib_build
import paper_1511_02494_gb300 as sp

HERE = os.path.dirname(os.path.abspath(__file__))
OK, NOMEM, CUDA = 0, 4, 5
CUDA_ERROR_MEMORY = 2


@pytest.fixture(scope="module")
def linked(tmp_path_factory):
    """The library's objects with the fake runtime in the place of CUDA's."""
    lib_build.build()
    objs = sorted(os.path.join(lib_build.OBJ, f) for f in os.listdir(lib_build.OBJ) if f.endswith(".cu.o"))
    objs = [o for o in objs if os.path.exists(os.path.join(lib_build.CSRC, os.path.basename(o)[:-2]))]
    out = str(tmp_path_factory.mktemp("fake") / "lib.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(lib_build._nvcc()))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I", inc, "-o", out,
                        os.path.join(HERE, "fake_cuda.cpp"), *objs, "-Wl,-Bsymbolic"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


class Fake:
    """A fresh instance of the library with its own runtime state."""

    def __init__(self, path, devices=1):
        self.lib = _abi.declare(C.CDLL(path))
        self.lib.fake_log.restype = C.c_char_p
        self.lib.fake_live.restype = self.lib.fake_reserved.restype = C.c_longlong
        self.lib.fake_lock.argtypes = [C.c_void_p, C.c_size_t]
        self.lib.fake_reset(devices)

    def fail(self, fn, code, after=0):
        self.lib.fake_fail(fn.encode(), after, code)

    def log(self):
        return self.lib.fake_log().decode().splitlines()

    def matrix(self, n, per_row=1):
        """n rows of per_row columns on the diagonal and after it."""
        self.rp = np.arange(n + 1, dtype=np.int32) * per_row
        self.ci = (np.arange(n, dtype=np.int32)[:, None] + np.arange(per_row, dtype=np.int32)).reshape(-1) % n
        self.ci = np.ascontiguousarray(self.ci)
        self.v = np.ones(n * per_row)
        return _abi.CSR(n, n, self.ci.size, self.rp.ctypes.data, self.ci.ctypes.data, self.v.ctypes.data)

    def prepare(self, A, variant="sliced", trusted=1, **kw):
        h, ch = C.c_void_p(), sp.make_choice(variant, **kw)
        st = self.lib.spmv_prepare(C.byref(A), C.byref(ch), trusted, C.byref(h), None)
        return st, h


@pytest.fixture
def fake(linked, tmp_path):
    def make(devices=1):
        path = str(tmp_path / f"lib{len(os.listdir(tmp_path))}.so")
        shutil.copy(linked, path)
        return Fake(path, devices)
    return make


def test_free_waits_for_the_device_that_owns_the_object(fake):
    f = fake(devices=2)
    st, h = f.prepare(f.matrix(1000))
    assert st == OK
    f.lib.cudaSetDevice(1)
    f.lib.fake_clear()
    f.lib.spmv_prepared_free(h)
    log = f.log()
    frees = [i for i, ln in enumerate(log) if ln.startswith("free ")]
    assert frees and "device 0 synchronize" in log[:frees[0]], log
    d = C.c_int(-1)
    f.lib.cudaGetDevice(C.byref(d))
    assert d.value == 1 and f.lib.fake_live() == 0


@pytest.mark.parametrize("fn,after", [("cudaMemPoolCreate", 0), ("cudaMallocFromPoolAsync", 0),
                                      ("cudaMallocFromPoolAsync", -1), ("cudaMallocHost", 1)])
def test_a_prepare_that_fails_leaves_no_validation_running(fake, fn, after):
    """The caller may free the matrix once spmv_prepare has returned."""
    f = fake()
    A = f.matrix(1000)
    f.fail(fn, CUDA_ERROR_MEMORY, after)
    st, h = f.prepare(A, trusted=0)
    assert (st == OK) == (fn == "cudaMallocFromPoolAsync" and after == 0) and bool(h) == (st == OK)   # tried once more
    log = f.log()
    runs = [i for i, ln in enumerate(log) if ln.startswith("kernel ")]
    assert not runs or "stream 0 synchronize" in log[runs[-1]:], log


def test_peers_reach_prepared_arrays(fake):
    """As they reach memory of cudaMalloc: every device that can, and no other."""
    f = fake(devices=4)
    for a, b in ((1, 0), (3, 0), (0, 2)):               # 1 and 3 reach 0; 0 reaches 2
        f.lib.fake_peer(a, b)
    st, h = f.prepare(f.matrix(1000))
    assert st == OK
    opened = [ln for ln in f.log() if ln.startswith("pool of device 0 open")]
    assert opened == ["pool of device 0 open to device 1", "pool of device 0 open to device 3"]
    f.lib.spmv_prepared_free(h)


def test_a_pool_that_cannot_be_opened_to_a_peer(fake):
    f = fake(devices=2)
    f.lib.fake_peer(1, 0)
    f.fail("cudaMemPoolSetAccess", 1, after=-1)
    st, h = f.prepare(f.matrix(1000))
    assert st == OK
    f.lib.spmv_prepared_free(h)


def _features(f, A):
    return f.lib.spmv_features(C.byref(A), 128, C.byref(_abi.Features()), None)


def _validate(f, A):
    return f.lib.spmv_validate(C.byref(A), None)


def _batch(f, A):
    B = C.c_void_p()
    st = f.lib.spmv_batch_create(C.byref(A), 1, None, None, C.byref(B), None)
    f.lib.spmv_batch_free(B)
    return st


def _train(f, A):
    m = np.ones(16 * 8 + 8 + 8 * 8 + 8 + 2 * 8 + 2, dtype=np.float32)
    g, loss, z, y = np.empty_like(m), np.zeros(1, np.float32), np.zeros((4, 16), np.float32), np.zeros(4, np.int32)
    return f.lib.spmv_mlp_loss_grad(m.ctypes.data, 8, 8, 2, z.ctypes.data, y.ctypes.data, 4, g.ctypes.data,
                                    loss.ctypes.data, None)


def _probe(f, A):
    x, s = np.ones(A.n_cols), np.zeros(1, np.uint64)
    return f.lib.spmv_gather_probe(C.byref(A), x.ctypes.data, s.ctypes.data, None)


def _profile_outputs(f, A):
    x, y = np.ones(A.n_cols), np.zeros(A.n_rows)
    return f.lib.spmv_profile_outputs(C.byref(A), x.ctypes.data, 4, None, y.ctypes.data, None, None, None, None)


@pytest.mark.parametrize("call,fn,after", [
    (_features, "cudaMalloc", 0), (_validate, "cudaMalloc", 0), (_batch, "cudaMalloc", 0), (_batch, "cudaMalloc", 1),
    (_batch, "cudaMalloc", 2), (_train, "cudaMallocAsync", 0), (_probe, "cudaMallocAsync", 0),
    (_profile_outputs, "cudaMallocAsync", 0), (_profile_outputs, "cudaMallocAsync", 4)])
def test_the_pools_idle_memory_is_given_back_before_a_call_fails(fake, call, fn, after):
    f = fake()
    A = f.matrix(1000)
    st, kept = f.prepare(A)
    st2, h = f.prepare(A)
    assert st == st2 == OK
    f.lib.spmv_prepared_free(h)                          # its arrays stay in the pool, which `kept` holds open
    f.lib.fake_clear()
    f.fail(fn, CUDA_ERROR_MEMORY, after)
    assert call(f, A) == OK
    assert "trim to 0" in f.log()
    f.fail(fn, CUDA_ERROR_MEMORY, -1)
    assert call(f, A) in (OK, NOMEM, CUDA)               # OK where an earlier call's scratch serves
    f.lib.fake_reset(1)
    f.lib.spmv_prepared_free(kept)


def test_the_pools_idle_memory_is_given_back_for_large_work_vectors(fake):
    f = fake()
    n = 12_000_000                                       # three vectors: more than the pool keeps for scratch
    st, h = f.prepare(f.matrix(n))
    assert st == OK
    f.lib.fake_clear()
    f.fail("cudaMallocAsync", CUDA_ERROR_MEMORY)
    assert _cg(f, h, n, iters=1) == OK and "trim to 0" in f.log()
    f.lib.spmv_prepared_free(h)


def test_scratch_of_many_calls_at_once_does_not_stay(fake):
    """40 solves in flight, 48 MB of work vectors each: once they have been
    waited for, the pool keeps 1 GB and a step of 256 MB beyond the objects;
    with the last object nothing, also not what was in flight then."""
    f = fake()
    n = 2_000_000
    st, h = f.prepare(f.matrix(n))
    assert st == OK
    objects = f.lib.fake_reserved()
    f.lib.fake_free_later(1)
    for _ in range(40):
        assert _cg(f, h, n, iters=1) == OK
    assert f.lib.fake_reserved() > objects + 40 * 24 * n - 1
    f.lib.cudaDeviceSynchronize()
    assert objects < f.lib.fake_reserved() <= objects + (1 << 30) + (1 << 28) + (1 << 20)
    assert _cg(f, h, n, iters=1) == OK
    f.lib.spmv_prepared_free(h)
    f.lib.cudaDeviceSynchronize()
    assert f.lib.fake_reserved() == 0 and f.lib.fake_live() == 0


# ---- page-locked vectors -------------------------------------------------------------

N = 1 << 19                       # columns from which the kernel pulls x
PAGE = 4096
X_PULLED, X_COPIED, Y_COPIED = "kernel k_sliced_host on stream 0", f"copy up {8 * N}", f"copy down {8 * N}"


def _paged(n):
    """n doubles from a page boundary on, and what keeps them."""
    raw = np.zeros(8 * n + PAGE, dtype=np.uint8)
    at = -raw.ctypes.data % PAGE
    return raw[at:at + 8 * n].view(np.float64)


@pytest.mark.parametrize("vector", ["x", "y"])
@pytest.mark.parametrize("locked,direct", [
    ([(0, 8 * N)], True),                                              # all of it
    ([(0, PAGE), (8 * N - PAGE, PAGE)], False),                        # a hole between two registrations
    ([(0, 8 * N - PAGE), (8 * N - PAGE, PAGE)], True),                 # two, end to end
    ([(0, PAGE), (PAGE, PAGE), (2 * PAGE, 8 * N)], True),              # three, and past the end
    ([(0, 8 * N - PAGE)], False), ([(PAGE, 8 * N - PAGE)], False), ([], False)])
def test_host_vectors_are_used_where_registrations_hold_all_of_them(fake, vector, locked, direct):
    f = fake()
    st, h = f.prepare(f.matrix(N), block_nnz=1, threads_per_row=1)
    assert st == OK
    x, y = _paged(N), _paged(N)
    for v, ranges in ((x, locked if vector == "x" else [(0, 8 * N)]), (y, locked if vector == "y" else [(0, 8 * N)])):
        for at, n in ranges:
            f.lib.fake_lock(v.ctypes.data + at, n)
    f.lib.fake_clear()
    assert f.lib.spmv_host(h, x.ctypes.data, y.ctypes.data, None) == OK
    log = f.log()
    assert ((X_PULLED in log), (X_COPIED in log)) == ((True, False) if direct or vector == "y" else (False, True))
    assert (Y_COPIED in log) == (vector == "y" and not direct)
    f.lib.fake_clear()
    assert f.lib.spmv_host_async(h, x.ctypes.data, y.ctypes.data, None) == OK
    assert X_COPIED in f.log() and Y_COPIED in f.log() and X_PULLED not in f.log()
    f.lib.spmv_prepared_free(h)


# ---- conjugate gradients ----------------------------------------------------------

COOPERATIVE_TOO_LARGE = 720


def _cg(f, h, n, iters=3, refine=0, graph=0):
    v = np.ones((2, n))
    return f.lib.spmv_cg(h, h, v[0].ctypes.data, v[1].ctypes.data, iters, refine, None, graph, None)


def _kernels(log):
    return [ln.split()[1] for ln in log if ln.startswith("kernel ")]


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("code", [COOPERATIVE_TOO_LARGE, 701, 801])
def test_cg_runs_in_three_kernels_where_the_one_launch_is_refused(fake, code, graph):
    f = fake()
    st, h = f.prepare(f.matrix(1000))
    assert st == OK
    f.lib.fake_clear()
    assert _cg(f, h, 1000, graph=graph) == OK
    assert _kernels(f.log()).count("k_cg_resident") == 1 and "begin capture" not in f.log()
    f.fail("cudaLaunchCooperativeKernel", code)
    f.lib.fake_clear()
    assert _cg(f, h, 1000, graph=graph) == OK
    ran = _kernels(f.log())
    assert "k_cg_resident" not in ran and ran.count("k_sliced_dot") == 3
    assert ("graph launch" in f.log()) == (graph == 1)
    f.lib.spmv_prepared_free(h)
    assert f.lib.fake_live() == 0


@pytest.mark.parametrize("fn,after,code,graph", [
    ("cudaLaunchCooperativeKernel", 0, 700, 0),      # an error that is not a refusal
    ("launch", 0, 98, 0), ("launch", 1, 98, 1),
    ("cudaStreamCreateWithFlags", 0, 2, 1), ("cudaStreamBeginCapture", 0, 900, 1),
    ("cudaGraphInstantiate", 0, 2, 1), ("cudaMemsetAsync", 0, 1, 0), ("cudaMemsetAsync", 1, 1, 0)])
def test_cg_frees_its_vectors_after_an_error(fake, fn, after, code, graph):
    f = fake()
    st, h = f.prepare(f.matrix(1000))
    assert st == OK
    assert _cg(f, h, 1000) == OK                       # what a first call allocates for good
    if graph:
        f.fail("cudaLaunchCooperativeKernel", COOPERATIVE_TOO_LARGE)
    before = f.lib.fake_live()
    f.fail(fn, code, after)
    assert _cg(f, h, 1000, graph=graph) == CUDA
    assert f.lib.fake_live() == before
    f.lib.spmv_prepared_free(h)
    assert f.lib.fake_live() == 0
