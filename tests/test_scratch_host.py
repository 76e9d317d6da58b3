"""Scratch of a plan across its calls, on the host alone: the library's objects
linked with a double of the CUDA runtime (cudart_double.cpp), which counts what
the plan allocates, frees, captures and launches."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2508_07476_gb300 import _lib, build

HERE = os.path.dirname(os.path.abspath(__file__))
MALLOCS, FREES, INSTANTIATED, LAUNCHED, STALE = range(5)
ADDRESS = 1 << 20  # a device address: the double's kernels read and write nothing


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    build.build()
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    objs = [os.path.join(build.BUILD, f) for f in sorted(os.listdir(build.BUILD)) if f.endswith(".o")]
    out = str(tmp_path_factory.mktemp("double") / "libct_double.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda,
                    os.path.join(HERE, "cudart_double.cpp"), *objs, "-o", out, "-ldl", "-lpthread"], check=True)
    lib = _lib.load(out)
    lib.double_count.restype = ctypes.c_int64
    lib.double_limit.argtypes = [ctypes.c_uint64]
    return lib


class Plan:
    """A plan on the double, and what its calls cost."""

    def __init__(self, lib, dims, rho=3.0):
        self.lib, self.dims, self.p = lib, dims, ctypes.c_void_p()
        params = _lib.make_params(1.0, rho, (300.0, 260.0, 10.0), (0.1, 0.1, 1.0), _lib.CT_PREC_MIXED)
        self.ok(lib.ct_plan_create(ctypes.byref(params), _lib._i64x3(dims), ctypes.byref(self.p)))

    def ok(self, status):
        assert status == _lib.CT_OK, (status, self.lib.ct_last_error())

    def box(self, n):
        i3 = _lib._i64x3
        self.ok(self.lib.ct_run_box(self.p, ADDRESS, i3((0, 0, 0)), i3(self.dims), i3((3, 2, 1)), i3(n), None, ADDRESS,
                                    ADDRESS, ADDRESS, ADDRESS, None))

    def batch(self, dims):
        items = [_lib.make_item(ADDRESS, d, None, ADDRESS, ADDRESS, ADDRESS, ADDRESS) for d in dims]
        self.ok(self.lib.ct_run_chunks(self.p, (_lib.ct_item * len(items))(*items), len(items), 0, None))

    def eig(self, n):
        self.ok(self.lib.ct_eig_smallest(self.p, ADDRESS, n, ADDRESS, ADDRESS, None))

    def counts(self):
        return [self.lib.double_count(k) for k in range(5)]


@pytest.fixture
def plan(lib):
    lib.double_limit(ctypes.c_uint64(-1).value)
    p = Plan(lib, (160, 90, 80))
    yield p
    lib.double_limit(ctypes.c_uint64(-1).value)
    lib.double_user_capture(0)
    lib.ct_plan_destroy(p.p)


BATCH = [(70, 40, 30), (65, 41, 20), (90, 33, 25)]


@pytest.mark.parametrize("grow", ["box", "eig"])
def test_a_batch_graph_is_recorded_anew_when_its_scratch_has_moved(plan, grow):
    """A batch's graph holds the addresses of its slots' scratch and re-solve lists.  Equal batches
    replay it; after a call that replaced one of them the next equal batch records it again."""
    before = plan.counts()
    plan.batch(BATCH)
    plan.batch(BATCH)
    after = plan.counts()
    assert after[INSTANTIATED] - before[INSTANTIATED] == 1 and after[LAUNCHED] - before[LAUNCHED] == 2
    if grow == "box":
        plan.box((150, 80, 70))
    else:
        plan.eig(1 << 22)
    moved = plan.counts()
    assert moved[FREES] > after[FREES]
    plan.batch(BATCH)
    plan.batch(BATCH)
    end = plan.counts()
    assert end[STALE] == before[STALE]
    assert end[INSTANTIATED] - moved[INSTANTIATED] == 1 and end[LAUNCHED] - moved[LAUNCHED] == 2
