"""Scratch of a plan across its calls, the tuner's candidates and the copies of host items, on the
host alone: the library's objects linked with a double of the CUDA runtime
(cudart_double.cpp), which counts what the plan allocates, frees, captures, launches and
copies."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2508_07476_gb300 import _lib, build

HERE = os.path.dirname(os.path.abspath(__file__))
MALLOCS, FREES, INSTANTIATED, LAUNCHED, STALE, STRIDED = range(6)
ADDRESS = 1 << 20  # a device address: the double's kernels read and write nothing


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    build.build()
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    objs = [os.path.join(build.BUILD, f[:-3] + ".o") for f in sorted(os.listdir(build.CSRC)) if f.endswith(".cu")]
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

    def __init__(self, lib, dims, rho=3.0, chunk=(0, 0, 0)):
        self.lib, self.dims, self.p = lib, dims, ctypes.c_void_p()
        params = _lib.make_params(1.0, rho, (300.0, 260.0, 10.0), (0.1, 0.1, 1.0), _lib.CT_PREC_MIXED, chunk=chunk)
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
        return [self.lib.double_count(k) for k in range(6)]


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


NARROW, WIDE = (63, 68, 50), (66, 60, 50)  # the narrow box's scratch holds the wide one's rows, but not padded


def test_padding_does_not_move_scratch_that_holds_the_plain_rows(plan):
    """The wide box recorded by the caller on the narrow one's scratch, then called directly: the
    buffers whose addresses the record holds stay."""
    plan.box(NARROW)
    before = plan.counts()
    plan.lib.double_user_capture(1)
    plan.box(WIDE)
    plan.lib.double_user_capture(0)
    plan.box(WIDE)
    assert plan.counts() == before


def refuse_padding(plan, call):
    """The smallest limit on a block under which a first `call` passes (its plain rows), above that
    of the re-solve lists; a smaller one refuses it."""
    lo, hi = 0, 1 << 40
    while hi - lo > 1:
        mid = (lo + hi) // 2
        plan.lib.double_limit(mid)
        probe = Plan(plan.lib, plan.dims)
        try:
            call(probe)
            hi = mid
        except AssertionError:
            lo = mid
        finally:
            plan.lib.ct_plan_destroy(probe.p)
    plan.lib.double_limit(hi)


@pytest.mark.parametrize("call", [lambda p: p.box(WIDE), lambda p: p.batch(BATCH)], ids=["box", "batch"])
def test_a_refused_padding_is_not_asked_for_again(plan, call):
    """Where the padded scratch is refused a call takes plain rows; the next equal call allocates
    and frees nothing, nor does one after the device has room again."""
    refuse_padding(plan, call)
    call(plan)
    before = plan.counts()
    call(plan)
    assert plan.counts()[:3] == before[:3]
    plan.lib.double_limit(ctypes.c_uint64(-1).value)
    call(plan)
    assert plan.counts()[:3] == before[:3] and plan.counts()[STALE] == before[STALE]


def test_a_first_call_allocates_its_scratch_once(plan):
    """Two buffers, the re-solve list and its two counters, and nothing given back."""
    before = plan.counts()
    plan.box(WIDE)
    after = plan.counts()
    assert after[MALLOCS] - before[MALLOCS] == 5 and after[FREES] == before[FREES]


@pytest.mark.parametrize("nx,blocks", [(62, 1), (63, 2), (64, 1), (65, 1), (161, 1)])
def test_the_tuner_times_a_block_size_only_where_a_kernel_takes_it(lib, nx, blocks):
    """The z pass over rows of odd length (narrow boxes: wider rows are padded) alone has two block
    sizes to choose from; elsewhere the stencils are one candidate, its block size not tuned."""
    params = _lib.make_params(1.0, 3.0, (0.0, 0.0, 0.0), (0.0, 0.0, 1.0))
    r = _lib.ct_tune_result()
    assert lib.ct_autotune(ctypes.byref(params), _lib._i64x3((nx, 40, 30)), None, 0, None, ctypes.byref(r)) == 0
    tensor_core = 6 if nx % 4 == 0 else 0
    assert r.candidates == 1 + tensor_core + blocks
    if not tensor_core:
        assert r.rho_path == 0 and (r.stream_block > 0) == (blocks == 2)


@pytest.mark.parametrize("chunk,slab_bytes,strided", [
    ((0, 0, 0), None, False), ((0, 0, 8), None, False), ((0, 33, 8), None, False), ((64, 33, 8), None, False),
    ((64, 33, 8), "1000000", True)])
@pytest.mark.parametrize("masked", [False, True])
def test_host_copies_of_whole_rows_are_no_strided_copies(lib, monkeypatch, chunk, slab_bytes, strided, masked):
    """Slabs of whole rows are copied as ranges, or a range per plane; only runs cut along x (here by
    the slab's bytes) are copied row by row."""
    if slab_bytes:
        monkeypatch.setenv("CT_TUNE_SLAB_BYTES", slab_bytes)
    plan = Plan(lib, (161, 90, 40), chunk=chunk)
    try:
        before = plan.counts()
        item = _lib.make_item(ADDRESS, plan.dims, ADDRESS if masked else None, ADDRESS, ADDRESS, ADDRESS, ADDRESS)
        plan.ok(lib.ct_run_chunks(plan.p, (_lib.ct_item * 1)(item), 1, 1, None))
        assert (plan.counts()[STRIDED] > before[STRIDED]) == strided
    finally:
        lib.ct_plan_destroy(plan.p)
