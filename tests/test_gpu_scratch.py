"""Scratch that a plan replaces between calls, on the GPU: what was recorded
before is recorded again, and what a caller recorded stays valid."""
import numpy as np
import pytest

from paper_2508_07476_gb300 import _lib, build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import gpu_util as G  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    _lib.load()


def _vol(shape, seed):
    return np.random.default_rng(seed).integers(500, 3000, size=shape).astype(np.uint16)


def _out(n):
    return [torch.empty((k,) * (k > 1) + (n[2], n[1], n[0]), device="cuda") for k in (3, 1, 1, 1)]


DIMS = (160, 90, 80)
PARAMS = dict(sigma=1.0, rho=3.0, lv_center=(300.0, 260.0, 10.0), lv_axis=(0.1, 0.1, 1.0),
              precision=_lib.CT_PREC_MIXED)


def test_equal_batches_around_calls_that_replace_the_scratch():
    """A batch, then a larger box and a larger eigen call on the same plan, other tensors where the
    old scratch was, then the same batch: the first outputs again, and the other tensors unharmed."""
    plan = _lib.ct_plan_create(_lib.make_params(**PARAMS), DIMS)
    try:
        dims = [(70, 40, 30), (65, 41, 20), (90, 33, 25)]
        vols = [G.dev_u16(_vol(d[::-1], k)) for k, d in enumerate(dims)]
        outs = [_out(d) for d in dims]
        items = [_lib.make_item(v, d, None, *o) for v, d, o in zip(vols, dims, outs)]
        _lib.ct_run_chunks(plan, items, False)
        torch.cuda.synchronize()
        first = [[t.cpu().numpy() for t in o] for o in outs]
        vol = G.dev_u16(_vol(DIMS[::-1], 9))
        S = torch.rand((6, 1 << 21), device="cuda")
        ev, vec = torch.empty((3, 1 << 21), device="cuda"), torch.empty((3, 1 << 21), device="cuda")
        others = []
        for call in ("box", "eig"):
            if call == "box":
                _lib.ct_run_box(plan, vol, (0, 0, 0), DIMS, (0, 0, 0), DIMS, None, *_out(DIMS))
            else:
                _lib.ct_eig_smallest(plan, S, 1 << 21, ev, vec)
            others += [torch.full((1 << 20,), 3.0, device="cuda") for _ in range(8)]
            for o in outs:
                for t in o:
                    t.fill_(-9.0)
            _lib.ct_run_chunks(plan, items, False)
            torch.cuda.synchronize()
            _lib.ct_plan_sync(plan)
            for a, b in zip(outs, first):
                for p, q in zip(a, b):
                    np.testing.assert_array_equal(p.cpu().numpy(), q, err_msg=call)
        assert all(bool((t == 3.0).all()) for t in others)
    finally:
        _lib.ct_plan_destroy(plan)


def test_a_recorded_box_after_the_same_direct_call():
    """A 66 x 60 x 50 box recorded into the caller's graph on scratch that a narrower box left (it holds
    the plain rows but not the padded ones), then called directly on the same plan: the direct
    call leaves the recorded scratch in place, and the graph replays to its outputs."""
    vol = G.dev_u16(_vol(DIMS[::-1], 3))
    params = _lib.make_params(**PARAMS)

    def run(plan, n, o):
        _lib.ct_run_box(plan, vol, (0, 0, 0), DIMS, (3, 2, 1), n, None, *o)

    first, box, plans = (63, 68, 50), (66, 60, 50), [_lib.ct_plan_create(params, DIMS) for _ in range(2)]
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    try:
        padded, warm, got, plain = _out(box), _out(first), _out(box), _out(box)
        run(plans[0], box, padded)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            run(plans[1], first, warm)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=st):
            run(plans[1], box, got)
        run(plans[1], box, plain)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for a, b, c in zip(got, plain, padded):
            np.testing.assert_array_equal(a.cpu().numpy(), c.cpu().numpy())
            np.testing.assert_array_equal(b.cpu().numpy(), c.cpu().numpy())
    finally:
        del graph
        for p in plans:
            _lib.ct_plan_destroy(p)
