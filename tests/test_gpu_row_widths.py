"""Row widths around every boundary of the stencil chain's work splitting: the
padding of scratch rows (from 64 columns on, to multiples of 8), the CTA widths of the
x/y kernels (64, 96, 128, 160, 256 columns), odd and even planes of the z
passes, walks cut into segments, and boxes whose haloed rows start anywhere.
The stage's tensor against the FP64 oracle, and every box equal to the whole
volume bit for bit."""
import numpy as np
import pytest

from oracle import oracle as O
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
    import scipy.ndimage as ndi
    rng = np.random.default_rng(seed)
    v = ndi.gaussian_filter(rng.integers(500, 3000, size=shape).astype(np.float64), 1.0)
    return np.clip(np.rint(v + rng.normal(0, 30, size=shape)), 0, 65535).astype(np.uint16)


@pytest.mark.parametrize("nx", [31, 63, 64, 65, 72, 95, 97, 129, 161, 193, 255, 257, 321])
@pytest.mark.parametrize("sigma,rho", [(1.0, 2.0), (0.7, 1.5), (2.0, 6.0)])
def test_tensor_of_every_row_width(nx, sigma, rho):
    shape = (7, 23, nx) if nx % 2 else (8, 9, nx)
    vol = _vol(shape, nx)
    S_o = O.structure_tensor(vol, sigma, rho)
    g = G.stages(vol, sigma, rho, (10.0, 10.0, 5.0), (0.0, 0.0, 1.0))
    err = np.abs(g["S"] - S_o) / (S_o[0] + S_o[1] + S_o[2])[None]
    assert err.max() <= 2e-5, err.max()  # the stage's tolerance (FP32 form)


@pytest.mark.parametrize("x0,n0", [(0, 64), (1, 70), (3, 101), (5, 66), (29, 131), (40, 129), (96, 73), (104, 65)])
@pytest.mark.parametrize("shape", [(40, 150, 169), (150, 20, 176)])
@pytest.mark.parametrize("prec", [_lib.CT_PREC_FP32, _lib.CT_PREC_MIXED])
def test_boxes_with_padded_rows_equal_the_whole(x0, n0, shape, prec):
    sigma, rho = 1.0, 4.0
    vol = _vol(shape, 5)
    nz, ny, nx = shape
    cen, ax = (80.0, 60.0, 10.0), (0.1, 0.1, 1.0)
    whole = G.fused(vol, sigma, rho, cen, ax, precision=prec, raw=True)
    h = O.radius(sigma) + O.radius(rho)
    lo, n = (x0, 3, 5), (n0, ny - 7, nz - 9)
    ilo = tuple(max(0, a - h) for a in lo)
    ihi = tuple(min(d, a + b + h) for a, b, d in zip(lo, n, (nx, ny, nz)))
    sub = vol[ilo[2]:ihi[2], ilo[1]:ihi[1], ilo[0]:ihi[0]]
    o = [torch.empty((k,) * (k > 1) + (n[2], n[1], n[0]), device="cuda") for k in (3, 1, 1, 1)]
    plan = _lib.ct_plan_create(_lib.make_params(sigma, rho, cen, ax, prec), (nx, ny, nz))
    try:
        _lib.ct_run_box(plan, G.dev_u16(sub), ilo, tuple(b - a for a, b in zip(ilo, ihi)), lo, n, None, *o)
        torch.cuda.synchronize()
        _lib.ct_plan_sync(plan)
    finally:
        _lib.ct_plan_destroy(plan)
    sl = (slice(lo[2], lo[2] + n[2]), slice(lo[1], lo[1] + n[1]), slice(lo[0], lo[0] + n[0]))
    for k, t in zip(("v", "ha", "ia", "fa"), o):
        np.testing.assert_array_equal(t.cpu().numpy(), whole[k][(slice(None),) * (k == "v") + sl], err_msg=k)


@pytest.mark.parametrize("ny,nz", [(1, 1), (31, 1), (33, 1), (32, 3), (127, 1), (129, 1), (20, 24), (25, 41)])
def test_tensor_core_rows_of_every_count(monkeypatch, ny, nz):
    """The tensor-core x pass takes each component's rows in groups of 128, the last one ragged
    (tensor maps read its missing rows as zeros and clip their stores): the tensor matches the
    oracle in every row, and nothing is written past the last component's last row."""
    monkeypatch.setenv("CT_TUNE_TC_RHO", "7")
    monkeypatch.setenv("CT_TUNE_TC_MIN_R", "0")
    monkeypatch.setenv("CT_TUNE_TC_ANY_BOX", "1")
    nx, sigma, rho = 192, 1.0, 3.0
    vol = _vol((nz, ny, nx), 17 * ny + nz)
    n = nx * ny * nz
    plan = _lib.ct_plan_create(_lib.make_params(sigma, rho, (0, 0, 0), (0, 0, 1)), (nx, ny, nz))
    try:
        S = torch.full((6 * n + 4096,), -7.0, device="cuda")
        _lib.ct_structure_tensor(plan, G.dev_u16(vol), (0, 0, 0), (nx, ny, nz), (0, 0, 0), (nx, ny, nz), S)
        torch.cuda.synchronize()
        _lib.ct_plan_sync(plan)
    finally:
        _lib.ct_plan_destroy(plan)
    S = S.cpu().numpy()
    assert np.all(S[6 * n:] == -7.0)
    S_o = O.structure_tensor(vol, sigma, rho)
    err = np.abs(S[:6 * n].reshape(S_o.shape) - S_o) / (S_o[0] + S_o[1] + S_o[2])[None]
    assert err.max() <= 2e-5, err.max()


@pytest.mark.parametrize("nx", [5, 63, 65, 511, 512, 513, 1030])
@pytest.mark.parametrize("types", [(_lib.CT_OUT_F32,) * 3, (_lib.CT_OUT_F16,) * 3,
                                   (_lib.CT_OUT_F32, _lib.CT_OUT_U8Q, _lib.CT_OUT_F16)])
def test_unmasked_eigen_rows_equal_the_masked_form(nx, types):
    """Without a mask a CTA walks a span of one row; with a mask of ones each row segment's voxels
    are listed first: the same arithmetic per voxel, so the same outputs to the bit, the
    re-solved voxels of a flat slab among them."""
    vol = _vol((5, 6, nx), nx)
    vol[:, :, : nx // 4] = 1500
    kw = dict(vec_type=types[0], angle_type=types[1], fa_type=types[2], raw=True)
    cen, ax = (nx / 2 + 0.3, 2.0, 1.0), (0.1, 0.0, 1.0)
    a = G.fused(vol, 1.0, 2.0, cen, ax, **kw)
    b = G.fused(vol, 1.0, 2.0, cen, ax, mask=np.ones_like(vol, dtype=np.uint8), **kw)
    for k in ("v", "ha", "ia", "fa"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert a["stats"]["fallback_voxels"] == b["stats"]["fallback_voxels"]


@pytest.mark.parametrize("first", [(65, 60, 50), (63, 62, 50)])
def test_captured_box_equals_the_direct_call(first):
    """A 65 x 60 x 50 box recorded into the caller's graph after a call that left scratch for
    padded rows (the same box), and after one that left room for plain rows only (a narrower,
    larger one): both replay to the direct call's outputs."""
    nx, ny, nz = 160, 90, 80
    vol = G.dev_u16(_vol((nz, ny, nx), 3))
    params = _lib.make_params(1.0, 3.0, (300.0, 260.0, 10.0), (0.1, 0.1, 1.0), _lib.CT_PREC_MIXED)

    def out(n):
        return [torch.empty((k,) * (k > 1) + (n[2], n[1], n[0]), device="cuda") for k in (3, 1, 1, 1)]

    def run(plan, n, o):
        _lib.ct_run_box(plan, vol, (0, 0, 0), (nx, ny, nz), (3, 2, 1), n, None, *o)

    box, plans = (65, 60, 50), [_lib.ct_plan_create(params, (nx, ny, nz)) for _ in range(2)]
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    try:
        direct, warm, got = out(box), out(first), out(box)
        run(plans[0], box, direct)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            run(plans[1], first, warm)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=st):
            run(plans[1], box, got)
        for t in got:
            t.fill_(-9.0)
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(got, direct):
            np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
    finally:
        del graph
        for p in plans:
            _lib.ct_plan_destroy(p)


@pytest.mark.parametrize("chunk", [(0, 0, 9), (0, 0, 16), (0, 0, 64), (0, 0, 149), (72, 0, 20), (72, 60, 33)])
@pytest.mark.parametrize("masked", [False, True])
def test_host_slabs_of_every_count_equal_the_device_call(chunk, masked):
    """Two host items of one call, in slabs of which each reuses its buffers two slabs later
    while the copies of others are in flight: both equal the call on device memory."""
    rng = np.random.default_rng(8)
    dims = [(200, 130, 150), (96, 70, 41)]
    vols = [_vol(d[::-1], 11 + k) for k, d in enumerate(dims)]
    masks = [(rng.random(d[::-1]) < 0.7).astype(np.uint8) if masked else None for d in dims]
    params = _lib.make_params(1.0, 3.0, (300.0, 260.0, 10.0), (0.1, 0.1, 1.0), _lib.CT_PREC_MIXED,
                              chunk=chunk)

    def run(on_host):
        outs, items, keep = [], [], []
        plan = _lib.ct_plan_create(params, dims[0])
        for (nx, ny, nz), vol, mask in zip(dims, vols, masks):
            v = torch.from_numpy(vol.view(np.int16))
            m = None if mask is None else torch.from_numpy(mask)
            kw = dict(pin_memory=True) if on_host else dict(device="cuda")
            v, m = [None if t is None else t.pin_memory() if on_host else t.cuda() for t in (v, m)]
            o = [torch.full((k,) * (k > 1) + (nz, ny, nx), -9.0, **kw) for k in (3, 1, 1, 1)]
            items.append(_lib.make_item(v, (nx, ny, nz), m, *o))
            outs.append(o)
            keep += [v, m]
        try:
            for _ in range(2 if on_host else 1):
                _lib.ct_run_chunks(plan, items, on_host)
            torch.cuda.synchronize()
        finally:
            _lib.ct_plan_destroy(plan)
        return outs

    for a, b in zip(run(True), run(False)):
        for p, q in zip(a, b):
            np.testing.assert_array_equal(p.numpy(), q.cpu().numpy())
