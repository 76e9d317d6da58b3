"""The stage kernels at the sizes where their work splitting can go wrong: tile
and vector-width remainders, single elements, misaligned pointers, lists that
fill and empty, and re-solved tensors at the ends of the accepted range."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from oracle import profile as OP
from paper_2508_07476_gb300 import _lib, build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

F32, F16, U8Q = _lib.CT_OUT_F32, _lib.CT_OUT_F16, _lib.CT_OUT_U8Q
DT = {F32: torch.float32, F16: torch.float16, U8Q: torch.uint8}


@pytest.fixture(scope="module", autouse=True)
def _ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    _lib.load()


def _off(a, dtype, shift):
    """A device copy of `a` starting `shift` elements past an aligned address."""
    t = torch.empty(a.size + shift, dtype=dtype, device="cuda")[shift:]
    t.copy_(torch.from_numpy(np.ascontiguousarray(a)).reshape(-1).to(dtype))
    return t


def _angles(dims, evec, evals, mask, types, shift=0):
    vt, at, ft = types
    nx, ny, nz = dims
    n = nx * ny * nz
    cen, ax = (nx / 2 + 0.3, ny / 2 - 0.2, 1.0), (0.1, -0.2, 1.0)
    plan = _lib.ct_plan_create(_lib.make_params(1.0, 2.0, cen, ax, vec_type=vt, angle_type=at, fa_type=ft), dims)
    try:
        o = [_off(np.zeros(k), DT[t], shift) for k, t in ((3 * n, vt), (n, at), (n, at), (n, ft))]
        m = None if mask is None else _off(mask, torch.uint8, shift)
        _lib.ct_angles(plan, _off(evec, torch.float32, shift), _off(evals, torch.float32, shift), (0, 0, 0), dims, m,
                       *o)
        torch.cuda.synchronize()
    finally:
        _lib.ct_plan_destroy(plan)
    return [t.cpu().numpy() for t in o], cen, ax


@pytest.mark.parametrize("dims", [(1, 1, 1), (4, 1, 1), (5, 1, 1), (2, 2, 3), (33, 5, 4), (64, 3, 2), (31, 17, 4)])
@pytest.mark.parametrize("types", [(F32, F32, F32), (F16, F16, F16), (F32, U8Q, F16), (F16, F32, F32)])
@pytest.mark.parametrize("masked", [False, True])
def test_angles_of_small_and_misaligned_boxes(dims, types, masked):
    rng = np.random.default_rng(sum(dims) + masked)
    n = int(np.prod(dims))
    shape = dims[::-1]
    v = rng.normal(size=(3, n))
    v = (v / np.linalg.norm(v, axis=0)).astype(np.float32)
    l = np.sort(rng.uniform(0.0, 5.0, size=(3, n)), axis=0).astype(np.float32)
    mask = (rng.random(n) < 0.5).astype(np.uint8) if masked else None
    got, cen, ax = _angles(dims, v, l, mask, types)
    ora = O.angles_field(v.astype(np.float64).reshape((3,) + shape), l.astype(np.float64).reshape((3,) + shape), dims,
                         (0, 0, 0), dims, cen, ax, mask=None if mask is None else mask.reshape(shape))
    ov, oha, oia, ofa = (np.asarray(a).reshape(-1) for a in ora)
    ins = np.ones(n, bool) if mask is None else mask.astype(bool)
    vt, at, ft = types
    # near v.e_t = 0 the orientation rule may flip the sign: compared up to it there
    flip = np.abs(oha) > 89.9
    ok = ins & ~flip
    half = {F32: 0.0, F16: 2.0 ** -12, U8Q: 0.0}  # relative half-ulp of the encoding
    if at == U8Q:
        for g, o in ((got[1], oha), (got[2], oia)):
            code = np.rint((o + 90.0) * 256.0 / 180.0)
            d = np.abs(g[ok].astype(int) - code[ok].astype(int)) % 256
            assert np.all((d <= 1) | (d >= 255))
            assert np.all(g[~ins] == 0)
    else:
        for g, o in ((got[1], oha), (got[2], oia)):
            assert np.all(np.abs(g[ok].astype(np.float64) - o[ok]) <= 1e-3 + 90.0 * half[at] * 2)
            assert np.all(np.isnan(g[~ins].astype(np.float64)))
    assert np.all(np.abs(got[3][ins].astype(np.float64) - ofa[ins]) <= 1e-5 + half[ft] * 2)
    gv, o3 = got[0].astype(np.float64).reshape(3, n), ov.reshape(3, n)
    assert np.all(np.abs(gv[:, ok] - o3[:, ok]) <= 1e-6 + half[vt] * 2)
    assert np.all(np.isnan(gv[:, ~ins]))
    # arrays off the vector boundary (one voxel per thread): the same values to the bit
    for a, b in zip(got, _angles(dims, v, l, mask, types, shift=1)[0]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 255, 256, 257, 4097, 70001])
@pytest.mark.parametrize("share", [1.0, 0.3])
def test_eig_list_fills_and_empties(n, share):
    """Every tensor (or a third of them) near-degenerate: the list takes each exactly once."""
    rng = np.random.default_rng(n)
    Q, _ = np.linalg.qr(rng.normal(size=(n, 3, 3)))
    lam = np.stack([np.full(n, 0.1), np.full(n, 0.1 + 1e-3), np.full(n, 1.0)], axis=1)
    listed = rng.random(n) < share
    lam[~listed, 1] = 0.5
    A = np.einsum("nij,nj,nkj->nik", Q, lam, Q)
    S = np.stack([A[:, 0, 0], A[:, 1, 1], A[:, 2, 2], A[:, 0, 1], A[:, 0, 2], A[:, 1, 2]]).astype(np.float32)
    plan = _lib.ct_plan_create(_lib.make_params(1.0, 2.0, (0, 0, 0), (0, 0, 1), _lib.CT_PREC_MIXED), (8, 8, 8))
    try:
        ev, vec = torch.empty((3, n), device="cuda"), torch.full((3, n), 7.0, device="cuda")
        _lib.ct_eig_smallest(plan, torch.from_numpy(S).cuda(), n, ev, vec)
        assert _lib.ct_plan_stats(plan)["fallback_voxels"] == int(listed.sum())
    finally:
        _lib.ct_plan_destroy(plan)
    _, v = O.eig_field(S.astype(np.float64))
    cosang = np.abs((vec.cpu().numpy().astype(np.float64) * v).sum(0))
    # the cosine of two unit vectors, one rounded to FP32, is within 4e-7 of 1: 0.06 deg
    assert cosang[listed].min(initial=1.0) >= 1 - 4e-7
    assert cosang.min() > math.cos(math.radians(0.15))


@pytest.mark.parametrize("scale", [1e-12, 1.0, 1e12, 1e30])
@pytest.mark.parametrize("gap", [5e-3, 1e-4, 1e-6, 0.0])
def test_fp64_resolve_over_gaps_and_scales(scale, gap):
    """The re-solve's eigenvalues and direction against FP64 LAPACK on the same FP32 tensor: the
    direction within 1e-15 / gap (the perturbation of FP64 rounding, with margin) and the FP32
    rounding of the outputs; any direction of the plane for an exact pair."""
    rng = np.random.default_rng(3)
    n = 4000
    Q, _ = np.linalg.qr(rng.normal(size=(n, 3, 3)))
    lam = np.stack([np.full(n, 0.2), np.full(n, 0.2 + 0.8 * gap), np.ones(n)], axis=1)
    if gap == 0.0:  # axis-aligned, so that the FP32 tensor holds the exact pair
        P = np.stack([np.roll(np.eye(3), k % 3, axis=0) for k in range(n)])
        Q = P
    A = np.einsum("nij,nj,nkj->nik", Q, lam, Q) * scale
    S = np.stack([A[:, 0, 0], A[:, 1, 1], A[:, 2, 2], A[:, 0, 1], A[:, 0, 2], A[:, 1, 2]]).astype(np.float32)
    plan = _lib.ct_plan_create(_lib.make_params(1.0, 2.0, (0, 0, 0), (0, 0, 1), _lib.CT_PREC_MIXED), (8, 8, 8))
    try:
        ev, vec = torch.empty((3, n), device="cuda"), torch.empty((3, n), device="cuda")
        _lib.ct_eig_smallest(plan, torch.from_numpy(S).cuda(), n, ev, vec)
        torch.cuda.synchronize()
    finally:
        _lib.ct_plan_destroy(plan)
    S = S.astype(np.float64) / scale
    M = np.stack([np.stack([S[0], S[3], S[4]]), np.stack([S[3], S[1], S[5]]), np.stack([S[4], S[5], S[2]])])
    l, V = np.linalg.eigh(M.transpose(2, 0, 1))
    v = vec.cpu().numpy().astype(np.float64)
    assert np.abs(np.linalg.norm(v, axis=0) - 1).max() <= 1e-6
    assert np.abs(ev.cpu().numpy().astype(np.float64) / scale - l.T).max() <= 1e-6
    # the angle of v out of the plane of the smallest pair, and within it
    out = np.abs((v * V[:, :, 2].T).sum(0))
    assert out.max() <= 1e-6
    if gap > 0.0:
        across = np.abs((v * V[:, :, 1].T).sum(0))
        real = l[:, 1] - l[:, 0]
        assert np.all(across <= 4e-7 + 4e-15 / real)


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 8), (3, 1, 9), (1, 7, 16), (40, 300, 24), (2, 2, 4096), (257, 3, 8)])
@pytest.mark.parametrize("ha_type", [F32, F16, U8Q])
@pytest.mark.parametrize("masked", [False, True])
def test_profile_counts_every_voxel_once(shape, ha_type, masked):
    """Totals and bins of small and degenerate boxes.  Depth edges and HA values lie well inside
    their bins (HA at bin centres, voxel radii on no edge), so the counts are exact."""
    rng = np.random.default_rng(sum(shape))
    nz, ny, nx = shape
    nd, nh = 3, 16
    code = rng.integers(0, nh, size=shape)
    ha = (code + 0.5) * (180.0 / nh) - 90.0
    if ha_type == U8Q:
        field = np.rint((ha + 90.0) * 256.0 / 180.0).astype(np.uint8)
        decoded = field.astype(np.float64) * 180.0 / 256.0 - 90.0
    else:
        field = ha.astype({F32: np.float32, F16: np.float16}[ha_type])
        field[rng.random(shape) < 0.1] = np.nan
        decoded = field.astype(np.float64)
    mask = (rng.random(shape) < 0.4).astype(np.uint8) if masked else None
    # axis far to the side: radii from about 5000 on, three depth bins over the box
    cen, ax = (-5000.123, ny / 2.0, 0.0), (0.0, 0.0, 1.0)
    r_in, r_out = 4999.7, 5000.123 + nx + 0.4
    d = OP.depth_field(shape, (0, 0, 0), cen, ax, r_in, r_out) * nd
    sure = np.abs(d - np.round(d)) > 1e-2
    m = sure if mask is None else sure & mask.astype(bool)
    spec = _lib.make_profile_spec(cen, ax, r_in, r_out, nd, nh, ha_type)
    hist = torch.zeros(nd * nh, dtype=torch.int64, device="cuda")
    dm = None if mask is None and sure.all() else torch.from_numpy(m.astype(np.uint8)).cuda()
    _lib.ct_transmural_profile(spec, (nx, ny, nz), (0, 0, 0), (nx, ny, nz), torch.from_numpy(field).cuda(), dm, hist)
    torch.cuda.synchronize()
    ora = OP.transmural_profile(decoded, m.astype(np.uint8), (0, 0, 0), cen, ax, r_in, r_out, nd, nh)
    np.testing.assert_array_equal(hist.cpu().numpy(), np.asarray(ora).reshape(-1).astype(np.int64))
