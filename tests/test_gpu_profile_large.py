"""The profile kernel where a CTA takes tiles of several segments per thread and several tiles, and
voxels whose radius lies exactly on a depth bin's edge: counts equal the oracle's.

No tolerance: HA lies at bin centres, and every depth either lies more than 1e-3 of a bin
from an edge (others are not counted) or is exact in FP32 and FP64 alike."""
import numpy as np
import pytest

from oracle import profile as OP
from paper_2508_07476_gb300 import _lib, build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

F32, F16, U8Q = _lib.CT_OUT_F32, _lib.CT_OUT_F16, _lib.CT_OUT_U8Q


@pytest.fixture(scope="module", autouse=True)
def _ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    _lib.load()


def _field(rng, shape, nh, ha_type, dropped):
    """(encoded HA at bin centres, its FP64 values), without a value where `dropped` is set."""
    ha = (rng.integers(0, nh, size=shape, dtype=np.int16) + 0.5) * (180.0 / nh) - 90.0
    if ha_type == U8Q:
        field = np.rint((ha + 90.0) * 256.0 / 180.0).astype(np.uint8)
        field[dropped] = 0
        return field, np.where(field == 0, np.nan, field * (180.0 / 256.0) - 90.0)
    field = ha.astype({F32: np.float32, F16: np.float16}[ha_type])
    field[dropped] = np.nan
    return field, field.astype(np.float64)


def _counts(field, mask, cen, ax, r_in, r_out, nd, nh, ha_type):
    nz, ny, nx = field.shape
    hist = torch.zeros(nd * nh, dtype=torch.int64, device="cuda")
    _lib.ct_transmural_profile(_lib.make_profile_spec(cen, ax, r_in, r_out, nd, nh, ha_type), (nx, ny, nz), (0, 0, 0),
                               (nx, ny, nz), torch.from_numpy(field).cuda(),
                               None if mask is None else torch.from_numpy(mask).cuda(), hist)
    torch.cuda.synchronize()
    return hist.cpu().numpy().reshape(nd, nh)


# 152 SMs, 5 CTAs of 256 threads each: 2 segments per thread and tile from 389 120 segments on, 16 from
# 3.1 million on, and more tiles than CTAs just above such a size
@pytest.mark.parametrize("shape,ha_type,masked", [
    ((40, 330, 256), F32, True),    # 2 per thread, 825 tiles
    ((40, 330, 251), U8Q, True),    # the same, rows of ragged segments
    ((47, 401, 256), F16, False),   # 3 per thread
    ((60, 300, 509), F32, True),    # 5 per thread, ragged
    ((64, 250, 520), U8Q, False),   # 5 per thread
    ((70, 347, 504), F16, True),    # 7 per thread
    ((200, 250, 504), F32, True),   # 16 per thread, 770 tiles
    ((203, 251, 497), F16, False),  # 16 per thread, ragged
])
def test_counts_of_large_fields(shape, ha_type, masked):
    rng = np.random.default_rng(sum(shape))
    nz, ny, nx = shape
    nd, nh = 20, 36
    cen, ax = (nx * 0.52 + 0.137, ny * 0.47 + 0.211, nz / 2.0), (0.17, -0.05, 0.98)
    r_in, r_out = 0.1 * nx + 0.03, 0.45 * nx + 0.3
    d = OP.depth_field(shape, (0, 0, 0), cen, ax, r_in, r_out) * nd
    near = np.abs(d - np.round(d)) <= 1e-3
    field, decoded = _field(rng, shape, nh, ha_type, near)
    mask = None
    if masked:  # whole segments, tiles and planes outside, and single voxels
        mask = (rng.random(shape) < 0.8).astype(np.uint8)
        mask[:, : ny // 3] = 0
        mask[nz // 3: nz // 2] = 0
    ora = OP.transmural_profile(decoded, mask, (0, 0, 0), cen, ax, r_in, r_out, nd, nh)
    assert ora.sum() > 100000
    got = _counts(field, mask, cen, ax, r_in, r_out, nd, nh, ha_type)
    np.testing.assert_array_equal(got, ora.astype(np.int64))


@pytest.mark.parametrize("shape", [(3, 150, 151), (5, 151, 152), (64, 250, 520)])
@pytest.mark.parametrize("masked", [False, True])
def test_radii_on_bin_edges(shape, masked):
    """Bins one voxel wide around an axis through voxel centres: every integer radius lies on an edge,
    the range's ends among them.  Squared radii are integers below 2^24 and bin widths powers of
    two, so the definition's FP32 arithmetic is exact on the edges and far from them elsewhere."""
    rng = np.random.default_rng(sum(shape))
    nz, ny, nx = shape
    nd, nh = 64, 30
    cen, ax = (float(nx // 2), float(ny // 2), 1.0), (0.0, 0.0, 1.0)
    field, decoded = _field(rng, shape, nh, F32, rng.random(shape) < 0.05)
    mask = (rng.random(shape) < 0.6).astype(np.uint8) if masked else None
    d = OP.depth_field((1, ny, nx), (0, 0, 1), cen, ax, 5.0, 69.0) * nd
    assert ((d == np.round(d)) & (d >= 0) & (d <= nd)).sum() > 300  # edge voxels of one plane
    ora = OP.transmural_profile(decoded, mask, (0, 0, 0), cen, ax, 5.0, 69.0, nd, nh)
    got = _counts(field, mask, cen, ax, 5.0, 69.0, nd, nh, F32)
    np.testing.assert_array_equal(got, ora.astype(np.int64))
