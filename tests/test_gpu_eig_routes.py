"""Unmasked eigen stages on either side of the widths that walk a row per CTA: the outputs of a
mask of ones, to the bit."""
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


@pytest.mark.parametrize("nx", [1, 31, 32, 33, 64, 66, 96, 97, 128, 130, 160, 161, 512, 514, 640, 641, 1024, 1026, 1152, 1153])
@pytest.mark.parametrize("types", [(_lib.CT_OUT_F32,) * 3, (_lib.CT_OUT_F32, _lib.CT_OUT_U8Q, _lib.CT_OUT_F16)])
def test_rows_of_every_route_equal_the_masked_form(nx, types):
    vol = np.random.default_rng(nx).integers(500, 3000, size=(4, 5, nx)).astype(np.uint16)
    vol[:, :, : nx // 4] = 1500
    kw = dict(vec_type=types[0], angle_type=types[1], fa_type=types[2], raw=True)
    cen, ax = (nx / 2 + 0.3, 2.0, 1.0), (0.1, 0.0, 1.0)
    a = G.fused(vol, 1.0, 2.0, cen, ax, **kw)
    b = G.fused(vol, 1.0, 2.0, cen, ax, mask=np.ones_like(vol, dtype=np.uint8), **kw)
    for k in ("v", "ha", "ia", "fa"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert a["stats"]["fallback_voxels"] == b["stats"]["fallback_voxels"]
