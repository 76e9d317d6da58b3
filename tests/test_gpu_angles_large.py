"""ct_angles on either side of the size from which a thread takes four voxels: the same values as
a voxel per thread (arrays off the vector boundary), to the bit."""
import numpy as np
import pytest

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


def _at(t, shift):
    o = torch.empty(t.numel() + shift, dtype=t.dtype, device="cuda")[shift:]
    o.copy_(t.reshape(-1))
    return o


# 2^18 - 4, 2^18 and 2^18 + 4 voxels, rows that groups of four cross, no multiple of four, several groups per thread
@pytest.mark.parametrize("dims", [(65535, 2, 2), (64, 64, 64), (65537, 2, 2), (31, 17, 500), (33, 5, 1589), (301, 263, 160)])
@pytest.mark.parametrize("types", [(F32, F32, F32), (F16, F16, F16), (F32, U8Q, F16), (F16, F32, F32)])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("spacing", [(0.0, 0.0, 0.0), (1.0, 1.5, 2.0)])
def test_four_voxels_per_thread_equal_one(dims, types, masked, spacing):
    n = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cuda").manual_seed(n)
    v = torch.randn((3, n), device="cuda", generator=g)
    v /= v.norm(dim=0)
    ev = torch.rand((3, n), device="cuda", generator=g).sort(dim=0).values
    mask = (torch.rand(n, device="cuda", generator=g) < 0.5).to(torch.uint8) if masked else None
    if masked:
        mask[n // 3: n // 2] = 0
    params = _lib.make_params(1.0, 2.0, (dims[0] / 2 + 0.3, dims[1] / 2 - 0.2, 1.0), (0.1, -0.2, 1.0),
                              vec_type=types[0], angle_type=types[1], fa_type=types[2], spacing=spacing)
    plan = _lib.ct_plan_create(params, dims)
    try:
        got = []
        for shift in (0, 1):
            o = [_at(torch.zeros(k * n, dtype=DT[t], device="cuda"), shift)
                 for k, t in zip((3, 1, 1, 1), (types[0], types[1], types[1], types[2]))]
            _lib.ct_angles(plan, _at(v, shift), _at(ev, shift), (0, 0, 0), dims, None if mask is None else _at(mask, shift),
                           *o)
            torch.cuda.synchronize()
            got.append([t.cpu().numpy() for t in o])
    finally:
        _lib.ct_plan_destroy(plan)
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
