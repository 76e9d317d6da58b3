"""The library's work as its users give it, one case each: whole volumes, padded
chunks, batches of crops, host-resident volumes and the single stages, through
the entry points of ``paper_2508_07476_gb300._lib``.

A case is a dict of plain values; ``kind`` names the call:

  volume   ct_run_chunks on one device-resident volume
  box      ct_run_box on one padded chunk of a larger volume
  crops    ct_run_chunks on a batch of uneven device-resident crops
  host     ct_run_chunks on a volume in pinned host memory, slab by slab
  tensor   ct_structure_tensor on a whole volume
  eig      ct_eig_smallest on a field of tensors
  angles   ct_angles on a field of eigenvectors and eigenvalues
  profile  ct_transmural_profile of an HA map
  track    ct_track through a fibre field

``exact`` computes the same outputs in FP64 with torch alone, from the
definitions in ``include/ct.h``.
"""
import dataclasses
import math
import random

import torch

from paper_2508_07476_gb300 import _lib, synth

PREC = {"fp32": _lib.CT_PREC_FP32, "mixed": _lib.CT_PREC_MIXED}
# encodings of (vector, HA / IA, FA); "u8q" has no vector output (the teravoxel stream's outputs)
ENC = {"f32": (_lib.CT_OUT_F32, _lib.CT_OUT_F32, _lib.CT_OUT_F32),
       "f16": (_lib.CT_OUT_F16, _lib.CT_OUT_F16, _lib.CT_OUT_F16),
       "u8q": (_lib.CT_OUT_F32, _lib.CT_OUT_U8Q, _lib.CT_OUT_F16)}
DTYPE = {_lib.CT_OUT_F32: torch.float32, _lib.CT_OUT_F16: torch.float16, _lib.CT_OUT_U8Q: torch.uint8}
TILT = (math.sin(math.radians(10.0)), 0.0, math.cos(math.radians(10.0)))


def listed():
    return [
        # one small volume on its own, FP32 form: the smallest call, where launches and latency count
        dict(name="volume64", kind="volume", nx=64, ny=64, nz=64, sigma=1.0, rho=3.0, prec="fp32", out="f32",
             masked=False),
        # one ragged crop of a scan, odd on every axis
        dict(name="volume_ragged", kind="volume", nx=173, ny=141, nz=118, sigma=1.5, rho=4.0, prec="mixed",
             out="f16", masked=False),
        # the benchmark's volume: a left-ventricle wall with its mask, everything resident
        dict(name="volume512", kind="volume", nx=512, ny=512, nz=512, sigma=2.0, rho=6.0, prec="mixed", out="f32",
             masked=True),
        # one chunk of a 2048 x 2048 x 1024 scan streamed in 256^3 chunks, half-precision outputs
        dict(name="chunk256", kind="box", dx=2048, dy=2048, dz=1024, r_in=480.0, r_out=880.0, period=8.0,
             x=1536, y=1024, z=512, nx=256, ny=256, nz=256, sigma=2.0, rho=8.0, prec="mixed", out="f16",
             masked=True),
        # one chunk of the teravoxel stream, quantised angles
        dict(name="chunk384_u8q", kind="box", dx=4096, dy=4096, dz=2048, r_in=1000.0, r_out=1800.0, period=10.0,
             x=3072, y=2304, z=768, nx=384, ny=384, nz=384, sigma=3.0, rho=9.0, prec="mixed", out="u8q",
             masked=True),
        # many uneven crops with their own scales and frames in one call
        dict(name="crops12", kind="crops", count=12, lo=64, hi=384, shape_seed=4, prec="mixed", out="f16"),
        # a scan held in pinned host memory, whole planes at a time
        dict(name="host_slabs", kind="host", nx=512, ny=512, nz=256, cx=0, cy=0, cz=64, sigma=2.0, rho=8.0,
             prec="mixed", out="f16", masked=True),
        # the tensor alone, FP32 form, for a caller with a solver of their own
        dict(name="tensor_ragged", kind="tensor", nx=250, ny=203, nz=190, sigma=2.0, rho=6.0, prec="fp32"),
        # the eigen-decomposition alone over a 256^3 field
        dict(name="eig_256", kind="eig", n=256 ** 3, prec="mixed"),
        # the angles alone over a masked 256^3 field
        dict(name="angles_256", kind="angles", nx=256, ny=256, nz=256, out="f16", masked=True),
        # the transmural HA profile of the benchmark's volume
        dict(name="profile512", kind="profile", nx=512, ny=512, nz=512, out="f32", masked=True, depth=20, bins=180),
        # tractography through the benchmark's wall
        dict(name="track_200k", kind="track", nx=512, ny=512, nz=512, seeds=200000, steps=200, step=0.5,
             masked=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["volume", "volume", "volume", "box", "crops", "host", "tensor", "eig", "angles", "profile",
                       "track"])
    sigma = rng.choice([1.0, 1.5, 2.0, 3.0])
    rho = rng.choice([2.0, 3.0, 4.0, 6.0, 8.0, 9.0])
    prec = rng.choice(["fp32", "mixed", "mixed"])
    masked = rng.random() < 0.6
    if kind in ("volume", "tensor"):
        top = _log_int(rng, 64, 384)  # one size class per case, its axes uneven within it
        n = [max(48, int(top * rng.uniform(0.6, 1.0))) for _ in range(3)]
        if rng.random() < 0.4:
            n[0] = (n[0] + 7) // 8 * 8
        c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], sigma=sigma, rho=rho, prec=prec)
        if kind == "volume":
            c.update(out=rng.choice(["f32", "f16", "u8q"]), masked=masked)
        return c
    if kind == "box":
        d = rng.choice([(1024, 1024, 512, 240.0, 440.0), (2048, 2048, 1024, 480.0, 880.0),
                        (4096, 4096, 2048, 1000.0, 1800.0)])
        n = [rng.choice([96, 128, 192, 256, 320, _log_int(rng, 90, 320)]) for _ in range(3)]
        a, r = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(d[3], d[4])
        at = [d[0] / 2 + r * math.cos(a), d[1] / 2 + r * math.sin(a), rng.uniform(0.0, d[2])]
        lo = [min(max(0, int(at[k] - n[k] / 2)), d[k] - n[k]) for k in range(3)]
        if rng.random() < 0.6:  # most chunk grids start on multiples of the chunk size
            lo = [lo[k] // n[k] * n[k] for k in range(3)]
        return dict(kind="box", dx=d[0], dy=d[1], dz=d[2], r_in=d[3], r_out=d[4], period=8.0, x=lo[0], y=lo[1],
                    z=lo[2], nx=n[0], ny=n[1], nz=n[2], sigma=sigma, rho=rho, prec=prec,
                    out=rng.choice(["f32", "f16", "u8q"]), masked=masked)
    if kind == "crops":
        return dict(kind="crops", count=rng.randint(2, 12), lo=64, hi=rng.choice([128, 192, 256, 384]),
                    shape_seed=rng.randint(5, 1 << 20), prec=prec, out=rng.choice(["f32", "f16"]))
    if kind == "host":
        n = [_log_int(rng, 96, 512) for _ in range(3)]
        ch = rng.choice([(0, 0, 0), (0, 0, 32), (0, 0, 64), (128, 128, 128), (256, 256, 256)])
        return dict(kind="host", nx=n[0], ny=n[1], nz=min(n[2], 256), cx=ch[0], cy=ch[1], cz=ch[2], sigma=sigma,
                    rho=rho, prec=prec, out=rng.choice(["f32", "f16", "u8q"]), masked=masked)
    if kind == "eig":
        return dict(kind="eig", n=_log_int(rng, 1 << 14, 1 << 25), prec=prec)
    if kind == "angles":
        n = [_log_int(rng, 32, 384) for _ in range(3)]
        return dict(kind="angles", nx=n[0], ny=n[1], nz=n[2], out=rng.choice(["f32", "f16", "u8q"]), masked=masked)
    if kind == "profile":
        n = [_log_int(rng, 64, 512) for _ in range(3)]
        return dict(kind="profile", nx=n[0], ny=n[1], nz=n[2], out=rng.choice(["f32", "f16", "u8q"]), masked=masked,
                    depth=rng.choice([10, 20, 50]), bins=rng.choice([36, 90, 180]))
    m = _log_int(rng, 128, 512)
    return dict(kind="track", nx=m, ny=m, nz=rng.choice([m // 2, m]), seeds=_log_int(rng, 1000, 200000),
                steps=rng.choice([50, 100, 200]), step=rng.choice([0.25, 0.5, 1.0]), masked=masked)


# ---------------------------------------------------------------- inputs

def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(seed)


def _dims(c):
    return (c["nx"], c["ny"], c["nz"])


def _wall(c, seed):
    """The wall a volume of the case's size holds: the benchmark's annulus, scaled to it."""
    m = min(c["nx"], c["ny"])
    return synth.AnnulusSpec(shape=(c["nz"], c["ny"], c["nx"]), r_in=m * 120.0 / 512.0, r_out=m * 220.0 / 512.0,
                             period=6.0, ha_in_deg=70.0, ha_out_deg=-70.0, axis=TILT, noise=("poisson_like", 0.05),
                             ia_std_deg=5.0, ia_corr=40.0, seed=seed)


def _scan(spec, dims, lo, n, masked):
    """(volume, mask or None) of the box (lo, n), generated on the device."""
    vol = torch.empty((n[2], n[1], n[0]), dtype=torch.int16, device="cuda")
    mask = torch.empty((n[2], n[1], n[0]), dtype=torch.uint8, device="cuda") if masked else None
    _lib.ct_synth_annulus(spec, dims, lo, n, vol, mask, flags=_lib.CT_SYNTH_FP32)
    return vol, mask


def _halo(c):
    return _radius(c["sigma"]) + _radius(c["rho"])


def _radius(s):
    return int(math.floor(4.0 * s + 0.5))


def _grow(lo, n, r, dims):
    a = [max(0, lo[k] - r) for k in range(3)]
    b = [min(dims[k], lo[k] + n[k] + r) for k in range(3)]
    return a, [b[k] - a[k] for k in range(3)]


def _box_inputs(c, seed):
    """(spec, volume dims, input box, output box, volume over the input box, mask over the output box)."""
    dims, lo, n = (c["dx"], c["dy"], c["dz"]), (c["x"], c["y"], c["z"]), _dims(c)
    spec = synth.AnnulusSpec(shape=(dims[2], dims[1], dims[0]), r_in=c["r_in"], r_out=c["r_out"], period=c["period"],
                             ha_in_deg=70.0, ha_out_deg=-70.0, axis=TILT, noise=("poisson_like", 0.05),
                             ia_std_deg=5.0, ia_corr=40.0, seed=seed)
    ilo, inn = _grow(lo, n, _halo(c), dims)
    vol, _ = _scan(spec, dims, ilo, inn, False)
    mask = None
    if c["masked"]:
        mask = torch.empty((n[2], n[1], n[0]), dtype=torch.uint8, device="cuda")
        _lib.ct_synth_annulus(spec, dims, lo, n, None, mask, flags=_lib.CT_SYNTH_FP32)
    return spec, dims, (ilo, inn), (lo, n), vol, mask


def _crop_inputs(c, seed):
    """[(workload, volume)] of the batch: sizes, scales and frames from the case, voxels from the seed."""
    got = []
    for j, w in enumerate(synth.crop_batch(c["count"], c["shape_seed"], (c["lo"], c["hi"]))):
        spec = dataclasses.replace(w.spec, seed=seed * 64 + j)
        nz, ny, nx = spec.shape
        got.append((w, _scan(spec, (nx, ny, nz), (0, 0, 0), (nx, ny, nz), False)[0]))
    return got


def _eig_inputs(c, seed):
    """n tensors as six planes: fibre-like spectra (one small eigenvalue, two larger ones) in random
    orientations; in one of 50 the two smallest meet within a few percent (texture without a
    direction), and one of 200 is zero (constant background)."""
    n, g = c["n"], _gen(seed)
    q = torch.randn((4, n), device="cuda", generator=g)
    q = q / q.norm(dim=0)
    w, x, y, z = q[0], q[1], q[2], q[3]
    rot = ((1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)),
           (2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)),
           (2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)))
    u = torch.rand((4, n), device="cuda", generator=g)
    top = 2000.0 * torch.exp(1.5 * torch.randn(n, device="cuda", generator=g))
    ev = [top * (0.02 + 0.2 * u[0]), top * (0.35 + 0.4 * u[1]), top]
    ev[1] = torch.where(u[2] < 0.02, ev[0] * (1 + 0.1 * u[1]), ev[1])
    zero = u[3] < 0.005
    ev = [torch.where(zero, torch.zeros_like(e), e) for e in ev]
    S = torch.empty((6, n), device="cuda")
    for k, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        S[k] = sum(ev[m] * rot[a][m] * rot[b][m] for m in range(3))
    return S


def _frame(dims):
    return tuple((d - 1) / 2.0 for d in dims), TILT


def _local(dims):
    """Voxel positions, their distance from the axis, height along it, and the frame (e_t, e_r), in FP32."""
    cen, ax = _frame(dims)
    pos = [torch.arange(dims[k], device="cuda", dtype=torch.float32) - cen[k] for k in range(3)]
    d = [pos[0][None, None, :], pos[1][None, :, None], pos[2][:, None, None]]
    h = d[0] * ax[0] + d[1] * ax[1] + d[2] * ax[2]
    r = [d[k] - h * ax[k] for k in range(3)]
    rr = (r[0] ** 2 + r[1] ** 2 + r[2] ** 2).sqrt()
    er = [q / rr.clamp_min(1e-6) for q in r]
    et = [ax[1] * er[2] - ax[2] * er[1], ax[2] * er[0] - ax[0] * er[2], ax[0] * er[1] - ax[1] * er[0]]
    return rr, et, er, ax


def _wall_field(c, seed, jitter):
    """(vectors, mask, depth) of a helical wall: HA from +70 deg to -70 deg through it, with `jitter`
    of noise per component; vectors unit, oriented along e_t."""
    dims = _dims(c)
    m = min(dims[0], dims[1])
    rr, et, er, ax = _local(dims)
    depth = (rr - m * 120.0 / 512.0) / (m * 100.0 / 512.0)
    mask = ((depth >= 0) & (depth <= 1)).to(torch.uint8)
    ha = torch.deg2rad(70.0 - 140.0 * depth.clamp(0, 1))
    co, si = ha.cos(), ha.sin()
    g = _gen(seed)
    v = torch.stack([co * et[k] + si * ax[k] for k in range(3)])
    del et, er, rr
    v += jitter * torch.randn(v.shape, device="cuda", generator=g)
    v /= v.norm(dim=0)
    return v, mask, depth


def _angle_inputs(c, seed):
    v, mask, _ = _wall_field(c, seed, 0.08)
    g = _gen(seed + 1)
    # the stage's input convention: the largest component positive
    big = v.gather(0, v.abs().argmax(dim=0, keepdim=True))
    v *= torch.where(big < 0, -1.0, 1.0)
    u = torch.rand(v.shape, device="cuda", generator=g)
    l3 = 5000.0 * torch.exp(1.2 * torch.randn(v.shape[1:], device="cuda", generator=g))
    ev = torch.stack([l3 * (0.3 * u[0]), l3 * (0.35 + 0.6 * u[1]), l3])
    return v.contiguous(), ev, (mask if c["masked"] else None)


def _profile_inputs(c, seed):
    """The HA map of a wall (noise of 6 deg, fill outside the mask) and its mask."""
    _, mask, depth = _wall_field(c, seed, 0.0)
    g = _gen(seed + 2)
    ha = 70.0 - 140.0 * depth.clamp(0, 1) + 6.0 * torch.randn(depth.shape, device="cuda", generator=g)
    ha = (ha + 90.0) % 180.0 - 90.0
    if c["out"] == "u8q":
        ha = torch.where(mask != 0, torch.round((ha + 90.0) * (256.0 / 180.0)) % 256, torch.zeros_like(ha))
        ha = ha.to(torch.uint8)
    else:
        ha = torch.where(mask != 0, ha, torch.full_like(ha, math.nan)).to(DTYPE[ENC[c["out"]][1]])
    return ha, (mask if c["masked"] else None)


def _track_inputs(c, seed):
    """A wall's fibre field (NaN outside), its FA, its mask, and seeds spread over the wall."""
    dims = _dims(c)
    v, mask, _ = _wall_field(c, seed, 0.05)
    v = torch.where(mask != 0, v, torch.full_like(v, math.nan))
    g = _gen(seed + 3)
    fa = 0.25 + 0.5 * torch.rand(mask.shape, device="cuda", generator=g)
    m, n = min(dims[0], dims[1]), c["seeds"]
    cen, ax = _frame(dims)
    u = torch.rand((3, n), device="cuda", generator=g)
    r = m * (130.0 + 80.0 * u[0]) / 512.0
    a = 2.0 * math.pi * u[1]
    h = (dims[2] - 1) * (0.1 + 0.8 * u[2]) - cen[2]
    # in the plane at height h: the axis crosses it at an offset along x
    seeds = torch.stack([cen[0] + h * ax[0] / ax[2] + r * a.cos(), cen[1] + r * a.sin(), cen[2] + h], dim=1)
    return v.contiguous(), fa, (mask if c["masked"] else None), seeds.contiguous()


# ---------------------------------------------------------------- the calls

class Plan:
    """A plan that goes with its state."""

    def __init__(self, dims, sigma, rho, cen, ax, prec, out, chunk=(0, 0, 0)):
        vt, at, ft = ENC[out]
        self.h = _lib.ct_plan_create(_lib.make_params(sigma, rho, cen, ax, PREC[prec], vt, at, ft, chunk=chunk), dims)

    def __del__(self):
        if getattr(self, "h", None):
            _lib.ct_plan_destroy(self.h)


def _outputs(out, n, **where):
    vt, at, ft = ENC[out]
    shape = (n[2], n[1], n[0])
    where = where or dict(device="cuda")
    o = {} if out == "u8q" else {"vec": torch.empty((3,) + shape, dtype=DTYPE[vt], **where)}
    o["ha"] = torch.empty(shape, dtype=DTYPE[at], **where)
    o["ia"] = torch.empty(shape, dtype=DTYPE[at], **where)
    o["fa"] = torch.empty(shape, dtype=DTYPE[ft], **where)
    return o


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("volume", "host", "tensor"):
        dims = _dims(c)
        spec = _wall(c, seed)
        vol, mask = _scan(spec, dims, (0, 0, 0), dims, c.get("masked", False))
        cen, ax = synth.frame_of(spec)
        chunk = (c["cx"], c["cy"], c["cz"]) if kind == "host" else (0, 0, 0)
        plan = Plan(dims, c["sigma"], c["rho"], cen, ax, c["prec"], c.get("out", "f32"), chunk)
        if kind == "tensor":
            return {"kind": kind, "plan": plan, "dims": dims, "vol": vol,
                    "S": torch.empty((6, dims[2], dims[1], dims[0]), device="cuda")}
        where = {}
        if kind == "host":
            where = dict(device="cpu", pin_memory=True)
            vol = vol.cpu().pin_memory()
            mask = None if mask is None else mask.cpu().pin_memory()
        o = _outputs(c["out"], dims, **where)
        item = _lib.make_item(vol, dims, mask, o.get("vec"), o["ha"], o["ia"], o["fa"])
        return {"kind": kind, "plan": plan, "items": [item], "out": o, "keep": (vol, mask)}
    if kind == "box":
        spec, dims, ib, ob, vol, mask = _box_inputs(c, seed)
        cen, ax = synth.frame_of(spec)
        plan = Plan(dims, c["sigma"], c["rho"], cen, ax, c["prec"], c["out"])
        return {"kind": kind, "plan": plan, "ib": ib, "ob": ob, "vol": vol, "mask": mask,
                "out": _outputs(c["out"], ob[1])}
    if kind == "crops":
        plan = Plan((1, 1, 1), 2.0, 6.0, (0.0, 0.0, 0.0), (0.0, 0.0, 1.0), c["prec"], c["out"])
        items, outs, keep = [], [], []
        for w, vol in _crop_inputs(c, seed):
            dims = w.spec.shape[::-1]
            o = _outputs(c["out"], dims)
            cen, ax = synth.frame_of(w.spec)
            items.append(_lib.make_item(vol, dims, None, o["vec"], o["ha"], o["ia"], o["fa"], sigma=w.sigma,
                                        rho=w.rho, lv_center=cen, lv_axis=ax))
            outs.append(o)
            keep.append(vol)
        return {"kind": kind, "plan": plan, "items": items, "out": outs, "keep": keep}
    if kind == "eig":
        S = _eig_inputs(c, seed)
        plan = Plan((64, 64, 64), 1.0, 3.0, (32.0, 32.0, 32.0), (0.0, 0.0, 1.0), c["prec"], "f32")
        return {"kind": kind, "plan": plan, "S": S, "n": c["n"], "evals": torch.empty((3, c["n"]), device="cuda"),
                "evec": torch.empty((3, c["n"]), device="cuda")}
    if kind == "angles":
        v, ev, mask = _angle_inputs(c, seed)
        dims = _dims(c)
        cen, ax = _frame(dims)
        return {"kind": kind, "plan": Plan(dims, 2.0, 6.0, cen, ax, "mixed", c["out"]), "dims": dims, "evec": v,
                "evals": ev, "mask": mask, "out": _outputs(c["out"], dims)}
    if kind == "profile":
        ha, mask = _profile_inputs(c, seed)
        dims = _dims(c)
        m = min(dims[0], dims[1])
        cen, ax = _frame(dims)
        spec = _lib.make_profile_spec(cen, ax, m * 120.0 / 512.0, m * 220.0 / 512.0, c["depth"], c["bins"],
                                      ENC[c["out"]][1])
        return {"kind": kind, "spec": spec, "dims": dims, "ha": ha, "mask": mask,
                "hist": torch.empty((c["depth"], c["bins"]), dtype=torch.int64, device="cuda")}
    v, fa, mask, seeds = _track_inputs(c, seed)
    n = seeds.shape[0]
    # points past a track's count are never written: they stay zero
    return {"kind": kind, "dims": _dims(c), "params": _lib.make_track_params(c["step"], c["steps"], 0.1, 60.0),
            "vec": v, "fa": fa, "mask": mask, "seeds": seeds, "n": n,
            "points": torch.zeros((n, 2, c["steps"] + 1, 3), device="cuda"),
            "count": torch.zeros((n, 2), dtype=torch.int32, device="cuda")}


def run(state):
    s, kind = state, state["kind"]
    if kind in ("volume", "crops"):
        _lib.ct_run_chunks(s["plan"].h, s["items"], False)
        return s["out"]
    if kind == "host":
        _lib.ct_run_chunks(s["plan"].h, s["items"], True)
        return s["out"]
    if kind == "box":
        o = s["out"]
        _lib.ct_run_box(s["plan"].h, s["vol"], *s["ib"], *s["ob"], s["mask"], o.get("vec"), o["ha"], o["ia"], o["fa"])
        return o
    if kind == "tensor":
        lo, n = (0, 0, 0), s["dims"]
        _lib.ct_structure_tensor(s["plan"].h, s["vol"], lo, n, lo, n, s["S"])
        return s["S"]
    if kind == "eig":
        _lib.ct_eig_smallest(s["plan"].h, s["S"], s["n"], s["evals"], s["evec"])
        return {"evals": s["evals"], "evec": s["evec"]}
    if kind == "angles":
        o = s["out"]
        _lib.ct_angles(s["plan"].h, s["evec"], s["evals"], (0, 0, 0), s["dims"], s["mask"], o.get("vec"), o["ha"],
                       o["ia"], o["fa"])
        return o
    if kind == "profile":
        s["hist"].zero_()
        _lib.ct_transmural_profile(s["spec"], s["dims"], (0, 0, 0), s["dims"], s["ha"], s["mask"], s["hist"])
        return s["hist"]
    _lib.ct_track(s["params"], s["dims"], s["vec"], s["fa"], s["mask"], s["seeds"], s["n"], s["points"], s["count"])
    return {"points": s["points"], "count": s["count"]}


# ---------------------------------------------------------------- what a pass cannot do without

def _fma(sigma, rho):
    """Multiply-adds per voxel of the separable definition: eight 1-D gradient passes, the six
    products, eighteen 1-D smoothing passes."""
    return 8 * (2 * _radius(sigma) + 1) + 6 + 18 * (2 * _radius(rho) + 1)


EIG_FLOPS, ANGLE_FLOPS = 150, 80  # operations of one 3x3 solve and of one voxel's angles and FA, about


def _out_bytes(out):
    size = {_lib.CT_OUT_F32: 4, _lib.CT_OUT_F16: 2, _lib.CT_OUT_U8Q: 1}
    vt, at, ft = ENC[out]
    return (0 if out == "u8q" else 3 * size[vt]) + 2 * size[at] + size[ft]


def work(case):
    c, kind = case, case["kind"]
    if kind == "crops":
        b = f = 0
        for w in synth.crop_batch(c["count"], c["shape_seed"], (c["lo"], c["hi"])):
            nz, ny, nx = w.spec.shape
            v = nx * ny * nz
            b += v * (2 + _out_bytes(c["out"]))
            f += v * (2 * _fma(w.sigma, w.rho) + EIG_FLOPS + ANGLE_FLOPS)
        return {"bytes": b, "flops": f}
    if kind == "eig":
        return {"bytes": c["n"] * 48, "flops": c["n"] * EIG_FLOPS}
    if kind == "track":
        # each track's points written, each step's cell of vectors, FA and mask read once
        steps = 2 * c["seeds"] * c["steps"]
        return {"bytes": steps * 12 + 12 * c["seeds"], "flops": steps * 4 * 120}
    v = c["nx"] * c["ny"] * c["nz"]
    if kind == "tensor":
        return {"bytes": v * (2 + 24), "flops": v * 2 * _fma(c["sigma"], c["rho"])}
    m = 1 if c["masked"] else 0
    if kind == "angles":
        return {"bytes": v * (24 + m + _out_bytes(c["out"])), "flops": v * ANGLE_FLOPS}
    if kind == "profile":
        return {"bytes": v * ({"f32": 4, "f16": 2, "u8q": 1}[c["out"]] + m), "flops": v * 20}
    read = v
    if kind == "box":
        _, n = _grow((c["x"], c["y"], c["z"]), _dims(c), _halo(c), (c["dx"], c["dy"], c["dz"]))
        read = n[0] * n[1] * n[2]
    return {"bytes": 2 * read + v * (m + _out_bytes(c["out"])),
            "flops": v * (2 * _fma(c["sigma"], c["rho"]) + EIG_FLOPS + ANGLE_FLOPS)}


# ---------------------------------------------------------------- the same in FP64

def _taps(s):
    r = _radius(s)
    k = torch.arange(-r, r + 1, dtype=torch.float64)
    w = torch.exp(-k * k / (2.0 * s * s))
    w /= w.sum()
    return w.tolist(), (k / (s * s) * w).tolist()


def _filter(x, xlo, dim, olo, on, t, axis):
    """Correlation of x (starting at position xlo on `axis`) with taps t for outputs olo .. olo + on - 1;
    positions outside the volume [0, dim) take the edge voxel."""
    d, r = 2 - axis, len(t) // 2
    a, b = max(0, olo - r), min(dim, olo + on + r)
    x = x.narrow(d, a - xlo, b - a)
    pad = []
    if olo - r < 0:
        pad.append(x.narrow(d, 0, 1).expand([r - olo if k == d else s for k, s in enumerate(x.shape)]))
    pad.append(x)
    if olo + on + r > dim:
        pad.append(x.narrow(d, b - a - 1, 1).expand([olo + on + r - dim if k == d else s
                                                     for k, s in enumerate(x.shape)]))
    x = torch.cat(pad, dim=d) if len(pad) > 1 else x
    y = torch.zeros([on if k == d else s for k, s in enumerate(x.shape)], dtype=torch.float64, device=x.device)
    for j, w in enumerate(t):
        if w != 0.0:
            y.add_(x.narrow(d, j, on), alpha=w)
    return y


def _tensor64(vol, ib, ob, dims, sigma, rho):
    """The six planes of S over the output box from the uint16 voxels of the input box."""
    ws, cs = _taps(sigma)
    wr, _ = _taps(rho)
    glo, gn = _grow(ob[0], ob[1], _radius(rho), dims)
    img = (vol.to(torch.int32) & 0xffff).double()
    g = []
    for k in range(3):
        f = img
        for a in (2, 1, 0):
            f = _filter(f, ib[0][a], dims[a], glo[a], gn[a], cs if a == k else ws, a)
        g.append(f)
    del img
    S = []
    for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)):
        f = g[a] * g[b]
        for x in (2, 1, 0):
            f = _filter(f, glo[x], dims[x], ob[0][x], ob[1][x], wr, x)
        S.append(f)
    return S


def _eig64(S):
    """Eigenvalues ascending and a unit eigenvector of the smallest, from six FP64 planes (flat)."""
    a, b, c, d, e, f = S
    q = (a + b + c) / 3.0
    aq, bq, cq = a - q, b - q, c - q
    p = ((aq * aq + bq * bq + cq * cq + 2.0 * (d * d + e * e + f * f)) / 6.0).sqrt()
    flat = p == 0
    ps = torch.where(flat, torch.ones_like(p), p)
    det = (aq * (bq * cq - f * f) - d * (d * cq - f * e) + e * (d * f - bq * e)) / ps ** 3
    phi = torch.acos((0.5 * det).clamp(-1.0, 1.0)) / 3.0
    l3 = q + 2.0 * p * torch.cos(phi)
    l1 = q + 2.0 * p * torch.cos(phi + 2.0 * math.pi / 3.0)
    l2 = 3.0 * q - l1 - l3
    l1, l2 = torch.minimum(l1, l2), torch.maximum(l1, l2)
    r = torch.stack([torch.stack([a - l1, d, e]), torch.stack([d, b - l1, f]), torch.stack([e, f, c - l1])])
    best, size = None, None
    for i, j in ((0, 1), (0, 2), (1, 2)):
        v = torch.cross(r[i], r[j], dim=0)
        n = (v * v).sum(0)
        if best is None:
            best, size = v, n
        else:
            best, size = torch.where(n > size, v, best), torch.maximum(n, size)
    none = flat | (size == 0)
    best = best / torch.where(none, torch.ones_like(size), size).sqrt()
    best[0] = torch.where(none, torch.ones_like(size), best[0])
    best[1:] = torch.where(none, torch.zeros_like(size), best[1:])
    return torch.stack([l1, l2, l3]), best


def _angles64(v, l, at, cen, ax):
    """(oriented vector, HA, IA, FA) of flat FP64 vectors and eigenvalues at voxel positions `at` (x, y, z)."""
    s = math.sqrt(sum(x * x for x in ax))
    a = [x / s for x in ax]
    d = [at[k] - cen[k] for k in range(3)]
    h = sum(d[k] * a[k] for k in range(3))
    r = [d[k] - h * a[k] for k in range(3)]
    rr = sum(x * x for x in r).sqrt()
    er = [x / rr for x in r]
    et = [a[1] * er[2] - a[2] * er[1], a[2] * er[0] - a[0] * er[2], a[0] * er[1] - a[1] * er[0]]
    vr, vt, vz = (sum(v[k] * w[k] for k in range(3)) for w in (er, et, a))
    sign = torch.where((vt < 0) | ((vt == 0) & (vz < 0)), -1.0, 1.0).double()
    vr, vt, vz = vr * sign, vt * sign, vz * sign
    l = l.clamp_min(0.0)
    den = (l * l).sum(0)
    num = (l[0] - l[1]) ** 2 + (l[1] - l[2]) ** 2 + (l[2] - l[0]) ** 2
    fa = torch.where(den == 0, torch.zeros_like(den), (0.5 * num / torch.where(den == 0, 1.0, den)).sqrt())
    return v * sign, torch.rad2deg(torch.atan2(vz, vt)), torch.rad2deg(torch.asin(vr.clamp(-1, 1))), fa


def _positions(lo, n, i):
    return [(i % n[0] + lo[0]).double(), (i // n[0] % n[1] + lo[1]).double(), (i // (n[0] * n[1]) + lo[2]).double()]


def _decode64(S, ev, vec, lo, n, mask, cen, ax, out):
    """The outputs over the box (lo, n) from its tensors, or from its eigenvalues and vectors.  Without a
    mask the background's texture has no direction of its own, and only FA has a value."""
    total = n[0] * n[1] * n[2]
    directed = mask is not None and out != "u8q"
    res = {"fa": torch.empty(total, dtype=torch.float64, device="cuda")}
    if directed:
        res.update(vec=torch.empty((3, total), dtype=torch.float64, device="cuda"),
                   ha=torch.empty(total, dtype=torch.float64, device="cuda"),
                   ia=torch.empty(total, dtype=torch.float64, device="cuda"))
    step = 1 << 23
    for i in range(0, total, step):
        sl = slice(i, min(total, i + step))
        if S is not None:
            l, v = _eig64([p.reshape(-1)[sl] for p in S])
        else:
            l, v = ev.reshape(3, -1)[:, sl].double(), vec.reshape(3, -1)[:, sl].double()
        at = _positions(lo, n, torch.arange(sl.start, sl.stop, device="cuda"))
        v, ha, ia, fa = _angles64(v, l, at, cen, ax)
        if mask is not None:
            hole = mask.reshape(-1)[sl] == 0
            v, ha, ia, fa = (torch.where(hole, math.nan, t) for t in (v, ha, ia, fa))
        res["fa"][sl] = fa
        if directed:
            res["vec"][:, sl], res["ha"][sl], res["ia"][sl] = v, ha, ia
    shape = (n[2], n[1], n[0])
    got = {k: t.reshape(((3,) if k == "vec" else ()) + shape) for k, t in res.items()}
    return {k: got.get(k) for k in (("ha", "ia", "fa") if out == "u8q" else ("vec", "ha", "ia", "fa"))}


def _cell64(q, n):
    """(inside, lowest corner, offsets) of positions q (3, m) in a volume of size n."""
    top = torch.tensor([float(x - 1) for x in n], dtype=torch.float64, device=q.device)[:, None]
    ok = ((q >= 0) & (q <= top)).all(dim=0)
    i = torch.minimum(torch.floor(torch.where(ok, q, torch.zeros_like(q))), top - 1)
    return ok, i.long(), q - i


def _corners(i, t, n):
    for k in range(8):
        b = (k & 1, k >> 1 & 1, k >> 2 & 1)
        w = 1.0
        for a in range(3):
            w = w * (t[a] if b[a] else 1.0 - t[a])
        yield ((i[2] + b[2]) * n[1] + i[1] + b[1]) * n[0] + i[0] + b[0], w


def _direction64(vec, q, ref, n):
    ok, i, t = _cell64(q, n)
    s = torch.zeros_like(q)
    for j, w in _corners(i, t, n):
        u = vec[:, j].double()
        ok = ok & torch.isfinite(u).all(dim=0)
        u = torch.where((u * ref).sum(0) < 0, -u, u)
        s = s + w * u
    n2 = (s * s).sum(0)
    ok = ok & (n2 > 0)
    return ok, s / torch.where(ok, n2, torch.ones_like(n2)).sqrt()


def _track64(c, seed):
    v, fa, mask, seeds = _track_inputs(c, seed)
    n, steps = _dims(c), c["steps"]
    h, fa_min, turn = c["step"], float(torch.tensor(0.1, dtype=torch.float32)), math.cos(math.radians(60.0))
    vec, fa = v.reshape(3, -1), fa.reshape(-1)
    p = seeds.t().double().repeat_interleave(2, dim=1)
    m = p.shape[1]
    pts = torch.zeros((m, steps + 1, 3), dtype=torch.float64, device="cuda")
    ok, _, _ = _cell64(p, n)
    pts[ok, 0] = p.t()[ok]
    near = lambda q: (torch.floor(q[2] + 0.5).long() * n[1] + torch.floor(q[1] + 0.5).long()) * n[0] + \
        torch.floor(q[0] + 0.5).long()  # noqa: E731
    ref = vec[:, near(torch.where(ok, p, torch.zeros_like(p)))].double()
    ok = ok & torch.isfinite(ref).all(dim=0) & (ref != 0).any(dim=0)
    good, d = _direction64(vec, p, ref, n)
    d[:, 1::2] *= -1
    live = torch.nonzero(ok & good).flatten()
    p, d = p[:, live], d[:, live]
    for s in range(steps):
        k1_ok, k1 = _direction64(vec, p, d, n)
        k2_ok, k2 = _direction64(vec, p + 0.5 * h * k1, k1, n)
        k3_ok, k3 = _direction64(vec, p + 0.5 * h * k2, k2, n)
        k4_ok, k4 = _direction64(vec, p + h * k3, k3, n)
        t = k1 + 2 * k2 + 2 * k3 + k4
        dn = t / t.norm(dim=0)
        q = p + h / 6.0 * t
        ok = k1_ok & k2_ok & k3_ok & k4_ok & ((dn * d).sum(0) >= turn)
        inside, i, o = _cell64(q, n)
        ok = ok & inside
        if mask is not None:
            ok = ok & (mask.reshape(-1)[near(torch.where(ok, q, torch.zeros_like(q)))] != 0)
        ok = ok & (sum(w * fa[torch.where(ok, j, torch.zeros_like(j))].double() for j, w in _corners(i, o, n)) >=
                   fa_min)
        live, p, d = live[ok], q[:, ok], dn[:, ok]
        pts[live, s + 1] = p.t()
    return {"points": pts.reshape(-1, 2, steps + 1, 3), "count": None}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "profile":
        return None  # whole numbers
    if kind == "track":
        return _track64(c, seed)
    if kind == "eig":
        S = _eig_inputs(c, seed)
        ev = torch.empty((3, c["n"]), dtype=torch.float64, device="cuda")
        vec = torch.empty_like(ev)
        for i in range(0, c["n"], 1 << 23):
            l, v = _eig64(list(S[:, i:i + (1 << 23)].double()))
            big = v.gather(0, v.abs().argmax(dim=0, keepdim=True))
            ev[:, i:i + (1 << 23)], vec[:, i:i + (1 << 23)] = l, v * torch.where(big < 0, -1.0, 1.0)
        return {"evals": ev, "evec": vec}
    if kind == "angles":
        v, ev, mask = _angle_inputs(c, seed)
        dims = _dims(c)
        return _decode64(None, ev, v, (0, 0, 0), dims, mask, *_frame(dims), c["out"])
    if kind == "crops":
        got = []
        for w, vol in _crop_inputs(c, seed):
            dims = w.spec.shape[::-1]
            box = ((0, 0, 0), dims)
            S = _tensor64(vol, box, box, dims, w.sigma, w.rho)
            got.append(_decode64(S, None, None, *box, None, *synth.frame_of(w.spec), c["out"]))
        return got
    if kind == "box":
        spec, dims, ib, ob, vol, mask = _box_inputs(c, seed)
        S = _tensor64(vol, ib, ob, dims, c["sigma"], c["rho"])
        return _decode64(S, None, None, *ob, mask, *synth.frame_of(spec), c["out"])
    spec, dims = _wall(c, seed), _dims(c)
    vol, mask = _scan(spec, dims, (0, 0, 0), dims, c.get("masked", False))
    box = ((0, 0, 0), dims)
    S = _tensor64(vol, box, box, dims, c["sigma"], c["rho"])
    if kind == "tensor":
        return torch.stack(S)
    return _decode64(S, None, None, *box, mask, *synth.frame_of(spec), c["out"])
