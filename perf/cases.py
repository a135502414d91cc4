"""The work this library does for its users, as cases to time.

Each case is one call, or one chain of calls, of the public binding
(`paper_2101_03240_gb300.ibip`) on images of the two kinds the method is used
on: smoothed-noise blobs (the paper's 60 %-porosity artificial images) and
packs of overlapping solid spheres.  Sizes, smoothing lengths, radii and
porosities are those of the repository's workloads (48^3 blobs, 200^3 pack,
512^3 blobs, mixed batches of 32^3-160^3, mixed request streams from 64^3)
with odd and uneven edges between them.  Images are built on the GPU from the
seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_03240_gb300 import ibip, synth

VOXEL_M, SIGMA, THETA = 5e-6, 0.072, 180.0


# ------------------------------------------------------------------ images --

def _blobs(shape, sigma, porosity, g):
    """Uniform noise under a wrapping Gaussian filter; the lowest `porosity`
    of its values (taken as normal, which the filter makes them) are pore."""
    f = torch.fft.rfftn(torch.rand(shape, generator=g, device="cuda"))
    for ax, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device="cuda") if ax == 2 else torch.fft.fftfreq(n, device="cuda")
        w = torch.exp(-2.0 * (math.pi * sigma[ax] * k) ** 2)
        f *= w.view([-1 if a == ax else 1 for a in range(3)])
    f = torch.fft.irfftn(f, s=shape)
    z = math.sqrt(2.0) * torch.erfinv(torch.tensor(2.0 * porosity - 1.0, dtype=torch.float64)).item()
    return (f <= f.mean() + z * f.std()).to(torch.uint8)


def _pack(shape, radius, porosity, g):
    """Overlapping solid spheres, centres uniform over the box and its rim;
    their number is the one that leaves `porosity` on average."""
    r, size = float(radius), torch.tensor(shape, device="cuda", dtype=torch.float64)
    box = math.prod(n + 2 * r for n in shape)
    n = max(1, round(-math.log(porosity) * box / (4.0 / 3.0 * math.pi * r ** 3)))
    c = torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64) * (size + 2 * r) - r
    o = torch.arange(-int(radius) - 1, int(radius) + 2, device="cuda")
    o = torch.cartesian_prod(o, o, o)
    pore = torch.ones(shape, dtype=torch.uint8, device="cuda")
    for part in c.split(1024):
        v = part.round().long()[:, None, :] + o
        hit = ((v - part[:, None, :]) ** 2).sum(-1) <= r * r
        hit &= ((v >= 0) & (v < size.long())).all(-1)
        x, y, z = v[hit].unbind(-1)
        pore[x, y, z] = 0
    return pore


def _image(case, g):
    shape = (case["nx"], case["ny"], case["nz"])
    if case["image"] == "blobs":
        return _blobs(shape, (case["sx"], case["sy"], case["sz"]), case["porosity"], g)
    return _pack(shape, case["radius"], case["porosity"], g)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _edges(case):
    n = case["images"]
    e = [round(case["lo"] * (case["hi"] / case["lo"]) ** ((i + 0.5) / n)) for i in range(n)]
    return e[::3] + e[1::3] + e[2::3]


def _mixed(case, g):
    """Uneven cubes, edges spread evenly over the logarithm of [lo, hi] in
    mixed order, blobs and packs in turn."""
    out = []
    for i, e in enumerate(_edges(case)):
        u = torch.rand(2, generator=g, device="cuda").tolist()
        if i % 2 == 0:
            s = 2.0 + 4.0 * u[0]
            out.append(_blobs((e, e, e), (s, s, s), 0.5 + 0.2 * u[1], g))
        else:
            out.append(_pack((e, e, e), 4 + int(7 * u[0]), 0.35 + 0.15 * u[1], g))
    return out


# ------------------------------------------------------------------- cases --

def _blob_case(name, call, shape, sigma, porosity, **more):
    return dict(name=name, call=call, image="blobs", nx=shape[0], ny=shape[1], nz=shape[2], sx=sigma[0], sy=sigma[1],
                sz=sigma[2], porosity=porosity, inlet=0, outlet=1, **more)


def _pack_case(name, call, shape, radius, porosity, **more):
    return dict(name=name, call=call, image="pack", nx=shape[0], ny=shape[1], nz=shape[2], radius=radius,
                porosity=porosity, inlet=0, outlet=1, **more)


def listed():
    iso3, aniso = (3.0, 3.0, 3.0), (4.0, 8.0, 4.0)
    return [
        # one distance map of a small sample: the shortest call, all latency
        _blob_case("edt_small", "edt", (48, 48, 48), iso3, 0.65),
        # the distance map of a full scan
        _blob_case("edt_large", "edt", (512, 512, 512), aniso, 0.60),
        # a small sample invaded straight from its image
        _blob_case("invade_small", "invade", (48, 48, 48), iso3, 0.65, dt2=False),
        # a laboratory-size pack, the distance map inside the call
        _pack_case("invade_pack", "invade", (200, 200, 200), 8, 0.40, dt2=False),
        # a full scan whose distance map the user already has
        _blob_case("invade_large", "invade", (512, 512, 512), aniso, 0.60, dt2=True),
        # the invasion as the paper prints it, all tied maxima at once
        _pack_case("literal_pack", "literal", (150, 161, 173), 8, 0.40),
        # the defending phase of a finished invasion, uneven edges
        _blob_case("trapping", "trapping", (301, 323, 347), aniso, 0.60),
        # pressure-based drainage at forty radii, from another face
        _blob_case("opening", "opening", (255, 260, 277), aniso, 0.60, levels=40),
        # saturation and pressure curve with the saturation image of a long
        # sequence
        dict(name="curve", call="curve", nx=400, ny=411, nz=423, steps=2500000, porosity=0.60),
        # a study of many small samples in one call
        dict(name="batch", call="batch", images=96, lo=32, hi=160),
        # the same through the request loop, which owns its memory
        dict(name="serve", call="serve", images=20, lo=64, hi=200, slots=16),
        # everything a user reports for one sample, call after call
        _blob_case("path", "path", (190, 200, 213), aniso, 0.60, levels=40),
    ]


def _log_edge(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["edt", "edt", "invade", "invade", "invade", "literal", "trapping", "opening", "curve", "batch",
                       "serve", "path"])
    if call in ("batch", "serve"):
        lo = _log_edge(rng, 24, 64)
        c = dict(call=call, images=rng.randint(24, 96) if call == "batch" else rng.randint(2, 20), lo=lo,
                 hi=_log_edge(rng, lo + 8, 160 if call == "batch" else 200))
        if call == "serve":
            c["slots"] = rng.choice([4, 8, 16])
        return c
    top = {"edt": 512, "invade": 400, "literal": 170, "trapping": 330, "opening": 260, "curve": 420, "path": 210}[call]
    least = 120 if call in ("trapping", "path") else 32
    e = _log_edge(rng, least, top)
    shape = [max(8, min(top, int(round(e * rng.uniform(0.7, 1.3))))) for _ in range(3)]
    if call == "curve":
        return dict(call=call, nx=shape[0], ny=shape[1], nz=shape[2], porosity=rng.uniform(0.35, 0.7),
                    steps=max(1, int(math.prod(shape) * rng.uniform(0.002, 0.06))))
    c = dict(call=call, nx=shape[0], ny=shape[1], nz=shape[2], inlet=rng.randint(0, 5))
    c["outlet"] = c["inlet"] ^ 1
    if rng.random() < 0.5:
        c.update(image="blobs", porosity=rng.uniform(0.5, 0.7), sx=rng.uniform(2.0, 6.0), sy=rng.uniform(2.0, 8.0),
                 sz=rng.uniform(2.0, 6.0))
    else:
        c.update(image="pack", porosity=rng.uniform(0.35, 0.5), radius=rng.randint(4, 10))
    if call == "invade":
        c["dt2"] = rng.random() < 0.5
    if call in ("opening", "path"):
        c["levels"] = rng.randint(10, 60)
    return c


def _sequence(case, g):
    """A sequence image as long invasions leave it: steps in the order of a
    smooth field (a step's voxels lie together), a tenth of the pore left
    uninvaded in clusters, most steps a few voxels and some very large."""
    shape, K = (case["nx"], case["ny"], case["nz"]), case["steps"]
    img = _blobs(shape, (4.0, 8.0, 4.0), case["porosity"], g)
    f = torch.fft.rfftn(torch.rand(shape, generator=g, device="cuda"))
    for ax, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device="cuda") if ax == 2 else torch.fft.fftfreq(n, device="cuda")
        f *= torch.exp(-2.0 * (math.pi * 4.0 * k) ** 2).view([-1 if a == ax else 1 for a in range(3)])
    f = torch.fft.irfftn(f, s=shape)
    f = (f - f.mean()) / f.std()
    u = 0.5 * (1.0 + torch.erf(f / math.sqrt(2.0)))
    step = (u / 0.9) ** 2 * K        # early steps are the large ones
    step += torch.rand(shape, generator=g, device="cuda") * 2.0
    seq = step.to(torch.int32).clamp_(1, K)
    seq[u > 0.9] = -1
    seq[img == 0] = 0
    r2 = (1.0 + 200.0 * torch.rand(K, generator=g, device="cuda") ** 12).to(torch.int32)
    return seq, r2


def prepare(case, seed):
    g, call = _generator(seed), case["call"]
    ctx = ibip.context()
    s = dict(case=case, ctx=ctx)
    if call == "curve":
        s["seq"], s["r2"] = _sequence(case, g)
        return s
    if call in ("batch", "serve"):
        s["images"] = _mixed(case, g)
        if call == "serve":
            need = sum(sorted((ibip.job_footprint(im.shape) for im in s["images"]), reverse=True)[:case["slots"]])
            s["server"] = ibip.Server(ctx, need, case["slots"])
        return s
    s["image"] = _image(case, g)
    if call == "trapping":
        s["seq"] = ctx.invade(s["image"], inlet=case["inlet"], centres=False)[0].clone()
    if call in ("invade", "path"):   # the step arrays a program keeps from one image to the next
        for k in ("r2", "centre"):
            s[k] = torch.zeros(s["image"].numel(), dtype=torch.int32, device="cuda")
    if call == "opening" or case.get("dt2"):
        s["dt2"] = ctx.edt(s["image"])
    if call == "opening":
        s["radii"] = synth.mio_levels(int(s["dt2"].max()), case["levels"])
    return s


def _whole(t, n):
    """A step array with zeros after its last step, so that its length does
    not depend on the image."""
    return torch.nn.functional.pad(t, (0, n - t.numel()))


def _counts(n, *lists):
    """Per-level counts, zeros after the last level."""
    return np.array([list(c) + [0] * (n - len(c)) for c in lists], np.int64)


def _many(out, voxels):
    """The results of many images, each kind end to end."""
    whole = [torch.cat([r[k].flatten() for r in out]) for k in ("seq", "trapped", "seq_out")]
    steps = [_whole(torch.cat([r[k] for r in out]), voxels) for k in ("step_r2", "step_centre", "S", "Pc")]
    return whole + steps + [np.array([[r["K"], r["status"]] for r in out], np.int64)]


def run(s):
    case, ctx = s["case"], s["ctx"]
    call = case["call"]
    if call == "edt":
        return ctx.edt(s["image"])
    if call == "invade":
        seq, _, _, K, status = ctx.invade(s["image"], s.get("dt2"), inlet=case["inlet"], step_r2=s["r2"],
                                          step_centre=s["centre"])
        return [seq, s["r2"], s["centre"], K, status]
    if call == "literal":
        seq, cstep, r2, count, K, status = ctx.invade_literal(s["image"], inlet=case["inlet"])
        return [seq, cstep, _whole(r2, seq.numel()), _whole(count, seq.numel()), K, status]
    if call == "trapping":
        return list(ctx.trapping(s["seq"], case["outlet"]))
    if call == "opening":
        level, counts = ctx.morph_drainage(s["image"], s["dt2"], s["radii"], inlet=case["inlet"])
        return [level, _counts(case["levels"], counts)]
    if call == "curve":
        return list(ctx.pc_curve(s["seq"], s["r2"], VOXEL_M, SIGMA, THETA, sat_image=True))
    if call == "batch":
        return _many(ctx.invade_batched(s["images"], 0, 1, voxel_m=VOXEL_M, sigma=SIGMA, theta_deg=THETA),
                     _voxels(case))
    if call == "serve":
        srv = s["server"]
        tickets = [srv.submit(im, 0, 1, voxel_m=VOXEL_M, sigma=SIGMA, theta_deg=THETA) for im in s["images"]]
        return _many([srv.wait(t) for t in tickets], _voxels(case))
    image, n = s["image"], s["image"].numel()
    dt2 = ctx.edt(image)
    seq, r2, centre, K, status = ctx.invade(image, dt2, inlet=case["inlet"], step_r2=s["r2"], step_centre=s["centre"])
    trapped, seq_out = ctx.trapping(seq, case["outlet"])
    S, pc, _ = ctx.pc_curve(seq_out, r2, VOXEL_M, SIGMA, THETA)
    radii = synth.mio_levels(int(dt2.max()), case["levels"])
    level, counts = ctx.morph_drainage(image, dt2, radii, inlet=case["inlet"])
    at, diff, found = ctx.equal_saturation(seq, level, K, len(radii))
    env_k, env_n = ctx.pc_envelope(seq, r2, radii)
    size = ctx.size_image(seq, r2)
    return [dt2, seq, s["r2"], s["centre"], K, status, trapped, seq_out, _whole(S, n), _whole(pc, n), level, size,
            _counts(case["levels"], counts, at, diff, found, env_k, env_n)]


def _voxels(case):
    if "images" in case:
        return sum(e ** 3 for e in _edges(case))
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes: inputs read once and outputs written once per voxel; step
    arrays (about one step per 25 voxels) 4 bytes an entry.  Operations: the
    few integer operations a voxel cannot do without."""
    N, call = _voxels(case), case["call"]
    per = {"edt": 1 + 4,                       # image in, dt2 out
           "invade": (4 if case.get("dt2") else 1) + 4 + 8 / 25,
           "literal": 1 + 4 + 4,               # image in, sequence and insertion steps out
           "trapping": 4 + 1 + 4,              # sequence in, mask and corrected sequence out
           "opening": 1 + 4 + 4,               # image and dt2 in, level out
           "curve": 4 + 4,                     # sequence in, saturation image out
           "batch": 1 + 4 + 1 + 4 + 16 / 25,   # image in, sequence, mask, corrected sequence, steps out
           "serve": 1 + 4 + 1 + 4 + 16 / 25,
           "path": 1 + 4 + 4 + 1 + 4 + 4 + 4 + 16 / 25}[call]
    extra = 12 * case["steps"] if call == "curve" else 0
    return {"bytes": int(N * per) + extra, "flops": 3 * N}


def exact(case, seed):
    """The curve in 64 bits; every other output is a whole number, or takes
    an invasion to compute."""
    if case["call"] != "curve":
        return None
    seq, r2 = _sequence(case, _generator(seed))
    seq, K = seq.flatten().long(), case["steps"]
    n = torch.bincount(seq.clamp(min=0), minlength=K + 1)[1:]
    S = n.cumsum(0).double() / (seq != 0).sum().double()
    pc = -2.0 * SIGMA * math.cos(THETA * math.pi / 180.0) / (r2.double().sqrt() * VOXEL_M)
    image = torch.full(seq.shape, math.inf, dtype=torch.float64, device=seq.device)
    on = seq >= 1
    image[on] = S[seq[on] - 1]
    return [S, pc, image.view(case["nx"], case["ny"], case["nz"])]
