"""The work a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values.  ``listed()`` names twelve of them, ``draw``
makes more over the same ranges, ``prepare`` builds what a program holds before
the call (scene handle, rays, output buffers), ``run`` is one pass through the
public entry points, ``work`` what that pass cannot do without and ``exact``
its floating results in binary64, where plain torch can afford them.

Every float4 hit is returned as two views: t, u, v and the triangle id's bits.
"""
import math
from functools import lru_cache

import numpy as np
import torch

from paper_2506_11273_gb300 import rr
from paper_2506_11273_gb300 import workloads as W

# Scenes by name: the tiny box soup, and terrains with boxes from 50 thousand
# triangles to the path tracer's 1,168,576.
TERRAINS = {
    "terrain50k": (107, 214, 334),
    "terrain250k": (240, 480, 1646),
    "terrain1M": (512, 1024, 10000),
}
SCENE_TRIS = {"soup": 4108, **{k: 2 * x * z + 12 * b for k, (x, z, b) in TERRAINS.items()}}
LAYOUTS = {"aila": rr.RR_KEY_AILA, "two_point": rr.RR_KEY_TWO_POINT, "costa": rr.RR_KEY_COSTA}
ESTIMATES = {"fixed": rr.RR_T_FIXED, "adaptive": rr.RR_T_ADAPTIVE}
EYE = (0.5, 0.6, 0.1)
LOOK_AT = (0.5, 0.2, 1.2)


def listed():
    return [
        # One bounce of the smallest served request (4,097 rays) on the tiny scene: launches and latency.
        dict(name="bounce_4k", op="bounce", scene="soup", n=4097, order="random", layout="two_point",
             estimate="fixed", bits=32),
        # One bounce of the tiny scene's 65,536 rays with the full 64-bit adaptive key.
        dict(name="bounce_64k", op="bounce", scene="soup", n=65536, order="random", layout="two_point",
             estimate="adaptive", bits=64),
        # The path tracer's third bounce: 1,196,335 secondary rays in pixel order, 64-bit adaptive key.
        dict(name="bounce_path", op="bounce", scene="terrain1M", n=1196335, order="pixel", layout="two_point",
             estimate="adaptive", bits=64),
        # The same bounce from page-locked host buffers and back, as an application outside the GPU calls it.
        dict(name="bounce_host", op="host", scene="terrain1M", n=1196335, order="pixel", layout="two_point",
             estimate="fixed", bits=32),
        # The cheapest reordering: a 16-bit direction-first key, its sort, and the trace through the
        # permutation; the path tracer's fourth bounce (689,149 rays).
        dict(name="indirect", op="indirect", scene="terrain1M", n=689149, order="pixel", layout="costa",
             estimate="fixed", bits=16),
        # Camera rays of a 1920x1080 frame, closest hit, natural order.
        dict(name="trace_camera", op="trace", scene="terrain1M", n=2073600, order="camera"),
        # A 3840x2160 frame's worth of secondary rays in random order, closest hit.
        dict(name="trace_large", op="trace", scene="terrain1M", n=8294400, order="random"),
        # Shadow rays of one bounce towards an area light, any hit.
        dict(name="trace_shadow", op="any", scene="terrain1M", n=986588, order="random"),
        # Keys and their sort for the second bounce, 32-bit keys.
        dict(name="key_sort_32", op="key_sort", scene="terrain1M", n=2071587, order="pixel", layout="two_point",
             estimate="fixed", bits=32),
        # Keys and their sort for the largest wavefront, 64-bit keys.
        dict(name="key_sort_64", op="key_sort", scene="terrain1M", n=8294400, order="random", layout="aila",
             estimate="fixed", bits=64),
        # The reorder of the largest wavefront with its payload.
        dict(name="reorder", op="permute", scene="terrain1M", n=8294400, order="random", layout="two_point",
             estimate="fixed", bits=32),
        # Twelve uneven wavefronts over three resident scenes as one batch, 24-bit keys.
        dict(name="batch", op="batch", scene="terrain250k", n=3700001, order="random", layout="two_point",
             estimate="fixed", bits=24, fronts=12),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["bounce", "bounce", "host", "indirect", "trace", "any", "key_sort", "permute", "batch"])
    most = {"bounce": 2073600, "host": 2073600, "indirect": 2073600, "any": 2073600, "batch": 3700001}.get(op, 8294400)
    c = dict(op=op, scene=rng.choice(["soup", "terrain50k", "terrain250k", "terrain1M"]), n=size(4097, most),
             order=rng.choice(["random", "pixel"]))
    if op == "trace" and rng.random() < 0.5:
        c["order"] = "camera"
    if op not in ("trace", "any"):
        c["layout"] = rng.choice(["aila", "two_point", "two_point", "costa"])
        c["estimate"] = rng.choice(["fixed", "adaptive"]) if c["layout"] == "two_point" and op in (
            "bounce", "host") else "fixed"
        c["bits"] = rng.choice([16, 24, 32] if op in ("indirect", "batch") else [24, 32, 48, 64])
    if op == "batch":
        c["fronts"] = rng.randint(2, 32)
    return c


# ------------------------------------------------------------------ scenes (resident, as a program keeps them)

@lru_cache(maxsize=None)
def _scene(name):
    if name == "soup":
        tris = W.scene_box_soup(seed=1)
    else:
        x, z, b = TERRAINS[name]
        tris = W.scene_terrain(seed=2, cells_x=x, cells_z=z, n_boxes=b)
    lo, hi = W.scene_aabb(tris)
    t = torch.from_numpy(tris).cuda().double()
    v0, e1, e2 = t[:, 0:3], t[:, 3:6] - t[:, 0:3], t[:, 6:9] - t[:, 0:3]
    c = torch.linalg.cross(e1, e2)
    area = c.norm(dim=1)
    return dict(tris=tris, bvh=rr.BVH(tris), lo=lo, hi=hi, v0=v0, e1=e1, e2=e2,
                normal=c / area.clamp_min(1e-30)[:, None], cdf=torch.cumsum(area, 0))


# ------------------------------------------------------------------ rays

def _unit(v):
    return v / v.norm(dim=1, keepdim=True).clamp_min(1e-30)


def _about(axis, cos_a, phi):
    """Directions at angle acos(cos_a) from the unit axes, turned by phi."""
    other = torch.where(axis[:, :1].abs() > 0.9, torch.tensor([[0.0, 1.0, 0.0]], device=axis.device, dtype=axis.dtype),
                        torch.tensor([[1.0, 0.0, 0.0]], device=axis.device, dtype=axis.dtype))
    t = _unit(torch.linalg.cross(axis, other))
    b = torch.linalg.cross(axis, t)
    sin_a = (1.0 - cos_a * cos_a).clamp_min(0.0).sqrt()
    return _unit(axis * cos_a[:, None] + t * (sin_a * phi.cos())[:, None] + b * (sin_a * phi.sin())[:, None])


def _camera_frame(dtype):
    eye = torch.tensor(EYE, device="cuda", dtype=dtype)
    fwd = _unit((torch.tensor(LOOK_AT, device="cuda", dtype=dtype) - eye)[None])[0]
    right = _unit(torch.linalg.cross(fwd, torch.tensor([0.0, 1.0, 0.0], device="cuda", dtype=dtype))[None])[0]
    return eye, fwd, right, torch.linalg.cross(right, fwd), math.tan(math.radians(30.0))


def _pack(o, d, tmin, tmax):
    n = o.shape[0]
    om, dm = torch.empty(n, 4, device="cuda"), torch.empty(n, 4, device="cuda")
    om[:, :3], om[:, 3] = o.float(), tmin
    dm[:, :3], dm[:, 3] = d.float(), tmax
    return om, dm


def _surface(s, n, g):
    """Points uniform by area, their triangles, and the direction from the eye."""
    r = torch.rand(3, n, generator=g, device="cuda", dtype=torch.float64)
    ids = torch.searchsorted(s["cdf"], r[0] * s["cdf"][-1]).clamp_max(s["cdf"].shape[0] - 1)
    b = r[1].sqrt()
    p = s["v0"][ids] + s["e1"][ids] * (b * (1 - r[2]))[:, None] + s["e2"][ids] * (b * r[2])[:, None]
    incoming = _unit(p - torch.tensor(EYE, device="cuda", dtype=torch.float64))
    nrm = s["normal"][ids]
    nrm = torch.where((nrm * incoming).sum(1, keepdim=True) > 0, -nrm, nrm)
    return p, ids, nrm, incoming


def _pixel_order(p, width=1920):
    """The order in which a compacted wavefront holds rays that leave the points p: by screen row and column."""
    eye, fwd, right, up, th = _camera_frame(torch.float64)
    v = p - eye
    z = (v * fwd).sum(1).abs().clamp_min(1e-3)
    height = width * 9 // 16
    x = ((v * right).sum(1) / z / (th * 16 / 9) * 0.5 + 0.5).clamp(0, 1) * (width - 1)
    y = (0.5 - (v * up).sum(1) / z / th * 0.5).clamp(0, 1) * (height - 1)
    return torch.sort(y.long() * width + x.long(), stable=True)[1]


def _secondary(s, n, order, g):
    """Rays that scatter off the scene: 70% diffuse, 30% Phong lobes about the mirror direction."""
    p, ids, nrm, incoming = _surface(s, n, g)
    r = torch.rand(2, n, generator=g, device="cuda", dtype=torch.float64)
    glossy = (ids * 2654435761 % 1000) < 300
    mirror = _unit(incoming - 2 * (incoming * nrm).sum(1, keepdim=True) * nrm)
    axis = torch.where(glossy[:, None], mirror, nrm)
    cos_a = torch.where(glossy, r[1] ** (1.0 / 101.0), r[1].sqrt())
    d = _about(axis, cos_a, 2 * math.pi * r[0])
    d = torch.where((d * nrm).sum(1, keepdim=True) <= 0, mirror, d)
    if order == "pixel":
        at = _pixel_order(p)
        p, d = p[at], d[at]
    return _pack(p, d, 1e-4, math.inf)


def _camera(n, g):
    """The first n pixels of a 16:9 frame with at least n pixels, one jittered ray each."""
    eye, fwd, right, up, th = _camera_frame(torch.float64)
    width = math.ceil(math.sqrt(n * 16 / 9))
    height = math.ceil(n / width)
    k = torch.arange(n, device="cuda")
    j = torch.rand(2, n, generator=g, device="cuda", dtype=torch.float64)
    x = (2 * (k % width + j[0]) / width - 1) * th * width / height
    y = (1 - 2 * (k // width + j[1]) / height) * th
    d = _unit(fwd + x[:, None] * right + y[:, None] * up)
    return _pack(eye.expand(n, 3), d, 0.0, math.inf)


def _shadow(s, n, order, g):
    """Segments from surface points to a square light above the scene, 5% of its largest extent wide."""
    p, _, _, _ = _surface(s, n, g)
    if order == "pixel":
        p = p[_pixel_order(p)]
    lo, hi = s["lo"].astype(np.float64), s["hi"].astype(np.float64)
    e = float((hi - lo).max())
    c = torch.tensor([(lo[0] + hi[0]) / 2, hi[1] + 0.05 * e, (lo[2] + hi[2]) / 2], device="cuda", dtype=torch.float64)
    j = (torch.rand(2, n, generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.05 * e
    light = c + torch.stack([j[0], torch.zeros_like(j[0]), j[1]], 1)
    return _pack(p, light - p, 1e-4, 1 - 1e-4)


def _rays(case, s, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    if case["op"] == "any":
        return _shadow(s, case["n"], case["order"], g)
    if case["order"] == "camera":
        return _camera(case["n"], g)
    return _secondary(s, case["n"], case["order"], g)


def _front_sizes(case):
    """Uneven wavefronts: weights from 1 to 20 in a fixed scatter, summing to n."""
    w = np.array([20.0 ** ((k * 7 % case["fronts"]) / max(1, case["fronts"] - 1)) for k in range(case["fronts"])])
    sizes = np.floor(case["n"] * w / w.sum()).astype(int)
    sizes[0] += case["n"] - sizes.sum()
    return [int(x) for x in sizes]


# ------------------------------------------------------------------ the calls

def _params(case, s, table=None):
    return rr.key_params(LAYOUTS[case["layout"]], case["bits"], s["lo"], s["hi"],
                         t_source=ESTIMATES[case["estimate"]], table=table)


def _hits(n):
    h = torch.empty(n, 4, device="cuda")
    return h, (h[:, :3], h.view(torch.int32)[:, 3])


def prepare(case, seed):
    op, n = case["op"], case["n"]
    s = _scene(case["scene"])
    st = dict(op=op, s=s, n=n)
    if op == "batch":
        g = torch.Generator("cuda").manual_seed(seed)
        scenes = [_scene(x) for x in (case["scene"], "soup", "terrain50k")]
        sizes = _front_sizes(case)
        parts = [_secondary(scenes[k % 3], m, case["order"], g) for k, m in enumerate(sizes)]
        st["o"], st["d"] = (torch.cat([p[i] for p in parts]) for i in (0, 1))
        st["batch"] = rr.Batch([(scenes[k % 3]["bvh"], None, scenes[k % 3]["lo"], scenes[k % 3]["hi"], m)
                                for k, m in enumerate(sizes)], LAYOUTS[case["layout"]])
        st["cfg"] = rr.Batch.config(case["bits"], 8, 128)
        st["perm"] = torch.empty(n, dtype=torch.int32, device="cuda")
        st["hits"], st["out"] = _hits(n)
        return st
    st["o"], st["d"] = _rays(case, s, seed)
    if op in ("trace", "any"):
        st["hits"], st["out"] = _hits(n)
        return st
    table = rr.LengthTable(s["lo"], s["hi"]) if case["estimate"] == "adaptive" else None
    st["params"] = _params(case, s, table)
    if op in ("bounce", "host"):
        st["pay"] = torch.arange(n, dtype=torch.int32, device="cuda")
        st["pipe"] = rr.Pipeline(s["bvh"], n, st["params"])
        st["hits"], st["out"] = _hits(n)
        st["pay_out"] = torch.empty_like(st["pay"])
        if op == "host":
            for k in ("o", "d", "pay", "hits", "pay_out"):
                st[k] = st[k].cpu().pin_memory()
            st["out"] = (st["hits"][:, :3], st["hits"].view(torch.int32)[:, 3])
        return st
    st["keys"] = torch.empty(n, dtype=rr.key_dtype(case["bits"]), device="cuda")
    st["perm"] = torch.empty(n, dtype=torch.int32, device="cuda")
    st["ws"] = rr.sort_workspace(n, case["bits"])
    if op == "indirect":
        st["hits"], st["out"] = _hits(n)
    elif op == "permute":
        rr.rr_key_sort(st["o"], st["d"], st["params"], st["keys"], st["perm"], 8, st["ws"])
        st["pay"] = torch.arange(n, dtype=torch.int32, device="cuda")
        st["o2"], st["d2"], st["pay2"] = (torch.empty_like(st[k]) for k in ("o", "d", "pay"))
        del st["keys"], st["ws"]
    return st


def run(st):
    op = st["op"]
    if op == "bounce":
        st["pipe"].run(st["o"], st["d"], st["pay"], st["hits"], st["pay_out"])
        return dict(hit=st["out"][0], tri=st["out"][1], payload=st["pay_out"])
    if op == "host":
        st["pipe"].run_host(st["o"], st["d"], st["pay"], st["hits"], st["pay_out"])
        return dict(hit=st["out"][0], tri=st["out"][1], payload=st["pay_out"])
    if op == "indirect":
        rr.rr_key_sort(st["o"], st["d"], st["params"], st["keys"], st["perm"], 8, st["ws"])
        rr.rr_trace_ex(st["s"]["bvh"], st["o"], st["d"], st["hits"], order=st["perm"])
        return dict(hit=st["out"][0], tri=st["out"][1], perm=st["perm"])
    if op == "trace":
        rr.rr_trace(st["s"]["bvh"], st["o"], st["d"], st["hits"])
        return dict(hit=st["out"][0], tri=st["out"][1])
    if op == "any":
        rr.rr_trace_ex(st["s"]["bvh"], st["o"], st["d"], st["hits"], flags=rr.RR_TRACE_ANY_HIT)
        return dict(hit=st["out"][0], tri=st["out"][1])
    if op == "key_sort":
        rr.rr_key_sort(st["o"], st["d"], st["params"], st["keys"], st["perm"], 8, st["ws"])
        return dict(keys=st["keys"], perm=st["perm"])
    if op == "permute":
        rr.rr_permute(st["o"], st["d"], st["pay"], st["perm"], st["o2"], st["d2"], st["pay2"])
        return dict(o=st["o2"], d=st["d2"], payload=st["pay2"])
    st["batch"].run(st["o"], st["d"], st["hits"], st["cfg"], st["perm"])
    return dict(hit=st["out"][0], tri=st["out"][1], perm=st["perm"])


def work(case):
    """Bytes: rays, payloads, keys and permutation in and out once.  Operations of a trace: the boxes of
    one 8-wide node per level and one triangle per ray; of a key, about 40."""
    op, n = case["op"], case["n"]
    kb = 8 if case.get("bits", 0) > 32 else 4
    per_trace = 30 + 8 * 12 * math.ceil(math.log(SCENE_TRIS[case["scene"]], 8))
    per_ray = {"bounce": 32 + 4 + 16 + 4, "host": 32 + 4 + 16 + 4, "indirect": 32 + 16 + 4 + kb, "trace": 32 + 16,
               "any": 32 + 16, "key_sort": 32 + kb + 4, "permute": 4 + 36 + 36, "batch": 32 + 16 + 4}[op]
    flops = (0 if op in ("key_sort", "permute") else per_trace) + (0 if op in ("trace", "any", "permute") else 40)
    return {"bytes": per_ray * n, "flops": flops * n}


# ------------------------------------------------------------------ binary64 results

def _exact_hits(tris, o, d):
    """Closest hits of every ray over all triangles, two-sided Moller-Trumbore in binary64; ties to the lowest id."""
    t = torch.from_numpy(tris).cuda().double()
    v0, e1, e2 = t[:, 0:3], t[:, 3:6] - t[:, 0:3], t[:, 6:9] - t[:, 0:3]
    out = torch.zeros(o.shape[0], 3, dtype=torch.float64, device="cuda")
    step = max(1, 40_000_000 // max(1, t.shape[0]))
    for a in range(0, o.shape[0], step):
        oo, dd = o[a:a + step].double(), d[a:a + step].double()
        org, dr = oo[:, None, :3], dd[:, None, :3].expand(-1, t.shape[0], -1)
        pv = torch.linalg.cross(dr, e2[None].expand_as(dr))
        det = (pv * e1).sum(2)
        tv = org - v0
        qv = torch.linalg.cross(tv, e1[None].expand_as(tv))
        u, v, tt = (tv * pv).sum(2) / det, (dr * qv).sum(2) / det, (e2 * qv).sum(2) / det
        ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (tt > oo[:, 3:]) & (tt < dd[:, 3:])
        best, at = torch.where(ok, tt, math.inf).min(1)
        hit = torch.isfinite(best)[:, None]
        uv = torch.stack([u.gather(1, at[:, None])[:, 0], v.gather(1, at[:, None])[:, 0]], 1)
        out[a:a + step, 0] = best
        out[a:a + step, 1:] = torch.where(hit, uv, 0.0)
    return out


def _two_point_order(o, d, bits, lo, hi):
    """The stable order of the Two Point keys with the estimate 0.25 E (also the first pass of an
    adaptive table), in binary32 as the key is defined."""
    f32 = np.float32
    o, d = o.cpu().numpy(), d.cpu().numpy()
    ext = hi - lo
    ln = np.sqrt((d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2], dtype=f32)
    dh = np.where(ln[:, None] > 0, d[:, :3] / np.where(ln > 0, ln, f32(1))[:, None], f32(0)).astype(f32)
    p = o[:, :3] + dh * (f32(0.25) * ext.max())

    def cells(x):
        x = (x - lo) * (f32(1) / ext)
        return np.where(x >= 1, 2.0 ** 32 - 1, np.floor(np.clip(x, f32(0), f32(1)).astype(np.float64) * 2.0 ** 32)).astype(np.uint64)

    c = np.concatenate([cells(o[:, :3]), cells(p)], 1)
    key = np.zeros(o.shape[0], np.uint64)
    for b in range(bits):
        key = (key << np.uint64(1)) | ((c[:, b % 6] >> np.uint64(31 - b // 6)) & np.uint64(1))
    return torch.from_numpy(np.argsort(key, kind="stable")).cuda()


def exact(case, seed):
    op = case["op"]
    if op == "key_sort":
        return None
    if op == "permute":
        st = prepare(case, seed)
        at = st["perm"].long()
        return dict(o=st["o"].double()[at], d=st["d"].double()[at], payload=None)
    if op not in ("bounce", "host", "trace") or case["n"] * SCENE_TRIS[case["scene"]] > 2_000_000_000:
        return None  # an any-hit ray may report any triangle; larger scenes take too long without a hierarchy
    if op != "trace" and case["layout"] != "two_point":
        return None
    s = _scene(case["scene"])
    o, d = _rays(case, s, seed)
    if op == "trace":
        return dict(hit=_exact_hits(s["tris"], o, d), tri=None)
    at = _two_point_order(o, d, case["bits"], s["lo"], s["hi"])
    return dict(hit=_exact_hits(s["tris"], o[at], d[at]), tri=None, payload=None)
