"""The calls that a user of this library makes in earnest, with inputs, work and tolerances.

Five kinds, each through the public entry points of paper_2305_16652_gb300.hcc:

bounce  hcc_run on device buffers: encode, sort, trace of one wavefront (closest hit, or any hit for
        shadow rays), for each method and node layout; method "nosort" is the plain trace
order   hcc_encode + hcc_sort: keys and permutation for a program that has its own tracer
split   the stages called one by one: encode, sort, gather into 32-byte records, trace with scatter
batch   two bounces of several scenes' wavefronts: hcc_batch_run, hcc_batch_spawn, hcc_batch_run
host    hcc_run_host: rays and hits in page-locked host memory

Scenes are the furnished rooms and the random-triangle cloud of paper_2305_16652_gb300.gen; they belong
to the case (resident geometry, its BVH handle and cut are kept by the program) and are built once per
process.  The rays belong to the seed: samples scattered over the camera's visible points, eight to a
pixel, each sending one cosine-weighted diffuse ray, or two shadow rays toward the ceiling lights.

Sizes: 1,024 rays to the 1920x1080x8 wavefront (16,588,800), scenes of 10,000 to 1,000,000 triangles,
keys of 16 to 64 bits.
"""
import math

import numpy as np
import torch

from paper_2305_16652_gb300 import gen, hcc

DEV = "cuda:0"
FULL_N = 1920 * 1080 * 8


def listed():
    return [
        # the smallest wavefront in use (the 64x64 image over 10,000 triangles): launches and latency
        dict(name="bounce_cloud_4k", kind="bounce", scene="cloud", tris=10_000, n=4096, method="hcc",
             layout="quantised", bits=32, any_hit=False, records=False),
        # the smallest serving request: a 65,536-ray window over a mid-sized scene
        dict(name="bounce_room_64k", kind="bounce", scene="room", tris=200_000, n=65_536, method="hcc",
             layout="exact", bits=32, any_hit=False, records=False),
        # the mean serving request, an odd number of rays, on the full room
        dict(name="bounce_room_958k", kind="bounce", scene="room", tris=1_000_000, n=957_759, method="hcc",
             layout="exact", bits=32, any_hit=False, records=False),
        # the headline wavefront: 1080p, 8 samples, 1M triangles, 32 cut nodes
        dict(name="bounce_1080p", kind="bounce", scene="room", tris=1_000_000, n=FULL_N, method="hcc",
             layout="exact", bits=32, any_hit=False, records=False),
        # the baseline every method is compared with: no sort, 4-ary nodes, one sample per 1080p pixel
        dict(name="unsorted_2m", kind="bounce", scene="room", tris=400_000, n=2_073_600, method="nosort",
             layout="wide", bits=32, any_hit=False, records=False),
        # shadow rays (two per sample), any hit, in key order
        dict(name="shadow_4m", kind="bounce", scene="room", tris=1_000_000, n=4_147_200, method="hcc",
             layout="exact", bits=32, any_hit=True, records=False),
        # two-level 16-bit keys on 32-byte ray records, a ragged count
        dict(name="mlhcc16_3m", kind="bounce", scene="room", tris=400_000, n=3_000_001, method="mlhcc",
             layout="exact", bits=16, any_hit=False, records=True),
        # long keys for a program's own tracer: 48-bit TwoPoint (64-bit key type)
        dict(name="order_48bit_4m", kind="order", scene="room", tris=50_000, n=4_000_003, method="twopoint",
             layout="exact", bits=48, any_hit=False, records=False),
        # a small wavefront's order, origin and direction key
        dict(name="order_20k", kind="order", scene="room", tris=50_000, n=20_011, method="origin_dir",
             layout="exact", bits=32, any_hit=False, records=False),
        # the stages one by one, rays gathered as records, quantised nodes
        dict(name="split_2m", kind="split", scene="room", tris=400_000, n=2_000_000, method="twopoint",
             layout="quantised", bits=32, any_hit=False, records=True),
        # six rooms, two bounces, one launch per stage
        dict(name="batch_6_rooms", kind="batch", scene="room", tris=400_000, n=2_600_017, method="hcc",
             layout="exact", bits=24, any_hit=False, records=False, scenes=6),
        # host buffers above one pipeline chunk: copies overlap kernels
        dict(name="host_6m", kind="host", scene="room", tris=400_000, n=6_000_000, method="hcc",
             layout="exact", bits=32, any_hit=False, records=False),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["bounce"] * 6 + ["order"] * 2 + ["split", "batch", "host"])
    method = rng.choice(["hcc", "hcc", "twopoint", "origin", "origin_dir"] +
                        ([] if kind == "batch" else ["mlhcc"]) + (["nosort"] if kind in ("bounce", "batch", "host") else []))
    case = dict(kind=kind, scene=rng.choice(["room"] * 4 + ["cloud"]), tris=log(10_000, 600_000), n=log(1_024, 8_000_000),
                method=method, layout=rng.choice(["exact", "exact", "quantised", "wide"]),
                bits=rng.choice([16, 24, 30, 32, 32, 48, 64]), any_hit=kind in ("bounce", "host") and rng.random() < 0.25,
                records=kind in ("bounce", "split") and rng.random() < 0.4)
    if method == "mlhcc":
        case["bits"] = rng.choice([16, 32])
    if kind == "batch":
        case["scenes"] = rng.randint(2, 8)
        case["n"] = min(max(case["n"], 8_192), 5_000_000)
        case["bits"] = rng.choice([16, 24, 28, 48])
        case["scene"] = "room"
    if case["n"] > 4096:
        case["n"] |= rng.randint(0, 1)
    return case


# ------------------------------------------------------------------ scenes

_scenes, _points = {}, {}


def _scene(kind, tris, number=0):
    """Host BVH of a case's scene, built once per process."""
    key = (kind, tris, number)
    if key not in _scenes:
        t = gen.random_tris(number, tris) if kind == "cloud" else gen.room_tris(1 + number, tris)
        _scenes[key] = gen.build_bvh(t)
    return _scenes[key]


def _visible(kind, tris, number, n):
    """Visible points of about n / 8 camera pixels: position, normal toward the camera, pixel
    footprint and camera distance, as GPU tensors (the camera belongs to the scene)."""
    pixels = (n + 7) // 8
    h = max(9, math.ceil(math.sqrt(pixels * 9 / 16)))
    w = math.ceil(h * 16 / 9)
    key = (kind, tris, number, w, h)
    if key in _points:
        return _points[key]
    bvh = _scene(kind, tris, number)
    if kind == "cloud":
        eye, target, fov = (0.5, 0.5, -1.2), (0.5, 0.5, 0.5), 45.0
    else:
        eye, target, fov = gen.ROOM_CAMERA
    sec, _, prim = gen.camera_rays(bvh.tris, eye, target, fov, w, h, 1, 7, sample_major=False)
    p = torch.from_numpy(np.ascontiguousarray(sec.org[:, :3])).to(DEV)
    tri = torch.from_numpy(bvh.tris[prim]).to(DEV).double()
    nrm = torch.linalg.cross(tri[:, 3:6] - tri[:, :3], tri[:, 6:] - tri[:, :3])
    nrm = torch.nn.functional.normalize(nrm, dim=1).float()
    to_eye = torch.tensor(eye, device=DEV) - p
    nrm = torch.where(((nrm * to_eye).sum(1) < 0)[:, None], -nrm, nrm)
    foot = to_eye.norm(dim=1) * (2 * math.tan(math.radians(fov) / 2) / h)
    if len(_points) > 8:
        _points.clear()
    _points[key] = (p, nrm, foot)
    return _points[key]


def _rays(case, seed, number=0, n=None, tris=None):
    """n rays (org_tmin, dir_tmax), float32 GPU tensors, drawn from the seed."""
    n = case["n"] if n is None else n
    tris = case["tris"] if tris is None else tris
    per = 2 if case["any_hit"] else 1
    p, nrm, foot = _visible(case["scene"], tris, number, -(-n // per))
    g = torch.Generator(device=DEV)
    g.manual_seed(1000 * seed + number)
    i = torch.arange(n, device=DEV) // (8 * per) % p.shape[0]
    p, nrm, foot = p[i], nrm[i], foot[i]
    # orthonormal basis about the normal
    a = torch.where((nrm[:, :1].abs() > 0.9), torch.tensor([0.0, 1, 0], device=DEV), torch.tensor([1.0, 0, 0], device=DEV))
    b1 = torch.nn.functional.normalize(torch.linalg.cross(a, nrm), dim=1)
    b2 = torch.linalg.cross(nrm, b1)
    jitter = (torch.rand(n, 2, device=DEV, generator=g) - 0.5) * foot[:, None]
    p = p + jitter[:, :1] * b1 + jitter[:, 1:] * b2
    if case["any_hit"]:
        lights = torch.tensor(gen.ROOM_LIGHTS, device=DEV, dtype=torch.float32)
        at = lights[torch.randint(0, 4, (n,), device=DEV, generator=g)]
        at = at + torch.cat([torch.rand(n, 1, device=DEV, generator=g) - 0.5, torch.zeros(n, 1, device=DEV),
                             torch.rand(n, 1, device=DEV, generator=g) - 0.5], 1) * 0.5
        d = at - p
        tmax = d.norm(dim=1, keepdim=True) * (1 - 1e-4)
        d = torch.nn.functional.normalize(d, dim=1)
    else:
        r2 = torch.rand(n, 1, device=DEV, generator=g)
        phi = torch.rand(n, 1, device=DEV, generator=g) * (2 * math.pi)
        r = r2.sqrt()
        d = (r * phi.cos()) * b1 + (r * phi.sin()) * b2 + (1 - r2).sqrt() * nrm
        tmax = torch.full((n, 1), math.inf, device=DEV)
    org = torch.cat([p, torch.full((n, 1), 1e-4, device=DEV)], 1).contiguous()
    return org, torch.cat([d, tmax], 1).contiguous()


def _batch_parts(case):
    """(triangles, rays) of each scene of a batch: mixed sizes that add up to n rays."""
    s = case["scenes"]
    share = [2.0 ** -(k % 4) for k in range(s)]
    ns = [int(case["n"] * w / sum(share)) for w in share]
    ns[-1] += case["n"] - sum(ns)
    return [(max(2_000, case["tris"] >> (k % 3)), ns[k]) for k in range(s)]


# ------------------------------------------------------------- state and pass

class _State:
    """What a program keeps: a context with reserved scratch, BVH and cut handles, buffers."""

    def __init__(self):
        self.ctx = hcc.hcc_create(0)
        self.bvhs, self.cuts, self.batch = [], [], None

    def add_scene(self, case, host_bvh):
        bvh = hcc.hcc_bvh_upload(self.ctx, host_bvh, layout=case["layout"])
        self.bvhs.append(bvh)
        if case["method"] == "hcc":
            self.cuts.append(hcc.hcc_select_cut(self.ctx, bvh, min(case["bits"], 64)))
        elif case["method"] == "mlhcc":
            self.cuts.append(hcc.hcc_select_cut_ml(self.ctx, bvh, case["bits"] // 2, case["bits"] // 2))
        else:
            self.cuts.append(None)

    def __del__(self):
        torch.cuda.synchronize()
        if self.batch is not None:
            hcc.hcc_batch_destroy(self.batch)
        for c in self.cuts:
            if c is not None:
                hcc.hcc_cut_destroy(c)
        for b in self.bvhs:
            hcc.hcc_bvh_destroy(b)
        hcc.hcc_destroy(self.ctx)


def _as_records(org, dir_):
    rec = torch.cat([org, dir_], 1).contiguous()
    return rec[:, :4], rec[:, 4:]


def prepare(case, seed):
    s = _State()
    n, kind = case["n"], case["kind"]
    s.case = case
    s.hits = torch.empty((n, 4), dtype=torch.int32, device=DEV)
    if kind == "batch":
        orgs, dirs, offsets = [], [], [0]
        for k, (tris, m) in enumerate(_batch_parts(case)):
            s.add_scene(case, _scene(case["scene"], tris, k))
            o, d = _rays(case, seed, k, m, tris)
            orgs.append(o)
            dirs.append(d)
            offsets.append(offsets[-1] + m)
        s.org, s.dir = torch.cat(orgs), torch.cat(dirs)
        s.batch = hcc.hcc_batch_create(s.ctx, s.bvhs, s.cuts if case["method"] == "hcc" else None, offsets)
        s.org2, s.dir2 = torch.empty_like(s.org), torch.empty_like(s.dir)
        s.hits2 = torch.empty_like(s.hits)
        s.seed = 12345 + seed
        hcc.hcc_reserve(s.ctx, n, case["bits"] + math.ceil(math.log2(case["scenes"])))
        return s
    s.add_scene(case, _scene(case["scene"], case["tris"]))
    s.org, s.dir = _rays(case, seed)
    if kind == "host":
        def pinned(t):
            return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
        s.org, s.dir, s.hits = pinned(s.org), pinned(s.dir), torch.empty((n, 4), dtype=torch.int32, pin_memory=True)
        return s
    if case["records"] and kind == "bounce":
        s.org, s.dir = _as_records(s.org, s.dir)
    if kind in ("order", "split"):
        s.keys = torch.empty(n, dtype=torch.int32 if case["bits"] <= 32 else torch.int64, device=DEV)
        s.perm = torch.empty(n, dtype=torch.int32, device=DEV)
    if kind == "split":
        s.gathered = torch.empty((n, 8), dtype=torch.float32, device=DEV)
        if not case["records"]:
            s.gathered = torch.empty((2, n, 4), dtype=torch.float32, device=DEV)
        else:
            s.org, s.dir = _as_records(s.org, s.dir)
    if case["method"] != "nosort":
        hcc.hcc_reserve(s.ctx, n, case["bits"])
    return s


def _hits(case, hits):
    if case["any_hit"]:  # which hit is unspecified: what a shadow ray asks is whether there is one
        return {"blocked": hits[:, 0] >= 0}
    return {"prim": hits[:, 0], "tuv": hits.view(torch.float32)[:, 1:]}


def run(s):
    c = s.case
    kind, bits = c["kind"], c["bits"]
    if kind == "bounce":
        hcc.hcc_run(s.ctx, c["method"], s.bvhs[0], s.cuts[0], s.org, s.dir, bits, s.hits, any_hit=c["any_hit"])
        return _hits(c, s.hits)
    if kind == "host":
        hcc.hcc_run_host(s.ctx, c["method"], s.bvhs[0], s.cuts[0], s.org, s.dir, bits, s.hits, any_hit=c["any_hit"])
        return _hits(c, s.hits)
    if kind == "order":
        hcc.hcc_encode(s.ctx, c["method"], s.bvhs[0], s.cuts[0], s.org, s.dir, bits, s.keys)
        hcc.hcc_sort(s.ctx, s.keys, bits, c["n"], s.perm)
        return {"keys": s.keys, "perm": s.perm}
    if kind == "split":
        hcc.hcc_encode(s.ctx, c["method"], s.bvhs[0], s.cuts[0], s.org, s.dir, bits, s.keys)
        hcc.hcc_sort(s.ctx, s.keys, bits, c["n"], s.perm)
        org, dir_ = (s.gathered[:, :4], s.gathered[:, 4:]) if c["records"] else (s.gathered[0], s.gathered[1])
        hcc.hcc_gather(s.ctx, s.org, s.dir, s.perm, org, dir_)
        hcc.hcc_trace(s.ctx, s.bvhs[0], org, dir_, s.hits, scatter=s.perm)
        return {"perm": s.perm, "gathered": s.gathered, **_hits(c, s.hits)}
    hcc.hcc_batch_run(s.ctx, s.batch, c["method"], s.org, s.dir, bits, s.hits)
    hcc.hcc_batch_spawn(s.ctx, s.batch, s.org, s.dir, s.hits, s.seed, 1e-4, s.org2, s.dir2)
    hcc.hcc_batch_run(s.ctx, s.batch, c["method"], s.org2, s.dir2, bits, s.hits2)
    return {"first": _hits(c, s.hits), "org": s.org2, "dir": s.dir2, "second": _hits(c, s.hits2)}


# ---------------------------------------------------------------- expectations

def work(case):
    """Rays read once, outputs written once, geometry read once; the arithmetic of the box and
    triangle tests that a traversal of a BVH2 of this size needs and of the key."""
    n, tris, kind = case["n"], case["tris"], case["kind"]
    key = 8 if case["bits"] > 32 else 4
    boxes = {"hcc": min(case["bits"], 64), "mlhcc": case["bits"]}.get(case["method"], 0)
    encode = 0 if case["method"] == "nosort" else 18 * boxes + 30
    trace = 2 * 18 * 1.8 * math.log2(tris) + 5 * 45
    if kind == "order":
        return {"bytes": n * (32 + key + 4), "flops": n * encode}
    if kind == "split":
        return {"bytes": n * (32 + 4 + 32 + 16) + 68 * tris, "flops": n * (encode + trace)}
    if kind == "batch":
        geometry = sum(68 * t for t, _ in _batch_parts(case))
        return {"bytes": n * (32 + 16 + 32 + 16) + geometry, "flops": 2 * n * (encode + trace)}
    return {"bytes": n * (32 + (1 if case["any_hit"] else 16)) + 68 * tris, "flops": n * (encode + trace)}


def tolerance(case):
    """Every output is a fixed function of the inputs: keys are whole numbers from a stated
    sequence of rounded operations, the permutation is that of a stable sort, a closest hit is the
    smallest (t, triangle id) of a stated Moller-Trumbore sequence whatever order the tree is
    walked in, and spawned rays follow from the hits."""
    return "exact"


def _closest64(case, org, dir_):
    """Closest hits by brute force over all triangles in 64 bits."""
    tri = torch.from_numpy(_scene(case["scene"], case["tris"]).tris).to(DEV).double()
    v0, e1, e2 = tri[:, :3], tri[:, 3:6] - tri[:, :3], tri[:, 6:] - tri[:, :3]
    n = org.shape[0]
    prim = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    tuv = torch.zeros((n, 3), dtype=torch.float64, device=DEV)
    step = max(1, 40_000_000 // v0.shape[0])

    def dot(a, b):
        return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

    def cross(a, b):
        return a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]

    V, A, B = ([x[None, :, k] for k in range(3)] for x in (v0, e1, e2))
    for i in range(0, n, step):
        o, d = org[i:i + step].double(), dir_[i:i + step].double()
        D = [d[:, k, None] for k in range(3)]
        P = cross(D, B)
        inv = 1 / dot(A, P)
        S = [o[:, k, None] - V[k] for k in range(3)]
        u = dot(S, P) * inv
        Q = cross(S, A)
        v = dot(D, Q) * inv
        t = dot(B, Q) * inv
        hit = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > o[:, 3, None]) & (t < d[:, 3, None])
        t = torch.where(hit, t, math.inf)
        best, at = t.min(dim=1)
        met = best < math.inf
        pick = at[:, None]
        prim[i:i + step] = torch.where(met, at, -1).int()
        tuv[i:i + step, 0] = best
        tuv[i:i + step, 1] = torch.where(met, u.gather(1, pick)[:, 0], 0.0)
        tuv[i:i + step, 2] = torch.where(met, v.gather(1, pick)[:, 0], 0.0)
    return {"prim": prim, "tuv": tuv}


def exact(case, seed):
    # brute force: wavefronts and scenes small enough for about 15 G ray-triangle tests
    if case["kind"] not in ("bounce", "host") or case["any_hit"] or case["n"] * case["tris"] > 15_000_000_000:
        return None
    return _closest64(case, *_rays(case, seed))
