"""The work that users of this package have it do, as cases that can be timed.

``listed()`` names the cases, ``draw(rng)`` makes another one of the same
ranges, ``prepare(case, seed)`` makes what a program has in hand before the call
(segments, workspace, outputs, a captured step, a batch, pinned host buffers),
``run(state)`` is one pass through the public entry points, ``work(case)`` the
bytes that pass cannot do without, and ``exact(case, seed)`` the same outputs
from plain torch in 64-bit integers.

A case's ``kind`` is the entry point:
  scene    vox_generate on one scene (count, scan, list and/or volume)
  step     batching.SceneStep: the same as a captured graph on two streams
  batch    batching.make_batch(...).run(): many scenes in one launch sequence
  serve    serving.GpuLauncher: a batch of requests from pinned host memory
  euclid   vox_euclid_generate (the Euclidean-N variant)
  bricked  vox_generate into a brick-major volume, then vox_unbrick
  host     vox_generate_host (host buffers in and out)
and its ``shape`` the segments: ``uniform`` endpoints, ``fixed`` lengths,
``loguniform`` lengths, ``giga`` (pairwise different lengths with a given
total), one ``single`` segment.
"""

import math

import numpy as np
import torch

from paper_2009_09500_gb300 import batching, serving, vox, workloads

EDGE_MAX = 1 << 21


def listed():
    return [
        # one segment of 10^5 voxels (the paper's Table 2 range): the smallest call
        {"name": "segment-100k", "kind": "scene", "shape": "single", "n": 1, "length": 100000, "w": EDGE_MAX,
         "h": EDGE_MAX, "d": EDGE_MAX, "list": 64, "volume": 0},
        # the quick start: a small scene, list and volume, a workspace of vox_workspace_size(n) bytes
        {"name": "scene-4096", "kind": "scene", "shape": "uniform", "n": 4096, "w": 256, "h": 256, "d": 256,
         "list": 32, "volume": 1, "fresh": 1, "bricks": 0},
        # a volume whose rows are not whole words, an odd number of segments, added to what it holds
        {"name": "ragged-volume", "kind": "scene", "shape": "uniform", "n": 60001, "w": 500, "h": 333, "d": 217,
         "list": 32, "volume": 1, "fresh": 0, "bricks": 0},
        # a million segments of 64 voxels (Table 3 shape): list and fresh volume
        {"name": "fixed64-1m", "kind": "scene", "shape": "fixed", "n": 1 << 20, "length": 64, "w": 1024, "h": 1024,
         "d": 1024, "list": 32, "volume": 1, "fresh": 1, "bricks": 1},
        # a list alone of segments of very different lengths
        {"name": "loguniform-300k-list", "kind": "scene", "shape": "loguniform", "n": 300007, "w": 2048, "h": 2048,
         "d": 2048, "list": 64, "volume": 0},
        # 1024 segments, 10^9 voxels (Table 4 shape)
        {"name": "giga-list", "kind": "scene", "shape": "giga", "n": 1024, "length": 10**9, "w": EDGE_MAX,
         "h": EDGE_MAX, "d": EDGE_MAX, "list": 64, "volume": 0},
        # the largest step: 4M segments in 4096^3, list and 8 GiB volume, captured with the list
        # kernel that the autotuner picks for such lengths
        {"name": "loguniform-4m-step", "kind": "step", "shape": "loguniform", "n": 4 << 20, "w": 4096, "h": 4096,
         "d": 4096, "list": 64, "volume": 1, "list_runs": 2},
        # uneven scenes in one launch sequence: lists and volumes
        {"name": "batch-48", "kind": "batch", "shape": "uniform", "scenes": 48, "s_lo": 1000, "s_hi": 100000,
         "list": 32, "volume": 1},
        # a few requests of a serving loop at its size range: volumes alone, segments from the host
        {"name": "serve-5", "kind": "serve", "shape": "uniform", "scenes": 5, "s_lo": 1000, "s_hi": 1000000},
        # the literal Euclidean N: compacted list and fresh volume
        {"name": "euclid-fixed64-1m", "kind": "euclid", "shape": "fixed", "n": 1 << 20, "length": 64, "w": 1024,
         "h": 1024, "d": 1024, "list": 32, "volume": 1, "fresh": 1, "bricks": 1},
        # a volume kept brick by brick, and its export to rows
        {"name": "bricked-1m", "kind": "bricked", "shape": "loguniform", "n": 1000003, "w": 2048, "h": 2048,
         "d": 2048},
        # host buffers in and out: list and volume
        {"name": "host-200k", "kind": "host", "shape": "uniform", "n": 200000, "w": 512, "h": 512, "d": 512,
         "list": 32, "volume": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A row length: whole words two times in three, else any."""
    w = _log(rng, lo, hi)
    return max(32, w // 32 * 32) if rng.random() < 0.67 else w


def draw(rng):
    kind = rng.choice(["scene", "scene", "scene", "step", "batch", "serve", "euclid", "bricked", "host"])
    if kind == "batch":
        return {"kind": kind, "shape": "uniform", "scenes": rng.randint(3, 56), "s_lo": 1000,
                "s_hi": _log(rng, 2000, 100000), "list": rng.choice([0, 32, 64]), "volume": 1}
    if kind == "serve":
        return {"kind": kind, "shape": "uniform", "scenes": rng.randint(1, 8), "s_lo": 1000,
                "s_hi": _log(rng, 5000, 1000000)}
    if kind in ("bricked", "step"):
        edge = 128 * rng.randint(2, 16) if kind == "bricked" else 32 * rng.randint(8, 80)
        c = {"kind": kind, "shape": "loguniform", "n": _log(rng, 3000, 1500000), "w": edge, "h": edge, "d": edge}
        if kind == "step":
            c.update({"list": 64 if edge > 1024 else rng.choice([32, 64]), "volume": rng.choice([0, 1, 1]),
                      "list_runs": rng.choice([0, 2])})
        return c
    if kind in ("euclid", "host"):
        w, h, d = _width(rng, 64, 1024), _log(rng, 64, 1024), _log(rng, 64, 1024)
        return {"kind": kind, "shape": "uniform", "n": _log(rng, 100, 200000), "w": w, "h": h, "d": d,
                "list": rng.choice([32, 64]), "volume": 1, "fresh": 1, "bricks": 1}
    shape = rng.choice(["single", "fixed", "uniform", "uniform", "loguniform", "giga"])
    c = {"kind": kind, "shape": shape, "list": 64, "volume": 0}
    if shape == "single":
        c.update({"n": 1, "length": _log(rng, 1000, 1000000), "w": EDGE_MAX, "h": EDGE_MAX, "d": EDGE_MAX})
    elif shape == "giga":
        c.update({"n": 1024, "length": _log(rng, 3 * 10**8, 10**9), "w": EDGE_MAX, "h": EDGE_MAX,
                  "d": EDGE_MAX})
    elif shape == "fixed":
        length = _log(rng, 20, 200000)
        edge = EDGE_MAX if length > 1000 else 1024
        c.update({"n": max(1, _log(rng, 1000, 1 << 20) * 64 // max(64, length)), "length": length, "w": edge,
                  "h": edge, "d": edge, "list": 64 if edge > 1024 else rng.choice([32, 64])})
    elif shape == "loguniform":
        edge = rng.randint(200, 3000)
        c.update({"n": _log(rng, 1000, 1500000), "w": edge, "h": edge, "d": edge})
    else:
        w, h, d = _width(rng, 64, 1024), _log(rng, 64, 1024), _log(rng, 64, 1024)
        c.update({"n": _log(rng, 100, 200000), "w": w, "h": h, "d": d, "list": rng.choice([0, 32, 32, 64]),
                  "volume": 1, "fresh": rng.choice([0, 1]), "bricks": rng.choice([0, 1])})
    return c


# ------------------------------------------------------------------- inputs
def _moved(segs, dims, seed):
    """The segments in another order, each mirrored along axes taken at random: as many
    voxels in all, so that the outputs of every seed have one size."""
    rng = np.random.default_rng(seed)
    segs = segs[rng.permutation(len(segs))]
    for a, edge in enumerate(dims):
        flip = rng.random(len(segs)) < 0.5
        for col in (a, a + 3):
            segs[flip, col] = edge - 1 - segs[flip, col]
    return np.ascontiguousarray(segs)


def _segments(case, seed, n=None):
    """The case's segments (numpy int32 [n, 6]) from the seed alone."""
    n = case["n"] if n is None else n
    shape, dims = case["shape"], _dims(case)
    if shape == "single":
        return workloads.sweep_single(case["length"], seed=seed, edge=case["w"]).segs
    if shape == "giga":
        return workloads.sweep_giga(case["length"], n=case["n"], seed=seed, edge=case["w"]).segs
    if shape == "fixed":
        if case["kind"] != "euclid":
            return workloads.sweep_fixed(case["length"], n=n, seed=seed, edge=case["w"]).segs
        segs = workloads.sweep_fixed(case["length"], n=n, edge=case["w"]).segs
    elif shape == "loguniform":
        segs = workloads.config3(n=n, edge=case["w"]).segs
    else:
        segs = workloads.uniform_segments(np.random.default_rng(0), n, dims)
    return _moved(segs, dims, seed)


def _dims(case):
    return (case["w"], case["h"], case["d"])


def _scenes(case, seed):
    """Scenes of a batch, or the requests of a serving loop (workloads.Workload)."""
    if case["kind"] == "batch":
        got = workloads.config4(n_scenes=case["scenes"], s_lo=case["s_lo"], s_hi=case["s_hi"])
    else:
        got = [r.workload() for r in workloads.config5(s_lo=case["s_lo"], s_hi=case["s_hi"],
                                                       max_requests=case["scenes"])]
    return [workloads.Workload(w.name, _moved(w.segs, w.dims, [seed, k]), w.dims) for k, w in enumerate(got)]


def _flags(case):
    f = {0: 0, 32: vox.OUT_LIST32, 64: vox.OUT_LIST64}[case["list"]]
    if case["volume"]:
        f |= vox.OUT_BITMASK
        if case.get("fresh", 1):
            f |= vox.OUT_FRESH
    return f


def _list(case, V, **kw):
    if not case["list"]:
        return None
    return torch.zeros(max(V, 1), dtype=torch.int64 if case["list"] == 64 else torch.int32, **kw)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        s["batch"] = batching.make_batch(_scenes(case, seed), _flags(case))
        return s
    if kind == "serve":
        s["reqs"] = [serving.ServeRequest(rid=i, arrival_s=0.0, n=w.n, dims=w.dims,
                                          segs_host=torch.from_numpy(w.segs).pin_memory())
                     for i, w in enumerate(_scenes(case, seed))]
        s["launcher"], s["slot"] = serving.GpuLauncher(4), 0
        return s
    dims = s["dims"] = _dims(case)
    segs_np = _segments(case, seed)
    n = len(segs_np)
    segs = s["segs"] = vox.segments_tensor(segs_np)
    if kind == "step":
        # the launch tuning that the autotuner left, in force while the step is captured
        vox.vox_set_tuning(list_runs=case["list_runs"])
        s["step"] = batching.SceneStep(segs, dims, vox.OUT_LIST64 if case["list"] == 64 else vox.OUT_LIST32,
                                       volume=bool(case["volume"]))
        vox.vox_reset_tuning()
        return s
    status = s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    words = vox.vox_mask_words(dims)
    if kind == "euclid":
        ws = torch.empty(vox.vox_euclid_workspace_size_volume(n, dims, 0), dtype=torch.uint8, device="cuda")
        V, _, P = vox.vox_euclid_plan(segs, dims, ws, status, with_pieces=True)
        s["ws"] = torch.empty(vox.vox_euclid_workspace_size_volume(n, dims, P), dtype=torch.uint8, device="cuda")
        s["offsets"] = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    else:
        ws = torch.empty(vox.vox_workspace_size_volume(n, dims, 0), dtype=torch.uint8, device="cuda")
        V, P = vox.vox_plan(segs, dims, ws, status)
        if kind == "host":
            f = _flags(case) & ~vox.OUT_FRESH
            s["segs"] = torch.from_numpy(segs_np).pin_memory()
            s["list"] = _list(case, V, pin_memory=True)
            s["mask"] = torch.zeros(words, dtype=torch.int32, pin_memory=True)
            s["arena"] = torch.empty(vox.vox_host_arena_size_volume(n, dims, f, V, P), dtype=torch.uint8,
                                     device="cuda")
            return s
        if kind == "bricked":
            s["ws"] = torch.empty(vox.vox_workspace_size_volume(n, dims, P), dtype=torch.uint8, device="cuda")
            s["bricked"] = torch.zeros(vox.vox_mask_words_bricked(dims), dtype=torch.int32, device="cuda")
            s["mask"] = torch.zeros(words, dtype=torch.int32, device="cuda")
            return s
        size = vox.vox_workspace_size_volume(n, dims, P) if case.get("bricks") else vox.vox_workspace_size(n)
        s["ws"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    s["list"] = _list(case, V, device="cuda")
    s["mask"] = torch.zeros(words, dtype=torch.int32, device="cuda") if case["volume"] else None
    s["flags"] = _flags(case)
    return s


# -------------------------------------------------------------------- a pass
def run(s):
    kind = s["kind"]
    if kind == "scene":
        vox.vox_generate(s["segs"], s["dims"], s["ws"], s["status"], s["list"], s["mask"], s["flags"])
        return {"list": s["list"], "volume": s["mask"], "status": s["status"]}
    if kind == "step":
        s["step"].replay()
        return {"list": s["step"].lst, "volume": s["step"].mask, "status": s["step"].status}
    if kind == "batch":
        b = s["batch"]
        b.run()
        return {"list": b.lst, "volumes": b.masks, "base": b.scene_base, "status": b.status}
    if kind == "serve":
        s["slot"] = (s["slot"] + 1) % 4
        h = s["launcher"](s["reqs"], s["slot"])
        return {"volumes": h.keep["masks"], "base": h.keep["base"], "status": h.keep["status"]}
    if kind == "euclid":
        vox.vox_euclid_generate(s["segs"], s["dims"], s["ws"], s["status"], s["list"], s["mask"], s["flags"],
                                s["offsets"])
        return {"list": s["list"], "volume": s["mask"], "offsets": s["offsets"], "status": s["status"]}
    if kind == "bricked":
        vox.vox_generate(s["segs"], s["dims"], s["ws"], s["status"], None, s["bricked"],
                         vox.OUT_BITMASK | vox.OUT_BRICKED)
        vox.vox_unbrick(s["bricked"], s["dims"], s["mask"], status=s["status"])
        return {"volume": s["mask"], "bricked": s["bricked"], "status": s["status"]}
    V = vox.vox_generate_host(s["segs"], s["dims"], s["arena"], s["list"], s["mask"])
    return {"list": s["list"], "volume": s["mask"], "voxels": V}


# ---------------------------------------------------------------- its bytes
def _mean_voxels(segs, euclid=False):
    if euclid:  # a few segments sampled as the variant does
        return len(_voxels(torch.from_numpy(segs[:512]), True)[0]) / min(len(segs), 512)
    d = np.abs(segs[:, 3:].astype(np.int64) - segs[:, :3])
    return float(d.max(axis=1).mean()) + 1.0


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        bytes_ = 0.0
        for w in _scenes(case, 1):
            bytes_ += 24 * w.n + w.dims[0] * w.dims[1] * w.dims[2] // 8
            bytes_ += case.get("list", 0) // 8 * w.n * _mean_voxels(w.segs[:4096])
        return {"bytes": float(bytes_), "flops": 0.0}
    segs = _segments(case, 1, None if case["shape"] in ("single", "giga") else min(case["n"], 1 << 14))
    voxels = case["n"] * _mean_voxels(segs, kind == "euclid")
    volume = case["w"] * case["h"] * case["d"] / 8
    bytes_ = 24 * case["n"] + case.get("list", 0) / 8 * voxels
    if kind == "euclid":
        bytes_ += 8 * case["n"]
    if kind == "bricked":  # the volume written, then read and written again
        bytes_ += 3 * volume
    elif case["volume"]:  # OR-ed into: the 32-byte sectors touched are read and written
        bytes_ += volume if case.get("fresh", 1) else min(2 * volume, 64 * voxels)
    return {"bytes": float(bytes_), "flops": 0.0}


# ------------------------------------------------------- in plain torch, 64 bits
def _voxels(segs, euclid=False):
    """(voxels int64 [V, 3], first voxel of every segment) of int32 [n, 6] segments."""
    p = segs.to(torch.int64)
    d = p[:, 3:] - p[:, :3]
    if euclid:
        sq = (d * d).sum(1)
        N = sq.double().sqrt().to(torch.int64)
        N = N - (N * N > sq).to(torch.int64)
        N = N + ((N + 1) * (N + 1) <= sq).to(torch.int64)
    else:
        N = d.abs().max(1).values
    ends = torch.cumsum(N + 1, 0)
    first = ends - (N + 1)
    seg = torch.repeat_interleave(torch.arange(len(p), device=p.device), N + 1)
    k = torch.arange(int(ends[-1]), device=p.device) - first[seg]
    Ns = N[seg][:, None]
    q = (2 * k[:, None] * d[seg].abs() + Ns) // (2 * Ns).clamp(min=1)
    v = p[seg, :3] + d[seg].sign() * q
    if not euclid:
        return v, first
    keep = torch.ones(len(v), dtype=torch.bool, device=v.device)
    keep[1:] = (k[1:] == 0) | (v[1:] != v[:-1]).any(1)
    at = torch.cumsum(keep.to(torch.int64), 0) - 1
    return v[keep], at[first]


def _scene_exact(segs_np, dims, bits, volume, euclid=False):
    """(list or None, volume or None, offsets with the total) of one scene."""
    w, h, d = dims
    lists, offs, total = [], [], 0
    vol = torch.zeros((w * h * d + 31) // 32 * 32, dtype=torch.uint8, device="cuda") if volume else None
    n = max(1, (1 << 23) // max(1, int(np.abs(segs_np[:, 3:].astype(np.int64) - segs_np[:, :3]).max()) + 1))
    for a in range(0, len(segs_np), n):
        v, first = _voxels(torch.from_numpy(segs_np[a:a + n]).cuda(), euclid)
        offs.append(first + total)
        total += len(v)
        if bits:
            sh = 10 if bits == 32 else 21
            packed = v[:, 0] | v[:, 1] << sh | v[:, 2] << 2 * sh
            lists.append(packed if bits == 64 else packed.to(torch.int32))
        if volume:
            vol[v[:, 0] + w * (v[:, 1] + h * v[:, 2])] = 1
    words = None
    if volume:
        words = torch.zeros(len(vol) // 32, dtype=torch.int32, device="cuda")
        for b in range(32):
            words |= vol[b::32].to(torch.int32) << b
    offs.append(torch.tensor([total], device="cuda"))
    return torch.cat(lists) if bits else None, words, torch.cat(offs)


def exact(case, seed):
    kind = case["kind"]
    status = torch.zeros(1, dtype=torch.int32)
    if kind in ("batch", "serve"):
        got = [_scene_exact(w.segs, w.dims, case.get("list", 0), True) for w in _scenes(case, seed)]
        base = torch.cumsum(torch.tensor([0] + [int(g[2][-1]) for g in got]), 0)
        out = {"volumes": [g[1] for g in got], "base": base, "status": status}
        if kind == "batch":
            out["list"] = torch.cat([g[0] for g in got]) if case["list"] else None
        return out
    if work(case)["bytes"] > 3e9:  # too much for a few seconds
        return None
    segs, dims = _segments(case, seed), _dims(case)
    lst, words, offs = _scene_exact(segs, dims, case.get("list", 0), bool(case.get("volume", 1)), kind == "euclid")
    if kind == "bricked":
        return {"volume": words, "bricked": None, "status": status}
    if kind == "host":
        return {"list": lst, "volume": words, "voxels": int(offs[-1])}
    out = {"list": lst, "volume": words, "status": status}
    if kind == "euclid":
        out["offsets"] = offs
    return out
